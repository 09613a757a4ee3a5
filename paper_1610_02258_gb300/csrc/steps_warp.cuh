// The operator-split step on warp tiles: 32 consecutive tets per warp, one
// per lane, for models with up to kWarpMaxSpecies species. Included after
// steps_step.cuh, whose building blocks it shares; every draw, formula and
// decision is the block-tile step's, so both give the same bits.
//
// Why a warp owns its tets from load to apply: the block-tile step packs the
// reacting tets of 256 or 512 into dense chunks, which costs four block
// barriers per tile (its largest stall) and walks species sets with one
// branchy loop per lane. Here nothing waits for another warp, the loops over
// species are unrolled with the model's species count as a constant, and
// what only some lanes need (occupancy rounding, Philox blocks, bit-plane
// groups, movers) is queued in the warp's shared memory and worked off 32 at
// a time.
//
// What bounds it: instruction issue. On the 294,780-tet box (14 to 18
// molecules per tet, 0.07 events per tet and window) a window is about 24M
// warp instructions, issued at two thirds of the slots; loading and applying
// alone take 7 us. us per window, block tiles -> warp tiles, flow launches:
// box 42.7 -> 28.6, at a tenth of the densities 24.0 -> 15.3, at ten times
// 139 -> 102; 1.05M tets in window launches 94 -> 65. Registers: 64 at 32
// warps per SM; 48 at 40 warps spilled and was 10 % slower. Items per warp
// instead of per block (warps out of step) missed the instruction cache: 35
// us on the box.
#pragma once

#include "steps_step.cuh"

namespace steps {
namespace {

// Philox4x32-10 with the round keys given: they are operands of the rounds'
// three-input XORs (constant bank in a plain launch), 18 instructions fewer
// per block, of about 65, than adding the Weyl constants each time.
__device__ __forceinline__ uint4 philox_rk(const uint4 *rk, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t k0 = (r & 1) ? rk[r >> 1].z : rk[r >> 1].x, k1 = (r & 1) ? rk[r >> 1].w : rk[r >> 1].y;
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c0 = n0;
        c1 = (uint32_t)p1;
        c2 = n2;
        c3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// floor(A R / 2^31): a cumulative face threshold (2^31 fixed point).
__device__ __forceinline__ uint32_t thr31(uint32_t A, uint32_t R) { return (uint32_t)(((uint64_t)A * R) >> 31); }

// round_trials in 64-bit integers. nbar = mant 2^-sh, f its fraction's sh
// bits: u < f 2^-sh with u = (2w + 1) 2^-33 means (2w + 1) 2^sh < f 2^33, that
// is 2w + 1 < f 2^(33 - sh) for sh <= 33 and, with k = sh - 33 and f >= 1,
// 2w + 1 <= floor((f - 1) / 2^k) beyond.
__device__ __forceinline__ int32_t round_trials32(double nbar, uint32_t w, int32_t most) {
    const uint64_t bits = (uint64_t)__double_as_longlong(nbar);
    const int e = (int)(bits >> 52);
    if (e == 0 || e >= 0x800) return 0;  // zero (or negative, not reached): no trials
    const uint64_t mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = 1075 - e;             // fraction bits of mant
    if (sh <= 20) return most;           // nbar >= 2^32: above every count
    uint64_t fl = 0, f = mant;
    if (sh < 64) {
        fl = mant >> sh;
        f = mant & ((1ull << sh) - 1);
    }
    const uint64_t u = 2ull * w + 1ull;
    const int k = sh - 33;
    const bool up = k <= 0 ? u < (f << -k) : f != 0 && k < 64 && u <= ((f - 1) >> k);
    fl += up ? 1u : 0u;
    return fl > (uint64_t)most ? most : (int32_t)fl;
}

// Model access for models given at run time: the reaction table, walked in a
// loop; the running sums are summed again for a pick instead of kept
// (unrolled by four, or with the sums kept, the loops were slower). 30,720
// tets at 151 molecules each, us per window: block tiles 79.7, this 63.8
// (compiled for the model 43); the 1,920-tet cuboid 9.7 -> 7.4.
struct RtWarp {
    static constexpr bool kExpLeave = false;
    __device__ static int S(const ModelDev &m) { return m.S; }
    __device__ static int R(const ModelDev &m) { return m.R; }
    __device__ static uint32_t diffusive(const ModelDev &m) { return m.diffusive; }
    template <int THREADS>
    __device__ static void build(const ModelDev &m, RxnTab &tb) {
        if (threadIdx.x < THREADS) build_rxn_tab<THREADS, 32>(m, tb);
    }
    template <class F>
    __device__ static void for_changes(const RxnTab &tb, int r, F f) {
        RtModel<false>::for_changes(tb, r, f);
    }
    template <int RM>
    __device__ __forceinline__ static float sums(const RxnTab &tb, const ModelDev &m, const int32_t *cnt, float inv_nav,
                                                 uint32_t active, bool, float *) {
        const bool z = m.order0 != 0u;
        float a0 = 0.0f;
#pragma unroll 2
        for (int r = 0; r < m.R; ++r)
            a0 = __fadd_rn(a0, ((active >> r) & 1u) ? propensity(tb.p[r], cnt, inv_nav, z) : 0.0f);
        return a0;
    }
    template <int RM>
    __device__ __forceinline__ static float first_sums(const RxnTab &tb, const ModelDev &m, const int32_t *cnt,
                                                       float inv_nav, uint32_t active, bool masked, float *psum) {
        const float a0 = sums<RM>(tb, m, cnt, inv_nav, active, masked, psum);
        if (a0 <= kPlainSums) return a0;
        return careful_sums(tb, m, cnt, inv_nav, active, nullptr);
    }
    template <int RM>
    __device__ __forceinline__ static int pick(const RxnTab &tb, const ModelDev &m, const float *, float target,
                                               const int32_t *cnt, float inv_nav, uint32_t active) {
        const bool z = m.order0 != 0u;
        float sum = 0.0f;
        for (int r = 0; r < m.R; ++r) {
            sum = __fadd_rn(sum, ((active >> r) & 1u) ? propensity(tb.p[r], cnt, inv_nav, z) : 0.0f);
            if (sum > target) return r;
        }
        // no sum exceeds the target, or the sums met an infinite rate of an
        // absent reactant and are not numbers from there on
        return careful_pick(tb, m, cnt, inv_nav, active, target);
    }
};

// The species factor of tet i's thresholds: the window's species scale R_s
// (EULER), or the tet's own leave value from the EXP table.
template <class P>
__device__ __forceinline__ uint32_t warp_R(const StepArgs &a, const uint32_t *s_scale, int s, int64_t i) {
    if constexpr (P::kExpLeave) return __ldg(a.leave + (size_t)((uint64_t)(uint32_t)s * (uint32_t)a.Tpad) + (size_t)i);
    else return s_scale[s];
}

// An attempt certain to end the window: -ln u >= 1 - u, so a waiting time of
// at least (1 - u) / a0 beyond tau_k needs neither the logarithm nor the
// division (the factor covers their rounding and that of the products).
__device__ __forceinline__ bool attempt_over(float u1, float a0, float tau_dn) {
    return __fmul_rn(__fsub_rn(1.0f, u1), 0.9999f) > __fmul_rn(a0, tau_dn);
}

// The SSA of one tet from its second event on (ssa_tet; counts in the lane's
// column of the warp tile, the first event already applied). An attempt
// whose waiting time alone exceeds the window ends it in float:
// (double)dt > tau_k <=> dt > tau_dn.
template <int RM, class P>
__device__ __forceinline__ uint32_t ssa_lane(const RxnTab &tb, const ModelDev &m, const StepArgs &a, int32_t *cnt,
                                             uint32_t tet, uint32_t c0, uint32_t c3, float inv_nav, uint32_t active,
                                             int pick0, float dt0, double *O, double *tS, uint32_t &touched) {
    double dt_acc = (double)dt0;
    P::for_changes(tb, pick0, [&](int s, int d) {
        O[s] = __dmul_rn((double)(cnt[s * 32] - d), dt_acc);
        tS[s] = dt_acc;
    });
    for (uint32_t j = 1;; ++j) {
        asm volatile("" ::: "memory");  // keep the reaction table out of registers across iterations
        const uint4 w = philox_rk(a.rk, c0, tet, j, (kPurposeReac << 28) | c3);
        float psum[RM];
        const float a0 = P::template sums<RM>(tb, m, cnt, inv_nav, active, a.rmask != nullptr, psum);
        if (!(a0 > 0.0f)) break;
        if (j >= kMaxEventsPerWindow) return 2u;  // pathological rates: stop and report, never spin
        const float u1 = unit24f(w.x);
        if (attempt_over(u1, a0, a.tau_dn)) break;
        const float dt = __fdiv_rn(-steps_logf(u1), a0);
        if (dt > a.tau_dn) break;
        const double dt_new = __dadd_rn(dt_acc, (double)dt);
        if (dt_new > a.tau_k) break;
        const int pick = P::template pick<RM>(tb, m, psum, __fmul_rn(unit24f(w.y), a0), cnt, inv_nav, active);
        if (pick < 0) break;
        dt_acc = dt_new;
        P::for_changes(tb, pick, [&](int s, int d) {
            const int32_t nn = cnt[s * 32];
            if ((touched >> s) & 1u) O[s] = __dadd_rn(O[s], __dmul_rn((double)nn, __dsub_rn(dt_acc, tS[s])));
            else O[s] = __dmul_rn((double)nn, dt_acc);
            tS[s] = dt_acc;
            touched |= 1u << s;
            cnt[s * 32] = nn + d;
        });
    }
    return 0u;
}

// Up to 32 queued (tet, species) pairs, one per lane: the trial count of a
// species a reaction changed (trial_count).
template <int SM>
__device__ __forceinline__ void round_pairs(const StepArgs &a, WarpTile<SM> &w, int first, int n, uint32_t c0,
                                            uint32_t c3) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint32_t ls = w.r.ls[first + lane];
        const int t = (int)(ls & 31u), s = (int)((ls >> 5) & 31u);
        const int32_t N = w.cnt[s][t];
        const uint64_t ob = w.r.O[first + lane], tb = w.r.tS[first + lane];
        double tS = __longlong_as_double((long long)tb), O = __longlong_as_double((long long)ob);
        if (ls >> 15) {  // one event, at a float time, changed N - d to N
            tS = (double)__uint_as_float((uint32_t)tb);
            O = __dmul_rn((double)(N - (int32_t)(uint32_t)ob), tS);
        }
        const double occ = __dadd_rn(O, __dmul_rn((double)N, __dsub_rn(a.tau_k, tS)));
        const double nbar = __dmul_rn(occ, a.inv_tau_k);
        const uint4 rb = philox_rk(a.rk, c0, w.tet[t], (uint32_t)(s >> 2), (kPurposeRound << 28) | c3);
        w.trial[s][t] = round_trials32(nbar, word_of(rb, (uint32_t)(s & 3)), N);
    }
}

// Up to 32 queued movers, one per lane: the face (face f when
// T_{f-1} <= x < T_f), one molecule into the neighbour's entry of nxt, one
// less in the tet.
template <int SM, class P>
__device__ __forceinline__ void move_out(const StepArgs &a, WarpTile<SM> &w, int32_t *nxt, const uint32_t *s_scale,
                                         int64_t i0, int first, int n) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint2 e = w.d.q[first + lane];
        const uint32_t x = e.x;
        const int t = (int)(e.y & 31u), s = (int)(e.y >> 5);
        const uint4 A = w.thr[t];
        const uint32_t R = warp_R<P>(a, s_scale, s, i0 + t);
        const int f = (x >= thr31(A.x, R)) + (x >= thr31(A.y, R)) + (x >= thr31(A.z, R));
        const uint32_t nb = (uint32_t)reinterpret_cast<const int32_t *>(w.nbr + t)[f];
        atomicAdd(nxt + ((uint64_t)(uint32_t)s * (uint32_t)a.Tpad + nb), 1);
        atomicSub(&w.cnt[s][t], 1);
    }
}

// The bit-plane draws of bulk_species for group g of species s: bit j of l[f]
// says that molecule 32 g + j is below threshold T_f. Called by the lanes of
// `lanes`. Planes above every lane's last threshold (slow species leave with a
// per cent or so) settle the molecules with a bit there, for all thresholds
// alike: four planes in six operations instead of eighty.
__device__ __forceinline__ void plane_group(uint32_t lanes, const StepArgs &a, const uint4 A, uint32_t R, uint32_t M, uint32_t g,
                                            uint32_t tet, int s, uint32_t c0, uint32_t c3, uint32_t l[4]) {
    const uint32_t m = min(32u, M - 32u * g);
    const uint32_t valid = m == 32u ? 0xFFFFFFFFu : (1u << m) - 1u;
    uint32_t T0, T1, T2, T3;
    species_thresholds(A, R, T0, T1, T2, T3);
    const uint32_t c3b = (kPurposeBulk << 28) | ((uint32_t)s << 23) | (c3 & 0x007FFFFFu);
    // T_f = 2^31: every x < T_f; T_f = 0: none
    uint32_t l0 = T0 >= 0x80000000u ? valid : 0u, u0 = (T0 >= 0x80000000u || T0 == 0u) ? 0u : valid;
    uint32_t l1 = T1 >= 0x80000000u ? valid : 0u, u1 = (T1 >= 0x80000000u || T1 == 0u) ? 0u : valid;
    uint32_t l2 = T2 >= 0x80000000u ? valid : 0u, u2 = (T2 >= 0x80000000u || T2 == 0u) ? 0u : valid;
    uint32_t l3 = T3 >= 0x80000000u ? valid : 0u, u3 = (T3 >= 0x80000000u || T3 == 0u) ? 0u : valid;
    const uint32_t zeros = __reduce_min_sync(lanes, (uint32_t)max(0, __clz((int)T3) - 1)) / 4u;
    for (uint32_t blk = 0; blk < 8u && (u0 | u1 | u2 | u3); ++blk) {
        const uint4 r = philox_rk(a.rk, c0, tet, (g << 3) | blk, c3b);
        const int sh = 30 - 4 * (int)blk;
        if (blk < zeros && blk < 7u) {
            const uint32_t rest = ~(r.x | r.y | r.z | r.w);
            u0 &= rest;
            u1 &= rest;
            u2 &= rest;
            u3 &= rest;
            continue;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q < 3 || blk < 7u) {  // 31 planes
                const uint32_t Rw = word_of(r, (uint32_t)q);
                plane_compare(T0, sh - q, Rw, u0, l0);
                plane_compare(T1, sh - q, Rw, u1, l1);
                plane_compare(T2, sh - q, Rw, u2, l2);
                plane_compare(T3, sh - q, Rw, u3, l3);
            }
        }
        // a molecule that stays needs no face
        const uint32_t may = u3 | l3;
        u0 &= may;
        u1 &= may;
        u2 &= may;
    }
    l[0] = l0;
    l[1] = l1;
    l[2] = l2;
    l[3] = l3;
}

// Up to 32 queued groups of 32 trial molecules, one per lane.
template <int SM, class P>
__device__ __forceinline__ void plane_groups(const StepArgs &a, WarpTile<SM> &w, int32_t *nxt, const uint32_t *s_scale,
                                             int64_t i0, int first, int n, uint32_t c0, uint32_t c3) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint2 e = w.d.q[first + lane];
        const int t = (int)(e.y & 31u), s = (int)(e.y >> 5);
        uint32_t l[4];
        plane_group(n == 32 ? 0xFFFFFFFFu : (1u << n) - 1u, a, w.thr[t], warp_R<P>(a, s_scale, s, i0 + t), (uint32_t)w.trial[s][t], e.x, w.tet[t], s, c0, c3, l);
        // cumulative thresholds: l[0] within l[1] within l[2] within l[3]
        const int32_t n0 = __popc(l[0]), n1 = __popc(l[1] & ~l[0]), n2 = __popc(l[2] & ~l[1]), n3 = __popc(l[3] & ~l[2]);
        const int4 nb = w.nbr[t];
        int32_t *row = nxt + (uint64_t)(uint32_t)s * (uint32_t)a.Tpad;
        if (n0) atomicAdd(row + nb.x, n0);
        if (n1) atomicAdd(row + nb.y, n1);
        if (n2) atomicAdd(row + nb.z, n2);
        if (n3) atomicAdd(row + nb.w, n3);
        if (l[3]) atomicSub(&w.cnt[s][t], n0 + n1 + n2 + n3);
    }
}

// The species of word v of a tet: how many species end at or before v. pre
// holds the words up to and including each species, a byte each, below 128;
// v's byte with the top bit set, minus that, keeps the top bit where v has
// reached it (no borrow between bytes). Rows past the last species hold 0x80,
// which no word reaches; with 32 species there is no such row, and a word past
// the tet's last molecule gives 32 (kScaleEntries). (The byte dot product __dp4a in place of the shifts
// and the population count took three times the instructions on this GPU.)
template <int NP>
__device__ __forceinline__ uint32_t species_of(const uint32_t *pre, uint32_t v4) {
    uint32_t u = (v4 - pre[0]) & 0x80808080u;
#pragma unroll
    for (int j = 1; j < NP; ++j) u |= ((v4 - pre[j]) >> j) & (0x80808080u >> j);
    return (uint32_t)__popc(u);
}

// The same for a tet of 128 words or more, species by species, from its trial
// counts (trial: its column).
__device__ __forceinline__ uint32_t species_of_wide(const int32_t *trial, int S, uint32_t v) {
    uint32_t end = 0;
    int c = 0;
    for (; c < S - 1; ++c) {
        const int32_t M = trial[c * 32];
        end += M < kBulkMin ? (uint32_t)M : 0u;
        if (v < end) break;
    }
    return (uint32_t)c;
}

// The listed Philox blocks, n of them, 32 at a time, one per lane: word v
// decides a tet's trial molecule v; below the species' last threshold it
// moves, else it stays. About one in seven moves on the benchmark box, so a
// lane only tests the last threshold; movers are queued and find their face
// 32 at a time. The code of a word is free of branches: short-circuit tests
// and a lane guard around the block cost twice the instructions, half of them
// control flow.
template <int SM, class P, bool WIDE>
__device__ __forceinline__ void draw_words(const ModelDev &m, const StepArgs &a, WarpTile<SM> &w, int32_t *nxt,
                                           const uint32_t *s_scale, int64_t i0, uint32_t n, uint32_t c0, uint32_t c3) {
    constexpr int NP = (SM + 3) / 4;
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
    int nq = 0;
    for (uint32_t b = 0; b < n; b += 32) {
        const uint32_t o = w.d.map[min(b + lane, n - 1u)];
        const int t = (int)(o & 31u);
        const uint32_t k = o >> 5, v4 = k * 0x04040404u + 0x80808080u;
        constexpr int NQ = WarpTile<SM>::kPre;
        uint32_t pre[4 * NQ];
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const uint4 x = w.pre[t][j];
            pre[4 * j] = x.x, pre[4 * j + 1] = x.y, pre[4 * j + 2] = x.z, pre[4 * j + 3] = x.w;
        }
        const int left = b + lane < n ? (int)(pre[4 * NQ - 1] - 4u * k) : 0;  // words that decide a molecule
        const uint32_t Aw = w.thr[t].w;
        const uint4 rw = philox_rk(a.rk, c0, w.tet[t], k, (kPurposeDiff << 28) | c3);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            uint32_t c;
            if constexpr (WIDE) c = species_of_wide(&w.trial[0][t], P::S(m), 4u * k + r);
            else c = species_of<NP>(pre, v4 + r * 0x01010101u);
            if constexpr (P::kExpLeave) c = min(c, (uint32_t)P::S(m) - 1u);  // (a word past the last molecule)
            const uint32_t x = word_of(rw, (uint32_t)r) >> 1;
            const bool moves = (r < left) & (x < thr31(Aw, warp_R<P>(a, s_scale, (int)c, i0 + t)));
            const uint32_t mv = __ballot_sync(0xFFFFFFFFu, moves);
            const int pos = nq + __popc(mv & below);
            if (moves) w.d.q[pos] = make_uint2(x, (uint32_t)t | (c << 5));
            nq += __popc(mv);
        }
        // one copy of the movers' code: full sets of lanes, and the rest after the last block
        const int keep = b + 32 < n ? 31 : 0;
        if (nq > keep) {
            __syncwarp();
            do {
                const int take = min(nq, 32);
                nq -= take;
                move_out<SM, P>(a, w, nxt, s_scale, i0, nq, take);
            } while (nq > keep);
            __syncwarp();
        }
    }
    __syncwarp();
}

template <int SM, class P>
__device__ __noinline__ void draw_words_wide(const ModelDev &m, const StepArgs &a, WarpTile<SM> &w, int32_t *nxt,
                                             const uint32_t *s_scale, int64_t i0, uint32_t n, uint32_t c0, uint32_t c3) {
    draw_words<SM, P, true>(m, a, w, nxt, s_scale, i0, n, c0, c3);
}

// Every species' trial count into w.trial, as draw_words_wide reads them: those
// in the word stream, 0 for the others, bit-plane species (bm) as they are.
// round: species whose trial count is there already.
template <int SM, class P>
__device__ __noinline__ void wide_trials(const ModelDev &m, const StepArgs &a, WarpTile<SM> &w, const uint32_t *s_scale,
                                         int64_t i, uint32_t Aw, uint32_t bm, uint32_t round) {
    const int lane = threadIdx.x & 31;
    for (int s = 0; s < P::S(m); ++s) {
        if ((bm >> s) & 1u) continue;
        int32_t M = (round >> s) & 1u ? w.trial[s][lane] : w.cnt[s][lane];
        if (!((P::diffusive(m) >> s) & 1u) || thr31(Aw, warp_R<P>(a, s_scale, s, i)) == 0u) M = 0;
        w.trial[s][lane] = max(M, 0);
    }
}

// Waits until the warp tiles holding the lanes' face neighbours, and the
// warp's own (word `own`, the tile of device tets i0 on), have published
// window word `need` (flow_deps_wait without lists: a lane checks the tiles
// of its own four neighbours, so that a simulation needs no table of
// neighbouring tiles). Relaxed loads, four in flight per lane, then one fence.
__device__ __forceinline__ bool flow_nbr_wait(const uint32_t *done, uint32_t own, int64_t i0, const int4 nb,
                                              uint32_t need, long long limit = 2ll << 30) {
    const uint32_t *base = done + own - (uint32_t)(i0 >> 5);
    const uint32_t *p[4] = {nb.x < 0 ? done + own : base + (nb.x >> 5), nb.y < 0 ? done + own : base + (nb.y >> 5),
                            nb.z < 0 ? done + own : base + (nb.z >> 5), nb.w < 0 ? done + own : base + (nb.w >> 5)};
    uint32_t v[5];
#pragma unroll
    for (int k = 0; k < 5; ++k)
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v[k]) : "l"(k < 4 ? p[k] : done + own) : "memory");
    uint32_t open = 0u;  // words not seen done yet: a lane reads only those again
#pragma unroll
    for (int k = 0; k < 5; ++k) open |= (int32_t)(v[k] - need) >= 0 ? 0u : 1u << k;
    if (!__all_sync(0xFFFFFFFFu, open == 0u)) {
        const long long t0 = clock64();
        uint32_t ns = 32;
        do {
            if (__any_sync(0xFFFFFFFFu, clock64() - t0 > limit)) return false;
            // every waiting warp polls: back off, so that the ones at work are not held up
            __nanosleep(ns);
            ns = min(2u * ns, 1024u);
            for (uint32_t left = open; left; left &= left - 1) {
                const int k = __ffs(left) - 1;
                const uint32_t *w = k == 0 ? p[0] : k == 1 ? p[1] : k == 2 ? p[2] : k == 3 ? p[3] : done + own;
                uint32_t x;
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(w) : "memory");
                if ((int32_t)(x - need) >= 0) open &= ~(1u << k);
            }
        } while (!__all_sync(0xFFFFFFFFu, open == 0u));
    }
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    __syncwarp();
    return true;
}

// One diffusion window for the `lanes` tets from i0 on, one warp. FLOW as in
// step_tile, with the finished-window words by warp tile
// (dep): window a.window + q, buffers swapped when q is odd. False when the
// tiles it waits for did not finish within the wait limit.
template <int RM, int SM, class P, int FLOW>
__device__ __forceinline__ bool warp_window(const ModelDev &m, const StepArgs &a, WarpTile<SM> &w, const RxnTab &tb,
                                            const uint32_t *s_scale, int64_t i0, const FlowArgs *f, uint32_t q,
                                            uint32_t dep, int lanes = 32) {
    constexpr int NP = (SM + 3) / 4;
    const int lane = threadIdx.x & 31;
    const int64_t i = i0 + lane;
    const bool live = i < a.T && lane < lanes;
    const uint32_t below = (1u << lane) - 1u;
    int32_t *const cur = (q & 1u) ? a.nxt : a.cur;
    int32_t *const nxt = (q & 1u) ? a.cur : a.nxt;
    const size_t Tpad = (size_t)a.Tpad;
    uint32_t bad = 0;

    // ---- load: the tables no window writes, then (once the previous window,
    // or in a flow launch the tiles this one depends on, is done) the counts,
    // one coalesced load per row, all in flight together
    uint4 A = make_uint4(0u, 0u, 0u, 0u);
    int4 nb4 = make_int4(-1, -1, -1, -1);
    float inv_nav = 1.0f;
    uint32_t tet = (uint32_t)i, active = 0u;
    if (live) {
        A = __ldg(a.thr + i);
        nb4 = __ldg(a.nbr + i);
        inv_nav = __ldg(a.inv_nav + i);
        if (a.orig) tet = (uint32_t)__ldg(a.orig + i);
        active = a.rmask ? __ldg(a.rmask + i) : 0xFFFFFFFFu;
    }
    w.thr[lane] = A;
    w.nbr[lane] = nb4;
    w.tet[lane] = tet;
    if constexpr (FLOW != 0) {
        if (q > 0 && !flow_nbr_wait(f->tile_done, dep, i0, nb4, (uint32_t)(a.window + q))) {
            if (lane == 0) atomicOr(a.err, 8u);
            return false;
        }
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    const uint64_t window = a.window + q + (a.window_base ? *a.window_base : 0ull);
    const uint32_t c0 = (uint32_t)window, c3 = (uint32_t)(window >> 32) & 0x0FFFFFFFu;
    int32_t any = 0;
    uint32_t nz = 0;  // the tet's species (models of many: a warp of which may lack every reaction's reactants)
    {
        int32_t n[SM];
        const int32_t *src = cur + i;
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            n[s] = live && s < P::S(m) ? __ldcg(src) : 0;
            src += Tpad;
        }
        // `cur` receives the window after next: zero its non-zero entries
        int32_t *row = cur + i;
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            w.cnt[s][lane] = s < P::S(m) ? n[s] : 1;  // (row S holds ones: a missing reactant)
            any |= n[s];
            if (SM > kManySpecies) nz |= n[s] != 0 ? 1u << s : 0u;
            if (n[s] != 0) *row = 0;
            row += Tpad;
        }
        w.cnt[SM][lane] = 1;
    }
    if (any < 0) bad |= 1u;
    __syncwarp();

    // ---- reactions: the tet's events inside the window. Most tets that react
    // fire once (0.07 events per tet and window on the benchmark box, averaged
    // over its run), so the first event and the attempt after it are
    // straight-line code for the whole warp, with both Philox blocks side by
    // side; only tets whose second attempt may fire run the event loop.
    uint32_t touched = 0;
    bool possible = P::R(m) > 0;
    if (SM > kManySpecies && possible) {  // lane r: can reaction r fire in any tet of the warp?
        const uint32_t wnz = __reduce_or_sync(0xFFFFFFFFu, nz), wact = __reduce_or_sync(0xFFFFFFFFu, active);
        const uint32_t need = lane < P::R(m) ? tb.need[lane] : 0u;
        possible = __any_sync(0xFFFFFFFFu, lane < P::R(m) && ((wact >> lane) & 1u) && (wnz & need) == need);
    }
    if (possible) {
        double O[SM], tS[SM];
        int32_t *const cnt = &w.cnt[0][lane];
        const bool masked = a.rmask != nullptr;
        int pick = -1;
        bool many = false;
        float psum[RM];
        float a0 = P::template first_sums<RM>(tb, m, cnt, inv_nav, active, masked, psum);
        const uint4 r0 = philox_rk(a.rk, c0, tet, 0u, (kPurposeReac << 28) | c3);
        const uint4 r1 = philox_rk(a.rk, c0, tet, 1u, (kPurposeReac << 28) | c3);
        const float dt = __fdiv_rn(-steps_logf(unit24f(r0.x)), a0);
        if (live & (a0 > 0.0f) & !(dt > a.tau_dn))
            pick = P::template pick<RM>(tb, m, psum, __fmul_rn(unit24f(r0.y), a0), cnt, inv_nav, active);
        if (__any_sync(0xFFFFFFFFu, pick >= 0)) {
            if (pick >= 0)
                P::for_changes(tb, pick, [&](int s, int d) {
                    cnt[s * 32] += d;
                    touched |= 1u << s;
                });
            a0 = P::template sums<RM>(tb, m, cnt, inv_nav, active, masked, psum);
            many = (pick >= 0) & (a0 > 0.0f) & !attempt_over(unit24f(r1.x), a0, a.tau_dn);
            if (many) bad |= ssa_lane<RM, P>(tb, m, a, cnt, tet, c0, c3, inv_nav, active, pick, dt, O, tS, touched);
            // occupancy rounding of the species the reactions changed, 32
            // (tet, species) pairs at a time: few tets have one, spread over
            // all species
            uint32_t todo = a.occ ? touched & P::diffusive(m) : 0u;
            const uint4 chg = tb.chg[max(pick, 0)];
            int np = 0;
            __syncwarp();
            for (uint32_t has = 1u; has || np;) {
                has = __ballot_sync(0xFFFFFFFFu, todo != 0u);
                if (todo) {
                    const int s = __ffs(todo) - 1, pos = np + __popc(has & below);
                    todo &= todo - 1;
                    // a single event: its change of s (the table is in species order)
                    const int e = __popc(touched & ((1u << s) - 1u));
                    const int32_t d = (int32_t)(int8_t)((e < 4 ? chg.z : chg.w) >> (8 * (e & 3)));
                    uint64_t o = (uint32_t)d, t = __float_as_uint(dt);
                    if (many) {
                        o = (uint64_t)__double_as_longlong(O[s]);
                        t = (uint64_t)__double_as_longlong(tS[s]);
                    }
                    w.r.O[pos] = o;
                    w.r.tS[pos] = t;
                    w.r.ls[pos] = (uint16_t)(lane | (s << 5) | (many ? 0 : 0x8000));
                }
                np += __popc(has);
                if (np >= 32 || (!has && np)) {  // a full set of lanes, or the rest
                    __syncwarp();
                    const int take = min(np, 32);
                    np -= take;
                    round_pairs<SM>(a, w, np, take, c0, c3);
                    __syncwarp();
                }
            }
            __syncwarp();
        }
    }

    // ---- trial counts of the diffusive species with a non-zero leave
    // threshold; those below kBulkMin join the tet's word stream
    uint32_t W = 0, bm = 0;
    const uint32_t round = a.occ ? touched : 0u;
    // species somewhere in the warp (models of many species skip the others)
    const uint32_t here = SM > kManySpecies ? __reduce_or_sync(0xFFFFFFFFu, nz | touched) : 0xFFFFFFFFu;
    {
        constexpr int NQ = WarpTile<SM>::kPre;
        uint32_t pre[4 * NQ] = {};
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            if (s < P::S(m) && ((P::diffusive(m) >> s) & 1u) && ((here >> s) & 1u)) {
                int32_t M = w.cnt[s][lane];
                if ((round >> s) & 1u) M = w.trial[s][lane];
                M = thr31(A.w, warp_R<P>(a, s_scale, s, i)) == 0u ? 0 : M;  // draws nothing
                const bool bulk = M >= kBulkMin;
                bm |= bulk ? 1u << s : 0u;
                if (bulk) w.trial[s][lane] = M;
                W += bulk ? 0u : (uint32_t)max(M, 0);
            }
            pre[s >> 2] |= W << (8 * (s & 3));
        }
#pragma unroll
        for (int s = SM; s < 4 * NP; ++s) pre[s >> 2] |= 0x80u << (8 * (s & 3));
        pre[4 * NQ - 1] = W;
#pragma unroll
        for (int j = 0; j < NQ; ++j)
            w.pre[lane][j] = make_uint4(pre[4 * j], pre[4 * j + 1], pre[4 * j + 2], pre[4 * j + 3]);
    }

    const bool wide = __any_sync(0xFFFFFFFFu, W > 127u);
    if (wide) wide_trials<SM, P>(m, a, w, s_scale, i, A.w, bm, round);

    // ---- bit-plane groups of the species with many trial molecules
    if (__any_sync(0xFFFFFFFFu, bm != 0u)) {
        __syncwarp();
        int32_t M = 0;
        uint32_t g = 0;
        int s = 0, ng = 0;
        for (;;) {
            if (32ll * g >= M && bm) {  // the lane's next species
                s = __ffs(bm) - 1;
                bm &= bm - 1;
                M = w.trial[s][lane];
                g = 0;
            }
            const bool more = 32ll * g < M;
            const uint32_t has = __ballot_sync(0xFFFFFFFFu, more);
            if (!(has | (uint32_t)ng)) break;
            if (more) {
                w.d.q[ng + __popc(has & below)] = make_uint2(g, (uint32_t)(lane | (s << 5)));
                ++g;
            }
            ng += __popc(has);
            if (ng >= 32 || !has) {  // a full set of lanes, or the rest
                __syncwarp();
                const int take = min(ng, 32);
                ng -= take;
                plane_groups<SM, P>(a, w, nxt, s_scale, i0, ng, take, c0, c3);
                __syncwarp();
            }
        }
    }
    __syncwarp();

    // ---- word stream: the tets' Philox blocks, listed kWarpMapCap at a time
    // and spread over the lanes
    {
        const uint32_t nb = (W + 3u) >> 2;
        uint32_t xs = nb;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, xs, d);
            if (lane >= d) xs += y;
        }
        const uint32_t first = xs - nb;
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, xs, 31);
        uint32_t k = 0;
        for (uint32_t base = 0; base < total; base += kWarpMapCap) {
            const uint32_t lim = min(total, base + (uint32_t)kWarpMapCap);
            for (; k < nb && first + k < lim; ++k) w.d.map[first + k - base] = (uint16_t)((uint32_t)lane | (k << 5));
            __syncwarp();
            if (wide) draw_words_wide<SM, P>(m, a, w, nxt, s_scale, i0, lim - base, c0, c3);
            else draw_words<SM, P, false>(m, a, w, nxt, s_scale, i0, lim - base, c0, c3);
        }
    }

    // ---- what stays is added to the tet's own entry of nxt (apply_remaining)
    {
        int32_t *out = nxt + i;
#pragma unroll
        for (int s = 0; s < SM; ++s) {
            if (s < P::S(m) && ((here >> s) & 1u)) {
                const int32_t N = w.cnt[s][lane];
                if (N) {
                    if ((P::diffusive(m) >> s) & 1u) atomicAdd(out, N);
                    else *out = N;
                }
            }
            out += Tpad;
        }
    }
    if (bad) atomicOr(a.err, bad);
    if constexpr (FLOW != 0) {
        // publish: every lane's writes of this tile come before the release
        __syncwarp();
        if (lane == 0) st_release_gpu(f->tile_done + dep, (uint32_t)(a.window + q + 1));
    }
    return true;
}

// The warps of a block: they share the reaction table and the species scales;
// after the barrier that publishes them every warp runs on its own. FLOW 0:
// the tiles of block tile `tile`. 1 (a launch of several windows): the block
// takes its item (window, block tile) from f's counter, as in flow_tiles. 2
// (batched): the caller took the block's item; dep is its work entry.
// BLOCK 0: as many threads as the launch has.
template <int BLOCK, int RM, int SM, class P, int FLOW = 0>
__device__ __forceinline__ void warp_step(const ModelDev &m, const StepArgs &a, int64_t tile,
                                          const FlowArgs *f = nullptr, uint32_t q = 0, uint32_t dep = 0) {
    extern __shared__ __align__(16) unsigned char warp_smem[];
    __shared__ RxnTab tb;
    __shared__ uint32_t s_scale[kScaleEntries];
    static_assert(SM <= kWarpMaxSpecies, "species bound");
    const int threads = BLOCK ? BLOCK : (int)blockDim.x, warps = threads / 32;
    constexpr bool PERSIST = warp_flow_persists(BLOCK);
    const int tid = threadIdx.x, warp = tid >> 5;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    P::template build<32>(m, tb);  // (of up to 32 reactions, by the first warp)
    if (tid < kMaxSpecies) s_scale[tid] = a.scale[tid];
    if (tid == 0) s_scale[kMaxSpecies] = 0u;
    __syncthreads();
    WarpTile<SM> &w = reinterpret_cast<WarpTile<SM> *>(warp_smem)[warp];
    if constexpr (FLOW == 1) {
        __shared__ uint32_t s_item;
        const uint32_t items = f->nwin * f->ntiles;
        uint32_t next = 0;
        if (tid == 0) next = atomicAdd(f->fetch, 1u);
        for (;;) {
            if (tid == 0) s_item = next;
            __syncthreads();
            const uint32_t item = s_item;
            if (item >= items) return;
            // the next item, fetched while this one runs
            if (PERSIST && tid == 0) next = atomicAdd(f->fetch, 1u);
            const uint32_t qq = item / f->ntiles, t = item - qq * f->ntiles;
            const int64_t i0 = (int64_t)t * threads + warp * 32;
            bool done = true;
            if (i0 < a.T)
                done = warp_window<RM, SM, P, FLOW>(m, a, w, tb, s_scale, i0, f, qq, t * (uint32_t)warps + (uint32_t)warp);
            if (!PERSIST || __syncthreads_or(!done)) return;  // (a wait that ran out ends the block)
        }
    } else {
        const int lanes = FLOW == 0 && BLOCK == 0 ? a.lanes : 32;
        const int64_t i0 = (tile * warps + warp) * lanes;
        if (i0 < a.T) warp_window<RM, SM, P, FLOW>(m, a, w, tb, s_scale, i0, f, q, dep * (uint32_t)warps + (uint32_t)warp, lanes);
    }
}
}  // namespace
}  // namespace steps
