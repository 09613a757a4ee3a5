// The operator-split step in the list form: models with many species, in
// states of few molecules per tet (a step over tiles reads every count of
// every tet). Included after steps_warp.cuh, whose building blocks it shares;
// the same draws, formulas and decisions, so the same bits.
//
// Every tet has a word of species bits beside its counts (StepArgs::tm_cur,
// tm_nxt, in step with the count buffers): a set bit says that the count may
// be non-zero. Warps work on 32 tets that hold something at a time, one per
// lane, reading only their non-zero counts and their tables; an empty tet
// costs nothing. Those tets are listed by the window before: whoever sets bits
// of a tet's word in tm_nxt appends the tet to the next window's list. Tets
// with an active order-0 reaction (sources) have a list of their own and are
// tested every window.
//
// What bounds it: scattered accesses to L2 and a chunk's chain of them (list
// entry, record, counts, atomics, append). On the 1.03M-tet dendrite (0.12
// molecules per tet) an empty launch takes 1.4 us, the chunks without
// reactions and draws 8.7, all of it 14.6 us per window; block tiles, which
// copied every count, took 39.8. Tried: one append per block, 14.5; places
// reserved at the start of a chunk, 16.9; a scan of tiles for listed tets
// instead of a list, 30.8.
#pragma once

#include "steps_warp.cuh"

namespace steps {
namespace {

template <class P>
__device__ __forceinline__ uint32_t list_R(const StepArgs &a, const uint32_t *s_scale, int s, int32_t i) {
    if constexpr (P::kExpLeave)
        return __ldg(a.leave + ((uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i));
    else return s_scale[s];
}

// What a chunk's helpers need.
template <int SM>
struct ListCtx {
    ListTile<SM> &w;
    int32_t *cur, *nxt;
    uint32_t *tm_nxt;
    const uint32_t *s_scale;
    uint32_t c0, c3;
    int32_t *list;      // the next window's list and its length
    uint32_t *lcnt;
};

// The whole warp calls. Lanes with bits != 0 set them in tet j's word of the
// next window and append the tet to its list unless it is a
// source (those have their own list). A tet's own warp (OWN) appends it
// without a look at the word, others only when they set its first bit: a tet
// is listed twice at most, and worked off by the warp that takes its word
// first (list_window).
template <bool OWN, int SM>
__device__ __forceinline__ void list_mark(const StepArgs &a, const ListCtx<SM> &x, uint32_t j, uint32_t bits) {
    bool add = bits != 0u;
    if constexpr (OWN) {
        if (add) atomicOr(x.tm_nxt + j, bits);
    } else {
        add = add && atomicOr(x.tm_nxt + j, bits) == 0u;
    }
    if (a.srcbits && add) add = ((__ldg(a.srcbits + (j >> 5)) >> (j & 31u)) & 1u) == 0u;
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, add);
    if (m) {
        const uint32_t lane = threadIdx.x & 31u;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(x.lcnt, (uint32_t)__popc(m));
        at = __shfl_sync(0xFFFFFFFFu, at, 0);
        if (add) x.list[at + __popc(m & ((1u << lane) - 1u))] = (int32_t)j;
    }
}

// Up to 32 queued (tet, species) pairs: the trial count of a species a
// reaction changed (round_pairs; the trial counts live in StepArgs::trial).
template <int SM>
__device__ __forceinline__ void list_round(const StepArgs &a, const ListCtx<SM> &x, int first, int n) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint32_t ls = x.w.r.ls[first + lane];
        const int t = (int)(ls & 31u), s = (int)((ls >> 5) & 31u);
        const int32_t N = x.w.cnt[s][t];
        const uint64_t ob = x.w.r.O[first + lane], tb = x.w.r.tS[first + lane];
        double tS = __longlong_as_double((long long)tb), O = __longlong_as_double((long long)ob);
        if (ls >> 15) {  // one event, at a float time, changed N - d to N
            tS = (double)__uint_as_float((uint32_t)tb);
            O = __dmul_rn((double)(N - (int32_t)(uint32_t)ob), tS);
        }
        const double occ = __dadd_rn(O, __dmul_rn((double)N, __dsub_rn(a.tau_k, tS)));
        const double nbar = __dmul_rn(occ, a.inv_tau_k);
        const uint4 rb = philox_rk(a.rk, x.c0, x.w.tet[t], (uint32_t)(s >> 2), (kPurposeRound << 28) | x.c3);
        a.trial[(uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)x.w.idx[t]] =
            round_trials32(nbar, word_of(rb, (uint32_t)(s & 3)), N);
    }
}

// Up to 32 queued movers (move_out); the whole warp calls.
template <int SM, class P>
__device__ __forceinline__ void list_move(const StepArgs &a, const ListCtx<SM> &x, int first, int n) {
    const int lane = threadIdx.x & 31;
    uint32_t j = 0, bits = 0;
    if (lane < n) {
        const uint2 e = x.w.d.q[first + lane];
        const int t = (int)(e.y & 31u), s = (int)(e.y >> 5);
        const int32_t i = x.w.idx[t];
        const uint4 A = __ldg(a.thr + i);
        const uint32_t R = list_R<P>(a, x.s_scale, s, i);
        const int f = (e.x >= thr31(A.x, R)) + (e.x >= thr31(A.y, R)) + (e.x >= thr31(A.z, R));
        j = (uint32_t)__ldg(reinterpret_cast<const int32_t *>(a.nbr + i) + f);
        bits = 1u << s;
        atomicAdd(x.nxt + ((uint64_t)(uint32_t)s * (uint32_t)a.Tpad + j), 1);
        atomicSub(&x.w.cnt[s][t], 1);
    }
    list_mark<false>(a, x, j, bits);
}

// Up to 32 queued groups of 32 trial molecules, one per lane (plane_groups);
// the whole warp calls.
template <int SM, class P>
__device__ __forceinline__ void list_planes(const StepArgs &a, const ListCtx<SM> &x, int first, int n) {
    const int lane = threadIdx.x & 31;
    uint32_t moved = 0;  // molecules through each face, a byte each
    int s = 0;
    int32_t i = 0;
    if (lane < n) {
        const uint2 e = x.w.d.q[first + lane];
        const int t = (int)(e.y & 31u);
        s = (int)(e.y >> 5);
        i = x.w.idx[t];
        const int32_t M = a.trial[(uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i];
        uint32_t l[4];
        plane_group(n == 32 ? 0xFFFFFFFFu : (1u << n) - 1u, a, __ldg(a.thr + i), list_R<P>(a, x.s_scale, s, i), (uint32_t)M, e.x, x.w.tet[t], s, x.c0, x.c3, l);
        // cumulative thresholds: l[0] within l[1] within l[2] within l[3]
        moved = (uint32_t)__popc(l[0]) | (uint32_t)__popc(l[1] & ~l[0]) << 8 | (uint32_t)__popc(l[2] & ~l[1]) << 16 |
                (uint32_t)__popc(l[3] & ~l[2]) << 24;
        if (l[3]) atomicSub(&x.w.cnt[s][t], __popc(l[3]));
    }
    for (int f = 0; f < 4; ++f, moved >>= 8) {
        const int32_t out = (int32_t)(moved & 255u);
        uint32_t j = 0;
        if (out) {
            j = (uint32_t)__ldg(reinterpret_cast<const int32_t *>(a.nbr + i) + f);
            atomicAdd(x.nxt + ((uint64_t)(uint32_t)s * (uint32_t)a.Tpad + j), out);
        }
        list_mark<false>(a, x, j, out ? 1u << s : 0u);
    }
}

// The chunk's reactions (warp_window's; `possible`: those with all reactants
// somewhere in the chunk, the others' propensities are 0), skipped by a chunk
// without any. Models with rates near the float range keep to the tiles
// (plain_rates): the sums are taken as they are. Returns the species changed
// and, above them, error bits.
template <int RM, int SM, class P>
__device__ __forceinline__ uint64_t list_react(const ModelDev &m, const StepArgs &a, const ListCtx<SM> &x,
                                              const RxnTab &tb, uint32_t possible, bool live, float inv_nav,
                                              uint32_t tet, uint32_t active) {
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    ListTile<SM> &w = x.w;
    int32_t *const cnt = &w.cnt[0][lane];
    uint32_t touched = 0, bad = 0;
    float a0 = 0.0f;
    float psum[RM];
    asm volatile("" ::: "memory");  // (no count in a register across the sweeps)
#pragma unroll
    for (int r = 0; r < RM; ++r) {
        float ar = 0.0f;
        if ((possible >> r) & 1u) ar = ((active >> r) & 1u) ? P::prop(tb, m, r, cnt, inv_nav) : 0.0f;
        a0 = __fadd_rn(a0, ar);
        psum[r] = a0;
    }
    if (__any_sync(0xFFFFFFFFu, live & (a0 > 0.0f))) {
        double O[SM], tS[SM];
        int pick = -1;
        bool many = false;
        const uint4 r0 = philox_rk(a.rk, x.c0, tet, 0u, (kPurposeReac << 28) | x.c3);
        const float dt = __fdiv_rn(-steps_logf(unit24f(r0.x)), a0);
        if (live & (a0 > 0.0f) & !(dt > a.tau_dn))
            pick = pick_reaction<P, RM>(tb, m, psum, __fmul_rn(unit24f(r0.y), a0), cnt, inv_nav, active);
        if (__any_sync(0xFFFFFFFFu, pick >= 0)) {
            if (pick >= 0) {
                P::for_changes(tb, pick, [&](int s, int d) {
                    cnt[s * 32] += d;
                    touched |= 1u << s;
                });
                const uint4 r1 = philox_rk(a.rk, x.c0, tet, 1u, (kPurposeReac << 28) | x.c3);
                asm volatile("" ::: "memory");
                a0 = propensity_sums<P, RM>(tb, m, cnt, inv_nav, active, psum);
                many = (a0 > 0.0f) & !attempt_over(unit24f(r1.x), a0, a.tau_dn);
                if (many)
                    bad |= ssa_lane<RM, P>(tb, m, a, cnt, tet, x.c0, x.c3, inv_nav, active, pick, dt, O, tS, touched);
            }
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
                    w.r.ls[pos] = (uint16_t)(lane | (uint32_t)(s << 5) | (many ? 0u : 0x8000u));
                }
                np += __popc(has);
                if (np >= 32 || (!has && np)) {  // a full set of lanes, or the rest
                    __syncwarp();
                    const int take = min(np, 32);
                    np -= take;
                    list_round<SM>(a, x, np, take);
                    __syncwarp();
                }
            }
            __syncwarp();
        }
    }
    return (uint64_t)bad << 32 | touched;
}

// One window for up to 32 listed tets, one per lane: the lane's tet is i
// (-1: none) with the species bits nz.
template <int RM, int SM, class P>
__device__ __forceinline__ uint32_t list_chunk(const ModelDev &m, const StepArgs &a, const ListCtx<SM> &x,
                                                 const RxnTab &tb, int32_t i, uint32_t nz) {
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    ListTile<SM> &w = x.w;
    const bool live = i >= 0;
    int32_t *const cnt = &w.cnt[0][lane];
    uint32_t bad = 0;

    // ---- load
    uint4 rec = make_uint4(0u, 0u, 0x3F800000u, 0u);
    if (live) rec = __ldg(a.rec + i);
    const uint32_t Aw = rec.x, tet = rec.y, active = rec.w;
    const float inv_nav = __uint_as_float(rec.z);
#pragma unroll
    for (int s = 0; s < SM; ++s) cnt[s * 32] = 0;
    cnt[SM * 32] = 1;
    // the listed counts, four in flight, each taken and zeroed by one access (the
    // buffer receives the window after next). What bounds a sparse window is
    // the number of scattered accesses, so a tet's tables are one 16-byte
    // record too: five per tet in place of nine.
    for (uint32_t left = nz; left;) {
        int32_t v[4];
        int sp[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sp[k] = left ? __ffs(left) - 1 : -1;
            left &= left - 1;
            v[k] = sp[k] >= 0 ? atomicExch(x.cur + ((uint64_t)(uint32_t)sp[k] * (uint32_t)a.Tpad + (uint32_t)i), 0) : 0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (v[k] != 0) {
                cnt[sp[k] * 32] = v[k];
                if (v[k] < 0) bad |= 1u;
            }
    }
    w.thr_w[lane] = Aw;
    w.tet[lane] = tet;
    w.idx[lane] = i;
    __syncwarp();

    // ---- reactions, if any has its reactants in the chunk (lane r decides
    // reaction r)
    uint32_t touched = 0;
    if (P::R(m) > 0) {
        const uint32_t wnz = __reduce_or_sync(0xFFFFFFFFu, nz);
        const uint32_t wact = __reduce_or_sync(0xFFFFFFFFu, active);
        const uint32_t need = lane < P::R(m) ? tb.need[lane] : 0u;
        const uint32_t possible =
            __ballot_sync(0xFFFFFFFFu, lane < P::R(m) && ((wact >> lane) & 1u) && (wnz & need) == need);
        if (possible) {
            const uint64_t r = list_react<RM, SM, P>(m, a, x, tb, possible, live, inv_nav, tet, active);
            touched = (uint32_t)r;
            bad |= (uint32_t)(r >> 32);
        }
    }

    // ---- trial counts: a lane walks its own species
    const uint32_t may = nz | touched;
    uint32_t round = a.occ ? touched : 0u;  // species whose trial count is in StepArgs::trial
    uint32_t W = 0, hm = 0, bm = 0;
    for (uint32_t walk = live ? may & P::diffusive(m) : 0u; walk; walk &= walk - 1) {
        const int s = __ffs(walk) - 1;
        const uint64_t at = (uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i;
        int32_t M = cnt[s * 32];
        if ((round >> s) & 1u) M = a.trial[at];
        if (M <= 0 || thr31(Aw, list_R<P>(a, x.s_scale, s, i)) == 0u) continue;  // draws nothing
        if (M >= kBulkMin) {
            bm |= 1u << s;
            a.trial[at] = M;
        } else {
            hm |= 1u << s;
            W += (uint32_t)M;
        }
    }

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
                M = a.trial[(uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i];
                g = 0;
            }
            const bool more = 32ll * g < M;
            const uint32_t has = __ballot_sync(0xFFFFFFFFu, more);
            if (!(has | (uint32_t)ng)) break;
            if (more) {
                w.d.q[ng + __popc(has & below)] = make_uint2(g, lane | (uint32_t)(s << 5));
                ++g;
            }
            ng += __popc(has);
            if (ng >= 32 || !has) {  // a full set of lanes, or the rest
                __syncwarp();
                const int take = min(ng, 32);
                ng -= take;
                list_planes<SM, P>(a, x, ng, take);
                __syncwarp();
            }
        }
    }
    __syncwarp();

    // ---- word stream: the tets' Philox blocks, kListMapCap at a time, with
    // the species of their four words
    {
        const uint32_t nb = (W + 3u) >> 2;
        uint32_t xs = nb;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, xs, d);
            if (lane >= (uint32_t)d) xs += y;
        }
        const uint32_t first = xs - nb;
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, xs, 31);
        uint32_t k = 0;   // the lane's next block
        int s = 0;        // species of its next word
        int32_t rem = 0;  // words of that species left
        w.words[lane] = (uint16_t)W;
        if (total > (uint32_t)kListMapCap) {  // later rounds list after counts have dropped
            for (uint32_t walk = hm & ~round; walk; walk &= walk - 1) {
                const int c = __ffs(walk) - 1;
                a.trial[(uint64_t)(uint32_t)c * (uint32_t)a.Tpad + (uint32_t)i] = cnt[c * 32];
            }
            round |= hm;
        }
        for (uint32_t base = 0; base < total; base += kListMapCap) {
            const uint32_t lim = min(total, base + (uint32_t)kListMapCap);
            for (; k < nb && first + k < lim; ++k) {
                uint32_t sp = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (rem == 0 && hm) {
                        s = __ffs(hm) - 1;
                        hm &= hm - 1;
                        rem = (round >> s) & 1u ? a.trial[(uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i]
                                                : cnt[s * 32];
                    }
                    --rem;
                    sp |= (uint32_t)s << (5 * q);
                }
                w.d.map[first + k - base] = lane | (k << 5) | (sp << 12);
            }
            __syncwarp();
            int nq = 0;
            for (uint32_t b = base; b < lim; b += 32) {
                const uint32_t o = w.d.map[min(b + lane, lim - 1u) - base];
                const int t = (int)(o & 31u);
                const uint32_t kk = (o >> 5) & 127u;
                const int left = b + lane < lim ? (int)w.words[t] - (int)(4u * kk) : 0;
                const uint32_t tw = w.thr_w[t];
                const int32_t ti = w.idx[t];
                const uint4 rw = philox_rk(a.rk, x.c0, w.tet[t], kk, (kPurposeDiff << 28) | x.c3);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t c = (o >> (12 + 5 * r)) & 31u;
                    const uint32_t u = word_of(rw, (uint32_t)r) >> 1;
                    const bool moves = (r < left) & (u < thr31(tw, list_R<P>(a, x.s_scale, (int)c, max(ti, 0))));
                    const uint32_t mv = __ballot_sync(0xFFFFFFFFu, moves);
                    const int pos = nq + __popc(mv & below);
                    if (moves) w.d.q[pos] = make_uint2(u, (uint32_t)t | (c << 5));
                    nq += __popc(mv);
                }
                const int keep = b + 32 < lim ? 31 : 0;
                if (nq > keep) {
                    __syncwarp();
                    do {
                        const int take = min(nq, 32);
                        nq -= take;
                        list_move<SM, P>(a, x, nq, take);
                    } while (nq > keep);
                    __syncwarp();
                }
            }
            __syncwarp();
        }
    }

    // ---- what stays
    uint32_t kept = 0;
    for (uint32_t walk = live ? may : 0u; walk; walk &= walk - 1) {
        const int s = __ffs(walk) - 1;
        const int32_t N = cnt[s * 32];
        if (N) {
            int32_t *out = x.nxt + ((uint64_t)(uint32_t)s * (uint32_t)a.Tpad + (uint32_t)i);
            if ((P::diffusive(m) >> s) & 1u) atomicAdd(out, N);
            else *out = N;
            kept |= 1u << s;
        }
    }
    list_mark<true>(a, x, (uint32_t)i, kept);
    __syncwarp();
    return bad;
}

// Whether an empty tet may fire an order-0 reaction in the window: all its other propensities are 0.
__device__ __forceinline__ bool source_fires(const ModelDev &m, const StepArgs &a, int32_t i, uint32_t c0, uint32_t c3) {
    const uint4 rec = __ldg(a.rec + i);
    const float inv_nav = __uint_as_float(rec.z);
    uint32_t act = rec.w & m.order0;
    float a0 = 0.0f;
    for (; act; act &= act - 1) a0 = __fadd_rn(a0, __fdiv_rn(m.reac[__ffs(act) - 1].k, inv_nav));
    const uint4 r = philox_rk(a.rk, c0, rec.y, 0u, (kPurposeReac << 28) | c3);
    return !attempt_over(unit24f(r.x), a0, a.tau_dn);
}

// One window: warp `wid` of `warps` takes every warps-th chunk
// of 32 entries of the window's list, then of the sources.
template <int RM, int SM, class P>
__device__ __forceinline__ void list_window(const ModelDev &m, const StepArgs &a, ListTile<SM> &w, const RxnTab &tb,
                                              const uint32_t *s_scale, uint32_t wid, uint32_t warps) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t window = a.window + (a.window_base ? *a.window_base : 0ull);
    const uint32_t w2 = (uint32_t)(window & 1ull), w3 = (uint32_t)(window % 3ull);
    const int32_t *const list = a.list[w2];
    int32_t i = wid * 32 + lane < 2u * (uint32_t)a.Tpad ? __ldcg(list + wid * 32 + lane) : -1;  // the first chunk's, at once
    const uint32_t n = __ldcg(a.lcnt + w3), nsrc = a.srcbits ? __ldcg(a.lcnt + 3) : 0u;
    // the length after next's: read by the window before, written by the next
    if (wid == 0 && lane == 0) a.lcnt[w3 == 0u ? 2u : w3 - 1u] = 0u;
    const ListCtx<SM> x{w, a.cur, a.nxt, a.tm_nxt, s_scale, (uint32_t)window, (uint32_t)(window >> 32) & 0x0FFFFFFFu,
                          a.list[w2 ^ 1u], a.lcnt + (w3 == 2u ? 0u : w3 + 1u)};
    // where half of the tets are listed, the window goes through all of them in order
    const bool scan = n >= (uint32_t)a.Tpad / 2u;
    const uint32_t chunks = scan ? (uint32_t)a.Tpad / 32u : (n + 31u) / 32u, total = chunks + (nsrc + 31u) / 32u;
    uint32_t bad = 0;
    for (uint32_t c = wid; c < total; c += warps) {
        uint32_t nz = 0;
        if (c < chunks) {
            const uint32_t at = c * 32 + lane;
            if (scan) {
                const uint32_t src = a.srcbits ? __ldg(a.srcbits + c) : 0u;
                i = at < (uint32_t)a.T && !((src >> lane) & 1u) ? (int32_t)at : -1;
            } else {
                if (c != wid) i = at < n ? __ldcg(list + at) : -1;
                if (at >= n) i = -1;
            }
            // whoever takes the word works the tet off; it receives the window after next
            if (i >= 0) nz = atomicExch(a.tm_cur + i, 0u);
            if (nz == 0u) i = -1;
        } else {
            const uint32_t at = (c - chunks) * 32 + lane;
            i = at < nsrc ? __ldcg(a.src + at) : -1;
            if (i >= 0) {
                nz = __ldcg(a.tm_cur + i);
                if (nz) a.tm_cur[i] = 0u;
                else if (!source_fires(m, a, i, x.c0, x.c3)) i = -1;
            }
        }
        if (__any_sync(0xFFFFFFFFu, i >= 0)) bad |= list_chunk<RM, SM, P>(m, a, x, tb, i, nz);
    }
    if (bad) atomicOr(a.err, bad);
}

// The warps of a block of a plain launch (of any number of blocks).
template <int BLOCK, int RM, int SM, class P>
__device__ __forceinline__ void list_step(const ModelDev &m, const StepArgs &a, uint32_t block, uint32_t blocks) {
    extern __shared__ __align__(16) unsigned char warp_smem[];
    __shared__ RxnTab tb;
    __shared__ uint32_t s_scale[kMaxSpecies];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    P::template build<BLOCK>(m, tb);
    if (threadIdx.x < kMaxSpecies) s_scale[threadIdx.x] = a.scale[threadIdx.x];
    __syncthreads();
    const uint32_t warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    list_window<RM, SM, P>(m, a, reinterpret_cast<ListTile<SM> *>(warp_smem)[warp], tb, s_scale,
                             block * (BLOCK / 32) + warp, blocks * (BLOCK / 32));
}

}  // namespace
}  // namespace steps
