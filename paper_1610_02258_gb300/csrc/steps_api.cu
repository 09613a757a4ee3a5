// C ABI of the library: mesh, model and simulation handles, the window loop
// of Algorithm 1 on the host, and the device buffers it drives.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <limits>
#include <algorithm>
#include <future>
#include <system_error>
#include <map>
#include <tuple>
#include <memory>
#include <mutex>
#include <new>
#include <string>

#include "steps_internal.h"

using namespace steps;

namespace steps {

static thread_local std::string g_last_error;

void set_error(const std::string &msg) { g_last_error = msg; }

}  // namespace steps

struct steps_mesh {
    HostMesh m;
};

struct steps_model {
    HostModel m;
};

namespace {

constexpr int kGraphWindows = 16;  // full windows per captured graph (even: buffer parity is restored)
// The list form runs a state of at most this many listed tets (or, from set
// counts, non-zero counts) per tet. us per window, warp tiles -> list form:
// 1.03M-tet dendrite, 0.12: 61.8 -> 14.6; 294,780-tet box with 14 and 20
// species at 0.2 and 0.31: 19.6 -> 15.3, 22.0 -> 16.2; but with 14 at 1.0: 23.3
// -> 28.3, and the 300k-tet dendrite, whose molecules crowd at one end, 0.37:
// 15.8 -> 19.1. One line for every species count, set by the crowded states:
// even ones gain beyond it (30 species at 0.48, 34.1 -> 16.7) and stay on tiles.
constexpr double kListFill = 0.33;
// On smaller meshes than this, or with more tets listed, the tiles are faster: a
// window in the list form takes some 11 us however little there is to do, and
// the scattered accesses of many tets miss L2. us per window, the best tiles ->
// list form, 14 and 30 species at 0.1 molecules per tet: 10,404 tets 5.5 -> 9.6
// and 6.5 -> 9.2, 138,720 9.0 -> 12.3 and 10.4 -> 12.1, 294,780 15.2 -> 14.5 and
// 18.3 -> 14.5, 599,964 30.7 -> 15.3 and 38.7 -> 15.5, 1,040,400 49.8 -> 20.6 and
// 61.8 -> 21.6; there at 0.3 59.0 -> 73.7 and 79.1 -> 87.2.
constexpr int64_t kListMinTets = 262144;
constexpr double kListMost = 250000.0;
constexpr uint64_t kListWindows = 128;       // windows after which a list is built afresh
constexpr uint64_t kListCheckWindows = 1024;  // windows after which a run looks at the list's length
constexpr int64_t kFlowTuneWindows = 72;  // windows the launch-form tuning takes (3 rounds of up to 3 groups)
constexpr int64_t kFormTuneWindows = 90;  // with block tiles as two more candidates
constexpr int kForms = 6;                 // window launches, flow, flow at 512; the same of block tiles (256)

// Tets a resident wave of compiled warp tiles covers (their shared memory, at
// most 32 warps per SM). Models of 13 or more species on larger meshes have
// compiled block tiles too, whose copies run ahead (TMA, L2 prefetch) with 40
// warps per SM. us per window in the best launch form, warp tiles -> block
// tiles, 14, 20 and 30 species: 138,720 tets at 0.1 molecules per tet 10.9, 12.0
// and 14.0 -> 9.0, 9.7 and 10.4, at 2 16.1, 17.9 and 18.8 -> 15.4, 18.4 and 19.4;
// 1,040,400 tets at 0.5 67.6, 80.0 and 132 -> 65.6, 78.2 and 89.3, at 5 98, 116 and
// 216 -> 124, 182 and 214. Within a wave warp tiles win throughout (69,360 tets,
// 14 species at 0.1: 7.2 -> 8.7).
int64_t warp_wave(int S) {
    const size_t block = 8 * warp_tile_bytes(S) + 3072;  // 256 threads, and the static arrays
    return (int64_t)152 * 32 * std::min<int64_t>(32, 8 * (int64_t)(227 * 1024 / block));
}
// The molecules per tet up to which, by those figures, window launches that were
// not timed go over block tiles, and the tuning times them.
double block_density(int S, int64_t T) { return S >= 24 ? 1.5 : T < kListMinTets ? 1.0 : 0.2; }
double tuned_block_density(int S) { return S >= 24 ? 5.0 : 2.0; }
// The same for a batch, by its members together: four of 69,360 tets and 30
// species at 2 molecules per tet, 65 us per window on warp tiles, 54 on block
// tiles.
double batch_block_density(int S) { return S >= 24 ? 2.0 : 0.5; }
// Batches of run-time models of 5 to 12 species go over block tiles up to this
// density. us per window of 16 members of 52,020 tets and 10 species, block ->
// warp tiles: 0.05 molecules per tet 55 -> 67, 0.2 65 -> 73, 0.5 76 -> 79, 1.0
// 88 -> 84, 3.0 113 -> 101; 3 species 40 -> 40, 44 -> 42, 51 -> 44, 59 -> 47, 72
// -> 59.
constexpr double kFewPerTet = 0.5;

__global__ void scatter_to_device_order(const int32_t *src, int64_t nt, int32_t S, const int32_t *inv_perm,
                                        int32_t *dst, size_t Tpad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nt) return;
    const int64_t d = inv_perm ? inv_perm[i] : i;
    for (int s = 0; s < S; ++s) dst[s * Tpad + d] = src[s * (size_t)nt + i];
}

__global__ void gather_to_original_order(const int32_t *src, int64_t nt, int32_t S, const int32_t *inv_perm,
                                         size_t Tpad, int32_t *dst) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nt) return;
    const int64_t d = inv_perm ? inv_perm[i] : i;
    for (int s = 0; s < S; ++s) dst[s * (size_t)nt + i] = src[s * Tpad + d];
}

// Species words (StepArgs::tm_cur, tm_nxt) of a count buffer, for the list form:
// one coalesced pass over the counts.
__global__ void build_species_words(const int32_t *cnt, int64_t T, size_t Tpad, int32_t S, uint32_t *cur, uint32_t *nxt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= T) return;
    uint32_t nz = 0;
#pragma unroll 4
    for (int s = 0; s < S; ++s) nz |= cnt[s * Tpad + i] != 0 ? 1u << s : 0u;
    cur[i] = nz;
    nxt[i] = 0u;
}

// The list of the next window: the tets with a species
// bit that are not sources, a block's together, in order.
__global__ void build_list(const uint32_t *tm, int64_t T, const uint32_t *srcbits, int32_t *list, uint32_t *n) {
    __shared__ uint32_t at[9];
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const bool in = i < T && tm[i] != 0u && !(srcbits && ((srcbits[i >> 5] >> (i & 31)) & 1u));
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
    if (lane == 0) at[warp] = (uint32_t)__popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t sum = 0;
        for (int k = 0; k < 8; ++k) {
            const uint32_t c = at[k];
            at[k] = sum;
            sum += c;
        }
        at[8] = sum ? atomicAdd(n, sum) : 0u;
    }
    __syncthreads();
    if (in) list[at[8] + at[warp] + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
}

// The tets' records, and those with an active order-0 reaction (rmask null:
// all are active): a bit each and a list (list null: the model has none).
__global__ void build_sources(const uint32_t *rmask, uint32_t order0, int64_t T, const uint4 *thr, const int32_t *orig,
                              const float *inv_nav, uint4 *rec, uint32_t *bits, int32_t *list, uint32_t *n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t act = i < T && rmask ? rmask[i] : 0xFFFFFFFFu;
    if (i < T)
        rec[i] = make_uint4(thr[i].w, orig ? (uint32_t)orig[i] : (uint32_t)i, __float_as_uint(inv_nav[i]), act);
    if (!list) return;
    const bool in = i < T && (act & order0) != 0u;
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
    uint32_t at = 0;
    if (lane == 0 && i < T) {
        bits[i >> 5] = m;
        if (m) at = atomicAdd(n, (uint32_t)__popc(m));
    }
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (in) list[at + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
}

// EXP leave law: out[s Tpad + d] = floor(2^31 (1 - exp(-(tau_k D_s) G_d))), the
// entries of exp_leave_table. That table is the C library's, bit for bit, and
// the device's exp is another function; but both are within an ulp of the
// exact value, so the two products differ by less than 2^-20, and the floors
// can differ only where the product lies that close to an integer >= 1. Those
// entries (one in 2^15 with the margin of 2^-16 taken here) go to a list: *n
// of them, list[k] = (species, tet), for the host to decide.
struct LeaveRates {
    double tauD[kMaxSpecies];  // tau_k D_s, 0 for immobile species
};
constexpr uint32_t kLeaveListCap = 4096;
// Up to so many entries the host computes the whole table, behind the windows
// already enqueued and without a wait (the copy, of 32 KB at most, is staged).
// A recording of 40 intervals of 2.5 windows, us, device -> host: 144 entries
// 1,770 -> 875, 1,440 entries 1,945 -> 996, 5,760 entries 1,980 -> 1,413. The
// host takes 4 ns an entry: 19,200 entries took 3,650 from the host (on the
// block tiles, whose windows were slower too), 2,990 from the device.
constexpr int64_t kLeaveHostEntries = 8192;
constexpr size_t kLeaveListBytes = (2 + 3 * (size_t)kLeaveListCap) * 4;

__global__ void leave_table(const double *G, int64_t T, size_t Tpad, int S, const __grid_constant__ LeaveRates r,
                            uint32_t *out, uint2 *list, uint32_t *n) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= T) return;
    const double g = G[d];
    for (int s = 0; s < S; ++s) {
        uint32_t v = 0;
        if (r.tauD[s] > 0.0) {
            const double y = __dmul_rn(1.0 - exp(-__dmul_rn(r.tauD[s], g)), 2147483648.0);
            const double near = rint(y);
            if (near >= 1.0 && fabs(y - near) < 1.52587890625e-05) {
                const uint32_t k = atomicAdd(n, 1u);
                if (k < kLeaveListCap) list[k] = make_uint2((uint32_t)s, (uint32_t)d);
            } else {
                v = (uint32_t)fmin(2147483648.0, fmax(0.0, floor(y)));
            }
        }
        out[s * Tpad + d] = v;
    }
}

__global__ void patch_leave(const uint2 *list, const uint32_t *value, uint32_t n, size_t Tpad, uint32_t *out) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[list[k].x * Tpad + list[k].y] = value[k];
}

__global__ void set_u64_kernel(uint64_t *p, uint64_t v) { *p = v; }

// What an input holds: word 0 |= 1 if any of src[0..n) is negative; asked for
// more, word 1 += the non-zero ones and words 2-3 (64 bits) += their sum.
// Bound by reading src: four counts per load where it is aligned for that, and
// one atomic per block and word (per warp they queued up on the three words:
// 2.9M counts took 45.7 us, now 5.7).
constexpr int kInputThreads = 256;

template <bool COUNT>
__global__ void __launch_bounds__(kInputThreads) any_negative(const int32_t *src, int64_t n, uint32_t *flag) {
    bool neg = false;
    uint32_t nz = 0;
    unsigned long long sum = 0;
    auto look = [&](int32_t v) {
        neg |= v < 0;
        if (COUNT) {
            nz += v != 0 ? 1u : 0u;
            sum += (unsigned long long)max(v, 0);
        }
    };
    const int64_t first = (int64_t)blockIdx.x * kInputThreads + threadIdx.x, step = (int64_t)gridDim.x * kInputThreads;
    const int64_t n4 = (reinterpret_cast<uintptr_t>(src) & 15u) == 0 ? n / 4 : 0;
    for (int64_t i = first; i < n4; i += step) {
        const int4 v = reinterpret_cast<const int4 *>(src)[i];
        look(v.x);
        look(v.y);
        look(v.z);
        look(v.w);
    }
    for (int64_t i = 4 * n4 + first; i < n; i += step) look(src[i]);
    if (__syncthreads_or(neg) && threadIdx.x == 0) atomicOr(flag, 1u);
    if (COUNT) {
        __shared__ uint32_t s_nz[kInputThreads / 32];
        __shared__ unsigned long long s_sum[kInputThreads / 32];
        nz = __reduce_add_sync(0xFFFFFFFFu, nz);
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, d);
        if ((threadIdx.x & 31) == 0) {
            s_nz[threadIdx.x / 32] = nz;
            s_sum[threadIdx.x / 32] = sum;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int k = 1; k < kInputThreads / 32; ++k) {
                nz += s_nz[k];
                sum += s_sum[k];
            }
            if (nz) {
                atomicAdd(flag + 1, nz);
                atomicAdd(reinterpret_cast<unsigned long long *>(flag + 2), sum);
            }
        }
    }
}

// blocks for n counts: two loads of four per thread, up to a resident wave
unsigned input_blocks(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, 8 * 152)); }

// The tiles every tile of a flow launch waits for (CSR): itself and every tile
// holding a face neighbour of one of its tets. Tiles of B tets in device order.
void flow_neighbours(const std::vector<int32_t> &nbr_dev, int64_t T, int64_t B, std::vector<int32_t> &off,
                     std::vector<int32_t> &nb) {
    std::vector<int32_t> tmp;
    for (int64_t t = 0; t * B < T; ++t) {
        tmp.assign(1, (int32_t)t);
        for (int64_t d = 4 * t * B; d < 4 * std::min(T, (t + 1) * B); ++d) {
            const int32_t j = nbr_dev[(size_t)d];
            if (j >= 0 && j / B != t) tmp.push_back((int32_t)(j / B));
        }
        std::sort(tmp.begin(), tmp.end());
        off.push_back((int32_t)nb.size());
        nb.insert(nb.end(), tmp.begin(), std::unique(tmp.begin(), tmp.end()));
    }
}

// Launch-form choices of tuned simulations, shared by every simulation of
// the same compiled kernel, tet count, block size and molecules per tet (to a
// power of two; clones of one prototype, the jobs of a stream): the first
// one's tuning run decides. (A tenth of the benchmark box's molecules runs 14 %
// faster in another form than the box.)
struct FlowChoice {
    int pick;
    float ms[kForms];
};
std::mutex g_flow_mu;
std::map<std::tuple<const void *, int64_t, int, int>, FlowChoice> g_flow_choice;

bool cuda_ok(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return true;
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return false;
}

// Device allocations of simulations and batches. A test makes one of its
// thread's fail (steps_debug_fail_alloc): the paths that follow cannot be
// reached by filling the device.
thread_local int32_t t_fail_alloc = 0;
thread_local int32_t t_form = 0;  // steps_debug_form
thread_local int64_t t_allocs = 0;

cudaError_t device_alloc(void **p, size_t bytes) {
    if (t_fail_alloc > 0 && --t_fail_alloc == 0) return cudaErrorMemoryAllocation;
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) ++t_allocs;
    else cudaGetLastError();
    return e;
}

}  // namespace

struct steps_sim {
    // the host tables, built once and shared by a simulation's clones (copied,
    // about 50 bytes a tet, they were half of what admitting a job cost)
    std::shared_ptr<Tables> tables;
    Tables &tab;
    HostModel model;
    steps_options opt{};
    cudaStream_t stream = nullptr;
    int device = -1;                // the device current at creation (owns every buffer below)
    bool failed = false;            // a bounded device wait ran out: later runs are refused
    int64_t T = 0;
    int64_t Tpad = 0;
    int S = 0;
    uint64_t seed = 0;
    // device state
    int32_t *d_cnt[2] = {nullptr, nullptr};
    int cur = 0;
    int4 *d_nbr = nullptr;
    uint4 *d_thr = nullptr;
    float *d_inv_nav = nullptr;
    int32_t *d_orig = nullptr;      // device index -> original id (null without reordering)
    int32_t *d_inv_perm = nullptr;  // original id -> device index (null without reordering)
    uint32_t *d_rmask = nullptr;
    std::vector<uint32_t> h_rmask;  // device order
    uint32_t *d_err = nullptr;      // [6]: window error word, unused, then any_negative's four
    uint64_t *d_window_base = nullptr;
    int32_t *d_stage = nullptr;     // [S * nt] original-order staging
    int32_t *d_rec = nullptr;       // recording selection (species, then tets)
    size_t rec_bytes = 0;
    void *spec = nullptr;           // step kernel compiled for this model (cached process-wide), or null
    int32_t *d_trial = nullptr;     // list form: [S][Tpad] trial counts that differ from the count
    uint32_t *d_leave[2] = {nullptr, nullptr};  // EXP leave law: [S][Tpad] tables of the full and the last window
    double *d_G = nullptr;          // [Tpad] the tets' total face rates, and
    uint32_t *d_leave_list = nullptr;  // the entries the host decides: their number, (species, tet) each, values
    std::string spec_why;           // why there is none
    // block tiles (steps_step.cuh) compiled for a model of many species, for
    // meshes of more than a resident wave of warp tiles, on first use
    void *spec_block = nullptr;
    bool block_tried = false;
    bool blocky = false;            // the present run's window launches go over block tiles
    int forced = 0;                 // a test's choice of form (steps_debug_form), or 0
    // list form (steps_list.cuh): its kernel, and per-simulation buffers
    void *spec_list = nullptr;
    uint32_t *d_tm[2] = {nullptr, nullptr};   // [Tpad] species words of both count buffers
    int32_t *d_list[2] = {nullptr, nullptr};  // [2 Tpad] the lists (a tet is listed twice at most)
    uint32_t *d_lcnt = nullptr;     // [4] their lengths (StepArgs::lcnt)
    uint4 *d_tetrec = nullptr;      // [Tpad] the tets' records (StepArgs::rec)
    int32_t *d_src = nullptr;       // models with order-0 reactions: the sources, a list
    uint32_t *d_srcbits = nullptr;  // and a bit each
    bool tm_valid = false;          // the species words match the counts
    bool list_valid = false;        // the next window's list matches the species words
    bool src_valid = false;         // the records and the sources match the reaction masks
    bool listing = false;           // the present run's windows go through the list form
    uint64_t list_built = 0;        // the window the list was last built for
    uint64_t looked = 0;            // the window its length was last looked at
    // Molecules per tet when all counts were last set; listed tets or non-zero
    // counts per tet, last known. Counts of single species leave both unknown
    // (negative): a run that needs one of them looks at the state (measure).
    double density = 0.0;
    double fill = 0.0;
    // time
    double t_base = 0.0;
    int64_t k_grid = 0;
    uint64_t k_total = 0;
    uint64_t launches = 0;
    uint32_t scale_full[kMaxSpecies] = {};
    // graphs of kGraphWindows full windows, one per starting buffer
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    // flow launches (a run's full windows in one launch), per block size: [0]
    // the simulation's, [1] 512 (a tuning candidate when the block is smaller),
    // [2] and [3] compiled block tiles of 256 and 512 tets.
    // Each holds its step kernel, the tiles' finished-window words and the item
    // counter (d_flow[nwords]) and, for a block-tile kernel, every tile's
    // neighbour tiles (tiles of `block` tets in device order, CSR).
    struct Flow {
        void *spec = nullptr;  // null with `generic`: the generic kernel's flow form (256-thread blocks)
        bool generic = false;
        int block = 0;
        bool tried = false;
        int32_t *d_tnb_off = nullptr;
        int32_t *d_tnb = nullptr;
        uint32_t *d_flow = nullptr;
        int64_t ntiles = 0;  // items per window
        int64_t nwords = 0;
        size_t bytes = 0;
    } flow[4];
    // flow = 0 (tuned): -1 not yet timed, 0 window launches, 1 + k flow launches
    // of flow[k] (k < 2); on block tiles 3 window launches, 2 + k flow[k] (k >= 2)
    int flow_pick = -1;
    int pick_bucket = 0;         // the bucket of the density it was made for
    float flow_ms[kForms] = {};  // tuning: ms per window of each

    // a clone's buffers: one allocation (a dozen, and as many frees, were most
    // of the time of admitting and retiring a served job)
    char *arena = nullptr;
    size_t arena_bytes = 0;
    void drop(void *p) {
        if (!(arena && static_cast<char *>(p) >= arena && static_cast<char *>(p) < arena + arena_bytes)) cudaFree(p);
    }

    using Request = std::pair<void **, size_t>;
    cudaError_t alloc_arena(const std::vector<Request> &want) {
        size_t n = 0;
        for (const Request &r : want) n += (r.second + 255) / 256 * 256;
        void *p = nullptr;
        const cudaError_t e = device_alloc(&p, n);
        if (e != cudaSuccess) return e;
        arena = static_cast<char *>(p);
        arena_bytes = n;
        size_t at = 0;
        for (const Request &r : want) {
            *r.first = arena + at;
            at += (r.second + 255) / 256 * 256;
        }
        return cudaSuccess;
    }

    explicit steps_sim(std::shared_ptr<Tables> t) : tables(std::move(t)), tab(*tables) {}

    double time() const { return k_grid == 0 ? t_base : t_base + (double)k_grid * tab.tau; }

    ~steps_sim() {
        for (auto &g : graph)
            if (g) cudaGraphExecDestroy(g);
        drop(d_cnt[0]);
        drop(d_cnt[1]);
        drop(d_nbr);
        drop(d_thr);
        drop(d_inv_nav);
        drop(d_orig);
        drop(d_inv_perm);
        drop(d_rmask);
        drop(d_err);
        drop(d_window_base);
        drop(d_stage);
        drop(d_rec);
        free_list();
        drop(d_leave[0]);
        drop(d_leave[1]);
        drop(d_G);
        drop(d_leave_list);
        for (Flow &f : flow) {
            cudaFree(f.d_tnb_off);
            cudaFree(f.d_tnb);
            cudaFree(f.d_flow);
        }
        cudaFree(arena);
    }

    // flow[k]'s kernel and tables (once): tile t lists itself and every tile
    // holding a face neighbour of one of its tets. flow[0] runs the
    // simulation's kernel (the generic one only at 256-thread blocks);
    // flow[1], 512-tet tiles of the specialised kernel, is compiled here. A
    // form without a kernel keeps no tables (d_flow null: no candidate).
    int ensure_flow(int k) {
        Flow &fl = flow[k];
        if (fl.d_flow || fl.tried) return STEPS_OK;
        fl.tried = true;
        const int64_t B = k == 0 ? opt.block : k == 2 ? 256 : 512;
        void *sp = k == 0   ? spec
                   : k == 2 ? spec_block
                   : !spec  ? nullptr
                            : k == 1 ? spec_kernel(model, 512, nullptr) : spec_block_kernel(model, 512);
        const bool generic = k == 0 && !spec;
        if (!sp && !(generic && B == 256)) return STEPS_OK;
        // a warp-tile kernel publishes per 32 tets and finds the tiles it waits
        // for from its tets' neighbours: it needs no lists
        const bool warp = k < 2 && (sp || model.dev.S <= kWarpGenericSpecies);
        const int64_t nt = (T + B - 1) / B, nwords = warp ? nt * (B / 32) : nt;
        std::vector<int32_t> off, nb;
        if (!warp) {
            try {
                flow_neighbours(tab.nbr_dev, T, B, off, nb);
                off.push_back((int32_t)nb.size());
            } catch (const std::bad_alloc &) {
                set_error("flow tables: out of host memory");
                return STEPS_ERR_OOM;
            }
        }
        int rc = STEPS_OK;
        if ((!warp && (!cuda_ok(device_alloc((void **)&fl.d_tnb_off, off.size() * 4), "flow tables") ||
                       !cuda_ok(device_alloc((void **)&fl.d_tnb, nb.size() * 4), "flow tables"))) ||
            !cuda_ok(device_alloc((void **)&fl.d_flow, ((size_t)nwords + 1) * 4), "flow tables"))
            rc = STEPS_ERR_OOM;
        // on the stream of the launches: a launch there waits for nothing the
        // default stream still has to do, and a word of an earlier simulation
        // in this memory would open a tile's wait at once
        if (!rc &&
            ((!warp && (!cuda_ok(cudaMemcpyAsync(fl.d_tnb_off, off.data(), off.size() * 4, cudaMemcpyHostToDevice, stream),
                                 "flow tables") ||
                        !cuda_ok(cudaMemcpyAsync(fl.d_tnb, nb.data(), nb.size() * 4, cudaMemcpyHostToDevice, stream),
                                 "flow tables"))) ||
             !cuda_ok(cudaMemsetAsync(fl.d_flow, 0, ((size_t)nwords + 1) * 4, stream), "flow tables")))
            rc = STEPS_ERR_CUDA;
        if (rc) {
            cudaFree(fl.d_tnb_off);
            cudaFree(fl.d_tnb);
            cudaFree(fl.d_flow);
            fl.d_tnb_off = fl.d_tnb = nullptr;
            fl.d_flow = nullptr;
            return rc;
        }
        fl.spec = sp;
        fl.generic = generic;
        fl.block = (int)B;
        fl.ntiles = nt;
        fl.nwords = nwords;
        fl.bytes = (off.size() + nb.size() + (size_t)nwords + 1) * 4;
        return STEPS_OK;
    }

    // EXP leave law: a table of more than kLeaveHostEntries waits for the stream,
    // so it comes before a run's windows
    bool leave_waits() const { return d_leave[0] && (int64_t)S * T > kLeaveHostEntries; }

    // the table of a window of length tau_k, smaller ones from the host
    int upload_leave(double tau_k, cudaStream_t st) {
        if (!d_leave[0]) return STEPS_OK;
        if (leave_waits() || !std::isfinite(tab.tau)) return device_leave(tau_k, st);
        try {
            std::vector<uint32_t> t;
            exp_leave_table(model, tab, tau_k, (size_t)Tpad, t);
            return cuda_ok(cudaMemcpyAsync(tau_k == tab.tau ? d_leave[0] : d_leave[1], t.data(), t.size() * 4,
                                           cudaMemcpyHostToDevice, st),
                           "leave table")
                       ? STEPS_OK
                       : STEPS_ERR_CUDA;
        } catch (const std::bad_alloc &) {
            set_error("leave table: out of host memory");
            return STEPS_ERR_OOM;
        }
    }

    // The table of a window of length tau_k, into the full window's buffer
    // (tau_k == tau) or the last window's, in stream order. The device computes
    // it and the host decides the entries it lists (leave_table); *decided, if
    // asked for, receives their number. Waits for the stream. 105,222 tets and
    // 10 species: 2.6 ms when the host computed all of it, 0.05 ms now.
    int device_leave(double tau_k, cudaStream_t st, uint32_t *decided = nullptr) {
        uint32_t *dst = tau_k == tab.tau ? d_leave[0] : d_leave[1];
        if (!std::isfinite(tab.tau))
            return cuda_ok(cudaMemsetAsync(dst, 0, (size_t)S * Tpad * 4, st), "leave table") ? STEPS_OK : STEPS_ERR_CUDA;
        LeaveRates r{};
        for (int s = 0; s < S; ++s) r.tauD[s] = model.D[(size_t)s] > 0.0 ? tau_k * model.D[(size_t)s] : 0.0;
        uint2 *d_list_ = reinterpret_cast<uint2 *>(d_leave_list + 2);
        uint32_t *d_value = d_leave_list + 2 + 2 * kLeaveListCap;
        if (!cuda_ok(cudaMemsetAsync(d_leave_list, 0, 4, st), "leave table")) return STEPS_ERR_CUDA;
        leave_table<<<(unsigned)((T + 255) / 256), 256, 0, st>>>(d_G, T, (size_t)Tpad, S, r, dst, d_list_, d_leave_list);
        constexpr uint32_t kFirst = 512;  // entries fetched with their number
        uint32_t h[2 + 2 * kFirst];
        if (!cuda_ok(cudaGetLastError(), "leave table") ||
            !cuda_ok(cudaMemcpyAsync(h, d_leave_list, sizeof(h), cudaMemcpyDeviceToHost, st), "leave table") ||
            !cuda_ok(cudaStreamSynchronize(st), "leave table"))
            return STEPS_ERR_CUDA;
        const uint32_t n = h[0];
        if (decided) *decided = n;
        if (n == 0) return STEPS_OK;
        try {
            if (n > kLeaveListCap) {  // not met by leave probabilities below 1: the whole table from the host
                std::vector<uint32_t> t;
                exp_leave_table(model, tab, tau_k, (size_t)Tpad, t);
                return cuda_ok(cudaMemcpyAsync(dst, t.data(), t.size() * 4, cudaMemcpyHostToDevice, st), "leave table") &&
                               cuda_ok(cudaStreamSynchronize(st), "leave table")
                           ? STEPS_OK
                           : STEPS_ERR_CUDA;
            }
            std::vector<uint32_t> at(2 * (size_t)n), value(n);
            std::memcpy(at.data(), h + 2, (size_t)std::min(n, kFirst) * 8);
            if (n > kFirst && (!cuda_ok(cudaMemcpyAsync(at.data() + 2 * kFirst, d_leave_list + 2 + 2 * kFirst,
                                                        (size_t)(n - kFirst) * 8, cudaMemcpyDeviceToHost, st),
                                        "leave table") ||
                               !cuda_ok(cudaStreamSynchronize(st), "leave table")))
                return STEPS_ERR_CUDA;
            for (uint32_t k = 0; k < n; ++k) value[k] = exp_leave_entry(tau_k * model.D[at[2 * k]], tab.G_dev[at[2 * k + 1]]);
            if (!cuda_ok(cudaMemcpyAsync(d_value, value.data(), (size_t)n * 4, cudaMemcpyHostToDevice, st), "leave table"))
                return STEPS_ERR_CUDA;
            patch_leave<<<(n + 255) / 256, 256, 0, st>>>(d_list_, d_value, n, (size_t)Tpad, dst);
            return cuda_ok(cudaGetLastError(), "leave table") ? STEPS_OK : STEPS_ERR_CUDA;
        } catch (const std::bad_alloc &) {
            set_error("leave table: out of host memory");
            return STEPS_ERR_OOM;
        }
    }

    // The windows of a run to t_end (the loop of Algorithm 1): full ones, and the
    // length of a shortened last one (0: none).
    void schedule(double t_end, int64_t *full, double *partial) const {
        const double tau = tab.tau;
        const bool finite = std::isfinite(tau);
        const double tol = finite ? 1e-9 * tau : 0.0;
        *partial = 0.0;
        for (*full = 0;; ++*full) {
            const int64_t k = k_grid + *full;
            const double t = k == 0 ? t_base : t_base + (double)k * tau;
            if (!(t_end - t > tol)) return;
            if (!finite || !(t + tau <= t_end + tol)) {
                *partial = t_end - t;
                return;
            }
        }
    }

    void free_list() {
        for (void **p : {(void **)&d_tm[0], (void **)&d_tm[1], (void **)&d_list[0], (void **)&d_list[1],
                         (void **)&d_lcnt, (void **)&d_tetrec, (void **)&d_trial, (void **)&d_src, (void **)&d_srcbits}) {
            drop(*p);
            *p = nullptr;
        }
    }

    // the list form's buffers
    std::vector<Request> list_requests() {
        const size_t n = (size_t)Tpad * 4;
        std::vector<Request> r = {{(void **)&d_tm[0], n},       {(void **)&d_tm[1], n}, {(void **)&d_list[0], 2 * n},
                                  {(void **)&d_list[1], 2 * n}, {(void **)&d_lcnt, 16}, {(void **)&d_tetrec, 4 * n},
                                  {(void **)&d_trial, (size_t)S * n}};
        if (model.dev.order0) {
            r.emplace_back((void **)&d_src, n);
            r.emplace_back((void **)&d_srcbits, n / 32);
        }
        return r;
    }

    bool wants_list() const {
        return spec_list && opt.flow != 1 && fill >= 0.0 && fill <= kListFill &&
               (forced || (T >= kListMinTets && fill * (double)T <= kListMost)) && plain_rates(model, tab);
    }

    // whether block tiles are a form of this simulation at all
    bool block_possible() const {
        return spec && S >= kListMinSpecies && (forced ? forced == 3 : opt.flow != 1 && T > warp_wave(S));
    }

    // their kernels, and the trial buffer they need
    bool ensure_block() {
        if (!spec_block && !block_tried && block_possible()) {
            block_tried = true;
            void *k = spec_block_kernel(model, 256);
            if (k && ensure_trial()) spec_block = k;
        }
        return spec_block != nullptr;
    }

    // window launches over block tiles, at a density of d molecules per tet
    bool wants_block(double d) {
        if (!block_possible()) return false;
        if (flow_pick >= 0 && !stale() ? flow_pick < 3 : !forced && !(d >= 0.0 && d <= block_density(S, T))) return false;
        return ensure_block();
    }

    // density and fill of the present state; waits for the stream
    int measure(cudaStream_t st) {
        uint32_t seen[4] = {0, 0, 0, 0};
        const int64_t n = (int64_t)S * Tpad;  // (the padding is zero)
        if (!cuda_ok(cudaMemsetAsync(d_err + 2, 0, 16, st), "state measure")) return STEPS_ERR_CUDA;
        any_negative<true><<<input_blocks(n), kInputThreads, 0, st>>>(d_cnt[cur], n, d_err + 2);
        if (!cuda_ok(cudaGetLastError(), "state measure") ||
            !cuda_ok(cudaMemcpyAsync(seen, d_err + 2, 16, cudaMemcpyDeviceToHost, st), "state measure") ||
            !cuda_ok(cudaStreamSynchronize(st), "state measure"))
            return STEPS_ERR_CUDA;
        found(seen);
        return STEPS_OK;
    }

    // density and fill from any_negative's words over all counts
    void found(const uint32_t seen[4]) {
        fill = seen[1] / (double)T;
        density = (double)((uint64_t)seen[3] << 32 | seen[2]) / (double)T;
    }

    // the trial buffer that block tiles of 16 or more species need
    bool ensure_trial() {
        if (d_trial || !spec_block_trial(model)) return true;
        if (device_alloc((void **)&d_trial, (size_t)S * (size_t)Tpad * 4) != cudaSuccess) return false;
        drop_graphs();  // (captured launches hold the arguments)
        return true;
    }

    // Before a run, and within long ones: the form of its windows, by what is
    // known of the state. A list's length is looked at (the stream waited for)
    // every kListCheckWindows, also over the intervals of a recording.
    int choose_form() {
        if (listing && k_total - looked >= kListCheckWindows) {
            uint32_t c[4];
            if (!cuda_ok(cudaMemcpyAsync(c, d_lcnt, 16, cudaMemcpyDeviceToHost, stream), "list length") ||
                !cuda_ok(cudaStreamSynchronize(stream), "list length"))
                return STEPS_ERR_CUDA;
            fill_from(c);
        }
        if ((spec_list && opt.flow != 1 && fill < 0.0) || (block_possible() && density < 0.0))
            if (int rc = measure(stream)) return rc;
        const bool want = wants_list(), block = !want && wants_block(density);
        if (want != listing || block != blocky) drop_graphs();
        if (want != listing) looked = k_total;
        listing = want;
        blocky = block;
        if (!listing) tm_valid = list_valid = false;  // the other kernels leave them behind
        return STEPS_OK;
    }

    // Before windows in the list form: the species words match the counts, the
    // records and sources the masks, and the list is window k_total's. Windows
    // append tets in the order their warps meet them; building the list afresh
    // now and then keeps neighbours together.
    int prepare_list(cudaStream_t st) {
        if (!listing || (tm_valid && src_valid && list_valid && k_total - list_built < kListWindows)) return STEPS_OK;
        const unsigned grid = (unsigned)((T + 255) / 256);
        if (!tm_valid)
            build_species_words<<<grid, 256, 0, st>>>(d_cnt[cur], T, (size_t)Tpad, S, d_tm[cur], d_tm[1 - cur]);
        if (!cuda_ok(cudaMemsetAsync(d_lcnt, 0, src_valid ? 12 : 16, st), "tet lists")) return STEPS_ERR_CUDA;
        if (!src_valid)
            build_sources<<<grid, 256, 0, st>>>(d_rmask, model.dev.order0, T, d_thr, d_orig, d_inv_nav, d_tetrec,
                                                    d_srcbits, d_src, d_lcnt + 3);
        build_list<<<grid, 256, 0, st>>>(d_tm[cur], T, d_srcbits, d_list[k_total & 1], d_lcnt + k_total % 3);
        if (!cuda_ok(cudaGetLastError(), "tet lists")) return STEPS_ERR_CUDA;
        tm_valid = src_valid = list_valid = true;
        list_built = k_total;
        return STEPS_OK;
    }

    // n full windows in the list form, as long as the state stays sparse: their
    // number into *done
    int list_windows(int64_t n, int64_t *done) {
        while (listing && *done < n) {
            int rc = choose_form();
            if (rc) return rc;
            if (!listing) break;
            const int64_t m = std::min(n - *done, (int64_t)(kListCheckWindows - (k_total - looked)));
            rc = window_launches(m);
            if (rc) return rc;
            *done += m;
        }
        return STEPS_OK;
    }

    // the fill from the list's lengths after the last window enqueued
    void fill_from(const uint32_t c[4]) {
        if (list_valid) fill = ((double)c[k_total % 3] + (d_src ? 0.5 * (double)c[3] : 0.0)) / (double)T;
        looked = k_total;
    }

    void drop_graphs() {
        for (auto &g : graph) {
            if (g) cudaGraphExecDestroy(g);
            g = nullptr;
        }
    }

    StepArgs args(int from, uint64_t window, const uint64_t *base, double tau_k, const uint32_t *scale) const {
        StepArgs a;
        std::memset(&a, 0, sizeof(a));
        a.cur = d_cnt[from];
        a.nxt = d_cnt[1 - from];
        a.nbr = d_nbr;
        a.thr = d_thr;
        a.inv_nav = d_inv_nav;
        a.orig = d_orig;
        a.rmask = d_rmask;
        a.err = d_err;
        a.T = (int32_t)T;
        a.Tpad = (int32_t)Tpad;
        a.key0 = (uint32_t)seed;
        a.key1 = (uint32_t)(seed >> 32);
        for (uint32_t k0 = a.key0, k1 = a.key1, r = 0; r < 10; ++r, k0 += 0x9E3779B9u, k1 += 0xBB67AE85u) {
            (r & 1 ? a.rk[r / 2].z : a.rk[r / 2].x) = k0;  // Philox key schedule: Weyl steps of the key
            (r & 1 ? a.rk[r / 2].w : a.rk[r / 2].y) = k1;
        }
        a.window = window;
        a.window_base = base;
        a.tau_k = tau_k;
        a.inv_tau_k = 1.0 / tau_k;
        a.tau_dn = (float)tau_k;
        if ((double)a.tau_dn > tau_k) a.tau_dn = std::nextafter(a.tau_dn, 0.0f);
        a.occ = opt.occupancy;
        a.lanes = 32;
        a.prefetch = 1;  // the launch sets the distance: half a resident wave
        a.trial = d_trial;
        a.tm_cur = d_tm[from];
        a.tm_nxt = d_tm[1 - from];
        a.rec = d_tetrec;
        a.list[0] = d_list[0];
        a.list[1] = d_list[1];
        a.lcnt = d_lcnt;
        a.src = d_src;
        a.srcbits = d_srcbits;
        a.leave = d_leave[0] ? (tau_k == tab.tau ? d_leave[0] : d_leave[1]) : nullptr;
        std::memcpy(a.scale, scale, sizeof(a.scale));
        return a;
    }

    // one window on the model-specialised kernel if there is one, else the generic one
    int launch(const StepArgs &a, cudaStream_t st) const {
        if (listing || blocky) return launch_spec(listing ? spec_list : spec_block, model.dev, a, opt.block, st);
        return spec ? launch_spec(spec, model.dev, a, opt.block, st) : launch_step(model.dev, a, opt.block, st);
    }

    int window_launch(double tau_k) {  // one window of explicit length, plain launch
        uint32_t scale[kMaxSpecies] = {};
        for (int s = 0; s < S; ++s) scale[s] = species_scale(model, tab, s, tau_k);
        if (d_leave[0] && !leave_waits() && tau_k != tab.tau)
            if (int rl = upload_leave(tau_k, stream)) return rl;
        StepArgs a = args(cur, k_total, nullptr, tau_k, scale);
        int rc = prepare_list(stream);
        if (!rc) rc = launch(a, stream);
        if (rc) return rc;
        ++launches;
        cur = 1 - cur;
        ++k_total;
        return STEPS_OK;
    }

    int capture_graph(int from) {
        cudaStream_t cs = nullptr;
        if (!cuda_ok(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "cudaStreamCreate")) return STEPS_ERR_CUDA;
        int rc = STEPS_OK;
        cudaGraph_t g = nullptr;
        if (!cuda_ok(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture")) {
            cudaStreamDestroy(cs);
            return STEPS_ERR_CUDA;
        }
        int b = from;
        for (int q = 0; q < kGraphWindows && rc == STEPS_OK; ++q) {
            StepArgs a = args(b, (uint64_t)q, d_window_base, tab.tau, scale_full);
            rc = launch(a, cs);
            b = 1 - b;
        }
        if (rc == STEPS_OK) rc = launch_add_u64(d_window_base, kGraphWindows, cs);
        cudaError_t e = cudaStreamEndCapture(cs, &g);
        if (rc == STEPS_OK && !cuda_ok(e, "cudaStreamEndCapture")) rc = STEPS_ERR_CUDA;
        if (rc == STEPS_OK && !cuda_ok(cudaGraphInstantiate(&graph[from], g, 0), "cudaGraphInstantiate"))
            rc = STEPS_ERR_CUDA;
        if (g) cudaGraphDestroy(g);
        cudaStreamDestroy(cs);
        return rc;
    }

    // a flow kernel exists for the simulation's block size
    bool flow_possible() const { return spec || opt.block == 256; }

    // the flow launches of a run's full windows: flow[k], or -1 for window launches
    int flow_form() const {
        if (!flow_possible()) return -1;
        if (opt.flow == 1) return blocky ? 2 : 0;
        return opt.flow != 0 ? -1 : flow_pick >= 4 ? (blocky ? flow_pick - 2 : -1) : flow_pick == 1 || flow_pick == 2 ? flow_pick - 1 : -1;
    }

    // n full windows: flow launches or window launches (all give the same bits)
    int full_windows(int64_t n) {
        int64_t listed = 0;
        if (int rl = list_windows(n, &listed)) return rl;
        n -= listed;
        if (n == 0) return STEPS_OK;
        if (opt.flow == 0 && (flow_pick < 0 || stale()) && flow_possible() && forced != 3 && n >= tune_windows()) {
            int64_t used = 0;
            int rc = tune_flow(&used);
            if (!rc) rc = choose_form();
            if (rc) return rc;
            n -= used;
        }
        const int k = n >= 2 ? flow_form() : -1;
        return k >= 0 ? flow_windows(n, k) : window_launches(n);
    }


    // molecules per tet, to a power of two
    int bucket() const { return (int)std::lrint(std::log2(std::max(density, 0.0) + 0.01)); }

    // whether a tuned choice was made for another state: the next run that is
    // long enough tunes again (or looks the choice up)
    bool stale() const { return flow_pick >= 0 && density >= 0.0 && bucket() != pick_bucket; }

    // full windows that the tuning takes
    int64_t tune_windows() const {
        return block_possible() && density <= tuned_block_density(S) ? kFormTuneWindows : kFlowTuneWindows;
    }

    // The first run with enough full windows times the launch forms on
    // alternating groups of windows: window launches, flow launches at the
    // simulation's block size and, when that is below 512, flow launches of
    // 512-tet tiles; then both forms of block tiles where the model and mesh
    // have them. One warm round, so that one-time costs do not decide, then two
    // timed rounds, so that the state's slow drift cancels. The fastest other
    // form is kept when it is more than 2 % faster than window launches. The
    // windows taken are ordinary windows of the run.
    int tune_flow(int64_t *used) {
        if (density < 0.0)
            if (int rc = measure(stream)) return rc;
        // the best form depends on the state: by powers of two of the molecules per tet
        const auto key = std::make_tuple((const void *)spec, T, opt.block, bucket());
        pick_bucket = bucket();
        {
            std::lock_guard<std::mutex> lock(g_flow_mu);
            auto it = g_flow_choice.find(key);
            if (it != g_flow_choice.end() && (it->second.pick < 3 || ensure_block())) {
                flow_pick = it->second.pick;
                std::memcpy(flow_ms, it->second.ms, sizeof(flow_ms));
                return STEPS_OK;
            }
        }
        int rc = ensure_flow(0);
        if (!rc && opt.block < 512) rc = ensure_flow(1);
        if (rc) return rc;
        int form[kForms] = {0}, nc = 1;
        for (int k = 0; k < 2; ++k)
            if (flow[k].d_flow) form[nc++] = 1 + k;
        const int64_t windows = tune_windows();
        if (windows == kFormTuneWindows && ensure_block()) {
            form[nc++] = 3;
            // (512-tet tiles, another program to compile, are only faster where a
            // window is few waves: 138,720 tets and 20 species 10.8 -> 9.1 us)
            for (int k = 2; k < (T < kListMinTets ? 4 : 3); ++k)
                if (ensure_flow(k) == STEPS_OK && flow[k].d_flow) form[nc++] = 2 + k;
        }
        flow_pick = 0;
        if (nc == 1) return STEPS_OK;
        cudaEvent_t e[kForms + 1] = {};
        for (auto &ev : e)
            if (!cuda_ok(cudaEventCreate(&ev), "flow tuning event")) {
                for (auto &x : e)
                    if (x) cudaEventDestroy(x);
                return STEPS_ERR_CUDA;
            }
        float tot[kForms] = {};
        const int64_t g = windows / (3 * nc);  // windows per group (too few for a graph)
        for (int round = 0; round < 3 && rc == STEPS_OK; ++round) {
            for (int c = 0; c < nc && rc == STEPS_OK; ++c) {
                if (!cuda_ok(cudaEventRecord(e[c], stream), "flow tuning")) rc = STEPS_ERR_CUDA;
                blocky = form[c] == 3;
                if (!rc) rc = form[c] % 3 == 0 ? window_launches(g) : flow_windows(g, form[c] >= 4 ? form[c] - 2 : form[c] - 1);
                *used += g;
            }
            if (!rc && !cuda_ok(cudaEventRecord(e[nc], stream), "flow tuning")) rc = STEPS_ERR_CUDA;
            if (!rc && !cuda_ok(cudaEventSynchronize(e[nc]), "flow tuning")) rc = STEPS_ERR_CUDA;
            for (int c = 0; c < nc && rc == STEPS_OK; ++c) {
                float ms = 0.f;
                if (!cuda_ok(cudaEventElapsedTime(&ms, e[c], e[c + 1]), "flow tuning")) rc = STEPS_ERR_CUDA;
                else if (round > 0) tot[c] += ms;
            }
        }
        if (windows == kFormTuneWindows) drop_graphs();  // (captured before, perhaps of another form)
        for (auto &x : e) cudaEventDestroy(x);
        if (rc) return rc;
        int best = 1;
        for (int c = 2; c < nc; ++c)
            if (tot[c] < tot[best]) best = c;
        for (int c = 0; c < nc; ++c) flow_ms[form[c]] = tot[c] / (2.f * (float)g);
        flow_pick = tot[best] < 0.98f * tot[0] ? form[best] : 0;
        std::lock_guard<std::mutex> lock(g_flow_mu);
        FlowChoice ch;
        ch.pick = flow_pick;
        std::memcpy(ch.ms, flow_ms, sizeof(flow_ms));
        g_flow_choice[key] = ch;
        return STEPS_OK;
    }

    // n full windows, one launch each (graph replay of kGraphWindows at a time)
    int window_launches(int64_t n) {
        int64_t done = 0;
        if (opt.use_graph && n >= kGraphWindows) {
            if (!graph[cur]) {
                int rc = capture_graph(cur);
                if (rc) return rc;
            }
            set_u64_kernel<<<1, 1, 0, stream>>>(d_window_base, k_total);
            if (!cuda_ok(cudaGetLastError(), "set window base")) return STEPS_ERR_CUDA;
            ++launches;
            while (n - done >= kGraphWindows) {
                int rc = prepare_list(stream);
                if (rc) return rc;
                if (!cuda_ok(cudaGraphLaunch(graph[cur], stream), "cudaGraphLaunch")) return STEPS_ERR_CUDA;
                launches += kGraphWindows + 1;
                done += kGraphWindows;
                k_total += kGraphWindows;  // even: cur unchanged
            }
        }
        for (; done < n; ++done) {
            StepArgs a = args(cur, k_total, nullptr, tab.tau, scale_full);
            int rc = prepare_list(stream);
            if (!rc) rc = launch(a, stream);
            if (rc) return rc;
            ++launches;
            cur = 1 - cur;
            ++k_total;
        }
        return STEPS_OK;
    }

    // n full windows through launches of flow[k]'s kernel (one per 2^31 items)
    int flow_windows(int64_t n, int k) {
        int rc = ensure_flow(k);
        if (rc) return rc;
        const Flow &fl = flow[k];
        if (!fl.d_flow) return window_launches(n);
        const int64_t ntiles = fl.ntiles;
        uint32_t *const d_flow = fl.d_flow;
        const int64_t cap = std::max<int64_t>(1, (int64_t)0x7FFFFFFF / ntiles);
        for (int64_t done = 0; done < n;) {
            const int64_t nw = std::min(n - done, cap);
            if (!cuda_ok(cudaMemsetAsync(d_flow + fl.nwords, 0, 4, stream), "flow counter")) return STEPS_ERR_CUDA;
            StepArgs a = args(cur, k_total, nullptr, tab.tau, scale_full);
            FlowArgs f;
            f.tnb_off = fl.d_tnb_off;
            f.tnb = fl.d_tnb;
            f.tile_done = d_flow;
            f.fetch = d_flow + fl.nwords;
            f.nwin = (uint32_t)nw;
            f.ntiles = (uint32_t)ntiles;
            rc = fl.generic ? launch_flow(model.dev, a, f, fl.block, stream)
                            : launch_spec_flow(fl.spec, model.dev, a, f, fl.block, stream);
            if (rc) return rc;
            ++launches;
            done += nw;
            k_total += (uint64_t)nw;
            if (nw & 1) cur = 1 - cur;
        }
        return STEPS_OK;
    }
};

#define CHECK_NULL(p, name)                                    \
    do {                                                       \
        if (!(p)) {                                            \
            set_error(std::string(name) + ": NULL argument");  \
            return STEPS_ERR_ARG;                              \
        }                                                      \
    } while (0)

extern "C" {

const char *steps_last_error(void) { return g_last_error.c_str(); }

void steps_options_default(steps_options *opt) {
    if (!opt) return;
    std::memset(opt, 0, sizeof(*opt));
    opt->occupancy = STEPS_OCC_MEAN;
    opt->reorder = STEPS_REORDER_MORTON;
    opt->block = 256;
    opt->use_graph = 1;
    opt->specialize = 0;
}

int steps_mesh_create(const double *verts_xyz, int64_t nv, const int32_t *tets, int64_t nt, steps_mesh **out) {
    CHECK_NULL(out, "steps_mesh_create");
    *out = nullptr;
    std::unique_ptr<steps_mesh> m(new (std::nothrow) steps_mesh);
    if (!m) {
        set_error("steps_mesh_create: out of host memory");
        return STEPS_ERR_OOM;
    }
    int rc;
    try {
        rc = build_mesh(verts_xyz, nv, tets, nt, m->m);
    } catch (const std::bad_alloc &) {
        set_error("steps_mesh_create: out of host memory");
        return STEPS_ERR_OOM;
    }
    if (rc) return rc;
    *out = m.release();
    return STEPS_OK;
}

void steps_mesh_destroy(steps_mesh *mesh) { delete mesh; }

int steps_mesh_num_tets(const steps_mesh *mesh, int64_t *nt) {
    CHECK_NULL(mesh, "steps_mesh_num_tets");
    CHECK_NULL(nt, "steps_mesh_num_tets");
    *nt = mesh->m.nt;
    return STEPS_OK;
}

int steps_model_create(int32_t n_species, const double *diff, int32_t n_reac, const int32_t *lhs,
                       const int32_t *rhs, const double *k, steps_model **out) {
    CHECK_NULL(out, "steps_model_create");
    *out = nullptr;
    std::unique_ptr<steps_model> m(new (std::nothrow) steps_model);
    if (!m) {
        set_error("steps_model_create: out of host memory");
        return STEPS_ERR_OOM;
    }
    int rc = build_model(n_species, diff, n_reac, lhs, rhs, k, m->m);
    if (rc) return rc;
    *out = m.release();
    return STEPS_OK;
}

void steps_model_destroy(steps_model *model) { delete model; }

int steps_sim_create(const steps_mesh *mesh, const steps_model *model, uint64_t seed, const steps_options *opt,
                     void *cuda_stream, steps_sim **out) try {
    CHECK_NULL(out, "steps_sim_create");
    *out = nullptr;
    CHECK_NULL(mesh, "steps_sim_create");
    CHECK_NULL(model, "steps_sim_create");
    std::unique_ptr<steps_sim> s;
    try {
        s.reset(new steps_sim(std::make_shared<Tables>()));
    } catch (const std::bad_alloc &) {
        set_error("steps_sim_create: out of host memory");
        return STEPS_ERR_OOM;
    }
    if (opt) {
        s->opt = *opt;
        if (s->opt.block == 0) s->opt.block = 256;
        if (s->opt.block != 64 && s->opt.block != 128 && s->opt.block != 256 && s->opt.block != 512) {
            set_error("steps_sim_create: block must be 64, 128, 256 or 512");
            return STEPS_ERR_ARG;
        }
        if (s->opt.occupancy != STEPS_OCC_MEAN && s->opt.occupancy != STEPS_OCC_END) {
            set_error("steps_sim_create: bad occupancy mode");
            return STEPS_ERR_ARG;
        }
        if (s->opt.leave_law != STEPS_LEAVE_EULER && s->opt.leave_law != STEPS_LEAVE_EXP) {
            set_error("steps_sim_create: bad leave law");
            return STEPS_ERR_ARG;
        }
        if (s->opt.reorder != STEPS_REORDER_NONE && s->opt.reorder != STEPS_REORDER_MORTON &&
            s->opt.reorder != STEPS_REORDER_RCM) {
            set_error("steps_sim_create: bad reorder");
            return STEPS_ERR_ARG;
        }
        if (s->opt.flow < -1 || s->opt.flow > 1) {
            set_error("steps_sim_create: flow must be 0 (tuned), 1 (on) or -1 (off)");
            return STEPS_ERR_ARG;
        }
        if (s->opt.leave_law == STEPS_LEAVE_EXP) {
            if (s->opt.specialize < 0) {
                set_error("steps_sim_create: the EXP leave law runs on the model-specialised kernel only "
                          "(specialize must be 0 or 1)");
                return STEPS_ERR_ARG;
            }
            s->opt.specialize = 1;
        }
    } else {
        steps_options_default(&s->opt);
    }
    s->forced = t_form;
    s->model = model->m;
    s->model.leave_exp = s->opt.leave_law == STEPS_LEAVE_EXP;
    s->stream = (cudaStream_t)cuda_stream;
    if (!cuda_ok(cudaGetDevice(&s->device), "steps_sim_create: cudaGetDevice")) return STEPS_ERR_CUDA;
    s->T = mesh->m.nt;
    s->Tpad = (s->T + 31) / 32 * 32;
    s->S = s->model.S;
    s->seed = seed;
    try {
        build_tables(mesh->m, s->model, s->opt.reorder, s->tab);
    } catch (const std::bad_alloc &) {
        set_error("steps_sim_create: out of host memory");
        return STEPS_ERR_OOM;
    }
    for (int sp = 0; sp < s->S; ++sp) s->scale_full[sp] = species_scale(s->model, s->tab, sp, s->tab.tau);

    const size_t T = (size_t)s->T, Tpad = (size_t)s->Tpad, S = (size_t)s->S;
    bool reordered = false;
    for (size_t d = 0; d < T && !reordered; ++d) reordered = s->tab.perm[d] != (int32_t)d;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) e = device_alloc(p, bytes);
    };
    alloc((void **)&s->d_cnt[0], S * Tpad * 4);
    alloc((void **)&s->d_cnt[1], S * Tpad * 4);
    // per-tet tables are padded to Tpad entries (zeros) so that the step
    // kernel's bulk copies of a block's tile are whole multiples of 16 bytes
    alloc((void **)&s->d_nbr, Tpad * 16);
    alloc((void **)&s->d_thr, Tpad * 16);
    alloc((void **)&s->d_inv_nav, Tpad * 4);
    alloc((void **)&s->d_err, 24);
    alloc((void **)&s->d_window_base, 8);
    alloc((void **)&s->d_stage, S * T * 4);
    if (reordered) {
        alloc((void **)&s->d_orig, Tpad * 4);
        alloc((void **)&s->d_inv_perm, T * 4);
    }
    if (s->model.leave_exp) {
        alloc((void **)&s->d_leave[0], S * Tpad * 4);
        alloc((void **)&s->d_leave[1], S * Tpad * 4);
        alloc((void **)&s->d_G, Tpad * 8);
        alloc((void **)&s->d_leave_list, kLeaveListBytes);
    }
    if (e != cudaSuccess) {
        set_error(std::string("steps_sim_create: device allocation failed: ") + cudaGetErrorString(e));
        cudaGetLastError();
        return STEPS_ERR_OOM;
    }
    // every upload on the simulation's stream, so that its launches come after
    // them whatever the default stream is busy with
    const cudaStream_t st = s->stream;
    auto fill = [&](void *p, int byte, size_t n) { return cuda_ok(cudaMemsetAsync(p, byte, n, st), "memset"); };
    auto put = [&](void *p, const void *src, size_t n, const char *what) {
        return cuda_ok(cudaMemcpyAsync(p, src, n, cudaMemcpyHostToDevice, st), what);
    };
    bool ok = fill(s->d_nbr, 0xFF, Tpad * 16) && fill(s->d_thr, 0, Tpad * 16) && fill(s->d_inv_nav, 0, Tpad * 4) &&
              put(s->d_nbr, s->tab.nbr_dev.data(), T * 16, "upload nbr") &&
              put(s->d_thr, s->tab.thr_dev.data(), T * 16, "upload thr") &&
              put(s->d_inv_nav, s->tab.inv_nav_dev.data(), T * 4, "upload inv_nav") &&
              fill(s->d_cnt[0], 0, S * Tpad * 4) && fill(s->d_cnt[1], 0, S * Tpad * 4) && fill(s->d_err, 0, 24) &&
              fill(s->d_window_base, 0, 8);
    if (ok && reordered)
        ok = fill(s->d_orig, 0, Tpad * 4) && put(s->d_orig, s->tab.perm.data(), T * 4, "upload perm") &&
             put(s->d_inv_perm, s->tab.inv_perm.data(), T * 4, "upload inv_perm");
    if (ok && s->model.leave_exp)
        ok = fill(s->d_leave[0], 0, S * Tpad * 4) && fill(s->d_leave[1], 0, S * Tpad * 4) &&
             put(s->d_G, s->tab.G_dev.data(), T * 8, "upload G") && s->upload_leave(s->tab.tau, st) == STEPS_OK;
    // (a clone on another stream reads the tables as soon as this call returns)
    if (!ok || !cuda_ok(cudaStreamSynchronize(st), "steps_sim_create")) return STEPS_ERR_CUDA;
    // the model-specialised step kernel (compiled once per model and block size)
    constexpr int64_t kSpecializeMinTets = 65536;
    if (s->opt.specialize > 0 || (s->opt.specialize == 0 && s->T >= kSpecializeMinTets)) {
        // the second program of a model of many species, compiled beside the
        // first (2.1 s each): the list form's, or on smaller meshes block tiles,
        // for this simulation or a batch of its clones (on meshes that have the
        // list form's they come on first use)
        const bool many = s->S >= kListMinSpecies && s->opt.flow != 1;
        const bool list = many && (s->forced ? s->forced == 2 : s->T >= kListMinTets);
        const bool block = many && !list && s->T < kListMinTets && (s->opt.specialize > 0 || s->T > warp_wave(s->S));
        std::future<void *> second;
        if (list || block) try {
                second = std::async(std::launch::async, [&s, list]() -> void * {
                    cudaSetDevice(s->device);
                    return list ? spec_list_kernel(s->model) : spec_block_kernel(s->model, 256);
                });
            } catch (const std::system_error &) {  // no thread: compiled when it is asked for below
            }
        s->spec = spec_kernel(s->model, s->opt.block, &s->spec_why);
        if (second.valid()) second.get();
        if (!s->spec && s->opt.specialize > 0) {
            set_error("steps_sim_create: the specialised step kernel could not be built: " + s->spec_why);
            return STEPS_ERR_CUDA;
        }
        if (s->spec && list) {
            s->spec_list = spec_list_kernel(s->model);
            if (s->spec_list)
                for (const steps_sim::Request &r : s->list_requests()) alloc(r.first, r.second);
            if (e != cudaSuccess) {  // no room for the list form: the simulation runs its tiles
                s->free_list();
                s->spec_list = nullptr;
            }
        }
    } else {
        s->spec_why = "not requested";
    }
    *out = s.release();
    return STEPS_OK;
} catch (const std::bad_alloc &) {
    set_error("steps_sim_create: out of host memory");
    return STEPS_ERR_OOM;
}

int steps_sim_clone(const steps_sim *src, uint64_t seed, void *cuda_stream, steps_sim **out) try {
    CHECK_NULL(out, "steps_sim_clone");
    *out = nullptr;
    CHECK_NULL(src, "steps_sim_clone");
    std::unique_ptr<steps_sim> s;
    try {
        s.reset(new steps_sim(src->tables));
        s->model = src->model;
        s->h_rmask = src->h_rmask;
    } catch (const std::bad_alloc &) {
        set_error("steps_sim_clone: out of host memory");
        return STEPS_ERR_OOM;
    }
    s->opt = src->opt;
    s->stream = (cudaStream_t)cuda_stream;
    s->device = src->device;
    s->T = src->T;
    s->Tpad = src->Tpad;
    s->S = src->S;
    s->seed = seed;
    s->spec = src->spec;
    s->spec_list = src->spec_list;
    s->forced = src->forced;
    s->spec_why = src->spec_why;
    std::memcpy(s->scale_full, src->scale_full, sizeof(s->scale_full));
    const size_t Tpad = (size_t)s->Tpad, S = (size_t)s->S, T = (size_t)s->T;
    std::vector<steps_sim::Request> want;
    auto alloc = [&](void **p, size_t bytes) { want.emplace_back(p, bytes); };
    alloc((void **)&s->d_cnt[0], S * Tpad * 4);
    alloc((void **)&s->d_cnt[1], S * Tpad * 4);
    alloc((void **)&s->d_nbr, Tpad * 16);
    alloc((void **)&s->d_thr, Tpad * 16);
    alloc((void **)&s->d_inv_nav, Tpad * 4);
    alloc((void **)&s->d_err, 24);
    alloc((void **)&s->d_window_base, 8);
    alloc((void **)&s->d_stage, S * T * 4);
    if (src->d_orig) {
        alloc((void **)&s->d_orig, Tpad * 4);
        alloc((void **)&s->d_inv_perm, T * 4);
    }
    if (src->d_rmask) alloc((void **)&s->d_rmask, Tpad * 4);
    if (src->d_leave[0]) {
        alloc((void **)&s->d_leave[0], S * Tpad * 4);
        alloc((void **)&s->d_leave[1], S * Tpad * 4);
        alloc((void **)&s->d_G, Tpad * 8);
        alloc((void **)&s->d_leave_list, kLeaveListBytes);
    }
    const size_t base = want.size();
    if (src->d_tm[0])
        for (const steps_sim::Request &r : s->list_requests()) want.push_back(r);
    cudaError_t e = s->alloc_arena(want);
    if (e != cudaSuccess && want.size() > base) {  // no room for the list form: the clone runs its tiles
        want.resize(base);
        s->spec_list = nullptr;
        e = s->alloc_arena(want);
    }
    if (e != cudaSuccess) {
        set_error(std::string("steps_sim_clone: device allocation failed: ") + cudaGetErrorString(e));
        cudaGetLastError();
        return STEPS_ERR_OOM;
    }
    cudaStream_t st = s->stream;
    bool ok = cuda_ok(cudaMemcpyAsync(s->d_nbr, src->d_nbr, Tpad * 16, cudaMemcpyDeviceToDevice, st), "clone") &&
              cuda_ok(cudaMemcpyAsync(s->d_thr, src->d_thr, Tpad * 16, cudaMemcpyDeviceToDevice, st), "clone") &&
              cuda_ok(cudaMemcpyAsync(s->d_inv_nav, src->d_inv_nav, Tpad * 4, cudaMemcpyDeviceToDevice, st), "clone") &&
              cuda_ok(cudaMemsetAsync(s->d_cnt[0], 0, S * Tpad * 4, st), "clone") &&
              cuda_ok(cudaMemsetAsync(s->d_cnt[1], 0, S * Tpad * 4, st), "clone") &&
              cuda_ok(cudaMemsetAsync(s->d_err, 0, 24, st), "clone") &&
              cuda_ok(cudaMemsetAsync(s->d_window_base, 0, 8, st), "clone");
    if (ok && src->d_orig)
        ok = cuda_ok(cudaMemcpyAsync(s->d_orig, src->d_orig, Tpad * 4, cudaMemcpyDeviceToDevice, st), "clone") &&
             cuda_ok(cudaMemcpyAsync(s->d_inv_perm, src->d_inv_perm, T * 4, cudaMemcpyDeviceToDevice, st), "clone");
    if (ok && src->d_rmask)
        ok = cuda_ok(cudaMemcpyAsync(s->d_rmask, src->d_rmask, Tpad * 4, cudaMemcpyDeviceToDevice, st), "clone");
    if (ok && src->d_leave[0])
        ok = cuda_ok(cudaMemcpyAsync(s->d_leave[0], src->d_leave[0], S * Tpad * 4, cudaMemcpyDeviceToDevice, st),
                     "clone") &&
             cuda_ok(cudaMemsetAsync(s->d_leave[1], 0, S * Tpad * 4, st), "clone") &&
             cuda_ok(cudaMemcpyAsync(s->d_G, src->d_G, T * 8, cudaMemcpyDeviceToDevice, st), "clone");
    if (!ok || !cuda_ok(cudaStreamSynchronize(st), "steps_sim_clone")) return STEPS_ERR_CUDA;
    *out = s.release();
    return STEPS_OK;
} catch (const std::bad_alloc &) {
    set_error("steps_sim_clone: out of host memory");
    return STEPS_ERR_OOM;
}

int steps_sim_device_bytes(const steps_sim *sim, int64_t *bytes) {
    CHECK_NULL(sim, "steps_sim_device_bytes");
    CHECK_NULL(bytes, "steps_sim_device_bytes");
    const int64_t Tpad = sim->Tpad, S = sim->S, T = sim->T;
    *bytes = 2 * S * Tpad * 4 + Tpad * 16 * 2 + Tpad * 4 + 16 + S * T * 4 + (sim->d_orig ? Tpad * 4 + T * 4 : 0) +
             (sim->d_trial ? S * Tpad * 4 : 0) + (sim->d_tm[0] ? 10 * Tpad * 4 + 16 : 0) +
             (sim->d_src ? Tpad * 4 + Tpad / 8 : 0) + (sim->d_leave[0] ? 2 * S * Tpad * 4 + Tpad * 8 + (int64_t)kLeaveListBytes : 0) +
             (sim->d_rmask ? Tpad * 4 : 0) + (int64_t)(sim->flow[0].bytes + sim->flow[1].bytes + sim->flow[2].bytes +
                       sim->flow[3].bytes);
    return STEPS_OK;
}

void steps_sim_destroy(steps_sim *sim) {
    if (!sim) return;
    if (sim->stream) cudaStreamSynchronize(sim->stream);
    else cudaDeviceSynchronize();
    delete sim;
}

static int put_counts(steps_sim *sim, int32_t s0, int32_t ns, const int32_t *counts) {
    const size_t T = (size_t)sim->T, Tpad = (size_t)sim->Tpad;
    if (!cuda_ok(cudaMemcpyAsync(sim->d_stage, counts, (size_t)ns * T * 4, cudaMemcpyHostToDevice, sim->stream),
                 "steps_set_counts: copy"))
        return STEPS_ERR_CUDA;
    // reject negative counts on the device, before anything of the state changes
    uint32_t seen[4] = {0, 0, 0, 0};  // a negative count; non-zero ones; their sum
    const int64_t n = (int64_t)ns * (int64_t)T;
    if (!cuda_ok(cudaMemsetAsync(sim->d_err + 2, 0, 16, sim->stream), "steps_set_counts: check"))
        return STEPS_ERR_CUDA;
    any_negative<true><<<input_blocks(n), kInputThreads, 0, sim->stream>>>(sim->d_stage, n, sim->d_err + 2);
    if (!cuda_ok(cudaGetLastError(), "steps_set_counts: check") ||
        !cuda_ok(cudaMemcpyAsync(seen, sim->d_err + 2, 16, cudaMemcpyDeviceToHost, sim->stream), "steps_set_counts: check") ||
        !cuda_ok(cudaStreamSynchronize(sim->stream), "steps_set_counts: check"))
        return STEPS_ERR_CUDA;
    if (seen[0]) {
        set_error("steps_set_counts: negative count");
        return STEPS_ERR_ARG;
    }
    sim->tm_valid = sim->list_valid = false;
    if (ns == sim->S) sim->found(seen);
    else sim->fill = sim->density = -1.0;
    scatter_to_device_order<<<(unsigned)((T + 255) / 256), 256, 0, sim->stream>>>(
        sim->d_stage, (int64_t)T, ns, sim->d_inv_perm, sim->d_cnt[sim->cur] + (size_t)s0 * Tpad, Tpad);
    if (!cuda_ok(cudaGetLastError(), "steps_set_counts: scatter")) return STEPS_ERR_CUDA;
    // the receiving buffer must start at zero (the step kernel writes only non-zero counts)
    if (!cuda_ok(cudaMemsetAsync(sim->d_cnt[1 - sim->cur] + (size_t)s0 * Tpad, 0, (size_t)ns * Tpad * 4,
                                 sim->stream),
                 "steps_set_counts: memset"))
        return STEPS_ERR_CUDA;
    if (!cuda_ok(cudaStreamSynchronize(sim->stream), "steps_set_counts")) return STEPS_ERR_CUDA;
    return STEPS_OK;
}


int steps_set_counts(steps_sim *sim, int32_t species, const int32_t *counts) {
    CHECK_NULL(sim, "steps_set_counts");
    CHECK_NULL(counts, "steps_set_counts");
    if (species < 0 || species >= sim->S) {
        set_error("steps_set_counts: species out of range");
        return STEPS_ERR_ARG;
    }
    return put_counts(sim, species, 1, counts);
}

int steps_set_counts_all(steps_sim *sim, const int32_t *counts) {
    CHECK_NULL(sim, "steps_set_counts_all");
    CHECK_NULL(counts, "steps_set_counts_all");
    return put_counts(sim, 0, sim->S, counts);
}

static int fetch_counts(const steps_sim *sim, int32_t s0, int32_t ns, int32_t *out) {
    const size_t T = (size_t)sim->T, Tpad = (size_t)sim->Tpad;
    gather_to_original_order<<<(unsigned)((T + 255) / 256), 256, 0, sim->stream>>>(
        sim->d_cnt[sim->cur] + (size_t)s0 * Tpad, (int64_t)T, ns, sim->d_inv_perm, Tpad, sim->d_stage);
    if (!cuda_ok(cudaGetLastError(), "steps_get_counts: gather")) return STEPS_ERR_CUDA;
    if (!cuda_ok(cudaMemcpyAsync(out, sim->d_stage, (size_t)ns * T * 4, cudaMemcpyDeviceToHost, sim->stream),
                 "steps_get_counts: copy"))
        return STEPS_ERR_CUDA;
    if (!cuda_ok(cudaStreamSynchronize(sim->stream), "steps_get_counts")) return STEPS_ERR_CUDA;
    return STEPS_OK;
}

int steps_get_counts(const steps_sim *sim, int32_t species, int32_t *out) {
    CHECK_NULL(sim, "steps_get_counts");
    CHECK_NULL(out, "steps_get_counts");
    if (species < 0 || species >= sim->S) {
        set_error("steps_get_counts: species out of range");
        return STEPS_ERR_ARG;
    }
    return fetch_counts(sim, species, 1, out);
}

int steps_get_counts_all(const steps_sim *sim, int32_t *out) {
    CHECK_NULL(sim, "steps_get_counts_all");
    CHECK_NULL(out, "steps_get_counts_all");
    return fetch_counts(sim, 0, sim->S, out);
}

int steps_set_reac_mask(steps_sim *sim, int32_t reac, const uint8_t *active) {
    CHECK_NULL(sim, "steps_set_reac_mask");
    if (reac < 0 || reac >= sim->model.R) {
        set_error("steps_set_reac_mask: reaction out of range");
        return STEPS_ERR_ARG;
    }
    const size_t T = (size_t)sim->T;
    if (sim->h_rmask.empty()) sim->h_rmask.assign(T, 0xFFFFFFFFu);
    const uint32_t bit = 1u << reac;
    for (size_t d = 0; d < T; ++d) {
        const bool on = !active || active[sim->tab.perm[d]] != 0;
        sim->h_rmask[d] = on ? (sim->h_rmask[d] | bit) : (sim->h_rmask[d] & ~bit);
    }
    if (!sim->d_rmask) {
        if (!cuda_ok(device_alloc((void **)&sim->d_rmask, (size_t)sim->Tpad * 4), "steps_set_reac_mask: alloc"))
            return STEPS_ERR_OOM;
        sim->drop_graphs();  // kernel arguments change
        if (!cuda_ok(cudaMemsetAsync(sim->d_rmask, 0, (size_t)sim->Tpad * 4, sim->stream), "steps_set_reac_mask: memset"))
            return STEPS_ERR_CUDA;
    }
    sim->src_valid = sim->list_valid = false;
    if (!cuda_ok(cudaMemcpyAsync(sim->d_rmask, sim->h_rmask.data(), T * 4, cudaMemcpyHostToDevice, sim->stream),
                 "steps_set_reac_mask: copy") ||
        !cuda_ok(cudaStreamSynchronize(sim->stream), "steps_set_reac_mask"))
        return STEPS_ERR_CUDA;
    return STEPS_OK;
}

}  // extern "C"

namespace {

// A simulation whose bounded wait ran out stays closed: the block that gave up
// may have left a bulk copy in flight, so its results cannot be trusted.
int refuse_failed(const steps_sim *sim, const char *who) {
    if (!sim->failed) return STEPS_OK;
    set_error(std::string(who) + ": an earlier run of this simulation timed out on the device; "
                                 "destroy it and create a new one");
    return STEPS_ERR_STATE;
}

// Enqueues the windows of Algorithm 1 from the simulation's time to t_end
// (full windows of tau, then a shortened last window). Waits for the stream
// only where the host has to see something first: the tuning of the launch
// form, a list's length (choose_form), a leave table of many entries.
int enqueue_run(steps_sim *sim, double t_end) {
    if (int rf = sim->choose_form()) return rf;
    if (sim->leave_waits()) {  // the shortened window's leave table first
        int64_t full;
        double partial;
        sim->schedule(t_end, &full, &partial);
        if (partial > 0.0 && partial != sim->tab.tau)
            if (int rl = sim->upload_leave(partial, sim->stream)) return rl;
    }
    const double tau = sim->tab.tau;
    const bool finite = std::isfinite(tau);
    const double tol = finite ? 1e-9 * tau : 0.0;
    for (;;) {
        const double t = sim->time();
        if (!(t_end - t > tol)) break;
        if (finite && t + tau <= t_end + tol) {
            // the consecutive full windows the loop of Algorithm 1 takes from here
            int64_t n = 0;
            while (n < kWindowBatch) {
                const int64_t k = sim->k_grid + n;
                const double tt = k == 0 ? sim->t_base : sim->t_base + (double)k * tau;
                if (!(t_end - tt > tol) || !(tt + tau <= t_end + tol)) break;
                ++n;
            }
            int rc = sim->full_windows(n);
            if (rc) return rc;
            sim->k_grid += n;
        } else {
            int rc = sim->window_launch(t_end - t);  // shortened last window (Algorithm 1)
            if (rc) return rc;
            sim->t_base = t_end;
            sim->k_grid = 0;
            break;
        }
    }
    return STEPS_OK;
}

// The return code of a device error word, with its message. *closed: a wait
// ran out, the counts are not valid and the simulations of the launch are
// closed to further runs.
int error_word(uint32_t err, const char *who, bool *closed) {
    *closed = (err & 12u) != 0u;
    if (err == 0) return STEPS_OK;
    set_error(std::string(who) +
              (err & 4u ? ": a bulk copy into shared memory did not complete within its wait limit; a copy may still "
                          "be in flight, so what the launch ran is closed to further runs"
               : err & 8u ? ": a tile of a flow launch waited beyond its limit for the tiles it depends on; the counts "
                            "are not valid, so what the launch ran is closed to further runs"
               : err & 2u ? ": a tet fired more than 2^24 reactions in one window (rates too large)"
                          : ": a negative count was seen on the device"));
    return *closed ? STEPS_ERR_TIMEOUT : STEPS_ERR_STATE;
}

// Waits for the simulation's stream and turns the device error word into a
// return code (and clears it).
int finish_run(steps_sim *sim, const char *who) {
    uint32_t err = 0, c[4];
    if (!cuda_ok(cudaMemcpyAsync(&err, sim->d_err, 4, cudaMemcpyDeviceToHost, sim->stream), "error word") ||
        (sim->listing && !cuda_ok(cudaMemcpyAsync(c, sim->d_lcnt, 16, cudaMemcpyDeviceToHost, sim->stream), who)) ||
        !cuda_ok(cudaStreamSynchronize(sim->stream), who))
        return STEPS_ERR_CUDA;
    if (sim->listing) sim->fill_from(c);
    if (err) cudaMemsetAsync(sim->d_err, 0, 4, sim->stream);
    bool closed = false;
    const int rc = error_word(err, who, &closed);
    if (closed) sim->failed = true;
    return rc;
}

// One recording: counts of the chosen species (rows of cur) at the chosen
// tets (device indices) into out[species][tet].
__global__ void gather_record(const int32_t *cur, size_t Tpad, const int32_t *species, int32_t ns,
                              const int32_t *tets, int32_t nr, int32_t *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)ns * nr) return;
    const int32_t q = (int32_t)(i / nr), j = (int32_t)(i % nr);
    out[i] = cur[(size_t)species[q] * Tpad + tets[j]];
}

}  // namespace

extern "C" {

int steps_run(steps_sim *sim, double t_end) {
    CHECK_NULL(sim, "steps_run");
    if (!std::isfinite(t_end)) {
        set_error("steps_run: t_end must be finite");
        return STEPS_ERR_ARG;
    }
    if (int rf = refuse_failed(sim, "steps_run")) return rf;
    int rc = enqueue_run(sim, t_end);
    return rc ? rc : finish_run(sim, "steps_run");
}

int steps_set_reac_rate(steps_sim *sim, int32_t reac, double k) {
    CHECK_NULL(sim, "steps_set_reac_rate");
    if (reac < 0 || reac >= sim->model.R) {
        set_error("steps_set_reac_rate: reaction out of range");
        return STEPS_ERR_ARG;
    }
    if (!(k >= 0.0) || !std::isfinite(k)) {
        set_error("steps_set_reac_rate: rate constant must be finite and >= 0");
        return STEPS_ERR_ARG;
    }
    sim->model.k[(size_t)reac] = k;
    sim->model.dev.reac[reac].k = (float)k;
    sim->drop_graphs();  // the captured launches hold the old model
    return STEPS_OK;
}

int steps_run_record(steps_sim *sim, double t_end, double dt_rec, int32_t n_species, const int32_t *species,
                     int32_t n_tets, const int32_t *tets, int32_t *d_out, int64_t max_records, int64_t *n_records) {
    CHECK_NULL(sim, "steps_run_record");
    CHECK_NULL(species, "steps_run_record");
    CHECK_NULL(tets, "steps_run_record");
    CHECK_NULL(d_out, "steps_run_record");
    if (n_records) *n_records = 0;
    if (!std::isfinite(t_end) || !(dt_rec > 0.0) || !std::isfinite(dt_rec)) {
        set_error("steps_run_record: t_end must be finite and dt_rec finite and > 0");
        return STEPS_ERR_ARG;
    }
    if (int rf = refuse_failed(sim, "steps_run_record")) return rf;
    if (n_species < 1 || n_species > sim->S || n_tets < 1 || max_records < 0) {
        set_error("steps_run_record: bad species or tet count");
        return STEPS_ERR_ARG;
    }
    for (int32_t q = 0; q < n_species; ++q)
        if (species[q] < 0 || species[q] >= sim->S) {
            set_error("steps_run_record: species out of range");
            return STEPS_ERR_ARG;
        }
    std::vector<int32_t> dev_tets((size_t)n_tets);
    for (int32_t j = 0; j < n_tets; ++j) {
        if (tets[j] < 0 || tets[j] >= sim->T) {
            set_error("steps_run_record: tet out of range");
            return STEPS_ERR_ARG;
        }
        dev_tets[(size_t)j] = sim->tab.inv_perm.empty() ? tets[j] : sim->tab.inv_perm[(size_t)tets[j]];
    }
    // recording times t0 + k dt_rec, k = 1, 2, ... up to t_end (recomputed, not accumulated)
    const double t0 = sim->time();
    const double tol = 1e-12 * std::max(std::fabs(t_end), dt_rec);
    int64_t nrec = 0;
    while (t0 + (double)(nrec + 1) * dt_rec <= t_end + tol) ++nrec;
    if (nrec > max_records) {
        set_error("steps_run_record: " + std::to_string(nrec) + " recordings do not fit max_records = " +
                  std::to_string(max_records));
        return STEPS_ERR_ARG;
    }
    // the selection, uploaded once
    const size_t need = ((size_t)n_species + (size_t)n_tets) * 4;
    if (sim->rec_bytes < need) {
        cudaFree(sim->d_rec);
        sim->d_rec = nullptr;
        sim->rec_bytes = 0;
        if (!cuda_ok(device_alloc((void **)&sim->d_rec, need), "steps_run_record: alloc")) return STEPS_ERR_OOM;
        sim->rec_bytes = need;
    }
    int32_t *d_species = sim->d_rec, *d_tets = sim->d_rec + n_species;
    if (!cuda_ok(cudaMemcpyAsync(d_species, species, (size_t)n_species * 4, cudaMemcpyHostToDevice, sim->stream),
                 "steps_run_record: upload") ||
        !cuda_ok(cudaMemcpyAsync(d_tets, dev_tets.data(), (size_t)n_tets * 4, cudaMemcpyHostToDevice, sim->stream),
                 "steps_run_record: upload"))
        return STEPS_ERR_CUDA;
    const int64_t per = (int64_t)n_species * n_tets;
    const unsigned grid = (unsigned)((per + 255) / 256);
    for (int64_t k = 1; k <= nrec; ++k) {
        int rc = enqueue_run(sim, t0 + (double)k * dt_rec);
        if (rc) return rc;
        gather_record<<<grid, 256, 0, sim->stream>>>(sim->d_cnt[sim->cur], (size_t)sim->Tpad, d_species, n_species,
                                                     d_tets, n_tets, d_out + (k - 1) * per);
        if (!cuda_ok(cudaGetLastError(), "steps_run_record: gather")) return STEPS_ERR_CUDA;
        ++sim->launches;
    }
    int rc = enqueue_run(sim, t_end);
    if (!rc) rc = finish_run(sim, "steps_run_record");
    // the host copy of dev_tets must outlive the async upload: finish_run synchronised
    if (n_records) *n_records = rc ? 0 : nrec;
    return rc;
}

int steps_sim_flow(const steps_sim *sim, int32_t *flow_block, float *tune_ms) {
    CHECK_NULL(sim, "steps_sim_flow");
    CHECK_NULL(flow_block, "steps_sim_flow");
    const int k = sim->flow_form();
    *flow_block = k < 0 ? 0 : k == 0 ? sim->opt.block : k == 2 ? 256 : 512;
    if (tune_ms)
        for (int c = 0; c < 3; ++c) tune_ms[c] = sim->flow_ms[c];
    return STEPS_OK;
}

int steps_sim_specialized(const steps_sim *sim, int32_t *specialized) {
    CHECK_NULL(sim, "steps_sim_specialized");
    CHECK_NULL(specialized, "steps_sim_specialized");
    *specialized = sim->spec ? 1 : 0;
    return STEPS_OK;
}

int steps_get_time(const steps_sim *sim, double *t) {
    CHECK_NULL(sim, "steps_get_time");
    CHECK_NULL(t, "steps_get_time");
    *t = sim->time();
    return STEPS_OK;
}

int steps_get_tau(const steps_sim *sim, double *tau) {
    CHECK_NULL(sim, "steps_get_tau");
    CHECK_NULL(tau, "steps_get_tau");
    *tau = sim->tab.tau;
    return STEPS_OK;
}

int steps_sim_shape(const steps_sim *sim, int64_t *nt, int32_t *n_species) {
    CHECK_NULL(sim, "steps_sim_shape");
    if (nt) *nt = sim->T;
    if (n_species) *n_species = sim->S;
    return STEPS_OK;
}

int steps_get_windows(const steps_sim *sim, uint64_t *windows, uint64_t *launches) {
    CHECK_NULL(sim, "steps_get_windows");
    if (windows) *windows = sim->k_total;
    if (launches) *launches = sim->launches;
    return STEPS_OK;
}

int steps_debug_philox(uint64_t seed, const uint32_t *ctr, int64_t n, uint32_t *out) {
    CHECK_NULL(ctr, "steps_debug_philox");
    CHECK_NULL(out, "steps_debug_philox");
    if (n < 0) return STEPS_ERR_ARG;
    if (n == 0) return STEPS_OK;
    uint32_t *dc = nullptr, *dout = nullptr;
    int rc = STEPS_OK;
    if (!cuda_ok(cudaMalloc((void **)&dc, (size_t)n * 16), "alloc") ||
        !cuda_ok(cudaMalloc((void **)&dout, (size_t)n * 16), "alloc"))
        rc = STEPS_ERR_OOM;
    if (!rc && !cuda_ok(cudaMemcpy(dc, ctr, (size_t)n * 16, cudaMemcpyHostToDevice), "copy")) rc = STEPS_ERR_CUDA;
    if (!rc) rc = launch_philox_test(seed, dc, n, dout, nullptr);
    if (!rc && !cuda_ok(cudaMemcpy(out, dout, (size_t)n * 16, cudaMemcpyDeviceToHost), "copy")) rc = STEPS_ERR_CUDA;
    cudaFree(dc);
    cudaFree(dout);
    return rc;
}

int steps_debug_host_tables(const steps_mesh *mesh, const steps_model *model, int32_t reorder, double *tau,
                            uint32_t *thr, int32_t *perm) {
    CHECK_NULL(mesh, "steps_debug_host_tables");
    CHECK_NULL(model, "steps_debug_host_tables");
    CHECK_NULL(tau, "steps_debug_host_tables");
    CHECK_NULL(thr, "steps_debug_host_tables");
    if (reorder != STEPS_REORDER_NONE && reorder != STEPS_REORDER_MORTON && reorder != STEPS_REORDER_RCM) {
        set_error("steps_debug_host_tables: bad reorder");
        return STEPS_ERR_ARG;
    }
    Tables t;
    try {
        build_tables(mesh->m, model->m, reorder, t);
    } catch (const std::bad_alloc &) {
        set_error("steps_debug_host_tables: out of host memory");
        return STEPS_ERR_OOM;
    }
    *tau = t.tau;
    const size_t nt = t.perm.size();
    for (size_t d = 0; d < nt; ++d)
        for (int f = 0; f < 4; ++f) thr[(size_t)t.perm[d] * 4 + f] = t.thr_dev[d * 4 + f];
    if (perm) std::memcpy(perm, t.perm.data(), nt * sizeof(int32_t));
    return STEPS_OK;
}

int steps_debug_leave_table(steps_sim *sim, double tau_k, uint32_t *out, uint32_t *decided) {
    CHECK_NULL(sim, "steps_debug_leave_table");
    CHECK_NULL(out, "steps_debug_leave_table");
    if (!sim->d_leave[0] || !(tau_k > 0.0) || !std::isfinite(tau_k)) {
        set_error("steps_debug_leave_table: needs the EXP leave law and a finite window > 0");
        return STEPS_ERR_ARG;
    }
    int rc = sim->device_leave(tau_k, sim->stream, decided);
    if (rc) return rc;
    const uint32_t *d = tau_k == sim->tab.tau ? sim->d_leave[0] : sim->d_leave[1];
    gather_to_original_order<<<(unsigned)((sim->T + 255) / 256), 256, 0, sim->stream>>>(
        (const int32_t *)d, sim->T, sim->S, sim->d_inv_perm, (size_t)sim->Tpad, sim->d_stage);
    if (!cuda_ok(cudaGetLastError(), "steps_debug_leave_table") ||
        !cuda_ok(cudaMemcpyAsync(out, sim->d_stage, (size_t)sim->S * sim->T * 4, cudaMemcpyDeviceToHost, sim->stream),
                 "steps_debug_leave_table") ||
        !cuda_ok(cudaStreamSynchronize(sim->stream), "steps_debug_leave_table"))
        return STEPS_ERR_CUDA;
    return STEPS_OK;
}

int steps_debug_fail_alloc(int32_t nth, int64_t *made) {
    if (nth < 0) {
        set_error("steps_debug_fail_alloc: nth must be >= 0");
        return STEPS_ERR_ARG;
    }
    t_fail_alloc = nth;
    if (made) *made = t_allocs;
    return STEPS_OK;
}

int steps_debug_form(int32_t form) {
    if (form != 0 && form != 2 && form != 3) {
        set_error("steps_debug_form: form must be 0, 2 or 3");
        return STEPS_ERR_ARG;
    }
    t_form = form;
    return STEPS_OK;
}

int steps_debug_error_word(uint32_t word, int32_t *closed) {
    bool c = false;
    const int rc = error_word(word, "steps_debug_error_word", &c);
    if (closed) *closed = c ? 1 : 0;
    return rc;
}

int steps_debug_wait(int32_t deliver, int64_t limit_cycles) {
    if (limit_cycles < 1 || limit_cycles > (int64_t)1 << 31) {
        set_error("steps_debug_wait: limit_cycles must be in [1, 2^31]");
        return STEPS_ERR_ARG;
    }
    void *src = nullptr;
    uint32_t *status = nullptr;
    int rc = STEPS_OK;
    if (!cuda_ok(cudaMalloc(&src, 16), "steps_debug_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&status, 4), "steps_debug_wait: alloc"))
        rc = STEPS_ERR_OOM;
    uint32_t st = 0;
    if (!rc && (!cuda_ok(cudaMemset(src, 0, 16), "steps_debug_wait") ||
                !cuda_ok(cudaMemset(status, 0xFF, 4), "steps_debug_wait")))
        rc = STEPS_ERR_CUDA;
    if (!rc) rc = launch_wait_test(src, deliver != 0, (long long)limit_cycles, status, nullptr);
    if (!rc && !cuda_ok(cudaMemcpy(&st, status, 4, cudaMemcpyDeviceToHost), "steps_debug_wait")) rc = STEPS_ERR_CUDA;
    cudaFree(src);
    cudaFree(status);
    if (rc) return rc;
    if (st == 4u) {
        set_error("steps_debug_wait: the bulk-copy wait did not complete within its limit");
        return STEPS_ERR_TIMEOUT;
    }
    if (st != 0u) {
        set_error("steps_debug_wait: unexpected status");
        return STEPS_ERR_STATE;
    }
    return STEPS_OK;
}

int steps_debug_flow_wait(int32_t deliver, int64_t limit_cycles) {
    if (limit_cycles < 1 || limit_cycles > (int64_t)1 << 31) {
        set_error("steps_debug_flow_wait: limit_cycles must be in [1, 2^31]");
        return STEPS_ERR_ARG;
    }
    // tile 0 lists 40 neighbour tiles (two rounds of the warp); all of them
    // have finished window 4 (word 5) when delivered, else the last has not
    constexpr int n = 40;
    int32_t h_off[2] = {0, n}, h_nb[n];
    uint32_t h_done[n];
    for (int j = 0; j < n; ++j) {
        h_nb[j] = j;
        h_done[j] = 5u + (uint32_t)(j % 3);
    }
    if (!deliver) h_done[n - 1] = 4u;
    int32_t *d_off = nullptr, *d_nb = nullptr;
    uint32_t *d_done = nullptr, *status = nullptr;
    int rc = STEPS_OK;
    if (!cuda_ok(cudaMalloc((void **)&d_off, sizeof(h_off)), "steps_debug_flow_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&d_nb, sizeof(h_nb)), "steps_debug_flow_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&d_done, sizeof(h_done)), "steps_debug_flow_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&status, 4), "steps_debug_flow_wait: alloc"))
        rc = STEPS_ERR_OOM;
    uint32_t st = 0;
    if (!rc && (!cuda_ok(cudaMemcpy(d_off, h_off, sizeof(h_off), cudaMemcpyHostToDevice), "steps_debug_flow_wait") ||
                !cuda_ok(cudaMemcpy(d_nb, h_nb, sizeof(h_nb), cudaMemcpyHostToDevice), "steps_debug_flow_wait") ||
                !cuda_ok(cudaMemcpy(d_done, h_done, sizeof(h_done), cudaMemcpyHostToDevice), "steps_debug_flow_wait") ||
                !cuda_ok(cudaMemset(status, 0xFF, 4), "steps_debug_flow_wait")))
        rc = STEPS_ERR_CUDA;
    if (!rc) rc = launch_flow_wait_test(d_off, d_nb, d_done, (long long)limit_cycles, status);
    if (!rc && !cuda_ok(cudaMemcpy(&st, status, 4, cudaMemcpyDeviceToHost), "steps_debug_flow_wait"))
        rc = STEPS_ERR_CUDA;
    cudaFree(d_off);
    cudaFree(d_nb);
    cudaFree(d_done);
    cudaFree(status);
    if (rc) return rc;
    if (st == 8u) {
        set_error("steps_debug_flow_wait: the dependency wait did not complete within its limit");
        return STEPS_ERR_TIMEOUT;
    }
    if (st != 0u) {
        set_error("steps_debug_flow_wait: unexpected status");
        return STEPS_ERR_STATE;
    }
    return STEPS_OK;
}

int steps_debug_flow_nbr_wait(int32_t late, int64_t limit_cycles) {
    constexpr int n = 40;  // warp tiles of 32 tets
    if (limit_cycles < 1 || limit_cycles > (int64_t)1 << 31 || late < -1 || late >= n) {
        set_error("steps_debug_flow_nbr_wait: limit_cycles must be in [1, 2^31], late in [-1, 39]");
        return STEPS_ERR_ARG;
    }
    // of the 128 faces of tile 1's tets, three reach each tile and eight are boundary faces
    int32_t h_nbr[128];
    for (int k = 0; k < 128; ++k) h_nbr[k] = k < 3 * n ? 32 * (k % n) + k / 4 : -1;
    uint32_t h_done[n];
    for (int j = 0; j < n; ++j) h_done[j] = j == late ? 4u : 5u + (uint32_t)(j % 3);
    void *d_nbr = nullptr;
    uint32_t *d_done = nullptr, *status = nullptr;
    int rc = STEPS_OK;
    if (!cuda_ok(cudaMalloc(&d_nbr, sizeof(h_nbr)), "steps_debug_flow_nbr_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&d_done, sizeof(h_done)), "steps_debug_flow_nbr_wait: alloc") ||
        !cuda_ok(cudaMalloc((void **)&status, 4), "steps_debug_flow_nbr_wait: alloc"))
        rc = STEPS_ERR_OOM;
    uint32_t st = 0;
    if (!rc && (!cuda_ok(cudaMemcpy(d_nbr, h_nbr, sizeof(h_nbr), cudaMemcpyHostToDevice), "steps_debug_flow_nbr_wait") ||
                !cuda_ok(cudaMemcpy(d_done, h_done, sizeof(h_done), cudaMemcpyHostToDevice), "steps_debug_flow_nbr_wait") ||
                !cuda_ok(cudaMemset(status, 0xFF, 4), "steps_debug_flow_nbr_wait")))
        rc = STEPS_ERR_CUDA;
    if (!rc) rc = launch_nbr_wait_test(d_done, d_nbr, (long long)limit_cycles, status);
    if (!rc && !cuda_ok(cudaMemcpy(&st, status, 4, cudaMemcpyDeviceToHost), "steps_debug_flow_nbr_wait"))
        rc = STEPS_ERR_CUDA;
    cudaFree(d_nbr);
    cudaFree(d_done);
    cudaFree(status);
    if (rc) return rc;
    if (st == 0u) return STEPS_OK;
    set_error(st == 8u ? "steps_debug_flow_nbr_wait: the neighbour wait did not complete within its limit"
                       : "steps_debug_flow_nbr_wait: unexpected status");
    return st == 8u ? STEPS_ERR_TIMEOUT : STEPS_ERR_STATE;
}

int steps_debug_logf(const float *x, int64_t n, float *out) {
    CHECK_NULL(x, "steps_debug_logf");
    CHECK_NULL(out, "steps_debug_logf");
    if (n < 0) return STEPS_ERR_ARG;
    if (n == 0) return STEPS_OK;
    float *dx = nullptr, *dout = nullptr;
    int rc = STEPS_OK;
    if (!cuda_ok(cudaMalloc((void **)&dx, (size_t)n * 4), "alloc") ||
        !cuda_ok(cudaMalloc((void **)&dout, (size_t)n * 4), "alloc"))
        rc = STEPS_ERR_OOM;
    if (!rc && !cuda_ok(cudaMemcpy(dx, x, (size_t)n * 4, cudaMemcpyHostToDevice), "copy")) rc = STEPS_ERR_CUDA;
    if (!rc) rc = launch_logf_test(dx, n, dout, nullptr);
    if (!rc && !cuda_ok(cudaMemcpy(out, dout, (size_t)n * 4, cudaMemcpyDeviceToHost), "copy")) rc = STEPS_ERR_CUDA;
    cudaFree(dx);
    cudaFree(dout);
    return rc;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched form: one launch per window over many simulations.
// ---------------------------------------------------------------------------
struct steps_batch {
    std::vector<steps_sim *> members;
    cudaStream_t stream = nullptr;
    int block = 256;
    bool autotune = false;
    bool use_graph = true;
    int max_S = 1, max_R = 0;
    bool any_order0 = false;
    RepEntry *h_reps = nullptr;  // pinned host mirror (full windows)
    RepEntry *h_last = nullptr;  // pinned host table of the shortened last windows: a second buffer, so
                                 // that filling it cannot change h_reps while its upload is still queued
    RepEntry *d_reps = nullptr;
    uint32_t *d_err = nullptr;
    uint32_t *h_err = nullptr;   // pinned copy of the error word, read after the stream completes
    struct Work {
        BlockWork *d = nullptr;
        int64_t n = 0;
        bool built = false;
        cudaGraphExec_t graph = nullptr;
    };
    Work work[4];  // block sizes 64, 128, 256, 512
    // members whose windows go through the list form in this run (their blocks
    // are not in `work`), its kernel and their blocks
    std::vector<char> listed;
    void *spec_list = nullptr;
    Work lwork;
    uint32_t *h_lcnt = nullptr;  // pinned: their list lengths after the run
    void *spec_block = nullptr;  // block tiles for the others (256-thread blocks)
    bool blocky = false;         // in this run
    bool few = false;            // run-time models of 5 to 12 species in sparse states: block tiles, in this run
    uint64_t launches = 0;
    bool use_spec = false;      // run the model-specialised batched kernel
    bool spec_forced = false;
    void *spec[4] = {};         // per block size, compiled on first use (before any capture)
    std::string spec_why;
    std::vector<float> tune_ms;  // autotune timings per candidate block (ms per window)
    bool flow = false;           // full windows of member groups as flow launches (specialised kernel)
    // flow launches, per block size: the finished-window words of every work
    // entry's warp tiles followed by the item counter, and the groups:
    // consecutive members whose tables fit in about half of L2 (at least one
    // member each), so that a group's windows run from L2
    struct Flow {
        uint32_t *d_flow = nullptr;
        std::vector<std::pair<int64_t, int64_t>> groups;  // (first work entry, entries)
        int64_t nwords = 0;
    } fl[4];
    uint64_t flow_launches = 0;

    static int slot(int b) { return b == 64 ? 0 : b == 128 ? 1 : b == 512 ? 3 : 2; }

    ~steps_batch() {
        for (auto &w : work) {
            if (w.graph) cudaGraphExecDestroy(w.graph);
            cudaFree(w.d);
        }
        for (auto &f : fl) cudaFree(f.d_flow);
        cudaFree(d_reps);
        cudaFree(d_err);
        cudaFree(lwork.d);
        cudaFreeHost(h_lcnt);
        cudaFreeHost(h_err);
        cudaFreeHost(h_last);
        cudaFreeHost(h_reps);
    }

    // `v` as a work list on the device; after a failure the list counts as not
    // built, so that a later run builds it or fails again
    int upload_work(Work &w, const std::vector<BlockWork> &v) {
        if (!v.empty()) {
            const size_t bytes = v.size() * sizeof(BlockWork);
            BlockWork *d = nullptr;
            if (!cuda_ok(device_alloc((void **)&d, bytes), "steps_batch: alloc work")) return STEPS_ERR_OOM;
            if (!cuda_ok(cudaMemcpyAsync(d, v.data(), bytes, cudaMemcpyHostToDevice, stream), "steps_batch: upload work")) {
                cudaFree(d);
                return STEPS_ERR_CUDA;
            }
            w.d = d;
        }
        w.n = (int64_t)v.size();
        w.built = true;
        return STEPS_OK;
    }

    int build_work(int b) try {
        Work &w = work[slot(b)];
        if (w.built) return STEPS_OK;
        std::vector<BlockWork> v;
        for (size_t j = 0; j < members.size(); ++j) {
            const int64_t tiles = listed[j] ? 0 : (members[j]->T + b - 1) / b;
            for (int64_t t = 0; t < tiles; ++t) v.push_back(BlockWork{(int32_t)j, (int32_t)t});
        }
        return upload_work(w, v);
    } catch (const std::bad_alloc &) {
        set_error("steps_batch: work list: out of host memory");
        return STEPS_ERR_OOM;
    }

    // the members whose windows go through the list form, by what is known of their states
    std::vector<char> wanted() const {
        std::vector<char> want(members.size(), 0);
        for (size_t j = 0; j < members.size(); ++j) {
            const steps_sim *m = members[j];
            want[j] = use_spec && !flow && m->wants_list();
        }
        return want;
    }

    // the blocks of the listed members
    int build_list_work() try {
        if (lwork.built) return STEPS_OK;
        std::vector<BlockWork> v;
        for (size_t j = 0; j < members.size(); ++j) {
            const int64_t n = listed[j] ? list_blocks(members[j]->T, 256) : 0;
            for (int64_t t = 0; t < n; ++t) v.push_back(BlockWork{(int32_t)j, (int32_t)t});
            if (listed[j]) spec_list = members[j]->spec_list;
        }
        return upload_work(lwork, v);
    } catch (const std::bad_alloc &) {
        set_error("steps_batch: work list: out of host memory");
        return STEPS_ERR_OOM;
    }

    // Before a run: its members of the list form; the work lists and graphs
    // follow when they change (a batch is created with those of its members'
    // states, since freeing a list waits for the device).
    int choose_forms() try {
        const bool many = use_spec && !flow && max_S >= kListMinSpecies;
        const bool generic = !use_spec && max_S > 4 && max_S <= kWarpGenericSpecies;
        for (steps_sim *m : members)
            if ((many || generic) && m->density < 0.0)  // (the fill is unknown with it)
                if (int rc = m->measure(stream)) return rc;
        std::vector<char> want = wanted();
        // block tiles for the members that are not listed, by their tets and molecules together
        int64_t tets = 0;
        double molecules = 0.0;
        bool forced = false;
        for (size_t j = 0; j < members.size(); ++j)
            if (!want[j]) {
                tets += members[j]->T;
                molecules += members[j]->density * (double)members[j]->T;
                forced = forced || members[j]->forced == 3;
            }
        bool block = many && (forced || (tets > warp_wave(max_S) && molecules <= batch_block_density(max_S) * (double)tets));
        if (block && !spec_block) spec_block = spec_block_kernel(members[0]->model, 256);
        block = block && spec_block;
        for (size_t j = 0; j < members.size() && block; ++j)
            block = want[j] || members[j]->ensure_trial();
        const bool sparse = generic && molecules <= kFewPerTet * (double)tets;
        if (block != blocky || sparse != few)
            for (Work &w : work) {
                if (w.graph) cudaGraphExecDestroy(w.graph);
                w.graph = nullptr;
            }
        blocky = block;
        few = sparse;
        if (want != listed) {
            for (Work *w : {&work[0], &work[1], &work[2], &work[3], &lwork}) {
                if (w->graph) cudaGraphExecDestroy(w->graph);
                cudaFree(w->d);
                *w = Work{};
            }
            listed = std::move(want);
        }
        if (int rc = build_list_work()) return rc;
        for (size_t j = 0; j < members.size(); ++j) {
            steps_sim *m = members[j];
            if (m->listing != (bool)listed[j]) {
                m->drop_graphs();
                m->looked = m->k_total;
            }
            m->listing = listed[j];
            if (!m->listing) m->tm_valid = m->list_valid = false;  // the other kernels leave them behind
            int rc = m->prepare_list(stream);
            if (rc) return rc;
        }
        return STEPS_OK;
    } catch (const std::bad_alloc &) {
        set_error("steps_batch: work list: out of host memory");
        return STEPS_ERR_OOM;
    }

    // the specialised batched kernel for block size b (compiled once); on
    // failure the generic kernel takes over unless specialisation was forced
    int prepare_spec(int b) {
        if (!use_spec || spec[slot(b)]) return STEPS_OK;
        spec[slot(b)] = spec_kernel(members[0]->model, b, &spec_why);
        if (spec[slot(b)]) return STEPS_OK;
        if (spec_forced) {
            set_error("steps_batch_run: the specialised batched kernel could not be built: " + spec_why);
            return STEPS_ERR_CUDA;
        }
        use_spec = false;
        return STEPS_OK;
    }

    // launches of a batched window: tiles, the list form, advance
    uint64_t per_window(int b) const { return (work[slot(b)].n ? 1 : 0) + (lwork.n ? 1 : 0) + 1; }

    int window(int b, cudaStream_t st) {  // one batched window + advance
        Work &w = work[slot(b)];
        int rc = use_spec && spec[slot(b)] ? launch_spec_batch(blocky ? spec_block : spec[slot(b)], w.d, w.n, d_reps, b, st)
                                           : launch_step_batch(w.d, w.n, d_reps, max_S, max_R, any_order0, few, b, st);
        if (!rc && lwork.n) rc = launch_spec_batch(spec_list, lwork.d, lwork.n, d_reps, 256, st);
        if (!rc) rc = launch_advance(d_reps, (int32_t)members.size(), st);
        launches += per_window(b);
        return rc;
    }

    int graph_for(int b) {
        Work &w = work[slot(b)];
        if (w.graph) return STEPS_OK;
        cudaStream_t cs = nullptr;
        if (!cuda_ok(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "cudaStreamCreate")) return STEPS_ERR_CUDA;
        cudaGraph_t g = nullptr;
        int rc = STEPS_OK;
        if (!cuda_ok(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture")) {
            cudaStreamDestroy(cs);
            return STEPS_ERR_CUDA;
        }
        const uint64_t before = launches;
        for (int q = 0; q < kGraphWindows && rc == STEPS_OK; ++q) rc = window(b, cs);
        launches = before;
        cudaError_t e = cudaStreamEndCapture(cs, &g);
        if (rc == STEPS_OK && !cuda_ok(e, "cudaStreamEndCapture")) rc = STEPS_ERR_CUDA;
        if (rc == STEPS_OK && !cuda_ok(cudaGraphInstantiate(&w.graph, g, 0), "cudaGraphInstantiate")) rc = STEPS_ERR_CUDA;
        if (g) cudaGraphDestroy(g);
        cudaStreamDestroy(cs);
        return rc;
    }

    // the flow words and groups of block size b (once; build_work(b) first)
    int build_flow(int b) {
        Flow &f = fl[slot(b)];
        if (f.d_flow) return STEPS_OK;
        int dev = 0, l2 = 0;
        if (!cuda_ok(cudaGetDevice(&dev), "steps_batch: device") ||
            !cuda_ok(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev), "steps_batch: L2 size"))
            return STEPS_ERR_CUDA;
        std::vector<std::pair<int64_t, int64_t>> groups;
        int64_t nwork = 0;
        try {
            int64_t gfirst = 0, gbytes = 0;
            for (steps_sim *m : members) {
                const int64_t T = m->T, tiles = (T + b - 1) / b;
                // counts (both buffers) and tables the member's windows touch
                const int64_t bytes = T * (8 * (int64_t)m->S + 40) + (m->d_rmask ? 4 * T : 0);
                if (nwork > gfirst && gbytes + bytes > (int64_t)l2 / 2) {
                    groups.emplace_back(gfirst, nwork - gfirst);
                    gfirst = nwork;
                    gbytes = 0;
                }
                gbytes += bytes;
                nwork += tiles;
            }
            if (nwork > gfirst) groups.emplace_back(gfirst, nwork - gfirst);
        } catch (const std::bad_alloc &) {
            set_error("steps_batch: flow tables: out of host memory");
            return STEPS_ERR_OOM;
        }
        if (nwork != work[slot(b)].n) {
            set_error("steps_batch: flow tables do not match the work list");
            return STEPS_ERR_STATE;
        }
        // flow runs on the specialised kernels only: warp tiles, which publish per 32 tets and need no lists
        const int64_t nwords = nwork * (b / 32);
        if (!cuda_ok(device_alloc((void **)&f.d_flow, ((size_t)nwords + 1) * 4), "steps_batch: flow words"))
            return STEPS_ERR_OOM;
        if (!cuda_ok(cudaMemsetAsync(f.d_flow, 0, ((size_t)nwords + 1) * 4, stream), "steps_batch: flow words")) {
            cudaFree(f.d_flow);
            f.d_flow = nullptr;
            return STEPS_ERR_CUDA;
        }
        f.nwords = nwords;
        f.groups = std::move(groups);
        return STEPS_OK;
    }

    // n full windows of every member as flow launches, one per group (the
    // device member table is not advanced: the table of any later window
    // is uploaded from the host)
    int flow_windows(int b, int64_t n) {
        int rc = build_flow(b);
        if (rc) return rc;
        Flow &f = fl[slot(b)];
        for (const auto &g : f.groups) {
            const int64_t cap = std::max<int64_t>(1, (int64_t)0x7FFFFFFF / g.second);
            for (int64_t done = 0; done < n;) {
                const int64_t nw = std::min(n - done, cap);
                if (!cuda_ok(cudaMemsetAsync(f.d_flow + f.nwords, 0, 4, stream), "steps_batch: flow counter"))
                    return STEPS_ERR_CUDA;
                FlowArgs a;
                a.tnb_off = a.tnb = nullptr;
                a.tile_done = f.d_flow;
                a.fetch = f.d_flow + f.nwords;
                a.nwin = (uint32_t)nw;
                a.ntiles = (uint32_t)g.second;
                rc = launch_spec_batch_flow(spec[slot(b)], work[slot(b)].d, d_reps, a, (uint32_t)g.first, b,
                                            stream);
                if (rc) return rc;
                ++launches;
                ++flow_launches;
                done += nw;
            }
        }
        return STEPS_OK;
    }

    // What windows at block size b need, allocated. Called for every size a run
    // may use before its first window: a run that fails in between would leave
    // the members' counts ahead of their clocks.
    int prepare(int b) {
        int rc = build_work(b);
        if (!rc) rc = prepare_spec(b);
        return !rc && flow && use_spec && spec[slot(b)] ? build_flow(b) : rc;
    }

    int run_windows(int b, int64_t n) {  // n windows at block size b
        int rc = prepare(b);
        if (rc) return rc;
        if (flow && use_spec && spec[slot(b)] && n >= 2) return flow_windows(b, n);
        int64_t done = 0;
        if (use_graph && n >= kGraphWindows) {
            rc = graph_for(b);
            if (rc) return rc;
            for (; n - done >= kGraphWindows; done += kGraphWindows) {
                if (!cuda_ok(cudaGraphLaunch(work[slot(b)].graph, stream), "cudaGraphLaunch")) return STEPS_ERR_CUDA;
                launches += per_window(b) * kGraphWindows;
            }
        }
        for (; done < n; ++done) {
            rc = window(b, stream);
            if (rc) return rc;
        }
        return STEPS_OK;
    }
};

extern "C" {

void steps_batch_options_default(steps_batch_options *opt) {
    if (!opt) return;
    std::memset(opt, 0, sizeof(*opt));
    opt->block = 0;
    opt->use_graph = 1;
}

int steps_batch_create(steps_sim *const *members, int32_t n, const steps_batch_options *opt, void *cuda_stream,
                       steps_batch **out) {
    CHECK_NULL(out, "steps_batch_create");
    *out = nullptr;
    CHECK_NULL(members, "steps_batch_create");
    if (n < 1) {
        set_error("steps_batch_create: need at least one member");
        return STEPS_ERR_ARG;
    }
    std::unique_ptr<steps_batch> b(new (std::nothrow) steps_batch);
    if (!b) return STEPS_ERR_OOM;
    steps_batch_options o;
    if (opt) o = *opt;
    else steps_batch_options_default(&o);
    if (o.block != 0 && o.block != 64 && o.block != 128 && o.block != 256 && o.block != 512) {
        set_error("steps_batch_create: block must be 0 (autotune), 64, 128, 256 or 512");
        return STEPS_ERR_ARG;
    }
    b->autotune = o.block == 0;
    b->block = o.block == 0 ? 256 : o.block;
    b->use_graph = o.use_graph != 0;
    if (o.flow != 0 && o.flow != 1) {
        set_error("steps_batch_create: flow must be 0 (window launches, default) or 1 (group flow launches)");
        return STEPS_ERR_ARG;
    }
    b->flow = o.flow == 1;
    b->stream = (cudaStream_t)cuda_stream;
    for (int32_t j = 0; j < n; ++j) {
        if (!members[j]) {
            set_error("steps_batch_create: NULL member");
            return STEPS_ERR_ARG;
        }
        for (int32_t q = 0; q < j; ++q)
            if (members[q] == members[j]) {
                set_error("steps_batch_create: a simulation appears twice");
                return STEPS_ERR_ARG;
            }
        b->members.push_back(members[j]);
        b->max_S = std::max(b->max_S, members[j]->S);
        b->max_R = std::max(b->max_R, members[j]->model.R);
        b->any_order0 = b->any_order0 || members[j]->model.dev.order0 != 0u;
    }
    if (!cuda_ok(cudaMallocHost((void **)&b->h_reps, sizeof(RepEntry) * n), "steps_batch_create: host alloc") ||
        !cuda_ok(cudaMallocHost((void **)&b->h_last, sizeof(RepEntry) * n), "steps_batch_create: host alloc") ||
        !cuda_ok(cudaMallocHost((void **)&b->h_err, 4), "steps_batch_create: host alloc") ||
        (std::any_of(b->members.begin(), b->members.end(), [](const steps_sim *m) { return m->spec_list != nullptr; }) &&
         !cuda_ok(cudaMallocHost((void **)&b->h_lcnt, (size_t)n * 16), "steps_batch_create: host alloc")) ||
        !cuda_ok(device_alloc((void **)&b->d_reps, sizeof(RepEntry) * n), "steps_batch_create: alloc") ||
        !cuda_ok(device_alloc((void **)&b->d_err, 4), "steps_batch_create: alloc") ||
        !cuda_ok(cudaMemsetAsync(b->d_err, 0, 4, b->stream), "steps_batch_create: memset"))
        return STEPS_ERR_OOM;
    // the model-specialised batched kernel: all members must share one model structure
    bool uniform = true;
    int64_t tets = 0;
    const std::string src0 = spec_program_source(members[0]->model, 256);
    for (int32_t j = 0; j < n; ++j) {
        tets += members[j]->T;
        if (j > 0 && uniform && spec_program_source(members[j]->model, 256) != src0) uniform = false;
    }
    if (o.specialize > 0 && !uniform) {
        set_error("steps_batch_create: specialize = 1 needs members that share one model structure");
        return STEPS_ERR_ARG;
    }
    constexpr int64_t kSpecializeMinTets = 65536;
    bool any_exp = false;
    for (int32_t j = 0; j < n; ++j) any_exp = any_exp || members[j]->model.leave_exp;
    if (any_exp && (!uniform || o.specialize < 0)) {
        set_error("steps_batch_create: members with the EXP leave law run on the model-specialised batched "
                  "kernel only: they need one model structure and specialize 0 or 1");
        return STEPS_ERR_ARG;
    }
    b->spec_forced = o.specialize > 0 || any_exp;
    b->use_spec = uniform && (o.specialize > 0 || any_exp || (o.specialize == 0 && tets >= kSpecializeMinTets));
    b->listed = b->wanted();
    int rc = b->build_work(b->block);
    if (!rc) rc = b->build_list_work();
    if (rc) return rc;
    *out = b.release();
    return STEPS_OK;
}

void steps_batch_destroy(steps_batch *b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    else cudaDeviceSynchronize();
    delete b;
}

}  // extern "C"

namespace steps {

// steps_batch_run without its final wait: every window is enqueued on the
// batch's stream, the members' clocks advanced and the error word's copy to
// the host enqueued. batch_finish waits and turns the word into a code. While
// members go through the list form, no member takes more than `most` full
// windows (0: no limit) and *more says that there are others to run: the next
// call looks at the lists' lengths and builds them afresh.
int batch_enqueue(steps_batch *b, const double *t_end, int64_t most, bool *more) {
    CHECK_NULL(b, "steps_batch_run");
    CHECK_NULL(t_end, "steps_batch_run");
    const size_t n = b->members.size();
    for (size_t j = 0; j < n; ++j)
        if (!std::isfinite(t_end[j])) {
            set_error("steps_batch_run: t_end must be finite");
            return STEPS_ERR_ARG;
        }
    for (steps_sim *m : b->members)
        if (int rf = refuse_failed(m, "steps_batch_run")) return rf;
    // members' own streams may still hold work
    for (steps_sim *m : b->members)
        if (!cuda_ok(cudaStreamSynchronize(m->stream), "steps_batch_run: member stream")) return STEPS_ERR_CUDA;
    if (int rf = b->choose_forms()) return rf;
    const bool sliced = most > 0 && std::count(b->listed.begin(), b->listed.end(), 1) > 0;
    // the window schedule of every member (the loop of steps_run)
    std::vector<int64_t> nfull(n, 0);
    std::vector<double> partial(n, 0.0);  // > 0: a shortened last window of this length
    int64_t nmax = 0;
    for (size_t j = 0; j < n; ++j) {
        steps_sim *m = b->members[j];
        m->schedule(t_end[j], &nfull[j], &partial[j]);
        if (sliced && nfull[j] > most) {
            nfull[j] = most;
            partial[j] = 0.0;
            *more = true;
        }
        // the shortened window's leave table first where it waits for the stream
        if (m->leave_waits() && partial[j] > 0.0 && partial[j] != m->tab.tau)
            if (int rl = m->upload_leave(partial[j], b->stream)) return rl;
        nmax = std::max(nmax, nfull[j]);
    }
    // table for the full windows
    for (size_t j = 0; j < n; ++j) {
        steps_sim *m = b->members[j];
        RepEntry &e = b->h_reps[j];
        std::memset(&e, 0, sizeof(e));
        e.model = m->model.dev;
        e.args = m->args(0, m->k_total, nullptr, std::isfinite(m->tab.tau) ? m->tab.tau : 1.0, m->scale_full);
        e.args.err = b->d_err;
        e.cnt[0] = m->d_cnt[0];
        e.cnt[1] = m->d_cnt[1];
        e.tm[0] = m->d_tm[0];
        e.tm[1] = m->d_tm[1];
        e.parity = (uint32_t)m->cur;
        e.window_end = m->k_total + (uint64_t)nfull[j];
    }
    if (!cuda_ok(cudaMemcpyAsync(b->d_reps, b->h_reps, sizeof(RepEntry) * n, cudaMemcpyHostToDevice, b->stream),
                 "steps_batch_run: upload"))
        return STEPS_ERR_CUDA;
    int64_t done = 0;
    int rc = STEPS_OK;
    const int cand[3] = {128, 256, 512};
    const bool tune = b->autotune && !b->blocky && nmax >= 12;
    const int block = b->blocky ? 256 : b->block;
    for (int c = 0; c < 3 && tune && rc == STEPS_OK; ++c) rc = b->prepare(cand[c]);
    if (rc == STEPS_OK) rc = b->prepare(block);
    if (rc) return rc;
    if (tune) {
        // time the candidate block sizes on alternating windows (one warm window
        // each, then two rounds of one timed window each), so that the state's
        // slow drift over the run cancels; keep 256 unless another is more than
        // 2 % faster
        b->tune_ms.assign(3, 0.f);
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        if (!cuda_ok(cudaEventCreate(&e0), "steps_batch_run: autotuner event") ||
            !cuda_ok(cudaEventCreate(&e1), "steps_batch_run: autotuner event")) {
            if (e0) cudaEventDestroy(e0);
            return STEPS_ERR_CUDA;
        }
        float total[3] = {0.f, 0.f, 0.f};
        for (int round = 0; round < 2 && rc == STEPS_OK; ++round) {
            for (int c = 0; c < 3 && rc == STEPS_OK; ++c) {
                if (round == 0) {
                    rc = b->run_windows(cand[c], 1);  // warm
                    if (rc) break;
                    done += 1;
                }
                float ms = 0.f;
                if (!cuda_ok(cudaEventRecord(e0, b->stream), "steps_batch_run: autotuner") ||
                    (rc = b->run_windows(cand[c], 1)) != STEPS_OK ||
                    !cuda_ok(cudaEventRecord(e1, b->stream), "steps_batch_run: autotuner") ||
                    !cuda_ok(cudaEventSynchronize(e1), "steps_batch_run: autotuner") ||
                    !cuda_ok(cudaEventElapsedTime(&ms, e0, e1), "steps_batch_run: autotuner")) {
                    if (rc == STEPS_OK) rc = STEPS_ERR_CUDA;
                    break;
                }
                total[c] += ms;
                done += 1;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        if (rc) return rc;
        int best_b = 256;
        float best = total[1];
        for (int c = 0; c < 3; ++c) {
            b->tune_ms[c] = total[c] / 2.f;
            if (total[c] < 0.98f * best) {
                best = total[c];
                best_b = cand[c];
            }
        }
        b->block = best_b;
        b->autotune = false;
    }
    rc = b->run_windows(tune ? b->block : block, nmax - done);
    if (rc) return rc;
    // shortened last windows: their table goes into the second pinned buffer
    // (h_reps may still be read by its queued upload)
    bool any_partial = false;
    for (size_t j = 0; j < n; ++j) {
        steps_sim *m = b->members[j];
        RepEntry &e = b->h_last[j];
        e = b->h_reps[j];
        const uint64_t w = m->k_total + (uint64_t)nfull[j];
        e.args.window = w;
        e.parity = (uint32_t)(m->cur ^ (int)(nfull[j] & 1));
        e.window_end = w;
        if (partial[j] > 0.0) {
            any_partial = true;
            uint32_t scale[kMaxSpecies] = {};
            for (int s = 0; s < m->S; ++s) scale[s] = species_scale(m->model, m->tab, s, partial[j]);
            if (m->d_leave[0] && !m->leave_waits() && partial[j] != m->tab.tau)
                if (int rl = m->upload_leave(partial[j], b->stream)) return rl;
            StepArgs a = m->args(0, w, nullptr, partial[j], scale);
            a.err = b->d_err;
            e.args = a;
            e.window_end = w + 1;
        }
    }
    if (any_partial) {
        if (!cuda_ok(cudaMemcpyAsync(b->d_reps, b->h_last, sizeof(RepEntry) * n, cudaMemcpyHostToDevice, b->stream),
                     "steps_batch_run: upload"))
            return STEPS_ERR_CUDA;
        rc = b->run_windows(tune ? b->block : block, 1);
        if (rc) return rc;
    }
    // members' clocks and buffers
    for (size_t j = 0; j < n; ++j) {
        steps_sim *m = b->members[j];
        const int64_t wins = nfull[j] + (partial[j] > 0.0 ? 1 : 0);
        m->k_total += (uint64_t)wins;
        m->launches += (uint64_t)wins;
        m->cur ^= (int)(wins & 1);
        if (partial[j] > 0.0) {
            m->t_base = t_end[j];
            m->k_grid = 0;
        } else {
            m->k_grid += nfull[j];
        }
    }
    for (size_t j = 0; j < n; ++j)
        if (b->listed[j] && !cuda_ok(cudaMemcpyAsync(b->h_lcnt + 4 * j, b->members[j]->d_lcnt, 16,
                                                     cudaMemcpyDeviceToHost, b->stream),
                                     "steps_batch_run: list length"))
            return STEPS_ERR_CUDA;
    if (!cuda_ok(cudaMemcpyAsync(b->h_err, b->d_err, 4, cudaMemcpyDeviceToHost, b->stream),
                 "steps_batch_run: error word"))
        return STEPS_ERR_CUDA;
    return STEPS_OK;
}

int batch_finish(steps_batch *b) {
    if (!cuda_ok(cudaStreamSynchronize(b->stream), "steps_batch_run")) return STEPS_ERR_CUDA;
    for (size_t j = 0; j < b->members.size(); ++j)
        if (b->listed[j]) b->members[j]->fill_from(b->h_lcnt + 4 * j);
    const uint32_t err = *b->h_err;
    if (err) cudaMemsetAsync(b->d_err, 0, 4, b->stream);
    bool closed = false;
    const int rc = error_word(err, "steps_batch_run", &closed);
    for (steps_sim *m : b->members) m->failed = m->failed || closed;
    return rc;
}

std::string sim_structure_key(const steps_sim *sim) { return spec_program_source(sim->model, 256); }

}  // namespace steps

extern "C" {

int steps_batch_run(steps_batch *b, const double *t_end) {
    for (bool more = true; more;) {
        more = false;
        int rc = steps::batch_enqueue(b, t_end, (int64_t)kListCheckWindows, &more);
        if (!rc) rc = steps::batch_finish(b);
        if (rc) return rc;
    }
    return STEPS_OK;
}

int steps_batch_specialized(const steps_batch *b, int32_t *specialized) {
    CHECK_NULL(b, "steps_batch_specialized");
    CHECK_NULL(specialized, "steps_batch_specialized");
    *specialized = b->use_spec ? 1 : 0;
    return STEPS_OK;
}

int steps_batch_info(const steps_batch *b, int32_t *block, uint64_t *launches, float *tune_ms) {
    CHECK_NULL(b, "steps_batch_info");
    if (block) *block = b->block;
    if (launches) *launches = b->launches;
    if (tune_ms)
        for (int c = 0; c < 3; ++c) tune_ms[c] = c < (int)b->tune_ms.size() ? b->tune_ms[c] : 0.f;
    return STEPS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free run on caller-owned device counts.
//
// Scratch for steps_run_noalloc lives in this file-scope device array: two
// receiving/sending count buffers of up to kNoAllocMaxCounts int32 each, then
// an error word. Every GPU that loads the library holds it (32 MiB + 256 B)
// until the process exits. Host code cannot use the array's name as a device
// address; the address is looked up once per device with
// cudaGetSymbolAddress, with that device current.
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocMaxCounts = (size_t)1 << 22;  // n_species * Tpad per buffer
static __device__ __align__(256) int32_t g_noalloc_scratch[2 * kNoAllocMaxCounts + 64];

namespace {

struct NoAllocScratch {
    bool ready = false;
    int32_t *counts = nullptr;  // [2][kNoAllocMaxCounts]
    uint32_t *err = nullptr;    // after the count buffers: window error word, unused, any_negative's four
};

constexpr int kNoAllocMaxDevices = 64;
NoAllocScratch g_noalloc_dev[kNoAllocMaxDevices];
std::mutex g_noalloc_mu;

int noalloc_scratch(NoAllocScratch &out) {
    int dev = -1;
    if (!cuda_ok(cudaGetDevice(&dev), "steps_run_noalloc: cudaGetDevice")) return STEPS_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) {
        set_error("steps_run_noalloc: device index out of range");
        return STEPS_ERR_ARG;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoAllocScratch &s = g_noalloc_dev[dev];
    if (!s.ready) {
        void *p = nullptr;
        if (!cuda_ok(cudaGetSymbolAddress(&p, g_noalloc_scratch), "steps_run_noalloc: cudaGetSymbolAddress"))
            return STEPS_ERR_CUDA;
        s.counts = static_cast<int32_t *>(p);
        s.err = reinterpret_cast<uint32_t *>(s.counts + 2 * kNoAllocMaxCounts);
        s.ready = true;
    }
    out = s;
    return STEPS_OK;
}

}  // namespace

extern "C" int steps_run_noalloc(steps_sim *sim, int32_t *d_counts, double t_end) {
    CHECK_NULL(sim, "steps_run_noalloc");
    CHECK_NULL(d_counts, "steps_run_noalloc");
    if (!std::isfinite(t_end)) {
        set_error("steps_run_noalloc: t_end must be finite");
        return STEPS_ERR_ARG;
    }
    const size_t S = (size_t)sim->S, T = (size_t)sim->T, Tpad = (size_t)sim->Tpad;
    if (S * Tpad > kNoAllocMaxCounts) {
        set_error("steps_run_noalloc: n_species * padded tets = " + std::to_string(S * Tpad) +
                  " exceeds the fixed scratch of " + std::to_string(kNoAllocMaxCounts) +
                  " counts; use steps_run");
        return STEPS_ERR_ARG;
    }
    if (int rf = refuse_failed(sim, "steps_run_noalloc")) return rf;
    if (sim->d_leave[0]) {
        set_error("steps_run_noalloc: the EXP leave law needs a leave table for a shortened window, which "
                  "this call has no room for; use steps_run");
        return STEPS_ERR_ARG;
    }
    // the scratch address is per device, and the simulation's stream and
    // tables belong to the device it was created on
    int dev = -1;
    if (!cuda_ok(cudaGetDevice(&dev), "steps_run_noalloc: cudaGetDevice")) return STEPS_ERR_CUDA;
    if (dev != sim->device) {
        set_error("steps_run_noalloc: the current device (" + std::to_string(dev) +
                  ") is not the one the simulation was created on (" + std::to_string(sim->device) +
                  "); make that device current first");
        return STEPS_ERR_ARG;
    }
    NoAllocScratch sc;
    int rc = noalloc_scratch(sc);
    if (rc) return rc;
    int32_t *buf[2] = {sc.counts, sc.counts + kNoAllocMaxCounts};
    cudaStream_t st = sim->stream;
    // the scratch keeps the previous call's contents: clear both buffers
    // (padding and receiving rows must be zero) and both error words
    if (!cuda_ok(cudaMemsetAsync(buf[0], 0, S * Tpad * 4, st), "steps_run_noalloc: clear") ||
        !cuda_ok(cudaMemsetAsync(buf[1], 0, S * Tpad * 4, st), "steps_run_noalloc: clear") ||
        !cuda_ok(cudaMemsetAsync(sc.err, 0, 24, st), "steps_run_noalloc: clear"))
        return STEPS_ERR_CUDA;
    // reject negative input counts before anything (clock, caller's buffer) changes
    double density = 0.0;
    {
        const int64_t n = (int64_t)(S * T);
        uint32_t seen[4] = {0, 0, 0, 0};  // (any_negative)
        if (sim->block_possible()) any_negative<true><<<input_blocks(n), kInputThreads, 0, st>>>(d_counts, n, sc.err + 2);
        else any_negative<false><<<input_blocks(n), kInputThreads, 0, st>>>(d_counts, n, sc.err + 2);
        if (!cuda_ok(cudaGetLastError(), "steps_run_noalloc: check") ||
            !cuda_ok(cudaMemcpyAsync(seen, sc.err + 2, 16, cudaMemcpyDeviceToHost, st), "steps_run_noalloc: check") ||
            !cuda_ok(cudaStreamSynchronize(st), "steps_run_noalloc: check"))
            return STEPS_ERR_CUDA;
        if (seen[0]) {
            set_error("steps_run_noalloc: negative count in d_counts");
            return STEPS_ERR_ARG;
        }
        density = (double)((uint64_t)seen[3] << 32 | seen[2]) / (double)T;
    }
    const unsigned grid = (unsigned)((T + 255) / 256);
    scatter_to_device_order<<<grid, 256, 0, st>>>(d_counts, (int64_t)T, (int32_t)S, sim->d_inv_perm, buf[0], Tpad);
    if (!cuda_ok(cudaGetLastError(), "steps_run_noalloc: scatter")) return STEPS_ERR_CUDA;

    // the window loop of steps_run (Algorithm 1), with plain launches on the scratch buffers (never the list form)
    const bool block = sim->spec_block && sim->wants_block(density);  // (nothing is allocated or compiled here)
    if (sim->listing || sim->blocky != block) sim->drop_graphs();
    sim->listing = sim->tm_valid = sim->list_valid = false;
    sim->blocky = block;
    const double tau = sim->tab.tau;
    const bool finite = std::isfinite(tau);
    const double tol = finite ? 1e-9 * tau : 0.0;
    int cur = 0;
    auto launch = [&](double tau_k, const uint32_t *scale) -> int {
        StepArgs a = sim->args(0, sim->k_total, nullptr, tau_k, scale);
        a.cur = buf[cur];
        a.nxt = buf[1 - cur];
        a.err = sc.err;
        int r = sim->launch(a, st);
        if (r) return r;
        ++sim->launches;
        ++sim->k_total;
        cur = 1 - cur;
        return STEPS_OK;
    };
    for (;;) {
        const double t = sim->time();
        if (!(t_end - t > tol)) break;
        if (finite && t + tau <= t_end + tol) {
            rc = launch(tau, sim->scale_full);
            if (rc) return rc;
            sim->k_grid += 1;
        } else {
            uint32_t scale[kMaxSpecies] = {};
            for (int s = 0; s < sim->S; ++s) scale[s] = species_scale(sim->model, sim->tab, s, t_end - t);
            rc = launch(t_end - t, scale);
            if (rc) return rc;
            sim->t_base = t_end;
            sim->k_grid = 0;
            break;
        }
    }
    gather_to_original_order<<<grid, 256, 0, st>>>(buf[cur], (int64_t)T, (int32_t)S, sim->d_inv_perm, Tpad, d_counts);
    if (!cuda_ok(cudaGetLastError(), "steps_run_noalloc: gather")) return STEPS_ERR_CUDA;
    uint32_t err = 0;
    if (!cuda_ok(cudaMemcpyAsync(&err, sc.err, 4, cudaMemcpyDeviceToHost, st), "steps_run_noalloc: error word") ||
        !cuda_ok(cudaStreamSynchronize(st), "steps_run_noalloc"))
        return STEPS_ERR_CUDA;
    bool closed = false;
    rc = error_word(err, "steps_run_noalloc", &closed);
    if (closed) sim->failed = true;
    return rc;
}
