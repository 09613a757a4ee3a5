// Model-specialised step kernels, compiled at run time.
//
// The step body (steps_step.cuh) reads the model through a policy class. The
// generic kernels use RtModel, which looks reactants, flags and
// stoichiometry up in a per-tile table. Here, for one model, a policy is
// generated as C++ source: the species count, the diffusive set, each
// reaction's reactant rows, propensity form and changes become constants.
// The same step body, specialised with it, is then compiled for the device
// by NVRTC. The rate constants stay kernel parameters, so
// steps_set_reac_rate needs no recompilation. The arithmetic is the generic
// kernel's, operation for operation, so both give the same bits.
//
// NVRTC is opened with dlopen: without it the library still loads and the
// generic kernels run. The code is loaded with the runtime's library API
// (cudaLibraryLoadData), and kernels are cached per generated source.
#include <cuda_runtime.h>
#include <dlfcn.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "steps_internal.h"

namespace steps {

extern const char *const kSrcDeviceH;  // steps_device.h, embedded at build time
extern const char *const kSrcStepCuh;  // steps_step.cuh, embedded at build time
extern const char *const kSrcWarpCuh;  // steps_warp.cuh, embedded at build time
extern const char *const kSrcListCuh;  // steps_list.cuh, embedded at build time

namespace {

// The few NVRTC entry points used (C ABI of libnvrtc).
typedef int nvrtc_result;
typedef struct nvrtc_program_st *nvrtc_program;
struct Nvrtc {
    void *handle = nullptr;
    nvrtc_result (*create)(nvrtc_program *, const char *, const char *, int, const char *const *,
                           const char *const *) = nullptr;
    nvrtc_result (*compile)(nvrtc_program, int, const char *const *) = nullptr;
    nvrtc_result (*log_size)(nvrtc_program, size_t *) = nullptr;
    nvrtc_result (*log)(nvrtc_program, char *) = nullptr;
    nvrtc_result (*cubin_size)(nvrtc_program, size_t *) = nullptr;
    nvrtc_result (*cubin)(nvrtc_program, char *) = nullptr;
    nvrtc_result (*destroy)(nvrtc_program *) = nullptr;
    std::string why;
};

Nvrtc &nvrtc() {
    static Nvrtc n = [] {
        Nvrtc x;
        const char *names[] = {"libnvrtc.so.13", "libnvrtc.so", "libnvrtc.so.12"};
        for (const char *nm : names)
            if ((x.handle = dlopen(nm, RTLD_NOW | RTLD_LOCAL)) != nullptr) break;
        if (!x.handle) {
            x.why = "libnvrtc not found";
            return x;
        }
        x.create = reinterpret_cast<decltype(x.create)>(dlsym(x.handle, "nvrtcCreateProgram"));
        x.compile = reinterpret_cast<decltype(x.compile)>(dlsym(x.handle, "nvrtcCompileProgram"));
        x.log_size = reinterpret_cast<decltype(x.log_size)>(dlsym(x.handle, "nvrtcGetProgramLogSize"));
        x.log = reinterpret_cast<decltype(x.log)>(dlsym(x.handle, "nvrtcGetProgramLog"));
        x.cubin_size = reinterpret_cast<decltype(x.cubin_size)>(dlsym(x.handle, "nvrtcGetCUBINSize"));
        x.cubin = reinterpret_cast<decltype(x.cubin)>(dlsym(x.handle, "nvrtcGetCUBIN"));
        x.destroy = reinterpret_cast<decltype(x.destroy)>(dlsym(x.handle, "nvrtcDestroyProgram"));
        if (!x.create || !x.compile || !x.log_size || !x.log || !x.cubin_size || !x.cubin || !x.destroy) {
            x.why = "libnvrtc lacks an entry point";
            x.handle = nullptr;
        }
        return x;
    }();
    return n;
}

}  // namespace

bool spec_block_trial(const HostModel &hm) { return hm.dev.S >= 16; }

namespace {

std::string hex_u32(uint32_t v) {
    std::ostringstream o;
    o << "0x" << std::hex << v << "u";
    return o.str();
}

// The generated policy of the list form and of block tiles: the functions of
// RtModel with the model's structure as constants (block: entries of a count
// row). Propensity forms (all in float, as RtModel):
//   order 0: k / inv_nav            order 1: k x
//   order 2: ((k inv_nav) x) y      dimer:   ((k inv_nav) x) (x - 1)
// (RtModel's extra factors of 1 are exact and left out.)
std::string table_policy_source(const HostModel &hm, int block) {
    const ModelDev &m = hm.dev;
    std::ostringstream o;
    o << "namespace steps {\nnamespace {\nstruct SpecModel {\n";
    o << "    static constexpr bool kGlobalTrial = " << (spec_block_trial(hm) ? "true" : "false") << ";\n";
    o << "    static constexpr bool kExpLeave = " << (hm.leave_exp ? "true" : "false") << ";\n";
    o << "    __device__ static int S(const ModelDev &) { return " << m.S << "; }\n";
    o << "    __device__ static int R(const ModelDev &) { return " << m.R << "; }\n";
    o << "    __device__ static uint32_t diffusive(const ModelDev &) { return " << hex_u32(m.diffusive) << "; }\n";
    o << "    __device__ static uint32_t need(const RxnTab &tb, int r) { return tb.need[r]; }\n";
    o << "    template <int BLOCK>\n    __device__ static void build(const ModelDev &m, RxnTab &tb) {\n";
    o << "        build_rxn_tab<BLOCK, " << block << ">(m, tb);\n    }\n";
    o << "    __device__ static float prop(const RxnTab &, const ModelDev &m, int r, const int32_t *cnt, float inv_nav) {\n";
    o << "        switch (r) {\n";
    for (int r = 0; r < m.R; ++r) {
        const ReacDesc &d = m.reac[r];
        const std::string k = "m.reac[" + std::to_string(r) + "].k";
        const std::string x = "__int2float_rn(cnt[" + std::to_string(d.ia * block) + "])";
        o << "        case " << r << ": return ";
        switch (d.type) {
        case kOrder0: o << "__fdiv_rn(" << k << ", inv_nav)"; break;
        case kOrder1: o << "__fmul_rn(" << k << ", " << x << ")"; break;
        case kOrder2:
            o << "__fmul_rn(__fmul_rn(__fmul_rn(" << k << ", inv_nav), " << x << "), __int2float_rn(cnt["
              << d.ib * block << "]))";
            break;
        default:
            o << "__fmul_rn(__fmul_rn(__fmul_rn(" << k << ", inv_nav), " << x << "), __int2float_rn(cnt["
              << d.ib * block << "] - 1))";
            break;
        }
        o << ";\n";
    }
    o << "        default: return 0.0f;\n        }\n    }\n";
    // the stoichiometry from the tile's table: a switch over reactions inside the
    // SSA loop would inline every reaction's occupancy update there
    o << "    template <class F>\n    __device__ static void for_changes(const RxnTab &tb, int r, F f) {\n";
    o << "        RtModel<false>::for_changes(tb, r, f);\n    }\n";
    o << "    template <int RM>\n    __device__ __forceinline__ static float sums(const RxnTab &tb, const ModelDev &m, "
             "const int32_t *cnt, float inv_nav, uint32_t active, bool, float *psum) {\n"
             "        return propensity_sums<SpecModel, RM>(tb, m, cnt, inv_nav, active, psum);\n    }\n"
             "    template <int RM>\n    __device__ __forceinline__ static int pick(const RxnTab &tb, const ModelDev &m, "
             "const float *psum, float target, const int32_t *cnt, float inv_nav, uint32_t active) {\n"
             "        return pick_reaction<SpecModel, RM>(tb, m, psum, target, cnt, inv_nav, active);\n    }\n";
    o << "};\n}  // namespace\n}  // namespace steps\n";

    return o.str();
}

// The generated policy of the warp-tile step. The counts of a tet are read and
// converted once per sweep; every propensity is then two or three products in
// registers (the forms above, the same operations in the same order), and one
// with an absent reactant is exactly 0 by itself.
std::string warp_policy_source(const HostModel &hm) {
    const ModelDev &m = hm.dev;
    std::ostringstream o;
    o << "namespace steps {\nnamespace {\nstruct SpecModel {\n";
    o << "    static constexpr bool kExpLeave = " << (hm.leave_exp ? "true" : "false") << ";\n";
    o << "    __device__ static constexpr int S(const ModelDev &) { return " << m.S << "; }\n";
    o << "    __device__ static constexpr int R(const ModelDev &) { return " << m.R << "; }\n";
    o << "    __device__ static constexpr uint32_t diffusive(const ModelDev &) { return " << hex_u32(m.diffusive)
      << "; }\n";
    o << "    template <int THREADS>\n    __device__ static void build(const ModelDev &m, RxnTab &tb) {\n";
    o << "        if (threadIdx.x < THREADS) build_rxn_tab<THREADS, 32>(m, tb);\n    }\n";
    o << "    template <class F>\n    __device__ static void for_changes(const RxnTab &tb, int r, F f) {\n";
    o << "        RtModel<false>::for_changes(tb, r, f);\n    }\n";
    o << "    template <int RM, bool MASKED>\n    __device__ __forceinline__ static float sums_of(const ModelDev &m, "
         "const int32_t *cnt, float inv_nav, uint32_t active, float *psum) {\n";
    uint32_t used = 0;
    for (int r = 0; r < m.R; ++r) {
        if (m.reac[r].ia < m.S) used |= 1u << m.reac[r].ia;
        if (m.reac[r].ib < m.S && m.reac[r].type == kOrder2) used |= 1u << m.reac[r].ib;
    }
    for (int s = 0; s < m.S; ++s)
        if ((used >> s) & 1u) o << "        const float x" << s << " = __int2float_rn(cnt[" << s * 32 << "]);\n";
    o << "        float a0 = 0.0f, ar;\n";
    for (int r = 0; r < m.R; ++r) {
        const ReacDesc &d = m.reac[r];
        const std::string k = "m.reac[" + std::to_string(r) + "].k", x = "x" + std::to_string(d.ia);
        o << "        ar = ";
        switch (d.type) {
        case kOrder0: o << "__fdiv_rn(" << k << ", inv_nav)"; break;
        case kOrder1: o << "__fmul_rn(" << k << ", " << x << ")"; break;
        case kOrder2:
            o << "__fmul_rn(__fmul_rn(__fmul_rn(" << k << ", inv_nav), " << x << "), x" << d.ib << ")";
            break;
        default:
            o << "__fmul_rn(__fmul_rn(__fmul_rn(" << k << ", inv_nav), " << x << "), __int2float_rn(cnt["
              << d.ib * 32 << "] - 1))";
            break;
        }
        o << ";\n        if (MASKED && !((active >> " << r << ") & 1u)) ar = 0.0f;\n";
        o << "        psum[" << r << "] = a0 = __fadd_rn(a0, ar);\n";
    }
    o << "        return a0;\n    }\n";
    o << "    template <int RM>\n    __device__ __forceinline__ static float sums(const RxnTab &, const ModelDev &m, "
         "const int32_t *cnt, float inv_nav, uint32_t active, bool masked, float *psum) {\n"
         "        return masked ? sums_of<RM, true>(m, cnt, inv_nav, active, psum)\n"
         "                      : sums_of<RM, false>(m, cnt, inv_nav, active, psum);\n    }\n";
    o << "    template <int RM>\n    __device__ __forceinline__ static float first_sums(const RxnTab &tb, const "
         "ModelDev &m, const int32_t *cnt, float inv_nav, uint32_t active, bool masked, float *psum) {\n"
         "        const float a0 = sums<RM>(tb, m, cnt, inv_nav, active, masked, psum);\n"
         "        if (a0 <= kPlainSums) return a0;\n"
         "        float ps[RM];\n"
         "        const float a1 = careful_sums(tb, m, cnt, inv_nav, active, ps);\n"
         "        for (int r = 0; r < " << m.R << "; ++r) psum[r] = ps[r];\n"
         "        return a1;\n    }\n";
    o << "    template <int RM>\n    __device__ __forceinline__ static int pick(const RxnTab &tb, const ModelDev &m, "
         "const float *psum, float target, const int32_t *cnt, float inv_nav, uint32_t active) {\n"
         "        int n = 0;\n"
         "#pragma unroll\n"
         "        for (int r = 0; r < " << m.R << "; ++r) n += psum[r] <= target ? 1 : 0;\n"
         "        return n < " << m.R << " ? n : last_positive_tab(tb, m, cnt, inv_nav, active);\n    }\n";
    o << "};\n}  // namespace\n}  // namespace steps\n";
    return o.str();
}

std::string program_source(const HostModel &hm, int block) {
    std::ostringstream o;
    const std::string b = std::to_string(block);
    const std::string args = "<" + b + ", " + std::to_string(std::max(1, hm.dev.R)) + ", " +
                             std::to_string(hm.dev.S) + ", steps::SpecModel";
    const std::string head = "extern \"C\" __global__ void __launch_bounds__(" + b + ", " +
                             std::to_string(1024 / block) + ")\n";
    const std::string member = "const steps::BlockWork *__restrict__ work, const steps::RepEntry *__restrict__ reps";
    o << "#include \"steps_warp.cuh\"\n" << warp_policy_source(hm);
    o << head << "steps_spec_step(const __grid_constant__ steps::ModelDev m, const __grid_constant__ "
      << "steps::StepArgs a) {\n    steps::warp_step" << args << ">(m, a, (int64_t)blockIdx.x);\n}\n";
    o << head << "steps_spec_flow(const __grid_constant__ steps::ModelDev m, const __grid_constant__ "
      << "steps::StepArgs a, const __grid_constant__ steps::FlowArgs f) {\n    steps::warp_step" << args
      << ", 1>(m, a, 0, &f);\n}\n";
    o << head << "steps_spec_batch(" << member << ") {\n"
      << "    steps::batch_member<" << b << ">(work, reps, 0, [](const steps::ModelDev &m, const "
      << "steps::StepArgs &a, int64_t tile) { steps::warp_step" << args << ">(m, a, tile); });\n}\n";
    o << head << "steps_spec_batch_flow(" << member << ", const __grid_constant__ steps::FlowArgs f, uint32_t work0) {\n"
      << "    steps::batch_flow_member<" << b << ">(work, reps, f, work0, [&f](const steps::ModelDev &m, "
      << "const steps::StepArgs &a, int64_t tile, uint32_t q, uint32_t dep) { steps::warp_step" << args
      << ", 2>(m, a, tile, &f, q, dep); });\n}\n";
    return o.str();
}

// The list form's program: a plain and a batched step kernel (256-thread blocks).
constexpr int kListBlock = 256;

std::string list_program_source(const HostModel &hm) {
    std::ostringstream o;
    const std::string b = std::to_string(kListBlock);
    o << "#include \"steps_list.cuh\"\n" << table_policy_source(hm, 32);
    o << "extern \"C\" __global__ void __launch_bounds__(" << b << ", " << 1024 / kListBlock << ")\n"
      << "steps_spec_list(const __grid_constant__ steps::ModelDev m, const __grid_constant__ steps::StepArgs a) {\n"
      << "    steps::list_step<" << b << ", " << std::max(1, hm.dev.R) << ", " << hm.dev.S
      << ", steps::SpecModel>(m, a, blockIdx.x, gridDim.x);\n}\n";
    o << "extern \"C\" __global__ void __launch_bounds__(" << b << ", " << 1024 / kListBlock << ")\n"
      << "steps_spec_list_batch(const steps::BlockWork *__restrict__ work, const steps::RepEntry *__restrict__ reps) {\n"
      << "    steps::batch_member<" << b << ">(work, reps, 0, [](const steps::ModelDev &m, const steps::StepArgs &a, "
      << "int64_t tile) {\n        steps::list_step<" << b << ", " << std::max(1, hm.dev.R) << ", " << hm.dev.S
      << ", steps::SpecModel>(m, a, (uint32_t)tile, (uint32_t)steps::list_blocks(a.T, " << b << "));\n    });\n}\n";
    return o.str();
}

// The block tiles' program: plain, flow and batched step kernels. With the
// trial counts in global memory, five blocks of 256 threads fit an SM with a
// 32-entry block map and 48 registers per thread.
int reaction_bucket(int R) { return R <= 8 ? 8 : R <= 16 ? 16 : R <= 24 ? 24 : 32; }

std::string block_program_source(const HostModel &hm, int block) {
    std::ostringstream o;
    const bool five = spec_block_trial(hm) && block == 256;
    const std::string b = std::to_string(block), per_sm = std::to_string(1024 / block);
    const std::string head = "extern \"C\" __global__ void __launch_bounds__(" + b + ", " + (five ? "5" : per_sm) + ")\n";
    const std::string args = "<" + b + ", " + std::to_string(reaction_bucket(hm.dev.R)) + ", steps::SpecModel>";
    if (five) o << "#define STEPS_MAP_CAP 32\n";
    o << "#include \"steps_step.cuh\"\n" << table_policy_source(hm, block);
    o << head << "steps_spec_step(const __grid_constant__ steps::ModelDev m, const __grid_constant__ steps::StepArgs a) "
      << "{\n    steps::step_tile" << args << "(m, a, (int64_t)blockIdx.x);\n}\n";
    o << head << "steps_spec_flow(const __grid_constant__ steps::ModelDev m, const __grid_constant__ steps::StepArgs a, "
      << "const __grid_constant__ steps::FlowArgs f) {\n    steps::flow_tiles" << args << "(m, a, f);\n}\n";
    o << "extern \"C\" __global__ void __launch_bounds__(" << b << ", " << per_sm << ")\n"
      << "steps_spec_batch(const steps::BlockWork *__restrict__ work, const steps::RepEntry *__restrict__ reps, "
      << "int32_t prefetch) {\n    steps::batch_tile" << args << "(work, reps, prefetch);\n}\n";
    return o.str();
}

enum class Form { tiles, list, block };

struct Compiled {
    Form form = Form::tiles;
    int block = 0;                      // threads per block
    cudaLibrary_t lib = nullptr;
    cudaKernel_t kern = nullptr;        // plain step kernel
    cudaKernel_t kern_batch = nullptr;  // batched step kernel
    cudaKernel_t kern_flow = nullptr;   // flow kernel of a simulation's full windows
    cudaKernel_t kern_batch_flow = nullptr;  // flow kernel of a group of batch members
    size_t smem_set = 0;                // dynamic shared memory the plain kernel was opted in to
    size_t smem_set_flow = 0;           // the flow kernel
    size_t smem_set_batch_flow = 0;     // the batched flow kernel
    size_t smem_set_batch = 0;          // and the batched one
    size_t smem = 0;                    // dynamic shared memory per block
};

std::mutex g_mu;
std::map<std::string, std::shared_ptr<Compiled>> g_cache;

}  // namespace

std::string spec_program_source(const HostModel &hm, int block) { return program_source(hm, block); }

namespace {

// A generated program's binary, or nothing and why.
std::vector<char> build_program(Nvrtc &nv, const std::string &src, std::string *why) {
    std::vector<char> cubin;
    nvrtc_program prog = nullptr;
    const char *hdr_src[4] = {kSrcDeviceH, kSrcStepCuh, kSrcWarpCuh, kSrcListCuh};
    const char *hdr_name[4] = {"steps_device.h", "steps_step.cuh", "steps_warp.cuh", "steps_list.cuh"};
    if (nv.create(&prog, src.c_str(), "steps_spec.cu", 4, hdr_src, hdr_name) != 0) {
        if (why) *why = "nvrtcCreateProgram failed";
        return cubin;
    }
    // the generic kernels' flags: no contraction, C++17, this GPU only
    const char *opts[] = {"--gpu-architecture=sm_103a", "-std=c++17", "-fmad=false", "-lineinfo", "--device-int128"};
    const int rc = nv.compile(prog, 5, opts);
    if (rc == 0) {
        size_t n = 0;
        if (nv.cubin_size(prog, &n) == 0 && n > 0) {
            cubin.resize(n);
            if (nv.cubin(prog, cubin.data()) != 0) cubin.clear();
        }
    } else if (why) {
        size_t n = 0;
        nv.log_size(prog, &n);
        std::string lg(n, '\0');
        if (n) nv.log(prog, &lg[0]);
        *why = "NVRTC compile failed: " + lg.substr(0, 2000);
    }
    nv.destroy(&prog);
    return cubin;
}

// Compiles (once per generated source) and loads a form's kernels. Compiled
// without the lock, so that two programs of a model are at the same time.
Compiled *compiled(const HostModel &hm, int block, Form form, std::string *why) {
    Nvrtc &nv = nvrtc();
    if (!nv.handle) {
        if (why) *why = nv.why;
        return nullptr;
    }
    const std::string src = form == Form::list    ? list_program_source(hm)
                            : form == Form::block ? block_program_source(hm, block)
                                                  : program_source(hm, block);
    const auto known = [&](Compiled **c) {
        auto it = g_cache.find(src);
        if (it == g_cache.end()) return false;
        if (!it->second && why) *why = "an earlier build of this kernel failed";
        *c = it->second.get();
        return true;
    };
    Compiled *done = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (known(&done)) return done;
    }
    const std::vector<char> cubin = build_program(nv, src, why);
    std::lock_guard<std::mutex> lock(g_mu);
    if (known(&done)) return done;
    if (cubin.empty()) {
        g_cache[src] = nullptr;
        return nullptr;
    }
    auto c = std::make_shared<Compiled>();
    const auto get = [&](cudaKernel_t *k, const char *name) { return cudaLibraryGetKernel(k, c->lib, name) == cudaSuccess; };
    bool ok = cudaLibraryLoadData(&c->lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0) == cudaSuccess;
    const size_t S = (size_t)hm.dev.S;
    c->form = form;
    c->block = block;
    if (form == Form::list) {
        c->smem = (size_t)(kListBlock / 32) * list_tile_bytes(hm.dev.S);
        ok = ok && get(&c->kern, "steps_spec_list") && get(&c->kern_batch, "steps_spec_list_batch");
    } else {
        c->smem = form == Form::block ? (S + 1 + (spec_block_trial(hm) ? 0 : S)) * (size_t)block * sizeof(int32_t)
                                      : (size_t)(block / 32) * warp_tile_bytes(hm.dev.S);
        ok = ok && get(&c->kern, "steps_spec_step") && get(&c->kern_batch, "steps_spec_batch") &&
             get(&c->kern_flow, "steps_spec_flow") &&
             (form == Form::block || get(&c->kern_batch_flow, "steps_spec_batch_flow"));
    }
    if (!ok) {
        cudaGetLastError();
        if (why) *why = "loading the compiled kernel failed";
        g_cache[src] = nullptr;
        return nullptr;
    }
    g_cache[src] = c;
    return c.get();
}

// Opts a kernel in to `smem` bytes of dynamic shared memory (once per size).
bool opt_in(const void *fn, size_t smem, size_t *done) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (*done >= smem) return true;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        set_error("specialised step kernel shared memory: " + std::string(cudaGetErrorString(cudaGetLastError())));
        return false;
    }
    *done = smem;
    return true;
}

}  // namespace

void *spec_kernel(const HostModel &hm, int block, std::string *why) {
    return (void *)compiled(hm, block, Form::tiles, why);
}

void *spec_list_kernel(const HostModel &hm) {
    return hm.dev.S >= kListMinSpecies ? (void *)compiled(hm, kListBlock, Form::list, nullptr) : nullptr;
}

void *spec_block_kernel(const HostModel &hm, int block) {
    return hm.dev.S >= kListMinSpecies ? (void *)compiled(hm, block, Form::block, nullptr) : nullptr;
}

int launch_spec(void *spec, const ModelDev &m, const StepArgs &a, int block, void *stream) {
    if (a.T <= 0) return STEPS_OK;
    Compiled *c = static_cast<Compiled *>(spec);
    const void *fn = (const void *)c->kern;
    block = c->block;
    const size_t smem = c->smem;
    if (!opt_in(fn, smem, &c->smem_set)) return STEPS_ERR_CUDA;
    StepArgs b = a;
    if (c->form == Form::block) b.prefetch = prefetch_distance(fn, block, smem);
    void *args[2] = {(void *)&m, (void *)&b};
    const unsigned grid = (unsigned)(c->form == Form::list ? list_blocks(a.T, block) : (a.T + block - 1) / block);
    // programmatic dependent launch, as the generic step kernel
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e != cudaSuccess) {
        set_error(std::string("specialised step kernel launch: ") + cudaGetErrorString(e));
        return STEPS_ERR_CUDA;
    }
    return STEPS_OK;
}

int launch_spec_flow(void *spec, const ModelDev &m, const StepArgs &a, const FlowArgs &f, int block, void *stream) {
    if (a.T <= 0 || f.nwin == 0) return STEPS_OK;
    Compiled *c = static_cast<Compiled *>(spec);
    const void *fn = (const void *)c->kern_flow;
    const size_t smem = c->smem;
    if (!opt_in(fn, smem, &c->smem_set_flow)) return STEPS_ERR_CUDA;
    int per_sm = 0, dev = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem) != cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || per_sm < 1) {
        set_error("flow kernel occupancy: " + std::string(cudaGetErrorString(cudaGetLastError())));
        return STEPS_ERR_CUDA;
    }
    StepArgs b = a;
    b.window_base = nullptr;
    // block tiles: the item taken about half a resident wave later, its tables into L2
    b.prefetch = std::max(1, per_sm * sms / 2);
    void *args[3] = {(void *)&m, (void *)&b, (void *)&f};
    // one item per block, or the blocks resident at once
    const unsigned items = f.nwin * f.ntiles;
    const unsigned grid = c->form == Form::tiles && warp_flow_persists(block) ? std::min(items, (unsigned)(per_sm * sms)) : items;
    cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3((unsigned)block), args, smem, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        set_error(std::string("flow step kernel launch: ") + cudaGetErrorString(e));
        return STEPS_ERR_CUDA;
    }
    return STEPS_OK;
}

int launch_spec_batch_flow(void *spec, const BlockWork *work, RepEntry *reps, const FlowArgs &f, uint32_t work0,
                           int block, void *stream) {
    if (f.nwin == 0 || f.ntiles == 0) return STEPS_OK;
    if (!work) {
        set_error("specialised batched flow kernel launch: no work list");
        return STEPS_ERR_STATE;
    }
    Compiled *c = static_cast<Compiled *>(spec);
    const void *fn = (const void *)c->kern_batch_flow;
    const size_t smem = c->smem;
    if (!opt_in(fn, smem, &c->smem_set_batch_flow)) return STEPS_ERR_CUDA;
    void *args[4] = {(void *)&work, (void *)&reps, (void *)&f, (void *)&work0};
    const unsigned grid = f.nwin * f.ntiles;  // one item per block
    cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3((unsigned)block), args, smem, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        set_error(std::string("batched flow step kernel launch: ") + cudaGetErrorString(e));
        return STEPS_ERR_CUDA;
    }
    return STEPS_OK;
}

int launch_spec_batch(void *spec, const BlockWork *work, int64_t nblocks, RepEntry *reps, int block,
                      void *stream) {
    if (nblocks <= 0) return STEPS_OK;
    if (!work) {
        set_error("specialised batched step kernel launch: no work list");
        return STEPS_ERR_STATE;
    }
    Compiled *c = static_cast<Compiled *>(spec);
    const void *fn = (const void *)c->kern_batch;
    const size_t smem = c->smem;
    if (!opt_in(fn, smem, &c->smem_set_batch)) return STEPS_ERR_CUDA;
    block = c->block;
    int32_t prefetch = c->form == Form::block ? prefetch_distance(fn, block, smem) : 0;
    void *args[3] = {(void *)&work, (void *)&reps, (void *)&prefetch};  // (the last one: block tiles)
    cudaError_t e = cudaLaunchKernel(fn, dim3((unsigned)nblocks), dim3((unsigned)block), args, smem, (cudaStream_t)stream);
    if (e != cudaSuccess) {
        set_error(std::string("specialised batched step kernel launch: ") + cudaGetErrorString(e));
        return STEPS_ERR_CUDA;
    }
    return STEPS_OK;
}

}  // namespace steps
