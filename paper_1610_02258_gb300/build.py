"""Build the CUDA library in-tree: nvcc for sm_103a, one translation unit per
process in parallel, then a shared-library link. No floating-point
contraction in device or host code (-fmad=false, -ffp-contract=off)."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB_PATH = os.path.join(HERE, "libsteps_gpu.so")
SOURCES = ["steps_host.cpp", "steps_kernels.cu", "steps_warp.cu", "steps_batch.cu", "steps_api.cu", "steps_spec.cpp",
           "steps_server.cpp"]
# device sources embedded into the library for the run-time compiler (NVRTC)
EMBEDDED = [("kSrcDeviceH", "steps_device.h"), ("kSrcStepCuh", "steps_step.cuh"),
            ("kSrcWarpCuh", "steps_warp.cuh"), ("kSrcListCuh", "steps_list.cuh")]
EMBED_CPP = "steps_rtc_sources.cpp"
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _flags(verbose: bool):
    f = ["-O3", "-std=c++17", "-lineinfo", "-fmad=false", "-Xcompiler", "-fPIC,-ffp-contract=off,-O2",
         "-I", os.path.join(HERE, "..", "include")] + ARCH
    if verbose:
        f += ["-Xptxas", "-v"]
    return f


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(HERE, "..", "include", "steps_gpu.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps)


def _write_embedded() -> str:
    """A C++ file holding the device sources as string constants."""
    out = ["// Generated by build.py: the device sources the run-time compiler builds", "namespace steps {"]
    for name, fn in EMBEDDED:
        with open(os.path.join(CSRC, fn)) as f:
            text = f.read()
        if ")STEPSRTC\"" in text:
            raise RuntimeError(f"{fn} contains the raw-string delimiter")
        out.append(f'extern const char *const {name};\nconst char *const {name} = R"STEPSRTC({text})STEPSRTC";')
    out.append("}  // namespace steps\n")
    path = os.path.join(BUILD, EMBED_CPP)
    with open(path, "w") as f:
        f.write("\n".join(out))
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB_PATH
    os.makedirs(BUILD, exist_ok=True)
    embedded = _write_embedded()

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        lang = ["-x", "cu"] if src.endswith(".cu") else []
        path = src if os.path.isabs(src) else os.path.join(CSRC, src)
        cmd = [nvcc()] + _flags(verbose) + lang + ["-c", path, "-o", obj]
        p = subprocess.run(cmd, capture_output=True, text=True)
        if p.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{p.stderr}")
        if verbose:
            sys.stderr.write(p.stderr)
        return obj

    srcs = SOURCES + [embedded]
    with ThreadPoolExecutor(max_workers=len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs + ["-lcudart_static", "-lrt", "-lpthread", "-ldl"]
    p = subprocess.run(cmd, capture_output=True, text=True)
    if p.returncode != 0:
        raise RuntimeError(f"link failed:\n{p.stderr}")
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
