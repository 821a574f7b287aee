"""Build libcupso.so (the C-ABI library) in-tree with nvcc for sm_103a.

Each .cu file compiles to an object in parallel; the objects link into
paper_2205_01313_gb300/_build/libcupso.so. No cmake, no torch extension
machinery: the library is plain CUDA C++ behind `include/cupso.h`.
"""
import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libcupso.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

SOURCES = ["cupso_api.cu", "cupso_batch.cu", "cupso_lsq.cu", "kernels_state.cu", "kernels_stream.cu", "kernels_pipelined.cu",
           "kernels_batch.cu", "kernels_batch_panel.cu", "kernels_lsq.cu", "kernels_lsq_exact.cu", "kernels_lsq_swarm.cu", "kernels_onchip.cu",
           "kernels_paper.cu", "kernels_sync64.cu", "kernels_tiled.cu", "kernels_panel.cu", "kernels_resident.cu", "cupso_noalloc.cu"]
HEADERS = ["cupso_device.cuh", "cupso_internal.h", "stream_common.cuh", "paper_kernels.h", "tiled_kernels.h",
           "async_common.cuh", "pdl.cuh", "lsq_internal.h", "tma_common.cuh", "fit_terms.cuh", "fp64_common.cuh", "panel_common.cuh", "resident.h"]

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVFLAGS = ARCH + [
    "-O3", "-std=c++17", "-lineinfo",
    # exact IEEE float: no fused multiply-add contraction, IEEE division and sqrt
    "-fmad=false", "-prec-div=true", "-prec-sqrt=true", "-ftz=false",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-I" + INCLUDE,
]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libcupso.so")


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, ptxas_v: bool = False) -> str:
    os.makedirs(OUT, exist_ok=True)
    nv = nvcc()
    hdrs = [os.path.join(CSRC, h) for h in HEADERS] + [os.path.join(INCLUDE, "cupso.h"), __file__]
    objs = []
    jobs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(OUT, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + hdrs):
            cmd = [nv, *NVFLAGS, "-c", s, "-o", o]
            if ptxas_v:
                cmd.insert(1, "-Xptxas=-v")
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n%s\n%s%s" % (" ".join(cmd), r.stdout, r.stderr))
        return r.stdout + r.stderr

    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 1))) as ex:
        for out in ex.map(run, jobs):
            if verbose and out.strip():
                print(out)
    if force or jobs or _stale(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        r = subprocess.run([nv, *ARCH, "-shared", "-o", tmp, *objs], capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n%s%s" % (r.stdout, r.stderr))
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force="--force" in sys.argv, verbose=True, ptxas_v="-v" in sys.argv))
