"""Build the CUDA library in-tree for sm_103a (GB300).

Compiles every csrc/*.cu translation unit with nvcc in parallel and links
_build/libgb300lobpcg.so against cuBLAS and cuSOLVER.  Run as
`python -m paper_1704_07458_gb300.build` or call build().
"""
import concurrent.futures as cf
import glob
import os
import re
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libgb300lobpcg.so")
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-fvisibility=hidden",
         "--expt-relaxed-constexpr"]


def _nvcc():
    for cand in [os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")]:
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _cuda_lib_dir(nvcc):
    root = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    for d in ["lib64", "lib", "targets/sbsa-linux/lib", "targets/x86_64-linux/lib"]:
        p = os.path.join(root, d)
        if os.path.exists(os.path.join(p, "libcusolver.so")):
            return p
    return os.path.join(root, "lib64")


# Kernels whose warps share out the registers of the launch among themselves
# (setmaxnreg): built with another count than the constant in their source says,
# their launches would wait for shares that never come free, so the library
# refuses them at run time.  (source, constant, kernels)
REGISTER_SHARES = [("ozaki_tc.cu", "kURegs", r"ozaki_(gram|update)_tc_kernel")]


def check_registers(src, log):
    """Raise when ptxas -v's output shows such a kernel with another count."""
    for name, const, kernels in REGISTER_SHARES:
        if os.path.basename(src) != name:
            continue
        want = int(re.search(rf"\b{const} = (\d+)", open(src).read()).group(1))
        found = [(f, int(r)) for f, r in
                 re.findall(r"Compiling entry function '(\w+)'.*?Used (\d+) registers", log, re.S)
                 if re.search(kernels, f)]
        bad = [f"{f}: {r}" for f, r in found if r != want]
        if bad or not found:
            raise RuntimeError(f"{name}: {const} = {want} registers a thread, but ptxas gave "
                               f"{', '.join(bad) or 'no kernel'}")


def build(verbose=False, extra=()):
    nvcc = _nvcc()
    os.makedirs(OUT, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(HERE, "..", "include", "*.h"))
    newest_hdr = max(os.path.getmtime(h) for h in headers)

    def compile_one(src):
        obj = os.path.join(OUT, os.path.basename(src)[:-3] + ".o")
        if (os.path.exists(obj) and os.path.getmtime(obj) > os.path.getmtime(src)
                and os.path.getmtime(obj) > newest_hdr):
            return obj
        usage = ["-Xptxas", "-v"] * any(os.path.basename(src) == s for s, _, _ in REGISTER_SHARES)
        cmd = [nvcc, *ARCH, *FLAGS, *usage, *extra, "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        try:
            check_registers(src, r.stdout + r.stderr)
        except RuntimeError:
            os.remove(obj)
            raise
        if verbose and (r.stdout or r.stderr):
            print(r.stdout, r.stderr, file=sys.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, len(srcs))) as ex:
        objs = list(ex.map(compile_one, srcs))
    libdir = _cuda_lib_dir(nvcc)
    if (not os.path.exists(LIB)
            or max(os.path.getmtime(o) for o in objs) > os.path.getmtime(LIB)):
        cmd = [nvcc, *ARCH, "-shared", "-o", LIB, *objs, f"-L{libdir}", "-lcusolver",
               "-lcublas", "-lcudart", f"-Xlinker=-rpath,{libdir}"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    return LIB


if __name__ == "__main__":
    print(build(verbose=True))
