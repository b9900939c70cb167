"""Build the CUDA library libcwt_gb300.so in-tree for sm_103a.

Every .cu file under csrc/ is compiled in parallel with nvcc, with the device
headers of the plan-time compiler embedded as a generated jit_headers.cpp, then
linked into paper_2506_07793_gb300/_lib/libcwt_gb300.so (static CUDA runtime;
NVRTC from the toolkit, found through an rpath; the driver's module calls are
fetched at run time through the runtime).  Objects go
to paper_2506_07793_gb300/_build/.  A source is rebuilt when it, any header
under csrc/ or include/, or this file (the flags) is newer than its object.
"""
import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIBDIR = os.path.join(PKG, "_lib")
LIB = os.path.join(LIBDIR, "libcwt_gb300.so")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC,-O2",
              "-I", os.path.join(ROOT, "include")]


def nvcc():
    exe = shutil.which("nvcc")
    if exe:
        return exe
    cand = "/usr/local/cuda/bin/nvcc"
    if os.path.exists(cand):
        return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libcwt_gb300.so")


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h")) + [os.path.abspath(__file__)]


def _compile(src, extra, verbose, bdir=BUILD, defs=()):
    obj = os.path.join(bdir, os.path.basename(src) + ".o")
    newest_dep = max([os.path.getmtime(src)] + [os.path.getmtime(h) for h in _headers()])
    if os.path.exists(obj) and os.path.getmtime(obj) >= newest_dep and not extra:
        return obj, ""
    cmd = [nvcc()] + ARCH + NVCC_FLAGS + list(defs) + list(extra) + ["-c", src, "-o", obj + ".tmp"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    os.replace(obj + ".tmp", obj)
    return obj, (r.stdout + r.stderr) if verbose else ""


CHECK_LIB = os.path.join(LIBDIR, "libcwt_gb300_check.so")

# The device headers the plan-time compiler (csrc/jit.cu) builds kernels from;
# their text is embedded in the library as jit_headers.cpp.
JIT_HEADERS = ["smooth_device.cuh", "smooth_cluster_device.cuh", "dsmem.cuh", "mixed_radix.cuh",
               "fft_core.cuh", "check.cuh", "phase.cuh"]


def _jit_headers_source(bdir):
    """Write bdir/jit_headers.cpp (only when its text changes) and return its path."""
    out = ["// generated by build.py: the device headers of csrc/jit.cu's plan-time compiles",
           "extern \"C\" {"]
    names, texts = [], []
    for i, h in enumerate(JIT_HEADERS):
        with open(os.path.join(CSRC, h)) as f:
            text = f.read()
        delim = "cwtjit"
        while (")" + delim + '"') in text:
            delim += "x"
        out.append(f'static const char cwt_jit_text_{i}[] = R"{delim}({text}){delim}";')
        names.append(f'"{h}"')
        texts.append(f"cwt_jit_text_{i}")
    out.append(f"extern const int cwt_jit_header_count = {len(JIT_HEADERS)};")
    out.append("extern const char *const cwt_jit_header_names[] = {" + ", ".join(names) + "};")
    out.append("extern const char *const cwt_jit_header_texts[] = {" + ", ".join(texts) + "};")
    out.append("}")
    src = "\n".join(out) + "\n"
    path = os.path.join(bdir, "jit_headers.cpp")
    old = None
    if os.path.exists(path):
        with open(path) as f:
            old = f.read()
    if old != src:
        with open(path, "w") as f:
            f.write(src)
    return path


def _cuda_lib_dir():
    """The CUDA toolkit's library directory (NVRTC)."""
    root = os.path.dirname(os.path.dirname(os.path.realpath(nvcc())))
    cands = [os.path.join(root, "lib64")] + sorted(glob.glob(os.path.join(root, "targets", "*", "lib")))
    return next((d for d in cands if glob.glob(os.path.join(d, "libnvrtc.so*"))), cands[0])


def build(force=False, verbose=False, extra_flags=(), check=False):
    """Compile and link; returns the library path.

    check=True builds the bounds-checked variant (-DCWT_BOUNDS_CHECK, see
    csrc/check.cuh) into _lib/libcwt_gb300_check.so, objects in _build_check/;
    load it by setting CWT_GB300_LIB to its path before importing the package."""
    bdir = BUILD + "_check" if check else BUILD
    lib = CHECK_LIB if check else LIB
    os.makedirs(bdir, exist_ok=True)
    os.makedirs(LIBDIR, exist_ok=True)
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu"))) + [_jit_headers_source(bdir)]
    if force:
        for o in glob.glob(os.path.join(bdir, "*.o")):
            os.remove(o)
    extra = list(extra_flags) + (["-Xptxas", "-v"] if verbose else [])
    # The checked variant's device code is compressed (library 232 -> 32 MB): with
    # both builds and their objects the tree passed 700 MB, too much to ship.  The
    # ordinary one is not: unpacking would add 17 ms to a process's first call.
    defs = ["-DCWT_BOUNDS_CHECK", "--compress-mode=size"] if check else []
    with cf.ThreadPoolExecutor(max_workers=min(len(srcs), os.cpu_count() or 4)) as ex:
        results = list(ex.map(lambda s: _compile(s, extra, verbose, bdir, defs), srcs))
    objs = [o for o, _ in results]
    if verbose:
        for _, log in results:
            if log:
                print(log)
    if (not os.path.exists(lib) or force or extra
            or max(os.path.getmtime(o) for o in objs) > os.path.getmtime(lib)):
        tmp = lib + f".tmp{os.getpid()}"
        cuda_lib = _cuda_lib_dir()
        cmd = [nvcc()] + ARCH + ["-shared", "-o", tmp] + objs + [
            "-L" + cuda_lib, "-lnvrtc", "-lpthread", "-Xlinker", "-rpath", "-Xlinker", cuda_lib]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, check="--check" in sys.argv))
