"""Builds libquads.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _native.so, the binding's ordinary calls
as native functions on top of it."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libquads.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_SOURCE = os.path.join(CSRC, "native.cpp")
SOURCES = ["api.cu", "quantize.cu", "front.cu", "small_batch.cu", "gemm.cu", "gemm_dense.cu", "gemm_swapped.cu", "gemm_bf16.cu", "fp8.cu", "probe.cu"]
HEADERS = ["common.cuh", "kernels.cuh", "routing.cuh", "select.cuh", "split_k.cuh", "tcgen05.cuh", os.path.join("..", "..", "include", "quads.h")]


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _older(target, deps):
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def native_tag():
    """What _native.so has to have been compiled for: it reads torch's C++ objects through inline code, so another torch or Python may
    load it (its symbols resolve) and then read wrong memory.  None without torch."""
    try:
        import torch
    except ImportError:
        return None
    return "torch %s, CUDA %s, cxx11 ABI %d, %s" % (torch.__version__, torch.version.cuda, int(torch._C._GLIBCXX_USE_CXX11_ABI),
                                                    sysconfig.get_config_var("SOABI"))


def native_matches():
    """Whether the built _native.so carries this process's tag, without loading it."""
    tag = native_tag()
    if tag is None or not os.path.exists(NATIVE):
        return False
    with open(NATIVE, "rb") as f:
        return ("built for " + tag + "\0").encode() in f.read()


def needs_build():
    return _older(LIB, [os.path.join(CSRC, s) for s in SOURCES + HEADERS])


def _without_native(why):
    """The binding does without _native.so; an object of older sources must not be what it finds."""
    if os.path.exists(NATIVE):
        os.remove(NATIVE)
    sys.stderr.write("_native.so is not built (%s): the ordinary calls go through ctypes, at more host time each\n" % why)


def _start_native():
    """The compiler of _native.so and the link behind it, or None where something that it needs is missing."""
    try:
        import torch
        from torch.utils import cpp_extension
    except ImportError as e:
        return _without_native(e)
    lib_dir = os.path.join(os.path.dirname(torch.__file__), "lib")
    if torch.version.cuda is None or not os.path.exists(os.path.join(lib_dir, "libc10_cuda.so")):
        return _without_native("a torch without CUDA")
    cuda_include = os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include") if os.path.isabs(_nvcc()) else "/usr/local/cuda/include"
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-c", NATIVE_SOURCE, "-o", os.path.join(CSRC, "native.o"),
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DQUADS_NATIVE_TAG="%s"' % native_tag()]
    for d in cpp_extension.include_paths() + [sysconfig.get_paths()["include"], cuda_include]:
        cmd += ["-isystem", d]
    link = ["g++", "-shared", "-o", NATIVE, os.path.join(CSRC, "native.o"), "-L" + HERE, "-l:libquads.so", "-Wl,-rpath,$ORIGIN",
            "-L" + lib_dir, "-Wl,-rpath," + lib_dir, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    try:
        return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True), link
    except OSError as e:
        return _without_native(e)


def _finish_native(compiler, link):
    out, _ = compiler.communicate()
    if compiler.returncode == 0:
        done = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if done.returncode == 0:
            return
        out += done.stdout
    sys.stderr.write(out)
    _without_native("g++ failed")


def build(force=False, verbose=False):
    """libquads.so, and where this machine has what it takes _native.so."""
    native = None
    if force or not native_matches() or _older(NATIVE, [NATIVE_SOURCE, os.path.join(CSRC, HEADERS[-1])]):
        native = _start_native()
    if force or needs_build():
        _build_lib(verbose)
    if native is not None:
        _finish_native(*native)
    return LIB


def _build_lib(verbose):
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
               "-Xcompiler", "-fPIC", "-Xptxas", "-v" if verbose else "-O3", "-c",
               os.path.join(CSRC, src), "-o", obj] + os.environ.get("QUADS_NVCC_FLAGS", "").split()
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError("nvcc failed on %s" % src)
    cmd = [_nvcc(), "-shared", "-o", LIB] + objs + ["-lcudart_static", "-ldl", "-lrt", "-lpthread"]
    subprocess.check_call(cmd)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
