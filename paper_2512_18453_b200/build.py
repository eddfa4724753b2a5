"""Build libnova.so in-tree with nvcc for sm_100a (no JIT, no torch extension)."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnova.so")
# named for this interpreter's ABI: another one does not import it and goes through ctypes
EXT = os.path.join(HERE, "_fastcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["plan.cpp", "transforms.cu", "filter_transform.cu", "gemm_simt.cu", "fp32_path.cu", "gemm_tcgen05.cu", "input_transform_tc.cu", "input_transform_n4.cu", "output_transform_tma.cu", "fabric_probe.cu", "fused_small_c.cu", "fused_fp32.cu", "product_output.cu", "few_tiles.cu", "conv.cu"]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def needs_build():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "fastcall.c"] + [os.path.join(ROOT, "include", "nova.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build_ext():
    """The CPython extension of the binding's hot calls; without headers of Python 3.9 or newer the binding uses ctypes."""
    src, inc = os.path.join(CSRC, "fastcall.c"), sysconfig.get_paths()["include"]
    untagged = os.path.join(HERE, "_fastcall.so")           # an earlier build's name, which any interpreter would import
    if untagged != EXT and os.path.exists(untagged):
        os.remove(untagged)
    if sys.version_info < (3, 9) or not os.path.exists(os.path.join(inc, "Python.h")):
        sys.stderr.write("no headers of Python 3.9 or newer in %s: calls go through ctypes\n" % inc)
        return
    newest = max(os.path.getmtime(f) for f in (src, os.path.join(ROOT, "include", "nova.h")))
    if not os.path.exists(EXT) or os.path.getmtime(EXT) < newest:
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"),
                               "-I", inc, src, "-o", EXT])


def build(force=False, verbose=False):
    """Compile every source for sm_100a and link the shared library."""
    build_ext()
    if not force and not needs_build():
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    common = [
        "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
        "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
    ]
    if verbose:
        common += ["-Xptxas", "-v"]
    procs = []
    objs = []
    # an object is rebuilt when its source, any header of csrc/ or the public header is newer
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    headers.append(os.path.join(ROOT, "include", "nova.h"))
    newest_header = max(os.path.getmtime(h) for h in headers)
    for src in SOURCES:
        obj = os.path.join(objdir, src.rsplit(".", 1)[0] + ".o")
        objs.append(obj)
        path = os.path.join(CSRC, src)
        if (not force and not verbose and os.path.exists(obj)
                and os.path.getmtime(obj) > max(os.path.getmtime(path), newest_header)):
            continue
        cmd = [_nvcc()] + common + ["-x", "cu", "-c", path, "-o", obj]
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write("[%s]\n%s\n" % (src, out))
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    cmd = [_nvcc(), "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static"]
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
