"""Build libacs.so in-tree with nvcc for sm_103a (translation units in parallel)."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libacs.so")
SOURCES = ["acs_api.cu", "acs_construct.cu", "acs_noalloc.cu", "acs_prior.cu", "acs_relaxed.cu"]
# the construct kernel, one translation unit per variant
VARIANT = "acs_construct_variant.cu"
# (memory, one CTA per instance, how lists are read)
VARIANTS = [(mode, alone, kind) for mode in (2, 1, 0) for alone in (0, 1) for kind in (2, 0)]
VARIANTS += [(mode, 0, 1) for mode in (0, 1, 2)]
HEADERS = ["acs_internal.cuh", "acs_device.cuh", "acs_construct.cuh", VARIANT]

NVCC_FLAGS = [
    "-gencode", "arch=compute_103a,code=sm_103a",
    "-lineinfo", "-O3", "-std=c++17",
    # IEEE FP32 without contraction: results must match the CPU oracle bit for bit
    "-fmad=false", "-prec-div=true", "-prec-sqrt=true", "-ftz=false",
    "-Xcompiler", "-fPIC,-ffp-contract=off",
    "-I" + os.path.join(ROOT, "include"), "-I" + CSRC,
]


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    deps.append(os.path.join(ROOT, "include", "acs.h"))
    deps.append(os.path.join(ROOT, "include", "acs_prior.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force=False, verbose=False):
    """Compile every translation unit and link libacs.so. Returns its path."""
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()
    procs = []
    objs = []
    units = [(VARIANT, "acs_construct_%d%d%d.o" % v,
              ["-DACS_MODE=%d" % v[0], "-DACS_ALONE=%d" % v[1], "-DACS_KIND=%d" % v[2]]) for v in VARIANTS]
    units += [(src, src.replace(".cu", ".o"), []) for src in SOURCES]
    for src, name, defines in units:
        obj = os.path.join(BUILD, name)
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, *defines, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    failed = []
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out.decode(errors="replace"))
        if p.returncode != 0:
            failed.append(" ".join(cmd))
    if failed:
        raise RuntimeError("nvcc failed:\n" + "\n".join(failed))
    tmp = LIB + ".tmp%d" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-o", tmp, *objs])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
