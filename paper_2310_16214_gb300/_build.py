"""Build the in-tree C-ABI library libbplg.so for sm_103a with nvcc.

Every translation unit under csrc/ is compiled in parallel with
``-gencode arch=compute_103a,code=sm_103a`` and linked into
``paper_2310_16214_gb300/_lib/libbplg.so`` (CUDA runtime linked statically).
The benchmark's external references (extref/extref.cu: CUB, cuFFT, cuSPARSE)
go into a separate ``_lib/libbplg_extref.so`` that the library never loads.
"""
from __future__ import annotations

import concurrent.futures as cf
import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OUT_DIR = os.path.join(HERE, "_lib")
OBJ_DIR = os.path.join(OUT_DIR, "obj")
LIB = os.path.join(OUT_DIR, "libbplg.so")
EXTREF_SRC = os.path.join(HERE, "extref", "extref.cu")
EXTREF_LIB = os.path.join(OUT_DIR, "libbplg_extref.so")

GEN_DIR = os.path.join(OUT_DIR, "gen")
NOALLOC_TABLE = os.path.join(GEN_DIR, "noalloc_twiddles.inc")
NOALLOC_MAX_LOG = 12  # the no-alloc FFT entry point's table holds the roots of unity of order M <= 4096

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
         "-I" + INCLUDE, "-I" + CSRC, "-I" + GEN_DIR]


def _sincospi(t: float):
    """(sin(pi t), cos(pi t)) in float64 for a dyadic t, with the argument
    reduced exactly: t = r + f, r a multiple of 1/2 and |f| <= 1/4, then a
    rotation by the quarter turns in r (so multiples of pi/2 give exact 0 and
    +-1)."""
    import math
    r = round(2.0 * t) / 2.0
    f = t - r  # exact: t is dyadic
    s0, c0 = math.sin(math.pi * f), math.cos(math.pi * f)
    q = int(round(2.0 * r)) % 4
    return [(s0, c0), (c0, -s0), (-s0, -c0), (-c0, s0)][q]


def write_noalloc_table() -> str:
    """Write the static initializer of the no-alloc FFT entry point's twiddle
    array, for M = 2, 4, ..., 2^NOALLOC_MAX_LOG the two blocks of M entries
    described in csrc/fft_common.cuh: W_M^e = exp(-2 pi i e / M) at [2 M + e]
    and, for M >= 16, W_M^(r k) at [3 M + r M / 16 + k] (1 in the unused
    places), in float64, rounded once to float32, as hexadecimal
    float literals.  The file is rewritten only when its text changes."""
    import struct
    total = 4 << NOALLOC_MAX_LOG

    def f32(v: float) -> str:
        r = struct.unpack("<f", struct.pack("<f", v))[0]  # round to nearest float32
        return (r.hex() if r != 0.0 else ("-0x0p+0" if math.copysign(1.0, r) < 0 else "0x0p+0")) + "f"

    import math
    lines = ["// generated by _build.py: W_M^e at [2 M + e], stage blocks at [3 M ..], M = 2 .. %d, float64 rounded to float32"
             % (1 << NOALLOC_MAX_LOG)]
    for i in range(total):
        M = 1 << (i.bit_length() - 2) if i >= 4 else 1
        k = i - 2 * M
        if M < 2 or (k >= M and M < 16):
            c, s_ = 1.0, 0.0
        else:
            if k >= M:
                r, kk = divmod(k - M, M // 16)
                k = r * kk
            s_, c = _sincospi(-2.0 * k / M)
        lines.append("{%s, %s}," % (f32(c), f32(s_)))
    text = "\n".join(lines) + "\n"
    os.makedirs(GEN_DIR, exist_ok=True)
    old = open(NOALLOC_TABLE).read() if os.path.exists(NOALLOC_TABLE) else None
    if old != text:
        with open(NOALLOC_TABLE + ".tmp", "w") as f:
            f.write(text)
        os.replace(NOALLOC_TABLE + ".tmp", NOALLOC_TABLE)
    return NOALLOC_TABLE


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _headers():
    return glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(INCLUDE, "*.h")) + glob.glob(os.path.join(GEN_DIR, "*.inc"))


def _compile(src: str, verbose_ptxas: bool) -> str:
    obj = os.path.join(OBJ_DIR, os.path.basename(src) + ".o")
    if _stale(obj, [src] + _headers()):
        cmd = [nvcc()] + ARCH + FLAGS + ["-c", src, "-o", obj + ".tmp"]
        if verbose_ptxas:
            cmd += ["-Xptxas", "-v"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed on %s:\n%s" % (src, r.stderr[-8000:]))
        if verbose_ptxas:
            with open(obj + ".ptxas.txt", "w") as f:
                f.write(r.stderr)
        os.replace(obj + ".tmp", obj)
    return obj


def _build_extref() -> str:
    if _stale(EXTREF_LIB, [EXTREF_SRC]):
        cuda_inc = os.path.join(os.path.dirname(os.path.dirname(nvcc())), "include")
        tmp = EXTREF_LIB + ".tmp.%d" % os.getpid()
        cmd = [nvcc()] + ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                                 "-I" + os.path.join(cuda_inc, "cccl"), EXTREF_SRC, "-o", tmp,
                                 "-lcufft", "-lcusparse"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("extref build failed:\n" + r.stderr[-8000:])
        os.replace(tmp, EXTREF_LIB)
    return EXTREF_LIB


def build(verbose_ptxas: bool = False, jobs: int = 0) -> str:
    os.makedirs(OBJ_DIR, exist_ok=True)
    write_noalloc_table()
    srcs = sources()
    jobs = jobs or min(len(srcs), os.cpu_count() or 4)
    with cf.ThreadPoolExecutor(max_workers=jobs + 1) as ex:
        ext = ex.submit(_build_extref)
        objs = list(ex.map(lambda s: _compile(s, verbose_ptxas), srcs))
        ext.result()
    if _stale(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        cmd = [nvcc()] + ARCH + ["-shared", "-Xcompiler", "-fPIC", "-o", tmp] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("link failed:\n" + r.stderr[-8000:])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose_ptxas="-v" in sys.argv))
