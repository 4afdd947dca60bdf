"""Build the CUDA library libsdeb.so in-tree (paper_1908_03869_gb300/_build/).

Each translation unit under csrc/ is compiled for sm_103a only
(-gencode arch=compute_103a,code=sm_103a), in parallel, then linked into one
shared library with the CUDA runtime linked statically.  No cmake, no
architecture flags for the host compiler (the same command builds on x86_64
and aarch64 hosts).
"""
import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(HERE, "_build")
LIB_NAME = "libsdeb.so"
LIB_PATH = os.path.join(BUILD_DIR, LIB_NAME)
# The bounds-checked build: the same sources compiled with SDEB_CHECKED.
CHECKED_BUILD_DIR = os.path.join(HERE, "_build_checked")
CHECKED_LIB_PATH = os.path.join(CHECKED_BUILD_DIR, "libsdeb_checked.so")

GEN_DIR = os.path.join(BUILD_DIR, "gen")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
              "-I" + INCLUDE, "-I" + CSRC, "-I" + GEN_DIR]

# Device sources compiled again at run time for user-defined models (NVRTC):
# embedded into the library as string constants, one per file.
FIXED_INC = os.path.join(GEN_DIR, "sdeb_fixed_tables.inc")
RTC_EMBED = [("kRtcCheck", os.path.join(CSRC, "check.cuh")), ("kRtcFixedTables", FIXED_INC),
             ("kRtcFixedMath", os.path.join(CSRC, "fixed_math.cuh")),
             ("kRtcEmDevice", os.path.join(CSRC, "em_device.cuh")), ("kRtcArgs", os.path.join(CSRC, "rtc_args.h")),
             ("kRtcKernel", os.path.join(CSRC, "rtc_kernel.cuh"))]
RTC_INC = os.path.join(GEN_DIR, "sdeb_rtc_sources.inc")

# Working precision (bits) of the table generator below.
_BITS = 200


def _sincos_bits(num, den):
    """(cos, sin) of num/den in [0, 2), scaled by 2^_BITS: the Taylor series in integers."""
    x = (num << _BITS) // den
    c = s = k = 0
    term = 1 << _BITS
    while term:
        if k % 2 == 0:
            c += term if k % 4 == 0 else -term
        else:
            s += term if k % 4 == 1 else -term
        k += 1
        term = (term * x >> _BITS) // k
    return c, s


def _ln_bits(num, den):
    """ln(num/den) scaled by 2^_BITS: 2 atanh((num - den) / (num + den))."""
    z = ((num - den) << _BITS) // (num + den)
    total, term, k = 0, z, 1
    while term:
        total += term // k
        term = (term * z >> _BITS) * z >> _BITS
        k += 2
    return 2 * total


def _rounded(v, q):
    return (v + (1 << (_BITS - q - 1))) >> (_BITS - q)


def _pi_bits():
    """pi scaled by 2^_BITS (Machin: 16 atan(1/5) - 4 atan(1/239))."""
    def atan_inv(n):
        total, term, k = 0, (1 << _BITS) // n, 1
        while term:
            total += term // k if k % 4 == 1 else -(term // k)
            term //= n * n
            k += 2
        return total
    return 16 * atan_inv(5) - 4 * atan_inv(239)


def fixed_tables(step=(1, 256), rows=403, q_cos=62, q_sin=62, q_log=58, up=(2, 0)):
    """(cos, sin)(j step) in Q(q_cos) and Q(q_sin), j < rows, the cosines up[0] units up (of use where rows pass
    pi/2: a rotation's rounding then leaves none below 0), and (ln c, c), c in Q15 the largest with m c <= 1 for
    every m below (257 + j) / 512, ln c in Q(q_log), up[1] units up."""
    trig = []
    for j in range(rows):
        c, s = _sincos_bits(j * step[0], step[1])
        trig.append((_rounded(c, q_cos) + up[0], _rounded(s, q_sin)))
    log = []
    for j in range(256):
        c = (512 << 15) // (257 + j)
        log.append((_rounded(_ln_bits(c, 1 << 15), q_log) + up[1], c))
    return trig, log


def _write_if_changed(path, content):
    os.makedirs(os.path.dirname(path), exist_ok=True)
    if os.path.exists(path):
        with open(path) as f:
            if f.read() == content:
                return
    with open(path, "w") as f:
        f.write(content)


def generate_fixed_tables():
    parts = ["// Generated by build.py: tables of fixed_math.cuh.\n#pragma once\nnamespace sdeb {\n"]
    tables = fixed_tables((_pi_bits(), 4096 << _BITS), 1024, 63, 64, 64, (0, 2))
    for name, rows in zip(("kFixedTrig", "kFixedLog"), tables):
        parts.append("static __device__ const __align__(16) unsigned long long %s[%d][2] = {\n" % (name, len(rows)))
        parts += ["{0x%016xull, 0x%016xull},\n" % row for row in rows]
        parts.append("};\n")
    _write_if_changed(FIXED_INC, "".join(parts) + "}  // namespace sdeb\n")


def generate_rtc_sources():
    parts = ["// Generated by build.py from csrc/: the device sources of the run-time compiled kernel.\n"]
    for name, path in RTC_EMBED:
        with open(path) as f:
            text = f.read()
        if ")SDEBRTC" in text:
            raise RuntimeError("%s contains the raw-string delimiter" % path)
        parts.append('static const char %s[] = R"SDEBRTC(%s)SDEBRTC";\n' % (name, text))
    _write_if_changed(RTC_INC, "".join(parts))


def _nvcc():
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found")
    return cand


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return hs + [os.path.join(INCLUDE, "sdeb.h")]


def needs_build(checked=False):
    lib = CHECKED_LIB_PATH if checked else LIB_PATH
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(p) > t for p in sources() + headers() + [os.path.abspath(__file__)])


def _compile(src, verbose_ptxas=False, checked=False):
    obj = os.path.join(CHECKED_BUILD_DIR if checked else BUILD_DIR, os.path.basename(src)[:-3] + ".o")
    cmd = [_nvcc()] + ARCH + NVCC_FLAGS + (["-DSDEB_CHECKED=1"] if checked else []) + ["-c", src, "-o", obj]
    if verbose_ptxas:
        cmd += ["-Xptxas", "-v"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s" % (src, r.stderr))
    return obj, r.stderr


def build(force=False, verbose_ptxas=False, jobs=None, checked=False):
    """Build libsdeb.so, or with checked=True the bounds-checked
    libsdeb_checked.so (every kernel compiled with SDEB_CHECKED)."""
    lib = CHECKED_LIB_PATH if checked else LIB_PATH
    if not force and not needs_build(checked):
        return lib
    os.makedirs(CHECKED_BUILD_DIR if checked else BUILD_DIR, exist_ok=True)
    os.makedirs(GEN_DIR, exist_ok=True)
    generate_fixed_tables()
    generate_rtc_sources()
    srcs = sources()
    jobs = jobs or min(len(srcs), os.cpu_count() or 4)
    with concurrent.futures.ThreadPoolExecutor(max_workers=jobs) as ex:
        results = list(ex.map(lambda s: _compile(s, verbose_ptxas, checked), srcs))
    if verbose_ptxas:
        for _, log in results:
            sys.stderr.write(log)
    tmp = lib + ".tmp%d" % os.getpid()
    cmd = [_nvcc()] + ARCH + ["-shared", "-o", tmp] + [o for o, _ in results] + ["-cudart", "static", "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stderr)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose_ptxas="-v" in sys.argv, checked="--checked" in sys.argv))
