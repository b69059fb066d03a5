"""Build libfpt_gb300.so (the C-ABI CUDA library) in-tree for sm_103a.

Each translation unit is compiled by nvcc in parallel, then linked into
paper_2206_11234_gb300/libfpt_gb300.so.  The binary64 stepper and the RNG
probe are compiled with FMA contraction off so that their arithmetic is
rounded exactly as written in the source.

build(debug=True) builds the same sources with -DFPT_DEBUG=1 into
libfpt_gb300_debug.so: kernels whose bounds checks (parameter set of a
ticket, replay-queue capacity, record index, histogram bin index) record a
status bit and skip the access, reported by the call as FPT_EDEVICE_STATUS.
The binding loads it instead of the default library when the environment
variable FPT_DEBUG_LIB is 1.
"""
import concurrent.futures as cf
import math
import os
import shutil
import struct
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libfpt_gb300.so")
INCLUDE = os.path.join(ROOT, "include")

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# Device code uncompressed: a unit is unpacked as a whole at its first call, which cost a process 15 ms
# for a binary32 stepper and 11 ms for the binary64 one (a library of 29 MB; 92 without).
COMMON = ["-O3", "-lineinfo", "--no-compress", "-std=c++17", "-Xcompiler", "-fPIC", "-I" + INCLUDE, "-I" + CSRC]
UNITS = {
    "abi.cu": [],
    "histogram.cu": [],
    "stepper_f32_kahan.cu": [],
    "stepper_f32_f64acc.cu": [],
    "stepper_pow.cu": [],
    "stepper_f64.cu": ["-fmad=false", "-DFPT_STEPPER_MAXNREG=128"],
    "rng_probe.cu": ["-fmad=false"],
    "noalloc.cu": [],
    "autotune.cu": [],
    "mlp.cu": [],
    "stepper_mlp.cu": [],
    "train.cu": [],
    "plan.cu": [],
    "estimate.cu": [],
    "pipes.cu": [],
    "hist_merge.cu": [],
}


def f64_tables() -> str:
    """The binary64 Box–Muller tables of csrc/rng64.cuh, rounded correctly from
    200-bit integer arithmetic: cosines and sines of the 2^16 angles 2 pi u1 (the
    binary64 product), the logarithm's 2^-20-grained reciprocals with 2 ln(2 inv),
    and the multiples of 2 ln 2."""
    bits = 200
    one = 1 << bits

    def series(n, odd_sign):  # atan(1/n) (odd_sign -1) or atanh(1/n) (odd_sign 1)
        t = one // n
        s, k, sign = t, 1, 1
        while t:
            t //= n * n
            k += 2
            sign *= odd_sign
            s += sign * (t // k)
        return s

    pi = 4 * (4 * series(5, -1) - series(239, -1))  # Machin
    ln2 = 2 * series(3, 1)

    def cos_sin(x):
        out = [0, 0]
        t, k = one, 0
        while t:
            out[k % 2] += t if k % 4 < 2 else -t
            k += 1
            t = (t * x >> bits) // k
        return out

    def ln_ratio(a, b):  # ln(a / b) = 2 atanh((a - b) / (a + b)), 1 <= a / b <= 2
        z = (a - b) * one // (a + b)
        z2 = z * z >> bits
        s, t, k = 0, z, 1
        while t:
            s += t // k
            t = t * z2 >> bits
            k += 2
        return 2 * s

    c, s = cos_sin(pi >> 16)
    dc, ds = cos_sin(pi >> 15)
    trig = []
    for h in range(1 << 16):
        num, den = (6.283185307179586 * ((h + 0.5) / 65536)).as_integer_ratio()
        e = num * one // den - (pi * (2 * h + 1) >> 16)  # the rounded angle less the angle
        trig.append(((c - (s * e >> bits)) / one, (s + (c * e >> bits)) / one))  # int / int rounds correctly
        c, s = (c * dc - s * ds) >> bits, (s * dc + c * ds) >> bits
    log = []
    for i in range(1 << 10):
        inv = ((1 << 21) * (1 << 11) // (2 * (1 << 10) + 2 * i + 1) + 1) >> 1  # 2^20 / (1 + (i + 1/2)/1024), rounded
        if i == (1 << 10) - 1:
            inv = 1 << 19  # exactly 1/2 next to u0 = 1
        log.append((-2.0 * inv / (1 << 20), 2 * ln_ratio(inv, 1 << 19) / one))
    word = lambda x: "0x%xull" % struct.unpack("<Q", struct.pack("<d", x))  # noqa: E731
    pairs = lambda rows: ",".join("{%s,%s}" % (word(a), word(b)) for a, b in rows)  # noqa: E731
    return ("__device__ const ulonglong2 kTrig64[65536] = {%s};\n__device__ const ulonglong2 kLog64[1024] = {%s};\n"
            "__device__ const unsigned long long kLn2N64[33] = {%s};\n"
            % (pairs(trig), pairs(log), ",".join(word(2 * n * ln2 / one) for n in range(33))))


def exp_table() -> str:
    """The exponential's table of csrc/histogram.cu: 2^(-j/4096) in units of 2^-62, ln 2 / 4096
    in units of 2^-98 as three words, and 4096 / ln 2 in units of 2^-19."""
    bits = 200
    one = 1 << bits
    root = 2 * one
    for _ in range(12):
        root = math.isqrt(root * one)
    ln2, t, k = 0, 2 * one // 3, 1  # 2 atanh(1/3)
    while t:
        ln2 += t // k
        t //= 9
        k += 2
    step = ln2 >> 12
    x, table = one, []
    for _ in range(1 << 12):
        table.append(f"{(x >> (bits - 63)) + 1 >> 1}ull")
        x = x * one // root
    c = (step >> (bits - 99)) + 1 >> 1
    return ("__device__ const unsigned long long kExp62[4096] = {%s};\nconstexpr unsigned kExpStep2 = %du, "
            "kExpStep1 = %du, kExpStep0 = %du, kExpPerStep = %du;\n"
            % (",".join(table), c >> 64, c >> 32 & 0xffffffff, c & 0xffffffff, ((one << 19) + step // 2) // step))


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _inputs():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "fpt.h"))
    files.append(os.path.abspath(__file__))
    return files


LIB_DEBUG = os.path.join(HERE, "libfpt_gb300_debug.so")


def lib_path(debug: bool = False) -> str:
    return LIB_DEBUG if debug else LIB


def up_to_date(debug: bool = False) -> bool:
    lib = lib_path(debug)
    if not os.path.exists(lib):
        return False
    t = os.path.getmtime(lib)
    return all(os.path.getmtime(f) <= t for f in _inputs())


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib = lib_path(debug)
    if not force and up_to_date(debug):
        return lib
    build_dir = BUILD + ("_debug" if debug else "")
    os.makedirs(build_dir, exist_ok=True)
    with open(os.path.join(build_dir, "f64_tables.inc"), "w") as f:
        f.write(f64_tables())
    with open(os.path.join(build_dir, "exp_table.inc"), "w") as f:
        f.write(exp_table())
    cc = nvcc()
    extra = ["-DFPT_DEBUG=1"] if debug else []

    def compile_unit(name):
        obj = os.path.join(build_dir, name.replace(".cu", ".o"))
        cmd = [cc, *ARCH, *COMMON, "-I" + build_dir, *extra, *UNITS[name], "-c", os.path.join(CSRC, name), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {name}:\n{r.stderr}")
        return obj, r.stderr

    with cf.ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        results = list(ex.map(compile_unit, sorted(UNITS)))
    if verbose:
        for obj, log in results:
            print(obj, log, file=sys.stderr)
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *[o for o, _ in results]]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stderr}")
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv))
