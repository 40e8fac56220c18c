"""The host rules that pick a kernel form (csrc/plans.h), for the tests: compiled as plain C++ and called through ctypes, so that
a test can say which form its shape takes."""
import ctypes
import functools
import os
import subprocess
import tempfile
from collections import namedtuple

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_WRAPPER = r"""
#include "%s/paper_2412_14363_b200/csrc/plans.h"
using namespace resq;
extern "C" {
void mid(int T, int N, int kbt, int* o) { MidPlan p = mid_plan(T, N, kbt); o[0] = p.use; o[1] = p.ntok; o[2] = p.tok_tiles; o[3] = p.splits; }
int together(int d, int kv_tiles, int tiles) { return append_tiles_together(d, kv_tiles, tiles); }
int few(int T, int K) { return quantizes_rows(T, K); }
int meet(size_t a, size_t an, size_t b, size_t bn) { return ranges_meet((const void*)a, an, (const void*)b, bn); }
int gptq(int N, int K) { return gptq_rows_per_cta(N, K); }
void prefill(int pos0, int T, int g, int Hkv, int d, int* o) {
    PrefillPlan p = prefill_plan(pos0, T, g, Hkv, d); o[0] = p.tiles_per_cta; o[1] = p.splits; o[2] = (int)p.row_groups; o[3] = p.pair; }
void rows64(int rows, int Hkv, int capacity, int* o) {
    Attn64Plan p = attention64_rows_plan(rows, Hkv, capacity); o[0] = p.warps; o[1] = p.splits; o[2] = p.pack; o[3] = p.short_steps; o[4] = (int)p.ctas; }
}
"""
Mid = namedtuple("Mid", "use ntok tok_tiles splits")
Prefill = namedtuple("Prefill", "tiles_per_cta splits row_groups pair")
Attn64 = namedtuple("Attn64", "warps splits pack short_steps ctas")


@functools.lru_cache(None)
def _lib():
    d = tempfile.mkdtemp()
    src, so = os.path.join(d, "plans.cpp"), os.path.join(d, "plans.so")
    with open(src, "w") as f:
        f.write(_WRAPPER % ROOT)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", src, "-o", so], check=True)
    return ctypes.CDLL(so)


def _call(fn, kind, *args):
    out = (ctypes.c_int * len(kind._fields))()
    getattr(_lib(), fn)(*args, out)
    return kind(*out)


def k_blocks(K, r):
    return (r + 127) // 128 + (K - r + 127) // 128


def mid(T, K, N, r):
    """The plan of the mixed GEMM at T > 16: use = 0 means the large-tile kernel."""
    return _call("mid", Mid, T, N, k_blocks(K, r))


def gptq_rows(N, K):
    return _lib().gptq(N, K)


def quantizes_rows(T, K):
    return _lib().few(T, K)


def ranges_meet(a, a_bytes, b, b_bytes):
    return bool(_lib().meet(*(ctypes.c_size_t(v) for v in (a, a_bytes, b, b_bytes))))


def append_together(d, T, Hq, Hkv):
    kv_tiles = 2 * -(-T // 16) * Hkv
    return bool(_lib().together(d, kv_tiles, kv_tiles + -(-T * Hq // 16)))


def prefill(pos0, T, Hq, Hkv, d=128):
    return _call("prefill", Prefill, pos0, T, Hq // Hkv, Hkv, d)


def rows64(rows, Hkv, capacity):
    return _call("rows64", Attn64, rows, Hkv, capacity)
