"""The library's own rules of which CTA of the fused attention does what (``csrc/baps_tile_order.cuh``), compiled as
plain C++ for the tests that have to know which form of the kernel a call takes."""
import ctypes
import functools
import os
import subprocess
import tempfile

from paper_2602_02071_b200 import build

SHIM = r"""
#include "baps_tile_order.cuh"
using namespace baps;
extern "C" int one_tile(long long heads, int nq, int causal, int sms) { return one_tile_per_cta(heads, nq, causal, sms); }
extern "C" int two_ctas(long long heads, int nq, int causal, int sms) { return two_ctas_per_sm(heads, nq, causal, sms); }
extern "C" void chunks(long long kv, long long bytes, long long per_kv, int causal, int sms, int per_sm, int *out)
{ const KvChunks c = kv_chunks(kv, bytes, per_kv, causal, sms, per_sm); out[0] = c.size; out[1] = c.wide; }
extern "C" void items(int H, int Hkv, int npairs, int size, int wide, int n, int *out)
{
    const KvChunks c = {size, wide};
    for (int i = 0; i < n; ++i) {
        const WorkItem w = work_item(H, Hkv, npairs, c, i);
        out[4 * i] = w.tile; out[4 * i + 1] = w.h; out[4 * i + 2] = w.hk; out[4 * i + 3] = w.b;
    }
}
"""
SMS = 148


@functools.lru_cache(maxsize=None)
def lib():
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "shim.cpp"), os.path.join(d, "shim.so")
        with open(src, "w") as f:
            f.write(SHIM)
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", build.CSRC, "-o", so, src], check=True)
        out = ctypes.CDLL(so)
    ll, i = ctypes.c_longlong, ctypes.c_int
    out.one_tile.argtypes = out.two_ctas.argtypes = [ll, i, i, i]
    out.chunks.argtypes = [ll, ll, ll, i, i, i, ctypes.POINTER(i)]
    out.items.argtypes = [i, i, i, i, i, i, ctypes.POINTER(i)]
    return out


def one_tile_per_cta(heads, nq, causal):
    return bool(lib().one_tile(heads, nq, causal, SMS))


def two_ctas_per_sm(heads, nq, causal):
    return bool(lib().two_ctas(heads, nq, causal, SMS))


def form(D, heads, nq, causal):
    """Form of the kernel that the usual call (Algorithm 1, B0 = the first tile) takes."""
    if D == 64:
        return "two CTAs per SM" if two_ctas_per_sm(heads, nq, causal) else "one tile"
    return "one tile" if one_tile_per_cta(heads, nq, causal) else "two tiles"


def tiles(B, H, Hkv, npairs, kv_bytes, causal, per_sm, whole=False):
    """((chunk size, chunks of one more), [(tile, h, hk, b) of every CTA in launch order])"""
    c = (ctypes.c_int * 2)(B * Hkv, 0)
    if not whole:
        lib().chunks(B * Hkv, kv_bytes, npairs * (H // Hkv), causal, SMS, per_sm, c)
    n = B * H * npairs
    out = (ctypes.c_int * (4 * n))()
    lib().items(H, Hkv, npairs, c[0], c[1], n, out)
    return (c[0], c[1]), [tuple(out[4 * k:4 * k + 4]) for k in range(n)]
