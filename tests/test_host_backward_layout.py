"""Launch layout of the backprojector, checked on the CPU with the library's own host code.

* backward_layout chooses tile, views per stage and staged rows; for every geometry spdhg_create admits
  (vx / d_radial up to 9.1, up to 256 slices) the pair lists stay within the 48 KB a kernel has by
  default and the whole launch within the limit of k_backward.
* Its staged rows and candidate bins cover every bin whose lines cross a pixel of the tile, by
  brute force over the kernel's FP32 formulas and the exact footprints.
* An item's record word names its kind and the staged slots of its lanes for components whose planes lie
  inside, across and wholly outside the image's slices.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1808_07150_gb300 import _build_ext

HELPER = r"""
#include "backward.cuh"
using namespace spdhg;
// in: nx ny nz V m bins taps R; seg_n[n_seg]; comps (seg, qlo, qhi, smask); out: cpw rows cand views batches, most
// bytes of the pair lists and of a launch, margin in 2^-40 bins
extern "C" void layout(const int* in, float inv, int n_seg, const int* seg_n, int n_comp, const int* comps, long long* out) {
  DevGeom g{};
  g.nx = in[0], g.ny = in[1], g.nz = in[2], g.V = in[3], g.m = in[4], g.bins = in[5], g.taps = in[6], g.R = in[7];
  g.inv_drp = inv, g.n_seg = n_seg, g.n_comp = n_comp;
  std::vector<SegDev> seg(n_seg);
  std::vector<CompDev> comp(n_comp);
  for (int k = 0, p = 0; k < n_seg; p += seg_n[k++]) seg[k] = SegDev{p, seg_n[k], 0.f, 0.f, 0, 0};
  for (int c = 0; c < n_comp; ++c)
    comp[c] = CompDev{comps[4 * c], comps[4 * c + 1], comps[4 * c + 2], comps[4 * c + 3], 0, 0, 0, 0};
  std::vector<int2> slots;
  std::vector<BwdBatch> batches;
  backward_layout(g, seg.data(), comp.data(), slots, batches);
  const int words = (g.nz + 31) / 32, zk = words <= 4 ? words : 8;
  out[0] = g.bw_cpw, out[1] = g.bw_rows, out[2] = g.bw_cand, out[3] = g.bw_views, out[4] = g.bw_nb;
  out[5] = (long long)bwd_pair_bytes(g);
  out[6] = (long long)bwd_smem(g, g.taps, zk, false, false, g.bw_step2);
  out[7] = kBwdMaxSmem;
  out[8] = llrint(ldexp((double)g.bw_margin, 40));
}
extern "C" unsigned word(int row_slot, int* jp, int* len, int taps, int lanes, int pad, int step2) {
  return item_word(row_slot, *jp, *len, taps, lanes, pad, step2 != 0);
}
"""


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    lib = _build_ext.build()
    d = tmp_path_factory.mktemp("layout")
    src, so = str(d / "layout.cu"), str(d / "layout.so")
    with open(src, "w") as f:
        f.write(HELPER)
    subprocess.run([_build_ext._nvcc(), *_build_ext.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    "-shared", "-I", _build_ext.CSRC, src, lib, "-o", so,
                    "-Xlinker", f"-rpath={os.path.dirname(lib)}"], check=True, capture_output=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def layout(helper):
    fn = helper.layout

    def run(nx, ny, nz, inv, views, subsets, taps, seg_n, comps, bins=0, radial=0):
        a = lambda v: np.ascontiguousarray(v, np.int32).ctypes.data_as(ctypes.POINTER(ctypes.c_int))
        head, sn, cm, out = [np.ascontiguousarray(v, np.int32) for v in
                             ([nx, ny, nz, views, subsets, bins, taps, radial or int(1.5 * max(nx, ny) * inv) + 3], seg_n, comps)] + [np.zeros(9, np.int64)]
        fn(a(head), ctypes.c_float(inv), len(sn), a(sn), len(cm), a(cm), out.ctypes.data_as(ctypes.POINTER(ctypes.c_longlong)))
        return dict(zip(("cpw", "rows", "cand", "views", "batches", "pairs", "smem", "limit", "margin"), out.tolist()))

    return run


def test_every_admitted_geometry_fits_its_launches(layout):
    rng = np.random.default_rng(0)
    worst = 0
    for k in range(4000):
        nx, ny = (int(v) for v in np.exp(rng.uniform(0, np.log(400), 2)))
        nz, taps = int(np.exp(rng.uniform(0, np.log(256.9)))), int(rng.integers(1, 5))
        inv = float(rng.choice([0.5, 1, 1.5, 2.2, 3, 4, 6, 9.1]))
        views = int(np.exp(rng.uniform(0, np.log(400))))
        seg_n = [int(v) for v in np.exp(rng.uniform(0, np.log(2 * nz), int(rng.integers(1, 6))))]
        comps = [(s, 0, n, 0) for s, n in enumerate(seg_n)]
        if k % 3 == 0:
            for s, n in enumerate(seg_n):
                comps += [(s, int(rng.integers(0, n)), n, 1)] * int(rng.integers(0, 3))
            comps.sort(key=lambda c: c[0])
        L = layout(nx, ny, nz, inv, views, int(rng.integers(1, views + 1)), taps, seg_n, comps, int(rng.integers(0, 2)))
        assert L["pairs"] <= 48 * 1024, (nx, ny, nz, inv, views)
        assert L["smem"] <= L["limit"], (nx, ny, nz, inv, views, taps, seg_n)
        worst = max(worst, L["pairs"])
    assert worst > 40 * 1024  # the bound is reached


@pytest.mark.parametrize("inv", [0.4, 1.0, 3.0, 9.1])
@pytest.mark.parametrize("n", [(344, 344), (171, 130), (23, 37)])
def test_staged_rows_and_candidates_cover_every_footprint(layout, n, inv):
    f = np.float32
    nx, ny = n
    L = layout(nx, ny, 4, inv, 24, 2, 1, [4], [(0, 0, 4, 0)])
    margin = f(math.ldexp(L["margin"], -40))
    assert L["cpw"] == (4 if nx > 100 else 1)
    TX, TY = 2 * L["cpw"], 4
    R = int(1.5 * max(n) * inv) + 3
    iv, half = f(inv), f(0.5 * (R - 1))
    ix, iy = (v.ravel() for v in np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij"))
    tx0, ty0 = ix // TX * TX, iy // TY * TY
    for v in range(24):
        c, s = math.cos(math.pi * v / 24), math.sin(math.pi * v / 24)
        c, s = 0.0 if abs(c) < 1e-12 else c, 0.0 if abs(s) < 1e-12 else s
        cf, sf = f(c), f(s)
        # the kernel's rows of the tile and candidates of the pixel
        mid = (f(1) * tx0.astype(f) + f(0.5 * TX) - f(0.5 * nx)) * cf + (ty0.astype(f) + f(0.5 * TY) - f(0.5 * ny)) * sf
        hwt = f(0.5) * (f(TX) * abs(cf) + f(TY) * abs(sf))
        r_min = np.maximum(0, np.ceil((mid - hwt) * iv + half - f(2) * margin)).astype(int)
        r_max = np.minimum(np.minimum(R - 1, r_min + L["rows"] - 1), np.floor((mid + hwt) * iv + half + f(2) * margin)).astype(int)
        hw = f(0.5) * (abs(cf) + abs(sf))
        sc = (ix.astype(f) + f(0.5) - f(0.5 * nx)) * cf + (iy.astype(f) + f(0.5) - f(0.5 * ny)) * sf
        lo = np.ceil((sc - hw) * iv + half - margin).astype(int)
        hi = np.minimum(np.floor((sc + hw) * iv + half + margin).astype(int), lo + L["cand"] - 1)
        # the bins whose line meets the pixel in more than a point
        s64, hw64 = (ix + 0.5 - 0.5 * nx) * c + (iy + 0.5 - 0.5 * ny) * s, 0.5 * (abs(c) + abs(s))
        e_lo = np.maximum(0, np.ceil((s64 - hw64) * inv + 0.5 * (R - 1) + 1e-9)).astype(int)
        e_hi = np.minimum(R - 1, np.floor((s64 + hw64) * inv + 0.5 * (R - 1) - 1e-9)).astype(int)
        some = e_lo <= e_hi
        assert (np.maximum(lo, r_min)[some] <= e_lo[some]).all()
        assert (np.minimum(hi, r_max)[some] >= e_hi[some]).all()


@pytest.mark.parametrize("step2", [0, 1])
@pytest.mark.parametrize("lanes", [32, 96, 256])
def test_record_words_name_their_kind_and_slots(helper, lanes, step2):
    helper.word.restype = ctypes.c_uint
    b = np.arange(lanes)
    for pad in range(4):
        for taps in range(1, pad + 2):
            for row_slot in (0, 1, 5000):
                for n in (1, 2, 31, 300):
                    for jp0 in [*range(-lanes - 6, 8), *range(n - 4, n + 4), -9000, -1000, -300, 300, 9000]:
                        jp, ln = ctypes.c_int(jp0), ctypes.c_int(n)
                        w = helper.word(row_slot, ctypes.byref(jp), ctypes.byref(ln), taps, lanes, pad, step2)
                        assert (w >> 31) == step2
                        off = ((w & 0x7FFFFFFF) >> 2) - 256
                        at = b + jp0 - (pad - 1 if step2 else 0)  # the run's lane of tap 0 (step 2: of taps 0 and 1)
                        sets = (0, 2) if step2 and taps > 2 else (0,)
                        seen = False
                        for add in sets:
                            want, got = (at + add >= 0) & (at + add < n), (b + jp.value + add >= 0) & (b + jp.value + add < ln.value)
                            assert (want == got).all()
                            if not want.any():
                                continue
                            seen = True
                            slot = off + (((b + (w & 1)) >> 1) + add // 2 if step2 else b)
                            assert (slot == row_slot + ((at + add) // 2 if step2 else at))[want].all()
                        more = (w & 3) if not step2 else (w >> 1) & 1
                        assert more == ((taps - 1 if not step2 else taps > 2) if seen else 0)


@pytest.mark.parametrize("inv", [1.0, 9.1])
@pytest.mark.parametrize("n", [344, 3413, 8192, 18900])
def test_margin_covers_the_rounding_of_footprint_ends(layout, n, inv):
    f = np.float32
    R = int(1.42 * n * inv) + 3
    L = layout(n, n, 1, inv, 180, 2, 1, [1], [(0, 0, 1, 0)], radial=R)
    margin = math.ldexp(L["margin"], -40)
    assert margin < 0.1 and (n > 344 or margin == f(0.01))
    rng = np.random.default_rng(n)
    v, ix, iy = rng.integers(0, 180, 300000), rng.integers(0, n, 300000), rng.integers(0, n, 300000)
    c, s = np.cos(np.pi * v / 180), np.sin(np.pi * v / 180)
    cf, sf = c.astype(f), s.astype(f)
    hw = f(0.5) * (np.abs(cf) + np.abs(sf))
    sc = (ix.astype(f) + f(0.5) - f(0.5 * n)) * cf + (iy.astype(f) + f(0.5) - f(0.5 * n)) * sf
    mid, half = ((ix + 0.5 - 0.5 * n) * c + (iy + 0.5 - 0.5 * n) * s) * inv + 0.5 * (R - 1), 0.5 * (np.abs(c) + np.abs(s)) * inv
    for sign in (-1, 1):
        end = (sc + f(sign) * hw) * f(inv) + f(0.5 * (R - 1))
        assert np.abs(end.astype(np.float64) - (mid + sign * half)).max() < margin
