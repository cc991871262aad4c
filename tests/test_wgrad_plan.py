"""How weight gradients are split (wgrad_plan.h), on the host: the tensor core's
sums truncate, so none may be longer than it was when a unit of work was a
tile of 128 (tap, channel) rows, whatever the batch, the image and the SMs."""
import ctypes
import os
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1304_2062_gb300", "csrc")

CODE = """
#include "wgrad_plan.h"
extern "C" int plan(int B, int H, int W, int C, int Cout, int sms, int *o) {
    se2n::nn::tma::WgradGeo g{};
    if (!se2n::nn::tma::wgrad_split(g, B, H, W, C, Cout, sms)) return 0;
    int widest = 0;
    for (int i = 0; i < g.cgroups * g.ngroups; ++i) {
        int s0, s1;
        se2n::nn::tma::wgrad_offsets(g, i % g.cgroups * 64, i / g.cgroups * 64, s0, s1);
        const int t = se2n::nn::tma::wgrad_tiles(s0, s1);
        widest = t > widest ? t : widest;
    }
    const int v[] = {g.F, g.W, g.bkx, g.kblocks, g.ksplit, g.tiles, g.parts, widest, g.len, g.per};
    for (int i = 0; i < 10; ++i) o[i] = v[i];
    return 1;
}
"""

# input and output channels of the network's layers, and the level of their images
LAYERS = [(8, 32, 0), (32, 32, 0), (32, 64, 1), (64, 64, 1), (64, 128, 2), (128, 128, 2), (128, 256, 3),
          (256, 256, 3), (384, 128, 2), (192, 64, 1), (96, 32, 0)]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("wgrad")
    src, lib = d / "plan.cpp", d / "plan.so"
    src.write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", SRC, "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).plan

    def call(*a):
        o = (ctypes.c_int * 10)()
        return list(o) if fn(*a, o) else None
    return call


@pytest.mark.parametrize("B,H,W", [(32, 256, 256), (1, 8, 8), (3, 64, 136), (8, 128, 128), (64, 256, 256),
                                   (1, 1024, 1024), (16, 64, 64), (5, 40, 72), (32, 192, 256)])
@pytest.mark.parametrize("sms", [152, 148])
def test_sums_are_no_longer_than_they_were(plan, B, H, W, sms):
    for C, Cout, level in LAYERS:
        h, w = H >> level, W >> level
        F, cols, bkx, kblocks, ksplit, tiles, parts, widest, length, per = plan(B, h, w, C, Cout, sms)
        assert cols * F == w and kblocks == B * -(-cols // bkx) * -(-h // 8)
        assert per >= 1 and (ksplit - 1) * per < kblocks <= ksplit * per
        assert parts * tiles >= widest       # every tile has a CTA
        # a column of F pixels adds one term to each sum
        run = min(w, 64)
        runs = B * h * -(-w // run)
        ranges = min(runs, -(-2 * sms // -(-9 * C // 128)))
        was = -(-runs // ranges) * run
        terms = min(per, length) * 8 * bkx
        assert length >= 1 and terms <= max(was, 8 * bkx), (C, Cout, terms, was)
        # the length is part of the result: not much shorter either
        assert terms >= min(0.6 * was, kblocks * 8 * bkx), (C, Cout, terms, was)
        assert terms + 1024 + 8 * bkx > min(was, kblocks * 8 * bkx), (C, Cout, terms, was)
