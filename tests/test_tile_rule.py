"""The tiling rule of packed fp32 products (host code, compiled by itself): the tiles
that it counts are those of the kernels, a split's CTAs all run at once, and products
measured apart get the tile that was the fastest."""
import ctypes
import random
import subprocess

import pytest

from paper_1110_5765_gb300 import build
from test_gpu_tile_shapes import BY_RULE

SHIM = r"""
#include "tdg_tile_rule.h"
#include "tdg_gemm_tiles.h"
extern "C" int rule(int sym, int W, int L, long long mrows, long long ncols, int slabs, int target,
                    int may_split, int sms, int *groups) {
    tdg::F32Tile t = tdg::f32_tile_rule({sym != 0, W, L, mrows, ncols, slabs, target != 0,
                                         may_split != 0}, sms);
    *groups = t.groups;
    return t.tile;
}
// the tile of the kernel that runs (launch_packed_gemm's choice of shapes)
extern "C" void shape(int sym, int W, int tile, int *bm, int *bn) {
    using namespace tdg;
    if (tile == F32_TILE_SMALL) { *bm = TilesF32Small::BM; *bn = TilesF32Small::BN; }
    else if (tile == F32_TILE_MID) { *bm = TilesF32Mid::BM; *bn = TilesF32Mid::BN; }
    else if (sym) { *bm = TilesF32::BM; *bn = TilesF32::BN; }
    else if (W <= 2) { *bm = TilesF32AsymW2::BM; *bn = TilesF32AsymW2::BN; }
    else { *bm = TilesF32Asym::BM; *bn = TilesF32Asym::BN; }
}
"""
BIG, MID, SMALL = 0, 1, 2


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "rule.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(so),
                    str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(so))


def _rule(host, form, W, L, M, N, K, target=0, may_split=1, sms=152):
    sym = form == "sym"
    mrows = M if sym else -(-M // L) * -(-L // W)
    g = ctypes.c_int()
    tile = host.rule(int(sym), W, L, ctypes.c_longlong(mrows), ctypes.c_longlong(N), -(-K // L),
                     target, may_split, sms, ctypes.byref(g))
    bm, bn = ctypes.c_int(), ctypes.c_int()
    host.shape(int(sym), W, tile, ctypes.byref(bm), ctypes.byref(bn))
    return tile, g.value, -(-mrows // bm.value) * -(-N // bn.value)


@pytest.mark.parametrize("form,W,L,shape,tile,split", [
    # (whole calls, us)
    ("asym", 4, 256, (2048, 2048, 1024), SMALL, False),   # split 147, 64 x 128 110, 64 x 64 102
    ("asym", 4, 256, (4096, 1024, 1024), SMALL, False),   # 147, 109, 101
    ("asym", 4, 128, (1500, 1300, 3000), SMALL, False),   # 205, 238, 147
    ("asym", 4, 128, (512, 512, 4096), BIG, True),        # 63, 300, 176
    ("asym", 2, 128, (3000, 3000, 1000), BIG, False),     # 128 x 128 216, 64 x 64 268
    ("asym", 3, 128, (100, 5000, 2000), BIG, True),       # 116, 192, 130
    ("sym", 4, 64, (512, 512, 4096), BIG, True),          # 89, 128 x 128 203, 64 x 64 100
    ("sym", 2, 128, (700, 700, 3000), SMALL, False),      # 96, 159, 128 x 64 106, 64 x 64 82
    ("sym", 2, 128, (1500, 1500, 1500), BIG, False),      # 128 x 128 95, 128 x 64 100, 110
    ("sym", 2, 128, (4096, 400, 2048), SMALL, False),     # 207, 127, 133, 119
])
def test_measured_products(host, form, W, L, shape, tile, split):
    t, groups, _ = _rule(host, form, W, L, *shape)
    assert (t, groups > 1) == (tile, split)


@pytest.mark.parametrize("form,W,L,shape,kw,tile,split", BY_RULE)
def test_tiles_of_the_gpu_cases(host, form, W, L, shape, kw, tile, split):
    target = "target" in kw
    t, groups, _ = _rule(host, form, 2 if target and form == "sym" else W, L, *shape, int(target))
    assert (t, groups > 1) == ({"big": BIG, "mid": MID, "small": SMALL}[tile], split)


def test_a_split_runs_at_once(host):
    rng = random.Random(7)
    splits = 0
    for _ in range(4000):
        form, W, L = rng.choice(("sym", "asym")), rng.randint(1, 4), rng.choice((16, 48, 64, 128, 512))
        M, N, K = (int(2 ** rng.uniform(5, 12.5)) for _ in range(3))
        sms = rng.choice((152, 132, 16))
        tile, groups, tiles = _rule(host, form, W, L, M, N, K, rng.randint(0, 1), 1, sms)
        assert 1 <= groups <= max(1, -(-K // L))
        if groups > 1:
            splits += 1
            assert tile != MID and tiles * groups <= 2 * sms
        assert _rule(host, form, W, L, M, N, K, 0, 0, sms)[1] == 1
    assert splits > 200
