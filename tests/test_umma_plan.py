"""The host's plan for the tensor-core kernels (csrc/umma_plan.h), over all shapes, without a GPU: the header is compiled by itself."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include "umma_plan.h"
using namespace qlora;
extern "C" int tiles(int bits, int g, int r, int M, int C, int T, int transposed, int wants_p /* 2: dropout, the product is there already */, int* out) {
    TilePlan p{};
    p.M = M; p.C = C; p.bits = bits; p.g = g; p.r = r; p.r_pad = lora_columns(r, g);
    const bool ok = plan_tiles(p, T, transposed != 0, wants_p == 1, wants_p == 2, GpuFit{148, 74, 33});
    const int v[] = {p.S, p.P, p.split, p.steps, p.down_bytes != 0, p.BT, (int)p.off_bar, (int)p.x_stage_bytes};
    for (int i = 0; i < 8; ++i) out[i] = v[i];
    return ok;
}
extern "C" int pair(int bits, int g, int r, int transposed, int* out) {
    const unsigned l = (unsigned)(kPairW * lora_columns(r, g) * 2), a = (unsigned)(2 * kPairTok * lora_columns(r, g) * 2);
    TilePlan p{};
    plan_packed_stage(p, bits, g, transposed != 0);
    return plan_pair_rings(p.packed_slot_bytes, l + a < 8192 ? 8192 : l + a, out[0], out[1]);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2306_08162_b200", "csrc"),
                    str(d / "shim.cpp"), "-o", str(d / "plan.so")], check=True)
    return ctypes.CDLL(str(d / "plan.so"))


def early_wait(S, P, groups, n=60):
    """A step at which a dequant group's wait may return a lap early: what it knows to be over before step t is every step whose products it has
    seen through (up to t - groups - S: it waited for its previous stage to be free) and its own steps."""
    for t in range(n):
        seen = t - groups - S
        if t - 2 * S >= 0 and t - 2 * S > seen:
            return t
        if t - P >= 0 and t - P > seen and (t - P) % groups != t % groups:
            return t
    return None


SHAPES = [(bits, g, r, tr) for bits in (2, 3, 4, 8) for g in (32, 64, 128) for r in range(0, 65, 8) for tr in (0, 1)]


def test_rings_of_the_single_cta_kernel(plan):
    out = (ctypes.c_int * 8)()
    seen_down = False
    for bits, g, r, tr in SHAPES:
        for M in list(range(1, 257, 15)) + [333, 512, 700, 1024]:
            for C, T in ((256, 512), (2048, 768), (4096, 4096), (4096, 11008), (11008, 4096)):
                for wants_p in (0, 1):
                    assert plan.tiles(bits, g, r, M, C, T, tr, wants_p, out), (bits, g, r, tr, M, C, T)
                    S, P, split, steps, down, BT, off_bar, _ = out
                    assert split * steps == T // 64 and off_bar + 512 + 1024 + 1024 <= 232448
                    assert early_wait(S, P, 3 if down else 2) is None, (bits, g, r, tr, M, C, T, S, P, down)
                    seen_down |= bool(down)
    assert seen_down


def test_rings_of_the_pair_kernel(plan):
    out = (ctypes.c_int * 2)()
    for bits, g, r, tr in SHAPES:
        assert plan.pair(bits, g, r, tr, out), (bits, g, r, tr)
        assert early_wait(out[0], out[1], 2) is None, (bits, g, r, tr, list(out))


@pytest.mark.parametrize("M,BT_tiles", [(17, 1), (128, 1), (200, 1), (333, 2)])
def test_split_tiles_run_in_one_wave(plan, M, BT_tiles):
    """33 clusters of four CTAs run at a time on 148 SMs, 74 of two."""
    out = (ctypes.c_int * 8)()
    for C in range(64, 12000, 64):
        for T in (512, 768, 1024, 4096, 11008):
            for wants_p in (0, 1):
                assert plan.tiles(4, 128, 8, M, C, T, 0, wants_p, out)
                tiles = BT_tiles * ((C + 127) // 128)
                assert out[2] == 1 or tiles <= {4: 33, 2: 74}[out[2]], (M, C, T, list(out))


@pytest.mark.parametrize("r,wants_p,M,T,C,split,steps", [
    (32, 1, 17, 512, 512, 2, 4), (32, 1, 128, 768, 2048, 2, 6), (64, 1, 128, 512, 4096, 2, 4), (24, 2, 96, 512, 1024, 2, 4),     # ranks above 16
    (0, 0, 64, 512, 4096, 2, 4), (0, 0, 17, 768, 3072, 2, 6), (0, 0, 128, 512, 2048, 2, 4), (0, 2, 48, 512, 4096, 2, 4),          # rank 0
    (8, 2, 128, 512, 2048, 2, 4), (16, 2, 65, 512, 512, 2, 4),                                                                  # dropout, many tokens
    (0, 0, 64, 512, 2048, 4, 2), (0, 0, 128, 768, 1024, 4, 3), (16, 2, 64, 512, 4096, 4, 2), (0, 2, 17, 512, 4096, 4, 2),        # where short ranks pay
    (8, 1, 128, 512, 512, 4, 2), (16, 1, 17, 768, 4096, 4, 3)])
def test_short_ranks_only_where_they_pay(plan, r, wants_p, M, T, C, split, steps):
    out = (ctypes.c_int * 8)()
    assert plan.tiles(4, 128, r, M, C, T, 0, wants_p, out)
    assert (out[2], out[3]) == (split, steps)


@pytest.mark.parametrize("bits,r,M,T,C,tr,split,steps,down", [
    (4, 8, 128, 1024, 8192, 0, 2, 8, 0), (4, 16, 80, 1024, 6016, 1, 2, 8, 0), (4, 16, 128, 896, 2048, 0, 2, 7, 0),       # two ranks, many tokens
    (4, 8, 112, 640, 8192, 0, 2, 5, 0), (4, 8, 112, 640, 512, 0, 2, 5, 1), (4, 8, 64, 1024, 6016, 0, 2, 8, 1),
    (4, 8, 64, 4096, 2048, 0, 4, 16, 0), (2, 8, 128, 4096, 512, 1, 4, 16, 0), (4, 8, 48, 4096, 2048, 0, 4, 16, 1),        # rank 8, long ranks
    (4, 8, 96, 4096, 2048, 1, 4, 16, 1), (3, 8, 96, 4096, 2048, 0, 4, 16, 1), (4, 8, 96, 4096, 4096, 0, 4, 16, 1),
    (4, 16, 128, 6144, 2048, 0, 4, 24, 0), (4, 16, 64, 8192, 512, 0, 4, 32, 0), (8, 16, 48, 11008, 512, 0, 4, 43, 0),     # rank 16
    (4, 16, 128, 3584, 2048, 0, 4, 14, 1), (4, 16, 128, 6144, 2048, 1, 4, 24, 1), (4, 16, 128, 11008, 4096, 0, 4, 43, 1)])
def test_ranks_form_their_part_of_the_down_projection_where_that_pays(plan, bits, r, M, T, C, tr, split, steps, down):
    out = (ctypes.c_int * 8)()
    assert plan.tiles(bits, 128, r, M, C, T, tr, 1, out)
    assert (out[2], out[3], out[4]) == (split, steps, down)


def test_the_split_tile_tests_run_the_build_they_are_for(plan):
    from test_gpu_split_tiles import CASES
    out = (ctypes.c_int * 8)()
    ranks = set()
    for bits, g in ((2, 64), (3, 128), (4, 32), (8, 128)):
        for M, K, N, r in CASES:
            took = 0
            for C, T, tr in ((N, K, 0), (K, N, 1)):
                assert plan.tiles(bits, g if K % g == 0 else 64, r, M, C, T, tr, 1, out)
                if out[4]:
                    took += 1
                    ranks.add((out[2], out[3]))
            assert took, (bits, M, K, N, r)
    assert {(4, 2), (2, 4), (4, 16), (4, 14), (4, 32)} <= ranks, ranks
