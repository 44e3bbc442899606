"""The down-projection forms of the CTA-pair kernel's producer clusters beyond plain ranks of up to 16: under a dropout mask (forward), for a
product the tiles do not use (backward under dropout) -- on pairs without a tile and on pairs that take tiles
afterwards, with ragged rows and a last chunk that is not full -- and ranks 17 to 32 at such sizes."""
import numpy as np
import pytest
import torch

import qlora_inputs as qi
from gpu_util import GpuLayer, to_f64
from helpers import REL_TOL, rel_err
from oracle import qlora_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,r", [(1025, 1088, 512, 8), (1499, 512, 1088, 16), (1100, 256, 10240, 8), (1100, 10240, 256, 16), (1030, 512, 256, 24), (1040, 320, 256, 40)])
def test_dropout_beside_the_tiles(M, K, N, r):
    import paper_2306_08162_b200 as ql
    layer = qi.random_codes_layer(K=K, N=N, bits=4, group_size=64, r=r, alpha=2.0 * r, M=M, seed=M + r)
    gl = GpuLayer(layer)
    p = 0.25
    keep = 1.0 / (1.0 - p)
    mask_np = (np.random.default_rng(M).random((M, K)) >= p).astype(np.uint8)
    mask = torch.from_numpy(mask_np).cuda()
    Y = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    dX = torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
    H = torch.empty((M, r), dtype=torch.float32, device="cuda")
    G = torch.empty_like(H)
    grads = [(torch.empty((r, K), device="cuda"), torch.empty((N, r), device="cuda")) for _ in range(2)]
    ql.qlora_fwd_dropout(gl.desc, M, gl.X, mask, keep, gl.Q, gl.scales, gl.zeros, gl.A, gl.B, Y, H, gl.ws)
    ql.qlora_bwd_input_dropout(gl.desc, M, gl.dY, mask, keep, gl.Q, gl.scales, gl.zeros, gl.A, gl.B, dX, G, gl.ws)
    for (dA, dB), (h, g) in zip(grads, ((H, G), (None, None))):
        ql.qlora_bwd_lora_dropout(gl.desc, M, gl.X, mask, keep, gl.dY, gl.A, gl.B, h, g, dA, dB, 0, gl.ws)
    torch.cuda.synchronize()
    assert ql.qlora_device_status() == 0
    f64 = orc.bf16_bits_to_f64
    W = orc.dequant(orc.pack(layer["codes"], 4), layer["scales"], layer["zeros"], 4, 64)
    X, dY, A, B = f64(layer["X"]), f64(layer["dY"]), f64(layer["A"]), f64(layer["B"])
    Yo, Ho = orc.forward_dropout(X, W, A, B, layer["alpha"], mask_np, p)
    dXo, dAo, dBo, Go = orc.backward_dropout(X, dY, W, A, B, layer["alpha"], mask_np, p)
    assert rel_err(to_f64(H), Ho) < 1e-4 and rel_err(to_f64(G), Go) < 1e-4          # fp32 sums of exact products
    for name, got, want in (("Y", Y, Yo), ("dX", dX, dXo), ("dA", grads[0][0], dAo), ("dB", grads[0][1], dBo)):
        assert rel_err(to_f64(got), want) <= REL_TOL, name
    for a, b in zip(*grads):                                                        # recomputed H / G: the same bits wherever they are formed
        assert torch.equal(a, b)


@pytest.mark.parametrize("M,K,N,r", [(1100, 1088, 512, 24), (1100, 256, 10240, 32), (1100, 10240, 256, 32)])
def test_ranks_17_to_32_many_tokens(M, K, N, r):
    layer = qi.random_codes_layer(K=K, N=N, bits=4, group_size=64, r=r, alpha=2.0 * r, M=M, seed=M + K + r)
    gl = GpuLayer(layer)
    saved = gl.run()
    ref = orc.layer_reference(layer)
    for name in ("H", "G"):
        assert rel_err(to_f64(saved[name]), ref[name]) < 1e-4, name                 # fp32 sums of exact products
    for name in ("Y", "dX", "dA", "dB"):
        assert rel_err(to_f64(saved[name]), ref[name]) <= REL_TOL, name
    again = gl.run(save_hg=False)
    assert torch.equal(saved["dA"], again["dA"]) and torch.equal(saved["dB"], again["dB"])


@pytest.mark.parametrize("M,K,N,r", [(1025, 64, 256, 8), (1184, 96, 64, 16), (1184, 1056, 64, 8), (1185, 2080, 128, 16), (2368, 480, 64, 8), (2369, 512, 64, 16),
                                     (2400, 1472, 256, 8), (4800, 448, 64, 16)])
def test_masked_product_as_a_launch_of_its_own(M, K, N, r):
    """H recomputed for the gradients: eight rows to a pair of CTAs, sixteen, and one CTA to sixteen rows (borders at 1184 and 2368 tokens on 148 SMs);
    one step of the contraction to a warp and none, a chunk that is not full; the bits of the H that the forward saved."""
    import paper_2306_08162_b200 as ql
    layer = qi.random_codes_layer(K=K, N=N, bits=4, group_size=32, r=r, alpha=2.0 * r, M=M, seed=M + K)
    gl = GpuLayer(layer)
    mask = torch.from_numpy((np.random.default_rng(M).random((M, K)) >= 0.25).astype(np.uint8)).cuda()
    Y, H, G = torch.empty_like(gl.dY), torch.empty((M, r), device="cuda"), torch.randn((M, r), device="cuda")
    ql.qlora_fwd_dropout(gl.desc, M, gl.X, mask, 1 / 0.75, gl.Q, gl.scales, gl.zeros, gl.A, gl.B, Y, H, gl.ws)
    grads = [(torch.empty((r, K), device="cuda"), torch.empty((N, r), device="cuda")) for _ in range(2)]
    for h, (dA, dB) in zip((H, None), grads):
        ql.qlora_bwd_lora_dropout(gl.desc, M, gl.X, mask, 1 / 0.75, gl.dY, gl.A, gl.B, h, G, dA, dB, 0, gl.ws)
    want = (gl.X.double() * mask / 0.75) @ gl.A.double().t()
    assert rel_err(to_f64(H), to_f64(want)) < 1e-4                                  # fp32 sums of exact products
    assert rel_err(to_f64(grads[1][1]), to_f64(gl.desc.alpha / r * gl.dY.double().t() @ want)) < 1e-2     # H once rounded to bf16 (2^-9)
    assert torch.equal(grads[0][0], grads[1][0]) and torch.equal(grads[0][1], grads[1][1])
    assert ql.qlora_device_status() == 0


@pytest.mark.parametrize("M,r", [(1536, 8), (1400, 16)])
def test_dropout_with_a_split_last_wave(M, r):
    """1024 -> 6656: 78 tiles on 74 SM pairs, so the forward's masked producers, their counters and four tiles that two pairs share are one launch."""
    import paper_2306_08162_b200 as ql
    test_dropout_beside_the_tiles(M, 1024, 6656, r)
    layer = qi.random_codes_layer(K=1024, N=6656, bits=4, group_size=64, r=r, alpha=2.0 * r, M=M, seed=M + r)
    gl = GpuLayer(layer)
    mask = torch.from_numpy((np.random.default_rng(M).random((M, 1024)) >= 0.25).astype(np.uint8)).cuda()
    runs = [(torch.empty_like(gl.dY), torch.empty((M, r), device="cuda")) for _ in range(3)]
    for Y, H in runs:
        ql.qlora_fwd_dropout(gl.desc, M, gl.X, mask, 1 / 0.75, gl.Q, gl.scales, gl.zeros, gl.A, gl.B, Y, H, gl.ws)
    for Y, H in runs[1:]:
        assert torch.equal(Y, runs[0][0]) and torch.equal(H, runs[0][1])
    assert ql.qlora_device_status() == 0


@pytest.mark.parametrize("M,K,N,r", [(1600, 512, 4096, 8), (2400, 512, 256, 16), (1100, 1152, 8192, 16), (1100, 2048, 8192, 8)])
def test_dropout_with_short_contractions(M, K, N, r):
    """Where the masked product is a launch ahead because the tiles are through too soon, and where a left-over tile is kept whole (18 steps) and
    split (32)."""
    test_dropout_beside_the_tiles(M, K, N, r)
