"""Parity of the fused LREC loss kernel with the oracle (needs a B200).  Logits are bf16 on both sides; the loss is compared
per token, the gradient with the layer tests' error measure (|got - ref| / max(|ref|, rms(ref)) <= 2e-2: the gradient is
stored in bf16)."""
import numpy as np
import pytest
import torch

import paper_2306_08162_b200 as ql
import qlora_inputs as qi
from oracle import qlora_oracle as orc
from gpu_util import bf16_from_bits, to_f64
from helpers import REL_TOL, rel_err

pytestmark = pytest.mark.gpu


def run_case(T, V, lkl, lce, seed, with_grad=True, scale=1.0, spread=3.0):
    z_bits = qi.normal_bf16(seed, 0, (T, V), spread)
    t_bits = qi.normal_bf16(seed, 1, (T, V), spread)
    labels = np.random.default_rng(seed).integers(-1, V, size=T).astype(np.int32)
    z, t = bf16_from_bits(z_bits), bf16_from_bits(t_bits)
    loss = torch.full((T,), float("nan"), dtype=torch.float32, device="cuda")
    grad = torch.full((T, V), float("nan"), dtype=torch.bfloat16, device="cuda") if with_grad else None
    ql.qlora_lrec_loss(z, t, torch.from_numpy(labels).cuda(), lkl, lce, scale, loss, grad)
    torch.cuda.synchronize()
    want_loss, want_grad = orc.lrec_loss(orc.bf16_bits_to_f64(z_bits), orc.bf16_bits_to_f64(t_bits), labels, lkl, lce)
    assert np.allclose(loss.cpu().numpy(), want_loss, rtol=2e-4, atol=2e-5)
    if with_grad:
        assert rel_err(to_f64(grad), scale * want_grad) <= REL_TOL
    return loss


@pytest.mark.parametrize("T,V", [(7, 32000), (64, 32768), (33, 4096), (5, 8), (300, 1000), (2, 12296)])
def test_loss_and_gradient_match_the_oracle(T, V):
    run_case(T, V, 0.8, 1.2, seed=T + V, scale=1.0 / T)


@pytest.mark.parametrize("V", [8, 256, 264, 2056, 8192, 8200, 20000, 24584, 32760])
@pytest.mark.parametrize("T", [1, 700])
def test_row_lengths_at_the_edges_of_the_block_plan(T, V):
    """One chunk, a full warp of chunks and one more, several short rows per SM, rows that need a third and fourth chunk per
    thread; more rows than resident blocks (700 x short rows) and a single one."""
    if T * V > 6_000_000:
        T = 160                                             # still more rows than SMs
    run_case(T, V, 0.7, 0.9, seed=T + V, scale=0.5)


def test_rows_with_infinitely_unlikely_teacher_tokens():
    """A stretch of -inf teacher logits (whole warps of them) where the student has mass: KL is infinite, not NaN; the other
    rows of the launch are untouched."""
    z = torch.randn((3, 32000), device="cuda").bfloat16()
    t = z.clone()
    t[1, :24000] = float("-inf")
    loss = torch.empty(3, dtype=torch.float32, device="cuda")
    ql.qlora_lrec_loss(z, t, None, 1.0, 0.0, 1.0, loss, None)
    assert torch.isinf(loss[1]) and loss[1] > 0 and loss[0].abs() < 1e-5 and loss[2].abs() < 1e-5


@pytest.mark.parametrize("mask", [-3.3895313892515355e38, -1e30, -1e10, -65504.0])
@pytest.mark.parametrize("student,teacher", [(True, True), (True, False), (False, True)])
def test_rows_with_masked_vocabulary_entries(mask, student, teacher):
    """Entries masked by a large negative logit (finfo.min among them), in stretches that fill whole warps and in single places, on
    either side: a masked student entry has probability zero and adds nothing; a masked teacher entry beside an unmasked
    student one is as expensive as the formula says.  With loss scaling: a probability of zero stays zero."""
    T, V, scale = 5, 8192, 1024.0
    z_bits, t_bits = qi.normal_bf16(91, 0, (T, V), 2.0), qi.normal_bf16(91, 1, (T, V), 2.0)
    z, t = bf16_from_bits(z_bits), bf16_from_bits(t_bits)
    for x, on in ((z, student), (t, teacher)):
        if on:
            x[1, 4096:] = mask
            x[2, :256] = mask
            x[3, 1::3] = mask
            x[4, 8:] = mask
    labels = torch.tensor([5, 7, 300, 0, 3], dtype=torch.int32, device="cuda")
    loss, grad = torch.empty(T, dtype=torch.float32, device="cuda"), torch.empty_like(z)
    ql.qlora_lrec_loss(z, t, labels, 0.9, 0.6, scale, loss, grad)
    want_loss, want_grad = orc.lrec_loss(to_f64(z), to_f64(t), labels.cpu().numpy(), 0.9, 0.6)
    assert np.allclose(loss.cpu().numpy(), want_loss, rtol=2e-4, atol=2e-5)
    if student or mask > -1e38:                                          # (finfo.min in the teacher alone: the scaled gradient leaves bf16's range)
        for row in range(T):
            assert rel_err(to_f64(grad[row]), scale * want_grad[row]) <= REL_TOL, row
    if student and teacher:
        assert torch.equal(grad[1, 4096:], torch.zeros_like(grad[1, 4096:]))


def test_loss_only_and_pure_terms_and_determinism():
    a = run_case(16, 32000, 1.0, 0.0, seed=1, with_grad=False)
    run_case(16, 32000, 0.0, 1.0, seed=2)
    b = run_case(16, 32000, 1.0, 0.0, seed=1, with_grad=False)
    assert torch.equal(a, b)
    run_case(8, 2048, 0.5, 0.5, seed=3, spread=12.0)        # peaked distributions: large logit range


def test_rejected_shapes():
    z = torch.zeros((2, 12), dtype=torch.bfloat16, device="cuda")
    out = torch.zeros(2, dtype=torch.float32, device="cuda")
    with pytest.raises(ql.QloraError) as e:
        ql.qlora_lrec_loss(z, z, None, 1.0, 1.0, 1.0, out, None)          # V % 8 != 0
    assert e.value.status == -2
