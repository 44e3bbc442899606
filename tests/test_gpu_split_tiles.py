"""Split tiles whose ranks form their parts of the down-projection themselves: 17 to 128 tokens, ranks 8 and 16, each case in one direction at
least (test_umma_plan.py holds which) -- smallest and largest token tile, ragged tokens, two and four ranks, of two to 32 steps, output columns that
do not fill the last tile, more tiles than clusters of four run at a time, adapter elements and products that are not finite."""
import pytest
import torch

import qlora_inputs as qi
from gpu_util import GpuLayer, to_f64
from helpers import REL_TOL, rel_err
from oracle import qlora_oracle as orc

pytestmark = pytest.mark.gpu


CASES = [(17, 512, 512, 8), (33, 1024, 640, 16), (64, 512, 2048, 8), (100, 2048, 256, 16), (127, 256, 1088, 8), (128, 1152, 2048, 16), (64, 512, 4352, 8),
         (20, 4736, 512, 8), (40, 4096, 256, 8), (128, 3584, 256, 16), (30, 8192, 384, 16), (90, 320, 3072, 8)]


@pytest.mark.parametrize("bits,g", [(2, 64), (3, 128), (4, 32), (8, 128)])
@pytest.mark.parametrize("M,K,N,r", CASES)
def test_ranks_form_their_parts_of_the_down_projection(bits, g, M, K, N, r):
    layer = qi.random_codes_layer(K=K, N=N, bits=bits, group_size=g if K % g == 0 else 64, r=r, alpha=2.0 * r, M=M, seed=M + K + bits)
    gl = GpuLayer(layer)
    out = gl.run()
    ref = orc.layer_reference(layer)
    for name in ("H", "G"):
        assert rel_err(to_f64(out[name]), ref[name]) < 1e-4, name                   # fp32 sums of exact products
    for name in ("Y", "dX", "dA", "dB"):
        assert rel_err(to_f64(out[name]), ref[name]) <= REL_TOL, name
    again = gl.run()
    for name in ("Y", "dX", "H", "G"):
        assert torch.equal(out[name], again[name]), name


@pytest.mark.parametrize("M,r", [(17, 8), (64, 16), (128, 8)])
def test_infinite_products_stay_infinite(M, r):
    """s * H that is infinite or overflows must not turn the sum into a NaN."""
    import paper_2306_08162_b200 as ql
    gl = GpuLayer(qi.random_codes_layer(K=512, N=256, bits=4, group_size=128, r=r, alpha=16.0, M=M, seed=M + r))
    A, B, X = torch.zeros_like(gl.A), torch.zeros_like(gl.B), torch.zeros_like(gl.X)
    A[0], B[:, 0], X[:, 0] = 3e38, 1.0, 1e30
    X[1::2] *= -1.0
    Y = torch.empty((M, gl.N), dtype=torch.bfloat16, device="cuda")
    ql.qlora_fwd(gl.desc, M, X, gl.Q, gl.scales, gl.zeros, A, B, Y, None, gl.ws)
    assert torch.isinf(Y).all() and (Y[0::2] > 0).all() and (Y[1::2] < 0).all()


@pytest.mark.parametrize("M,g,r", [(17, 128, 8), (64, 32, 16), (128, 64, 8), (100, 128, 16)])
def test_infinite_adapter_elements_give_infinities(M, g, r):
    """An infinite element of the adapter applied second makes its column of Y / dX infinite with the sign of s * H / s * G, and changes no other bit;
    one of the adapter applied first makes its rank's column of H / G infinite (or NaN), and no other."""
    import paper_2306_08162_b200 as ql
    gl = GpuLayer(qi.random_codes_layer(K=512, N=512, bits=4, group_size=g, r=r, alpha=16.0, M=M, seed=M + g + r))
    clean = gl.run()
    A, B = gl.A.clone(), gl.B.clone()
    A[3, 70], B[100, 5] = float("-inf"), float("inf")
    Y, dX = torch.empty_like(clean["Y"]), torch.empty_like(clean["dX"])
    H, G = torch.empty_like(clean["H"]), torch.empty_like(clean["G"])
    ql.qlora_fwd(gl.desc, M, gl.X, gl.Q, gl.scales, gl.zeros, gl.A, B, Y, H, gl.ws)
    ql.qlora_bwd_input(gl.desc, M, gl.dY, gl.Q, gl.scales, gl.zeros, A, gl.B, dX, G, gl.ws)
    for got, was, col, want in ((Y, clean["Y"], 100, torch.sign(H[:, 5])), (dX, clean["dX"], 70, -torch.sign(G[:, 3]))):
        assert torch.isinf(got[:, col]).all() and torch.equal(torch.sign(got[:, col].float()), want)
        rest = torch.arange(got.shape[1], device="cuda") != col
        assert torch.equal(got[:, rest], was[:, rest])
    ql.qlora_fwd(gl.desc, M, gl.X, gl.Q, gl.scales, gl.zeros, A, gl.B, Y, H, gl.ws)
    ql.qlora_bwd_input(gl.desc, M, gl.dY, gl.Q, gl.scales, gl.zeros, gl.A, B, dX, G, gl.ws)
    for got, was, col in ((H, clean["H"], 3), (G, clean["G"], 5)):
        rest = torch.arange(r, device="cuda") != col
        assert not torch.isfinite(got[:, col]).any() and torch.equal(got[:, rest], was[:, rest])
