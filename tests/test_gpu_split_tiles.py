"""Split tiles whose ranks form their parts of the down-projection themselves: 17 to 128 tokens, short contractions, ranks 8 and 16, both
directions -- smallest and largest token tile, ragged tokens, two and four ranks, output columns that do not fill the last tile, more tiles than
clusters of four run at a time."""
import pytest
import torch

import qlora_inputs as qi
from gpu_util import GpuLayer, to_f64
from helpers import REL_TOL, rel_err
from oracle import qlora_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,g", [(2, 64), (3, 128), (4, 32), (8, 128)])
@pytest.mark.parametrize("M,K,N,r", [(17, 512, 512, 8), (33, 1024, 640, 16), (64, 512, 2048, 8), (100, 2048, 256, 16), (127, 256, 1088, 8), (128, 1152, 2048, 16), (64, 512, 4352, 8), (20, 4736, 512, 8)])
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
