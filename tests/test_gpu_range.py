"""Results that use most of the fp32 range: the small-batch kernels multiply half of a tile's rows in other units (2- and
3-bit codes), and the sums of those rows must not leave the range where the result does not."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests.test_gpu_forward import _pack

pytestmark = pytest.mark.gpu


# 32-warp, 16-warp (two and four token tiles), runs of row tiles, persistent (one and four token tiles)
@pytest.mark.parametrize("tiles_per_sm,T", [(0, 8), (0, 16), (0, 32), (4, 8), (7, 8), (2, 32)])
@pytest.mark.parametrize("bits", [2, 3])
def test_large_results_stay_finite(bits, tiles_per_sm, T):
    # Nothing but a permutation in front, the identity.  Activations +a, -a, ... meet codes top, 0, ... with the zero-point
    # half-way: every product is z a, the activations of a step add up to nothing, and no partial sum exceeds the result.
    n, g, top = 1024, 64, 2 ** bits - 1
    m = 16 * (tiles_per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 4)
    flip = (np.arange(m) // 3 % 2)[:, None]                                   # rows of either sign
    codes = np.where((np.arange(n)[None, :] + flip) % 2 == 0, top, 0).astype(np.uint8)
    layer = dict(codes=codes, scales=synth.f32_to_f16_bits(np.full((m, n // g), 60000.0)),
                 zeros=synth.f32_to_f16_bits(np.full((m, n // g), top / 2)), perm=np.arange(n, dtype=np.int32),
                 A=np.zeros((m, 0), np.uint16), B=np.zeros((0, n), np.uint16))
    a = torch.tensor(2.5e38 / (60000.0 * n * top / 2)).to(torch.bfloat16)
    x = (a * torch.tensor([1.0, -1.0]).repeat(n // 2)).to(torch.bfloat16).repeat(T, 1)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=n, rank=0)
    y = lopro.linear_fwd(d, _pack(layer, d), x.cuda(), lopro.OUT_F32)
    torch.cuda.synchronize()
    s = float(np.float16(60000.0))
    want = s * n * (top / 2) * float(a) * (1.0 - 2.0 * torch.from_numpy(flip[:, 0].astype(np.float64)))
    assert 2e38 < want.abs().max() < 3.4e38
    # n products, each rounded to 24 bits where it is added
    assert ((y.cpu().double() - want).abs() <= n * 2.0 ** -24 * want.abs()).all()
