"""Which kernels serve a little more than 32 tokens: the small-batch kernels, which apply scale and zero-point in fp32, up
to the line that small_batch_chunks draws.  The tensor-core kernels round the dequantized weights to bf16, so a call must
not cross that line because they became faster."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_forward import _pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,bits,g,r,T", [(2048, 2048, 4, 64, 128, 100), (4096, 2816, 3, 64, 64, 64), (2048, 2048, 4, 64, 32, 96),
                                            (8192, 1024, 2, 64, 128, 33), (1024, 4096, 2, 64, 16, 40)])
def test_rows_of_a_short_prompt_equal_those_of_small_batches(n, m, bits, g, r, T):
    layer = random_layer_np(n, m, bits, g, r, seed=n + T)
    d = lopro.make_desc(n, m, bits, g, 128, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] in (lopro.PATH_STREAM, lopro.PATH_TALL)
    blob = _pack(layer, d)
    x = bf16_bits_to_device(synth.activations(T, n, seed=T, outlier_frac=0.01))
    y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    parts = torch.cat([lopro.linear_fwd(d, blob, x[t:t + 32], lopro.OUT_F32) for t in range(0, T, 32)])
    torch.cuda.synchronize()
    # the same arithmetic, fp32 sums at most in another order; weights rounded to bf16 would differ by about 1e-3
    assert (y - parts).norm().item() <= 1e-5 * parts.norm().item()
