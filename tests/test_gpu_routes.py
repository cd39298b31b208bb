"""Which kernels serve a little more than 32 tokens: the small-batch kernels, which apply scale and zero-point in fp32, up
to the line that small_batch_chunks draws.  The tensor-core kernels round the dequantized weights to bf16, so a call must
not cross that line because they became faster."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_forward import _pack
from tests.test_gpu_vq import _check as _check_vq
from tests.test_gpu_vq import _random_record

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


# on both sides of the line between the two vector-quantized products for chunks of 32 tokens
@pytest.mark.parametrize("n,m,cr,cc,dim", [(4096, 192, 64, 256, 4), (4096, 512, 512, 256, 2), (4160, 576, 512, 64, 4), (4352, 320, 256, 256, 2),
                                           (256, 65536, 512, 256, 4), (256, 66048, 512, 256, 4)])
@pytest.mark.parametrize("T", [33, 70])
def test_vector_quantized_chunks(n, m, cr, cc, dim, T):
    d = lopro.make_vq_desc(n, m, cr, cc, 64, rank=16, dim=dim)
    rows = np.unique(np.concatenate([[0, 15, 16, m - 17, m - 1], np.random.default_rng(m).integers(0, m, 40)])) if m > 2048 else None
    _check_vq(d, *_random_record(n, m, cr, cc, 16, seed=n + T, dim=dim), T, seed=T, rows=rows)
