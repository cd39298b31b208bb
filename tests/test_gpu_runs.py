"""Taller layers of up to 16 tokens in runs of row tiles (launch_stream, in_runs): run lengths at the edges of each kernel
variant, one wave and two, a ragged last stage of K, against the oracle and against the kernel of short runs."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_forward import _check_forward, _pack

pytestmark = pytest.mark.gpu


def _rows(per_sm, extra):
    return 16 * (torch.cuda.get_device_properties(0).multi_processor_count * per_sm + extra)


# (row tiles per multiprocessor, further tiles): runs of 3, 4, 5 and 6; of 7 and 8 in two waves where K has eight stages
@pytest.mark.parametrize("n,per_sm,extra", [(576, 2, 1), (1088, 4, 0), (1088, 4, 1), (1024, 5, 147), (8192, 13, 1), (8256, 15, 147)])
@pytest.mark.parametrize("bits,g,T", [(4, 64, 8), (3, 64, 1), (2, 64, 5), (4, 64, 16)])
def test_runs_of_row_tiles(n, per_sm, extra, bits, g, T):
    m, r = _rows(per_sm, extra), 16
    layer = random_layer_np(n, m, bits, g, r, seed=n + T + bits)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL
    x_bits = synth.activations(T, n, seed=T, outlier_frac=0.01)
    rows = np.unique(np.concatenate([[0, 15, 16, m - 17, m - 1], np.random.default_rng(m).integers(0, m, 40)]))
    _check_forward(layer, d, x_bits, rows=rows)
    # the same products in fp32 in another order, every row (K = 8256: 2^-24 times the square root of the terms, times 16)
    blob, x = _pack(layer, d), bf16_bits_to_device(x_bits)
    y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    with lopro.configured(lopro.OPT_NO_TALL, 1):
        y_short = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    torch.cuda.synchronize()
    assert (y - y_short).abs().max().item() <= 2e-5 * y_short.abs().max().item()


def test_short_rows_of_more_than_eight_tokens_stay_with_the_persistent_kernel():
    # with a whole stage of K the two kernels add a row's products in different orders, so equal sums name the kernel
    for n, per_sm, same in ((512, 3, True), (960, 3, True), (1024, 3, False), (512, 4, False)):
        m = _rows(per_sm, 5)      # 3 or 4 tiles per CTA; 4 or 5
        layer = random_layer_np(n, m, 4, 64, 16, seed=n)
        d = lopro.make_desc(n, m, 4, 64, 64, identity_cols=64, rank=16)
        blob, x = _pack(layer, d), bf16_bits_to_device(synth.activations(12, n, seed=n))
        y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
        with lopro.configured(lopro.OPT_ONE_KERNEL_SET, 1):
            assert torch.equal(lopro.linear_fwd(d, blob, x, lopro.OUT_F32), y) == same
