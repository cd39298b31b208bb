"""Taller layers of up to 16 tokens in runs of row tiles (launch_stream, in_runs): run lengths at the edges of each kernel
variant, one wave and two, a ragged last stage of K, rings that hold all of K and rings that are refilled, against the oracle and
against the kernel of short runs; and the layers that stay with the persistent kernel."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np, takes_runs_of_row_tiles
from tests.test_gpu_forward import _check_forward, _pack

pytestmark = pytest.mark.gpu


def _rows(per_sm, extra):
    return 16 * (torch.cuda.get_device_properties(0).multi_processor_count * per_sm + extra)


_ANY = [(4, 64, 8), (3, 64, 1), (2, 64, 5)]
_CASES = (
    # (columns, row tiles per multiprocessor, further tiles, bits, group, tokens): runs of 3, 4, 5 and 6, all of K in the ring
    [(n, per_sm, extra, *q) for n, per_sm, extra in ((576, 2, 1), (1088, 4, 0), (1088, 4, 1), (1024, 5, 147)) for q in _ANY]
    + [(1088, 2, 1, 4, 64, 16), (1088, 4, 0, 3, 64, 9), (1088, 4, 1, 4, 64, 16), (2048, 4, 147, 2, 64, 16)]
    # rings of three or four slots that are refilled (K of four and of five or nine stages)
    + [(4096, 4, 1, 4, 128, 8), (4096, 5, 147, 4, 128, 1), (4160, 5, 3, 2, 64, 3), (8256, 4, 1, 3, 64, 2),
       (4096, 3, 5, 4, 128, 16), (5120, 4, 9, 2, 128, 12)]
    # five tiles of rows shorter than a stage
    + [(512, 4, 100, 2, 64, 9), (960, 4, 5, 4, 64, 16)]
    # two waves with runs of 7 and 8, K of eight stages and more
    + [(8192, 13, 1, 2, 64, 5), (8256, 15, 147, 2, 64, 8), (8192, 15, 147, 3, 256, 4)])
# no two waves for 16 tokens nor for short rows, no room for three stages of eight tiles, runs of six with 16 tokens, up to four
# tiles of rows shorter than a stage with more than eight
_PERSISTENT = [(8192, 13, 1, 2, 64, 16), (4096, 13, 1, 2, 64, 5), (8192, 13, 1, 4, 64, 8), (8256, 15, 147, 3, 64, 1),
               (1024, 5, 147, 4, 64, 16), (960, 3, 5, 4, 64, 12), (512, 4, 0, 2, 64, 9)]


@pytest.mark.parametrize("n,per_sm,extra,bits,g,T,runs", [(*c, True) for c in _CASES] + [(*c, False) for c in _PERSISTENT])
def test_runs_of_row_tiles(n, per_sm, extra, bits, g, T, runs):
    m, r = _rows(per_sm, extra), 16
    layer = random_layer_np(n, m, bits, g, r, seed=n + T + bits)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL
    x_bits = synth.activations(T, n, seed=T, outlier_frac=0.01)
    blob, x = _pack(layer, d), bf16_bits_to_device(x_bits)
    assert takes_runs_of_row_tiles(d, blob, x) == runs
    rows = np.unique(np.concatenate([[0, 15, 16, m - 17, m - 1], np.random.default_rng(m).integers(0, m, 40)]))
    _check_forward(layer, d, x_bits, rows=rows)
    # the same products in fp32 in another order, every row (K = 8256: 2^-24 times the square root of the terms, times 16)
    y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    with lopro.configured(lopro.OPT_NO_TALL, 1):
        y_short = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    torch.cuda.synchronize()
    assert (y - y_short).abs().max().item() <= 2e-5 * y_short.abs().max().item()
