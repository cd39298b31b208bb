"""Layers whose warps each take a run of tile steps of their own (launch_warp_runs): batches of four and of two steps, rings of three
and of two batches, fewer batches than warps, warps that cross several tiles, one and two token tiles, both low-rank records, layers and
experts that share a launch -- against the oracle and against the kernels that take the layers without it."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_experts import _check_experts, _experts
from tests.test_gpu_forward import _check_forward, _pack
from tests.test_gpu_group import _check_group, _siblings

pytestmark = pytest.mark.gpu


def _rows(per_sm, extra):
    return 16 * (torch.cuda.get_device_properties(0).multi_processor_count * per_sm + extra)


@pytest.mark.parametrize("n,per_sm,extra,bits,g,r,T", [
    (256, 7, 1, 4, 128, 16, 1),       # one batch of four steps per tile: warps without a batch, tiles of one warp
    (128, 8, 5, 2, 128, 0, 8),        # a tile is one batch of two steps; no low-rank term
    (2304, 7, 3, 3, 64, 17, 5),       # batches of four, a ragged last stage of activations
    (1152, 9, 100, 4, 64, 40, 3),     # batches of two steps (18 steps per tile), three tiles of ranks
    (4096, 4, 1, 4, 128, 128, 8),     # longer runs instead of runs of row tiles; ranks in two passes
    (4096, 3, 100, 2, 64, 32, 16),    # two token tiles, a ring of two batches
    (4096, 7, 9, 3, 256, 16, 9),      # groups as long as a batch
    (4096, 7, 9, 4, 128, 32, 13),     # four bits and two token tiles: batches of two
    (8192, 13, 3, 2, 64, 64, 2),      # eight stages of activations
    (4096, 40, 11, 2, 2048, 16, 4),   # forty tiles per CTA, groups longer than a stage
    (512, 2, 3, 4, 64, 16, 32),       # four token tiles
    (1024, 8, 3, 2, 64, 32, 17),      # two bits: a ring of four batches, where the sums of four token tiles fit
    (2048, 3, 1, 3, 128, 0, 25),      # no low-rank term
    (2304, 5, 3, 3, 64, 40, 32),      # two CTAs share K and the second begins in the middle of a stage
    (4096, 4, 77, 4, 128, 32, 31),    # a ring of two batches of two
    (4224, 4, 9, 4, 128, 17, 24),     # an odd number of batches of two: the CTAs' parts of K differ
    (8192, 7, 5, 2, 64, 128, 16),     # two token tiles, eight stages shared by two CTAs
    (11008, 8, 1, 3, 128, 16, 8),     # one token tile, eleven stages shared by two CTAs
])
def test_runs_of_tile_steps(n, per_sm, extra, bits, g, r, T):
    m = _rows(per_sm, extra)
    layer = random_layer_np(n, m, bits, g, r, seed=n + T + bits)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL
    x_bits = synth.activations(T, n, seed=T, outlier_frac=0.01)
    blob, x = _pack(layer, d), bf16_bits_to_device(x_bits)
    rows = np.unique(np.concatenate([[0, 15, 16, m - 17, m - 1], np.random.default_rng(m).integers(0, m, 40)]))
    _check_forward(layer, d, x_bits, rows=rows)
    # the same products in fp32 in another order, every row (2^-24 times the square root of the terms, times 16); rows behind y stay
    buf = torch.full((T + 1, m), 7.0, dtype=torch.float32, device="cuda")
    y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32, y=buf[:T])
    with lopro.configured(lopro.OPT_NO_TALL, 1):
        y_short = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    torch.cuda.synchronize()
    assert torch.all(buf[T:] == 7.0)
    assert (y - y_short).abs().max().item() <= 2e-5 * y_short.abs().max().item()


@pytest.mark.parametrize("n,m,bits,T", [(11008, 320, 4, 1), (10240, 2400, 3, 4), (8192, 1024, 4, 8), (11008, 16, 4, 7)])
def test_long_rows_of_few_tiles(n, m, bits, T):
    # fewer row tiles than multiprocessors, some CTAs without any
    layer = random_layer_np(n, m, bits, 128, 32, seed=n + m)
    d = lopro.make_desc(n, m, bits, 128, 128, identity_cols=128, rank=32)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_STREAM
    _check_forward(layer, d, synth.activations(T, n, seed=T, outlier_frac=0.01), rows=np.arange(0, m, 7))


@pytest.mark.parametrize("n,T", [(1024, 1), (1024, 8), (1024, 11), (1024, 32), (3072, 30)])
def test_siblings_of_unequal_rows(n, T):
    # the smallest layer gets a CTA (at 3072 columns and 30 tokens two that share K) or two, the tallest most of them
    layers, descs, blobs = _siblings(n, (64, _rows(9, 3), 272), 4, 128, 128, 17, seed=T)
    rows = np.arange(0, 64, 5)
    _check_group(layers, descs, blobs, synth.activations(T, n, seed=T + 50, outlier_frac=0.01), rows=rows, shared=True, bit_equal=False)


@pytest.mark.parametrize("counts", [[1, 9, 8, 0, 16, 3], [2] * 8, [9, 1] * 4])
def test_experts_of_one_and_of_two_token_tiles(counts):
    # in a launch shaped for up to 16 rows the experts with at most eight run the loop of one token tile
    n, m = 1024, _rows(1, 5)
    d, layers, blobs = _experts(n, m, 3, 64, 128, 16, len(counts), seed=3)
    _check_experts(d, layers, blobs, counts, seed=9, shared=True, bit_equal=False)
