"""The product kernels of the small-batch launches by name (lopro_product_kernel): the persistent kernel and runs of row tiles with runs of
tile steps, which take most of their layers, switched off; the forms of runs of tile steps; and the row CTAs of the prologue, against
the oracle and against each other."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_experts import _check_experts, _experts
from tests.test_gpu_forward import _check_forward, _pack, _tall_rows
from tests.test_gpu_group import _check_group, _persistent_rows, _siblings
from tests.test_gpu_runs import _CASES, _PERSISTENT, _rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,g,r", [(4, 128, 32), (3, 64, 17), (2, 64, 128), (4, 256, 0)])
@pytest.mark.parametrize("T", [1, 8, 16, 32])
@pytest.mark.parametrize("per_sm,extra", [(6, 3), (8, 1), (9, 100), (10, 7)])
def test_tall_layers_persistent_kernel(bits, g, r, T, per_sm, extra):
    # too many tiles for runs of row tiles: with runs of tile steps off the persistent kernel, whose runs of tiles per CTA end in
    # groups of 1, 2 and 3 tiles (4+2/4+3, 8/8+1, 8+1/8+2, 8+2/8+3 tiles per CTA) and a ragged last stage (36 steps)
    n, m = 2304, _tall_rows(per_sm, extra)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL
    layer = random_layer_np(n, m, bits, g, r, seed=m + bits + T)
    x_bits = synth.activations(T, n, seed=T + 11, outlier_frac=0.01)
    # the rows of the first CTAs and of the last ones, and some between
    rows = np.unique(np.concatenate([np.arange(16 * 24), m - 1 - np.arange(16 * 24), np.random.default_rng(m).integers(0, m, 64)]))
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
        assert lopro.product_kernel([d], T)[0] == lopro.PRODUCT_PERSISTENT
        _check_forward(layer, d, x_bits, rows=rows)
    _check_forward(layer, d, x_bits, rows=rows)


@pytest.mark.parametrize("g", [1024, 2048, 4096])
@pytest.mark.parametrize("T,m", [(8, 160), (16, 160), (8, 2), (8, 7), (32, 7)])
def test_groups_as_long_as_or_longer_than_a_stage(g, T, m):
    # a stage of the small-batch kernels holds 1024 columns: groups of exactly one stage, of two stages and of
    # the whole row (one scale per row), on the 32-warp and the 16-warp kernel, in runs of row tiles and, with runs of tile steps
    # off, on the persistent kernel (m below 16: tiles per multiprocessor, and a few)
    n, per_sm = 4096, m
    m = _tall_rows(m, 5) if m < 16 else m
    d = lopro.make_desc(n, m, 4, g, 128, identity_cols=128, rank=16)
    want = {(8, False): lopro.PATH_WIDE, (16, False): lopro.PATH_STREAM}.get((T, m > 160), lopro.PATH_TALL)
    assert lopro.linear_fwd_path(d, T)[0] == want
    layer = random_layer_np(n, m, 4, g, 16, seed=g + T)
    x_bits = synth.activations(T, n, seed=T + g)
    rows = None if m <= 160 else np.unique(np.concatenate([np.arange(160), np.arange(0, m, 37)]))
    if want == lopro.PATH_TALL:
        with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
            assert lopro.product_kernel([d], T)[0] == (lopro.PRODUCT_ROW_RUNS if per_sm == 2 else lopro.PRODUCT_PERSISTENT)
            _check_forward(layer, d, x_bits, rows=rows)
    _check_forward(layer, d, x_bits, rows=rows)


def test_tall_kernels_agree_with_the_per_group_kernel():
    # the small-batch kernels sum the same products in fp32 in different orders: outputs agree to fp32 rounding
    n, m, bits, g, r, T = 1024, _tall_rows(8, 9), 4, 128, 32, 8
    d = lopro.make_desc(n, m, bits, g, 128, rank=r)
    layer = random_layer_np(n, m, bits, g, r, seed=3)
    blob = _pack(layer, d)
    x = bf16_bits_to_device(synth.activations(T, n, seed=4))
    assert lopro.product_kernel([d], T)[0] == lopro.PRODUCT_STEP_RUNS
    y_steps = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
        assert lopro.product_kernel([d], T)[0] == lopro.PRODUCT_PERSISTENT
        y_persistent = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    with lopro.configured(lopro.OPT_NO_TALL, 1):
        assert lopro.linear_fwd_path(d, T)[0] in (lopro.PATH_STREAM, lopro.PATH_WIDE)
        y_stream = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    torch.cuda.synchronize()
    scale = y_stream.abs().max().item()
    for y in (y_steps, y_persistent):
        assert (y - y_stream).abs().max().item() <= 1e-5 * scale


@pytest.mark.parametrize("n,per_sm,extra,bits,g,T,runs", [(*c, True) for c in _CASES] + [(*c, False) for c in _PERSISTENT])
def test_runs_of_row_tiles(n, per_sm, extra, bits, g, T, runs):
    m, r = _rows(per_sm, extra), 16
    layer = random_layer_np(n, m, bits, g, r, seed=n + T + bits)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL
    x_bits = synth.activations(T, n, seed=T, outlier_frac=0.01)
    blob, x = _pack(layer, d), bf16_bits_to_device(x_bits)
    rows = np.unique(np.concatenate([[0, 15, 16, m - 17, m - 1], np.random.default_rng(m).integers(0, m, 40)]))
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
        assert lopro.product_kernel([d], T)[0] == (lopro.PRODUCT_ROW_RUNS if runs else lopro.PRODUCT_PERSISTENT)
        _check_forward(layer, d, x_bits, rows=rows)
        y = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    # the same products in fp32 in another order, every row (K = 8256: 2^-24 times the square root of the terms, times 16)
    with lopro.configured(lopro.OPT_NO_TALL, 1):
        y_short = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    torch.cuda.synchronize()
    assert (y - y_short).abs().max().item() <= 2e-5 * y_short.abs().max().item()


@pytest.mark.parametrize("n,per_sm,extra,bits,g,r,T,form", [
    # form: token tiles, tile steps of a batch, batches of a ring, CTAs that share K
    (256, 7, 1, 4, 128, 16, 1, (1, 4, 3, 1)),       # one batch per tile: warps without a batch, tiles of one warp
    (128, 8, 5, 2, 128, 0, 8, (1, 2, 3, 1)),        # a tile is one batch of two steps; no low-rank term
    (2304, 7, 3, 3, 64, 17, 5, (1, 4, 3, 1)),       # a ragged last stage of activations
    (1152, 9, 100, 4, 64, 40, 3, (1, 2, 3, 1)),     # 18 steps per tile, three tiles of ranks
    (4096, 4, 1, 4, 128, 128, 8, (1, 4, 3, 1)),     # longer runs instead of runs of row tiles; ranks in two passes
    (4096, 3, 100, 2, 64, 32, 16, (2, 4, 3, 1)),    # two token tiles
    (4096, 7, 9, 3, 256, 16, 9, (2, 4, 3, 1)),      # groups as long as a batch
    (4096, 7, 9, 4, 128, 32, 13, (2, 4, 2, 1)),     # a ring of two batches
    (4096, 5, 9, 4, 128, 64, 16, (2, 4, 2, 1)),
    (8192, 8, 3, 4, 128, 16, 8, (1, 4, 2, 1)),
    (1152, 6, 3, 2, 64, 16, 9, (2, 2, 3, 1)),       # two token tiles, batches of two, at every number of bits
    (1152, 6, 3, 3, 64, 32, 16, (2, 2, 3, 1)),
    (1152, 6, 3, 4, 128, 17, 12, (2, 2, 3, 1)),
    (8192, 13, 3, 2, 64, 64, 2, (1, 4, 3, 1)),      # eight stages of activations
    (4096, 40, 11, 2, 2048, 16, 4, (1, 4, 3, 1)),   # forty tiles per CTA, groups longer than a stage
    (512, 2, 3, 4, 64, 16, 32, (4, 2, 4, 1)),       # four token tiles
    (1024, 8, 3, 2, 64, 32, 17, (4, 2, 4, 1)),      # two bits: a ring of four batches, where the sums of four token tiles fit
    (2048, 3, 1, 3, 128, 0, 25, (4, 2, 4, 1)),      # no low-rank term
    (2304, 5, 3, 3, 64, 40, 32, (4, 2, 4, 2)),      # two CTAs share K and the second begins in the middle of a stage
    (4096, 4, 77, 4, 128, 32, 31, (4, 2, 4, 2)),
    (4096, 4, 96, 4, 128, 32, 32, (4, 2, 3, 2)),
    (4096, 12, 9, 4, 128, 64, 32, (4, 2, 2, 2)),    # a ring of two batches of two
    (4224, 4, 9, 4, 128, 17, 24, (4, 2, 2, 2)),     # an odd number of batches of two: the CTAs' parts of K differ
    (8192, 7, 5, 2, 64, 128, 16, (2, 4, 3, 2)),     # two token tiles, eight stages shared by two CTAs
    (11008, 8, 1, 3, 128, 16, 8, (1, 4, 3, 2)),     # one token tile, eleven stages shared by two CTAs
])
def test_runs_of_tile_steps(n, per_sm, extra, bits, g, r, T, form):
    m = _rows(per_sm, extra)
    layer = random_layer_np(n, m, bits, g, r, seed=n + T + bits)
    d = lopro.make_desc(n, m, bits, g, 64, identity_cols=64, rank=r)
    assert lopro.product_kernel([d], T)[0] == lopro.PRODUCT_STEP_RUNS and lopro.product_kernel([d], T)[1][:4] == form
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


@pytest.mark.parametrize("n,m,bits,T", [(11008, 320, 4, 1), (10240, 2400, 3, 4), (8192, 1024, 4, 8), (11008, 16, 4, 7),
                                        (7424, 2416, 4, 2), (9216, 2400, 3, 4)])
def test_long_rows_of_few_tiles(n, m, bits, T):
    # fewer row tiles than multiprocessors, some CTAs without any, and a few tiles more
    layer = random_layer_np(n, m, bits, 128, 32, seed=n + m)
    d = lopro.make_desc(n, m, bits, 128, 128, identity_cols=128, rank=32)
    assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_STREAM and lopro.product_kernel([d], T)[0] == lopro.PRODUCT_STEP_RUNS
    _check_forward(layer, d, synth.activations(T, n, seed=T, outlier_frac=0.01), rows=np.arange(0, m, 7))


@pytest.mark.parametrize("n,T", [(1024, 1), (1024, 8), (1024, 11), (1024, 32), (3072, 30)])
def test_siblings_of_unequal_rows(n, T):
    # the smallest layer gets a CTA (at 3072 columns and 30 tokens two that share K) or two, the tallest most of them
    layers, descs, blobs = _siblings(n, (64, _rows(9, 3), 272), 4, 128, 128, 17, seed=T)
    rows = np.arange(0, 64, 5)
    kernel, form = lopro.product_kernel(descs, T)
    assert kernel == lopro.PRODUCT_STEP_RUNS and form[3] == (2 if n == 3072 else 1)
    _check_group(layers, descs, blobs, synth.activations(T, n, seed=T + 50, outlier_frac=0.01), rows=rows, shared=True, bit_equal=False)


def test_a_sibling_of_one_row_tile_beside_pairs_of_ctas():
    # the second CTA of the pair that shares the small layer's K adds up no tile: it has no use for the low-rank intermediate, and
    # must not leave with a copy of it under way
    layers, descs, blobs = _siblings(4096, (4096, 4096, 16), 4, 128, 128, 32, seed=32)
    assert lopro.product_kernel(descs, 32)[0] == lopro.PRODUCT_STEP_RUNS and lopro.product_kernel(descs, 32)[1][3] == 2
    rows = np.unique(np.concatenate([np.arange(16), np.random.default_rng(1).integers(0, 4096, 30)]))
    _check_group(layers, descs, blobs, synth.activations(32, 4096, seed=3, outlier_frac=0.01), rows=rows, shared=True, bit_equal=False)


@pytest.mark.parametrize("counts", [[1, 9, 8, 0, 16, 3], [2] * 8, [9, 1] * 4])
def test_experts_of_one_and_of_two_token_tiles(counts):
    # in a launch shaped for up to 16 rows the experts with at most eight run the loop of one token tile
    n, m = 1024, _rows(2, 5)
    d, layers, blobs = _experts(n, m, 3, 64, 128, 16, len(counts), seed=3)
    with_rows = [c for c in counts if c]
    assert lopro.product_kernel([d] * len(with_rows), rows=with_rows)[1][:4] == ((2, 4, 3, 1) if max(counts) > 8 else (1, 4, 3, 1))
    _check_experts(d, layers, blobs, counts, seed=9, shared=True, bit_equal=False)


@pytest.mark.parametrize("T", [1, 8, 16, 32])
@pytest.mark.parametrize("bits,g,extra", [(4, 128, (1, 1)), (2, 64, (7, 130)), (3, 64, (3, 40, 90))])
def test_sibling_layers_through_the_persistent_kernel(T, bits, g, extra):
    n, r = 512, 16
    ms = tuple(_persistent_rows(e) for e in extra)
    layers, descs, blobs = _siblings(n, ms, bits, g, 128, r, seed=T + bits)
    assert all(lopro.linear_fwd_path(d, T)[0] == lopro.PATH_TALL for d in descs)
    x_bits = synth.activations(T, n, seed=T + 50, outlier_frac=0.01)
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
        assert lopro.product_kernel(descs, T)[0] == lopro.PRODUCT_PERSISTENT
        _check_group(layers, descs, blobs, x_bits, shared=True, bit_equal=False)
    _check_group(layers, descs, blobs, x_bits, shared=True, bit_equal=False)


@pytest.mark.parametrize("T,per_sm", [(1, 4), (8, 4), (16, 4), (1, 8), (7, 12), (16, 8), (17, 2), (24, 4), (32, 8)])
def test_one_kernel_set_gives_single_layers_the_sums_of_a_group(T, per_sm):
    # four (eight, twelve) row tiles per multiprocessor and layer: a CTA owns four alone and eight in the group of two, i.e. whole
    # groups of four tiles (two with more than 16 tokens) either way, so the persistent kernel adds a row's products in one
    # order -- and another kernel would not
    n, m = 1024, 16 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    layers, descs, blobs = _siblings(n, (m, m), 4, 128, 128, 16, seed=T)
    x = bf16_bits_to_device(synth.activations(T, n, seed=T + 3))
    with lopro.configured(lopro.OPT_ONE_KERNEL_SET, 1):
        assert lopro.product_kernel(descs, T)[0] == lopro.product_kernel(descs[:1], T)[0] == lopro.PRODUCT_PERSISTENT
        together = lopro.linear_fwd_group(descs, blobs, x, lopro.OUT_F32)
        for d, blob, y in zip(descs, blobs, together):
            assert torch.equal(lopro.linear_fwd(d, blob, x, lopro.OUT_F32), y)


def test_experts_through_the_persistent_kernel():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, m, r = 512, 16 * (2 * sms + 5), 16
    d, layers, blobs = _experts(n, m, 4, 128, 128, r, 5, seed=2)
    assert lopro.linear_fwd_path(d, 8)[0] == lopro.PATH_TALL
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, 1):
        assert lopro.product_kernel([d] * 4, rows=[8, 3, 20, 1])[0] == lopro.PRODUCT_PERSISTENT
        _check_experts(d, layers, blobs, [8, 0, 3, 20, 1], seed=9, shared=True, bit_equal=False)


@pytest.mark.parametrize("per_sm,extra,counts,off,kernel", [
    (7, 3, [8] * 8 + [3], 1, lopro.PRODUCT_PERSISTENT),             # up to 8 rows
    (2, 5, [20] + [1] * 7 + [2], 1, lopro.PRODUCT_PERSISTENT),      # and more than 16
    (7, 3, [8] * 8 + [3], 0, lopro.PRODUCT_STEP_RUNS),
    (2, 5, [20] + [1] * 7 + [2], 0, lopro.PRODUCT_STEP_RUNS),
    (2, 5, [8] * 8 + [1], 0, lopro.PRODUCT_ROW_RUNS)])              # the last layer alone
def test_an_expert_alone_in_the_last_launch_writes_its_own_rows_only(per_sm, extra, counts, off, kernel):
    with lopro.configured(lopro.OPT_NO_STEP_RUNS, off):
        _last_expert_alone(per_sm, extra, counts, kernel)


def _last_expert_alone(per_sm, extra, counts, kernel):
    # eight experts share a pair of launches, the ninth has one of its own, shaped for the largest row count: its rows end
    # where y ends, and the rows behind keep their pattern
    n, m = 512, 16 * (torch.cuda.get_device_properties(0).multi_processor_count * per_sm + extra)
    d, _, blobs = _experts(n, m, 4, 128, 128, 16, 1, seed=per_sm)
    blobs = blobs * len(counts)                                   # what an expert's weights are does not matter here
    offs = np.concatenate([[0], np.cumsum(counts)]).tolist()
    total, spare = offs[-1], max(counts)
    x = bf16_bits_to_device(synth.activations(total, n, seed=total))
    assert lopro.product_kernel([d], max(counts))[0] == kernel
    buf = torch.full((total + spare, m), 7.0, dtype=torch.float32, device="cuda")
    y = lopro.linear_fwd_experts(d, blobs, offs, x, lopro.OUT_F32, y=buf[:total])
    torch.cuda.synchronize()
    assert torch.all(buf[total:] == 7.0)
    for e in (0, len(counts) - 1):
        rows = slice(offs[e], offs[e + 1])
        alone = lopro.linear_fwd(d, blobs[e], x[rows], lopro.OUT_F32)
        # the same products in fp32 in another order
        assert (alone - y[rows]).abs().max().item() <= 2e-5 * alone.abs().max().item()


@pytest.mark.parametrize("n,count,r,T", [(512, 4, 16, 16), (1024, 3, 96, 8), (1024, 3, 96, 5), (4096, 2, 128, 1), (4096, 2, 128, 3),
                                         (4096, 8, 32, 1), (8192, 2, 128, 8), (8192, 2, 128, 4), (8192, 2, 64, 2), (2048, 3, 32, 16),
                                         (4096, 3, 32, 32), (2048, 3, 16, 14)])
def test_row_ctas_of_sibling_layers(n, count, r, T):
    # the low-rank rows of all siblings in one launch: one, two, four and eight tokens per CTA, two rows per CTA, long rows
    layers, descs, blobs = _siblings(n, (64, 80, 48, 16, 32, 64, 16, 96)[:count], 4, 64, 64, r, seed=T + r)
    _check_group(layers, descs, blobs, synth.activations(T, n, seed=T + 60, outlier_frac=0.01), shared=True, bit_equal=n < 8192)
