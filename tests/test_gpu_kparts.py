"""More than 32 tokens with tiles cut along K: the one-CTA-per-tile tensor-core kernel (one- and two-block tiles, an odd
number of row blocks, parts that hold low-rank stages only), more parts of the two-CTA kernel, and K slices of the low-rank
product that do not divide the width; the same layers in a workspace without room for the parts; and the rotation's CTAs."""
import numpy as np
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np
from tests.test_gpu_forward import GATE_A, GATE_B, _check_forward_once, _pack
from tests.test_gpu_rotate import _run as _run_rotation, _ulp_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,bits,g,b,r,T", [
    (2048, 400, 4, 128, 128, 32, 33),      # 4 row blocks, the last ragged; one token tile of 64
    (1024, 1680, 3, 64, 64, 17, 64), (1024, 1680, 2, 64, 64, 64, 65),
    (832, 560, 2, 64, 64, 128, 129),       # 13 steps of K: uneven slices; 5 row blocks
    (1088, 640, 4, 64, 64, 16, 256), (1856, 912, 3, 64, 64, 40, 257), (5696, 256, 4, 64, 64, 64, 133),
    (512, 272, 2, 64, 128, 512, 100),      # as many low-rank stages as weight stages
    (512, 272, 4, 128, 64, 0, 511),
    (704, 528, 2, 64, 64, 32, 544), (832, 560, 2, 64, 64, 128, 590), (320, 208, 4, 64, 64, 16, 1100),
])
def test_tiles_cut_along_k_and_uneven_slices(n, m, bits, g, b, r, T):
    layer = random_layer_np(n, m, bits, g, r, seed=n + m + T + 1)
    d = lopro.make_desc(n, m, bits, g, b, identity_cols=b, rank=r)
    x_bits = synth.activations(T, n, seed=T + 2, outlier_frac=0.01)
    with lopro.configured(lopro.OPT_NO_CHUNKS, 1):
        assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_PREFILL
        _check_forward_once(layer, d, x_bits, None, GATE_A, GATE_B)
        with lopro.configured(lopro.OPT_NO_CTA_PAIRS, 1):
            if (n, T) in ((2048, 33), (1856, 257)):
                assert lopro.linear_fwd_path(d, T)[1] >= 4          # the launch that adds the parts is there
            _check_forward_once(layer, d, x_bits, None, GATE_A, GATE_B)


@pytest.mark.parametrize("T", [40, 64, 200])
def test_the_general_product_with_the_tensor_core_path_off(T):
    # it needs the 64-column sums, which the rotation writes as a launch of its own only
    layer = random_layer_np(832, 272, 4, 64, 32, seed=T)
    d = lopro.make_desc(832, 272, 4, 64, 64, rank=32)
    with lopro.configured(lopro.OPT_NO_TCGEN05, 1):
        assert lopro.linear_fwd_path(d, T)[0] == lopro.PATH_GENERAL
        _check_forward_once(layer, d, synth.activations(T, 832, seed=T + 1), None, GATE_A, GATE_B)


@pytest.mark.parametrize("n,m,T", [(4096, 1024, 100), (1856, 912, 300)])
def test_the_fixed_scratch_takes_fewer_parts(n, m, T):
    # the workspace entry point wants more than the built-in scratch for its K parts; without a workspace fewer run
    layer = random_layer_np(n, m, 4, 64, 32, seed=n)
    d = lopro.make_desc(n, m, 4, 64, 64, rank=32)
    assert lopro.workspace_bytes(d, T) > lopro.NOALLOC_SCRATCH_BYTES
    blob = _pack(layer, d)
    x = bf16_bits_to_device(synth.activations(T, n, seed=T))
    want = lopro.linear_fwd(d, blob, x, lopro.OUT_F32)
    y = torch.empty_like(want)
    lopro.linear_fwd_noalloc(d, blob, x, y, lopro.OUT_F32)
    torch.cuda.synchronize()
    assert (y - want).abs().max().item() <= 1e-5 * want.abs().max().item()


# 1, 2, 4 and 8 token rows per CTA of the rotation (148 multiprocessors, up to 2048 columns), odd numbers of 16-column tiles in the prefix and of
# rotated blocks, and a last CTA with rows missing
@pytest.mark.parametrize("n,b_i,b_h", [(832, 64, 64), (320, 80, 16), (1088, 64, 256), (512, 0, 32), (448, 64, 128)])
@pytest.mark.parametrize("T", [16, 73, 75, 147, 149, 591, 593])
def test_rotation_with_every_number_of_rows_per_cta(n, b_i, b_h, T):
    got, exact, _, _ = _run_rotation(n, b_i, b_h, T, seed=T)
    assert np.all(np.abs(got - exact) <= _ulp_bf16(exact) + 1e-6 * np.abs(exact).max())


# the prologue's row CTAs of B x with two rows and 8, 4 or 2 tokens (more than eight tokens, by rows, columns and tokens), the
# last group of tokens short
# (25600 columns: past the default limit of shared memory; 8192 and 25600 at up to eight tokens: several passes at once)
@pytest.mark.parametrize("n,r,T", [(1024, 128, 21), (4096, 64, 30), (4160, 64, 32), (4096, 32, 17), (2560, 16, 31), (1024, 17, 27),
                                   (25600, 16, 17), (8192, 16, 1), (8256, 64, 3), (10304, 128, 8), (25600, 16, 2)])
def test_row_ctas_of_the_down_factor(n, r, T):
    layer = random_layer_np(n, 272, 4, 64, r, seed=n + T)
    d = lopro.make_desc(n, 272, 4, 64, 64, identity_cols=64, rank=r)
    _check_forward_once(layer, d, synth.activations(T, n, seed=T, outlier_frac=0.01), None, GATE_A, GATE_B)
