"""Residual, rotation and grid of the offline step with several rows per CTA: the same bits as one row per CTA and as the
steps one by one, at both numbers of rows, at widths that are no multiple of a warp's 256 columns, and where the kernel does
not apply (blocks or groups beyond a warp's columns)."""
import numpy as np
import pytest
import torch

from oracle import lopro_oracle as o
from paper_2601_19675_b200 import lopro, synth

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _layer(n, m, b_i, b_h, g, r, bits=4):
    d = lopro.make_desc(n, m, bits, g, b_h, identity_cols=b_i, rank=r)
    w = synth.weights(m, n, seed=n + m)
    w[1, :g], w[2, :g] = 0.375, -0.0123            # constant groups where the permutation leaves them together
    return d, w, synth.permutation(n, seed=n + 1)


# four rows per CTA up to 4608 columns, two beyond
@pytest.mark.parametrize("n,m,b_i,b_h,g,r", [(512, 48, 64, 64, 64, 16), (4608, 16, 128, 128, 128, 5), (4672, 16, 64, 64, 64, 17),
                                             (5184, 32, 64, 64, 64, 16), (11008, 16, 256, 256, 256, 32), (320, 16, 0, 2, 64, 3),
                                             (24576, 16, 128, 128, 128, 512), (640, 16, 640, 64, 64, 0)])
def test_rows_together_give_the_bits_of_a_row_alone(n, m, b_i, b_h, g, r):
    d, w, perm = _layer(n, m, b_i, b_h, g, r)
    a_bits, b_bits = synth.factors(m, n, max(r, 1), seed=n, std=0.05)
    af, bf = (_dev(o.f16_bits_to_f64(a_bits)[:, :r].astype(np.float32)), _dev(o.f16_bits_to_f64(b_bits)[:r].astype(np.float32))) if r else (None, None)
    together, st = lopro.residual_rotate(d, _dev(w), af, bf, _dev(perm))
    off = torch.empty(w.size + 1, dtype=torch.float32, device="cuda")[1:].view(w.shape)   # not on 16 bytes: a row at a time
    off.copy_(_dev(w))
    alone, st2 = lopro.residual_rotate(d, off, af, bf, _dev(perm))
    torch.cuda.synchronize()
    assert int(st.item()) == int(st2.item()) == lopro.OK
    assert torch.equal(together, alone)


@pytest.mark.parametrize("n,m,b_i,b_h,g,r,bits", [(1024, 48, 64, 64, 64, 8, 4), (5184, 32, 64, 64, 64, 4, 2), (11008, 32, 128, 128, 128, 8, 3),
                                                  (1024, 32, 0, 512, 128, 4, 4), (1024, 32, 128, 128, 512, 4, 2), (1216, 32, 192, 256, 64, 0, 3)])
def test_a_layer_in_one_call_has_the_bits_of_its_steps(n, m, b_i, b_h, g, r, bits):
    d, w, perm = _layer(n, m, b_i, b_h, g, r, bits)
    sk = synth.sketches(max(r, 1), n, seed=3).astype(np.float32)
    out = lopro.quantize_layer(d, _dev(w), _dev(perm), _dev(sk) if r else None, it=2)
    af, bf = (out["A"].view(torch.float16).float(), out["B"].view(torch.float16).float()) if r else (None, None)
    resid, _ = lopro.residual_rotate(d, _dev(w), af, bf, _dev(perm))
    codes, scales, zeros, _ = lopro.rtn_quantize(d, resid)
    torch.cuda.synchronize()
    assert lopro.workspace_status(out["workspace"]) == lopro.OK
    assert torch.equal(out["codes"], codes) and torch.equal(out["scales"], scales) and torch.equal(out["zeros"], zeros)
