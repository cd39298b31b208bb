"""The persistent rank-1 sketch: every number of threads per row, resident rows and rows that stream, and the launches that
stand in for it, against the oracle; what is not finite gives zero triples and touches nothing else; a wait that gives up
is reported and leaves the matrix."""
import time

import numpy as np
import pytest
import torch

from oracle import lopro_oracle as o
from paper_2601_19675_b200 import lopro, synth

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _check_against_the_oracle(m, n, r, it):
    w = synth.weights(m, n, seed=m + n, spikes=r + 2)
    sk = synth.sketches(r, n, seed=5).astype(np.float32)
    wd = _dev(w.copy())
    ws = torch.zeros(lopro.r1svd_workspace_bytes(m, n), dtype=torch.uint8, device="cuda")
    U, sigma, V = lopro.r1svd(wd, r, it, _dev(sk), workspace=ws)
    torch.cuda.synchronize()
    assert lopro.workspace_status(ws) == lopro.OK
    u_ref, s_ref, v_ref = o.r1svd(w.astype(np.float64), r, it, sk.astype(np.float64))
    # the tolerances of the oracle test of r1svd: unit vectors absolutely, the remainder in the Frobenius norm
    np.testing.assert_allclose(sigma.cpu().numpy(), s_ref, rtol=2e-4)
    assert np.max(np.abs(U.cpu().numpy() - u_ref)) <= 5e-4 and np.max(np.abs(V.cpu().numpy() - v_ref)) <= 5e-4
    rem_ref = w.astype(np.float64) - (u_ref * s_ref[None, :]) @ v_ref
    assert np.linalg.norm(wd.cpu().numpy() - rem_ref) <= 1e-4 * np.linalg.norm(w)


# threads per row and float4 columns per thread by width (512, 1024, 2048, 4096, 8192, 12288 columns at most), the last four
# columns alone in theirs, fewer rows than CTAs, rows that stay in the ring and rows that stream, one group of threads and
# several, ranks in a second and a fourth warp of a row's threads
@pytest.mark.parametrize("m,n,r,it", [(60, 512, 20, 2), (15000, 512, 3, 2), (300, 516, 40, 1), (7500, 1024, 3, 2), (148, 1536, 40, 1),
                                      (4000, 2048, 3, 2), (300, 2052, 5, 2), (1800, 4096, 3, 1), (1000, 5000, 3, 2), (200, 8192, 20, 1),
                                      (700, 11008, 3, 2), (160, 12288, 33, 1), (256, 512, 128, 1), (256, 1536, 128, 0)])
def test_every_form_of_the_persistent_kernel(m, n, r, it):
    _check_against_the_oracle(m, n, r, it)


# rows past the persistent kernel's 12288 columns, ranks past its 128
@pytest.mark.parametrize("m,n,r,it", [(96, 12292, 3, 2), (160, 256, 129, 1)])
def test_the_launches_that_stand_in_for_the_persistent_kernel(m, n, r, it):
    _check_against_the_oracle(m, n, r, it)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("m,n", [(200, 512), (72, 2052)])
def test_an_entry_that_is_not_finite_gives_zero_triples_and_leaves_the_matrix(m, n, bad):
    w = synth.weights(m, n, seed=n)
    w[m // 2, 17] = bad
    for cast in (False, True):
        wd = _dev(w.copy())
        U, sigma, V = lopro.r1svd(wd, 3, 2, _dev(synth.sketches(3, n, seed=1).astype(np.float32)), cast=cast)
        torch.cuda.synchronize()
        assert not U.any() and not sigma.any() and not V.any()
        np.testing.assert_array_equal(wd.cpu().numpy(), w)


def test_a_sketch_vector_that_is_not_finite_costs_its_own_rank_only():
    m, n, r, it = 160, 1536, 5, 4
    w = synth.weights(m, n, seed=4, spikes=8)
    sk = synth.sketches(r, n, seed=2).astype(np.float32)
    keep = [0, 2, 4]
    sk[1, 5], sk[3, 9] = np.nan, np.inf
    U, sigma, V = lopro.r1svd(_dev(w.copy()), r, it, _dev(sk))
    torch.cuda.synchronize()
    assert not U[:, [1, 3]].any() and not sigma[[1, 3]].any() and not V[[1, 3]].any()
    u_ref, s_ref, v_ref = o.r1svd(w.astype(np.float64), len(keep), it, sk[keep].astype(np.float64))
    np.testing.assert_allclose(sigma.cpu().numpy()[keep], s_ref, rtol=2e-4)   # tolerances of the oracle test of r1svd
    assert np.max(np.abs(U.cpu().numpy()[:, keep] - u_ref)) <= 5e-4 and np.max(np.abs(V.cpu().numpy()[keep] - v_ref)) <= 5e-4


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("fp8", [False, True])
def test_a_bad_weight_spoils_its_own_group_only(fp8, bad):
    n, m, g = 512, 64, 64
    d = lopro.make_desc(n, m, 4, g, 64, identity_cols=n, rank=4,
                        lowrank_format=lopro.LOWRANK_FP8 if fp8 else lopro.LOWRANK_FOLDED_F16)
    w = synth.weights(m, n, seed=9)
    w[11, 200] = bad
    perm, sk = np.arange(n, dtype=np.int32), synth.sketches(4, n, seed=3).astype(np.float32)
    out = lopro.quantize_layer(d, _dev(w), _dev(perm), _dev(sk), it=2)
    torch.cuda.synchronize()
    assert lopro.workspace_status(out["workspace"]) == lopro.ERR_INVALID_DATA
    for name in ("U", "V", "sigma") if fp8 else ("A", "B"):
        assert not out[name].any()
    # without a low-rank part the residual is the matrix itself (no rotation here): the other groups are its grid
    codes, scales, zeros = (out[k].cpu().numpy() for k in ("codes", "scales", "zeros"))
    w[11, 192:256] = 0.0
    c_ref, s_ref, z_ref = o.rtn_quantize(w, 4, g, dtype=np.float32)
    ok = np.ones((m, n // g), dtype=bool)
    ok[11, 200 // g] = False
    np.testing.assert_array_equal(codes.reshape(m, -1, g)[ok], c_ref.reshape(m, -1, g)[ok])
    np.testing.assert_array_equal(scales.view(np.float16).astype(np.float64)[ok], s_ref[ok])
    np.testing.assert_array_equal(zeros.view(np.float16).astype(np.float64)[ok], z_ref[ok])
    assert not codes.reshape(m, -1, g)[~ok].any()


@pytest.mark.parametrize("m,n,r,it", [(4096, 4096, 64, 64), (16384, 512, 64, 64)])   # one and four groups of threads per CTA
def test_a_sketch_that_gives_up_reports_it_and_leaves_the_matrix(m, n, r, it):
    # what a wait that ran out does -- raise the abort flag, the highest bit of word 2 of the workspace -- is done from another
    # stream while the kernel runs (some 100 ms if nothing stops it): every CTA leaves at its next barrier
    w = torch.randn((m, n), device="cuda")
    keep, sk = w.clone(), torch.randn((r, n), device="cuda")
    ws = torch.zeros(lopro.r1svd_workspace_bytes(m, n), dtype=torch.uint8, device="cuda")
    flag = torch.tensor([-2 ** 31], dtype=torch.int32).pin_memory()
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    lopro.r1svd(w, r, it, sk, workspace=ws)
    done.record()
    time.sleep(0.02)
    assert not done.query()
    with torch.cuda.stream(other):
        ws[8:12].view(torch.int32).copy_(flag, non_blocking=True)
    torch.cuda.synchronize()
    assert lopro.workspace_status(ws) == lopro.ERR_TIMEOUT
    assert torch.equal(w, keep)
    # the next call on the same workspace starts over
    U, sigma, V = lopro.r1svd(w, 2, 1, sk[:2], workspace=ws)
    torch.cuda.synchronize()
    assert lopro.workspace_status(ws) == lopro.OK
    assert torch.dist(w + (U * sigma) @ V, keep).item() <= 1e-5 * keep.norm().item()
