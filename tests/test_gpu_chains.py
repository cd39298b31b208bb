"""Launches that follow one another without a synchronisation: buffers reused inside a chain of early-launched kernels,
host buffers read and written in place, and attention at the edges of its split over half-warps and CTAs."""
import numpy as np
import pytest
import torch

from oracle import glue_oracle as g
from oracle import lopro_oracle as o
from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, device_bf16_to_f64, random_layer_np, to_device

pytestmark = pytest.mark.gpu


def _layer(n, m, seed, rank=32):
    dev = to_device(random_layer_np(n, m, 4, 128, rank, seed=seed))
    d = lopro.make_desc(n, m, 4, 128, 128, rank=rank)
    return d, lopro.pack(d, dev["codes"], dev["scales"], dev["zeros"], dev["perm"], dev["A"], dev["B"])


@pytest.mark.parametrize("T", [1, 8, 16, 32])
def test_a_buffer_rewritten_inside_a_chain_is_read_as_last_written(T):
    # two norms share one output buffer, as in a decoder layer; each feeds a group of linear layers
    n, m = 4096, 2048
    (d, a), (_, b) = _layer(n, m, 1), _layer(n, m, 2)
    h = bf16_bits_to_device(synth.activations(T, n, seed=3))
    w = [bf16_bits_to_device(synth.activations(1, n, seed=s))[0] for s in (4, 5)]
    xn = torch.empty_like(h)
    ws = torch.zeros(lopro.group_workspace_bytes([d, d], T), dtype=torch.uint8, device="cuda")
    ys = [[torch.empty((T, m), dtype=torch.bfloat16, device="cuda") for _ in range(2)] for _ in range(2)]

    def chain(synced):
        for k in range(2):
            lopro.block_add_rmsnorm(h, None, w[k], 1e-5, out=xn)
            if synced:
                torch.cuda.synchronize()
            lopro.linear_fwd_group([d, d], [a, b], xn, lopro.OUT_BF16, workspace=ws, ys=ys[k])
            if synced:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return [y.clone() for pair in ys for y in pair]

    want = chain(True)
    for _ in range(20):
        assert all(torch.equal(x, y) for x, y in zip(chain(False), want))


# pairs of (sequence, head) on both sides of every cluster size the launch chooses
@pytest.mark.parametrize("H", [1, 4, 8, 16, 32, 46, 57, 92])   # (from 46 on more pairs than one wave: 6, 149 and 12 in the last)
def test_attention_at_the_edges_of_its_splits(H):
    ctx = np.array([1, 2, 7, 8, 9, 31, 32, 33, 64, 65, 255, 257, 300], dtype=np.int32)
    T, hd, ctx_max = len(ctx), 128, 300
    gen = np.random.Generator(np.random.Philox(key=[H, 3]))
    qb, kb, vb = (synth.f32_to_bf16_bits(gen.standard_normal(s, dtype=np.float32))
                  for s in ((T, H * hd), (T, H, ctx_max, hd), (T, H, ctx_max, hd)))
    ws = torch.empty(lopro.block_attention_workspace_bytes(T, H, hd, ctx_max), dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    scale = hd ** -0.5
    out = lopro.block_attention_decode(bf16_bits_to_device(qb), bf16_bits_to_device(kb), bf16_bits_to_device(vb),
                                       torch.from_numpy(ctx).cuda(), scale, ws, st)
    torch.cuda.synchronize()
    assert int(st.item()) == lopro.OK
    ref = g.attention_decode(o.bf16_bits_to_f64(qb).reshape(T, H, hd), o.bf16_bits_to_f64(kb), o.bf16_bits_to_f64(vb), ctx, scale)
    got = device_bf16_to_f64(out).reshape(T, H, hd)
    assert np.max(np.abs(got - ref)) <= 2.0 ** -8 * np.abs(ref).max() + 1e-4


@pytest.mark.parametrize("d", [8, 4096, 4104, 12288])
def test_rmsnorm_of_unaligned_rows(d):
    # rows that do not start on 16 bytes take two-byte accesses; results are those of aligned rows
    T = 3
    hb, yb = synth.activations(T, d, seed=1), synth.activations(T, d, seed=2)
    w = bf16_bits_to_device(synth.activations(1, d, seed=3))[0]
    h, y = bf16_bits_to_device(hb), bf16_bits_to_device(yb)
    want = lopro.block_add_rmsnorm(h, y, w, 1e-5)
    wide = torch.zeros((T, d + 3), dtype=torch.bfloat16, device="cuda")
    h2 = wide[:, 1:1 + d]
    h2.copy_(bf16_bits_to_device(hb))
    got = lopro.block_add_rmsnorm(h2, y, w, 1e-5)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and torch.equal(h2, h)
    assert torch.all(wide[:, 0] == 0) and torch.all(wide[:, 1 + d:] == 0)


@pytest.mark.parametrize("T", [1, 8, 40, 260])     # 260 rows: activations beyond the size that kernels copy
@pytest.mark.parametrize("where", ["pinned", "pageable", "pinned, unaligned"])
def test_host_buffers_in_place_or_copied(T, where):
    n, m = 2048, 512
    d, blob = _layer(n, m, 7)
    xb = synth.activations(T, n, seed=T)
    x = torch.from_numpy(xb.view(np.int16)).view(torch.bfloat16)

    def host(shape):
        off = 1 if "unaligned" in where else 0
        flat = torch.zeros(shape[0] * shape[1] + off, dtype=torch.bfloat16)
        flat = flat.pin_memory() if "pinned" in where else flat
        return flat[off:].view(shape)

    xh, yh = host((T, n)), host((T, m))
    ws = torch.zeros(lopro.workspace_bytes(d, T) + lopro.host_staging_bytes(d, T), dtype=torch.uint8, device="cuda")
    want = lopro.linear_fwd(d, blob, x.cuda())
    for _ in range(3):                              # other contents of the same buffer in between
        xh.copy_(-x)
        lopro.linear_fwd_host(d, blob, xh, yh, ws)
        torch.cuda.synchronize()
        xh.copy_(x)
        lopro.linear_fwd_host(d, blob, xh, yh, ws)
        torch.cuda.synchronize()
        assert torch.equal(yh, want.cpu())
