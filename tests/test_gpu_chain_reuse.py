"""One activation buffer rewritten between forwards that start before its writer has ended: every kernel that reads it -- the
small-batch prologue, chunks of 32 tokens, the grid of rotation and B x, the vector-quantized chain -- takes the last
contents.  A run with a synchronisation after every call is the reference, bit for bit."""
import pytest
import torch

from paper_2601_19675_b200 import lopro, synth
from tests._layers import bf16_bits_to_device, random_layer_np, to_device
from tests.test_gpu_vq import _dev16, _random_record

pytestmark = pytest.mark.gpu


def _same_without_synchronising(forward, n, T, outs):
    h = bf16_bits_to_device(synth.activations(T, n, seed=3))
    w = [bf16_bits_to_device(synth.activations(1, n, seed=s))[0] for s in range(4, 4 + len(outs))]
    x = torch.empty_like(h)

    def chain(after_each):
        for k, y in enumerate(outs):
            lopro.block_add_rmsnorm(h, None, w[k], 1e-5, out=x)
            after_each()
            forward(x, y)
            after_each()
        torch.cuda.synchronize()
        got = [y.clone() for y in outs]
        for y in outs:
            y.zero_()
        return got

    want = chain(torch.cuda.synchronize)
    for _ in range(20):
        assert all(torch.equal(a, b) for a, b in zip(chain(lambda: None), want))


@pytest.mark.parametrize("T", [1, 2, 3, 5, 12, 33, 64, 150, 300, 600])
@pytest.mark.parametrize("n,r", [(2048, 64), (1088, 16)])
def test_linear_layers_on_a_reused_buffer(n, r, T):
    m = 1024
    layer = to_device(random_layer_np(n, m, 4, 64, r, seed=1))
    d = lopro.make_desc(n, m, 4, 64, 64, rank=r)
    blob = lopro.pack(d, layer["codes"], layer["scales"], layer["zeros"], layer["perm"], layer["A"], layer["B"])
    ws = torch.zeros(lopro.workspace_bytes(d, T), dtype=torch.uint8, device="cuda")
    outs = [torch.empty((T, m), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    _same_without_synchronising(lambda x, y: lopro.linear_fwd(d, blob, x, lopro.OUT_BF16, workspace=ws, y=y), n, T, outs)


@pytest.mark.parametrize("T", [1, 8, 20, 32, 40])
def test_vector_quantized_layers_on_a_reused_buffer(T):
    n, m, r = 1024, 1024, 16
    d = lopro.make_vq_desc(n, m, 512, 256, 64, rank=r)
    idx, books, perm, a, b = _random_record(n, m, 512, 256, r, seed=2)
    blob = lopro.vq_pack(d, torch.from_numpy(idx).cuda(), _dev16(books), torch.from_numpy(perm).cuda(), _dev16(a), _dev16(b))
    ws = torch.zeros(lopro.vq_workspace_bytes(d, T), dtype=torch.uint8, device="cuda")
    outs = [torch.empty((T, m), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    _same_without_synchronising(lambda x, y: lopro.vq_linear_fwd(d, blob, x, lopro.OUT_BF16, workspace=ws, y=y), n, T, outs)
