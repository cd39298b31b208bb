"""Tensors without an address of their own -- batched by vmap, or fake -- are refused with an exception, in every per-call
entry point, and the interpreter goes on."""
import pytest
import torch
from torch._subclasses.fake_tensor import FakeTensorMode

from paper_2601_19675_b200 import lopro
from tests._layers import random_layer_np, to_device

pytestmark = pytest.mark.gpu

BF16 = torch.bfloat16


def _calls():
    n, m = 512, 128
    dev = to_device(random_layer_np(n, m, 4, 128, 16, seed=1))
    d = lopro.make_desc(n, m, 4, 128, 64, rank=16)
    blob = lopro.pack(d, dev["codes"], dev["scales"], dev["zeros"], dev["perm"], dev["A"], dev["B"])
    ws = torch.zeros(lopro.workspace_bytes(d, 4) * 4, dtype=torch.uint8, device="cuda")
    y, out = torch.empty((4, m), dtype=BF16, device="cuda"), torch.empty((4, n), dtype=BF16, device="cuda")
    w, st = torch.ones(n, dtype=BF16, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    cache = torch.zeros((4, 4, 8, 128), dtype=BF16, device="cuda")
    pos = torch.ones(4, dtype=torch.int32, device="cuda")
    return {
        "linear_fwd": lambda x: lopro.linear_fwd(d, blob, x, workspace=ws, y=y),
        "linear_fwd_noalloc": lambda x: lopro.linear_fwd_noalloc(d, blob, x, y),
        "linear_fwd_group": lambda x: lopro.linear_fwd_group([d, d], [blob, blob], x, workspace=ws, ys=[y, y.clone()]),
        "linear_fwd_experts": lambda x: lopro.linear_fwd_experts(d, [blob], [0, 4], x, workspace=ws, y=y),
        "rotate": lambda x: lopro.rotate(d, dev["perm"], x, out=out),
        "block_add_rmsnorm": lambda x: lopro.block_add_rmsnorm(x, None, w, 1e-5, out=out),
        "block_rope_append": lambda x: lopro.block_rope_append(x, x, x, pos, cache, cache, 10000.0, st),
        "block_attention_decode": lambda x: lopro.block_attention_decode(x, cache, cache, pos, 1.0, ws, st, out=out),
        "block_silu_mul": lambda x: lopro.block_silu_mul(x, x, out=out),
    }


@pytest.mark.parametrize("name", ["linear_fwd", "linear_fwd_noalloc", "linear_fwd_group", "linear_fwd_experts", "rotate",
                                  "block_add_rmsnorm", "block_rope_append", "block_attention_decode", "block_silu_mul"])
def test_a_tensor_without_an_address_is_refused(name):
    call = _calls()[name]
    x = torch.zeros((4, 512), dtype=BF16, device="cuda")
    with pytest.raises(RuntimeError):
        torch.vmap(call)(torch.stack([x, x]))
    with FakeTensorMode(allow_non_fake_inputs=True) as mode:
        fake = mode.from_tensor(x)
    with pytest.raises(RuntimeError):     # (lopro.LoproError is one)
        call(fake)
    call(x)                               # the same call with a tensor of its own
    torch.cuda.synchronize()
