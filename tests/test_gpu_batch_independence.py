"""An image's merged rows are the same bits alone, in a batch and in the groups of a host-buffer call: what else a
thread block has to do must not change the order of a sum."""
import numpy as np
import pytest
import torch

from paper_2411_17686_b200 import binding

pytestmark = pytest.mark.gpu


def images(seed, batch, n, dim, heads, dtype):
    """Tokens around a few dozen centres (so that some preserved tokens collect many sources) and attention."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    centres = torch.randn((40, dim), generator=g, device="cuda")
    near = torch.randint(0, 40, (batch, n), generator=g, device="cuda")
    x = centres[near] + 0.7 * torch.randn((batch, n, dim), generator=g, device="cuda")
    attn = torch.softmax(torch.randn((batch, heads, n), generator=g, device="cuda"), dim=2)
    return x.to(torch.float32 if dtype == "fp32" else torch.bfloat16).contiguous(), attn


CASES = [
    ("fp32", 16, 40, 40, 1024, 800, 2),      # several parts per row, hubs of every length
    ("fp32", 8, 24, 24, 4096, 64, None),     # rows wide enough for every warp to have a part
    ("bf16", 32, 24, 24, 1024, 96, 3),
    ("fp32", 160, 30, 37, 64, 4, 1),         # in the batch a block meets more sources than it files, alone it does not
]


@pytest.mark.parametrize("dtype,batch,gh,gw,dim,keep,k", CASES, ids=["half", "wide", "bf16", "rescan"])
def test_image_alone_and_in_a_batch(dtype, batch, gh, gw, dim, keep, k):
    n = gh * gw
    x, attn = images(3, batch, n, dim, 2, dtype)
    prm = binding.make_params(has_cls=False, max_targets=k)
    c = binding.Context(max_tokens=batch * n, max_dim=dim, max_batch=batch)
    try:
        def run(b0, b1):
            r = c.ficoco_v_reduce(x[b0:b1].reshape(-1, dim), attn[b0:b1].contiguous(), keep, gh, gw, 2, n_tokens=n, params=prm)
            return r.out_tokens.reshape(b1 - b0, keep, dim), r.kept_idx.reshape(b1 - b0, keep)

        out, kept = run(0, batch)
        for b0, b1 in [(0, 1), (batch - 1, batch), (1, 4)]:
            o, i = run(b0, b1)
            assert torch.equal(kept[b0:b1], i)
            assert torch.equal(out[b0:b1], o), f"images {b0}..{b1 - 1}: {int((out[b0:b1] != o).sum())} values differ"
        assert c.ficoco_status() == 0
    finally:
        c.close()


def test_host_groups_and_device_call():
    """fp32 tokens, whose sums no rounding to storage hides, in eight groups."""
    batch, gh, gw, dim, keep = 16, 40, 40, 1024, 800
    x, attn = images(4, batch, gh * gw, dim, 2, "fp32")
    prm = binding.make_params(has_cls=False, max_targets=2)
    c = binding.Context(max_tokens=batch * gh * gw, max_dim=dim, max_batch=batch)
    try:
        d = c.ficoco_v_reduce(x.reshape(-1, dim), attn, keep, gh, gw, 2, n_tokens=gh * gw, params=prm)
        torch.cuda.synchronize()
        h = c.ficoco_v_reduce_host(x.reshape(-1, dim).cpu().pin_memory(), attn.cpu().pin_memory(), keep, gh, gw, 2,
                                   n_tokens=gh * gw, params=prm)
        assert np.array_equal(binding.to_numpy(d.kept_idx), h.kept_idx.numpy())
        assert np.array_equal(binding.to_numpy(d.out_tokens), h.out_tokens.numpy())
    finally:
        c.close()
