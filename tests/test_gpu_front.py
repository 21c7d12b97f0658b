"""Routing and sort of batches that no cluster routes, against the oracle: the layer's front (router, then the sort with the offsets
as its by-product) and the separate calls (router and offsets; count and scatter), at the lines between their forms."""
import numpy as np
import pytest
import torch

from _gpu_util import dev
from oracle import moe_oracle as O
from paper_2609_15627_b200 import inputs, moe

pytestmark = pytest.mark.gpu


def _check(logits, k, buf, x=None):
    ids, w, off = O.route(logits, k)
    assert np.array_equal(buf.topk_ids.cpu().numpy(), ids) and np.array_equal(buf.topk_w.cpu().numpy().view(np.uint32), w.view(np.uint32))
    assert np.array_equal(buf.expert_offsets.cpu().numpy(), off)
    perm = np.argsort(ids.reshape(-1), kind="stable")
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))
    assert np.array_equal(buf.perm.cpu().numpy(), perm) and np.array_equal(buf.inv_perm.cpu().numpy().reshape(-1), inv)
    if x is not None:
        assert np.array_equal(buf.x_perm.view(torch.int16).cpu().numpy().view(np.uint16), x[perm // k])


FRONTS = [  # T, E, k
    (257, 256, 8), (512, 256, 8), (513, 256, 8), (1365, 40, 3), (1366, 40, 3),   # up to 4096 slots and beyond
    (300, 10, 5), (2100, 10, 2), (2049, 33, 2),                                  # numbers of experts that are no multiple of four
    (33, 300, 8), (600, 300, 8), (40, 1024, 32), (4100, 1024, 1), (5000, 1, 1), (9001, 8, 8)]


@pytest.mark.parametrize("T,E,k", FRONTS)
def test_front_of_a_layer(T, E, k):
    H, I = 128, 128
    sh = moe.shape(T, H, I, E, k)
    logits, x = inputs.make_logits(T, E, 21), inputs.make_x(T, H, 22)
    logits[0] = 0.25                                      # ties, the lowest ids first
    logits[T // 2, : E // 2 + 1] = np.float32(-0.0)
    logits[T - 1, 0] = np.float32(3.0e38)
    logits[T - 1, E - 1] = np.float32(-3.0e38)
    w = tuple(dev(a) for a in inputs.make_expert_weights(H, I, E, seed=1))
    buf = moe.LayerBuffers(sh)
    for _ in range(2):                                    # twice on one workspace, which holds anything before
        buf.ws.fill_(0xA5)
        for v in (buf.topk_ids, buf.expert_offsets, buf.perm, buf.inv_perm):
            v.fill_(-7)
        moe.moe_layer(dev(logits), dev(x), w, buf)
        torch.cuda.synchronize()
        assert int(buf.status.item()) == 0
        _check(logits, k, buf, x)


@pytest.mark.parametrize("T,E,k", [(257, 256, 8), (512, 256, 8), (513, 256, 8), (1537, 256, 8), (4100, 1024, 1), (2000, 37, 6), (60, 300, 4)])
def test_separate_calls(T, E, k):
    H = 128
    sh = moe.shape(T, H, 128, E, k)
    logits, x = inputs.make_logits(T, E, 31), inputs.make_x(T, H, 32)
    buf = moe.LayerBuffers(sh)
    for _ in range(2):
        buf.ws.fill_(0xA5)
        moe.moe_route(dev(logits), k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
        moe.moe_permute(dev(x), buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
        torch.cuda.synchronize()
        _check(logits, k, buf, x)


@pytest.mark.parametrize("T", [65536, 65664])
def test_sort_of_the_most_chunks_the_scatter_sums_itself_and_beyond(T):
    E, k, H = 16, 8, 128
    sh = moe.shape(T, H, 128, E, k)
    g = torch.Generator(device="cuda").manual_seed(5)
    logits = torch.randn((T, E), device="cuda", generator=g)
    x = torch.randn((T, H), device="cuda", generator=g).to(torch.bfloat16)
    buf = moe.LayerBuffers(sh)
    moe.moe_route(logits, k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(x, buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
    torch.cuda.synchronize()
    flat = buf.topk_ids.reshape(-1).long()
    want = torch.argsort(flat, stable=True)
    assert torch.equal(buf.topk_ids.long(), torch.sort(logits, dim=1, descending=True, stable=True).indices[:, :k])
    assert torch.equal(buf.expert_offsets.long(), torch.cat([torch.zeros(1, dtype=torch.long, device="cuda"), torch.bincount(flat, minlength=E).cumsum(0)]))
    assert torch.equal(buf.perm.long(), want) and torch.equal(buf.inv_perm.reshape(-1).long()[want], torch.arange(T * k, device="cuda"))
    assert torch.equal(buf.x_perm, x[want // k])
