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


def _gpu_weights(g, H, I, E):
    def codes(rows, K):
        return torch.randint(0, 256, (E, rows, K // 2), dtype=torch.uint8, device="cuda", generator=g)

    def scales(rows, K):
        return torch.randint(119, 123, (E, rows, K // 32), dtype=torch.uint8, device="cuda", generator=g)

    return codes(2 * I, H), scales(2 * I, H), codes(H, I), scales(H, I)


# every kernel that may follow the front (only the eight-term one reads the offsets before it waits), above 256 tokens and above 256 experts
NATIVE, TWOTERM = "ffn_native_mxf4_block_scaled", "ffn_mxf8_two_term_cta_pair"
FOLLOWERS = [  # T, H, I, E, k, kernel
    (40, 1024, 512, 512, 8, NATIVE), (300, 1024, 512, 256, 2, NATIVE), (257, 256, 256, 64, 6, NATIVE), (40, 512, 512, 300, 8, NATIVE),
    (300, 512, 256, 256, 8, TWOTERM), (1366, 256, 256, 256, 3, TWOTERM), (512, 512, 512, 8, 2, "ffn_umma_tcgen05_grouped"),
    (300, 384, 256, 40, 3, "ffn_stream_bulk_ring_mma16816")]


@pytest.mark.parametrize("T,H,I,E,k,kernel", FOLLOWERS)
def test_expert_ffn_behind_the_front(T, H, I, E, k, kernel):
    """Batches of other routings one behind the other on one workspace, nothing waited for between the calls: the offsets of a call
    are never the last one's.  Every call has the separate calls' bits."""
    sh = moe.shape(T, H, I, E, k)
    g = torch.Generator(device="cuda").manual_seed(T)
    w, shared = _gpu_weights(g, H, I, E), _gpu_weights(g, H, I, 1)
    wr = (torch.randn((E, H), device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    n = 4
    x = [torch.randn((T, H), device="cuda", generator=g).to(torch.bfloat16) for _ in range(n)]
    slope = torch.linspace(-4.0, 4.0, E, device="cuda")
    lg = [torch.randn((T, E), device="cuda", generator=g) + slope * s for s in (0.0, 1.0, -1.0, 0.5)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    c, want, want_block = moe.LayerBuffers(sh), [], []
    sh1, off1 = moe.shape(T, H, I, 1, 1), torch.tensor([0, T], dtype=torch.int32, device="cuda")
    ys, ws1, lgb = torch.empty((T, H), device="cuda"), moe.alloc_workspace(moe.shape(T, H, I, 1, 1)), torch.empty((T, E), device="cuda")

    def separate(logits, rows):
        moe.moe_route(logits, k, c.topk_ids, c.topk_w, c.expert_offsets, c.ws)
        moe.moe_permute(rows, c.topk_ids, c.expert_offsets, sh, c.x_perm, c.perm, c.inv_perm, c.ws)
        torch.cuda.synchronize()
        moe.moe_expert_ffn(c.x_perm, c.expert_offsets, *w, sh, c.y_perm, c.status, c.ws)
        assert moe.moe_last_kernel_name() == kernel

    for i in range(n):
        separate(lg[i], x[i])
        moe.moe_combine(c.y_perm, c.inv_perm, c.topk_w, sh, c.out)
        torch.cuda.synchronize()
        want.append([v.clone() for v in (c.out, c.y_perm, c.expert_offsets, c.perm, c.x_perm)])
        moe.moe_router_logits(x[i], wr, lgb, c.status)
        separate(lgb, x[i])
        moe.moe_expert_ffn(x[i], off1, *shared, sh1, ys, c.status, ws1)
        moe.moe_combine_shared(c.y_perm, c.inv_perm, c.topk_w, ys, sh, c.out)
        torch.cuda.synchronize()
        want_block.append(c.out.clone())
    assert int(c.status.item()) == 0
    assert not torch.equal(want[0][2], want[1][2]) and not torch.equal(want[1][2], want[2][2])

    order = [0, 1, 2, 3, 1, 0, 3, 2] * 2
    b, got = moe.LayerBuffers(sh), []
    for i in order:
        moe.moe_layer(lg[i], x[i], w, b)
        got.append([v.clone() for v in (b.out, b.y_perm, b.expert_offsets, b.perm, b.x_perm)])
    torch.cuda.synchronize()
    assert int(b.status.item()) == 0
    for i, r in zip(order, got):
        for name, u, v in zip(("out", "y_perm", "expert_offsets", "perm", "x_perm"), r, want[i]):
            assert torch.equal(u, v), ("moe_layer", name, i)

    ws, packed = moe.alloc_forward_workspace(sh), moe.moe_prepack(*w, sh)
    moe.moe_expert_ffn_packed(c.x_perm, c.expert_offsets, packed, sh, c.y_perm, c.status, c.ws)
    assert moe.moe_last_kernel_name() == kernel
    outs = [torch.empty_like(b.out) for _ in order]
    for i, o in zip(order, outs):
        moe.moe_forward_packed(lg[i], x[i], packed, sh, o, None, None, status, ws)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, o in zip(order, outs):
        assert torch.equal(o, want[i][0]), ("moe_forward_packed", i)

    wsb = moe.alloc_block_workspace(sh)
    for i, o in zip(order, outs):
        moe.moe_ffn_block(x[i], wr, w, shared, sh, o, None, None, status, wsb)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, o in zip(order, outs):
        assert torch.equal(o, want_block[i]), ("moe_ffn_block", i)
