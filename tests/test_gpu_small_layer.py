"""The layer in one launch of one cluster (layers whose weights fit its shared memory) against the four calls, every buffer bit for
bit: few and many tokens, fewer experts than CTAs, several experts per CTA, experts without rows and with more than one block of
eight, odd token counts, widths that are odd multiples of 128."""
import numpy as np
import pytest
import torch

from _gpu_util import bits, check_out, dev
from oracle import moe_oracle as O
from paper_2609_15627_b200 import inputs, moe

pytestmark = pytest.mark.gpu

SHAPES = [  # T, H, I, E, k
    (1, 256, 128, 8, 2), (16, 256, 128, 8, 2), (32, 256, 128, 8, 4), (31, 128, 128, 3, 3), (8, 256, 128, 32, 8), (17, 128, 128, 64, 4),
    (7, 384, 128, 9, 1), (5, 128, 640, 5, 2), (1, 1024, 128, 8, 8), (2, 128, 128, 60, 32)]


def _weights(H, I, E, seed=0):
    return tuple(dev(a) for a in inputs.make_expert_weights(H, I, E, seed=seed))


@pytest.mark.parametrize("T,H,I,E,k", SHAPES)
def test_small_layer_has_the_four_calls_bits(T, H, I, E, k):
    sh, w = moe.shape(T, H, I, E, k), _weights(H, I, E)
    logits, x = dev(inputs.make_logits(T, E, 11)), dev(inputs.make_x(T, H, 11))
    b, c = moe.LayerBuffers(sh), moe.LayerBuffers(sh)
    for buf in (b, c):
        for v in (buf.x_perm, buf.y_perm, buf.out, buf.topk_w):
            v.fill_(float("nan"))
        for v in (buf.topk_ids, buf.expert_offsets, buf.perm, buf.inv_perm):
            v.fill_(-7)
    moe.moe_layer(logits, x, w, b)
    assert moe.moe_last_kernel_name() == "layer_one_cluster"
    moe.moe_route(logits, k, c.topk_ids, c.topk_w, c.expert_offsets, c.ws)
    moe.moe_permute(x, c.topk_ids, c.expert_offsets, sh, c.x_perm, c.perm, c.inv_perm, c.ws)
    moe.moe_expert_ffn(c.x_perm, c.expert_offsets, *w, sh, c.y_perm, c.status, c.ws)
    assert moe.moe_last_kernel_name() == "ffn_stream_bulk_ring_mma16816"
    moe.moe_combine(c.y_perm, c.inv_perm, c.topk_w, sh, c.out)
    torch.cuda.synchronize()
    for n in ("topk_ids", "topk_w", "expert_offsets", "x_perm", "perm", "inv_perm", "y_perm", "out"):
        assert torch.equal(getattr(b, n), getattr(c, n)), n
    out = torch.empty_like(b.out)
    ids, wt, st = torch.empty_like(b.topk_ids), torch.empty_like(b.topk_w), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = moe.alloc_forward_workspace(sh)
    moe.moe_forward(logits, x, *w, sh, out, ids, wt, st, ws)
    packed = moe.moe_prepack(*w, sh)
    out_p = torch.empty_like(out)
    moe.moe_forward_packed(logits, x, packed, sh, out_p, None, None, st, ws)
    torch.cuda.synchronize()
    assert torch.equal(out, b.out) and torch.equal(out_p, b.out) and torch.equal(ids, b.topk_ids) and torch.equal(wt, b.topk_w) and int(st.item()) == 0


def test_small_layer_against_the_oracle_with_equal_logits_and_infinities():
    T, H, I, E, k = 9, 256, 128, 8, 3
    sh, raw = moe.shape(T, H, I, E, k), inputs.make_expert_weights(H, I, E, seed=4)
    logits, x = inputs.make_logits(T, E, 12), inputs.make_x(T, H, 12)
    logits[2] = 0.0                                   # ties: the lowest ids
    logits[3, :4] = np.float32(-3.0e38)
    logits[5, 1] = np.float32(3.0e38)
    buf = moe.LayerBuffers(sh)
    moe.moe_layer(dev(logits), dev(x), tuple(dev(a) for a in raw), buf)
    torch.cuda.synchronize()
    r = O.forward_staged(logits, x, *raw, k)
    assert np.array_equal(buf.topk_ids.cpu().numpy(), r["ids"]) and np.array_equal(buf.topk_w.cpu().numpy().view(np.uint32), r["w"].view(np.uint32))
    check_out(bits(buf.out), r["out"], r["out_f32"], "small layer")
    x[4, 7] = 0x7F80                                  # an infinite activation: that token's output is not finite, the others stay
    want = buf.out.clone()
    moe.moe_layer(dev(logits), dev(x), tuple(dev(a) for a in raw), buf)
    torch.cuda.synchronize()
    keep = torch.arange(T, device="cuda") != 4
    assert torch.equal(buf.out[keep], want[keep]) and not bool(torch.isfinite(buf.out[4].float()).all())


def test_small_layers_one_behind_the_other_in_a_graph():
    """Nothing but the layers' launches, each of which lets the next one start at once: a layer's rows are the one before's output, and
    its output lies where the one before reads its rows, so neither reads nor writes may be early."""
    T, H, I, E, k, n = 16, 256, 128, 8, 2, 40
    sh, w = moe.shape(T, H, I, E, k), _weights(H, I, E)
    lg = [dev(inputs.make_logits(T, E, 50 + i)) for i in range(n)]
    x0 = dev(inputs.make_x(T, H, 1))
    bufs = [moe.LayerBuffers(sh) for _ in range(2)]

    def chain():
        x = x0
        for i in range(n):
            x = moe.moe_layer(lg[i], x, w, bufs[i & 1])
            assert moe.moe_last_kernel_name() == "layer_one_cluster"
        return x

    chain()
    torch.cuda.synchronize()
    x = x0
    for i in range(n):   # one at a time
        x = moe.moe_layer(lg[i], x, w, bufs[i & 1]).clone()
        torch.cuda.synchronize()
    want = x
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            chain()
        for _ in range(20):
            g.replay()
            s.synchronize()
            assert torch.equal(bufs[(n - 1) & 1].out, want)


def test_small_layer_reads_weights_that_the_kernel_in_front_writes():
    """moe_combine lets its dependents go before it writes; here its output is the expert codes of the layer behind it."""
    T, H, I, E, k = 16, 256, 128, 8, 2
    sh, g = moe.shape(T, H, I, E, k), torch.Generator(device="cuda").manual_seed(9)
    _, s13, _, s2 = _weights(H, I, E)
    n13, n2 = E * H * I, E * H * I // 2               # bytes of the codes
    Tc, Hc = 4096, 4096                               # a combine that writes for a while, the codes last
    shc = moe.shape(Tc, Hc, 128, 1, 1)
    ys = [torch.randn((Tc, Hc), device="cuda", generator=g).to(torch.bfloat16) for _ in range(2)]
    inv, one = torch.arange(Tc, dtype=torch.int32, device="cuda"), torch.ones(Tc, device="cuda")

    def codes(out):
        tail = out.view(torch.uint8).reshape(-1)[-(n13 + n2):]
        return tail[:n13].view(E, 2 * I, H // 2), s13, tail[n13:].view(E, H, I // 2), s2

    logits, x = dev(inputs.make_logits(T, E, 13)), dev(inputs.make_x(T, H, 13))
    b, want = moe.LayerBuffers(sh), []
    for y in ys:
        moe.moe_layer(logits, x, tuple(v.clone() for v in codes(y)), b)
        torch.cuda.synchronize()
        want.append(b.out.clone())
    assert moe.moe_last_kernel_name() == "layer_one_cluster" and not torch.equal(want[0], want[1])
    yf, out = [y.float() for y in ys], torch.zeros_like(ys[0])
    w, got = codes(out), []
    for i in (0, 1, 0, 1, 1, 0):
        moe.moe_combine(yf[i], inv, one, shc, out)
        moe.moe_layer(logits, x, w, b)
        got.append((i, b.out.clone()))
    torch.cuda.synchronize()
    for i, o in got:
        assert torch.equal(o, want[i])


@pytest.mark.parametrize("T,H,I,E,k,one", [
    (32, 512, 128, 8, 4, True), (32, 512, 128, 4, 4, False), (32, 512, 128, 4, 2, True), (31, 384, 256, 8, 4, False), (32, 640, 128, 3, 2, False)])
def test_small_layer_up_to_a_cta_s_share_of_the_work(T, H, I, E, k, one):
    """Either side of the line (2^20 weights times rows per CTA with an expert): the same bits by either path."""
    sh, w = moe.shape(T, H, I, E, k), _weights(H, I, E)
    logits, x = dev(inputs.make_logits(T, E, 15)), dev(inputs.make_x(T, H, 15))
    b, c = moe.LayerBuffers(sh), moe.LayerBuffers(sh)
    b.out.fill_(float("nan"))
    moe.moe_layer(logits, x, w, b)
    assert (moe.moe_last_kernel_name() == "layer_one_cluster") == one
    moe.moe_route(logits, k, c.topk_ids, c.topk_w, c.expert_offsets, c.ws)
    moe.moe_permute(x, c.topk_ids, c.expert_offsets, sh, c.x_perm, c.perm, c.inv_perm, c.ws)
    moe.moe_expert_ffn(c.x_perm, c.expert_offsets, *w, sh, c.y_perm, c.status, c.ws)
    assert moe.moe_last_kernel_name() == "ffn_stream_bulk_ring_mma16816"
    moe.moe_combine(c.y_perm, c.inv_perm, c.topk_w, sh, c.out)
    torch.cuda.synchronize()
    assert torch.equal(b.out, c.out) and torch.equal(b.y_perm, c.y_perm)
