"""GPU parity of the steps either side of the routed path - router projection, shared expert, join - and of the FFN block
they make with it (paper, figure "Execution structure"), against the CPU oracle, through the C ABI."""
import numpy as np
import pytest
import torch

from _gpu_util import bits, check_out, check_y, dev, weights_dev
from oracle import moe_oracle as O
from paper_2609_15627_b200 import inputs, moe

pytestmark = pytest.mark.gpu

bf = inputs.bf16_bits_to_f32


def _router_weights(E, H, seed):
    return inputs.f32_to_bf16_bits(bf(inputs.make_x(E, H, seed)) * np.float32(0.03))


@pytest.mark.parametrize("T,H,E,kernel", [
    (1, 4096, 256, "router_gemv_warp_per_expert"), (7, 512, 8, "router_gemv_warp_per_expert"),
    (16, 1024, 100, "router_gemv_warp_per_expert"), (17, 512, 64, "router_gemm_tcgen05_128x64"),
    (200, 512, 40, "router_gemm_tcgen05_128x64"), (1000, 1024, 256, "router_gemm_tcgen05_128x64"),
    (64, 4096, 256, "router_gemm_tcgen05_128x64"), (300, 256, 1024, "router_gemm_tcgen05_128x64")])
def test_router_logits_against_oracle(T, H, E, kernel):
    x, wr = inputs.make_x(T, H, 3), _router_weights(E, H, 4)
    lg = torch.full((T, E), float("nan"), dtype=torch.float32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    moe.moe_router_logits(dev(x), dev(wr), lg, st)
    torch.cuda.synchronize()
    assert moe.moe_last_kernel_name() == kernel and int(st.item()) == 0
    ref = O.router_logits(x, wr)
    got = lg.cpu().numpy()
    # both sum exact products in fp32, in different orders: each is within H * 2^-24 * sum |terms| of the true value
    bound = 2 * H * 2.0 ** -24 * (np.abs(bf(x).astype(np.float64)) @ np.abs(bf(wr).astype(np.float64)).T) + 1e-30
    assert np.isfinite(got).all() and np.all(np.abs(got.astype(np.float64) - ref) <= bound)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-5


def test_router_logits_exact_on_small_integers():
    # every partial sum is an integer below 2^24: any summation order gives the exact result
    rng = np.random.default_rng(0)
    for T in (3, 150):
        xi = rng.integers(-8, 9, (T, 512)).astype(np.float32)
        wi = rng.integers(-8, 9, (72, 512)).astype(np.float32)
        lg = torch.empty((T, 72), dtype=torch.float32, device="cuda")
        moe.moe_router_logits(dev(inputs.f32_to_bf16_bits(xi)), dev(inputs.f32_to_bf16_bits(wi)), lg)
        torch.cuda.synchronize()
        assert np.array_equal(lg.cpu().numpy().astype(np.int64), xi.astype(np.int64) @ wi.astype(np.int64).T)


@pytest.mark.parametrize("T,H,k", [(16, 256, 2), (1, 4096, 8), (1000, 512, 6)])
def test_combine_shared_bit_exact_given_oracle_inputs(T, H, k):
    rng = np.random.default_rng(1)
    y = (rng.standard_normal((T * k, H)) * 10).astype(np.float32)
    ys = (rng.standard_normal((T, H)) * 10).astype(np.float32)
    w = rng.random((T, k)).astype(np.float32)
    inv = rng.permutation(T * k).astype(np.int32)
    out = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    moe.moe_combine_shared(dev(y), dev(inv), dev(w), dev(ys), moe.shape(T, H, 128, 8, k), out)
    torch.cuda.synchronize()
    ref, _ = O.combine_shared(y, inv, w, ys)
    assert np.array_equal(bits(out), ref)


def _run_block(wl, x, wr, routed, shared, rdev=None):
    sh = moe.shape(wl.T, wl.H, wl.I, wl.E, wl.k)
    ws = moe.alloc_block_workspace(sh)
    out = torch.full((wl.T, wl.H), float("nan"), dtype=torch.bfloat16, device="cuda")
    ids = torch.empty((wl.T, wl.k), dtype=torch.int32, device="cuda")
    w = torch.empty((wl.T, wl.k), dtype=torch.float32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    rdev = rdev if rdev is not None else tuple(dev(a) for a in routed)
    sdev = tuple(dev(a) for a in shared)
    xd, wrd = dev(x), dev(wr)
    for _ in range(2):   # twice on one workspace
        moe.moe_ffn_block(xd, wrd, rdev, sdev, sh, out, ids, w, st, ws)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
    logits = ws[:wl.T * wl.E * 4].view(torch.float32).reshape(wl.T, wl.E).cpu().numpy()   # the block keeps them first in ws
    return out, ids.cpu().numpy(), w.cpu().numpy(), logits


def _check_block(wl, seed, routed=None, rdev=None, sample=None):
    routed = routed if routed is not None else inputs.make_expert_weights(wl.H, wl.I, wl.E, seed=0)
    shared = inputs.make_expert_weights(wl.H, wl.I, 1, seed=21)
    x, wr = inputs.make_x(wl.T, wl.H, seed), _router_weights(wl.E, wl.H, seed + 1)
    out, ids, w, logits = _run_block(wl, x, wr, routed, shared, rdev)
    ref_logits = O.router_logits(x, wr)
    assert np.linalg.norm(logits - ref_logits) / np.linalg.norm(ref_logits) < 1e-5
    # everything after the projection is checked on the logits the GPU computed (a last-bit difference in a logit may
    # legitimately change a near-tie of the Top-k)
    if sample is None:
        r = O.ffn_block(x, wr, *routed, *shared, wl.k, logits=logits)
        assert np.array_equal(ids, r["ids"]) and np.array_equal(w.view(np.uint32), r["w"].view(np.uint32))
        return check_out(bits(out), r["out"], r["out_f32"], wl.name)
    rids, rw, _ = O.route(logits, wl.k)
    assert np.array_equal(ids, rids) and np.array_equal(w.view(np.uint32), rw.view(np.uint32))
    tok = np.array(sample, np.int32)
    rt = O.forward_tokens(logits, x, *routed, wl.k, tok)
    ys = O.shared_expert(np.ascontiguousarray(x[tok]), *shared)
    want_f32 = (rt["out_f32"].astype(np.float64) + ys.astype(np.float64)).astype(np.float32)
    got = bits(out[torch.from_numpy(tok.astype(np.int64)).cuda()])
    return check_out(got, inputs.f32_to_bf16_bits(want_f32), want_f32, wl.name)


@pytest.mark.parametrize("T,H,I,E,k", [
    (16, 256, 128, 8, 2),      # streaming expert kernel for both calls
    (4, 512, 512, 8, 2),       # decode-sized kernel, router by warps
    (24, 1024, 512, 32, 6),    # decode-sized routed call, shared call of 24 rows on one expert
    (512, 512, 512, 8, 2),     # prefill-sized routed call, router GEMM
    (1100, 512, 512, 16, 6),   # prefill-sized kernel for both calls
    (1, 512, 512, 8, 2),       # one token: the router projection, then one launch with the shared expert as a third slot
    (1, 1024, 512, 16, 6),
    (1, 512, 1024, 4, 4)])
def test_ffn_block_small_shapes(T, H, I, E, k):
    _check_block(inputs.Workload("block", T, H, I, E, k), seed=5)
    if T == 1:
        assert moe.moe_last_kernel_name() == "block_one_launch_mxf4_pair_split_k"


@pytest.mark.parametrize("name", ["decode_c1", "decode_c64"])
def test_ffn_block_production_decode(name):
    wl = inputs.WORKLOADS[name]
    _check_block(wl, seed=7)
    if wl.T == 1:   # 9 slots x 16 CTAs on 144 of the 148 SMs
        assert moe.moe_last_kernel_name() == "block_one_launch_mxf4_pair_split_k"


def test_ffn_block_prefill_8k_sampled():
    wl = inputs.WORKLOADS["prefill_8k"]
    rng = np.random.default_rng(0)
    _check_block(wl, seed=9, sample=sorted(set([0, wl.T - 1] + rng.integers(0, wl.T, 30).tolist())))


# The calls that read logits before they wait (up to 32 tokens) directly behind the projection that writes them, queued up in a
# graph: every pair finds the logits of other tokens, or ones that choose other experts, in the buffer
@pytest.mark.parametrize("T", [1, 2, 16, 17, 32])
@pytest.mark.parametrize("call", ["route", "layer", "forward"])
def test_what_follows_the_router_projection_reads_its_logits(T, call):
    H, I, E, k = 4096, 256, 32, 4
    sh = moe.shape(T, H, I, E, k)
    w = tuple(dev(a) for a in inputs.make_expert_weights(H, I, E, seed=0))
    wr, xs = dev(_router_weights(E, H, 5)), [dev(inputs.make_x(T, H, 50 + i)) for i in range(6)]
    lg, buf, fws = torch.empty((T, E), device="cuda"), moe.LayerBuffers(sh), moe.alloc_forward_workspace(sh)
    ids = [torch.zeros((T, k), dtype=torch.int32, device="cuda") for _ in xs]
    outs = [torch.zeros((T, H), dtype=torch.bfloat16, device="cuda") for _ in xs]

    def pair(x, ids, out):
        moe.moe_router_logits(x, wr, lg, buf.status)
        if call == "route":
            moe.moe_route(lg, k, ids, buf.topk_w, buf.expert_offsets, buf.ws)
        elif call == "layer":
            buf.topk_ids, buf.out = ids, out
            moe.moe_layer(lg, x, w, buf)
        else:
            moe.moe_forward(lg, x, *w, sh, out, ids, buf.topk_w, buf.status, fws)
    want = []
    for x, i, o in zip(xs, ids, outs):
        pair(x, i, o)
        torch.cuda.synchronize()
        want.append((O.route(lg.cpu().numpy(), k)[0], o.clone()))
        assert np.array_equal(i.cpu().numpy(), want[-1][0])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for a in zip(xs, ids, outs):
            pair(*a)
    for _ in range(5):
        lg.copy_(torch.arange(E, device="cuda").expand(T, E))
        for t in (*ids, *outs):
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert int(buf.status.item()) == 0
        for (wi, wo), i, o in zip(want, ids, outs):
            assert np.array_equal(i.cpu().numpy(), wi) and torch.equal(o.view(torch.int16), wo.view(torch.int16))


# Up to 256 tokens the shared expert, the router projection and the routing run beside one another: the block is its steps, bit for
# bit, also where calls follow one another on one workspace and in a graph (17 tokens: router GEMM; above 32 the shared expert's
# kernel is another)
@pytest.mark.parametrize("T,H,I,E,k", [(4, 1024, 512, 32, 4), (17, 1024, 512, 64, 6), (48, 4096, 2048, 16, 6), (130, 4096, 2048, 32, 2), (256, 512, 512, 64, 8)])
def test_ffn_block_is_its_steps(T, H, I, E, k):
    routed = tuple(dev(a) for a in inputs.make_expert_weights(H, I, E, seed=0))
    shared = tuple(dev(a) for a in inputs.make_expert_weights(H, I, 1, seed=21))
    wr = dev(_router_weights(E, H, 3))
    sh, sh1 = moe.shape(T, H, I, E, k), moe.shape(T, H, I, 1, 1)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    xs, want = [dev(inputs.make_x(T, H, 30 + i)) for i in range(3)], []
    buf, lg, ys = moe.LayerBuffers(sh), torch.empty((T, E), device="cuda"), torch.empty((T, H), device="cuda")
    off2, ws1 = torch.tensor([0, T], dtype=torch.int32, device="cuda"), moe.alloc_workspace(sh1)
    for x in xs:
        moe.moe_router_logits(x, wr, lg, st)
        moe.moe_layer(lg, x, routed, buf)
        moe.moe_expert_ffn(x, off2, *shared, sh1, ys, st, ws1)
        moe.moe_combine_shared(buf.y_perm, buf.inv_perm, buf.topk_w, ys, sh, buf.out)
        torch.cuda.synchronize()
        want.append(buf.out.clone())
    ws, ids, w = moe.alloc_block_workspace(sh), torch.empty((T, k), dtype=torch.int32, device="cuda"), torch.empty((T, k), device="cuda")
    outs = [torch.empty((T, H), dtype=torch.bfloat16, device="cuda") for _ in range(9)]

    def calls():
        for i, o in enumerate(outs):
            moe.moe_ffn_block(xs[i % 3], wr, routed, shared, sh, o, ids, w, st, ws)
    calls()
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and all(torch.equal(o.view(torch.int16), want[i % 3].view(torch.int16)) for i, o in enumerate(outs))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    for o in outs:
        o.zero_()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and all(torch.equal(o.view(torch.int16), want[i % 3].view(torch.int16)) for i, o in enumerate(outs))


# The same with what a network does around it: the rows are rewritten in place between calls, in stream order only; blocks of
# them that two terms hold too little of, so that a shared expert on the two-term kernel is done again behind the join; and
# without a status word, where the steps run one after the other
@pytest.mark.parametrize("T,H,I,E,k,again", [(4, 1024, 512, 32, 4, False), (20, 1024, 512, 32, 4, False), (48, 4096, 2048, 16, 6, True),
                                             (130, 4096, 2048, 32, 2, True)])
@pytest.mark.parametrize("status", [True, False])
def test_ffn_block_on_rows_rewritten_in_place(T, H, I, E, k, again, status):
    routed = tuple(dev(a) for a in inputs.make_expert_weights(H, I, E, seed=0))
    shared = tuple(dev(a) for a in inputs.make_expert_weights(H, I, 1, seed=21))
    wr = dev(_router_weights(E, H, 3))
    sh, sh1 = moe.shape(T, H, I, E, k), moe.shape(T, H, I, 1, 1)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    xs, want = [], []
    for i in range(3):
        xf = bf(inputs.make_x(T, H, 40 + i)).copy()
        if i != 1:                       # 2^15 and eight values below 2^-14 of it, in a block of two rows
            xf[[0, T - 1], 64 * i:64 * i + 32] = 64.0
            xf[[0, T - 1], 64 * i + 5] = 2.0 ** 15
            xf[[0, T - 1], 64 * i + 8:64 * i + 16] = 1.0 + 2.0 ** -7
        xs.append(dev(inputs.f32_to_bf16_bits(xf)))
    buf, lg = moe.LayerBuffers(sh), torch.empty((T, E), device="cuda")
    ys, alone = torch.empty((T, H), device="cuda"), torch.empty((T, H), device="cuda")
    off2, ws1 = torch.tensor([0, T], dtype=torch.int32, device="cuda"), moe.alloc_workspace(sh1)
    for i, x in enumerate(xs):
        moe.moe_router_logits(x, wr, lg, st)
        moe.moe_layer(lg, x, routed, buf)
        moe.moe_expert_ffn(x, off2, *shared, sh1, ys, st, ws1)
        assert (moe.moe_last_kernel_name() == "ffn_mxf8_two_term_cta_pair") == again
        moe.moe_combine_shared(buf.y_perm, buf.inv_perm, buf.topk_w, ys, sh, buf.out)
        if again:
            moe.moe_debug_expert_ffn_variant(x, off2, *shared, sh1, alone, st, ws1, moe.VARIANT_TWOTERM)
            assert torch.equal(ys, alone) == (i == 1)
        torch.cuda.synchronize()
        want.append(buf.out.clone())
    ws, ids, w = moe.alloc_block_workspace(sh), torch.empty((T, k), dtype=torch.int32, device="cuda"), torch.empty((T, k), device="cuda")
    outs = [torch.empty((T, H), dtype=torch.bfloat16, device="cuda") for _ in range(7)]
    x = torch.empty_like(xs[0])

    def calls():
        for i, o in enumerate(outs):
            x.copy_(xs[i % 3])
            moe.moe_ffn_block(x, wr, routed, shared, sh, o, ids, w, st if status else None, ws)
    calls()
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and all(torch.equal(o.view(torch.int16), want[i % 3].view(torch.int16)) for i, o in enumerate(outs))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    for o in outs:
        o.zero_()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and all(torch.equal(o.view(torch.int16), want[i % 3].view(torch.int16)) for i, o in enumerate(outs))
