"""The expert FFN on two E4M3 terms per activation (CTA pairs, kind::mxf8f6f4) against the oracle: every form of a pass and
its edges, every way its scale bytes are read, both weight layouts, expert-parallel ranks, non-finite tokens."""
import numpy as np
import pytest
import torch

from _gpu_util import check_y, dev
from oracle import moe_oracle as O
from test_gpu_quant import _check_rows
from paper_2609_15627_b200 import ep, inputs, moe

pytestmark = pytest.mark.gpu
NAME = "ffn_mxf8_two_term_cta_pair"


def _weights(H, I, E, seed):
    w = inputs.make_expert_weights(H, I, E, seed=seed)
    return w[0], inputs.index_scales(2 * I, H, E, lo=117, span=6), w[2], inputs.index_scales(H, I, E, lo=118, span=5)


def _ffn(x, off, wdev, H, I, E):
    sh = moe.shape(x.shape[0], H, I, E, 1)
    S = x.shape[0]
    need = moe.moe_workspace_bytes(sh) + 2 * S * (H + I) + (E + S // 64 + 1) * (H + I) // 128 * 2048 + 4096
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    y = torch.full((S, H), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    moe.moe_debug_expert_ffn_variant(dev(x), dev(off), *wdev, sh, y, status, ws, moe.VARIANT_TWOTERM)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and moe.moe_last_kernel_name() == NAME
    return y.cpu().numpy()


# rows per expert.  On average up to 56: passes of at most 64 tokens; up to 96: of 112; more: of 224
_NARROW = [1, 16, 17, 0, 48, 49, 64, 65, 130]
_MID = [112, 113, 0, 97, 80, 96, 128, 1]
_WIDE = [224, 225, 113, 112, 0, 129, 450, 160]


@pytest.mark.parametrize("counts,H,I", [
    (_NARROW, 512, 256),   # down: 512 rows per item, scale rows of 8 bytes in one piece
    (_NARROW, 256, 512),   # down: 256 rows per item; gate/up: scale rows of 8 bytes
    (_NARROW, 768, 768),   # scale rows of 24 bytes
    (_MID, 512, 512),
    (_WIDE, 512, 512),
    (_WIDE, 1024, 256),
    ([0, 0, 3, 0], 4096, 256),
])
def test_against_oracle(counts, H, I):
    E, S = len(counts), sum(counts)
    w = _weights(H, I, E, seed=S)
    xf = inputs.bf16_bits_to_f32(inputs.make_x(S, H, seed=H + I))
    xf[:, ::7] *= 2.0 ** -9    # a wide range inside blocks: the second term and its scale matter
    xf[:, 5::11] *= 64.0
    xf[:, 64:96] = 0.0         # a block of zeros
    x = inputs.f32_to_bf16_bits(xf)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    check_y(_ffn(x, off, [dev(a) for a in w], H, I, E), O.expert_ffn(x, off, *w, 1), "two terms")


@pytest.mark.parametrize("counts", [[3, 0, 122, 130], [3, 0, 123, 130]])
@pytest.mark.parametrize("H", [256, 2304])
def test_rows_split_in_short_and_in_long_tasks(counts, H):   # below 256 rows two pieces of 256 values a task, from there on eight
    E, S, I = len(counts), sum(counts), 512
    w, x = _weights(H, I, E, seed=S), inputs.make_x(S, H, seed=H)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    check_y(_ffn(x, off, [dev(a) for a in w], H, I, E), O.expert_ffn(x, off, *w, 1), "two terms")


def test_non_finite_tokens_stay_non_finite_and_to_themselves():
    H, I, counts = 512, 256, [40, 130]
    E, S = len(counts), sum(counts)
    wdev = [dev(a) for a in _weights(H, I, E, seed=1)]
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    x = inputs.make_x(S, H, seed=2)
    want = _ffn(x, off, wdev, H, I, E)
    bad = x.copy()
    bad[3, 100], bad[41, 7], bad[169, 300] = 0x7F80, 0xFF80, 0x7FC0   # +inf, -inf, NaN
    got = _ffn(bad, off, wdev, H, I, E)
    rows = np.array([3, 41, 169])
    assert not np.isfinite(got[rows]).any()
    rest = np.setdiff1d(np.arange(S), rows)
    assert np.array_equal(got[rest], want[rest])


@pytest.mark.parametrize("T,k,world", [(512, 2, 4), (3100, 2, 2)])   # 16 and 97 rows per expert
def test_chosen_by_shape_the_same_on_packed_weights_and_on_expert_parallel_ranks(T, k, world):
    H, I, E = 512, 512, 64
    w = _weights(H, I, E, seed=4)
    wdev = tuple(dev(a) for a in w)
    logits, x = inputs.make_logits(T, E, 5), inputs.make_x(T, H, 6)
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    moe.moe_route(dev(logits), k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(dev(x), buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
    moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *wdev, sh, buf.y_perm, buf.status, buf.ws)
    assert moe.moe_last_kernel_name() == NAME
    want = buf.y_perm.clone()
    packed = moe.moe_prepack(*wdev, sh)
    buf.y_perm.fill_(float("nan"))
    moe.moe_expert_ffn_packed(buf.x_perm, buf.expert_offsets, packed, sh, buf.y_perm, buf.status, buf.ws)
    torch.cuda.synchronize()
    assert moe.moe_last_kernel_name() == NAME and torch.equal(buf.y_perm, want)
    r = O.forward_staged(logits, x, *w, k)
    check_y(want.cpu().numpy(), r["y_perm"], "two terms, chosen by shape")
    moe.moe_combine(buf.y_perm, buf.inv_perm, buf.topk_w, sh, buf.out)
    out, ranks = ep.run_emulated(torch, moe, sh, world, dev(logits), dev(x), wdev)
    assert all(int(b.layer.status.item()) == 0 for b in ranks) and torch.equal(out, buf.out)
    out1 = torch.empty_like(buf.out)
    moe.moe_forward_packed(dev(logits), dev(x), packed, sh, out1, None, None, buf.status, moe.alloc_forward_workspace(sh))
    torch.cuda.synchronize()
    assert int(buf.status.item()) == 0 and torch.equal(out1, buf.out)


# Rows split once per token and copied to their sorted places: rows of one, three, nine, sixteen and 28 pieces of 256 values, a
# warp's share of them from four to sixteen, one slot per token and thirty-two
@pytest.mark.parametrize("T,H,I,E,k", [(4200, 256, 256, 128, 1), (600, 768, 256, 128, 5), (1100, 2304, 256, 128, 2), (128, 4096, 256, 128, 32),
                                       (9000, 4096, 256, 128, 1), (520, 7168, 256, 128, 6)])
def test_rows_split_by_token_are_the_rows_split_in_sorted_order(T, H, I, E, k):
    wdev = tuple(dev(a) for a in _weights(H, I, E, seed=14))
    logits, x = inputs.make_logits(T, E, 15), inputs.make_x(T, H, 16)
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    moe.moe_route(dev(logits), k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(dev(x), buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
    moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *wdev, sh, buf.y_perm, buf.status, buf.ws)
    assert moe.moe_last_kernel_name() == NAME
    moe.moe_combine(buf.y_perm, buf.inv_perm, buf.topk_w, sh, buf.out)
    out = torch.empty_like(buf.out)
    moe.moe_forward(dev(logits), dev(x), *wdev, sh, out, None, None, buf.status, moe.alloc_forward_workspace(sh))
    torch.cuda.synchronize()
    assert int(buf.status.item()) == 0 and torch.equal(out.view(torch.int16), buf.out.view(torch.int16))
    buf2 = moe.LayerBuffers(sh)
    moe.moe_layer(dev(logits), dev(x), wdev, buf2)
    torch.cuda.synchronize()
    assert all(torch.equal(getattr(buf2, n).view(torch.int16), getattr(buf, n).view(torch.int16)) for n in ("x_perm", "perm", "inv_perm", "y_perm", "out"))


@pytest.mark.parametrize("T,H,I,E,k,packed", [(1100, 1024, 512, 32, 2, False), (1100, 1024, 512, 32, 2, True),   # 69 rows per expert
                                              (4200, 512, 256, 64, 1, False), (600, 768, 768, 43, 5, False)])
def test_quantised_activations_on_cta_pairs(T, H, I, E, k, packed):
    w = _weights(H, I, E, seed=9)
    x = inputs.make_x(T, H, 10)
    logits = inputs.make_logits(T, E, 11)
    logits[:, 3] += 1.0          # an expert of several passes
    logits[:, E - 1] -= 50.0     # an empty one
    ids, _, off = O.route(logits, k)
    x_perm, _, _ = O.permute(x, ids, off)
    sh = moe.shape(T, H, I, E, k)
    wdev = tuple(dev(a) for a in w)
    y = torch.full((T * k, H), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    moe.moe_expert_ffn_q(dev(x_perm), dev(off), moe.moe_prepack(*wdev, sh) if packed else wdev, sh, y, status, moe.alloc_ffn_q_workspace(sh))
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and moe.moe_last_kernel_name() == "ffn_mxf4_quantised_cta_pair"
    _check_rows(y.cpu().numpy(), O.expert_ffn_q(x_perm, off, *w, k), "quantised, CTA pairs")


# ---- blocks that two terms hold too little of: their experts are done again by the kernel that holds every value ----
_UMMA, _STREAM = "ffn_umma_tcgen05_grouped", "ffn_stream_bulk_ring_mma16816"
_AGAIN = [(2048, 1024, _UMMA, False), (2048, 1024, _UMMA, True), (2048, 1280, _STREAM, False)]


def _at_16(t):
    """A copy at an address that is a multiple of 16 bytes and not of 32."""
    room = torch.empty(t.numel() + 48, dtype=torch.uint8, device="cuda")
    lead = (16 - room.data_ptr()) % 32
    return room[lead:lead + t.numel()].copy_(t.reshape(-1)).view(t.shape)


def _bits(t):
    return t.contiguous().view(torch.int32)


def _three_ways(x, off, wdev, sh, kernel, packed):
    """y_perm of the public call, of the kernel that takes the shape without this one, and of this one alone."""
    xd, offd = dev(x), dev(off)
    buf = moe.LayerBuffers(sh)
    ys = []

    def run(call, *args, name=NAME):
        buf.y_perm.fill_(float("nan"))
        call(xd, offd, *args)
        torch.cuda.synchronize()
        assert int(buf.status.item()) == 0 and moe.moe_last_kernel_name() == name
        ys.append(buf.y_perm.clone())

    if packed:
        run(moe.moe_expert_ffn_packed, moe.moe_prepack(*wdev, sh), sh, buf.y_perm, buf.status, buf.ws)
    else:
        run(moe.moe_expert_ffn, *wdev, sh, buf.y_perm, buf.status, buf.ws)
    w16 = (_at_16(wdev[0]), wdev[1], _at_16(wdev[2]), wdev[3])
    run(moe.moe_expert_ffn, *w16, sh, buf.y_perm, buf.status, buf.ws, name=kernel)
    run(moe.moe_debug_expert_ffn_variant, *wdev, sh, buf.y_perm, buf.status, buf.ws, moe.VARIANT_TWOTERM)
    return ys


def _done_again(ys, off):
    """Experts whose rows are the other kernel's bits; every expert's rows are either that or this kernel's."""
    got, other, alone = (_bits(y) for y in ys)
    again = []
    for e in range(len(off) - 1):
        r = slice(int(off[e]), int(off[e + 1]))
        if torch.equal(got[r], other[r]) and not torch.equal(other[r], alone[r]):
            again.append(e)
        else:
            assert torch.equal(got[r], alone[r]), e
    return again


@pytest.mark.parametrize("H,I,kernel,packed", _AGAIN)
def test_experts_done_again(H, I, kernel, packed):
    E, counts = 16, [66 + (7 * e) % 11 for e in range(16)]
    S = sum(counts)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    w = [a.copy() for a in _weights(H, I, E, seed=21)]
    xf = inputs.bf16_bits_to_f32(inputs.make_x(S, H, seed=22))

    def block(row, c0, n_small, edge):
        """2^15, n_small values below 2^-14 of it, `edge` at that bound, the rest between"""
        xf[row, c0:c0 + 32] = 64.0
        xf[row, c0 + 5] = 2.0 ** 15
        xf[row, c0 + 8:c0 + 8 + n_small] = 1.0 + 2.0 ** -7
        xf[row, c0 + 20:c0 + 20 + edge] = 2.0

    block(int(off[1]), 0, 6, 0)                    # six: the first row of expert 1
    block(int(off[4]) - 1, H - 32, 5, 3)           # five, and three at the bound: not enough
    block(int(off[5]) + 3, 256 - 32, 9, 0)
    xf[int(off[7]) + 1, 300] = np.inf
    xf[int(off[9]) - 1, 17] = np.nan
    w[1][10, I:, :] = 105                          # up rows of expert 10: one of a block 2^15 times the others
    w[1][10, I + 101, :] = 120
    w[1][12, I:, :] = 105                          # of expert 12: half of a block
    w[1][12, I + 96:I + 112, :] = 120
    x = inputs.f32_to_bf16_bits(xf)
    sh = moe.shape(S, H, I, E, 1)
    ys = _three_ways(x, off, [dev(a) for a in w], sh, kernel, packed)
    assert _done_again(ys, off) == [1, 5, 7, 8, 10]


@pytest.mark.parametrize("where", ["tokens", "intermediate"])
@pytest.mark.parametrize("p", [10, 14, 18])
def test_rows_keep_their_precision_beside_an_outlier_of_every_block(where, p):
    """One element of every block of 32 is 2^p times the others and meets zero weights only, so every output is a sum over
    the others.  By the median over rows (a row in ten holds a bf16 rounding of the intermediate that falls the other way,
    2^-9 of one value): an fp32 sum of 2048 terms is off by 5e-7 of its norm, the two terms would be by 5e-5 (2^10) to 0.5."""
    H, I, E, counts = 2048, 1024, 16, [66] * 16
    S = sum(counts)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    w = [a.copy() for a in _weights(H, I, E, seed=31)]
    xf = inputs.bf16_bits_to_f32(inputs.make_x(S, H, seed=32))
    if where == "tokens":
        xf[:, 5::32] *= 2.0 ** p
        w[0][:, :, 2::16] &= 0x0F                  # element 5 of a block: the high nibble of byte 2
    else:
        w[1][:, I:, :] = 108
        w[1][:, I + 5::32, :] = 108 + p
        w[2][:, :, 2::16] &= 0x0F
    x = inputs.f32_to_bf16_bits(xf)
    sh = moe.shape(S, H, I, E, 1)
    buf = moe.LayerBuffers(sh)
    moe.moe_expert_ffn(dev(x), dev(off), *[dev(a) for a in w], sh, buf.y_perm, buf.status, buf.ws)
    torch.cuda.synchronize()
    assert int(buf.status.item()) == 0 and moe.moe_last_kernel_name() == NAME
    rows = np.concatenate([np.arange(off[e], off[e] + 8) for e in (0, 7, 15)])
    sub = np.zeros(E + 1, np.int32)
    sub[1:] = np.cumsum([8 if e in (0, 7, 15) else 0 for e in range(E)])
    ref = O.expert_ffn(x[rows], sub, *w, 1).astype(np.float64)
    got = buf.y_perm.cpu().numpy()[rows].astype(np.float64)
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.median(err) <= 5e-6 and err.max() <= 5e-3, (np.median(err), err.max())


@pytest.mark.parametrize("I,kernel", [(1024, _UMMA), (1280, _STREAM)])
def test_whole_layer_and_expert_parallel_ranks_do_experts_again(I, kernel):
    T, k, H, E = 536, 2, 2048, 16
    wdev = tuple(dev(a) for a in _weights(H, I, E, seed=41))
    xf = inputs.bf16_bits_to_f32(inputs.make_x(T, H, 42))
    xf[::3, 64] = 2.0 ** 20                        # tokens of every expert
    logits, x = dev(inputs.make_logits(T, E, 43)), dev(inputs.f32_to_bf16_bits(xf))
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    w16 = (_at_16(wdev[0]), wdev[1], _at_16(wdev[2]), wdev[3])
    want = moe.moe_layer(logits, x, w16, buf).clone()
    moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *w16, sh, buf.y_perm, buf.status, buf.ws)
    assert moe.moe_last_kernel_name() == kernel
    assert torch.equal(moe.moe_layer(logits, x, wdev, buf), want)
    out = torch.empty_like(want)
    fws = moe.alloc_forward_workspace(sh)
    fws[moe.moe_forward_sync_bytes():].fill_(0xFF)
    for call, weights in ((moe.moe_forward, wdev), (moe.moe_forward_packed, (moe.moe_prepack(*wdev, sh),))):
        out.fill_(float("nan"))
        call(logits, x, *weights, sh, out, None, None, buf.status, fws)
        assert torch.equal(out, want)
    out, ranks = ep.run_emulated(torch, moe, sh, 2, logits, x, wdev)
    assert all(int(b.layer.status.item()) == 0 for b in ranks) and torch.equal(out, want)
    assert int(buf.status.item()) == 0


# moe_forward_host where the two-term kernel runs: rows and logits read in place up to 256 tokens (by the gather of experts that are
# done again as well), the output written in place at any size; and the bf16 kernel's output
@pytest.mark.parametrize("T,H,I,E,k,ffn,again", [(256, 512, 512, 64, 4, NAME, False), (256, 1024, 512, 64, 32, NAME, True), (300, 512, 512, 64, 4, NAME, False),
                                                 (1300, 1024, 512, 64, 8, NAME, True), (1500, 512, 512, 8, 2, _UMMA, False)])
def test_host_buffers_in_place_and_copied(T, H, I, E, k, ffn, again):
    wdev = tuple(dev(a) for a in _weights(H, I, E, seed=61))
    xf = inputs.bf16_bits_to_f32(inputs.make_x(T, H, 62))
    if again:
        xf[::5, 64] = 2.0 ** 20
    x, logits = inputs.f32_to_bf16_bits(xf), inputs.make_logits(T, E, 63)
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    moe.moe_layer(dev(logits), dev(x), wdev, buf)
    want = buf.out.clone()
    moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *wdev, sh, buf.y_perm, buf.status, buf.ws)
    assert moe.moe_last_kernel_name() == ffn
    if again:                                      # (it does some experts again: alone the kernel gives other bits)
        alone = torch.empty_like(buf.y_perm)
        moe.moe_debug_expert_ffn_variant(buf.x_perm, buf.expert_offsets, *wdev, sh, alone, buf.status, buf.ws, moe.VARIANT_TWOTERM)
        assert not torch.equal(alone, buf.y_perm)
    ws = moe.alloc_workspace(sh, host_path=True)
    lh, xh = torch.from_numpy(logits), torch.from_numpy(x.view(np.int16))
    for pin in (True, False):
        oh = torch.zeros((T, H), dtype=torch.int16)
        bufs = [t.pin_memory() for t in (lh, xh, oh)] if pin else [lh, xh, oh]
        assert all((moe.lib().moe_debug_host_view(t.data_ptr(), t.numel() * t.element_size()) is not None) == pin for t in bufs)
        ws.fill_(0x5A)
        moe.moe_forward_host(bufs[0], bufs[1], *wdev, sh, bufs[2], buf.status, ws)
        assert int(buf.status.item()) == 0 and torch.equal(bufs[2], want.view(torch.int16).cpu())


# (33 and 97 rows per expert: passes of 64 and of 224 tokens; the quantised variant above 64)
@pytest.mark.parametrize("T,k,H,I,quantised", [(2112, 2, 512, 512, False), (3100, 4, 512, 512, False), (3100, 4, 512, 512, True)])
def test_offsets_may_come_from_the_launch_in_front(T, k, H, I, quantised):
    """moe_route lets its dependents start before it has written expert_offsets; a call right behind it on rows sorted
    earlier has to see the new ones.  (The old ones in the buffer are valid too, so a call that read them too early would
    give other rows, not stray ones.)"""
    E = 128
    w = tuple(dev(a) for a in _weights(H, I, E, seed=51))
    logits, x = dev(inputs.make_logits(T, E, 52)), dev(inputs.make_x(T, H, 53))
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    qws = moe.alloc_ffn_q_workspace(sh)
    moe.moe_route(logits, k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(x, buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)

    def ffn():
        if quantised:
            moe.moe_expert_ffn_q(buf.x_perm, buf.expert_offsets, w, sh, buf.y_perm, buf.status, qws)
            assert moe.moe_last_kernel_name() == "ffn_mxf4_quantised_cta_pair"
        else:
            moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *w, sh, buf.y_perm, buf.status, buf.ws)
            assert moe.moe_last_kernel_name() == NAME

    torch.cuda.synchronize()
    ffn()
    torch.cuda.synchronize()
    want = buf.y_perm.clone()
    stale = torch.full_like(buf.expert_offsets, T * k)
    stale[0] = 0
    for _ in range(5):
        buf.expert_offsets.copy_(stale)
        buf.y_perm.fill_(float("nan"))
        torch.cuda.synchronize()
        moe.moe_route(logits, k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
        ffn()
        torch.cuda.synchronize()
        assert int(buf.status.item()) == 0 and torch.equal(buf.y_perm, want)


@pytest.mark.parametrize("T,I,kernel", [(512, 512, "ffn_native_mxf4_block_scaled"), (1120, 512, _UMMA), (1120, 256, _STREAM)])
def test_weights_aligned_to_16_bytes_take_the_other_kernels(T, I, kernel):
    """16 and 35 rows per expert, where 32-byte aligned weights take the two-term kernel."""
    H, E, k = 512, 64, 2
    w = _weights(H, I, E, seed=61)
    x, ids = inputs.make_x(T, H, 62), O.route(inputs.make_logits(T, E, 63), k)
    x_perm, _, _ = O.permute(x, ids[0], ids[2])
    want = O.expert_ffn(x_perm, ids[2], *w, k)
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    wdev = [dev(a) for a in w]
    for weights, name in ((wdev, NAME), ([_at_16(wdev[0]), wdev[1], wdev[2], wdev[3]], kernel),
                          ([wdev[0], wdev[1], _at_16(wdev[2]), wdev[3]], kernel)):
        buf.y_perm.fill_(float("nan"))
        moe.moe_expert_ffn(dev(x_perm), dev(ids[2]), *weights, sh, buf.y_perm, buf.status, buf.ws)
        torch.cuda.synchronize()
        assert int(buf.status.item()) == 0 and moe.moe_last_kernel_name() == name
        check_y(buf.y_perm.cpu().numpy(), want, name)


@pytest.mark.parametrize("T,H,I,E,name,other", [
    (768, 4096, 1024, 256, "ffn_native_mxf4_block_scaled", moe.VARIANT_TWOTERM),   # 6 rows per expert
    (769, 4096, 1024, 256, NAME, moe.VARIANT_NATIVE),
    (1792, 1024, 512, 32, NAME, moe.VARIANT_UMMA),                                  # 112
    (1793, 1024, 512, 32, _UMMA, moe.VARIANT_TWOTERM)])
def test_lines_of_the_choice(T, H, I, E, name, other):
    k = 2
    g = torch.Generator(device="cuda").manual_seed(71)
    w = [torch.randint(lo, hi, (E, rows, cols), dtype=torch.uint8, device="cuda", generator=g)
         for lo, hi, rows, cols in ((0, 256, 2 * I, H // 2), (119, 123, 2 * I, H // 32), (0, 256, H, I // 2), (119, 123, H, I // 32))]
    sh = moe.shape(T, H, I, E, k)
    buf = moe.LayerBuffers(sh)
    moe.moe_route(dev(inputs.make_logits(T, E, 72)), k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(dev(inputs.make_x(T, H, 73)), buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
    moe.moe_expert_ffn(buf.x_perm, buf.expert_offsets, *w, sh, buf.y_perm, buf.status, buf.ws)
    assert moe.moe_last_kernel_name() == name
    got = buf.y_perm.clone()
    packed = moe.moe_prepack(*w, sh)
    buf.y_perm.fill_(float("nan"))
    moe.moe_expert_ffn_packed(buf.x_perm, buf.expert_offsets, packed, sh, buf.y_perm, buf.status, buf.ws)
    torch.cuda.synchronize()
    assert moe.moe_last_kernel_name() == name and torch.equal(buf.y_perm, got)     # the same choice, the same bits
    ws = torch.empty(buf.ws.numel() + 9 * T * k * (H + I), dtype=torch.uint8, device="cuda")
    moe.moe_debug_expert_ffn_variant(buf.x_perm, buf.expert_offsets, *w, sh, buf.y_perm, buf.status, ws, other)
    torch.cuda.synchronize()
    want = buf.y_perm.double()
    diff = got.double() - want                       # the tolerance of the fp32 per-slot rows
    assert int(buf.status.item()) == 0
    assert float(diff.norm() / want.norm()) <= 5e-4 and float(diff.abs().max()) <= 2e-2 * float(want.pow(2).mean().sqrt())


@pytest.mark.parametrize("S,H", [(8192, 1024), (8200, 1024), (8200, 2048), (16384, 2048), (16392, 2048)])
def test_sort_at_the_lines_between_its_forms(S, H):
    """The direct count and the chunked sort give the one stable order, rows copied along (the whole layer sorts without
    them: the line for short rows)."""
    k, E = 8, 40
    T = S // k
    logits, x = inputs.make_logits(T, E, 81), inputs.make_x(T, H, 82)
    sh = moe.shape(T, H, 256, E, k)
    buf = moe.LayerBuffers(sh)
    moe.moe_route(dev(logits), k, buf.topk_ids, buf.topk_w, buf.expert_offsets, buf.ws)
    moe.moe_permute(dev(x), buf.topk_ids, buf.expert_offsets, sh, buf.x_perm, buf.perm, buf.inv_perm, buf.ws)
    torch.cuda.synchronize()
    direct = S <= (16384 if H >= 2048 else 8192)
    assert moe.moe_last_kernel_name() == ("permute_rank_by_count" if direct else "permute_chunked_scan")
    ids, off = buf.topk_ids.cpu().numpy(), buf.expert_offsets.cpu().numpy()
    x_perm, perm, inv = O.permute(x, ids, off)
    assert np.array_equal(buf.perm.cpu().numpy(), perm) and np.array_equal(buf.inv_perm.cpu().numpy().reshape(-1), inv.reshape(-1))
    assert np.array_equal(buf.x_perm.view(torch.int16).cpu().numpy().view(np.uint16), x_perm)
