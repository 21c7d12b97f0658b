"""The two-term kernel with few rows per expert, whose K steps lie one behind the other in the ring, as large as their pass needs: equal and
uneven experts (passes of 16 to 64 rows, several per expert), a few and many K steps, weights in rows and in tiles."""
import pytest
import torch

from _gpu_util import bits, check_out, dev
from oracle import moe_oracle as O
from paper_2609_15627_b200 import inputs, moe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,I,E,k,skew", [
    (300, 512, 256, 256, 8, False), (300, 512, 512, 256, 8, True), (512, 512, 256, 256, 8, False), (128, 1024, 512, 64, 8, True),
    (260, 2560, 256, 128, 5, True), (333, 512, 768, 128, 6, True)])
def test_against_the_oracle(T, H, I, E, k, skew):
    sh = moe.shape(T, H, I, E, k)
    raw = inputs.make_expert_weights(H, I, E, seed=3)
    w = tuple(dev(a) for a in raw)
    logits, x = inputs.make_logits(T, E, 41, skew), inputs.make_x(T, H, 42)
    r = O.forward_staged(logits, x, *raw, k)
    b = moe.LayerBuffers(sh)
    for _ in range(2):
        b.out.fill_(float("nan"))
        moe.moe_layer(dev(logits), dev(x), w, b)
        torch.cuda.synchronize()
        assert int(b.status.item()) == 0
        check_out(bits(b.out), r["out"], r["out_f32"], "rows")
    y = torch.full_like(b.y_perm, float("nan"))
    moe.moe_expert_ffn(b.x_perm, b.expert_offsets, *w, sh, y, b.status, b.ws)
    assert moe.moe_last_kernel_name() == "ffn_mxf8_two_term_cta_pair"
    assert torch.equal(y, b.y_perm)
    out, st = torch.empty_like(b.out), torch.zeros(1, dtype=torch.int32, device="cuda")
    moe.moe_forward_packed(dev(logits), dev(x), moe.moe_prepack(*w, sh), sh, out, None, None, st, moe.alloc_forward_workspace(sh))
    torch.cuda.synchronize()
    assert torch.equal(out, b.out) and int(st.item()) == 0
