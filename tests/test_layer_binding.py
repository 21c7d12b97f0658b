"""moe_layer's binding on the host: what it refuses (no GPU call is reached)."""
import pytest
import torch

from paper_2609_15627_b200 import moe


@pytest.mark.parametrize("missing", ["x_perm", "perm", "y_perm", "expert_offsets"])
def test_a_missing_buffer_is_an_error_of_the_call(missing):
    sh = moe.shape(4, 128, 128, 8, 2)
    buf = moe.LayerBuffers(sh, device="cpu")
    setattr(buf, missing, None)
    w = tuple(torch.zeros(64, dtype=torch.uint8) for _ in range(4))
    with pytest.raises(moe.MoeError, match="moe_layer failed: invalid argument"):
        moe.moe_layer(torch.zeros(4, 8), torch.zeros(4, 128, dtype=torch.bfloat16), w, buf, stream=0)


def test_a_missing_weight_is_an_error_of_the_call():
    sh = moe.shape(4, 128, 128, 8, 2)
    buf = moe.LayerBuffers(sh, device="cpu")
    w = tuple(torch.zeros(64, dtype=torch.uint8) for _ in range(3)) + (None,)
    with pytest.raises(moe.MoeError, match="moe_layer failed: invalid argument"):
        moe.moe_layer(torch.zeros(4, 8), torch.zeros(4, 128, dtype=torch.bfloat16), w, buf, stream=0)


def test_a_library_without_the_call_is_not_an_argument_s_fault(monkeypatch):
    class Empty:
        pass

    sh = moe.shape(4, 128, 128, 8, 2)
    buf = moe.LayerBuffers(sh, device="cpu")
    monkeypatch.setattr(moe, "_lib", Empty())
    w = tuple(torch.zeros(64, dtype=torch.uint8) for _ in range(4))
    with pytest.raises(AttributeError, match="moe_layer"):
        moe.moe_layer(torch.zeros(4, 8), torch.zeros(4, 128, dtype=torch.bfloat16), w, buf, stream=0)


@pytest.mark.parametrize("where", ["weights", "perm"])
def test_what_is_no_tensor_is_not_taken_for_a_missing_buffer(where):
    sh = moe.shape(4, 128, 128, 8, 2)
    buf, w = moe.LayerBuffers(sh, device="cpu"), [torch.zeros(64, dtype=torch.uint8)] * 4
    if where == "weights":
        w[1] = [0]
    else:
        buf.perm = [0]
    with pytest.raises(AttributeError, match="data_ptr"):
        moe.moe_layer(torch.zeros(4, 8), torch.zeros(4, 128, dtype=torch.bfloat16), w, buf, stream=0)
