"""Host side of the learned correction, the library's calls replaced by stand-ins."""
import pytest
import torch

from paper_1004_1680_gb300 import learned


@pytest.mark.parametrize("default", [torch.float32, torch.float64, torch.bfloat16])
def test_gradients_have_the_parameters_type(monkeypatch, default):
    """The library adds FP32 into the gradients it is given, whatever torch's
    default type is when backward runs."""
    monkeypatch.setattr(learned.mhd, "conv_pack", lambda w, transpose=False: w)
    calls = []
    monkeypatch.setattr(learned.mhd, "cnn_backward", lambda *a: calls.append(a))
    net = learned.CorrectionNet(device="cpu")
    acts = [torch.zeros((4, c), dtype=torch.bfloat16) for c in (8, 32, 32, 32)]
    before = torch.get_default_dtype()
    try:
        torch.set_default_dtype(default)
        net.backward(torch.zeros((4, 8), dtype=torch.bfloat16), acts, (4, 1, 1))
    finally:
        torch.set_default_dtype(before)
    assert [(g.dtype, g.shape) for g in net.grads] == [(torch.float32, p.shape) for p in net.params]
    assert all(g.is_contiguous() and not g.any() for g in net.grads)
    assert [t.data_ptr() for t in calls[0][4] + calls[0][5]] == [g.data_ptr() for g in net.grads]
