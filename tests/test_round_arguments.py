"""``Round``'s arguments on the way to the library's calls (recorders in their place, no GPU)."""
import pytest
import torch


@pytest.fixture()
def recorded(dqlib, monkeypatch):
    from paper_2107_14575_b200 import dq
    from paper_2107_14575_b200.pipeline import Round
    made = []
    monkeypatch.setattr(dq, "norms_quantize_average", lambda *a: made.append(a))
    return Round([100], 32, 2, device="cpu"), dq, made


def test_an_update_needs_a_step_size(recorded):
    """Without one the average must not land in the parameters."""
    rnd, dq, made = recorded
    g, x = torch.zeros(2, 128), torch.ones(128)
    rule = dq.Rule.fixed(4)
    with pytest.raises(TypeError):
        rnd.step_fused(g, rule, 1, 0, params=x, lr=None)
    assert not made
    assert rnd.step_fused(g, rule, 1, 0, params=x, lr=0.5) is x
    assert made[-1][10] is x and made[-1][-1] == 0.5
    rnd.step_fused(g, rule, 1, 0, params=x)                   # (an eta of 0: the parameters stay)
    assert made[-1][-1] == 0.0
    assert rnd.step_fused(g, rule, 1, 0) is rnd.out
    assert made[-1][10] is rnd.out and made[-1][-1] is None
