"""What the Python entry points take and refuse before they reach the library, which a stand-in
replaces here (no GPU)."""

import pytest
import torch

from paper_1808_07284_gb300 import _binding as B


class Device(torch.Tensor):
    """A host tensor that says it is on the GPU: its pointer is taken, never followed."""
    is_cuda = property(lambda self: True)


def grid(*shape):
    return torch.zeros(shape).as_subclass(Device)


@pytest.fixture
def calls(monkeypatch):
    seen = []

    class Lib:
        def emd_dyn_solve_batched(self, *args):
            seen.append(args)
            return B.EMD_OK

    monkeypatch.setattr(B, "lib", Lib)
    monkeypatch.setattr(B, "_stream", lambda s: None)
    return seen


def solve(f_obs, f_pred, phis, ms):
    n = len(f_obs)
    return B.emd_dyn_solve_batched(f_obs, f_pred, [1.0] * n, [1.0] * n, B.EmdParams(), phis, ms, torch.zeros(256))


def lists(n=2, shape=(3, 8)):
    return ([grid(*shape) for _ in range(n)] for _ in range(3)), [grid(2, *shape) for _ in range(n)]


@pytest.mark.parametrize("shape", [(3, 8), (3, 8, 1), (3, 8, 1, 1)])
def test_batched_solve_reads_the_first_two_sizes(calls, shape):
    (obs, pred, phis), ms = lists(2, shape)
    solve(obs, pred, phis, ms)
    args = calls[0]
    assert args[0] == 2 and list(args[3]) == [8, 8] and list(args[4]) == [3, 3]
    for got, want in ((args[1], obs), (args[2], pred), (args[8], phis), (args[9], ms)):
        assert list(got) == [t.data_ptr() for t in want]


@pytest.mark.parametrize("which", [1, 2, 3])
@pytest.mark.parametrize("change", [-1, 1])
def test_batched_solve_refuses_lists_of_another_length(calls, which, change):
    (obs, pred, phis), ms = lists()
    args = [obs, pred, phis, ms]
    args[which] = args[which][:-1] if change < 0 else args[which] + args[which][:1]
    with pytest.raises(IndexError):
        solve(*args)
    assert not calls


def test_batched_solve_names_the_wrong_tensor(calls):
    (obs, pred, phis), ms = lists()
    ms[1] = grid(3, 8)
    with pytest.raises(ValueError, match=r"m\[1\]"):
        solve(obs, pred, phis, ms)
    phis[0] = torch.zeros(3, 8)
    with pytest.raises(TypeError, match=r"phi\[0\]"):
        solve(obs, pred, phis, ms)
    assert not calls


@pytest.mark.parametrize("value", [0.0, 0.1, -1e-50, 3.4028235e38, 3.4028236e38, -3.5e38, 1e300,
                                   float("inf"), float("nan")])
def test_losses_round_to_float32_as_a_conversion_does(monkeypatch, value):
    """A misfit beyond the range of float32 is an infinite loss."""
    import paper_1808_07284_gb300 as P
    f = torch.zeros(3, 8, requires_grad=True)
    monkeypatch.setattr(P, "emd_lsd", lambda *a, **k: value)
    monkeypatch.setattr(P, "emd", lambda *a, **k: (value, torch.zeros(3, 8), None, {}))
    want = torch.tensor(value, dtype=torch.float32)
    for loss in (P.lsd_loss(f, torch.zeros(3, 8), 1.0, 1.0), P.emd_loss(f, torch.zeros(3, 8), 1.0, 1.0)):
        assert loss.dtype == torch.float32 and loss.shape == () and loss.requires_grad
        assert torch.equal(loss.detach().view(torch.int32), want.view(torch.int32)) or value != value and loss != loss
