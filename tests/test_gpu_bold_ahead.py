"""BOLD of short and uneven lengths (the rates are fetched in blocks of eight
samples) and of drives on both sides of the short series' bounds, against the
FP64 oracle, and in two pieces bit for bit."""
import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import bold as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


@pytest.mark.parametrize("n_samples", [1, 7, 8, 9, 16, 17, 31, 4001])
@pytest.mark.parametrize("n_sets", [2, 3])
def test_bold_lengths(tvbx, n_samples, n_sets):
    import torch
    rng = np.random.default_rng(n_samples)
    # set 0 at 5 Hz, the others from rest to 150 Hz (f - 1 from 0 to 0.37)
    X = 5e-3 * rng.uniform(0.5, 1.5, (n_samples, 3, n_sets))
    X[:, :, 1:] += np.linspace(0.0, 0.15, n_samples)[:, None, None]
    X = X.astype(np.float32)
    x = torch.from_numpy(X).cuda()
    st = torch.zeros((4, 3, n_sets), device="cuda")
    y = tvbx.bold(x, 1.0, 1, state=st, reset_state=True)
    for p in range(n_sets):
        want, state = B.bold(X[:, :, p].T, 1.0, 1)
        state[1:] -= 1.0
        # Euler steps of FP32 roundings: 4,000 steps of 2^-24 of the largest term
        assert np.abs(y[:, :, p].cpu().numpy().T - want).max() <= 1e-4 * np.abs(want).max() + 1e-12
        assert np.abs(st[:, :, p].cpu().numpy() - state).max() <= 1e-4 * np.abs(state).max() + 1e-12
    half = n_samples // 2
    st2 = torch.zeros_like(st)
    parts = [tvbx.bold(x[:half].contiguous(), 1.0, 1, state=st2, reset_state=True)] if half else []
    parts.append(tvbx.bold(x[half:].contiguous(), 1.0, 1, state=st2, reset_state=not half))
    assert torch.equal(torch.cat(parts), y) and torch.equal(st, st2)


@pytest.mark.parametrize("beside", [0.0, 0.2, 3.0, float("nan"), float("inf")])
def test_bold_of_an_element_does_not_depend_on_its_neighbour(tvbx, beside):
    """Two elements share a thread: one at rates from 2.5 Hz to 2.7 kHz, from near
    rest to beyond the bounds of every series, beside one of any other rates."""
    import torch
    T, P = 3000, 500
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    amp = torch.exp(7.0 * torch.rand(P, generator=g, device="cuda") - 6.0)
    a = amp * torch.rand((T, 1, P), generator=g, device="cuda")
    b = beside * torch.rand((T, 1, P), generator=g, device="cuda")
    alone = tvbx.bold(torch.stack((a, a), dim=-1).view(T, 1, 2 * P), 1.0, 10).view(-1, P, 2)
    assert torch.equal(alone[..., 0], alone[..., 1]) and torch.isfinite(alone).all()
    for lane in (0, 1):
        pair = (a, b) if lane == 0 else (b, a)
        got = tvbx.bold(torch.stack(pair, dim=-1).view(T, 1, 2 * P), 1.0, 10).view(-1, P, 2)
        assert torch.equal(got[..., lane], alone[..., lane])
        assert torch.isfinite(got[..., 1 - lane]).all().item() == (beside < 3.5)


@pytest.mark.parametrize("peak", [0.02, 0.3, 3.0])
def test_bold_of_odd_counts_and_unaligned_rates(tvbx, peak):
    """One element per thread gives what two give."""
    import torch
    T, N = 3001, 33
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    a = peak * torch.rand((T, N, 1), generator=g, device="cuda")
    st, st2 = torch.zeros((4, N, 1), device="cuda"), torch.zeros((4, N, 2), device="cuda")
    odd, even = tvbx.bold(a, 1.0, 7, state=st), tvbx.bold(a.expand(T, N, 2).contiguous(), 1.0, 7, state=st2)
    assert torch.equal(odd[..., 0], even[..., 0]) and torch.equal(st[..., 0], st2[..., 1])
    x = torch.empty(T * N * 2 + 1, device="cuda")[1:].view(T, N, 2)
    x.copy_(a.expand(T, N, 2))
    assert x.data_ptr() % 8 == 4 and torch.equal(tvbx.bold(x, 1.0, 7), even)
