"""FP32 FC at the edges of its moment kernel: several groups of sets per CTA,
regions on both sides of a tile, samples split over moment blocks, both
layouts with and without 16-byte rows, against the FP64 Pearson FC."""
import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


@pytest.mark.parametrize("n_regions,n_sets,n_samples", [
    (3, 5000, 65), (7, 2433, 130), (8, 9741, 40), (16, 4867, 70), (24, 6, 1500), (71, 3, 700), (72, 1, 129), (130, 9, 333),
    (383, 2, 200)])
@pytest.mark.parametrize("layout", ["tnp", "set4"])
def test_fp32_fc_against_fp64(tvbx, n_regions, n_sets, n_samples, layout):
    import torch
    N, P, T = n_regions, n_sets, n_samples
    g = torch.Generator(device="cuda")
    g.manual_seed(N + P)
    x = 5e-3 + 1e-3 * (torch.randn((T, N, P), generator=g, device="cuda") + torch.randn((T, 1, P), generator=g, device="cuda"))
    at = np.unique(np.linspace(0, P - 1, 40).astype(int))
    ref = x[:, :, torch.as_tensor(at, device="cuda")].permute(2, 1, 0).double().cpu().numpy()
    y, lay = x, tvbx.LAYOUT_TNP
    if layout == "set4":
        y = torch.nn.functional.pad(x, (0, -P % 4)).view(T, N, -1, 4).permute(2, 0, 1, 3).contiguous()
        lay = tvbx.LAYOUT_SET4
    fc = torch.empty((P, N, N), device="cuda")
    chi, mfc = torch.empty(P, device="cuda"), torch.empty(P, device="cuda")
    tvbx.fc_series(y, N, P, T, fc_out=fc, chi=chi, mean_fc=mfc, layout=lay)
    # FP32 sums of T products of order-one relative rounding 2^-24: well below 5e-5
    want = O.fc_pearson(ref)
    got = fc[torch.as_tensor(at, device="cuda")].cpu().numpy()
    assert np.abs(got - want).max() < 5e-5
    assert np.array_equal(got, np.swapaxes(got, 1, 2))
    assert np.abs(chi.cpu().numpy()[at] - O.chi(ref)).max() < 5e-5
    assert np.abs(mfc.cpu().numpy()[at] - O.mean_offdiag(want)).max() < 5e-5


@pytest.mark.parametrize("n_regions", [16, 68])
def test_fp32_fc_of_a_set_does_not_depend_on_the_others(tvbx, n_regions):
    import torch
    T = 1100
    x = 5e-3 + 1e-3 * torch.randn((T, n_regions, 5000), device="cuda")
    out = []
    for P in (5000, 777, 5):
        fc, chi = torch.empty((P, n_regions, n_regions), device="cuda"), torch.empty(P, device="cuda")
        tvbx.fc_series(x[:, :, :P].contiguous(), n_regions, P, T, fc_out=fc, chi=chi)
        out.append((fc[:5].clone(), chi[:5].clone()))
    for fc, chi in out[1:]:
        assert torch.equal(fc, out[0][0]) and torch.equal(chi, out[0][1])


@pytest.mark.parametrize("n_regions", [5, 130])
@pytest.mark.parametrize("window", [0, 32])
def test_a_variance_beyond_fp32_is_flagged(tvbx, n_regions, window):
    """A region whose squares overflow has no FC row, with windows and without."""
    import torch
    N, P, T = n_regions, 6, 64   # 64 samples: the shift is the mean of all of them
    x = 5e-3 + 1e-3 * torch.randn((T, N, P), device="cuda")
    x[:, 1, 2] = 3e18 * (1.0 - 2.0 * (torch.arange(T, device="cuda") % 2))   # sum of squares 5.8e38, of 32 samples 2.9e38
    x[:, 1, 3] = 2e-3
    fc, status = torch.empty((P, N, N), device="cuda"), torch.zeros(P, dtype=torch.int32, device="cuda")
    fcd = torch.empty((P, 3, 3), device="cuda") if window else None
    tvbx.fc_series(x, N, P, T, fc_out=fc, fcd_out=fcd, fcd_window=window, fcd_step=window // 2, set_status=status)
    flagged = (status.cpu().numpy() & tvbx.SET_ZERO_VAR) != 0
    assert flagged.tolist() == [False, False, True, True, False, False]
