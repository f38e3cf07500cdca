"""Table 2 metrics at the edges of the phase-lag tiles and of the UP / DOWN
counts: region counts on both sides of a block, tile sizes for many regions,
odd and short lengths, rows that repeat, are constant, or leave a state once,
against the FP64 oracle."""
import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import analysis as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


def mean_pli(x):
    """Mean phase lag index with every row transformed on its own: a batched
    transform may round identical rows differently, and their lag sign is 0."""
    z = np.stack([A.analytic_signal(row) for row in x])
    n = x.shape[1]
    lag = [abs(np.sign(z[k].imag * z[k + 1:].real - z[k].real * z[k + 1:].imag).sum(axis=1)) / n
           for k in range(len(z) - 1)]
    return np.concatenate(lag).mean()


@pytest.mark.parametrize("n_regions,n_samples", [(2, 2), (3, 4), (5, 33), (8, 100), (9, 6), (101, 130), (197, 64),
                                                 (360, 40), (752, 12), (21, 8191), (4, 1025)])
def test_metrics_at_edges(tvbx, n_regions, n_samples):
    import torch
    rng = np.random.default_rng(n_regions + n_samples)
    x = (5e-3 + 1e-3 * rng.standard_normal((3, n_regions, n_samples))).astype(np.float32)
    x[1, 0] = 2e-3                      # no transition
    x[1, -1] = x[1, n_regions // 2]     # identical rows: lag sign 0
    x[2, 0] = np.where(np.arange(n_samples) < n_samples // 2, 1e-3, 4e-3)   # one transition
    out, used = tvbx.series_analysis(torch.from_numpy(x).cuda(), 1.0)
    got = out.cpu().numpy().astype(np.float64)
    for p in range(3):
        want = A.table2_metrics(x[p], 1.0)
        assert used == want["n_samples"]
        want["mean_pli"] = mean_pli(x[p].astype(np.float64)[:, n_samples - used:])
        for i, name in enumerate(tvbx.AN_FIELDS):
            g, w = got[p, i], want[name]
            if np.isnan(w):
                assert np.isnan(g), name
            elif name in ("n_up", "up_samples", "n_down", "down_samples"):
                assert g == w, name
            elif name == "mean_pli":
                # a sign may flip where |sin| of the phase difference is below the transforms'
                # relative error (about 1e-6): one of n samples of one pair in 1e5
                assert abs(g - w) < 1e-3, name
            elif name == "psd_b":
                assert abs(g - w) <= 1e-3 * abs(w), name
            else:
                assert abs(g - w) <= 1e-4 * abs(w) + 1e-7, name


@pytest.mark.parametrize("n_regions,n_samples", [(6, 100), (68, 1301), (101, 64)])
def test_phase_lag_without_sign(tvbx, n_regions, n_samples):
    """A region of NaN or infinities has no sign in any pair, like a silent one,
    and the other pairs keep theirs; a set of silent regions has none."""
    import torch
    rng = np.random.default_rng(n_regions)
    x = (5e-3 + 1e-3 * rng.standard_normal((4, n_regions, n_samples))).astype(np.float32)
    x[1:] = x[0]
    x[0, 2] = 2e-3
    x[1, 2] = np.nan
    x[2, 2, 7] = np.inf
    x[3] = 2e-3
    out, _ = tvbx.series_analysis(torch.from_numpy(x).cuda(), 1.0)
    lag = out.cpu().numpy()[:, tvbx.AN_FIELDS.index("mean_pli")]
    assert lag[0] > 0 and lag[1] == lag[0] and lag[2] == lag[0] and lag[3] == 0


@pytest.mark.parametrize("scale", [1e-19, 1e-21, 1e-22, 1e-23, 1e-24, 1e-30])
@pytest.mark.parametrize("n_regions,n_samples", [(6, 100), (33, 1301)])
def test_phase_lag_of_signals_whose_products_underflow(tvbx, scale, n_regions, n_samples):
    """A sample has a sign where its two products, rounded to FP32, differ: none
    where both underflow to zero, of either sign."""
    import torch
    rng = np.random.default_rng(n_samples)
    x = (scale * rng.standard_normal((2, n_regions, n_samples))).astype(np.float32)
    x[1, 0] = 5e-3   # a silent region beside them
    out, used = tvbx.series_analysis(torch.from_numpy(x).cuda(), 1.0)
    got = out.cpu().numpy()[:, tvbx.AN_FIELDS.index("mean_pli")]
    for p in range(2):
        z = [A.analytic_signal(row) for row in x[p].astype(np.float64)[:, n_samples - used:]]
        re, im = np.float32([v.real for v in z]), np.float32([v.imag for v in z])
        if p == 1:
            re[0] = im[0] = 0.0
        lag = []
        for k in range(n_regions - 1):
            a, b = im[k] * re[k + 1:], re[k] * im[k + 1:]
            lag.append(abs((a > b).sum(axis=1) - (a < b).sum(axis=1)) / used)
        want = np.concatenate(lag).mean()
        # the transforms' relative error (about 1e-6) moves the rounding of one product
        # of some 1e4 at most (products of 1e-43 are 100 units of the least FP32 number)
        assert abs(got[p] - want) < 1e-3
        if scale <= 1e-24:
            assert got[p] == 0.0


def test_threshold_keeps_the_last_bits_of_the_sum(tvbx):
    """Three samples of one thread whose FP64 sum, 1 + 2^-24 + 2^-50, lies just
    above a tie of the threshold's FP32 rounding: the sample at the threshold is
    not above it."""
    import torch
    n = 1024
    x = np.zeros((1, 2, n), dtype=np.float32)
    x[0, 0, [0, 256, 512]] = 1.0, 2.0 ** -24, 2.0 ** -50
    at = np.float32((1.0 + 2.0 ** -23) / n)
    x[0, 0, [5, 261]] = at, -at
    x[0, 1, ::3] = 1e-3
    assert x[0, 0].sum(dtype=np.float64) == 1.0 + 2.0 ** -24 + 2.0 ** -50
    out, used = tvbx.series_analysis(torch.from_numpy(x).cuda(), 1.0)
    want = A.table2_metrics(x[0], 1.0)
    assert used == n
    got = out.cpu().numpy()[0]
    for name in ("n_up", "up_samples", "n_down", "down_samples"):
        assert got[tvbx.AN_FIELDS.index(name)] == want[name], name
