"""The windowed simulation kernel (the automatic choice) against the general kernel on the edges of its windows, tiles and gather
passes: state, series, status and checkpoint equal bit for bit (both sum the
coupling in the same order and share the integrator)."""
import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

DT = 0.1


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


def _inputs(tvbx, n_regions, n_sets, d_min, speeds=(4.0,)):
    """Connectome whose shortest delay is d_min steps at the fastest speed,
    with a region without input and one fully connected."""
    rng = np.random.default_rng(100 * n_regions + n_sets + d_min)
    W = rng.uniform(0.1, 1.0, (n_regions, n_regions)) * (rng.random((n_regions, n_regions)) < 0.3)
    W[0] = 0.0
    W[-1] = rng.uniform(0.1, 1.0, n_regions)
    L = rng.uniform(d_min, 3 * d_min + 20, (n_regions, n_regions)) * DT * max(speeds)
    L[-1, 0] = d_min * DT * max(speeds)
    L[-1, -1] = (3 * d_min + 20) * DT * max(speeds)
    m = tvbx.make_model()
    pts = np.tile(np.array([m.defaults[i] for i in range(tvbx.N_AXES)]), (n_sets, 1))
    ix = tvbx.AXES.index
    pts[:, ix("g")] = rng.uniform(0.0, 10.0 / n_regions, n_sets)
    pts[:, ix("b_e")] = rng.uniform(0.0, 120.0, n_sets)
    pts[:, ix("E_L_i")] = rng.uniform(-80.0, -66.0, n_sets)
    pts[:, ix("speed")] = np.asarray(speeds)[rng.integers(0, len(speeds), n_sets)]
    return W, L, pts


def _run(tvbx, inputs, kernel, n_steps, more=0, **kw):
    W, L, pts = inputs
    sw = tvbx.Sweep(W, L, points=pts)
    sw.run(dt_ms=DT, n_steps=n_steps, seed=5, kernel=kernel, **kw)
    if more:
        sw.run_continue(more)
    out = [sw.state(), sw.series(), sw.summary()["status"]]
    ck = sw.checkpoint()
    sw.close()
    return out, ck


# d_min (windows of up to one step more): zero delays; far entries apart with
# windows of 2 to 6 steps; windows of 8, 16, 24 and 32 steps and ends with gather
# passes of 4, 2 and 1; sets: one, odd pairs, tiles of 64 and a rest
@pytest.mark.parametrize("n_regions,n_sets,d_min,n_steps,tavg,noise", [
    (5, 1, 1, 40, 4, False), (5, 1, 2, 41, 4, False), (7, 3, 7, 100, 10, True), (68, 2, 9, 130, 10, False),
    (68, 65, 16, 147, 7, False), (33, 131, 40, 90, 1, True), (68, 1203, 5, 63, 9, False), (68, 1251, 19, 50, 10, True),
    (200, 450, 12, 55, 5, False),
    (200, 401, 3, 50, 10, True), (16, 70, 15, 64, 8, False), (68, 701, 9, 44, 4, False), (100, 401, 2, 30, 3, True),
    (5, 1, 0, 40, 4, False), (68, 131, 0, 50, 10, True), (100, 401, 0, 30, 3, False), (200, 450, 0, 45, 5, False),
    (68, 1203, 6, 48, 8, False), (68, 701, 7, 45, 9, False), (33, 70, 31, 99, 3, False), (33, 70, 30, 99, 3, False),
])
def test_window_equals_general_kernel(tvbx, n_regions, n_sets, d_min, n_steps, tavg, noise):
    inputs = _inputs(tvbx, n_regions, n_sets, d_min)
    kw = dict(tavg_steps=tavg, noise_per_set=noise, chunk_steps=3 * tavg)
    more = 2 * tavg if n_steps % tavg == 0 else 0
    want, ck_want = _run(tvbx, inputs, tvbx.KERNEL_GENERAL, n_steps, more, **kw)
    got, ck_got = _run(tvbx, inputs, tvbx.KERNEL_AUTO, n_steps, more, **kw)
    for a, b in zip(want, got):
        assert np.isfinite(a).all() and np.array_equal(a, b)
    # the checkpoint's body (state, rings, noise) does not depend on the kernel
    header = 15 * 8
    assert np.array_equal(ck_want[header:], ck_got[header:])


def test_window_of_the_general_template(tvbx):
    """Unequal synaptic time constants take the template itself, one set per thread."""
    W, L, pts = _inputs(tvbx, 30, 40, 6)
    out = []
    for kernel in (tvbx.KERNEL_GENERAL, tvbx.KERNEL_AUTO):
        sw = tvbx.Sweep(W, L, points=pts, model=tvbx.make_model({"tau_i": 6.0}))
        sw.run(dt_ms=DT, n_steps=50, tavg_steps=5, seed=3, kernel=kernel)
        out.append((sw.state(), sw.series()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_window_with_several_speeds_restores_from_a_checkpoint(tvbx):
    W, L, pts = _inputs(tvbx, 40, 77, 6, speeds=(1.0, 2.0, 4.0))
    a = tvbx.Sweep(W, L, points=pts)
    a.run(dt_ms=DT, n_steps=150, tavg_steps=10, seed=2)
    ck = a.checkpoint()
    a.run_continue(70)
    b = tvbx.Sweep(W, L, points=pts)
    b.restore(ck)
    b.run_continue(70)
    assert np.array_equal(a.state(), b.state()) and np.array_equal(a.series(), b.series())
    g = tvbx.Sweep(W, L, points=pts)
    g.run(dt_ms=DT, n_steps=220, tavg_steps=10, seed=2, kernel=tvbx.KERNEL_GENERAL)
    assert np.array_equal(a.state(), g.state())


def test_a_set_does_not_depend_on_the_other_speeds(tvbx):
    """Short delays of one speed change how the sweep runs, not what a set of
    another speed gives."""
    W, L, pts = _inputs(tvbx, 40, 30, 3, speeds=(1.0, 4.0))
    slow = pts[:, tvbx.AXES.index("speed")] == 1.0
    both, alone = tvbx.Sweep(W, L, points=pts), tvbx.Sweep(W, L, points=pts[slow])
    for sw in (both, alone):
        sw.run(dt_ms=DT, n_steps=100, tavg_steps=10, seed=4)
    assert np.array_equal(both.state()[slow], alone.state())
    assert np.array_equal(both.series()[slow], alone.series())


@pytest.mark.parametrize("d_min,steps", [(0, 1), (5, 6), (12, 8), (18, 16), (40, 32)])
def test_reports_tell_windows_from_the_other_kernels(tvbx, d_min, steps):
    W, L, pts = _inputs(tvbx, 30, 10, d_min)
    sw = tvbx.Sweep(W, L, points=pts)
    for kernel, want in ((tvbx.KERNEL_AUTO, steps), (tvbx.KERNEL_DIRECT, 0), (tvbx.KERNEL_GENERAL, 0)):
        tvbx.profile_enable(sw.h)
        sw.run(dt_ms=DT, n_steps=90, tavg_steps=10, kernel=kernel, chunk_steps=50)
        _, launches, updates = tvbx.profile_read(sw.h)
        assert tvbx.last_window(sw.h) == want and ("window" in tvbx.kernel_name(sw.h)) == (want > 0)
        assert updates == 30 * 10 * 90
        # far sums once every 16 steps beside windows of fewer than 8, which end with them
        count = sum((n // 16 * -(-16 // steps) + -(-(n % 16) // steps) + -(-n // 16)) if steps < 8 else -(-n // steps)
                    for n in (50, 40))
        assert launches == (count if want else 2)
    sw.close()
