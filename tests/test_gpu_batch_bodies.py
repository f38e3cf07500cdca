"""The bodies of a batch against its jobs run alone by the kernels without
windows, bit for bit: windows over ragged tiles, several speeds, shortest
delays of 0, 3 and 20 steps, noise of each set's own, a streamed job and both
transfer functions; and the persistent body, which jobs of different models
take, in its general and its register-tile form."""
import numpy as np
import pytest

from gpu_common import require_gpu
from test_gpu_window import _inputs

pytestmark = pytest.mark.gpu

DT = 0.1


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


def _results(tvbx, sw, kw):
    if kw.get("series_mode", tvbx.SERIES_KEEP) == tvbx.SERIES_STREAM:
        return [sw.state(), sw.fc(), *sw.summary().values()]
    summ = sw.summary() if sw.n_regions <= 384 else {}   # the FC behind it takes no more
    return [sw.state(), sw.series(), *summ.values()]


def _compare(tvbx, jobs, sweeps):
    for (inputs, model, kw), sw in zip(jobs, sweeps):
        alone = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2], model=model)
        alone.run(kernel=tvbx.KERNEL_GENERAL if sw.n_regions <= 360 else tvbx.KERNEL_DIRECT, **kw)
        for a, b in zip(_results(tvbx, alone, kw), _results(tvbx, sw, kw)):
            assert np.isfinite(a).all() and np.array_equal(a, b)
        alone.close()


def _batch(tvbx, jobs):
    sweeps = [tvbx.Sweep(x[0], x[1], points=x[2], model=model) for x, model, _ in jobs]
    return sweeps, tvbx.Batch([(sw, kw) for sw, (_, _, kw) in zip(sweeps, jobs)])


def _close(sweeps, b):
    b.close()
    for sw in sweeps:
        sw.close()


def _cfg(n_steps, tavg, **kw):
    return dict(dt_ms=DT, n_steps=n_steps, tavg_steps=tavg, seed=5, **kw)


@pytest.mark.parametrize("tau_i", [None, 6.0])
def test_windows_equal_the_jobs_alone(tvbx, tau_i):
    model = None if tau_i is None else tvbx.make_model({"tau_i": tau_i})
    jobs = [(_inputs(tvbx, 68, 65, 0), model, _cfg(100, 10)),
            (_inputs(tvbx, 68, 131, 3, speeds=(1.0, 2.0, 4.0)), model, _cfg(130, 10, noise_per_set=True)),
            (_inputs(tvbx, 40, 131, 20, speeds=(1.0, 4.0)), model, _cfg(147, 5)),
            (_inputs(tvbx, 33, 70, 5), model,
             _cfg(190, 10, series_mode=tvbx.SERIES_STREAM, chunk_steps=50, transient_samples=3))]
    sweeps, b = _batch(tvbx, jobs)
    for _ in range(2):
        b.run()
        assert b.info()["threads"] == 128 and b.info()["grid"] == b.info()["items"]   # windows
        _compare(tvbx, jobs, sweeps)
    _close(sweeps, b)


def test_jobs_of_two_models_take_the_persistent_body(tvbx):
    jobs = [(_inputs(tvbx, 68, 65, 0), None, _cfg(100, 10)),
            (_inputs(tvbx, 84, 33, 9, speeds=(1.0, 4.0)), tvbx.make_model({"tau_i": 6.0}), _cfg(130, 10)),
            (_inputs(tvbx, 200, 20, 3), tvbx.make_model({"E_L_i": -66.0, "T": 25.0}), _cfg(90, 10, noise_per_set=True)),
            (_inputs(tvbx, 33, 70, 5), None,
             _cfg(190, 10, series_mode=tvbx.SERIES_STREAM, chunk_steps=50, transient_samples=3))]
    sweeps, b = _batch(tvbx, jobs)
    b.run()
    info = b.info()
    assert (info["threads"], info["smem_kb"]) == (512, 200)
    _compare(tvbx, jobs, sweeps)
    b.tune(trial_steps=50)   # whichever body is the fastest
    b.run()
    _compare(tvbx, jobs, sweeps)
    _close(sweeps, b)


def test_register_tiles_of_a_batch(tvbx):
    """400 regions do not fit the general body: the tuner can only take the register tiles."""
    jobs = [(_inputs(tvbx, 400, 21, 6), None, _cfg(60, 10)),
            (_inputs(tvbx, 68, 65, 2, speeds=(1.0, 4.0)), tvbx.make_model({"tau_i": 6.0}), _cfg(100, 10)),
            (_inputs(tvbx, 520, 9, 14), None, _cfg(50, 10, noise_per_set=True))]
    sweeps, b = _batch(tvbx, jobs)
    threads, _, trials = b.tune(trial_steps=50)
    assert threads == 768 and np.isfinite(trials).tolist() == [False] * 7 + [True]
    b.run()
    _compare(tvbx, jobs, sweeps)
    _close(sweeps, b)
