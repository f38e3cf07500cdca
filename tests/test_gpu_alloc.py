"""The handles' device memory through a caller's allocator
(tvbx_set_allocator): PyTorch's caching allocator behind a counting wrapper
serves a sweep, and the sweep's series, state and FC equal those of a run on
the default cudaMalloc; every block is returned when the handle closes."""
import numpy as np
import pytest

from gpu_common import require_gpu
from paper_2311_13337_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tvbx():
    return require_gpu()


def test_sweep_on_the_torch_caching_allocator(tvbx, oracle):
    import torch
    W, L = synth.connectome(68)
    pts = oracle.expand_grid([("g", [0.1, 0.4]), ("b_e", [0.0, 60.0]), ("speed", [3.0, 6.0])])
    kw = dict(dt_ms=0.1, n_steps=3000, tavg_steps=10, seed=5)

    def run():
        sw = tvbx.Sweep(W, L, points=pts).run(**kw)
        out = (sw.series(), sw.state(), sw.fc(fcd_window=100, fcd_step=50, precision=tvbx.FC_BF16X3))
        return sw, out

    ref_sw, ref = run()
    ref_sw.close()
    live = {}

    def alloc(n):
        p = torch.cuda.caching_allocator_alloc(n)
        live[p] = n
        return p

    def free(p):
        assert p in live
        del live[p]
        torch.cuda.caching_allocator_delete(p)

    before = torch.cuda.memory_allocated()
    tvbx.set_allocator(alloc, free)
    try:
        sw, got = run()
        assert len(live) > 10 and torch.cuda.memory_allocated() - before >= sum(live.values())
        assert all(p % 256 == 0 for p in live)
        sw.run_continue(1000)            # grows and reuses buffers through the same pair
        sw.close()
        assert not live
    finally:
        tvbx.set_allocator()
    for a, b in zip(got[:2], ref[:2]):
        assert np.array_equal(a, b, equal_nan=True)
    for a, b in zip(got[2], ref[2]):
        assert np.array_equal(a, b, equal_nan=True)
    # the default allocator is back: a handle made now takes nothing from the pool
    n_before = torch.cuda.memory_allocated()
    sw = tvbx.Sweep(W, L, points=pts).run(**kw)
    assert torch.cuda.memory_allocated() == n_before
    sw.close()


def test_surrogate_and_batch_on_a_caller_allocator(tvbx, oracle):
    import torch
    live = {}

    def alloc(n):
        p = torch.cuda.caching_allocator_alloc(n)
        live[p] = n
        return p

    def free(p):
        del live[p]
        torch.cuda.caching_allocator_delete(p)

    tvbx.set_allocator(alloc, free)
    try:
        W, L = synth.connectome(68)
        jobs = [tvbx.Sweep(W, L, points=oracle.expand_grid([("g", [0.1, 0.3]), ("b_e", [0.0, 30.0 * j])]))
                for j in range(2)]
        cfg = dict(dt_ms=0.1, n_steps=1000, tavg_steps=10, seed=3)
        b = tvbx.Batch([(j, cfg) for j in jobs])
        b.run()
        assert jobs[1].series().shape == (4, 68, 100)
        b.close()
        for j in jobs:
            j.close()
        assert not live
        s = tvbx.Surrogate(np.zeros(5), np.ones(5), 24, n_hidden=64, n_layers=2, n_members=2, seed=1)
        assert live
        s.close()
        assert not live
    finally:
        tvbx.set_allocator()


class CappedAllocator:
    """Device memory through PyTorch's allocator, refused beyond `cap` live bytes."""

    callbacks = []   # for as long as a handle may hold memory of theirs

    def __init__(self, tvbx, cap=None):
        self.live, self.cap = {}, cap
        tvbx.set_allocator(self.alloc, self.free)
        self.callbacks.append(tvbx._allocator_refs)

    def alloc(self, n):
        import torch
        used = sum(self.live.values()) + n
        if self.cap is not None and used > self.cap:
            return 0
        p = torch.cuda.caching_allocator_alloc(n)
        self.live[p] = n
        return p

    def free(self, p):
        import torch
        del self.live[p]
        torch.cuda.caching_allocator_delete(p)


SLACK = 1 << 16   # small tables whose sizes depend on the tile width


def _window_inputs(tvbx, n_regions, n_sets, speed):
    """Delays of a few steps, where windows need the most memory beside the others."""
    W, L = synth.connectome(n_regions)
    m = tvbx.make_model()
    pts = np.tile(np.array([m.defaults[i] for i in range(tvbx.N_AXES)]), (n_sets, 1))
    rng = np.random.default_rng(n_sets)
    pts[:, tvbx.AXES.index("g")] = rng.uniform(0.0, 0.4, n_sets)
    pts[:, tvbx.AXES.index("b_e")] = rng.uniform(0.0, 120.0, n_sets)
    pts[:, tvbx.AXES.index("speed")] = speed
    return W, L, pts


def _peak(tvbx, inputs, kernel, kw):
    """Bytes a run holds, and its results."""
    mem = CappedAllocator(tvbx)
    sw = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2]).run(kernel=kernel, **kw)
    peak = sum(mem.live.values())
    out = (sw.series(), sw.state()) if kw.get("series_mode", 0) == 0 else (sw.state(),)
    sw.close()
    tvbx.set_allocator()
    return peak, out


@pytest.mark.parametrize("speed,streamed", [(100.0, False), (30.0, False), (30.0, True)])
def test_a_run_that_only_fits_without_windows_runs_without_them(tvbx, speed, streamed):
    inputs = _window_inputs(tvbx, 68, 640, speed)
    kw = dict(dt_ms=0.1, n_steps=200, tavg_steps=10, seed=5, keep_i_series=not streamed,
              series_mode=tvbx.SERIES_STREAM if streamed else tvbx.SERIES_KEEP)
    try:
        general, want = _peak(tvbx, inputs, tvbx.KERNEL_GENERAL, kw)
        windowed, got = _peak(tvbx, inputs, tvbx.KERNEL_AUTO, kw)
        for a, b in zip(want, got):
            assert np.array_equal(a, b)
        assert windowed > general + 2 * SLACK
        # the rings' own allocation refused, the last one, and between them the series'
        for cap in (general + SLACK, (general + windowed) // 2, windowed - SLACK):
            mem = CappedAllocator(tvbx, cap)
            sw = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2]).run(**kw)
            mem.cap = None
            got = (sw.series(), sw.state()) if not streamed else (sw.state(),)
            for a, b in zip(want, got):
                assert np.array_equal(a, b)
            sw.run_continue(50)
            again = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2]).run(**kw).run_continue(50)
            assert np.array_equal(sw.state(), again.state())
            again.close()
            sw.close()
            tvbx.set_allocator()
    finally:
        tvbx.set_allocator()


def test_a_batch_that_only_fits_without_windows_runs_without_them(tvbx):
    inputs = [_window_inputs(tvbx, n, p, v) for n, p, v in ((68, 640, 100.0), (84, 512, 30.0))]
    kw = dict(dt_ms=0.1, n_steps=1000, tavg_steps=5, seed=5)
    try:
        peaks = [[_peak(tvbx, x, kernel, kw) for kernel in (tvbx.KERNEL_GENERAL, tvbx.KERNEL_AUTO)] for x in inputs]
        more = sum(w[0] - g[0] for g, w in peaks)
        assert more > 4 * SLACK
        for tune in (False, True):
            cap = None
            for step in range(2):   # uncapped, then with room for half of what windows need more
                mem = CappedAllocator(tvbx, cap)
                sweeps = [tvbx.Sweep(W, L, points=pts) for W, L, pts in inputs]
                b = tvbx.Batch([(sw, kw) for sw in sweeps])
                if tune and step:
                    b.tune(trial_steps=50)
                b.run()
                if cap is None:
                    cap = sum(mem.live.values()) - more // 2
                mem.cap = None
                for sw, ((_, want), _) in zip(sweeps, peaks):
                    assert np.array_equal(sw.series(), want[0]) and np.array_equal(sw.state(), want[1])
                b.close()
                for sw in sweeps:
                    sw.close()
                tvbx.set_allocator()
    finally:
        tvbx.set_allocator()


def test_a_batch_returns_to_windows_once_they_fit(tvbx):
    """Without room for windows the untuned body is the documented one, and the
    next rebuild tries windows again."""
    inputs = [_window_inputs(tvbx, n, p, v) for n, p, v in ((68, 640, 100.0), (84, 512, 30.0))]
    kw = dict(dt_ms=0.1, n_steps=100, tavg_steps=10, seed=5)
    try:
        peaks = [[_peak(tvbx, x, kernel, kw)[0] for kernel in (tvbx.KERNEL_GENERAL, tvbx.KERNEL_AUTO)] for x in inputs]
        mem = CappedAllocator(tvbx)
        sweeps = [tvbx.Sweep(W, L, points=pts) for W, L, pts in inputs]
        b = tvbx.Batch([(sw, kw) for sw in sweeps]).run()
        info = b.info()
        assert info["threads"] == 128 and info["grid"] == info["items"] > 0
        want = [sw.state() for sw in sweeps]
        b.close()
        for sw in sweeps:
            sw.close()
        assert not mem.live
        mem = CappedAllocator(tvbx)
        sweeps = [tvbx.Sweep(W, L, points=pts) for W, L, pts in inputs]
        b = tvbx.Batch([(sw, kw) for sw in sweeps])
        mem.cap = sum((g + w) // 2 for g, w in peaks)   # of the jobs; the batch's own tables are below half the difference
        b.run()
        info = b.info()
        assert (info["threads"], info["smem_kb"]) == (512, 200)
        mem.cap = None
        sweeps[0].run(**kw)   # the job's buffers changed
        b.run()
        assert b.info()["threads"] == 128
        for sw, x in zip(sweeps, want):
            assert np.array_equal(sw.state(), x)
        b.close()
        for sw in sweeps:
            sw.close()
    finally:
        tvbx.set_allocator()


def test_fc_of_few_sets_without_room_for_their_moment_blocks(tvbx):
    """Few sets store up to 12 moment blocks each; where only one fits, the same
    sums are added up as they are formed."""
    inputs = _window_inputs(tvbx, 68, 16, 4.0)
    kw = dict(dt_ms=0.1, n_steps=4000, tavg_steps=1, seed=5)
    out, grown = [], []
    try:
        for _ in range(2):
            mem = CappedAllocator(tvbx)
            sw = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2]).run(**kw)
            run = sum(mem.live.values())
            mem.cap = run + grown[0] // 2 if grown else None
            summ = sw.summary()
            out.append((sw.fc(), summ["chi"], summ["mean_fc"]))
            grown.append(sum(mem.live.values()) - run)
            sw.close()
            tvbx.set_allocator()
    finally:
        tvbx.set_allocator()
    assert grown[0] > 4 * 12 * 16 * 68 * 69 and all(np.array_equal(a, b) for a, b in zip(*out))


def test_checkpoint_of_windows_with_little_memory_left(tvbx):
    """The ring is converted through as few slots at a time as fit."""
    inputs = _window_inputs(tvbx, 68, 640, 10.0)
    kw = dict(dt_ms=0.1, n_steps=100, tavg_steps=10, seed=5)
    cks = []
    try:
        for short in (False, True):
            mem = CappedAllocator(tvbx)
            sw = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2]).run(**kw)
            assert tvbx.last_window(sw.h) > 0
            if short:
                mem.cap = sum(mem.live.values()) + 3 * 4 * 68 * 672   # three slots
            cks.append(sw.checkpoint())
            again = tvbx.Sweep(inputs[0], inputs[1], points=inputs[2])
            mem.cap = None
            again.run(**kw)
            if short:
                mem.cap = sum(mem.live.values()) + 3 * 4 * 68 * 672
            again.restore(cks[-1])
            mem.cap = None
            assert np.array_equal(again.run_continue(20).state(), sw.run_continue(20).state())
            again.close()
            sw.close()
            tvbx.set_allocator()
    finally:
        tvbx.set_allocator()
    assert np.array_equal(*cks)
