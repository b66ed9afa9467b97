"""What the library's host code does around its kernels, on a CUDA runtime of
host memory (host_runtime.cpp): which buffers outlive which work, what a failed
allocation leaves behind, what a call reports."""
import ctypes

import numpy as np
import pytest

import host_runtime


@pytest.fixture()
def rc(tmp_path):
    return host_runtime.load(tmp_path)


def tile(H, W, value=9):
    """(mask, marker, descriptor); the stand-in reconstruction sets the marker to the mask."""
    I, J = np.full((H, W), value, np.uint8), np.zeros((H, W), np.uint8)
    return I, J, (I.ctypes.data, J.ctypes.data, H, W, W, 8)


def done(tiles):
    return all((J == I).all() for I, J, _ in tiles)


def test_graph_is_not_replayed_from_a_staging_buffer_that_is_gone(rc):
    """An explicit schedule is replayed as a graph that copies from the staging
    buffer; a larger batch on the other engine in between replaces that buffer."""
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    one, many = tile(10, 12), [tile(5, 5) for _ in range(40)]
    for _ in range(3):
        one[1][:] = 0
        assert rc.recon_batch_ex(c, [one[2]], [1], [0]) == rc.RECON_OK and done([one])
        assert rc.recon_batch(c, [t[2] for t in many]) == rc.RECON_OK and done(many)
    assert rc.lib().ht_faults() == 0
    assert host_runtime.counts(rc)["graph"] == 3
    rc.recon_free(c)


def mix(z):
    z = (z + 0x9E3779B97F4A7C15) % (1 << 64)
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) % (1 << 64)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) % (1 << 64)
    return z ^ (z >> 31)


def order(n, seed, epoch):
    perm, st = list(range(n)), mix(seed ^ mix(epoch + 1))
    for i in range(n - 1, 0, -1):
        st = mix(st)
        perm[i], perm[st % (i + 1)] = perm[st % (i + 1)], perm[i]
    return perm


@pytest.mark.parametrize("n,epochs", [(1, 3), (7, 1), (50, 2), (1000, 6), (20000, 3)])
def test_every_epoch_trains_on_its_own_order(rc, n, epochs):
    """The host shuffles ahead; an order is copied only when the device gets to it."""
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    a = np.zeros(3 * rc.RECON_MLP_NPARAMS, np.float32)
    X = np.zeros((n, 22), np.float32)
    st, losses = rc.recon_mlp_train(c, a.ctypes.data, X.ctypes.data, X.ctypes.data, n, epochs, n, 1e-3, 5)
    assert st == rc.RECON_OK and losses == [1.0] * epochs
    st, step, losses = rc.recon_mlp_train_resume(c, a.ctypes.data, a.ctypes.data, epochs, epochs, X.ctypes.data,
                                                 X.ctypes.data, n, 2, n, 1e-3, 5)
    assert st == rc.RECON_OK and step == epochs + 2
    got = (ctypes.c_int * (n * (epochs + 2)))()
    assert rc.lib().ht_orders(got, len(got)) == len(got)
    for e in range(epochs + 2):
        assert list(got[e * n:(e + 1) * n]) == order(n, 5, e), e
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


@pytest.mark.parametrize("flag", [0, "RECON_FLAG_NO_GRAPH"])
@pytest.mark.parametrize("wavefront", [False, True])
@pytest.mark.parametrize("n", [1, 3])
def test_a_capturing_stream_is_refused_untouched(rc, flag, wavefront, n):
    L, st = rc.lib(), ctypes.c_void_p()
    assert L.cudaStreamCreateWithFlags(ctypes.byref(st), 0) == 0
    c = rc.recon_init(0, st.value, rc.RECON_FLAG_SYNC | (getattr(rc, flag) if flag else 0))
    tiles = [tile(70, 65) for _ in range(n)]
    def run():
        desc = [t[2] for t in tiles]
        return rc.recon_batch_ex(c, desc, [1] * n, list(range(n))) if wavefront else rc.recon_batch(c, desc)
    for warm in range(2):
        assert L.cudaStreamBeginCapture(st, 0) == 0
        assert run() == rc.RECON_ECUDA
        g = ctypes.c_void_p()
        assert L.cudaStreamEndCapture(st, ctypes.byref(g)) == 0
        assert L.ht_broken_captures() == 0 and L.ht_graph_nodes(g) == 0 and L.cudaGraphDestroy(g) == 0
        assert run() == rc.RECON_OK and done(tiles)
        for t in tiles:
            t[1][:] = 0
    rc.recon_free(c)


@pytest.mark.parametrize("first_wavefront", [False, True])
@pytest.mark.parametrize("then_wavefront", [False, True])
@pytest.mark.parametrize("violation", [False, True])
def test_a_failed_allocation_leaves_nothing_stale(rc, first_wavefront, then_wavefront, violation):
    """A call that cannot grow its buffers: the status of the call before it stays,
    its counters are refused (their buffer may be gone), and the next call works."""
    c = rc.recon_init(0, 0, 0)

    def run(tiles, wavefront):
        n, desc = len(tiles), [t[2] for t in tiles]
        return rc.recon_batch_ex(c, desc, [1] * n, list(range(n))) if wavefront else rc.recon_batch(c, desc)
    few, many = [tile(5, 5) for _ in range(3)], [tile(2, 2) for _ in range(3000)]
    if violation:
        few[1][1][0, 0] = 10
    assert run(few, first_wavefront) == rc.RECON_OK
    status = rc.RECON_EMARKER if violation else rc.RECON_OK
    if not violation:
        assert [w["visits"] for w in rc.recon_get_work(c, 3)] == [1, 1, 1]
    rc.lib().ht_device_limit(rc.lib().ht_device_bytes())
    assert run(many, then_wavefront) == rc.RECON_ENOMEM
    assert rc.recon_sync(c) == status and rc.recon_last_error_tile(c) == (1 if violation else -1)
    with pytest.raises(rc.ReconError):
        rc.recon_get_work(c, 1)
    assert rc.lib().ht_faults() == 0
    rc.lib().ht_device_limit(1 << 40)
    assert run(many, then_wavefront) == rc.RECON_OK and rc.recon_sync(c) == rc.RECON_OK and done(many)
    assert len(rc.recon_get_work(c, 3000)) == 3000
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


@pytest.mark.parametrize("n", [1, 4])
def test_the_wavefront_engine_takes_over_without_scratch(rc, n):
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    tiles = [tile(700, 900) for _ in range(n)]
    rc.lib().ht_device_limit(rc.lib().ht_device_bytes() + (1 << 19))
    assert rc.recon_batch(c, [t[2] for t in tiles]) == rc.RECON_OK and done(tiles)
    assert host_runtime.counts(rc)["wavefront"] == 1 and host_runtime.counts(rc)["merging"] == 0
    assert all(w["scan_rows"] for w in rc.recon_get_work(c, n))
    rc.lib().ht_device_limit(1 << 40)
    for t in tiles:
        t[1][:] = 0
    assert rc.recon_batch(c, [t[2] for t in tiles]) == rc.RECON_OK and done(tiles)
    assert host_runtime.counts(rc)["merging"] == 1
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


def test_a_host_batch_on_the_wavefront_engine_is_one_launch(rc):
    """Below 256 Mpx: one launch, replayed as a graph, reported as a whole."""
    c = rc.recon_init(0, 0, 0)
    assert rc.recon_set_param(c, rc.RECON_P_REVISIT_SCANS, 1) == rc.RECON_OK
    tiles = [tile(1800, 1700) for _ in range(4)]
    for k in (1, 2):
        assert rc.recon_batch_host(c, [t[2] for t in tiles]) == rc.RECON_OK and done(tiles)
        assert host_runtime.counts(rc) == dict(merging=0, wavefront=k, graph=k, plan=0)
        assert [w["scan_rows"] for w in rc.recon_get_work(c, 4)] == [1800] * 4
        for t in tiles:
            t[1][:] = 0
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


@pytest.mark.parametrize("bad", [None, 0, 4])
def test_a_host_batch_in_segments_reports_as_a_whole(rc, bad):
    """8 to 256 Mpx on the merging engine: several runs, but the counters are those
    of all tiles and the time (a nanosecond a pixel here) that of all runs, also
    when a tile is refused."""
    c = rc.recon_init(0, 0, 0)
    tiles = [tile(64 * (20 + k), 1700) for k in range(5)]
    for rep in range(2):
        if bad is not None:
            tiles[bad][1][5, 6] = 10
        want = rc.RECON_OK if bad is None else rc.RECON_EMARKER
        assert rc.recon_batch_host(c, [t[2] for t in tiles]) == want
        assert rc.recon_last_error_tile(c) == (-1 if bad is None else bad) and rc.recon_sync(c) == want
        assert [w["visits"] for w in rc.recon_get_work(c, 5)] == [27 * (20 + k) for k in range(5)]
        px = sum(I.size for k, (I, _, _) in enumerate(tiles) if k != bad)
        assert rc.recon_last_kernel_ms(c) == pytest.approx(1e-6 * px, rel=1e-5)
        assert host_runtime.counts(rc)["merging"] == 4 * (rep + 1)
        for _, J, _ in tiles:
            J[:] = 0
    small = tile(70, 70)   # the next call's own figures
    assert rc.recon_batch(c, [small[2]]) == rc.RECON_OK and rc.recon_sync(c) == rc.RECON_OK
    assert [w["visits"] for w in rc.recon_get_work(c, 1)] == [4]
    assert rc.recon_last_kernel_ms(c) == pytest.approx(1e-6 * 4900, rel=1e-2)
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


@pytest.mark.parametrize("op", ["RECON_OP_DILATE", "RECON_OP_FILL_HOLES"])
@pytest.mark.parametrize("bad", [0, 4])
def test_a_refused_host_batch_changes_nothing(rc, op, bad):
    """The markers are as they were when any tile is refused (a FillHoles tile's J is
    output only; in a batch with others it is left alone too)."""
    c = rc.recon_init(0, 0, 0)
    tiles = [tile(1300 + k, 1700) for k in range(5)]
    tiles[bad][1][5, 6] = 10
    desc = [t[2] + (rc.RECON_OP_DILATE if k == bad else getattr(rc, op),) for k, t in enumerate(tiles)]
    before = [J.copy() for _, J, _ in tiles]
    for _ in range(2):
        assert rc.recon_batch_host(c, desc) == rc.RECON_EMARKER and rc.recon_last_error_tile(c) == bad
        assert all((J == b).all() for (_, J, _), b in zip(tiles, before))
    tiles[bad][1][5, 6] = 0
    assert rc.recon_batch_host(c, desc) == rc.RECON_OK and done(tiles)
    assert host_runtime.counts(rc)["merging"] == 12
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


def test_the_autotuner_tunes_the_wavefront_engine_and_moves_no_call(rc):
    """Every trial runs on the wavefront engine; what it installs, from trials or from
    a cache, applies there, and a call on default settings stays where it was."""
    c, c2 = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC), rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    t = tile(70, 80)

    def installed(ctx):
        return tuple(rc.recon_get_param(ctx, k) for k in (rc.RECON_P_BLOCK_H, rc.RECON_P_BANDS, rc.RECON_P_SWEEPS,
                                                          rc.RECON_P_SCAN_GAIN))

    def engine(ctx):
        before = host_runtime.counts(rc)
        t[1][:] = 0
        assert rc.recon_batch(ctx, [t[2]]) == rc.RECON_OK and done([t])
        return [k for k in ("merging", "wavefront") if host_runtime.counts(rc)[k] > before[k]]
    st, best = rc.recon_autotune(c, [t[2]], 1)
    assert st == rc.RECON_OK and not t[1].any() and best == installed(c) != (128, 4, 1, 2048)
    assert host_runtime.counts(rc)["merging"] == 0 and host_runtime.counts(rc)["wavefront"] == 2 * 36
    assert engine(c) == ["merging"]
    assert rc.recon_autotune_cache_load(c2, rc.recon_autotune_cache(c)[1]) == rc.RECON_OK
    t[1][:] = 0
    assert rc.recon_autotune(c2, [t[2]], 1) == (rc.RECON_OK, best) and installed(c2) == best
    assert engine(c2) == ["merging"]
    assert rc.recon_set_param(c2, rc.RECON_P_REVISIT_SCANS, 1) == rc.RECON_OK and engine(c2) == ["wavefront"]
    assert installed(c2) == best
    rc.recon_free(c)
    rc.recon_free(c2)
    assert rc.lib().ht_faults() == 0


def test_the_learned_schedule_is_planned_where_the_wavefront_engine_runs(rc):
    """Once a batch in recon_batch, once a segment in a host batch; never for the
    merging engine, which has no schedule."""
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC | rc.RECON_FLAG_LEARNED)
    assert rc.recon_sched_set_model(c, [0.0] * rc.RECON_MLP_NPARAMS, [0, 1, 0, 1], 1, 2) == rc.RECON_OK
    small = [tile(40, 50) for _ in range(3)]
    large = [tile(8192, 8256) for _ in range(4)]   # 271 Mpx: four segments on either engine
    plans = []
    for setting in (0, 1):
        assert rc.recon_set_param(c, rc.RECON_P_REVISIT_SCANS, setting) == rc.RECON_OK
        for run, tiles in ((rc.recon_batch, small), (rc.recon_batch_host, large)):
            for t in tiles:
                t[1][:] = 0
            before = host_runtime.counts(rc)
            assert run(c, [t[2] for t in tiles]) == rc.RECON_OK and done(tiles)
            now = host_runtime.counts(rc)
            plans.append(tuple(now[k] - before[k] for k in ("merging", "wavefront", "plan")))
    assert plans == [(1, 0, 0), (4, 0, 0), (0, 1, 1), (0, 4, 4)]
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


@pytest.mark.parametrize("n,batch", [(5, 2), (64, 64), (10, 100)])
def test_training_without_the_cluster_takes_the_same_steps(rc, n, batch):
    """A device that cannot place sixteen CTAs together: gradient and Adam launches, the
    same samples in the same order, the steps numbered on."""
    rc.lib().ht_train_fits(0)
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    a = np.zeros(3 * rc.RECON_MLP_NPARAMS, np.float32)
    X = np.zeros((n, 22), np.float32)
    per = -(-n // batch)
    st, losses = rc.recon_mlp_train(c, a.ctypes.data, X.ctypes.data, X.ctypes.data, n, 3, batch, 1e-3, 5)
    assert st == rc.RECON_OK and losses == [1.0] * 3
    st, step, _ = rc.recon_mlp_train_resume(c, a.ctypes.data, a.ctypes.data, 3 * per, 3, X.ctypes.data, X.ctypes.data,
                                            n, 1, batch, 1e-3, 5)
    assert st == rc.RECON_OK and step == 4 * per
    got, steps = (ctypes.c_int * (4 * n))(), (ctypes.c_int * (4 * per))()
    assert rc.lib().ht_orders(got, 4 * n) == 4 * n and rc.lib().ht_steps(steps, 4 * per) == 4 * per
    assert list(got) == [i for e in range(4) for i in order(n, 5, e)]
    assert list(steps) == list(range(1, 4 * per + 1))
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


def test_a_host_batch_in_segments_without_scratch_for_the_merging_engine(rc):
    """The wavefront engine takes over segment by segment; its control word and its
    counters lie in buffers of their own."""
    c = rc.recon_init(0, 0, 0)
    tiles = [tile(64 * (20 + k), 1700) for k in range(5)]
    px = sum(I.size for I, _, _ in tiles)
    rc.lib().ht_device_limit(rc.lib().ht_device_bytes() + 2 * px + (3 << 20))
    assert rc.recon_batch_host(c, [t[2] for t in tiles]) == rc.RECON_OK and done(tiles)
    assert host_runtime.counts(rc)["wavefront"] == 4 and host_runtime.counts(rc)["merging"] == 0
    assert [w["scan_rows"] for w in rc.recon_get_work(c, 5)] == [64 * (20 + k) for k in range(5)]
    assert rc.recon_last_kernel_ms(c) == pytest.approx(1e-6 * px, rel=1e-5)
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0


def test_a_failed_pinned_allocation_is_reported_once(rc):
    """Its error must not show again in the check after the next launch."""
    c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
    few, many = [tile(5, 5) for _ in range(2)], [tile(2, 2) for _ in range(2000)]
    a, X = np.zeros(3 * rc.RECON_MLP_NPARAMS, np.float32), np.zeros((5000, 22), np.float32)

    def train(n):
        return rc.recon_mlp_train(c, a.ctypes.data, X.ctypes.data, X.ctypes.data, n, 2, 10, 1e-3)[0]
    rc.lib().ht_pinned_limit(1 << 12)
    assert rc.recon_batch(c, [t[2] for t in many]) == rc.RECON_ENOMEM
    assert rc.recon_batch(c, [t[2] for t in few]) == rc.RECON_OK and done(few)
    assert train(5000) == rc.RECON_ENOMEM and train(20) == rc.RECON_OK
    rc.lib().ht_pinned_limit(1 << 40)
    assert rc.recon_batch(c, [t[2] for t in many]) == rc.RECON_OK and done(many)
    assert train(5000) == rc.RECON_OK
    rc.recon_free(c)
    assert rc.lib().ht_faults() == 0
