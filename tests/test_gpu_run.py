"""The resident run kernel (small systems: many steps in one launch) against the
same steps launched one kernel at a time: the same bits, at the sizes where
its forms change and across list rebuilds, Hilbert resorts and calls of odd
lengths; and a run it cannot finish reports what stopped it."""
import ctypes

import numpy as np
import pytest

from paper_2608_14911_gb300 import espp, inputs as I

from _systems import WCA_RC, kg_case

pytestmark = pytest.mark.gpu
FP32, FP64 = espp.ESPP_FP32, espp.ESPP_FP64


def _melt(chains, beads, prec, chunk=None):
    c = I.kg_lattice(chains, beads, density=0.85, seed=4)
    s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=4)
    s.set_wca()
    s.set_fene()
    if chunk is not None:
        s.set_graph_chunk(chunk)
    s.set_resort_interval(20)
    s.set_state(c.x, I.maxwell_velocities(c.n, 1.0, seed=4), c.img)
    s.build_neighbors(WCA_RC, 0.4)
    return s


@pytest.mark.parametrize("prec,chains,beads", [
    (FP32, 3, 43),        # a partial tile (129)
    (FP32, 40, 100),
    (FP32, 304, 128),     # the last size with 16 entries in flight
    (FP32, 305, 128),     # and the next
    (FP64, 3, 43),
    (FP64, 114, 128),     # the last size with four lanes per particle
    (FP64, 115, 128),
])
def test_run_equals_single_launches(prec, chains, beads):
    a, b = _melt(chains, beads, prec), _melt(chains, beads, prec, chunk=0)
    for n in (1, 2, 19, 33):
        a.integrate(n, 0.005, 1.0, 1.0)
        b.integrate(n, 0.005, 1.0, 1.0)
        assert a.step == b.step and a.n_rebuilds == b.n_rebuilds
        for p, q in zip(a.get_state(), b.get_state()):
            assert np.array_equal(p, q)
    assert a.n_rebuilds > 4
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_direct_launches_keep_the_list_of_the_last_build(prec):
    # the rebuild kernels launched at every step build only when a replica asked:
    # the list held at the end is the last build's, whose pairs at the list radius
    # are no longer where they were
    lists = []
    for chunk in (None, 0):
        s = _melt(200, 100, prec, chunk)
        s.integrate(57, 0.005, 1.0, 1.0)
        lists.append((s.n_rebuilds, s.step) + tuple(s.get_neighbors()))
        s.close()
    a, b = lists
    assert a[:2] == b[:2]
    assert np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_broken_bond_stops_the_run(prec):
    # a bond pulled past R0 by its beads' velocities, some steps into the run
    s = _melt(20, 50, prec)
    x, v, img = s.get_state()
    v[0], v[1] = (-30.0, 0.0, 0.0), (30.0, 0.0, 0.0)
    s.set_state(x, v, img)
    with pytest.raises(espp.EsppError) as e:
        s.integrate(200, 0.005, 0.0, 0.0)
    assert e.value.code in (espp.ESPP_ERR_BOND_BROKEN, espp.ESPP_ERR_NONFINITE)
    assert s.step < 200
    # a new state clears the error, and the handle runs again
    s.set_state(x, np.zeros_like(v), img)
    s.integrate(5, 0.001, 1.0, 0.1)
    s.close()


def test_handles_on_streams_and_threads_run_together():
    # resident kernels of several handles, each on its own stream and host
    # thread: the same bits as one after the other
    import threading
    import torch
    sizes = [(FP32, 20, 50), (FP32, 40, 100), (FP64, 20, 50), (FP32, 200, 128), (FP64, 100, 64), (FP32, 300, 128)]

    def go(k, stream, out):
        prec, chains, beads = sizes[k]
        c = I.kg_lattice(chains, beads, density=0.85, seed=k)
        s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=k, stream=stream)
        s.set_wca()
        s.set_fene()
        s.set_state(c.x, I.maxwell_velocities(c.n, 1.0, seed=k), c.img)
        s.build_neighbors(WCA_RC, 0.4)
        for n in (120, 1, 79):
            s.integrate(n, 0.005, 1.0, 1.0)
        out[k] = s.get_state()
        s.close()

    alone, together = {}, {}
    for k in range(len(sizes)):
        go(k, 0, alone)
    streams = [torch.cuda.Stream() for _ in sizes]
    threads = [threading.Thread(target=go, args=(k, streams[k].cuda_stream, together)) for k in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k in range(len(sizes)):
        for p, q in zip(alone[k], together[k]):
            assert np.array_equal(p, q), k


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("barrier,shear", [(1, False), (2, False), (4, False), (1, True), (5, True), (-1, False),
                                           (-4, False)])
def test_grid_barrier_timeout_is_reported_and_cleared(prec, barrier, shear, monkeypatch, tmp_path):
    # host-side fault injection: one grid barrier's bounded wait of the binning
    # (barrier > 0) or run kernel (< 0) runs out.  The call reports it, and a new
    # state (or a loaded checkpoint) leaves nothing of it behind: the lists and
    # trajectories are those of a handle that never failed
    c = I.kg_lattice(40, 100, density=0.85, seed=4)
    v = I.maxwell_velocities(c.n, 1.0, seed=4)

    def handle():
        s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=4)
        s.set_wca()
        s.set_fene()
        if shear:
            s.set_lees_edwards(True, 0.1, 0.5)
        s.set_state(c.x, v, c.img)
        return s

    good = handle()
    good.build_neighbors(WCA_RC, 0.4)
    path = str(tmp_path / "start")
    good.checkpoint_save(path)
    lists = good.get_neighbors()
    good.integrate(40, 0.005, 1.0, 1.0)
    for how in ("state", "checkpoint"):
        monkeypatch.setenv("ESPP_FAULT_GRID_TIMEOUT", str(barrier))
        s = handle()
        monkeypatch.delenv("ESPP_FAULT_GRID_TIMEOUT")
        with pytest.raises(espp.EsppError) as e:
            s.build_neighbors(WCA_RC, 0.4)
            s.integrate(40, 0.005, 1.0, 1.0)
        assert e.value.code == espp.ESPP_ERR_TIMEOUT
        with pytest.raises(espp.EsppError) as e:
            s.compute_forces()
        assert e.value.code == espp.ESPP_ERR_TIMEOUT
        if how == "state":
            s.set_step(0)
            if shear:
                s.set_lees_edwards(True, 0.1, 0.5)
            s.set_state(c.x, v, c.img)
            s.build_neighbors(WCA_RC, 0.4)
        else:
            s.checkpoint_load(path)
        for a, b in zip(lists, s.get_neighbors()):
            assert np.array_equal(a, b)
        s.integrate(40, 0.005, 1.0, 1.0)
        assert s.error_word == 0 and s.step == 40
        for a, b in zip(good.get_state(), s.get_state()):
            assert np.array_equal(a, b)
        s.close()
    good.close()


def test_new_state_after_an_error_under_shear():
    # a run frozen by a broken bond had the positions of the step after; a new
    # state's belong to the step itself, Lees-Edwards offset included
    c = I.kg_lattice(40, 100, density=0.85, seed=4)
    v = I.maxwell_velocities(c.n, 1.0, seed=4)
    fast = v.copy()
    fast[0], fast[1] = (-60.0, 0.0, 0.0), (60.0, 0.0, 0.0)
    out = []
    for fails in (False, True):
        s = espp.System(c.box, c.n, c.types, c.bonds, precision=FP64, seed=4)
        s.set_wca()
        s.set_fene()
        s.set_lees_edwards(True, 0.4, 0.5)
        s.set_state(c.x, fast if fails else v, c.img)
        s.build_neighbors(WCA_RC, 0.4)
        if fails:
            with pytest.raises(espp.EsppError):
                s.integrate(100, 0.005, 0.0, 0.0)
        else:
            s.integrate(1, 0.005, 0.0, 0.0)
        s.set_step(0)
        s.set_lees_edwards(True, 0.4, 0.5)
        s.set_state(c.x, v, c.img)
        obs = s.observables()
        del obs["n_rebuilds"]  # (of the handle's life)
        out.append((s.get_neighbors(), obs, s.compute_forces()))
        s.close()
    (la, oa, fa), (lb, ob, fb) = out
    assert np.array_equal(la[0], lb[0]) and np.array_equal(la[1], lb[1])
    assert oa == ob and np.array_equal(fa, fb)


class _Green:
    """A green context of `sms` SMs (eight or the device's smallest part) with a
    stream."""

    class Res(ctypes.Structure):
        _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sm_count", ctypes.c_uint),
                    ("rest", ctypes.c_ubyte * 44)]

    def __init__(self):
        import torch
        torch.zeros(1, device="cuda")  # the device's primary context, current
        self.cu = ctypes.CDLL("libcuda.so.1")
        whole, part, rest = self.Res(), self.Res(), self.Res()
        groups = ctypes.c_uint(1)
        desc = ctypes.c_void_p()
        self.green, self.ctx, self.stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        self.call("cuDeviceGetDevResource", 0, ctypes.byref(whole), 1)
        self.call("cuDevSmResourceSplitByCount", ctypes.byref(part), ctypes.byref(groups), ctypes.byref(whole),
                  ctypes.byref(rest), 0, 8)
        self.call("cuDevResourceGenerateDesc", ctypes.byref(desc), ctypes.byref(part), 1)
        self.call("cuGreenCtxCreate", ctypes.byref(self.green), desc, 0, 1)
        self.call("cuCtxFromGreenCtx", ctypes.byref(self.ctx), self.green)
        self.call("cuGreenCtxStreamCreate", ctypes.byref(self.stream), self.green, 1, 0)
        self.sms = part.sm_count

    def call(self, name, *args):
        if not hasattr(self.cu, name):
            pytest.skip("no green contexts: " + name)
        rc = getattr(self.cu, name)(*args)
        assert rc == 0, (name, rc)

    def close(self):
        self.call("cuStreamDestroy_v2", self.stream)
        self.call("cuGreenCtxDestroy", self.green)


@pytest.mark.parametrize("how", ["stream", "current"])
@pytest.mark.parametrize("prec,chains,beads", [(FP32, 3, 43), (FP32, 40, 100), (FP32, 304, 128), (FP64, 3, 43),
                                               (FP64, 40, 100), (FP64, 300, 200)])
def test_a_part_of_the_sms(prec, chains, beads, how):
    # the blocks of a cooperative launch fit at once on the SMs of its stream and of
    # the context its graph was captured under, or the step graphs run
    g = _Green()
    assert g.sms < 64
    c = I.kg_lattice(chains, beads, density=0.85, seed=4)

    def go(stream):
        s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=4, stream=stream)
        s.set_wca()
        s.set_fene()
        s.set_resort_interval(20)
        s.set_state(c.x, I.maxwell_velocities(c.n, 1.0, seed=4), c.img)
        s.build_neighbors(WCA_RC, 0.4)
        for n in (33, 1, 20):
            s.integrate(n, 0.005, 1.0, 1.0)
        assert s.error_word == 0
        out = s.get_state()
        s.close()
        return out

    ref = go(0)
    if how == "stream":
        got = go(g.stream.value)
    else:
        g.call("cuCtxPushCurrent_v2", g.ctx)
        try:
            got = go(0)
        finally:
            g.call("cuCtxPopCurrent_v2", ctypes.byref(ctypes.c_void_p()))
    g.close()
    for p, q in zip(ref, got):
        assert np.array_equal(p, q)


def _integrate(case, prec, shape=0, chunk=64, timing=False, calls=(150,)):
    """State after the calls, rebuilds, and kernel launches counted in them."""
    s = case.system(prec, seed=8)
    s.set_step_shape(shape)
    s.set_graph_chunk(chunk)
    s.set_kernel_timing(timing)
    before = s.kernel_launches
    for n in calls:
        s.integrate(n, 0.005, 1.0, 1.0)
    out = s.get_state(), s.n_rebuilds, s.kernel_launches - before
    s.close()
    return out


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_step_graphs_equal_direct_launches(prec):
    # graphs of the step kernel behind conditional rebuild nodes, of several step
    # counts, on handles whose other runs stay in one kernel: a launch a step at least
    case = kg_case()
    ref, rebuilds, _ = _integrate(case, prec, chunk=0)
    assert rebuilds > 4
    forms = [dict(timing=True)] + [dict(shape=1)] * (prec == FP32)
    for form in forms:
        for chunk, calls in ((5, (150,)), (64, (1, 2, 20, 3, 124)), (7, (33, 117))):
            got, rb, launches = _integrate(case, prec, chunk=chunk, calls=calls, **form)
            assert launches >= 150 and rb == rebuilds, (form, chunk)
            for a, b in zip(ref, got):
                assert np.array_equal(a, b), (form, chunk)


@pytest.mark.parametrize("shape", range(espp.STEP_SHAPES))
def test_a_chosen_step_shape_is_the_step_kernels(shape):
    # shape 0 leaves a small handle to the resident kernel, the others launch the
    # step kernel in that shape: blocks of several tiles, the last one partial
    case = kg_case(23, 56, seed=12, jitter=0.06)
    ref, rebuilds, _ = _integrate(case, FP32, chunk=0)
    got, rb, launches = _integrate(case, FP32, shape=shape)
    assert rb == rebuilds and (launches >= 150) == (shape != 0)
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
    # (FP64 handles have one shape)
    assert _integrate(case, FP64, shape=shape)[2] < 150


@pytest.mark.parametrize("prec,tol", [(FP32, 2e-4), (FP64, 1e-11)])
def test_list_overflow_inside_a_resident_run(prec, tol, monkeypatch):
    # a dilute gas drawn together: its lists outgrow their capacity some rebuilds
    # into one call, which grows them and goes on from the step it had reached.
    # (The order of storage and of the sums is another afterwards: rounding only,
    # over 100 steps without many collisions; coordinates of 40 sigma)
    g = np.random.default_rng(3)
    k = np.arange(512)
    x = I.f32(20.0 + 2.2 * (np.stack([k % 8, k // 8 % 8, k // 64], 1) - 3.5) + g.uniform(-0.2, 0.2, (512, 3)))
    v = -0.9 * (x - 20.0)
    out = []
    for cap in (256, 8):
        monkeypatch.setenv("ESPP_FAULT_LIST_CAP", str(cap))
        s = espp.System((40.0, 40.0, 40.0), 512, None, None, precision=prec, seed=4)
        s.set_lj(1.0, 1.0, 1.5)
        s.set_state(x, v, None)
        s.build_neighbors(1.5, 0.4)
        assert s.list_capacity == cap  # (the first lists fit)
        s.integrate(100, 0.005, 0.0, 0.0)
        assert s.error_word == 0 and s.step == 100 and s.n_rebuilds > 5
        assert (s.list_capacity > cap) == (cap == 8)
        out.append(s.get_state())
        s.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= tol
