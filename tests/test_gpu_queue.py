"""The step kernel's pair queue (FP64 handles and the DPD thermostat): forces and
trajectories at the counts where a warp's queue can go wrong (a single
particle, partial warps, lists longer than one block of the queue, more results
than are held at a time) against the oracle, and the same bits whichever way
particles are spread over lanes.  FP64 forces to 1e-12 relative RMS; DPD in
FP32 one step to 1e-5, the tolerances of the other parity tests."""
import numpy as np
import pytest

import oracle as O
from paper_2608_14911_gb300 import espp, inputs as I

from _systems import rel_rms

pytestmark = pytest.mark.gpu
FP32, FP64 = espp.ESPP_FP32, espp.ESPP_FP64
CAP = ("lj_capped", 1.0, 1.0, 1.1, True, 0.8)


def _gas(n, density, seed, types=1):
    L = max(4.6, (n / density) ** (1 / 3))
    c = I.random_positions(n, (L, L, L), seed=seed)
    if types == 2:
        c.types = (np.random.default_rng(seed).random(n) < 0.5).astype(np.int32)
    c.v = I.maxwell_velocities(n, 1.0, seed=seed) if n > 1 else np.zeros((1, 3))
    return c


def _handle(cs, prec, types=1):
    reps = [dict(box=c.box, n=c.n, types=c.types, bonds=c.bonds, seed=9) for c in cs]
    s = espp.System(precision=prec, replicas=reps)
    for a in range(types):
        for b in range(a, types):
            s.set_lj_capped(1.0, 1.0, 1.1, 0.8, ta=a, tb=b)
    s.set_state(np.concatenate([c.x for c in cs]), np.concatenate([c.v for c in cs]),
                np.concatenate([c.img for c in cs]))
    s.build_neighbors(1.1, 0.4)
    return s


@pytest.mark.parametrize("types", [1, 2])
@pytest.mark.parametrize("n,density", [(1, 0.8), (31, 0.3), (33, 0.3), (129, 0.8), (700, 6.0), (1500, 12.0)])
def test_fp64_forces(n, density, types):
    c = _gas(n, density, 5, types)
    types = int(c.types.max()) + 1
    s = _handle([c], FP64, types)
    f = s.compute_forces()
    s.close()
    m = O.Model(types, {(a, b): CAP for a in range(types) for b in range(a, types)}, None)
    fo, _ = O.forces(m, c.box, c.x, c.types, c.bonds)
    if n == 1:
        assert np.array_equal(f, np.zeros((1, 3)))
    else:
        assert rel_rms(f, fo) <= 1e-12


@pytest.mark.parametrize("n,density", [(33, 0.3), (700, 6.0), (1500, 12.0)])
def test_dpd_fp32_step(n, density):
    c = _gas(n, density, 6)
    s = _handle([c], FP32)
    s.set_thermostat(espp.ESPP_THERMO_DPD, 1.1)
    s.integrate(1, 0.002, 4.5, 1.0)
    _, v, _ = s.get_state()
    s.close()
    O.set_dpd(True, 1.1)
    try:
        st = O.State(c.box, c.x, c.v, c.img, c.types, c.bonds)
        O.integrate(O.Model(1, {(0, 0): CAP}, None), st, 1, 0.002, 4.5, 1.0, seed=9)
    finally:
        O.set_dpd(False)
    assert rel_rms(v, st.v) <= 1e-5


@pytest.mark.parametrize("prec,dpd,n", [(FP64, False, 7000), (FP64, True, 7000), (FP32, True, 30000)])
def test_spread_does_not_change_the_bits(prec, dpd, n):
    # each replica alone takes four lanes per particle, both together one
    cs = [_gas(n, 0.7, seed) for seed in (3, 4)]
    out = []
    for group in ([cs[0]], [cs[1]], cs):
        s = _handle(group, prec)
        if dpd:
            s.set_thermostat(espp.ESPP_THERMO_DPD, 1.1)
        s.integrate(12, 0.002, 1.0, 1.0)
        out.append(s.get_state())
        s.close()
    for a, b, both in zip(*out):
        assert np.array_equal(np.concatenate([a, b]), both)


@pytest.mark.parametrize("prec,tol", [(FP32, 1e-5), (FP64, 1e-12)])
@pytest.mark.parametrize("n,density", [(33, 0.3), (129, 0.8), (700, 6.0), (1500, 12.0)])
def test_cell_forces(n, density, prec, tol):
    # the list-free force kernel: partial warps, columns that fill inside a row
    c = _gas(n, density, 8)
    s = _handle([c], prec)
    s.set_force_method(espp.ESPP_FORCES_CELLS)
    f = s.compute_forces()
    o = s.observables()
    s.close()
    m = O.Model(1, {(0, 0): CAP}, None)
    fo, _ = O.forces(m, c.box, c.x, c.types, c.bonds)
    assert rel_rms(f, fo) <= tol
    oo = O.observables(m, O.State(c.box, c.x, c.v, c.img, c.types, c.bonds))
    for k in ("pe_pair", "virial"):
        assert abs(o[k] - oo[k]) <= tol * abs(oo[k]), k


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_cell_forces_spread_does_not_change_the_bits(prec):
    # each replica alone takes eight lanes per particle, both together one
    cs = [_gas(22000, 0.7, seed) for seed in (3, 4)]
    out = []
    for group in ([cs[0]], [cs[1]], cs):
        s = _handle(group, prec)
        s.set_thermostat(espp.ESPP_THERMO_DPD, 1.1)
        s.set_force_method(espp.ESPP_FORCES_CELLS)
        s.integrate(6, 0.002, 1.0, 1.0)
        out.append(s.get_state())
        s.close()
    for a, b, both in zip(*out):
        assert np.array_equal(np.concatenate([a, b]), both)


@pytest.mark.parametrize("le", [False, True])
@pytest.mark.parametrize("types,pair", [(1, "lj"), (1, "capped"), (2, "lj")])
def test_dpd_walk_does_not_change_the_bits(types, pair, le):
    # long lists with few entries inside the thermostat's cutoff: each replica alone
    # takes the queue (four lanes per particle), both together walk their lists
    m = 19
    c0 = I.lj_fcc(m, m, m, density=0.8442)
    cs = []
    for seed in (3, 4):
        g = np.random.default_rng(seed)
        x = I.f32(np.mod(c0.x + g.uniform(-0.06, 0.06, c0.x.shape), c0.box))
        x[x >= c0.box] = 0.0
        cs.append((x, I.maxwell_velocities(c0.n, 0.72, seed=seed)))
    t = (np.arange(c0.n) % types).astype(np.int32)
    out = []
    for group in ([cs[0]], [cs[1]], cs):
        s = espp.System(precision=FP32, replicas=[dict(box=c0.box, n=c0.n, types=t, bonds=None, seed=9) for _ in group])
        for a in range(types):
            for b in range(a, types):
                if pair == "lj":
                    s.set_lj(1.0, 1.0, 2.5, True, a, b)
                else:
                    s.set_lj_capped(1.0, 1.0, 2.5, 0.9, True, a, b)
        if le:
            s.set_lees_edwards(True, 0.1, 0.4)
        s.set_thermostat(espp.ESPP_THERMO_DPD, 1.1)
        s.set_state(np.concatenate([x for x, _ in group]), np.concatenate([v for _, v in group]), None)
        s.build_neighbors(2.5, 0.3)
        s.integrate(12, 0.004, 4.5, 0.72)
        out.append(s.get_state())
        s.close()
    for a, b, both in zip(*out):
        assert np.array_equal(np.concatenate([a, b]), both)
