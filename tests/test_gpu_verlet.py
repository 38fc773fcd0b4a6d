"""The Verlet list search at the sizes where it can go wrong: boxes of the
fewest cells (every row wraps), long flat boxes, rows and lists longer than a
lane's buffer, both forms of the search (one thread or a team of lanes per
particle) and particle counts at the tile edges.  The neighbour sets are the
oracle's brute-force ones, FP32 outside a band of 1e-6 sigma at the list radius
(the rounding of coordinates up to a few tens of sigma), FP64 exactly."""
import numpy as np
import pytest

import oracle as O
from paper_2608_14911_gb300 import espp, inputs as I

from _systems import rel_rms

pytestmark = pytest.mark.gpu
FP32, FP64 = espp.ESPP_FP32, espp.ESPP_FP64
RL = 1.5


def _gas(n, box, seed, blob=0):
    """n uniform positions, the first `blob` of them in a ball of radius 0.9."""
    c = I.random_positions(n, box, seed=seed)
    g = np.random.default_rng(seed)
    if blob:
        d = g.normal(size=(blob, 3))
        d *= 0.9 * g.random((blob, 1)) ** (1 / 3) / np.linalg.norm(d, axis=1, keepdims=True)
        c.x[:blob] = I.f32(np.mod(0.25 + d, c.box))
        c.x[c.x >= c.box] = 0.0
    return c


def _handle(c, prec, w):
    s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=3)
    s.set_lj_capped(1.0, 1.0, 1.1, 0.8)
    s.set_cell_subdivision(w)
    s.set_state(c.x, None, c.img)
    s.build_neighbors(1.1, RL - 1.1)
    return s


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("w", [1, 2, 3])
@pytest.mark.parametrize("n,box,blob", [
    (1, (4.6, 4.6, 4.6), 0),
    (129, (4.6, 4.7, 4.8), 0),             # the fewest cells: every row crosses a face
    (1500, (40.0, 4.6, 5.3), 0),           # long rows along x
    (2000, (5.0, 4.6, 60.0), 0),
    (900, (9.0, 8.0, 7.7), 140),           # lists longer than a lane's buffer, around a corner
    (8191, (22.0, 20.0, 21.0), 60),        # the team form's last size (FP32)
    (8192, (22.0, 20.0, 21.0), 60),
])
def test_neighbour_sets(prec, w, n, box, blob):
    c = _gas(n, box, 11 + n, blob)
    s = _handle(c, prec, w)
    row, cols = s.get_neighbors()
    s.close()
    orow, ocols = O.neighbors(c.box, c.x, RL, method="brute")
    band = 1e-6 if prec == FP32 else 0.0
    for i in range(c.n):
        got = cols[row[i]:row[i + 1]].tolist()
        assert len(set(got)) == len(got)
        for j in set(got) ^ set(ocols[orow[i]:orow[i + 1]].tolist()):
            d = c.x[i] - c.x[j]
            d -= c.box * np.round(d / c.box)
            assert abs(np.linalg.norm(d) - RL) <= band, (i, j)


@pytest.mark.parametrize("prec,n", [(FP32, 5000), (FP64, 20000)])
def test_both_forms_build_the_same_lists(prec, n):
    # two replicas together are past the size up to which a team of lanes
    # shares a particle, each alone is below it: the same forces and
    # trajectories (rebuilds included) bit for bit
    cs = [_gas(n, (19.0 * (n / 5000) ** (1 / 3),) * 3, seed) for seed in (5, 6)]
    alone = []
    for c in cs:
        s = _handle(c, prec, 1)
        f = s.compute_forces()
        s.integrate(25, 0.002, 1.0, 1.0)
        alone.append((f, s.get_state()))
        assert s.n_rebuilds >= 2
        s.close()
    b = espp.System(precision=prec, replicas=[dict(box=c.box, n=c.n, types=c.types, bonds=c.bonds, seed=3)
                                              for c in cs])
    b.set_lj_capped(1.0, 1.0, 1.1, 0.8)
    b.set_cell_subdivision(1)
    b.set_state(np.concatenate([c.x for c in cs]), None, np.concatenate([c.img for c in cs]))
    b.build_neighbors(1.1, RL - 1.1)
    fb = b.compute_forces()
    b.integrate(25, 0.002, 1.0, 1.0)
    st = b.get_state()
    b.close()
    for k, (f, q) in enumerate(alone):
        sl = slice(k * n, (k + 1) * n)
        assert np.array_equal(f, fb[sl])
        for a, p in zip(q, st):
            assert np.array_equal(a, p[sl])


@pytest.mark.parametrize("prec,tol,band", [(FP32, 1e-5, 1e-6), (FP64, 1e-12, 0.0)])
@pytest.mark.parametrize("n,box", [
    (1, (30.0, 4.6, 45.0)),           # 1800 cells, one particle
    (100, (9.5, 24.2, 16.6)),         # 1056 cells: just past a block's share
    (1000, (151.0, 64.0, 47.0)),      # 130,000 cells
    (3000, (700.0, 31.0, 5.0)),       # a long flat box
    (1500, (160.0, 151.0, 155.0)),    # 1.1 million cells: past the shares of all resident blocks
])
def test_dilute_boxes(prec, tol, band, n, box):
    # many more cells than particles, whose scan has blocks of its own
    c = _gas(n, box, 7 + n, min(n, 60))
    s = _handle(c, prec, 1)
    row, cols = s.get_neighbors()
    s.set_force_method(espp.ESPP_FORCES_CELLS)
    f = s.compute_forces()
    s.close()
    orow, ocols = O.neighbors(c.box, c.x, RL, method="brute")
    for i in range(c.n):
        for j in set(cols[row[i]:row[i + 1]].tolist()) ^ set(ocols[orow[i]:orow[i + 1]].tolist()):
            d = c.x[i] - c.x[j]
            d -= c.box * np.round(d / c.box)
            assert abs(np.linalg.norm(d) - RL) <= band, (i, j)
    m = O.Model(1, {(0, 0): ("lj_capped", 1.0, 1.0, 1.1, True, 0.8)}, None)
    fo, _ = O.forces(m, c.box, c.x, c.types, c.bonds)
    assert rel_rms(f, fo) <= tol


@pytest.mark.parametrize("prec,n_chains", [(FP32, 40), (FP32, 90), (FP64, 40), (FP64, 330)])
@pytest.mark.parametrize("w", [1, 2, 3])
@pytest.mark.parametrize("variant", ["lees_edwards", "exclusions"])
def test_sheared_and_excluded_lists(prec, n_chains, w, variant):
    # the search's other instances, a team of lanes and one thread per particle,
    # against the oracle.  FP32 under shear: the offset and each of the three
    # differences it enters are rounded at up to 32 sigma, 1e-6 each
    c = I.kg_lattice(n_chains, 100, density=0.85, seed=5, jitter=0.1)
    le = variant == "lees_edwards"
    shear, t = 0.4, 3.3
    s = espp.System(c.box, c.n, c.types, c.bonds, precision=prec, seed=3)
    s.set_wca()
    s.set_fene()
    s.set_cell_subdivision(w)
    if le:
        s.set_lees_edwards(True, shear, t)
    else:
        s.set_exclude_bonded(True)
    s.set_state(c.x, None, c.img)
    s.build_neighbors(1.1225, RL - 1.1225)
    row, cols = s.get_neighbors()
    s.close()
    O.set_lees_edwards(le, shear)
    try:
        orow, ocols = O.neighbors(c.box, c.x, RL, time=t if le else 0.0)
    finally:
        O.set_lees_edwards(False)
    i = np.repeat(np.arange(c.n), np.diff(orow))
    want = i * c.n + ocols
    if not le:
        b = np.asarray(c.bonds)
        want = np.setdiff1d(want, np.concatenate([b[:, 0] * c.n + b[:, 1], b[:, 1] * c.n + b[:, 0]]))
    got = np.repeat(np.arange(c.n), np.diff(row)) * c.n + cols
    assert len(np.unique(got)) == len(got)
    delta = shear * c.box[2] * t if le else 0.0
    for q in np.setxor1d(got, want):
        d = c.x[q // c.n] - c.x[q % c.n]
        k = np.rint(d[2] / c.box[2])
        d[2] -= k * c.box[2]
        d[0] -= k * delta
        d -= c.box * np.rint(d / c.box)
        assert abs(np.linalg.norm(d) - RL) <= (0.0 if prec == FP64 else 1e-5 if le else 1e-6), (q // c.n, q % c.n)
