"""The one-pass step (tile codes 40xx and 41xx: both halves in one kernel, two
field sets) against the FP64 oracle, element by element, at the sizes where its
tiling can go wrong, and beside the rest of the handle's calls."""
import os
import tempfile

import numpy as np
import pytest

import oracle
from paper_2302_13907_gb300 import workloads as W
from tests.helpers import rel_l2

pytestmark = pytest.mark.gpu
FIELD_TOL = 2e-5  # of a field's maximum: the bar of the split kernels' element-wise tests
TILES = (4001, 4002, 4102, 4201, 4304)


def sim(sc, **kw):
    from paper_2302_13907_gb300.binding import Simulation
    return Simulation(sc, **kw)


def scenario(seed, nth, nr, nz, pml_r=3, pml_z=3, steps=60):
    """Random heterogeneous medium (liquid ring 0), off-axis source, receivers on and off the axis."""
    g = W.Grid(nr=nr, nth=nth, nz=nz, pml_r=pml_r, pml_z=pml_z, dr=0.004, dz=0.003)
    rng = np.random.default_rng(seed)
    mats = [W.FLUID, W.STEEL, W.CEMENT, W.ROCK, (2000.0, 2500.0, 0.0)]
    cid = rng.integers(0, len(mats), size=g.shape).astype(np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    rec = W.Receivers(r=np.array([0.0, 0.013]), theta=np.array([0.0, 1.1]), z=np.array([0.02, 0.06]))
    return W.Scenario("ragged", med, W.Source(r=0.014, theta=2.0, z=0.06, f0=60e3), rec, steps=steps)


def fields_match(s, o):
    for n in oracle.FIELDS:
        a, b = s.field(n), o.field(n)
        scale = np.abs(b).max()
        assert scale > 0, n
        assert np.abs(a - b).max() <= FIELD_TOL * scale, (n, np.abs(a - b).max() / scale)


def start(sc, *engines):
    """Random velocities everywhere (v_r on the axis and v_z past the end are no unknowns)."""
    rng = np.random.default_rng(5)
    for n in ("vr", "vp", "vz"):
        v = 1e-7 * rng.standard_normal(sc.grid.shape).astype(np.float32)
        if n == "vr":
            v[:, 0] = 0
        if n == "vz":
            v[:, :, -1] = 0
        for e in engines:
            if isinstance(e, oracle.Oracle):
                e.field(n)[...] = v
            else:
                e.set_field(n, v)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("nth,nr,nz,pml_r,pml_z,pml_on", [
    (12, 14, 301, 3, 3, True),    # two row tiles, three z tiles, uneven theta runs
    (8, 21, 126, 2, 5, True),     # rows one past a tile, z region one group past a tile
    (6, 5, 44, 0, 0, False),      # rigid walls: the last row's outer neighbour is the wall
    (4, 31, 250, 1, 1, True),     # one-cell layers
])
def test_fields_elementwise(tile, nth, nr, nz, pml_r, pml_z, pml_on):
    if 2 * (tile % 100) > nth:
        pytest.skip("more runs than half the planes")
    sc = scenario(nth + nz, nth, nr, nz, pml_r, pml_z)
    sc.pml_on = pml_on
    o = oracle.Oracle(sc)
    with sim(sc, tile=tile) as s:
        assert s.config() == (6, tile)
        start(sc, s, o)
        s.step(sc.steps)
        o.step(sc.steps)
        fields_match(s, o)
        assert rel_l2(s.traces(), o.traces()) <= 1e-4


@pytest.mark.parametrize("kind,r,z", [(1, 0.0, 0.06), (1, 0.014, 0.06), (2, 0.0, 0.06), (2, 0.014, 0.06),
                                      (1, 0.0, 0.0), (2, 0.0145, 0.0)])
def test_point_forces(kind, r, z):
    """Forces on and off the axis, inside the pass (z = 0.06) and on a z-end cell beside it (z = 0)."""
    sc = scenario(7, 8, 14, 141)
    sc.source = W.Source(kind=kind, r=r, theta=0.7, z=z, f0=60e3)
    o = oracle.Oracle(sc)
    with sim(sc, tile=4002) as s:
        s.step(sc.steps)
        o.step(sc.steps)
        fields_match(s, o)


def test_torsion_ring():
    sc = W.realistic_well_section(z0=107.5, length=1.0, nth=4, nr=64, pml_r=6, pml_z=6, source_depth=108.0, steps=60)
    o = oracle.Oracle(sc)
    with sim(sc, tile=4001) as s:
        start(sc, s, o)
        s.step(sc.steps)
        o.step(sc.steps)
        fields_match(s, o)


def test_other_calls_between_passes():
    """Odd step counts, half steps (in place, on whichever set holds the
    state), plane copies, a field written between steps and a checkpoint give
    what the split kernels give."""
    sc = scenario(3, 8, 14, 141, steps=90)
    with sim(sc, tile=4002, graph_chunk=8, max_steps=90) as a, sim(sc, kernel="split", tile=2004, max_steps=90) as b, \
            tempfile.TemporaryDirectory() as d:
        for s in (a, b):
            start(sc, s)
            s.step(27)
            s.half_step(0)
            s.half_step(1)
            s.set_field("vz", s.field("vz") * np.float32(0.5))
            s.step(33)
            p = s.get_planes(1, 3, 20, np.zeros((6, sc.grid.nth * sc.grid.NR, 17), np.float32))
            s.sync()
            s.put_planes(1, 3, 20, p)
            s.save(os.path.join(d, "ck"))
            s.step(28)
            end = s.field("srr")
            s.load(os.path.join(d, "ck"))
            s.step(28)
            assert np.array_equal(s.field("srr"), end)
        for n in oracle.FIELDS:
            y = b.field(n)
            assert np.abs(a.field(n) - y).max() <= FIELD_TOL * np.abs(y).max(), n
        assert rel_l2(a.traces(), b.traces()) <= 1e-5


def test_refused_where_it_cannot_run():
    from paper_2302_13907_gb300.binding import SIM_EINVAL, SimError
    sc = scenario(1, 8, 14, 141)
    for kw in (dict(kernel="split", tile=4001), dict(storage="f16", tile=4001), dict(tile=4000), dict(tile=4400)):
        with pytest.raises(SimError) as ei:
            sim(sc, **kw)
        assert ei.value.code == SIM_EINVAL


def test_largest_material_table():
    """2196 materials fill the shared memory beside the staged planes; one more is
    refused for a tile asked for and runs the other kernels under AUTO."""
    from paper_2302_13907_gb300.binding import SIM_EINVAL, SimError
    for n_mat in (2196, 2197):
        sc = scenario(11, 8, 14, 141, steps=40)
        m = sc.medium
        rng = np.random.default_rng(n_mat)
        q = np.arange(n_mat) % 4
        f = 1 + 1e-4 * (np.arange(n_mat) // 4)
        m.rho, m.vp, m.vs = m.rho[q], m.vp[q] * f, m.vs[q] * f
        m.cell_id = rng.integers(0, n_mat, size=m.grid.shape).astype(np.uint16)
        m.cell_id[:, 0] = 0
        if n_mat == 2197:
            with pytest.raises(SimError) as ei:
                sim(sc, tile=4001)
            assert ei.value.code == SIM_EINVAL
        o = oracle.Oracle(sc)
        with sim(sc, tile=4001 if n_mat == 2196 else 0) as s:
            assert (s.config()[0] == 6) == (n_mat == 2196)
            start(sc, s, o)
            s.step(sc.steps)
            o.step(sc.steps)
            fields_match(s, o)
