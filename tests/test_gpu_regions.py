"""Split half steps at the edges of their regions: where the lean z cells start
or end inside a tile, on a tile, or in a sliver of one that goes to the z ends,
and where the rows fill no whole tile."""
import numpy as np
import pytest

import oracle
from paper_2302_13907_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [2224, 2256, 2285, 2294, 2334])
@pytest.mark.parametrize("nr,pml_r,nz,pml_z", [
    (6, 1, 117, 2),     # lean cells 4 .. 116: one tile, cut at both ends
    (5, 3, 146, 3),     # lean cells 4 .. 148: the second tile would hold 20, so the z ends take them
    (7, 2, 60, 98),     # lean cells 100 .. 156: the first tile's 28 go to the z ends
    (4, 4, 252, 4),     # rows and z cells fill whole tiles
    (9, 1, 8, 5),       # no lean cell at all
])
def test_fields_at_region_edges(tile, nr, pml_r, nz, pml_z):
    """Every field against the oracle, element by element (2e-5 of its maximum,
    the bar of the split kernels' other element-wise tests)."""
    from paper_2302_13907_gb300.binding import Simulation
    g = W.Grid(nr=nr, nth=4, nz=nz, pml_r=pml_r, pml_z=pml_z, dr=0.004, dz=0.003)
    rng = np.random.default_rng(nz)
    mats = [W.FLUID, W.STEEL, W.CEMENT, W.ROCK]
    cid = rng.integers(0, len(mats), size=g.shape).astype(np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    sc = W.Scenario("edges", med, W.Source(r=0.009, theta=2.0, z=0.012, f0=60e3), W.on_axis_receivers([0.0]), steps=50)
    o = oracle.Oracle(sc)
    with Simulation(sc, kernel="split", tile=tile) as s:
        for n in ("vr", "vp", "vz"):  # waves everywhere (v_r on the axis, v_z past the end are no unknowns)
            v = 1e-7 * rng.standard_normal(g.shape).astype(np.float32)
            if n == "vr":
                v[:, 0] = 0
            if n == "vz":
                v[:, :, -1] = 0
            s.set_field(n, v)
            o.field(n)[...] = v
        s.step(sc.steps)
        o.step(sc.steps)
        for n in oracle.FIELDS:
            b = o.field(n)
            assert np.abs(b).max() > 0, n
            assert np.abs(s.field(n) - b).max() <= 2e-5 * np.abs(b).max(), n


@pytest.mark.parametrize("tile", [2275, 2324])
@pytest.mark.parametrize("storage", ["f32", "bf16", "f16", "f16sr"])
@pytest.mark.parametrize("nth,nr,pml_r,nz,pml_z,pml_on,n_mat", [
    (10, 6, 1, 117, 2, True, 5),        # two runs of five planes, one z tile cut at both ends
    (22, 5, 3, 146, 3, True, 2048),     # runs of five and a last one of two; the largest table in shared memory
    (4, 7, 2, 252, 4, True, 2049),      # one run; a table that stays in L1
    (6, 9, 0, 140, 0, False, 5),        # rigid walls: the last row has no outer neighbour
])
def test_march_along_theta(tile, storage, nth, nr, pml_r, nz, pml_z, pml_on, n_mat):
    """The interior marched along theta against the tile-by-tile kernels, every
    field: the same bits.  (Tile 2324 in FP32 marches the radial layer too, whose
    products and sums may be fused differently: 2e-5 of the maximum.)"""
    from paper_2302_13907_gb300.binding import Simulation
    if storage == "f16sr" and tile < 2300:
        pytest.skip("the stochastic rounding runs on the 23xx codes")
    g = W.Grid(nr=nr, nth=nth, nz=nz, pml_r=pml_r, pml_z=pml_z, dr=0.004, dz=0.003)
    rng = np.random.default_rng(nz)
    base = [W.FLUID, W.STEEL, W.CEMENT, W.ROCK]
    mats = [base[q % 4] for q in range(n_mat)]
    cid = rng.integers(0, n_mat, size=g.shape).astype(np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    steps = 8
    sc = W.Scenario("march", med, W.Source(r=0.009, theta=2.0, z=0.012, f0=60e3), W.on_axis_receivers([0.0]), steps=steps)
    sc.pml_on = pml_on
    scale = 1.0 / (1000.0 * 1500.0) if storage.startswith("f16") else 1e-7
    v0 = {n: (scale * rng.standard_normal(g.shape)).astype(np.float32) for n in ("vr", "vp", "vz")}
    v0["vr"][:, 0] = 0
    v0["vz"][:, :, -1] = 0
    exact = tile != 2324 or storage != "f32" or not pml_on or n_mat > 2048
    with Simulation(sc, kernel="split", tile=tile, storage=storage) as a, \
            Simulation(sc, kernel="split", tile=2335, storage=storage) as b:
        for n in v0:
            a.set_field(n, v0[n])
            b.set_field(n, v0[n])
        a.step(steps)
        b.step(steps)
        for n in oracle.FIELDS:
            x, y = a.field(n), b.field(n)
            assert np.abs(y).max() > 0, n
            assert np.abs(x - y).max() <= (0 if exact else 2e-5) * np.abs(y).max(), n


@pytest.mark.parametrize("tile", [2204, 2216, 2224, 2256, 2275, 2285, 2304, 2314, 2324])
@pytest.mark.parametrize("storage,steps", [("f32", 3), ("bf16", 40), ("f16", 40)])
@pytest.mark.parametrize("nz,pml_z", [
    (146, 3),   # the z ends hold a sliver of lean groups and an odd pair at either side
    (60, 98),   # the same below the lean cells
    (117, 2),   # lean cells up to one pair from the layer
    (252, 4),   # cuts on the layer's first cell
])
def test_no_trace_of_the_cut_in_the_fields(tile, storage, steps, nz, pml_z):
    """Where a split code cuts a row into lean cells and z ends does not show:
    every field has the bits of the kernel that decides per pair of cells (2106).
    (No radial layer: its body has its own order of sums.)"""
    from paper_2302_13907_gb300.binding import Simulation
    g = W.Grid(nr=9, nth=6, nz=nz, pml_r=0, pml_z=pml_z, dr=0.004, dz=0.003)
    rng = np.random.default_rng(nz)
    mats = [W.FLUID, W.STEEL, W.CEMENT, W.ROCK]
    cid = rng.integers(0, len(mats), size=g.shape).astype(np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    sc = W.Scenario("cut", med, W.Source(r=0.009, theta=2.0, z=0.012, f0=60e3), W.on_axis_receivers([0.0]), steps=steps)
    v = {n: rng.standard_normal(g.shape).astype(np.float32) / (1000 * 1500) for n in ("vr", "vp", "vz")}
    v["vr"][:, 0] = 0
    v["vz"][:, :, -1] = 0
    with Simulation(sc, kernel="split", tile=tile, storage=storage) as a, \
            Simulation(sc, kernel="split", tile=2106, storage=storage) as b:
        for n in v:
            a.set_field(n, v[n])
            b.set_field(n, v[n])
        a.step(steps)
        b.step(steps)
        for n in oracle.FIELDS:
            x, y = a.field(n), b.field(n)
            assert np.abs(y).max() > 0, n
            assert np.array_equal(x, y), (n, np.flatnonzero((x != y).any((0, 1))))


def _noisy_well(nr, pml_r, nz, pml_z, steps):
    g = W.Grid(nr=nr, nth=6, nz=nz, pml_r=pml_r, pml_z=pml_z, dr=0.004, dz=0.003)
    rng = np.random.default_rng(nz)
    mats = [W.FLUID, W.STEEL, W.CEMENT, W.ROCK]
    cid = rng.integers(0, len(mats), size=g.shape).astype(np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    sc = W.Scenario("cut", med, W.Source(r=0.009, theta=2.0, z=0.012, f0=60e3), W.on_axis_receivers([0.0]), steps=steps)
    v = {n: rng.standard_normal(g.shape).astype(np.float32) / (1000 * 1500) for n in ("vr", "vp", "vz")}
    v["vr"][:, 0] = 0
    v["vz"][:, :, -1] = 0
    return sc, v


@pytest.mark.parametrize("tile", [2204, 2216, 2224, 2256, 2275, 2285, 2304, 2314, 2324])
@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("nr,pml_r,nz,pml_z", [(9, 5, 146, 3), (10, 3, 300, 9), (8, 4, 252, 4)])
def test_radial_layer_in_16_bit_storage(tile, storage, nr, pml_r, nz, pml_z):
    """The radial layer's own bodies, wherever their region starts and ends, give the
    bits of the general body (2106), every field."""
    from paper_2302_13907_gb300.binding import Simulation
    sc, v = _noisy_well(nr, pml_r, nz, pml_z, 160)
    with Simulation(sc, kernel="split", tile=tile, storage=storage) as a, \
            Simulation(sc, kernel="split", tile=2106, storage=storage) as b:
        for n in v:
            a.set_field(n, v[n])
            b.set_field(n, v[n])
        a.step(sc.steps)
        b.step(sc.steps)
        for n in oracle.FIELDS:
            x, y = a.field(n), b.field(n)
            assert np.abs(y).max() > 0, n
            assert np.array_equal(x, y), (n, np.flatnonzero((x != y).any((0, 2))))


@pytest.mark.parametrize("tile", [2304, 2305, 2314, 2324, 2335])
@pytest.mark.parametrize("nr,pml_r,nz,pml_z,crc", [
    (10, 5, 300, 9, 0x25d6cab3),    # two rows above the layer share its first tile
    (9, 3, 500, 15, 0xe9d95514),
    (11, 4, 250, 3, 0xa9d32746),
])
def test_stochastic_rounding_keeps_its_bits(tile, nr, pml_r, nz, pml_z, crc):
    """FP16 with stochastic rounding, 60 steps: the fields of the kernels that cut
    their regions at whole tiles of 4 rows x 128 z cells (all 23xx codes gave these)."""
    import zlib
    from paper_2302_13907_gb300.binding import Simulation
    sc, v = _noisy_well(nr, pml_r, nz, pml_z, 60)
    with Simulation(sc, kernel="split", tile=tile, storage="f16sr") as s:
        for n in v:
            s.set_field(n, v[n])
        s.step(60)
        got = 0
        for n in oracle.FIELDS:
            got = zlib.crc32(np.ascontiguousarray(s.field(n)).tobytes(), got)
    assert got == crc
