"""Captured chunks of steps against steps enqueued one by one: the step number
of a captured step is an offset from the device counter, and its receivers run
beside the next step's first half.  Both orders compute the same bits."""
import numpy as np
import pytest

from paper_2302_13907_gb300 import workloads as W

pytestmark = pytest.mark.gpu
STEPS = 8 * 5 + 3


def scenario(kind, nth=8, nz=146):
    g = W.Grid(nr=20, nth=nth, nz=nz, pml_r=4, pml_z=4, dr=0.004, dz=0.004)
    med = W.cased_well(g, z_top=0.3, ramp=0.05, top_frac=0.5, casing_in=0.03, casing_t=0.008, cement_out=0.06)
    rec = W.Receivers(r=np.array([0.0, 0.01, 0.03]), theta=np.array([0.0, 0.4, 1.3]), z=np.array([0.3, 0.3, 0.36]))
    src = W.Source(kind=kind, r=0.034 if kind == 3 else 0.013,  # a ring of torsion in the steel
                   theta=0.4, z=0.3, f0=60e3)
    return W.Scenario("chunks", med, src, rec, steps=STEPS)


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("kw", [
    dict(kernel="split", tile=2004), dict(kernel="split", tile=2224), dict(kernel="split", tile=22852334), dict(tile=4002),
    dict(kernel="march", tile=1416), dict(kernel="fused"), dict(storage="f16sr", kernel="split", tile=2334, watchdog_every=3),
    dict(tile=4102, watchdog_every=8)])
def test_single_well(kind, kw):
    from paper_2302_13907_gb300.binding import Simulation
    if kind and (kw.get("kernel") == "fused" or kw.get("storage") == "f16sr"):
        pytest.skip("monopole only")
    sc = scenario(kind)
    with Simulation(sc, graph_chunk=8, **kw) as a, Simulation(sc, graph_chunk=-1, **kw) as b:
        a.step(3)
        a.step(40)
        for _ in range(STEPS):
            b.step(1)
        assert np.abs(a.field("vp")).max() > 0 and (kind == 3 or np.abs(a.traces()).max() > 0)  # torsion: no pressure
        assert np.array_equal(a.traces(), b.traces())
        for n in ("srr", "vz", "vp"):
            assert np.array_equal(a.field(n), b.field(n)), n
        if "watchdog_every" in kw:
            (ea, ra, na), (eb, rb, nb) = a.watchdog(), b.watchdog()
            assert na == nb > 0
            # FP64 atomic sums of at most a few thousand blocks, in any order
            assert abs(ea - eb) <= 1e-12 * eb and abs(ra - rb) <= 1e-12 * rb


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
def test_refined_well(kind):
    from paper_2302_13907_gb300.binding import RefinedSimulation
    sc = scenario(kind, nth=16)
    with RefinedSimulation(sc, [4, 8], graph_chunk=8) as a, RefinedSimulation(sc, [4, 8], graph_chunk=-1) as b:
        a.step(3)
        a.step(40)
        for _ in range(STEPS):
            b.step(1)
        assert kind == 3 or np.abs(a.traces()).max() > 0
        assert np.array_equal(a.traces(), b.traces())
        assert all(np.array_equal(a.field("vp", z), b.field("vp", z)) for z in range(3))


@pytest.mark.parametrize("tile", [0, 1])
def test_batch(tile):
    from paper_2302_13907_gb300.binding import BatchSimulation
    cases = [scenario(0, nz=nz) for nz in (146, 160, 211)]
    with BatchSimulation(cases, graph_chunk=8, tile=tile) as a, BatchSimulation(cases, graph_chunk=-1, tile=tile) as b:
        a.run(3)
        a.run(40)
        for _ in range(STEPS):
            b.run(1)
        for c in range(3):
            assert np.abs(a.traces(c)).max() > 0
            assert np.array_equal(a.traces(c), b.traces(c)), c
