"""Which kernels the zones of a refined grid run, on the CPU against a stand-in for
the CUDA runtime (fake_runtime.py)."""
import pytest

from fake_runtime import run


def kernels(nr, nth, nz, rows, **kw):
    """(one launch per half, marched interior, marched radial layer) of a step"""
    r = run(f"""
g = W.Grid(nr={nr}, nth={nth}, nz={nz}, pml_r=4, pml_z=4, dr=0.004, dz=0.003)
cid = np.ones(g.shape, np.uint16)
cid[:, 0] = 0
med = W.Medium(g, cid, *(np.array([m[q] for m in (W.FLUID, W.ROCK)]) for q in range(3)))
sc = W.Scenario("t", med, W.Source(z=0.03, f0=60e3), W.on_axis_receivers([0.0]), steps=4)
with B.RefinedSimulation(sc, {rows}, max_steps=4, **{kw!r}) as s:
    fake.fake_log_clear()
    s.step(1)
    out["launches"] = [x.split()[3] for x in fake.fake_log().decode().splitlines() if x.startswith("launch")]
""")["launches"]
    has = lambda *names: any(all(n in x for n in names) for x in r)  # noqa: E731
    # template flags of hoist_run<T, MINB, VEL, RAD, OUT> in the mangled name
    return has("hoist_batch"), has("hoist_run", "Lb1ELb0ELb0E"), has("hoist_run", "Lb1ELb1ELb0E")


@pytest.mark.parametrize("rows", [[], [8]])
def test_a_zone_that_fills_the_gpu_has_its_own_launches(rows):
    """A largest zone of 8 Mi cells and more, whether or not there are others; below
    that the zones share one launch."""
    nz = 4096 + 4  # x 64 x 32 rows
    rows_of = 28 + (rows[0] if rows else 0)
    assert not kernels(rows_of, 64, nz, rows)[0]
    assert kernels(rows_of, 64, nz - 16, rows)[0]


@pytest.mark.parametrize("rows", [[], [8]])
def test_the_radial_layer_is_marched_in_large_zones(rows):
    """The interior of every zone with launches of its own is marched along theta,
    the radial layer from 38 Mi cells on."""
    skip = rows[0] if rows else 0
    assert kernels(28 + skip, 64, 4096 + 4, rows) == (False, True, False)
    assert kernels(147 + skip, 64, 4096 + 4, rows) == (False, True, False)   # x 151 rows
    assert kernels(148 + skip, 64, 4096 + 4, rows) == (False, True, True)    # x 152 rows
