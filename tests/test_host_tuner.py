"""The kernel choice of AUTO and the memory it keeps, on the CPU against a
stand-in for the CUDA runtime (fake_runtime.py): kernels cost what the test says."""
import pytest

from fake_runtime import run

WELLS = """
for k, us in ((b"fused", 100.0), (b"march", 100.0), (b"sweep", 100.0), (b"hoist", 10.0), (b"split", 10.0),
              (b"hoist_edge", 0.1), (b"hoist_rim", 0.1)):
    fake.fake_cost(k, us)

def well(nr=24, nth=8, nz=80, pml_r=4, pml_z=4, n_mat=4, kind=0, receivers=1):
    g = W.Grid(nr=nr, nth=nth, nz=nz, pml_r=pml_r, pml_z=pml_z, dr=0.004, dz=0.003)
    mats = [(W.FLUID, W.ROCK)[min(q, 1)] for q in range(n_mat)]
    cid = np.ones(g.shape, np.uint16)
    cid[:, 0, :] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in mats]) for q in range(3)))
    rec = W.on_axis_receivers([0.0] * receivers)
    return W.Scenario("t", med, W.Source(z=0.03, f0=60e3, kind=kind), rec, steps=4)

def step(sc, **kw):
    with B.Simulation(sc, **kw) as s:
        try:
            s.step(4)
            ok = ""
        except B.SimError as e:
            ok = str(e)
        return [s.config()[0], ok]
"""


@pytest.mark.parametrize("other", [
    "n_mat=2197",              # a table that leaves no room beside the staged planes
    "nz=20, pml_z=34",         # the same stored cells, 16 of a row lean
    "nr=4, pml_r=24",          # the same rows, three lean
])
def test_a_cached_one_pass_choice_goes_to_wells_that_can_run_it_only(other):
    """The tuner's cache hands a well the choice of an earlier one only where all
    that decides whether the choice runs is the same, in either order."""
    r = run(WELLS + f"""
fake.fake_cost(b"pass_step", 0.01)
out["first"] = step(well())
out["other"] = step(well({other}))
out["again"] = step(well())
out["forced"] = step(well(), tile=4001)
""")
    assert r["first"] == [6, ""] and r["again"] == [6, ""] and r["forced"] == [6, ""], r
    assert r["other"][1] == "" and r["other"][0] != 6, r
    r = run(WELLS + f"""
fake.fake_cost(b"pass_step", 0.01)
out["other"] = step(well({other}))
out["first"] = step(well())
""")
    assert r["first"] == [6, ""] and r["other"][1] == "" and r["other"][0] != 6, r


@pytest.mark.parametrize("kind", [1, 2, 3])
def test_the_second_field_set_is_held_by_the_one_pass_step_only(kind):
    """A point force or the torsion ring under AUTO: the second set is there while
    the one-pass step runs, and neither with a split code asked for or picked nor
    where the step cannot run."""
    r = run(WELLS + f"""
def size(sc, **kw):
    with B.Simulation(sc, **kw) as s:
        return [s.config()[0], s.device_bytes, fake.fake_used()]
sc = lambda **kw: well(kind={kind}, **kw)
if {kind} == 3:  # the ring lies in the rock
    def sc(**kw):
        x = well(kind=3, **kw)
        x.source.r = 0.02
        return x
base = fake.fake_used()
out["one set"] = size(sc(), kernel="split")
out["tile"] = size(sc(), tile=2224)
out["no room"] = size(sc(n_mat=2197))
out["no room, split"] = size(sc(n_mat=2197), kernel="split")
fake.fake_cost(b"pass_step", 0.01)
out["picked"] = size(sc())
fake.fake_cost(b"pass_step", 1000.0)
out["not picked"] = size(sc(nz=81))
out["not picked, split"] = size(sc(nz=81), kernel="split")
fake.fake_cost(b"pass_step", 0.01)
fake.fake_total(base + 3 * out["one set"][1])
out["little memory"] = size(sc(nz=82))
out["left"] = fake.fake_used() - base
""")
    assert r["tile"] == r["one set"]
    assert r["no room"] == r["no room, split"]
    assert r["picked"][0] == 6 and r["picked"][1] > 1.3 * r["one set"][1]
    assert r["not picked"] == r["not picked, split"]
    assert r["little memory"][0] == 1 and r["left"] == 0


def test_a_memory_cap_that_held_one_set_still_does():
    """A cap just above what one set of fields, the layers and the traces take:
    the well is created without the second set."""
    r = run(WELLS + """
sc = well(kind=1, receivers=8)
with B.Simulation(sc, kernel="split", max_steps=65536) as s:
    out["bytes"] = s.device_bytes
fake.fake_cost(b"pass_step", 0.01)
with B.Simulation(sc, max_steps=65536, mem_cap=out["bytes"]) as s:
    out["capped"] = [s.config()[0], s.device_bytes]
    s.step(4)
with B.Simulation(sc, max_steps=65536) as s:
    out["free"] = s.config()[0]
    set_bytes = s.device_bytes - out["bytes"]
with B.Simulation(sc, max_steps=65536, mem_cap=out["bytes"] + set_bytes) as s:
    out["room"] = s.config()[0]
with B.Simulation(sc, max_steps=65536, mem_cap=out["bytes"] + set_bytes - 256) as s:
    out["short"] = [s.config()[0], s.device_bytes]
""")
    assert r["capped"] == [1, r["bytes"]] and r["short"] == [1, r["bytes"]]
    assert r["free"] == 6 and r["room"] == 6


@pytest.mark.parametrize("kernel,kind,us,storage", [
    ("sweep", 5, 30.0, "f32"), ("sweep", 5, 90.0, "f16sr"), ("fused", 2, 30.0, "f16")])
def test_families_are_compared_as_they_run(kernel, kind, us, storage):
    """A kernel of fewer launches that leads where each launch costs something by
    itself is picked only if it also leads in a captured graph."""
    r = run(WELLS + f"""
def pick(sc):
    with B.Simulation(sc, storage={storage!r}) as s:
        s.step(4)
        return s.config()[0]
fake.fake_launch_cost(40.0)  # split halves: one launch of 10 us each, with stochastic rounding three
fake.fake_cost(b"pass_step", 1000.0)
fake.fake_cost({kernel!r}.encode(), {us})
out["slower in a graph"] = pick(well())
fake.fake_cost({kernel!r}.encode(), 2.0)
out["faster in a graph"] = pick(well(nz=84))
""")
    assert r == {"slower in a graph": 1, "faster in a graph": kind}
