"""What a batch reports about its launches, on the CPU against a stand-in for the
CUDA runtime (fake_runtime.py)."""
from fake_runtime import run


def test_blocks_of_the_largest_shared_launch():
    """130 cases of two sizes: three launches a half step, the counts those of the
    launches themselves."""
    r = run("""
def well(nz):
    g = W.Grid(nr=12, nth=4, nz=nz, pml_r=2, pml_z=2, dr=0.004, dz=0.003)
    cid = np.ones(g.shape, np.uint16)
    cid[:, 0] = 0
    med = W.Medium(g, cid, *(np.array([m[q] for m in (W.FLUID, W.ROCK)]) for q in range(3)))
    return W.Scenario("t", med, W.Source(z=0.03, f0=60e3), W.on_axis_receivers([0.0]), steps=4)
with B.BatchSimulation([well(60 if c < 64 else 150) for c in range(130)], graph_chunk=-1, max_steps=4) as b:
    out["config"] = b.config()
    fake.fake_log_clear()
    b.run(1)
    out["grids"] = [int(x.split()[2], 16) for x in fake.fake_log().decode().splitlines() if "hoist_batch" in x]
""")
    grids = r["grids"]
    assert len(grids) == 6 and grids[:3] == grids[3:]
    assert r["config"] == [130, sum(grids[:3]), max(grids)]
