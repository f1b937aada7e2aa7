"""The sizes up to which the march along theta runs (32-bit offsets, material table
in shared memory): host arithmetic, on the CPU against a stand-in for the CUDA
runtime (fake_runtime.py)."""
import os
import subprocess

import pytest

from fake_runtime import ROOT, run

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def launcher(tmp_path_factory):
    from paper_2302_13907_gb300 import build
    lib = os.environ.get("CWELL_LIB") or build.build()
    out = str(tmp_path_factory.mktemp("march") / "march_limits.so")
    subprocess.run([build.nvcc(), "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC", *build.ARCH, "-I",
                    os.path.join(ROOT, "include"), os.path.join(HERE, "march_limits.cu"), "-o", out], check=True)
    return lib, out


def test_limits_of_the_march(launcher):
    lib, so = launcher
    r = run(f"""
cwell = ctypes.CDLL({os.path.abspath(lib)!r}, ctypes.RTLD_GLOBAL)
L = ctypes.CDLL({so!r})
def kernels(*a):
    fake.fake_log_clear()
    rc = L.launch_with(*a)
    names = [x.split()[3] for x in fake.fake_log().decode().splitlines() if x.startswith("launch")]
    return [rc, sum("9hoist_run" in x for x in names), len(names)]
# 4096 bytes short of 4 GB: FP32 64 x 1024 x 16384 cells is 4 GB exactly
for nth, name in ((64, "at"), (62, "below")):
    for storage, nr in ((0, 1000), (1, 2000), (2, 2000), (3, 2000)):
        NR = nr + (24 if storage == 0 else 48)
        out[f"{{name}} {{storage}}"] = kernels(storage, 2324, nth, NR, nr, 16384, 16384, 10, 16)
for n in (2048, 2049):
    out[f"materials {{n}}"] = kernels(0, 2324, 8, 40, 36, 512, 512, 4, n)
# the radial layer's memory variables beside 16-bit fields: 4 bytes a cell of it
out["layer at"] = kernels(1, 2275, 64, 1025, 1, 16384, 16384, 10, 16)
out["layer below"] = kernels(1, 2275, 64, 1024, 1, 16384, 16384, 10, 16)
""")
    for s in range(4):  # FP32: interior and radial layer of both halves
        assert r[f"at {s}"][:2] == [0, 0] and r[f"at {s}"][2] == 6, r
        assert r[f"below {s}"] == [0, 4 if s == 0 else 2, 6], r
    assert r["materials 2048"][:2] == [0, 4] and r["materials 2049"][:2] == [0, 0], r
    assert r["layer at"][:2] == [0, 0] and r["layer below"][:2] == [0, 2], r
