"""Host logic of the surrogate's training, on the CPU against a stand-in for the
CUDA runtime (fake_runtime.py)."""
from fake_runtime import run

NET = """
def net(max_batch=8):
    return B.Surrogate(max_batch=max_batch, in_dim=4, h1=32, h2=32, l0=16, chans=(16, 16, 8), out_ch=8)
"""


def test_side_streams_are_joined_after_a_failure():
    """Whichever launch of a gradient fails: every stream that was given work is
    waited for by the handle's stream behind its last launch."""
    r = run(NET + """
X, Y = np.zeros((8, 4), np.float32), np.zeros((8, 8, 64), np.float32)
calls = []
with net() as s:
    fake.fake_log_clear()
    s.loss_grad(X, Y)
    n = sum(x.startswith("launch") for x in fake.fake_log().decode().splitlines())
    for k in range(n + 1):
        fake.fake_log_clear()
        fake.fake_fail_launch(k)
        try:
            s.loss_grad(X, Y)
            failed = False
        except B.SimError:
            failed = True
        calls.append([failed, fake.fake_log().decode().splitlines()])
        fake.fake_fail_launch(-1)
out["calls"] = calls
""")
    calls = [(failed, [x.split() for x in log]) for failed, log in r["calls"]]
    assert len(calls) > 20 and not calls[-1][0]
    main = next(x[1] for x in calls[-1][1] if x[0] == "launch")
    sides = {x[1] for x in calls[-1][1] if x[0] == "launch"} - {main}
    assert len(sides) == 3
    left = 0
    for failed, log in calls:
        assert failed or log is calls[-1][1]
        for s in sides:
            given = [q for q, x in enumerate(log) if x[0] == "launch" and x[1] == s]
            if not given:
                continue
            left += failed
            done = [(q, x[2]) for q, x in enumerate(log) if x[0] == "record" and x[1] == s and q > given[-1]]
            assert done, log
            assert any(x[0] == "wait" and x[1] == main and x[2] == done[0][1] for x in log[done[0][0]:]), log
    assert left > 20  # failures with work on a side stream


def test_training_memory_does_not_grow_with_the_number_of_minibatches():
    """Beside the data and the order of the cases, an epoch takes a few MB however
    many minibatches it has."""
    r = run(NET + """
n = 40000
X, Y = np.zeros((n, 4), np.float32), np.zeros((n, 8, 64), np.float32)
with net() as s:
    before = fake.fake_used()
    fake.fake_peak(1)
    s.train(X, Y, epochs=0, batch=1)
    out["extra"] = fake.fake_peak(0) - before - X.nbytes - Y.nbytes - 4 * n
    out["left"] = fake.fake_used() - before
""")
    assert r["extra"] <= 8 << 20 and r["left"] == 0, r
