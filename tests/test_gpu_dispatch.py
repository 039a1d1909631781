"""Which launches a lattice or a batch takes (mdf_plan, mdf_batch_get_path), and
their bits against single updates where the kernel under test is known to run."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,path,updates", [
    ((2, 4), "resident", 64), ((64, 64), "resident", 64), ((129, 130), "resident", 64), ((1200, 16), "resident", 64),
    ((1201, 16), "fused", 2), ((300, 131), "fused", 2), ((2000, 2), "fused", 2), ((400001, 2), "fused", 2),
    ((250001, 3), "fused", 2), ((190001, 4), "fused", 4), ((1003, 751), "fused", 4),
    ((119, 121, 151), "fused", 2), ((960, 6, 200), "fused", 2), ((64, 64, 64), "single", 1)])
def test_default_path_of_a_run(shape, path, updates):
    from paper_2108_08591_gb300 import Lattice

    for q in (0, 4 if len(shape) == 2 else 6):
        lat = Lattice(shape, s1=1.7, q=q)
        got = lat.plan(64)
        lat.close()
        assert (got["path"], got["updates"]) == (path, updates) and got["launches"] == 64 // updates
        lat = Lattice(shape, s1=1.7, q=q, vx=1)  # a launch shape of the caller's own
        assert lat.plan(64)["path"] == "single" and lat.plan(64)["launches"] == 64
        lat.close()


# fused with and without walls and a force: 59 and 113 columns (60 stored),
# 5 and 1 rows beyond a multiple of 6
@pytest.mark.parametrize("shape", [(59, 65, 211), (59, 85, 199), (113, 89, 88)])
@pytest.mark.parametrize("forcing", ["none", "eq3-21", "scheme2"])
@pytest.mark.parametrize("wall", [(0, 0, 0), (1, 1, 1)])
@pytest.mark.parametrize("q", [0, 6])
def test_fused_3d_updates_equal_single_updates(shape, forcing, wall, q):
    import torch
    from paper_2108_08591_gb300 import Lattice

    N = int(np.prod(shape))
    rng = np.random.default_rng([*shape, q])
    P = 1.0 + 1e-3 * rng.standard_normal(N)
    u, F = 0.01 * rng.standard_normal((3, N)), 1e-5 * rng.standard_normal((3, N))
    outs = []
    for kw, path in (({}, "fused"), ({"vx": 1}, "single")):
        # a stream of its own: 64 updates and more replay a captured chunk
        lat = Lattice(shape, s1=1.8, s2=1.0, wall=wall, lid=bool(wall[2]), lid_u=(0.05, 0.01, 0.0), q=q,
                      stream=torch.cuda.Stream(), **kw)
        if forcing != "none":
            lat.set_forcing(forcing)
            lat.set_force(F)
        assert lat.plan(5)["path"] == path
        lat.init(P, u)
        got = []
        for n in (5, 64 + 3):
            lat.step(n)
            got += lat.fields_host(("P", "u", "rho", "G")).values()
        lat.close()
        outs.append(got)
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("sides,path,updates", [([128], "resident", 0), ([65] * 3 + [97] * 5 + [129] * 4, "resident", 0),
                                                ([300, 240], "fused", 2), ([113] * 6 + [267], "fused", 2),
                                                ([2, 870, 56], "fused", 4)])
def test_batch_path_and_bits(sides, path, updates):
    """The path of a batch; the state after steps and periods of every length is
    the persistent kernel's; a way there and back."""
    from paper_2108_08591_gb300 import CavityBatch

    got = []
    for own in (False, True):
        b = CavityBatch(sides, [50.0] * len(sides), lid_speed=0.1)
        assert b.path == {"path": path, "updates": updates}
        if own:
            b.set_path("persistent")
            assert b.path == {"path": "persistent", "updates": 0}
        b.step(11)
        b.run(tol=1e-12, max_steps=12, check_every=6)
        b.run(tol=1e-12, max_steps=200, check_every=100)
        got.append([b.fields_host(c, ("P", "u", "rho")) for c in range(b.n)])
        b.set_schedule(64, 0, 3)
        b.autotune(reps=4)
        assert b.path["path"] in (path, "persistent")
        b.set_path("default")
        assert b.path["path"] == path
        for c in range(b.n):
            now = b.fields_host(c, ("P", "u", "rho"))
            assert all(np.array_equal(now[k], got[-1][c][k]) for k in now)
        b.close()
    for x, y in zip(*got):
        for k in x:
            assert np.array_equal(x[k], y[k]), k
