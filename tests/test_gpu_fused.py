"""Fused updates (several per pass over memory, FP32) and the resident kernel
(small 2D lattices kept on chip) against single updates: the same bits for
every boundary, force scheme, width and number of steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# kept on chip by a cluster: fewer rows than CTAs, odd rows, the largest that fit
RESIDENT = [(2, 4), (3, 5), (24, 7), (57, 2), (64, 64), (129, 130), (300, 41), (1200, 16), (60, 319)]
# beyond that: strip edges (56 and 60 stored columns of 64), odd and even rows,
# rows too short for the deeper kernels, one to several strips
SHAPES = RESIDENT + [(1201, 16), (95, 310), (2000, 2), (1999, 3), (1921, 4), (2019, 9), (55, 560), (56, 550), (57, 545), (60, 512),
                     (61, 511), (113, 301), (128, 257), (300, 131)]
# from 750 000 nodes on: by fours
SHAPES += [(400001, 2), (250001, 3), (190001, 4), (150001, 5), (55, 13637), (56, 13400), (57, 13159), (113, 6638), (1003, 751)]
BCS = [((0, 0), False), ((1, 0), False), ((0, 1), True), ((1, 1), True)]


@pytest.mark.parametrize("q", [0, 4])
@pytest.mark.parametrize("forcing", ["none", "eq3-21", "scheme2"])
@pytest.mark.parametrize("shape", SHAPES)
def test_fused_updates_equal_single_updates(shape, forcing, q):
    import torch
    from paper_2108_08591_gb300 import Lattice

    N = shape[0] * shape[1]
    rng = np.random.default_rng([*shape, q])
    P = 1.0 + 1e-3 * rng.standard_normal(N)
    u, F = 0.01 * rng.standard_normal((2, N)), 1e-5 * rng.standard_normal((2, N))
    for wall, lid in BCS:
        outs = []
        for kw in ({}, {"vx": 1}):  # an own launch shape keeps to single updates
            lat = Lattice(shape, s1=1.8, wall=wall, lid=lid, lid_u=(0.05, 0.01, 0.0), q=q, **kw)
            if forcing != "none":
                lat.set_forcing(forcing)
                lat.set_force(F)
            lat.init(P, u)
            got = []
            for n in (1, 2, 3, 4, 7):  # fused: 1: single; the others by twos, or fours and a two
                lat.step(n)
                got += [v.clone() for v in lat.fields(("P", "u", "rho", "G")).values()]
            lat.close()
            outs.append(got)
        for a, b in zip(*outs):
            assert torch.equal(a, b), (wall, lid)


# boxes large enough for the fused kernel to be chosen (single updates below);
# tile edges (60 of 64 columns, 6 of 8 rows), odd rows, one segment and many
SHAPES3 = [(119, 61, 151), (59, 59, 211), (300, 120, 25), (960, 6, 200), (119, 121, 151)]
BCS3 = [((0, 0, 0), False), ((1, 0, 0), False), ((0, 1, 0), False), ((0, 0, 1), True), ((1, 1, 1), True)]


@pytest.mark.parametrize("q", [0, 6])
@pytest.mark.parametrize("forcing", ["none", "eq3-21", "scheme2"])
@pytest.mark.parametrize("shape", SHAPES3)
def test_fused_3d_updates_equal_single_updates(shape, forcing, q):
    import torch
    from paper_2108_08591_gb300 import Lattice

    N = int(np.prod(shape))
    rng = np.random.default_rng([*shape, q])
    P = 1.0 + 1e-3 * rng.standard_normal(N)
    u, F = 0.01 * rng.standard_normal((3, N)), 1e-5 * rng.standard_normal((3, N))
    for wall, lid in BCS3:
        outs = []
        for kw in ({}, {"vx": 1}):
            lat = Lattice(shape, s1=1.8, s2=1.0, wall=wall, lid=lid, lid_u=(0.05, 0.01, 0.0), q=q, **kw)
            if forcing != "none":
                lat.set_forcing(forcing)
                lat.set_force(F)
            lat.init(P, u)
            got = []
            for n in (2, 3, 1, 6):
                lat.step(n)
                got += [v.clone() for v in lat.fields(("P", "u", "rho", "G")).values()]
            lat.close()
            outs.append(got)
        for a, b in zip(*outs):
            assert torch.equal(a, b), (wall, lid)


def test_resident_updates_without_the_continuity_set():
    import torch
    from paper_2108_08591_gb300 import Lattice

    P, u = np.ones(70 * 33), 0.01 * np.random.default_rng(2).standard_normal((2, 70 * 33))
    outs = []
    for kw in ({}, {"vx": 1}):
        lat = Lattice((70, 33), s1=1.7, with_rho=False, wall=(0, 1), **kw)
        lat.init(P, u)
        lat.step(40000)  # three launches
        lat.step(3)
        outs.append(lat.fields(("P", "u", "G")))
        lat.close()
    for k in outs[0]:
        assert torch.equal(outs[0][k], outs[1][k]), k


@pytest.mark.parametrize("nx", [97, 777, 15777])
def test_fused_updates_in_a_captured_chunk(nx):
    import torch
    from paper_2108_08591_gb300 import Lattice

    P = np.ones(nx * 50)
    u = 0.01 * np.random.default_rng(1).standard_normal((2, nx * 50))
    outs = []
    for kw in ({}, {"vx": 1}):
        s = torch.cuda.Stream()
        lat = Lattice((nx, 50), s1=1.7, stream=s, **kw)
        lat.init(P, u)
        lat.step(64 * 2 + 3)
        lat.step(64 + 1)
        outs.append(lat.fields_host(("P", "u", "G")))
        lat.close()
    for k in outs[0]:
        assert np.array_equal(outs[0][k], outs[1][k]), k


# on chip: one CTA each, teams of several sizes and empty seats, the largest
# team; by fused launches: boxes beyond that, alone and with small ones, by twos
# and (750 000 nodes) by fours
@pytest.mark.parametrize("sides", [[2, 3, 4, 5, 7], [55, 36, 57, 64, 37], [113, 30, 65], [128],
                                   [65] * 3 + [97] * 5 + [129] * 4, [175, 20], [2, 267, 56], [2, 870, 56]])
def test_fused_cavities_equal_the_persistent_kernel(sides):
    """Batched cavities on chip or by fused launches (the default) against the
    persistent kernel: the same bits after steps and after a run, with its
    step counts, statuses and residuals."""
    from paper_2108_08591_gb300 import CavityBatch

    Re = [20.0 + 3.0 * s for s in sides]
    got = []
    for own in (False, True):
        b = CavityBatch(sides, Re, lid_speed=0.1)
        if own:
            b.set_schedule(64, 0, 3)
        out = []
        for n in (1, 2, 3, 7, 4):
            b.step(n)
        out += [b.fields_host(c, ("P", "u", "rho", "G")) for c in range(b.n)]
        b.init()
        for period in (6, 4, 100):  # by twos with a four for 6 and 100, or by fours and twos
            r = b.run(tol=1e-4, max_steps=3 * period, check_every=period)
        out += [{"steps": r[0], "status": r[1], "res": r[2]}]
        out += [b.fields_host(c, ("P", "u", "rho", "G")) for c in range(b.n)]
        b.close()
        got.append(out)
    for a, b in zip(*got):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("last", [129, 177, 866])
def test_fused_cavities_as_they_retire(last):
    """Most cavities converge early: the last one goes on alone in its cluster,
    or on the lists of shorter segments, and keeps the persistent kernel's
    bits."""
    from paper_2108_08591_gb300 import CavityBatch

    sides, Re = [33] * 40 + [last], [40.0] * 40 + [300.0]
    got = []
    for own in (False, True):
        b = CavityBatch(sides, Re, lid_speed=0.1)
        if own:
            b.set_schedule(64, 0, 3)
        r = b.run(tol=1e-6, max_steps=6000, check_every=100)
        got.append((*r, b.fields_host(0, ("u",))["u"], b.fields_host(40, ("u", "P"))["u"]))
        b.close()
    assert (got[0][1][:40] == 0).all() and got[0][0][:40].max() < got[0][0][40]
    for a, b in zip(*got):
        assert np.array_equal(a, b)
