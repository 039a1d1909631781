"""FP64 initialisation against NumPy: the equilibrium of every set and
direction (Eq. 2-4) rounded operation by operation, so the bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

AXES2, AXES3 = [(1, 0), (0, 1), (-1, 0), (0, -1)], [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
LATTICES = {(2, 0): ([(0, 0)] + AXES2, [1 / 3] + [1 / 6] * 4, 1 / 3), (2, 4): (AXES2, [0.25] * 4, 0.5),
            (3, 0): ([(0, 0, 0)] + AXES3, [0.25] + [0.125] * 6, 0.25), (3, 6): (AXES3, [1 / 6] * 6, 1 / 3)}


def equilibrium(c, w, cs2, P, u):
    """[1 + d][q][N]: the alpha = 0 set, then the velocity sets."""
    d, out = len(u), []
    for alpha in range(d + 1):
        for ci, wi in zip(c, w):
            cu = np.zeros_like(P)
            for b in range(d):
                if ci[b]:
                    cu = cu + u[b] if ci[b] > 0 else cu - u[b]
            if alpha == 0:
                out.append(wi * cu * (1 / cs2))
                continue
            ua, k = u[alpha - 1], ci[alpha - 1]
            cP = k * (P - 1.0) if k else np.zeros_like(P)
            out.append(wi * (ua + (cu * ua + cP) * (1 / cs2)))
    return np.array(out)


@pytest.mark.parametrize("shape,q", [((67, 45), 0), ((67, 45), 4), ((33, 20, 18), 0), ((33, 20, 18), 6)])
@pytest.mark.parametrize("with_rho", [True, False])
def test_f64_initial_state_is_the_equilibrium_bit_for_bit(tmp_path, shape, q, with_rho):
    from paper_2108_08591_gb300 import Lattice

    d, N = len(shape), int(np.prod(shape))
    rng = np.random.default_rng([*shape, q])
    P = 1.0 + 1e-3 * rng.standard_normal(N)
    u = 0.03 * rng.standard_normal((d, N))
    # the in-place layout holds each node's own populations
    lat = Lattice(shape, s1=1.7, storage="f64", q=q, inplace=True, with_rho=with_rho)
    lat.init(P, u)
    lat.save(str(tmp_path / "state"))
    px = lat.info.pitch
    lat.close()
    want = equilibrium(*LATTICES[d, q], P, u)[0 if with_rho else len(LATTICES[d, q][0]):]
    raw = np.fromfile(tmp_path / "state", np.uint8)[-len(want) * px * (N // shape[0]) * 8:].view(np.float64)
    got = raw.reshape(len(want), N // shape[0], px)[:, :, :shape[0]].reshape(len(want), N)
    assert np.array_equal(got, want)
