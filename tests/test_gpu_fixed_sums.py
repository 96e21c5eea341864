"""Sums of populations in 64-bit fixed point (density, momentum, second
moments): populations that are zero or far below the largest of their node
count for what they are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    return L


def lattice(lbm, D, storage, n=7):
    from paper_2112_01975_gb300 import inputs
    w = inputs.DROP_D2Q9_64
    return lbm.LBM(0 if D == 2 else 1, n, n, n if D == 3 else 1, w.eos, w.t_over_tc, w.kappa, 1.0, a=w.a, b=w.b,
                   storage=storage)


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("small", [0.0, 2.0 ** -70, 2.0 ** -59, 2.0 ** -56, 2.0 ** -53])
def test_small_populations(lbm, D, storage, small):
    """One population of 1, the others `small`: the density is the exact sum
    rounded once to FP64 (all of them are whole units of 2^-57, or below half
    of one and then nothing)."""
    g = lattice(lbm, D, storage)
    Q = g.Q
    f = np.full((Q, g.N), small)
    f[Q // 2] = 1.0   # the population at rest
    g.set_populations(f.ravel())
    rho, u, _ = g.moments()
    assert np.all(rho == 1.0 + (Q - 1) * small) and not u.any()
    # the largest one moving: the momentum is its own
    f[Q // 2], f[0] = small, 1.0
    g.set_populations(f.ravel())
    rho, u, _ = g.moments()
    j = -(1.0 - small)   # the other end of its pair moves the other way
    assert np.all(rho == 1.0 + (Q - 1) * small)
    assert np.all(abs(u - j / rho[0]) <= 2.0 ** -51)
