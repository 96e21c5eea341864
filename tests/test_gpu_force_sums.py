"""Rounding of the FP64 force sweeps: they take differences along each axis
before they smooth them, so the error is that of the differences and not of
the fields, also where a field is nearly uniform. (Lattices of fewer than
about 45^3 nodes sum node by node, differences of opposite nodes, and do not
take the sweeps.)

A fluid at rest (u = 0 exactly: opposite populations equal) with a capillary
coefficient so large that the rho stencil dominates: U = F / (2 rho) against
the same sums in extended precision. Bound: 16 roundings between the stored
densities and U (the difference 1, two smoothings 4, the sums along z 4, the
rings 1, their coefficient 3, force and U 3), each at most 2^-53 of the sum
of the terms' magnitudes; and 1e-9 of them for the psi part, 1e-8 of the
whole and formed here from the equation of state."""
import numpy as np
import pytest

from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

KAPPA = 1e8
LD = np.longdouble


def at(v, a, k):
    return np.roll(v, -k, a)


def sums(v, scale):
    """Per axis (x last) sum_i (w_i / cs2) c_i v(r + k c_i), k = 1, 2, scaled and
    added, and the same of the terms' magnitudes."""
    D = v.ndim
    out = []
    for ax in range(D):
        tot, mag = np.zeros_like(v), np.zeros_like(v)
        for k, s in zip((1, 2), scale):
            d = (at(v, D - 1 - ax, k) - at(v, D - 1 - ax, -k)) / 2
            m = abs(d)
            for b in range(D):
                if b != ax:
                    d = (4 * d + at(d, D - 1 - b, k) + at(d, D - 1 - b, -k)) / 6
                    m = (4 * m + at(m, D - 1 - b, k) + at(m, D - 1 - b, -k)) / 6
            tot, mag = tot + s * d, mag + abs(s) * m
        out.append((tot, mag))
    return out


@pytest.mark.parametrize("shape", [(64, 64), (37, 29), (301, 202), (70, 50, 41), (64, 64, 64), (97, 61, 75)])
def test_force_rounds_at_the_differences(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    w = inputs.DROP_D2Q9_64
    nx, ny = shape[:2]
    nz = shape[2] if len(shape) == 3 else 1
    D, Q = len(shape), 3 ** len(shape)
    rho0 = inputs.add_noise(inputs.drop(nx, ny, nz, min(shape) / 4, w.rho_v, w.rho_l), 1e-4, 7)
    w1 = (1 / 6, 2 / 3, 1 / 6)
    f = np.concatenate([rho0.ravel() * (w1[i % 3] * w1[i // 3 % 3] * (w1[i // 9] if D == 3 else 1.0))
                        for i in range(Q)])
    g = L.LBM(0 if D == 2 else 1, nx, ny, nz, w.eos, w.t_over_tc, KAPPA, 1.0, a=w.a, b=w.b)
    g.set_populations(f)
    rho, u, U = g.moments()
    assert not u.any()
    r = rho.reshape(shape[::-1]).astype(LD)
    rt = LD(w.t_over_tc * (8.0 * w.a / (27.0 * w.b)))
    d = r * rt / (1 - LD(w.b) * r) - LD(w.a) * r * r - r / 3
    psi = np.sqrt(abs(d))
    s = np.where(d > 0, 1, -1)
    Sr, Sp = sums(r, (2, -1)), sums(psi, (LD(4) / 3, -LD(1) / 6))
    for a in range(D):
        want = (-2 * s * psi * Sp[a][0] - LD(KAPPA) * r * Sr[a][0]) / (2 * r)
        err = abs(U[a * r.size:(a + 1) * r.size].reshape(r.shape) - want)
        bound = 16 * LD(2) ** -53 * (LD(KAPPA) / 2) * Sr[a][1] + LD(1e-9) * 2 * psi * Sp[a][1] / (2 * r)
        assert np.all(err <= bound), (a, float(np.max(err / bound)))
