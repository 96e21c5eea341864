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


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("storage", [2, 3])
@pytest.mark.parametrize("ratio", [1.0, 3.0, 200.0])
@pytest.mark.parametrize("solid", [False, True])
def test_shifted_sums(lbm, D, storage, ratio, solid):
    """Density and bare velocity of 16-bit shifted storage against exact sums
    of (w_i + h_i) rho(source), h_i found again from the decoded populations,
    for densities that differ by up to `ratio` between neighbours. Fixed point:
    1.5 units of 2^-56 of the largest population each; nodes whose largest
    population is below 1/16 of a source, or with an h of 1 or more (both at 200):
    FP64, 2 roundings per population and one per addition."""
    from paper_2112_01975_gb300 import inputs
    LD = np.longdouble
    n = (20, 13, 9 if D == 3 else 1)
    N = n[0] * n[1] * n[2]
    rng = np.random.default_rng(11)
    rho0 = np.exp(rng.uniform(0, np.log(ratio), N)) if ratio > 1 else 1 + 1e-3 * rng.random(N)
    w1 = np.array([1 / 6, 2 / 3, 1 / 6])
    Q = 3 ** D
    c = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1 if D == 3 else 0) for i in range(Q)]
    w = [w1[a + 1] * w1[b + 1] * (w1[d + 1] if D == 3 else 1.0) for a, b, d in c]
    f = np.array([w[i] * rho0 * (1 + 0.05 * rng.standard_normal(N)) for i in range(Q)])
    mask = inputs.block_mask(*n, (4, 3, 2 if D == 3 else 0), (9, 7, 6 if D == 3 else 1)) if solid else None
    fl = np.ones(N, bool) if mask is None else mask.ravel() == 0
    p = inputs.DROP_D2Q9_64
    g = lbm.LBM(0 if D == 2 else 1, *n, p.eos, p.t_over_tc, p.kappa, 1.0, a=p.a / 50, b=p.b / 50, storage=storage,
                mask=mask, rho_w=1.0)
    g.set_populations(f.ravel())
    dec = g.get_populations().reshape(Q, N)
    rho, u, _ = g.moments()
    own = np.float32(f.astype(LD).sum(0)).astype(np.float64)   # the source densities
    pops, big_src, big_h = [], np.zeros(N), np.zeros(N)
    grid = n[::-1]
    for i in range(Q):
        src = np.roll(own.reshape(grid), (c[i][2], c[i][1], c[i][0]), (0, 1, 2)).ravel()
        if mask is not None:
            bounced = np.roll(mask.reshape(grid), (c[i][2], c[i][1], c[i][0]), (0, 1, 2)).ravel() != 0
            src = np.where(bounced, own, src)
        h = (dec[i] / src - w[i]).astype(np.float32)
        if storage == 2:
            h = h.astype(np.float16).astype(np.float64)
        else:   # to nearest with 8 bits
            h = (((h.view(np.uint32) + 0x8000) >> 16) << 16).astype(np.uint32).view(np.float32).astype(np.float64)
        assert np.array_equal(((w[i] + h) * src)[fl], dec[i][fl])   # h is the stored one
        pops.append((LD(w[i]) + h.astype(LD)) * src.astype(LD))
        big_src, big_h = np.maximum(big_src, src), np.maximum(big_h, abs(h))
    pops = np.array(pops)
    largest, mag = abs(pops).max(0), abs(pops).sum(0)
    slow = (big_src > 15 * largest) | (big_h >= 1)   # may be summed in FP64
    unit = 1.5 * LD(2) ** -56 * largest
    slack = np.where(slow, (Q + 2) * LD(2) ** -53 * mag, Q * unit)
    want = pops.sum(0)
    assert np.all((abs(rho - want) <= slack + LD(2) ** -53 * want)[fl])
    for a in range(D):
        j = sum(c[i][a] * pops[i] for i in range(Q))
        jslack = np.where(slow, slack, Q * 2 / 3 * unit)
        err = abs(u[a * N:(a + 1) * N] - j / want)
        assert np.all((err <= jslack / want + abs(j / want) * (slack / want + 4 * LD(2) ** -53))[fl])
