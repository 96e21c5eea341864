"""The FP64 kernels at the edges of their tiles and chunks against the FP64
oracle: direct force sums (small D3Q27), the marching tiles (larger ones), the
two row heights of the D2Q9 tile, and nodes whose populations are negative,
tiny or of far apart exponents (summed in FP64 instead of fixed point). Three
steps from one state; tolerance 1e-10 of each field's largest value, as the
other FP64 comparisons (single roundings of 1e-16, grown by at most 1e2 per
field in the force sums)."""
import numpy as np
import pytest

from oracle.lbm import OracleLBM
from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    return L


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("shape", [(5, 5, 1), (31, 9, 1), (65, 130, 1), (300, 333, 1), (513, 161, 1), (5, 5, 5),
                                   (9, 7, 5), (33, 12, 11), (70, 41, 37), (30, 65, 66), (97, 61, 33)])
def test_fp64_tiles(lbm, shape, solid, tau):
    w = inputs.DROP_D3Q27_128
    nx, ny, nz = shape
    lat, n = int(nz > 1), nx * ny * nz
    mask = inputs.block_mask(nx, ny, nz, (nx - 2, 1, 0), (nx, 3, min(nz, 2))) if solid else None
    kw = dict(mask=mask, a=w.a, b=w.b, rho_w=w.rho_v)
    rho = inputs.add_noise(inputs.drop(nx, ny, nz, min(nx, ny) / 4, w.rho_v, w.rho_l), 1e-2, 5)
    g = lbm.LBM(lat, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, tau, **kw)
    o = OracleLBM(lat, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, tau, **kw)
    o.init(rho)
    g.init(rho)
    f = o.get_populations().reshape(-1, n)
    # a few nodes outside the range of the fixed-point sums
    rest, some = f[0], np.arange(0, n, 17)
    moved = 1.5 * f[1, some]
    f[1, some] -= moved
    rest[some] += moved
    f[2, some[::2]] = 1e-300
    f[3, some[::3]] = 0.0
    for h in (g, o):
        h.set_populations(f.reshape(-1))
        h.step(3)
    fl = np.ones(n, bool) if mask is None else mask == 0
    err = {}
    fields = {"f": (g.get_populations(), o.get_populations())}
    fields.update(zip(("rho", "u", "U"), zip(g.moments(), o.moments())))
    fields["P"] = (g.pressure_tensor().reshape(-1), o.pressure_tensor().reshape(-1))
    for k, (a, b) in fields.items():
        keep = np.tile(fl, a.size // n)
        err[k] = float(np.max(np.abs(a - b)[keep]) / np.max(np.abs(b[keep])))
    assert max(err.values()) < TOL, err
    a, b = g.reduce(), o.reduce()
    assert abs(a[0] / b[0] - 1) < TOL
