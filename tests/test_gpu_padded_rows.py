"""D3Q27 lattices of reduced storage whose rows the library pads to 16 bytes,
and tiles cut by the lattice's edge in the TMA-staged forms: a handle left to
choose its form against the plain form (bitwise), and one step from an
identical state against the FP64 oracle at the single-step tolerances (2e-6
of max f for FP32, the 16-bit rounding of h for shifted storage)."""
import numpy as np
import pytest

from oracle.lbm import OracleLBM
from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

STEP_TOL = {1: 2e-6, 2: 2e-4, 3: 2e-3}


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    return L


@pytest.mark.parametrize("storage", [1, 2, 3])
@pytest.mark.parametrize("shape", [(5, 5, 5), (31, 7, 6), (33, 9, 11), (34, 8, 7), (35, 17, 9), (40, 6, 12),
                                   (62, 16, 7), (94, 97, 5), (95, 15, 6), (97, 21, 8)])
@pytest.mark.parametrize("solid", [False, True])
def test_padded_rows(lbm, storage, shape, solid):
    import torch
    w = inputs.DROP_D3Q27_128
    nx, ny, nz = shape
    n = nx * ny * nz
    mask = inputs.block_mask(nx, ny, nz, (nx - 2, 1, 0), (nx, 3, 2)) if solid else None
    rho = inputs.add_noise(inputs.drop(nx, ny, nz, min(shape) / 4, w.rho_v, w.rho_l), 1e-2, 3)
    kw = dict(mask=mask, a=w.a, b=w.b, rho_w=w.rho_v)
    g = lbm.LBM(1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, 0.8, storage=storage, **kw)
    g.init(rho)
    stray = nx % (4 if storage == lbm.F32 else 8) == 1
    use = nx * ny / (-(-nx // 32) * 32 * -(-ny // 8) * 8)
    assert g.fused_variant == (lbm.FUSED_TMEM if stray or (storage != lbm.F32 and use < 0.9) else
                               lbm.FUSED_WS_TMA if storage == lbm.F32 else lbm.FUSED_TM_TMA)
    p = lbm.LBM(1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, 0.8, storage=storage, **kw)
    p.set_fused_variant(lbm.FUSED_PLAIN)
    p.init(rho)
    g.step(5)
    p.step(5)
    f = g.get_populations()
    assert np.all(np.isfinite(f)) and np.array_equal(f, p.get_populations())
    # read-back through the host and the device, and a restart from it
    host = g.moments() + (g.pressure_tensor().reshape(-1),)
    dev = tuple(torch.empty(k * n, dtype=torch.float64, device="cuda") for k in (1, 3, 3, 6, 27))
    g.moments(out=dev[:3])
    g.pressure_tensor(out=dev[3])
    g.get_populations(dev[4])
    for a, b in zip(host, dev):
        assert np.array_equal(a, b.cpu().numpy())
    fl = np.ones(n, bool) if mask is None else mask == 0
    fl27 = np.tile(fl, 27)
    assert np.array_equal(dev[4].cpu().numpy()[fl27], f[fl27])
    assert abs(g.reduce()[0] / f[fl27].sum() - 1) < 1e-12
    o = OracleLBM(1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, 0.8, **kw)
    o.init(rho)
    o.set_populations(f)
    g.set_populations(dev[4] if not solid else f)
    g.step(1)
    o.step(1)
    fg, fo = g.get_populations(), o.get_populations()
    assert float(np.max(np.abs(fg - fo)[fl27])) < STEP_TOL[storage] * float(np.max(np.abs(fo[fl27])))
