"""The D2Q9 step of reduced storage (32 x 8 tiles) at the edges of its tiles,
one step from an identical state against the FP64 oracle. Tolerances as for
the other single-step comparisons: 2e-6 of max f for FP32, the 16-bit
rounding of h for shifted storage (2e-4 FP16, 2e-3 BF16)."""
import numpy as np
import pytest

from oracle.lbm import OracleLBM
from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

STEP_TOL = {1: 2e-6, 2: 2e-4, 3: 2e-3}


@pytest.mark.parametrize("storage", [1, 2, 3])
@pytest.mark.parametrize("shape", [(5, 5), (31, 7), (32, 8), (33, 9), (64, 17), (7, 150), (130, 12)])
@pytest.mark.parametrize("solid,flags", [(False, 0), (True, 0), (True, 2)])
def test_step2d_tile_edges(storage, shape, solid, flags):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    w = inputs.DROP_D2Q9_64
    nx, ny = shape
    rho = inputs.add_noise(inputs.drop(nx, ny, 1, min(nx, ny) / 4, w.rho_v, w.rho_l), 1e-2, 3)
    mask = inputs.block_mask(nx, ny, 1, (nx - 2, 1, 0), (nx, 3, 1)) if solid else None
    kw = dict(mask=mask, a=w.a, b=w.b, rho_w=w.rho_v, g=(1e-4, -2e-4, 0.0))
    g = L.LBM(0, nx, ny, 1, w.eos, w.t_over_tc, w.kappa, 0.8, storage=storage, flags=flags, **kw)
    o = OracleLBM(0, nx, ny, 1, w.eos, w.t_over_tc, w.kappa, 0.8, **kw)
    g.init(rho)
    o.init(rho)
    g.step(3)
    o.set_populations(g.get_populations())
    g.step(1)
    o.step(1)
    fg, fo = g.get_populations(), o.get_populations()
    fl = np.ones(9 * nx * ny, bool) if mask is None else np.tile(mask == 0, 9)
    assert float(np.max(np.abs(fg - fo)[fl])) < STEP_TOL[storage] * float(np.max(np.abs(fo[fl])))
