"""Reduced storage with relaxation time 1, whose steps are kernels of their own
(no f and feq): cut tiles, padded rows and solid nodes, one step from an
identical state against the FP64 oracle at the single-step tolerances (2e-6 of
max f for FP32, the 16-bit rounding of h for shifted storage); and every form
of the D3Q27 step bitwise as the plain one."""
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
@pytest.mark.parametrize("shape", [(5, 5, 1), (31, 7, 1), (33, 9, 1), (130, 12, 1), (5, 5, 5), (33, 9, 11), (35, 17, 9),
                                   (40, 6, 12), (97, 21, 8)])
@pytest.mark.parametrize("solid", [False, True])
def test_relaxation_time_1(lbm, storage, shape, solid):
    nx, ny, nz = shape
    three = nz > 1
    w = inputs.DROP_D3Q27_128 if three else inputs.DROP_D2Q9_64
    side = min(shape) if three else min(nx, ny)
    rho = inputs.add_noise(inputs.drop(nx, ny, nz, side / 4, w.rho_v, w.rho_l), 1e-2, 3)
    mask = inputs.block_mask(nx, ny, nz, (nx - 2, 1, 0), (nx, 3, 2 if three else 1)) if solid else None
    kw = dict(mask=mask, a=w.a, b=w.b, rho_w=w.rho_v, g=(1e-4, -2e-4, 0.0))
    args = (1 if three else 0, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, 1.0)

    def make(form=None):
        g = lbm.LBM(*args, storage=storage, **kw)
        g.init(rho)
        if form is not None:
            g.set_fused_variant(form)
        g.step(3)
        return g

    g = make()
    o = OracleLBM(*args, **kw)
    o.init(rho)
    f = g.get_populations()
    o.set_populations(f)
    forms = []
    if three:
        forms = [0, 1, 2, 3, 4] if storage == 1 else [0, 2, 3, 4, 5]
    for form in forms:
        assert np.array_equal(make(form).get_populations(), f), form
    g.step(1)
    o.step(1)
    fg, fo = g.get_populations(), o.get_populations()
    fl = np.ones(g.Q * g.N, bool) if mask is None else np.tile(mask == 0, g.Q)
    assert float(np.max(np.abs(fg - fo)[fl])) < STEP_TOL[storage] * float(np.max(np.abs(fo[fl])))
