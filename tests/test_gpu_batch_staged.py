"""Batches of D3Q27 lattices in the TMA-staged forms: more members than one
launch takes, rows of any width, members with and without solids and of two
equations of state, each bitwise as the same lattice stepped alone."""
import numpy as np
import pytest

from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [1, 2])
@pytest.mark.parametrize("count,mixed", [(1, False), (5, False), (5, True), (35, True)])
def test_staged_batch_equals_alone(storage, count, mixed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    pr, vdw = inputs.DROP_D3Q27_128, inputs.DROP_D2Q9_64

    def make(k):
        nx, ny, nz = 20 + 7 * (k % 6), 9 + 5 * (k % 4), 30 - 4 * (k % 5)
        w = vdw if mixed and k % 3 == 1 else pr
        mask = inputs.block_mask(nx, ny, nz, (2, 3, 1), (6, 7, 4)) if mixed and k % 4 == 2 else None
        g = L.LBM(1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, 0.9, a=w.a, b=w.b, mask=mask, rho_w=w.rho_v,
                  storage=storage)
        g.init(inputs.add_noise(inputs.drop(nx, ny, nz, min(nx, ny, nz) / 4, w.rho_v, w.rho_l), 1e-4, k))
        return g

    alone = []
    for k in range(count):
        g = make(k)
        g.step(7)
        alone.append(g.get_populations())
    members = [make(k) for k in range(count)]
    b = L.Batch(members)
    b.step(7)
    b.sync()
    assert b.launches == 7
    for g, ref in zip(members, alone):
        f = g.get_populations()
        assert np.all(np.isfinite(f)) and np.array_equal(f, ref)
