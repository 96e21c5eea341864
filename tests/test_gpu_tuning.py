"""lbm_autotune of D2Q9 lattices, whose step has nothing to tune: a state that
is not finite is still reported."""
import numpy as np
import pytest

from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

ENONFINITE, ESTATE = 4, 6


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    return L


@pytest.mark.parametrize("lattice", [0, 1])
@pytest.mark.parametrize("storage", [1, 2, 3])
@pytest.mark.parametrize("seen", [False, True])
def test_autotune_reports_a_diverged_state(lbm, lattice, storage, seen):
    w = inputs.DROP_D2Q9_64
    n = (32, 16, 8 if lattice else 1)
    g = lbm.LBM(lattice, *n, w.eos, w.t_over_tc, w.kappa, 1.0, a=w.a, b=w.b, storage=storage)
    rho = np.full(n[0] * n[1] * n[2], w.rho_l)
    g.init(rho)
    assert g.autotune() >= 1
    f = g.get_populations()
    f[5] = np.nan
    g.set_populations(f)
    g.step(1)
    if seen:   # the divergence has been reported before
        with pytest.raises(lbm.LBMError) as e:
            g.sync()
        assert e.value.code == ENONFINITE
    with pytest.raises(lbm.LBMError) as e:
        g.autotune()
    assert e.value.code == (ESTATE if seen else ENONFINITE)
    g.init(rho)
    assert g.autotune() >= 1
