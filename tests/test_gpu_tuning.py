"""lbm_autotune of D2Q9 lattices, whose step has nothing to tune: a state that
is not finite is still reported. And the form that a lattice of any width
reports, by its own choice or tuned, can be set on it and on another."""
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


@pytest.mark.parametrize("storage", [1, 2, 3])
@pytest.mark.parametrize("nx", [38, 41, 64, 97])
def test_a_reported_form_can_be_set(lbm, storage, nx):
    w = inputs.DROP_D3Q27_128
    n = (nx, 24, 16)
    rho = inputs.add_noise(inputs.drop(*n, 5.0, w.rho_v, w.rho_l), 1e-3, 5)

    def make():
        g = lbm.LBM(1, *n, w.eos, w.t_over_tc, w.kappa, 0.8, a=w.a, b=w.b, storage=storage)
        g.init(rho)
        return g

    ref = make()
    ref.set_fused_variant(lbm.FUSED_PLAIN)
    ref.step(5)
    want = ref.get_populations()
    tuned = make()
    own = tuned.fused_variant
    chunk = tuned.autotune()
    # the TMA-staged forms of the storage run at any width
    staged = lbm.FUSED_WS_TMA if storage == lbm.F32 else lbm.FUSED_TM_TMA
    for v in {own, tuned.fused_variant, staged, lbm.FUSED_WS_TMA}:
        g = make()
        g.set_fused_variant(v)
        g.set_chunk(chunk)
        assert g.fused_variant == v
        g.step(5)
        assert np.array_equal(g.get_populations(), want)
    tuned.set_fused_variant(tuned.fused_variant)
    tuned.step(5)
    assert np.array_equal(tuned.get_populations(), want)
