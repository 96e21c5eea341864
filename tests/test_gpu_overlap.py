"""Steps in one call, replayed from graphs of 2 and of 16 steps whose kernels
may overlap at their ends, against the same steps one call and one wait at a
time, where none can: bitwise equal. Lattices on both sides of the rules that
let kernels overlap, with relaxation time 1 (which has kernels of its own)
and another, with and without solid nodes; and batches, whose members all
relax with time 1 or all with another, against the members alone."""
import numpy as np
import pytest

from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu

F64, F32, F16S, BF16S = 0, 1, 2, 3


@pytest.fixture(scope="module")
def lbm():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    return L


def make(lbm, storage, shape, tau, solid, seed=3, flags=0):
    nx, ny, nz = shape
    w = inputs.DROP_D2Q9_64 if nz == 1 else inputs.DROP_D3Q27_128
    side = min(nx, ny) if nz == 1 else min(shape)
    mask = inputs.block_mask(nx, ny, nz, (nx - 2, 1, 0), (nx, 3, min(nz, 2))) if solid else None
    g = lbm.LBM(0 if nz == 1 else 1, nx, ny, nz, w.eos, w.t_over_tc, w.kappa, tau, storage=storage, mask=mask,
                a=w.a, b=w.b, rho_w=w.rho_v, flags=flags)
    g.init(inputs.add_noise(inputs.drop(nx, ny, nz, side / 4, w.rho_v, w.rho_l), 1e-3, seed))
    return g


def one_by_one(g, n):
    for _ in range(n):
        g.step(1)
        g.sync()
    return g.get_populations()


# 2D: kernels side by side, in between, and 1024 blocks of 32 x 8 nodes, more than
# any SM count's residents leave room beside; 3D: whole and cut tiles, and a row
# of ny = 9, whose lower halo lies in no box (read from memory)
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("storage,shape", [
    (F64, (32, 20, 1)), (F64, (61, 37, 1)), (F32, (64, 64, 1)), (F32, (1000, 256, 1)), (F16S, (64, 64, 1)),
    (F16S, (1000, 256, 1)), (BF16S, (250, 200, 1)), (F32, (64, 24, 20)), (F32, (64, 9, 12)), (F32, (37, 21, 11)),
    (F16S, (64, 24, 20)), (BF16S, (40, 16, 12))])
def test_steps_at_once_equal_steps_one_by_one(lbm, storage, shape, solid, tau):
    a, b = make(lbm, storage, shape, tau, solid), make(lbm, storage, shape, tau, solid)
    a.step(35)   # an odd number: a plain launch, graphs of 16 and of 2
    f = a.get_populations()
    assert np.all(np.isfinite(f)) and np.array_equal(f, one_by_one(b, 35))


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("solid", [False, True])
@pytest.mark.parametrize("storage,shapes", [
    (F32, [(64, 64, 1), (96, 33, 1), (31, 70, 1)]), (F16S, [(64, 64, 1), (96, 33, 1), (31, 70, 1)]),
    (BF16S, [(512, 256, 1), (480, 500, 1), (64, 64, 1)]), (F32, [(512, 256, 1), (480, 500, 1), (64, 64, 1)]),
    (F32, [(32, 16, 12), (45, 9, 14), (64, 24, 10)]), (F16S, [(32, 16, 12), (45, 9, 14), (64, 24, 10)])])
def test_batch_of_one_relaxation_equals_members_alone(lbm, storage, shapes, solid, tau):
    # (solid: one member with solid nodes makes its launch the one for them)
    alone = [one_by_one(make(lbm, storage, s, tau, solid and k == 1, k), 35) for k, s in enumerate(shapes)]
    members = [make(lbm, storage, s, tau, solid and k == 1, k) for k, s in enumerate(shapes)]
    b = lbm.Batch(members)
    b.step(35)
    b.sync()
    for g, ref in zip(members, alone):
        f = g.get_populations()
        assert np.all(np.isfinite(f)) and np.array_equal(f, ref)
