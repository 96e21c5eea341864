"""Encoding of 16-bit shifted storage, h = f / rho(source) - w rounded to FP32
and then to 16 bits, against numpy's division over populations of very
different sizes and signs: the same stored values. (The library forms the
quotient from an FP32 one and corrects it by its remainder; its FP64 rounding
may differ from the division's, which reaches the 16 bits once in 2^29 or
less.)"""
import numpy as np
import pytest

from paper_2112_01975_gb300 import inputs

pytestmark = pytest.mark.gpu


def to_16(h, storage):
    """FP32 -> 16 bits, to nearest even -> FP64."""
    if storage == 2:
        return h.astype(np.float16).astype(np.float64)
    b = h.view(np.uint32).astype(np.uint64)
    b = (b + 0x7fff + ((b >> 16) & 1)) >> 16 << 16
    return b.astype(np.uint32).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("storage", [2, 3])
@pytest.mark.parametrize("scale", [1e-25, 1e-15, 1e-3, 1.0, 1e12, 1e25])
def test_encoding_is_the_division(D, storage, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_01975_gb300 import build
    build.build()
    from paper_2112_01975_gb300 import lbm as L
    n = (40, 33, 11 if D == 3 else 1)
    N, Q = n[0] * n[1] * n[2], 3 ** D
    rng = np.random.default_rng(5)
    w1 = (1 / 6, 2 / 3, 1 / 6)
    c = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1 if D == 3 else 0) for i in range(Q)]
    w = [w1[a + 1] * w1[b + 1] * (w1[d + 1] if D == 3 else 1.0) for a, b, d in c]
    rho = scale * np.exp(rng.uniform(-1, 1, N))
    f = np.array([w[i] * rho * (1 + 0.1 * rng.standard_normal(N)) for i in range(Q)])
    odd = rng.random(f.shape) < 0.05   # some far from equilibrium, small, negative or zero
    f[odd] *= rng.choice([0.0, -0.3, 1e-3, 1e-9, -1e-25], int(odd.sum()))
    p = inputs.DROP_D2Q9_64
    g = L.LBM(0 if D == 2 else 1, *n, p.eos, p.t_over_tc, p.kappa, 1.0, a=p.a, b=p.b, storage=storage)
    g.set_populations(f.ravel())
    got = g.get_populations().reshape(Q, N)
    own = f.astype(np.longdouble).sum(0).astype(np.float32).astype(np.float64)
    for i in range(Q):
        src = np.roll(own.reshape(n[::-1]), (c[i][2], c[i][1], c[i][0]), (0, 1, 2)).ravel()
        h = to_16((f[i] / src - w[i]).astype(np.float32), storage)
        assert np.array_equal(got[i], (w[i] + h) * src), i
