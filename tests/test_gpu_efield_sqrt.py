"""|E| against the same expression in numpy FP64, bit for bit (numpy's sqrt is
correctly rounded): random fields over the range of exponents, squares,
neighbours of squares, zeros, and sums that are subnormal or overflow."""

import numpy as np
import pytest


def _field(a, c):
    ax, ay, az = a
    ex = (((ax[:-1, :-1, :-1] + ax[1:, :-1, :-1]) + ax[:-1, 1:, :-1]) + ax[1:, 1:, :-1]) * c
    ey = (((ay[:-1, :-1, :-1] + ay[1:, :-1, :-1]) + ay[:-1, :-1, 1:]) + ay[1:, :-1, 1:]) * c
    ez = (((az[:-1, :-1, :-1] + az[:-1, 1:, :-1]) + az[:-1, :-1, 1:]) + az[:-1, 1:, 1:]) * c
    with np.errstate(over="ignore", under="ignore"):
        return np.sqrt((ex * ex + ey * ey) + ez * ez)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["uniform", "exponents", "squares", "extremes"])
def test_field_magnitude_bits(kind):
    torch = pytest.importorskip("torch")
    import paper_2010_12879_gb300 as spfd
    nx, ny, nz = 67, 50, 61
    shape = (3, nz + 1, ny + 1, nx + 1)
    rng = np.random.default_rng(5)
    if kind == "uniform":
        a = rng.normal(size=shape)
    elif kind == "exponents":
        a = np.ldexp(rng.normal(size=shape), rng.integers(-500, 480, size=shape))
    elif kind == "squares":  # E_x alone: x = 4 a, and x^2 or its neighbours
        a = np.zeros(shape)
        a[0] = rng.integers(0, 1 << 26, size=shape[1:])[:, :, :1]
        a[1, ..., 0] = rng.integers(0, 2, size=shape[1:-1])
    else:
        a = rng.choice([0.0, 1e-170, 3e-162, 1e153, 2e-160, 1.0], size=shape)
    omega = 2.0
    with spfd.Solver(torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda"), 0.5) as S:
        psi = torch.zeros(S.node_shape, dtype=torch.float64, device="cuda")
        E = S.efield(torch.from_numpy(a).cuda(), psi, omega).cpu().numpy()
    # a + 0 - 0 leaves every term as it is; c = omega / (4 h) = 1
    ref = _field(a, omega / (4 * 0.5))
    assert np.array_equal(E, ref)
