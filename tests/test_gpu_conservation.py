"""Mass and momentum of a periodic box without forces: the collision keeps both up to rounding.

Stored FP32 populations are deviations from w_i rho_ref.  What a sound collision may change per step is
 - what the rounded weights make of sum w = 1 and 3 sum w c_x c_x = 1 (a factor of om times their defect), and
 - the rounding errors themselves, which have no common sign: a quarter of the unit roundoff per step is allowed
   for what remains of them.
A collision whose constants do not add up to one multiplies mass and momentum by the same factor in every step; for
the relaxation times below that is up to a full unit roundoff (2^-24)."""
import math

import numpy as np
import pytest

from paper_2502_12955_gb300.lbm import Solver

pytestmark = pytest.mark.gpu

STEPS = 2000
C2 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
C3 += [(s * a, s * b, s * d) for (a, b, d) in ((1, 1, 0), (1, 0, 1), (0, 1, 1), (1, -1, 0), (1, 0, -1), (0, 1, -1)) for s in (1, -1)]
W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _box(dim, n, tau, precision, **kw):
    shape = (n, n, n) if dim == 3 else (1, n, n)
    cfg = dict(dim=dim, nx=n, ny=n, nz=shape[0], n_comp=1, tau=[tau], n_scal=0, periodic=[1, 1, 1], precision=precision, **kw)
    rng = np.random.default_rng(7)
    ph = 2 * math.pi * np.arange(n) / n
    x, y = ph[None, None, :], ph[None, :, None]
    rho = (1.02 + 0.01 * np.sin(x) * np.cos(y) + 0.0007 * rng.uniform(-1, 1, shape))[None]
    u = np.zeros((3,) + shape)
    u[0] += 0.02 + 0.01 * np.cos(y)
    u[1] += 0.01 * np.sin(x)
    s = Solver(cfg)
    s.set_geometry(np.zeros(shape, np.uint8))
    s.set_fields(rho, u, None)
    return s


def _totals(s, c, w, ref):
    f = s.pops()[0][0] - ref * np.asarray(w)[:, None]
    return math.fsum(f.ravel()), math.fsum((f * np.array([v[0] for v in c], float)[:, None]).ravel())


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("tau", [0.55, 0.6, 0.7, 0.9, 1.1])
@pytest.mark.parametrize("kw", [{}, {"forcing": "sc_shift"}, {"collision": "mrt"}], ids=["guo", "shift", "mrt"])
def test_fp32_mass_and_momentum_stay(dim, tau, kw):
    c, w = (C3, W3) if dim == 3 else (C2, W2)
    s = _box(dim, 16 if dim == 3 else 32, tau, "fp32", **kw)
    m0, p0 = _totals(s, c, w, 1.0)
    s.step(STEPS)
    m, p = _totals(s, c, w, 1.0)
    s.close()
    w32 = np.array(w, np.float32).astype(np.float64)
    defect_m = abs(w32.sum() - 1.0)
    defect_p = abs(3.0 * (w32 * np.array([v[0] ** 2 for v in c])).sum() - 1.0)
    assert abs(m / m0 - 1.0) <= STEPS * (defect_m / tau + 2.0 ** -26)
    assert abs(p / p0 - 1.0) <= STEPS * (defect_p / tau + 2.0 ** -26)


@pytest.mark.parametrize("tau", [0.55, 0.7, 0.8])
def test_fp64_mass_stays(tau):
    """FP64 stores full values.  Errors without a common sign of at most four unit roundoffs per node and step add up
    to 2^-51 sqrt(steps / nodes) of the mass; eight times that is allowed beside the rounded weights' share."""
    n, steps = 64, 400
    s = _box(2, n, tau, "fp64")
    m0, _ = _totals(s, C2, W2, 0.0)
    s.step(steps)
    m, _ = _totals(s, C2, W2, 0.0)
    s.close()
    # the rounded weights' sum exceeds 1 by w_defect, exactly representable products of 1/9
    from fractions import Fraction
    defect = float(sum(Fraction(float(v)) for v in W2) - 1)
    assert abs(m / m0 - 1.0 - steps * defect / tau) <= 8 * 2.0 ** -51 * math.sqrt(steps / (n * n))
