"""The monitors and the residual add a thread's nodes without loss: FP32 sums of nodes of very different size come out
exact (every value below is a power of two or an exact sum of a few, so the expected totals are exact in FP64)."""
import math

import numpy as np
import pytest

from paper_2502_12955_gb300.lbm import Ensemble, Solver

pytestmark = pytest.mark.gpu

N = 64   # 4096 nodes: several per thread
W2 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _solver(n_scal, make):
    cfg = dict(dim=2, nx=N, ny=N, nz=1, n_comp=1, tau=[1.0], n_scal=n_scal, tau_c=[1.0], J0=0.4, periodic=[1, 1, 1],
               precision="fp32", N_mon=0)
    s, owner = make(cfg)
    s.set_geometry(np.zeros((1, N, N), np.uint8))
    s.set_fields(np.ones((1, 1, N, N)), np.zeros((3, 1, N, N)), np.zeros((n_scal, 1, N, N)) if n_scal else None)
    return s, owner


def _single(cfg):
    return Solver(cfg), None


def _member(cfg):
    e = Ensemble([cfg])
    return e.members[0], e


def _mixed(seed):
    return np.random.default_rng(seed).random(N * N) < 0.5


@pytest.mark.parametrize("make", [_single, _member])
def test_mass_momentum_and_species_are_exact(make):
    s, owner = _solver(1, make)
    big = _mixed(1)
    v = np.where(big, 2.0 ** 24, 0.25)
    f = np.repeat(W2[:, None], N * N, 1)[None].copy()   # stored deviations 0
    f[0, 1] += v                                        # direction +x
    h = np.zeros((1, 5, N * N))
    h[0, 0] = v
    s.set_pops(f, h)
    m = s.monitors()
    total = math.fsum(v)
    assert m["momx"] == total and m["momy"] == 0.0
    assert m["mass0"] == total + N * N
    assert m["species0"] == total
    assert m["nonfinite"] == 0.0


def test_a_non_finite_node_stays_visible():
    s, _ = _solver(0, _single)
    f = np.repeat(W2[:, None], N * N, 1)[None].copy()
    f[0, 0, 7] = np.inf
    s.set_pops(f)
    m = s.monitors()
    assert m["nonfinite"] == 1.0 and m["mass0"] == np.inf


def test_the_residual_is_exact():
    s, _ = _solver(0, _single)
    big = _mixed(2)

    def state(u):   # rho = 1, velocity u along x
        f = np.repeat(W2[:, None], N * N, 1)[None].copy()
        f[0, 1] += 0.5 * u
        f[0, 3] -= 0.5 * u
        return f

    s.set_pops(state(np.where(big, 0.0, 2.0 ** -13)))
    assert s.residual() == -1.0
    s.set_pops(state(np.where(big, 1.0, 2.0 ** -13)))
    nb, ns = int(big.sum()), int((~big).sum())
    want = math.sqrt(nb / (nb + ns * 2.0 ** -26))   # the slow nodes are 2^-27 of it
    assert abs(s.residual() - want) <= 1e-14
