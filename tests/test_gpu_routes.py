"""The step's routes against one another: blocks of any size walk the node list back and forth over every entry once,
one launch for all members of an ensemble evaluates what a single domain's monitors evaluate, and the
network's layers give the same results by rows and by implicit GEMM.  All comparisons are bitwise: each pair of routes
does the same arithmetic in the same order per node, partial sum or output."""
import numpy as np
import pytest

from paper_2502_12955_gb300 import inputs
from paper_2502_12955_gb300.lbm import Ensemble, LbmError, Solver

pytestmark = pytest.mark.gpu


def _solver(cfg, geom, fields):
    s = Solver(cfg)
    s.set_geometry(geom)
    rho, u, C = fields
    s.set_fields(rho, u, C if s.n_scal else None)
    return s


def _geometry(nfluid, seed):
    """An 8 x 8 x 5 box with nfluid fluid nodes; 0: a box of 129 k fluid nodes, more than one wave of blocks."""
    if nfluid == 0:
        return inputs.random_solids((40, 64, 72), 0.3, seed=seed, reactive_fraction=0.5)
    g = np.full(5 * 8 * 8, inputs.REACTIVE, np.uint8)
    g[np.random.default_rng(seed).permutation(g.size)[:nfluid]] = 0
    return g.reshape(5, 8, 8)


# one node, around a block of 256, a whole box, more than one wave
@pytest.mark.parametrize("nfluid", [1, 255, 256, 257, 320, 0])
@pytest.mark.parametrize("kind,precision", [("flow", "fp32"), ("flow", "fp16"), ("flow", "fp64"), ("droplet", "fp32")])
def test_walk_covers_the_list_at_any_block_size(nfluid, kind, precision):
    geom = _geometry(nfluid, 3)
    nz, ny, nx = geom.shape
    if kind == "flow":
        cfg, _, _ = inputs.dissolution_3d(shape=geom.shape, g=1e-4, radius=(2.0, 3.0), seed=1)
        cfg = dict(cfg, geo_mode="none", precision=precision)
        fields = inputs.perturbed_fields(geom.shape, 1, 1, seed=5)
    else:
        cfg = dict(dim=3, nx=nx, ny=ny, nz=nz, n_comp=2, tau=[1.0, 1.0], G=[[0.0, 2.7], [2.7, 0.0]], psi_kind="identity",
                   periodic=[1, 1, 1], precision=precision)
        fields = inputs.perturbed_fields(geom.shape, 2, 0, seed=5, rho0=[1.0, 0.05])
    a = _solver(dict(cfg, block_x=256), geom, fields)
    others = [_solver(dict(cfg, block_x=b), geom, fields) for b in (0, 64, 128)]
    for n in (1, 1, 9):   # an even step, an odd step, a graph of eight and one more
        a.step(n)
        fa, ha = a.pops()
        assert np.isfinite(fa).all()
        for s in others:
            s.step(n)
            f, h = s.pops()
            assert np.array_equal(fa, f)
            assert ha is None or np.array_equal(ha, h)


@pytest.mark.parametrize("precision", ["fp32", "fp16", "fp64"])
@pytest.mark.parametrize("intervals", [(20, 20, 20, 20), (20, 10, 20, 20)])   # together, one by one
def test_ensemble_evaluates_as_single_domains(precision, intervals):
    mem = []
    for k, shape in enumerate([(4, 4, 4), (9, 10, 13), (16, 16, 16), (24, 20, 40)]):   # one block of partial sums to 19
        cfg, geom, fields = inputs.dissolution_3d(shape=shape, g=1e-4 * (1 + k), radius=(1.0, 2.0), seed=k)
        mem.append((dict(cfg, geo_mode="none", precision=precision, N_mon=intervals[k]), geom, fields))
    ens = Ensemble([c for c, _, _ in mem])
    singles = []
    for (cfg, geom, fields), m in zip(mem, ens.members):
        m.set_geometry(geom)
        m.set_fields(*fields)
        singles.append(_solver(cfg, geom, fields))
    ens.step(41)
    for s, m in zip(singles, ens.members):
        s.step(41)
        got, want = m.monitors(), s.monitors()
        assert want["residual"] > 0.0
        assert got["residual"] == want["residual"]
        for key in ("step", "mass0", "species0", "nfluid", "nsolid", "nonfinite"):
            assert got[key] == want[key], key
    ens.close()


def test_network_layers_by_rows_and_by_implicit_gemm(monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2502_12955_gb300 import surrogate as sg

    width, shape = (16, 16, 32), (16, 16, 32)
    V = shape[0] * shape[1] * shape[2]
    g = torch.Generator().manual_seed(7)
    x = torch.randn((V, 4), generator=g).to(torch.bfloat16).cuda()
    t = torch.randn((V, 4), generator=g).cuda()
    fluid = (torch.rand(V, generator=g) > 0.4).to(torch.uint8).cuda()
    nets = [sg.WarmStartNet(width=width, c_in=4, seed=2)]
    monkeypatch.setattr(sg, "lbm_nn_conv3_fits", lambda *a: 0)
    nets.append(sg.WarmStartNet(width=width, c_in=4, seed=2))
    assert not any(nets[0].rows.values()) and all(nets[1].rows.values())
    ys = [n.forward(x, shape) for n in nets]
    assert torch.equal(ys[0], ys[1])
    for n, y in zip(nets, ys):
        _, dy = n.loss_and_grad(y, t, fluid, int(fluid.sum()))
        n.backward(dy)
        n.check()
    for k in nets[0].g:
        if k.endswith(".w") and k != "head.w":
            assert torch.equal(nets[0].g[k], nets[1].g[k]), k
    # an input of 12 channels goes by rows; a number of voxels that is no multiple of 128 is refused by both
    monkeypatch.undo()
    wide = sg.WarmStartNet(width=width, c_in=12, seed=2)
    assert wide.rows["enc0a"] and not wide.rows["enc0b"]
    wide.forward(torch.zeros((V, 12), dtype=torch.bfloat16, device="cuda"), shape)
    wide.check()
    for n, c in ((nets[0], 4), (wide, 12)):
        with pytest.raises(LbmError):
            n.forward(torch.zeros((64, c), dtype=torch.bfloat16, device="cuda"), (4, 4, 4))
