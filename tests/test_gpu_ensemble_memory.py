"""An ensemble gives back all device memory that stepping and evaluating it has taken."""
import numpy as np
import pytest

from paper_2502_12955_gb300.lbm import Ensemble

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_create_step_close_keeps_free_memory():
    # 400 blocks of partial sums: 4.8 KB of work list for the evaluation.  The driver hands out device memory in
    # chunks of 2 MB, so a list left behind by each of 600 ensembles costs more than one chunk
    n = 640
    cfg = dict(dim=2, nx=n, ny=n, nz=1, n_comp=1, tau=[0.8], n_scal=0, periodic=[1, 1, 1], precision="fp32", N_mon=2)
    geom = np.zeros((1, n, n), np.uint8)
    rho, u = np.ones((1, 1, n, n)), np.zeros((3, 1, n, n))

    def cycle():
        e = Ensemble([cfg])
        e.members[0].set_geometry(geom)
        e.members[0].set_fields(rho, u, None)
        e.step(2)
        e.close()

    for _ in range(5):
        cycle()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(600):
        cycle()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free - (1 << 21)
