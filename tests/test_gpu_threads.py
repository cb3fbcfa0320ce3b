"""Contexts of different block sizes stepped from several host threads at once, each on its own stream, give what they
give alone: launch shapes are kept per block size and shared safely."""
import threading

import numpy as np
import pytest

from paper_2502_12955_gb300 import inputs
from paper_2502_12955_gb300.lbm import Solver

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _solver(block_x, stream=None):
    cfg, geom, fields = inputs.dissolution_3d(shape=(24, 40, 32), g=1e-4, radius=(2.0, 4.0), seed=3)
    s = Solver(dict(cfg, geo_mode="none", precision="fp32", block_x=block_x), stream=stream)
    s.set_geometry(geom)
    s.set_fields(*fields)
    return s


def test_threads_with_different_block_sizes():
    blocks = [64, 256, 96, 128]
    want = []
    for b in blocks:
        s = _solver(b)
        s.step(45)
        want.append(s.pops()[0])
        s.close()
    streams = [torch.cuda.Stream() for _ in blocks]
    solvers = [_solver(b, st.cuda_stream) for b, st in zip(blocks, streams)]
    errors = []

    def run(s):
        try:
            for _ in range(45):   # single steps: every launch looks its shape up
                s.step(1)
            s.sync()
        except Exception as e:   # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=(s,)) for s in solvers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for s, w in zip(solvers, want):
        assert np.array_equal(s.pops()[0], w)
        s.close()
