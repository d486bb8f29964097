"""Boards past L2 fetch the slab boxes' next plane ahead: the same fields, bit
for bit, as the resident launches, which do not.  Both field sets of the boards
here hold more than 100 MB; rows whole and ragged, runs of one to four planes."""
import numpy as np
import pytest

from paper_1008_2602_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,depth", [(161, 131, 101, (5, 5, 5, 5, 5, 5)), (204, 172, 63, (8, 4, 6, 10, 0, 7))])
def test_prefetched_slabs_equal_the_resident_steps(nx, ny, nz, depth):
    import torch
    assert torch.cuda.is_available()
    from paper_1008_2602_gb300 import solver
    p = W.random_problem(81, nx, ny, nz, upml=5, n_steps=20).replace(upml_depth=depth)
    assert 48 * (nx + 1) * (ny + 1) * (nz + 1) > 100e6
    a, b = solver.Solver(p), solver.Solver(p)
    a.step(9)
    b.step_profiled(9)
    for c in range(6):
        assert np.array_equal(a.field(c), b.field(c)), c
    assert np.array_equal(a.traces(), b.traces()) and np.any(a.field(2))
    a.close()
    b.close()
