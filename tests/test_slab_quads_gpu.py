"""The slab kernels work column quads: boxes whose rows, walls and auxiliaries
do not fall on multiples of four, in both storage types, against the oracle.
Bounds: 1e-4 for FP32 traces, 1e-2 for FP16 storage (the storage mode's bar)."""
import numpy as np
import pytest

import oracle
from paper_1008_2602_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "odd_columns": W.random_problem(61, 37, 29, 23, upml=3, n_steps=60),
    "three_columns_over": W.random_problem(62, 75, 33, 21, upml=5, n_steps=50).replace(upml_kappa_max=5.0),
    "pmc_high_walls": W.random_problem(63, 42, 31, 22, upml=0, n_steps=60).replace(walls=(0, 1, 0, 1, 0, 1)),
    "mixed_depths": W.random_problem(64, 45, 36, 28, upml=4, n_steps=60).replace(upml_depth=(4, 0, 3, 5, 0, 6),
                                                                              walls=(0, 1, 0, 0, 1, 0)),
}


@pytest.mark.parametrize("precision,bound", [("fp32", 1e-4), ("fp16", 1e-2)])
@pytest.mark.parametrize("name", list(CASES))
def test_slab_boxes_against_the_oracle(name, precision, bound):
    import torch
    assert torch.cuda.is_available()
    from paper_1008_2602_gb300 import solver
    p = CASES[name]
    ref = oracle.run(p, n_threads=4)["trace"]
    s = solver.Solver(p, precision=precision)
    s.step_profiled(p.n_steps)
    tr = s.traces().astype(np.float64)
    s.close()
    err = np.linalg.norm(tr - ref) / np.linalg.norm(ref)
    assert err <= bound, err
