"""A batch of more instances than a grid has rows (65,535): the residual pass
takes the instance as the grid's second index and runs in slices."""

from types import SimpleNamespace

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_more_instances_than_grid_rows():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr

    build.build()
    count = 65535 + 2
    row_ptr, col = np.array([0, 1, 1], np.int64), np.array([1], np.int32)
    s, t = np.array([0], np.int32), np.array([1], np.int32)
    # one edge and one commodity of demand 1; every third edge holds half of it
    insts = [SimpleNamespace(n=2, row_ptr=row_ptr, col=col, u=np.array([0.5 if i % 3 == 0 else 2.0]), s=s, t=t,
                             d=np.array([1.0])) for i in range(count)]
    with pdr.Batch(insts, eps_obj=0.0, resid_tol=0.0, max_sweeps=2) as B:
        res = B.solve()
    # f = 1/3, then 5/9 or beyond u: every instance of a kind as the first of it
    for i in (0, 1):
        with pdr.Solver.from_instance(insts[i], eps_obj=0.0, resid_tol=0.0, max_sweeps=2) as one:
            want = one.solve()
        for k in range(i, count, 3):
            assert res[k]["z"] == want["z"] and res[k]["cons_abs"] == want["cons_abs"], k
            assert res[k]["sweeps"] == 2
