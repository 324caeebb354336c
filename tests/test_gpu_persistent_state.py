"""After a solve on the persistent engine the congestion partials are those of
the returned flows, in whichever buffer they lie: the objective is the residual
pass's, and a second solve goes on as the graph's does."""

import numpy as np
import pytest

from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sweeps", [1, 4, 5])
@pytest.mark.parametrize("precision", [0, 1])
def test_objective_after_a_persistent_solve(precision, sweeps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr

    build.build()
    rng = np.random.default_rng(8)
    inst = I.make_instance("dg60_k40", I.random_digraph(60, 3, rng), 40, ("uniform_int", 1, 9), 1.2, rng)
    opts = dict(precision=precision, eps_obj=0.0, resid_tol=0.0, max_sweeps=sweeps, trace_len=10)
    got = []
    for use_graph, form in ((2, -1), (1, 0)):
        with pdr.Solver.from_instance(inst, use_graph=use_graph, excess_variant=form, **opts) as s:
            r = s.solve()
            assert s.debug_engine(precision)[0] == use_graph
            z = s.objective()
            np.testing.assert_allclose(z, r["z"], rtol=1e-5 if precision == 0 else 1e-12)
            s.solve()
            got.append((s.flows(), s.trace()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=1e-6 if precision == 0 else 1e-12)
