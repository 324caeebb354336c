"""What a batch's solve leaves behind for the calls that follow it, and what
the captured loop of its larger instances does after options change."""

import numpy as np
import pytest

from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu

# excess_variant 0 keeps the instances off the cluster engine: they run in the batch's captured loop
LOOP = dict(excess_variant=0, edge_variant=3, eps_rel=0.0)


@pytest.fixture(scope="module")
def pdr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr as _pdr

    build.build()
    _pdr.load()
    return _pdr


def insts(count=3):
    out = []
    for b in range(count):
        rng = np.random.default_rng([41, b])
        out.append(I.make_instance(f"b{b}", I.random_digraph(60 + 30 * b, 3, rng), 40 + b, ("uniform_int", 1, 9), 1.2,
                                   rng))
    return out


@pytest.mark.parametrize("use_graph", [1, 0])
@pytest.mark.parametrize("precision", [0, 1])
def test_congestion_after_a_stop_is_that_of_the_returned_flows(pdr, precision, use_graph):
    """A solve that stops by a rule has run the edge QPs of the sweep that stopped; the objective and the next
    solve still start from the returned flows.  (An objective rule this wide fires at the second evaluation,
    where successive flows differ by tens of percent.)"""
    opts = dict(LOOP, precision=precision, use_graph=use_graph, eps_obj=1e30, resid_tol=0.0, max_sweeps=50,
                trace_len=60)
    group = insts()
    with pdr.Batch(group, **opts) as B:
        first = B.solve()
        views = [B.solver(i) for i in range(len(group))]
        z = [v.objective() for v in views]
        again = B.solve()
        traces = [v.trace() for v in views]
    for x, r, zx, r2, tr in zip(group, first, z, again, traces):
        assert r["stop_name"] == "objective" and r["sweeps"] == 1
        np.testing.assert_allclose(zx, r["z"], rtol=1e-5, err_msg=x.name)  # FP32 terms against the FP64 pass
        with pdr.Solver.from_instance(x, **opts) as s:
            s.solve()
            want = s.solve()
            np.testing.assert_allclose(tr, s.trace(), rtol=1e-12, err_msg=x.name)
        assert r2["sweeps"] == want["sweeps"]
        np.testing.assert_allclose(r2["z"], want["z"], rtol=1e-12)


@pytest.mark.parametrize("change", [dict(algo=3), dict(algo=1), dict(algo=2), dict(edge_variant=4),
                                    dict(excess_variant=2), dict(trace_len=40)])
def test_options_of_an_instance_reach_its_next_batch_solve(pdr, change):
    opts = dict(LOOP, eps_obj=0.0, resid_tol=0.0, max_sweeps=25)
    group = insts()
    with pdr.Batch(group, **opts) as B:
        B.solve()
        view = B.solver(1)
        view.set_options(**change)
        B.reset()
        B.solve()
        flows = [B.solver(i).flows() for i in range(len(group))]
        trace = view.trace() if "trace_len" in change else None
    for i, x in enumerate(group):
        with pdr.Solver.from_instance(x, **dict(opts, **(change if i == 1 else {}))) as s:
            s.solve()
            np.testing.assert_array_equal(flows[i], s.flows(), err_msg=x.name)
            if i == 1 and trace is not None:
                assert len(trace) == 26
                np.testing.assert_allclose(trace, s.trace(), rtol=1e-12)
