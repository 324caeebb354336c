"""The library's own choice of forms on both sides of its size rules: the
flows are those of every other form bit for bit, and a change of algorithm,
which changes the edge kernel's form and its partials, leaves an objective
that is the residual pass's."""

import numpy as np
import pytest

from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pdr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr as _pdr

    build.build()
    _pdr.load()
    return _pdr


# sides of grids whose edges take one round of a part of the ring's warps, of most of them (the plain form and
# gathers up to 512 values, gathers beyond), and two rounds
@pytest.mark.parametrize("a,K", [(28, 500), (30, 500), (32, 500), (35, 512), (38, 500), (28, 640), (30, 640), (31, 449)])
def test_default_forms_around_a_crowded_ring(pdr, a, K):
    rng = np.random.default_rng([a, K])
    inst = I.make_instance(f"grid{a}_k{K}", I.grid_graph(a), K, ("lognormal", 1.0, 0.5), 1.2, rng)
    opts = dict(eps_obj=0.0, resid_tol=0.0, max_sweeps=21)
    flows = []
    for kw in (dict(), dict(excess_variant=0), dict(excess_variant=2), dict(use_graph=0)):
        with pdr.Solver.from_instance(inst, **kw, **opts) as s:
            s.solve()
            flows.append(s.flows())
            if not kw:
                for algo in (pdr.ALGO_AGD, pdr.ALGO_ESO, pdr.ALGO_CK, pdr.ALGO_GDM, pdr.ALGO_ESO):
                    s.set_options(algo=algo)
                    np.testing.assert_allclose(s.objective(), s.residuals()["z"], rtol=1e-5)
                s.reset()
                s.solve()
                flows.append(s.flows())
    for f in flows[1:]:
        np.testing.assert_array_equal(f, flows[0])


@pytest.mark.parametrize("a,K", [(7, 600), (15, 600), (20, 600), (25, 130), (22, 130), (15, 1100)])
@pytest.mark.parametrize("algo", [1, 2])
def test_fp64_gradient_steps_with_and_without_early_launches(pdr, algo, a, K):
    """The captured loop on both sides of the FP64 rule against plain launches from the host."""
    rng = np.random.default_rng([a, K])
    inst = I.make_instance(f"grid{a}_k{K}", I.grid_graph(a), K, ("uniform_int", 1, 9), 1.2, rng)
    got = []
    for use_graph in (1, 0):
        with pdr.Solver.from_instance(inst, precision=pdr.PREC_FP64, algo=algo, use_graph=use_graph, eps_obj=0.0,
                                      resid_tol=0.0, max_sweeps=23) as s:
            s.solve()
            got.append(s.flows())
    np.testing.assert_array_equal(got[0], got[1])
