"""The cluster engine against the captured loop of standalone kernels, and the
way out where a device refuses its launch."""

import numpy as np
import pytest

from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu

HOST, GRAPH, CLUSTER = 0, 1, 3
FREE = dict(eps_obj=0.0, resid_tol=0.0)


@pytest.fixture(scope="module")
def pdr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr as _pdr

    build.build()
    _pdr.load()
    return _pdr


def digraph(n, K, seed):
    rng = np.random.default_rng([seed, n, K])
    return I.make_instance(f"dg{n}_{K}", I.random_digraph(n, 3, rng), K, ("uniform_int", 1, 9), 1.2, rng)


# ------------------------------------------------------------------ a refused launch


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("use_graph", [1, 3])
def test_a_refused_launch_falls_back_to_the_graph(pdr, use_graph, precision):
    inst = I.grid5_k10(1.3)
    opts = dict(precision=precision, use_graph=use_graph, eps_obj=0.0, resid_tol=1e-4, max_sweeps=3000)
    with pdr.Solver.from_instance(inst, **opts) as s:
        want = s.solve()
        f = s.flows()
        assert s.debug_engine() == (CLUSTER, 1)
    with pdr.Solver.from_instance(inst, **opts) as s:
        pdr.load().pdr_debug_fail_cluster(1)
        try:
            for _ in range(2):  # the second solve does not try again
                s.reset()
                r = s.solve()
                assert s.debug_engine() == (GRAPH, 0)
                assert (r["sweeps"], r["stop_reason"], r["verdict"]) == (want["sweeps"], want["stop_reason"],
                                                                        want["verdict"])
                np.testing.assert_array_equal(s.flows(), f)
        finally:
            pdr.load().pdr_debug_fail_cluster(0)


def test_a_refused_launch_in_a_batch(pdr):
    """Two launch groups (one and several blocks), either refused: its instances go with the larger ones."""
    group = [I.grid5_k10(1.3), digraph(150, 60, 1), I.grid5_k10(0.6), digraph(160, 60, 2)]
    opts = dict(FREE, max_sweeps=75)
    with pdr.Batch(group, **opts) as B:
        want = B.solve()
        flows = [B.solver(i).flows() for i in range(4)]
        kinds = [B.solver(i).debug_engine() for i in range(4)]
    assert all(k[0] == CLUSTER for k in kinds) and kinds[0][1] != kinds[1][1]
    for nth in (1, 2):
        with pdr.Batch(group, **opts) as B:
            pdr.load().pdr_debug_fail_cluster(nth)
            try:
                for _ in range(2):
                    B.reset()
                    res = B.solve()
                    engines = [B.solver(i).debug_engine()[0] for i in range(4)]
                    assert sorted(set(engines)) == [GRAPH, CLUSTER]
                    for i in range(4):
                        assert res[i]["sweeps"] == want[i]["sweeps"] == 75
                        np.testing.assert_array_equal(B.solver(i).flows(), flows[i])
            finally:
                pdr.load().pdr_debug_fail_cluster(0)


def test_a_refusal_in_mid_solve_is_an_error(pdr):
    with pdr.Solver.from_instance(I.grid5_k10(1.3), max_sweeps=8192 + 10, **FREE) as s:
        pdr.load().pdr_debug_fail_cluster(2)
        try:
            with pytest.raises(pdr.PdrError) as e:
                s.solve()
            assert e.value.status == pdr.ERR_CUDA
        finally:
            pdr.load().pdr_debug_fail_cluster(0)
        s.reset()
        assert s.solve()["sweeps"] == 8192 + 10 and s.debug_engine() == (CLUSTER, 1)


# ------------------------------------------------------------------ the objective's sum


def test_blocks_sums_are_added_in_64_bits(pdr):
    """An objective whose terms are powers of two over 51 binary places, the largest and the smallest in different
    blocks: a 64-bit sum of the blocks' pairs is exact.  Vertices of a ring with two arcs out and two in, no
    capacity: a flow f on one arc adds f^2 as congestion and 4 (f/4)^2 at each of its ends."""
    n, K = 256, 32
    tail = np.repeat(np.arange(n), 2)
    row_ptr, col = I._csr(n, tail, (tail + np.tile([1, 2], n)) % n)
    f = np.zeros((2 * n, K))
    for vertex, k, x in ((0, 0, 1.0), (2, 1, 2.0**-12), (250, 2, 2.0**-25)):
        f[2 * vertex, k] = x
    s, t = np.full(K, 100), np.full(K, 150)
    d = np.full(K, 2.0**-60)  # squares far below the last place
    for use_graph, engine in ((0, HOST), (1, CLUSTER)):
        with pdr.Solver(n, row_ptr, col, np.zeros(2 * n), s, t, d, use_graph=use_graph, max_sweeps=1, trace_len=2,
                        **FREE) as solver:
            solver.set_flows(f)
            solver.solve()
            assert solver.debug_engine()[0] == engine and (engine == HOST or solver.debug_engine()[1] > 1)
            assert solver.trace()[0] == 0.75 * (1.0 + 2.0**-24 + 2.0**-50)
