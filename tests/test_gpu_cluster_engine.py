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


# ------------------------------------------------------------------ against the captured loop


def parallel(n, extra, K, seed):
    """n vertices with `extra` arcs among them (many parallel): fewer vertices than a cluster has blocks."""
    rng = np.random.default_rng([seed, n, K])
    src = np.concatenate([np.arange(n), rng.integers(0, n, extra)])
    dst = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, n, extra)])
    keep = src != dst
    row_ptr, col = I._csr(n, src[keep], dst[keep])
    s = rng.integers(0, n, K)
    t = (s + rng.integers(1, n, K)) % n
    u = rng.uniform(0, 4, col.shape[0]) * (rng.random(col.shape[0]) < 0.7) / 20
    return I.Instance(name=f"par{n}_{K}", n=n, row_ptr=row_ptr, col=col, u=u, s=s.astype(np.int32),
                      t=t.astype(np.int32), d=rng.uniform(0.5, 3, K), factor=1.0, load=u, hops=np.ones(K, np.int64))


CASES = {"grid5": (1, lambda: I.grid5_k10(1.3)), "tight": (1, lambda: I.grid5_k10(0.6)),
         "few3": (8, lambda: parallel(3, 1500, 32, 1)), "few6": (8, lambda: parallel(6, 1200, 61, 2)),
         "large": (8, lambda: digraph(400, 90, 3)), "wide": (8, lambda: digraph(60, 500, 4))}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("algo", [0, 3])
def test_flows_equal_the_graph_over_several_launches(pdr, algo, name):
    """Two whole launches of 8192 sweeps and an odd remainder, then a second solve from the returned flows."""
    blocks, make = CASES[name]
    inst = make()
    got = []
    for kw in (dict(use_graph=1), dict(use_graph=1, excess_variant=0)):
        with pdr.Solver.from_instance(inst, algo=algo, max_sweeps=2 * 8192 + 1, **kw, **FREE) as s:
            r1 = s.solve()
            f1 = s.flows()
            s.set_options(max_sweeps=8192 + 2)
            r2 = s.solve()
            got.append((r1, f1, r2, s.flows(), s.debug_engine()))
    a, b = got
    assert a[4] == (CLUSTER, blocks) and b[4] == (GRAPH, 0)
    assert a[0]["sweeps"] == b[0]["sweeps"] == 2 * 8192 + 1 and a[2]["sweeps"] == b[2]["sweeps"] == 8192 + 2
    np.testing.assert_array_equal(a[1], b[1])
    np.testing.assert_array_equal(a[3], b[3])
    for q in (0, 2):
        assert a[q]["z"] == b[q]["z"] and a[q]["cap_rel"] == b[q]["cap_rel"] and a[q]["cons_rel"] == b[q]["cons_rel"]
        assert abs(a[q]["dz"] - b[q]["dz"]) <= 1e-12 * max(1.0, a[q]["z"])


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("rules", [dict(eps_rel=1e-3), dict(resid_tol=0.5), dict(eps_rel=1e-6, trace_len=9000)])
def test_rules_fire_where_the_graph_s_do(pdr, rules, name):
    inst = CASES[name][1]()
    got = []
    for kw in (dict(use_graph=1), dict(use_graph=1, excess_variant=0)):
        with pdr.Solver.from_instance(inst, max_sweeps=9000, **dict(FREE, **rules), **kw) as s:
            r = s.solve()
            got.append((r["sweeps"], r["stop_reason"], s.flows(), s.trace() if "trace_len" in rules else np.ones(1)))
    assert got[0][:2] == got[1][:2]
    np.testing.assert_array_equal(got[0][2], got[1][2])
    np.testing.assert_allclose(got[0][3], got[1][3], rtol=1e-12)
