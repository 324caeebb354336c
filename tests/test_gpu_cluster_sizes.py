"""The cluster engine at the sizes where its work is split another way: fewer
vertices than blocks, one edge, vertices without edges, degrees around a
multiple of four (its row lists are padded to fours), rows at both ends of
every lane-group variant, stop rules at the first sweeps, a trace.  Its flows
equal the host loop's standalone kernels bit for bit; the objective trace
agrees to the pair sums' rounding (1e-12)."""

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


def ring(n, extra, K, seed):
    """A directed ring of n vertices and `extra` random arcs (parallel arcs and sinks of high degree among them),
    with isolated vertices at the end; some capacities 0."""
    rng = np.random.default_rng([seed, n, K])
    src = np.concatenate([np.arange(n), rng.integers(0, n, extra)])
    dst = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, max(1, n // 3), extra)])
    keep = src != dst
    row_ptr, col = I._csr(n + 2, src[keep], dst[keep])
    s = rng.integers(0, n, K)
    t = (s + rng.integers(1, n, K)) % n
    u = rng.uniform(0, 4, col.shape[0]) * (rng.random(col.shape[0]) < 0.7)
    return I.Instance(name="ring", n=n + 2, row_ptr=row_ptr, col=col, u=u, s=s.astype(np.int32), t=t.astype(np.int32),
                      d=rng.uniform(0.5, 3, K), factor=1.0, load=u, hops=np.ones(K, np.int64))


def run(pdr, inst, engine, **opts):
    with pdr.Solver.from_instance(inst, use_graph=engine, **opts) as s:
        r = s.solve()
        return r, s.flows(), s.trace() if opts.get("trace_len") else None, s.residuals()


@pytest.mark.parametrize("K", [1, 4, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 512])
@pytest.mark.parametrize("n,extra", [(2, 0), (3, 2), (7, 40), (40, 90)])
@pytest.mark.parametrize("algo", [0, 3])
def test_flows_equal_the_host_loop(pdr, n, extra, K, algo):
    inst = ring(n, extra, K, 5)
    opts = dict(algo=algo, eps_obj=0.0, resid_tol=0.0, max_sweeps=43)
    a, fa, _, ra = run(pdr, inst, 0, **opts)
    b, fb, _, rb = run(pdr, inst, 1, **opts)
    assert a["sweeps"] == b["sweeps"] == 43 and a["stop_reason"] == b["stop_reason"]
    np.testing.assert_array_equal(fa, fb)
    assert ra["z"] == rb["z"] and ra["cap_rel"] == rb["cap_rel"] and ra["cons_rel"] == rb["cons_rel"]


@pytest.mark.parametrize("rules", [dict(max_sweeps=0), dict(max_sweeps=1), dict(max_sweeps=2),
                                   dict(eps_obj=1e9, max_sweeps=50), dict(resid_tol=1e9, max_sweeps=50),
                                   dict(eps_rel=0.02, max_sweeps=400), dict(eps_obj=1e-3, max_sweeps=20000),
                                   dict(resid_tol=0.2, max_sweeps=20000)])
def test_stop_rules_fire_at_the_same_sweep(pdr, rules):
    inst = I.grid5_k10(1.3)
    opts = {**dict(eps_obj=0.0, resid_tol=0.0), **rules}
    for trace_len in (0, 30000):  # a traced sweep takes the full decision, an untraced one the short one
        a, fa, ta, _ = run(pdr, inst, 0, trace_len=trace_len, **opts)
        b, fb, tb, _ = run(pdr, inst, 1, trace_len=trace_len, **opts)
        assert (a["sweeps"], a["stop_reason"]) == (b["sweeps"], b["stop_reason"])
        np.testing.assert_array_equal(fa, fb)
        if trace_len:
            np.testing.assert_allclose(tb, ta, rtol=1e-12, atol=0)
        assert a["dz"] == b["dz"] or abs(a["dz"] - b["dz"]) <= 1e-12 * max(1.0, a["z"])  # -inf at the first sweep


def test_tail_mode_hands_over_at_the_same_sweep(pdr):
    inst = I.grid5_k10(1.3)
    opts = dict(precision=pdr.PREC_FP32_FP64TAIL, eps_obj=0.0, resid_tol=1e-6, max_sweeps=40000)
    a, fa, _, _ = run(pdr, inst, 0, **opts)
    b, fb, _, _ = run(pdr, inst, 1, **opts)
    assert a["verdict"] == b["verdict"] and a["stop_reason_fp32"] == b["stop_reason_fp32"]
    assert abs(a["sweeps"] - b["sweeps"]) <= 2 and abs(a["sweeps_fp64"] - b["sweeps_fp64"]) <= 2
