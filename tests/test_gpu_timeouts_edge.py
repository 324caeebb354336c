"""Time limits of the edge QP's shared-memory waits, and that a limit made
shorter than a copy takes leaves no copy behind.

pdr_debug_wait with hold_end makes the ring form's barriers want one arrival
more than a copy makes: every warp's wait runs out, its copies land, and the
call returns PDR_ERR_TIMEOUT.  With a limit of a thousand cycles ordinary
waits may run out too; a kernel that gives up still waits for the copies it
started.  Nothing faults, traps or hangs the GPU."""

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


def grid(a, K):
    rng = np.random.default_rng([a, K])
    return I.make_instance(f"grid{a}_k{K}", I.grid_graph(a), K, ("lognormal", 1.0, 0.5), 1.2, rng)


def start(inst):
    rng = np.random.default_rng(2)
    return rng.exponential(1.0, (inst.m, inst.K)) * (rng.random((inst.m, inst.K)) < 0.4)


@pytest.mark.parametrize("K", [129, 501])
def test_ring_wait_runs_out_and_the_context_recovers(pdr, K):
    inst = grid(30, K)
    f = start(inst)
    opts = dict(excess_variant=0, max_sweeps=100)  # gathers: no wait but the ring's
    with pdr.Solver.from_instance(inst, **opts) as s:
        s.set_flows(f)
        s.sweeps(3)
        want = s.flows()
        L = s.backward(3, 1)
    with pdr.Solver.from_instance(inst, **opts) as s:
        s.debug_wait(2_000_000, hold_end=True)
        s.set_flows(f)
        with pytest.raises(pdr.PdrError) as e:
            s.sweeps(1)
        assert e.value.status == pdr.ERR_TIMEOUT and "excess" not in str(e.value)
        for eng in (0, 1):
            s.set_options(use_graph=eng)
            with pytest.raises(pdr.PdrError) as e:
                s.solve()
            assert e.value.status == pdr.ERR_TIMEOUT
        with pytest.raises(pdr.PdrError) as e:
            s.backward(3, 1)
        assert e.value.status == pdr.ERR_TIMEOUT
        s.debug_wait(1 << 32, hold_end=False)
        s.set_flows(f)
        s.sweeps(3)
        np.testing.assert_array_equal(s.flows(), want)
        again = s.backward(3, 1)
        assert again[0] == L[0]
        np.testing.assert_array_equal(again[1], L[1])


@pytest.mark.parametrize("a,K,kw", [(30, 501, dict(excess_variant=0)), (30, 501, dict(excess_variant=1)),
                                    (30, 501, dict(excess_variant=2)), (30, 501, dict(excess_variant=5)),
                                    (10, 9000, dict(excess_variant=0, edge_variant=19)),
                                    (10, 9000, dict(excess_variant=3, edge_variant=20))])
def test_a_limit_shorter_than_a_copy(pdr, a, K, kw):
    inst = grid(a, K)
    f = start(inst)
    with pdr.Solver.from_instance(inst, **kw) as s:
        s.set_flows(f)
        s.sweeps(3)
        want = s.flows()
        s.debug_wait(1000)
        for _ in range(3):
            s.set_flows(f)
            try:
                s.sweeps(3)
            except pdr.PdrError as e:
                assert e.status == pdr.ERR_TIMEOUT
            else:
                np.testing.assert_array_equal(s.flows(), want)
        s.debug_wait()
        s.set_flows(f)
        s.sweeps(3)
        np.testing.assert_array_equal(s.flows(), want)
