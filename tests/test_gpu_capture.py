"""A context on a stream that is being captured: pdr_reset refuses, as the
calls that wait for the stream do, and changes nothing."""

import numpy as np
import pytest

from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["solver", "batch"])
def test_reset_is_refused_under_capture(what):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_07549_gb300 import build, pdr

    build.build()
    inst = I.grid5_k10(1.3)
    stream = torch.cuda.Stream()
    opts = dict(stream=stream.cuda_stream, eps_obj=0.0, resid_tol=0.0, max_sweeps=30)
    owner = pdr.Solver.from_instance(inst, **opts) if what == "solver" else pdr.Batch([inst, inst], **opts)
    with owner:
        view = owner if what == "solver" else owner.solver(1)
        owner.solve()
        want = view.flows()
        x = torch.zeros(4, device="cuda")
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            x += 1.0
            with pytest.raises(pdr.PdrError) as e:
                owner.reset()
            assert e.value.status == pdr.ERR_CUDA
        graph.replay()
        torch.cuda.synchronize()
        assert x.tolist() == [1.0] * 4
        np.testing.assert_array_equal(view.flows(), want)
        owner.reset()
        assert not view.flows().any()
