"""pdr_set_data from device arrays: the checks and the mean positive capacity,
formed by one block in the order the host path uses."""

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


@pytest.mark.parametrize("m_side", [2, 40])
def test_device_set_data_scales_as_the_host_path(pdr, m_side):
    """Fewer edges than the check kernel has threads, and more: the residuals
    (whose cap_rel the mean capacity scales) equal the host path's, and a bad
    last entry is found."""
    import torch

    rng = np.random.default_rng(m_side)
    K = 2 if m_side == 2 else 1500
    inst = I.make_instance("d", I.grid_graph(m_side), K, ("uniform_int", 1, 9), 0.7, rng)
    u, d = rng.uniform(0, 3, inst.m) * (rng.random(inst.m) < 0.6), rng.uniform(1, 2, K)
    with pdr.Solver.from_instance(inst) as s:
        s.sweeps(5)
        s.set_data(u=u, d=d)
        want = s.residuals()
        s.set_data(u=inst.u, d=inst.d)
        tu, td = torch.from_numpy(u).cuda(), torch.from_numpy(d).cuda()
        s.set_data_device(tu.data_ptr(), td.data_ptr())
        got = s.residuals()
        assert {k: got[k] for k in ("z", "cap_rel", "cons_rel", "margin")} == {
            k: want[k] for k in ("z", "cap_rel", "cons_rel", "margin")}
        for bad in (0, 1):
            bu, bd = tu.clone(), td.clone()
            (bd if bad else bu)[-1] = float("nan")
            with pytest.raises(pdr.PdrError) as e:
                s.set_data_device(bu.data_ptr(), bd.data_ptr())
            assert e.value.status == pdr.ERR_INVALID_ARG


@pytest.mark.parametrize("x", [0.0, -0.0, 5e-324, 1e308, -5e-324, -1.0, float("inf"), -float("inf"), float("nan")])
def test_device_set_data_domain(pdr, x):
    """A capacity is finite and not below 0 (-0 included), a demand finite and above 0."""
    import torch

    inst = I.grid5_k10(1.0)
    with pdr.Solver.from_instance(inst) as s:
        for u_side in (True, False):
            u, d = torch.from_numpy(inst.u.copy()).cuda(), torch.from_numpy(inst.d.copy()).cuda()
            (u if u_side else d)[3] = x
            if np.isfinite(x) and (x >= 0 if u_side else x > 0):
                s.set_data_device(u.data_ptr(), d.data_ptr())
            else:
                with pytest.raises(pdr.PdrError) as e:
                    s.set_data_device(u.data_ptr(), d.data_ptr())
                assert e.value.status == pdr.ERR_INVALID_ARG
