"""The residual pass of FP32 flows and the widening read-out at the sizes
where their kernels take another branch.

The pass decides in FP32 which elements need FP64 (the largest imbalances and
the certificate lengths); ties and near-ties, rows shorter than a warp, padded
rows and all-zero rows are where a screen could drop the maximum.  The oracle
evaluates the same FP32-representable flows in FP64; the tolerance is the
parity tests' 1e-12 of the quantity (FP64 sums of at most a few thousand
terms, each exact to 2^-45).
"""

import ctypes

import numpy as np
import pytest

import oracle
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


def flows_of(kind, m, K, rng):
    f = rng.exponential(1.0, (m, K)) * (rng.random((m, K)) < 0.5)
    if kind == "ties":  # small integers: equal heights and equal differences everywhere
        f = rng.integers(0, 3, (m, K)).astype(np.float64)
    elif kind == "near":  # values one rounding apart
        f = 1.0 + rng.integers(0, 3, (m, K)) * 2.0**-23
    elif kind == "wide":  # forty orders of magnitude
        f = 10.0 ** rng.uniform(-30, 10, (m, K)) * (rng.random((m, K)) < 0.7)
    elif kind == "zero":
        f = np.zeros((m, K))
    return f.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("K", [1, 3, 4, 5, 127, 128, 129, 300])
@pytest.mark.parametrize("kind", ["random", "ties", "near", "wide", "zero"])
def test_residuals_equal_the_oracle(pdr, kind, K):
    rng = np.random.default_rng([K, 3])
    n = max(8, int(np.sqrt(K)) + 2)
    inst = I.make_instance("r", I.random_digraph(n, 3, rng), K, ("uniform_int", 1, 9), 0.8, rng)
    f = flows_of(kind, inst.m, K, rng)
    ref = oracle.Problem.from_instance(inst).residuals(f)
    with pdr.Solver.from_instance(inst, precision=pdr.PREC_FP32) as s:
        s.set_flows(f)
        got = s.residuals()
    for key in ("z", "cap_abs", "cap_rel", "cons_abs", "cons_rel", "f_min", "margin_scale"):
        assert abs(got[key] - ref[key]) <= 1e-12 * abs(ref[key]), (key, got[key], ref[key])
    assert abs(got["margin"] - ref["margin"]) <= 1e-12 * ref["margin_scale"]


@pytest.mark.parametrize("K", [1, 2, 4, 6, 7, 64, 129])
@pytest.mark.parametrize("shift", [0, 1])
def test_flows_into_device_memory_at_any_alignment(pdr, K, shift):
    """Rows with and without padding, 16-byte aligned or not: the FP32 values
    (a subnormal and a negative zero among them) widened bit for bit."""
    import torch

    rng = np.random.default_rng(K)
    inst = I.make_instance("w", I.grid_graph(5), K, ("uniform_int", 1, 9), 1.2, rng)
    f = flows_of("wide", inst.m, K, rng)
    f[0, 0], f[1, 0], f[2, 0] = 2.0**-140, -0.0, np.finfo(np.float32).max
    with pdr.Solver.from_instance(inst) as s:
        s.set_flows(f)
        buf = torch.full((inst.m * K + 2,), -7.0, dtype=torch.float64, device="cuda")
        s._check(s._lib.pdr_flows(s._h, ctypes.c_void_p(buf.data_ptr() + 8 * shift)))
        out = buf.cpu().numpy()
    np.testing.assert_array_equal(out[shift:shift + inst.m * K].reshape(inst.m, K).view(np.int64), f.view(np.int64))
    assert out[shift + inst.m * K] == -7.0 and (shift == 0 or out[0] == -7.0)
