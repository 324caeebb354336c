"""Reverse mode at the row lengths where the backward edge step changes its form
(1 to 8 vectors per lane of a warp, then blocks): the longest row of a form and
the shortest of the next, and a short last segment.  Against the oracle's reverse
mode, FP64 to 1e-9, FP32 to 1e-4 element by element (test_gpu_adjoint.py)."""

import numpy as np
import pytest

import oracle
from test_gpu_adjoint import elementwise_close, jittered, pdr  # noqa: F401
from paper_2108_07549_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo", ["eso", "ck"])
@pytest.mark.parametrize("lanes", [1, 32, 33, 64, 65, 96, 97, 128, 129, 160, 161, 192, 193, 256, 257])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_rows_at_the_ends_of_every_form(pdr, prec, lanes, algo):  # noqa: F811
    K = lanes * (2 if prec == "fp64" else 4) - 1  # ragged: padded to `lanes` vectors (FP64: an even number of them)
    rng = np.random.default_rng(31)
    inst = jittered(I.make_instance("dg", I.random_digraph(40, 3, rng), K, ("lognormal", 1.0, 0.5), 0.9, rng), lanes)
    ref = oracle.Problem.from_instance(inst)
    Lr, gur, gdr = ref.adjoint_eso(7) if algo == "eso" else ref.adjoint_ck(7)
    with pdr.Solver.from_instance(inst, precision=pdr.PREC_FP64 if prec == "fp64" else pdr.PREC_FP32,
                                  algo=pdr.ALGO_ESO if algo == "eso" else pdr.ALGO_CK) as s:
        L, gu, gd = s.backward(7, 3)
    if prec == "fp64":
        assert abs(L - Lr) <= 1e-12 * Lr
        np.testing.assert_allclose(gd, gdr, rtol=1e-9, atol=1e-12 * np.abs(gdr).max())
        np.testing.assert_allclose(gu, gur, rtol=1e-9, atol=1e-12 * max(1.0, np.abs(gur).max()))
    else:
        assert abs(L - Lr) <= 1e-5 * Lr
        worst = elementwise_close(np.concatenate([gu, gd]), np.concatenate([gur, gdr]))
        assert worst <= 1.0, worst
