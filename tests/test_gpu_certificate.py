"""The certificate's potentials are one fixed vector: every difference the
residual pass forms is that of the same rounded heights, so sums of differences
along a path telescope and a margin above 0 is a proof.  A product fused into
the subtraction would let a height enter with two roundings, and a path of
exactly the demand's capacity would then seem too short for it.

Three vertices s -> a -> t of degree 5 and one commodity, u = d on both edges,
so the instance is feasible and the margin d (h_s - h_t) - u (h_s - h_a) -
u (h_a - h_t) is 0 exactly.  Flows from a fourth vertex set the imbalances to
1 + j 2^-52, for which the heights lie a few ulps apart and are all rounded up
("up") or all rounded down.  All other edges have no capacity."""

from fractions import Fraction

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


def imbalances(up):
    """Three j with falling heights (1 + j 2^-52) / 5, each rounded the given way."""
    w = 1.0 / 5.0
    found = []
    for j in range(64):
        delta = 1.0 + j * 2.0**-52
        exact, h = Fraction(delta) * Fraction(w), delta * w
        if (Fraction(h) < exact) if up else (Fraction(h) > exact):
            found.append((h, j))
    (_, jt), (_, ja), (_, js) = found[0], found[len(found) // 2], found[-1]
    return js, ja, jt


@pytest.mark.parametrize("up", [True, False])
def test_a_feasible_path_is_not_refuted(pdr, up):
    s, a, t, v = 0, 1, 2, 3
    js, ja, jt = imbalances(up)
    d = 0.5
    arcs = [(s, a, d, 0.0), (a, t, d, 0.0)]  # tail, head, capacity, flow
    # what each imbalance takes beyond the demand, as two FP32 values, and zeros up to degree 5
    for vertex, whole, j, more in ((s, 1.0 - d, js, 2), (a, 1.0, ja, 1), (t, 1.0 + d, jt, 2)):
        arcs += [(v, vertex, 0.0, whole), (v, vertex, 0.0, j * 2.0**-52)] + [(v, vertex, 0.0, 0.0)] * more
    arcs.sort(key=lambda x: x[0])
    row_ptr, col = I._csr(4, np.array([x[0] for x in arcs]), np.array([x[1] for x in arcs]))
    u = np.array([x[2] for x in arcs])
    f = np.array([[x[3]] for x in arcs])
    with pdr.Solver(4, row_ptr, col, u, [s], [t], [d], precision=pdr.PREC_FP32) as solver:
        solver.set_flows(f)
        np.testing.assert_array_equal(solver.flows(), f)
        r = solver.residuals()
    h = [(1.0 + j * 2.0**-52) * (1.0 / 5.0) for j in (js, ja, jt)]
    assert h[0] > h[1] > h[2]
    assert r["margin"] == 0.0 and r["margin_scale"] == 2.0 * d * (h[0] - h[2])
    assert r["verdict"] != pdr.VERDICT_INFEASIBLE
