"""FP64 edge QPs with several shares of a row per lane (edge_shares: 4, 2 or 1
by the number of edges), rows at both ends of every lane-group variant, edges
that leave a last warp partly empty.  The flows equal, bit for bit, the
persistent engine's, whose groups run on all their lanes; z agrees to the
rounding of an FP64 sum of at most 1e5 non-negative terms."""

import numpy as np
import pytest

from test_gpu_edge_ring import digraph, pdr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,out", [(7, 1), (611, 1), (401, 3), (1217, 2), (3001, 3), (8111, 3)])
@pytest.mark.parametrize("K", [3, 8, 9, 16, 17, 32, 33, 64, 65, 100, 128, 129, 256, 257, 510])
def test_flows_equal_the_persistent_engine(pdr, n, out, K):  # noqa: F811
    inst = digraph(n, out, K)
    got = []
    for engine in (2, 1):
        with pdr.Solver.from_instance(inst, use_graph=engine, precision=pdr.PREC_FP64, eps_obj=0.0, resid_tol=0.0,
                                      max_sweeps=7) as s:
            r = s.solve()
            got.append((r["sweeps"], r["z"], s.flows()))
    assert got[0][0] == got[1][0] == 7
    assert abs(got[0][1] - got[1][1]) <= 1e5 * 2.0**-53 * abs(got[0][1])
    np.testing.assert_array_equal(got[0][2], got[1][2])
