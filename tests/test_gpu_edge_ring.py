"""The edge QP's ring form (32-lane variants with about as many edges as resident
warps, or more): fewer and more edges than warps, an uneven last round, rows
at both ends of every variant.  Its flows equal, bit for bit, the persistent
engine's, whose warps load their rows directly."""

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


def digraph(n, out, K, seed=3):
    rng = np.random.default_rng([seed, n, K])
    src = np.repeat(np.arange(n), out)
    row_ptr, col = I._csr(n, src, (src + rng.integers(1, n, n * out)) % n)
    s = rng.integers(0, n, K)
    u = rng.uniform(0, 6, n * out) * (rng.random(n * out) < 0.5)
    return I.Instance(name="dg", n=n, row_ptr=row_ptr, col=col, u=u, s=s.astype(np.int32),
                      t=((s + rng.integers(1, n, K)) % n).astype(np.int32), d=rng.uniform(0.5, 3, K), factor=1.0, load=u,
                      hops=np.ones(K, np.int64))


@pytest.mark.parametrize("n,out", [(700, 3), (3001, 3), (4100, 5)])
@pytest.mark.parametrize("K", [65, 100, 128, 129, 256, 257, 510, 512, 513, 1000, 1024])
def test_flows_equal_the_persistent_engine(pdr, n, out, K):
    inst = digraph(n, out, K)
    got = []
    for engine in (2, 0, 1):
        with pdr.Solver.from_instance(inst, use_graph=engine, excess_variant=2, eps_obj=0.0, resid_tol=0.0,
                                      max_sweeps=7) as s:
            r = s.solve()
            got.append((r["sweeps"], r["z"], s.flows()))
    for sweeps, z, f in got[1:]:
        assert sweeps == got[0][0] == 7 and z == got[0][1]
        np.testing.assert_array_equal(f, got[0][2])
