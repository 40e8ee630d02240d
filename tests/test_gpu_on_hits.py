"""The O(N) hits drawn four at a time and the FP64 Metropolis test decided in FP32
where its error bound allows: visits whose hits are not a multiple of four, that
cross the 128-hit flush of the summed moves, and couplings and fields for which
the bound never decides (every test in FP64).  Each against the oracle: equal
accepted hits, fields within 1e-12 of their size (a visit rounds its sum of
moves once, the oracle once per accepted hit, 2^-53 each, at most 300 times; two
sweeps amplify little)."""
import numpy as np
import pytest

import oracle
from workloads import FP64_PLAIN, HOT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nhit,kappa,lam,delta,scale", [
    (4, 1, 0.3, 1.0, 0.8, 1.0), (1, 6, 0.2, 0.5, 1.5, 1.0), (3, 131, 0.3, 1.0, 0.8, 1.0), (2, 300, 0.25, 2.0, 0.5, 1.0),
    (4, 7, 0.3, 1e6, 1e-3, 1.0),     # a stiff constraint: the bound is loose
    (2, 5, -0.3, -1e-9, 0.8, 1.0),   # signs turned
    (4, 9, 0.3, 0.0, 1e45, 1e45),    # beyond FP32: every test in FP64
    (4, 9, 0.3, 0.0, 1e-36, (1e-36, 1e36)),  # even and odd sites: steps that FP32 cannot hold
])
def test_fp64_hits(N, nhit, kappa, lam, delta, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1310_7087_gb300 import build
    build.build()
    import paper_1310_7087_gb300 as q
    oracle.build()
    m = q.ONModel(N, 4, 6, kappa, lam, delta, FP64_PLAIN, HOT, 9, nhit=nhit)
    o = oracle.OracleON(N, 4, 6, kappa, lam, delta, nhit)
    s = np.arange(4 ** 3 * 6)
    odd = (s + s // 4 + s // 16 + s // 64) & 1
    size = np.take(np.broadcast_to(scale, 2), odd)[:, None]
    start = m.get_field() * size
    m.set_field(start)
    o.set_field(start)
    m.sweep(2, 9)
    o.sweep(2, 9)
    a, b = m.get_field(), o.get_field()
    assert m.accepted == o.accepted
    for p in (0, 1):
        w = odd == p
        assert np.abs(a - b)[w].max() <= 1e-12 * max(size[w].max(), np.abs(b[w]).max())
    m.close()
    o.close()
