"""FP64 scans of more lattices than CTAs of the faster kernel are resident (each
lattice of a wave needs one): one wave of tiny lattices, tuned, and 512-thread CTAs."""
import numpy as np
import pytest

import oracle
from workloads import FP64_PLAIN, HOT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Ns,threads", [(1300, 2, 0), (2400, 2, 64), (200, 4, 512)])
def test_many_lattices(n, Ns, threads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_1310_7087_gb300 as q
    beta = np.linspace(2.2, 2.5, n)
    b = q.Batch([Ns] * n, [2] * n, list(beta), [i % 4 for i in range(n)], FP64_PLAIN, HOT, 5)
    if threads:
        q.qcd_batch_set_block(b.h, threads)
    start = {i: b.get_links(i) for i in (0, n // 2, n - 1)}
    got = b.sweep(1, 1, 5)
    for i, links in start.items():
        o = oracle.OracleLattice(2, Ns, 2, beta[i], i % 4, 10, i)
        o.set_links(links)
        o.sweep(1, 1, 5)
        assert np.abs(b.get_links(i) - o.get_links()).max() < 1e-9, i
        p, l = o.measure()
        np.testing.assert_allclose(got[i, 0], list(p) + list(l), atol=1e-12)
    b.close()


def test_refused_shape_leaves_the_layout():
    """A launch shape that is refused (400 lattices, at most 304 CTAs of 512 threads) changes nothing: the sweeps
    after it run every lattice, in a graph of their own."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_1310_7087_gb300 as q
    n = 400
    b = q.Batch([4] * n, [2] * n, [2.3] * n, [1] * n, FP64_PLAIN, HOT, 5)
    q.qcd_batch_set_block(b.h, 128)
    shape = q.qcd_batch_get_shape(b.h)
    o = oracle.OracleLattice(2, 4, 2, 2.3, 1, 10, n - 1)
    o.set_links(b.get_links(n - 1))
    b.sweep(1, 1, 5)
    o.sweep(1, 1, 5)
    with pytest.raises(q.QcdError):
        q.qcd_batch_set_block(b.h, 512)
    assert q.qcd_batch_get_shape(b.h) == shape
    b.sweep(1, 1, 6)
    o.sweep(1, 1, 6)
    assert np.abs(b.get_links(n - 1) - o.get_links()).max() < 1e-9
    b.close()
