"""The fixed-point FP64 phase kernels where they can go wrong: each split of the
warps (at the sizes that choose it), a ragged last tile, links outside the
fixed-point range (which take the FP64 path) and staples that vanish, each phase
against the oracle.  An update divides by the norm of a subgroup block, at least
1e-4 among these links, so FP64 rounding stays below 1e-10."""
import numpy as np
import pytest

import oracle
from workloads import FP64_PLAIN, HOT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1310_7087_gb300 import build
    build.build()
    import paper_1310_7087_gb300 as q
    oracle.build()
    return q


def links_of(kind, links, rng):
    links = links.copy()
    V = links.shape[0]
    if kind == "scaled":  # a tenth of the links far from unitary
        pick = rng.random((V, 4)) < 0.1
        links[pick] *= rng.choice([1e-3, 1.5, 3.0, 100.0], pick.sum())[:, None, None]
    elif kind == "zero":  # every staple of an x-link vanishes
        links[:, 1:] = 0.0
    return links


@pytest.mark.parametrize("kind", ["unitary", "scaled", "zero"])
@pytest.mark.parametrize("group,Ns,Nt,flux,flux8", [(3, 6, 2, 1, 0), (3, 6, 6, 0, 0), (3, 18, 4, 1, 1), (3, 20, 4, 2, 0),
                                                    (2, 6, 2, 1, 0), (2, 6, 6, 0, 0), (2, 18, 4, 2, 0), (2, 20, 6, 1, 0)])
def test_phases(q, group, Ns, Nt, flux, flux8, kind):
    beta = 5.7 if group == 3 else 2.3
    lat = q.Lattice(group, Ns, Nt, beta, flux, FP64_PLAIN, HOT, 7, flux8=flux8)
    orc = oracle.OracleLattice(group, Ns, Nt, beta, flux, 10, 0, flux8=flux8)
    start = links_of(kind, lat.get_links(), np.random.default_rng(3))
    for step, parity, mu in ((q.QCD_HEATBATH, 1, 0), (q.QCD_OVERRELAX, 0, 0), (q.QCD_HEATBATH, 0, 1),
                             (q.QCD_OVERRELAX, 1, 1), (q.QCD_OVERRELAX_REUNIT, 0, 3)):
        if kind == "zero" and mu > 0:
            continue
        lat.set_links(start)
        orc.set_links(start)
        if step == q.QCD_OVERRELAX_REUNIT:
            if kind == "scaled":  # (a zero or huge row has no reunitarization to agree on)
                continue
            lat.phase(step, parity, mu, 5)
            orc.phase(q.QCD_OVERRELAX, parity, mu, 5)
            orc.reunitarize_phase(parity, mu)
        else:
            lat.phase(step, parity, mu, 5)
            orc.phase(step, parity, mu, 5)
        a, b = lat.get_links(), orc.get_links()
        err = np.abs(a - b).max(axis=(2, 3)) / np.maximum(1.0, np.abs(b).max(axis=(2, 3)))
        assert err.max() < 1e-10, (step, parity, mu, err.max())
    assert lat.exhausted == orc.exhausted
    lat.close()


@pytest.mark.parametrize("kind", ["unitary", "scaled"])
@pytest.mark.parametrize("Ns,Nt,flux,flux8", [(6, 2, 1, 0), (18, 4, 1, 1), (20, 4, 0, 0)])
def test_su3_working_sweep_measurement(q, Ns, Nt, flux, flux8, kind):
    """The plaquette sums on the last pass and the Polyakov loop in fixed point:
    the links of the same sweep without them, and the numbers of the separate
    measurement on those links (FP64 sums of 10^4 to 10^5 terms of order 1)."""
    a = q.Lattice(3, Ns, Nt, 5.7, flux, FP64_PLAIN, HOT, 7, flux8=flux8)
    b = q.Lattice(3, Ns, Nt, 5.7, flux, FP64_PLAIN, HOT, 7, flux8=flux8)
    start = links_of(kind, a.get_links(), np.random.default_rng(3))
    a.set_links(start)
    b.set_links(start)
    got = np.array(q.qcd_working_sweep(a.h, 1, 1, 5))
    b.sweep(1, 1, 5)
    assert np.array_equal(a.get_links(), b.get_links())
    p, l = b.measure()
    assert np.abs(got - np.array(p + l)).max() < 1e-13
    a.close()
    b.close()


@pytest.mark.parametrize("kind", ["unitary", "scaled"])
@pytest.mark.parametrize("group,Ns,Nt,flux,flux8", [(3, 6, 2, 1, 0), (3, 10, 4, 1, 1), (2, 6, 2, 0, 0), (2, 10, 4, 2, 0)])
def test_measurement(q, group, Ns, Nt, flux, flux8, kind):
    """Ragged blocks, fields, and links out of the fixed-point range (their sites in
    FP64) against the oracle: sums of 10^3 to 10^4 terms of the size of the largest."""
    lat = q.Lattice(group, Ns, Nt, 5.7, flux, FP64_PLAIN, HOT, 7, flux8=flux8)
    orc = oracle.OracleLattice(group, Ns, Nt, 5.7, flux, 10, 0, flux8=flux8)
    start = links_of(kind, lat.get_links(), np.random.default_rng(3))
    lat.set_links(start)
    orc.set_links(start)
    (p, l), (op, ol) = lat.measure(), orc.measure()
    for got, ref in ((p, op), (l, ol), (lat.measure_bare(), orc.measure_bare())):
        size = 1.0 if kind == "unitary" else 100.0 ** Nt
        assert np.abs(np.array(got) - np.array(ref)).max() < 1e-12 * size, (got, ref)
    lat.close()
