"""FP64 links at the ends of the fixed-point range, each phase against the oracle:
links that are centre elements, signs or elements of the quaternion group, whose
staples are exact multiples of group elements (or vanish).  An update divides by the norm of a
subgroup block, at least 1 among these unless it is 0, so FP64 rounding stays far below 1e-10."""
import numpy as np
import pytest

import oracle
from workloads import COLD, FP64_PLAIN, HOT

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


def exact_links(kind, group, V, rng):
    """(V, 4, N, N) links: a few centre elements in a cold lattice, or random signs or random elements of a finite group."""
    one = np.eye(group, dtype=complex)
    if group == 2:
        i, j = np.array([[1j, 0], [0, -1j]]), np.array([[0, 1], [-1, 0]], complex)
        elements = np.array([one, i, j, i @ j])
        elements = np.concatenate([elements, -elements])
    else:
        elements = np.array([np.diag(d) for d in ((1, 1, 1), (1, -1, -1), (-1, 1, -1), (-1, -1, 1))], complex)
    links = np.broadcast_to(one, (V, 4, group, group)).copy()
    if kind == "centre":  # the links around one see staples of 5 - 1; SU(3): diagonal signs
        for s in range(0, V, 37):
            links[s, s % 4] = -one if group == 2 else elements[1 + s % 3]
    elif kind == "signs":
        links *= rng.choice([1.0, -1.0], (V, 4))[:, :, None, None]
    elif kind == "group":
        links = elements[rng.integers(0, len(elements), (V, 4))]
    return links


def step(q, lat, orc, kind, parity, mu):
    lat.phase(kind, parity, mu, 5)
    if kind == q.QCD_OVERRELAX_REUNIT:
        orc.phase(q.QCD_OVERRELAX, parity, mu, 5)
        orc.reunitarize_phase(parity, mu)
    else:
        orc.phase(kind, parity, mu, 5)
    return np.abs(lat.get_links() - orc.get_links()).max()


@pytest.mark.parametrize("group,Ns,Nt,kind", [(2, 4, 4, "centre"), (2, 4, 4, "signs"), (2, 4, 4, "group"),
                                              (2, 20, 6, "centre"), (2, 20, 6, "signs"), (2, 20, 6, "group"),
                                              (3, 4, 4, "centre"), (3, 4, 4, "group"), (3, 18, 4, "group"),
                                              (3, 20, 6, "centre"), (3, 20, 6, "group")])
def test_overrelaxation_of_exact_links(q, group, Ns, Nt, kind):
    lat = q.Lattice(group, Ns, Nt, 2.3, 0, FP64_PLAIN, COLD, 7)
    orc = oracle.OracleLattice(group, Ns, Nt, 2.3, 0, 10, 0)
    start = exact_links(kind, group, Ns ** 3 * Nt, np.random.default_rng(3))
    for k, parity, mu in ((q.QCD_OVERRELAX, 0, 0), (q.QCD_OVERRELAX, 1, 3), (q.QCD_OVERRELAX_REUNIT, 1, 1)):
        lat.set_links(start)
        orc.set_links(start)
        assert step(q, lat, orc, k, parity, mu) < 1e-10, (k, parity, mu)
    lat.close()


@pytest.mark.parametrize("group,Ns,Nt,flux,kind", [(2, 4, 4, 0, "centre"), (2, 4, 4, 4, "cold"), (2, 2, 2, 1, "cold"),
                                                   (2, 20, 6, 100, "cold"), (2, 4, 4, 0, "group"), (3, 4, 4, 0, "centre"),
                                                   (3, 4, 4, 4, "cold"), (3, 18, 4, 0, "centre"), (3, 20, 6, 100, "cold")])
def test_heatbath_of_exact_links(q, group, Ns, Nt, flux, kind):
    """Field phases of a quarter turn from site to site (flux = Ns^2 / 4) make staples 4 and 2 of a cold lattice."""
    lat = q.Lattice(group, Ns, Nt, 2.3, flux, FP64_PLAIN, COLD, 7)
    orc = oracle.OracleLattice(group, Ns, Nt, 2.3, flux, 10, 0)
    start = exact_links(kind, group, Ns ** 3 * Nt, np.random.default_rng(3))
    for parity, mu in ((0, 0), (1, 1), (1, 3)):
        lat.set_links(start)
        orc.set_links(start)
        assert step(q, lat, orc, q.QCD_HEATBATH, parity, mu) < 1e-10, (parity, mu)
    assert lat.exhausted == orc.exhausted
    lat.close()


@pytest.mark.parametrize("group,Ns,Nt,flux", [(2, 4, 4, 1), (2, 6, 6, 0), (2, 20, 6, 1), (3, 4, 4, 1), (3, 20, 6, 0)])
def test_links_off_the_group(q, group, Ns, Nt, flux):
    """A third of the links with norms of 1.2 to 4: components below 2 among them, their products and reflections
    beyond it.  The bound is for links of norm 4."""
    lat = q.Lattice(group, Ns, Nt, 2.3, flux, FP64_PLAIN, HOT, 7)
    orc = oracle.OracleLattice(group, Ns, Nt, 2.3, flux, 10, 0)
    start, rng = lat.get_links(), np.random.default_rng(3)
    pick = rng.random(start.shape[:2]) < 1 / 3
    start[pick] *= rng.uniform(1.2, 4.0, pick.sum())[:, None, None]
    for kind, parity, mu in ((q.QCD_OVERRELAX, 0, 0), (q.QCD_OVERRELAX, 1, 1), (q.QCD_OVERRELAX_REUNIT, 0, 1),
                             (q.QCD_HEATBATH, 0, 3)):
        lat.set_links(start)
        orc.set_links(start)
        assert step(q, lat, orc, kind, parity, mu) < 4e-10, (kind, parity, mu)
    lat.close()


def test_batch_overrelaxation_of_exact_links(q):
    """At a coupling where every heat-bath try fails the links reach the overrelaxation as they were set."""
    Ns, Nt = [4, 6], [4, 2]
    b = q.Batch(Ns, Nt, [1e-300] * 2, [0, 0], FP64_PLAIN, COLD, 5)
    for i in range(2):
        start = exact_links("centre" if i else "group", 2, Ns[i] ** 3 * Nt[i], np.random.default_rng(3))
        b.set_links(i, start)
        orc = oracle.OracleLattice(2, Ns[i], Nt[i], 1e-300, 0, 10, i)
        orc.set_links(start)
        orc.sweep(1, 1, 5)
        if i == 0:
            first = orc
    got = b.sweep(1, 1, 5)
    for i, o in enumerate((first, orc)):
        assert np.abs(b.get_links(i) - o.get_links()).max() < 1e-10, i
        p, l = o.measure()
        np.testing.assert_allclose(got[i, 0], list(p) + list(l), atol=1e-12)
    b.close()


@pytest.mark.parametrize("scale", [0.3, 1e-3, 1e-6])
@pytest.mark.parametrize("group,Ns,Nt,flux", [(2, 4, 4, 1), (2, 20, 6, 0), (3, 4, 4, 1), (3, 18, 4, 0), (3, 20, 6, 1)])
def test_small_links(q, group, Ns, Nt, flux, scale):
    """All links scaled: fixed point has no digits of its own for small numbers, so these take the FP64 path where
    they would lose some.  Errors relative to the sizes; a hot lattice's blocks (6 terms of order 1) are at least
    1e-4 of theirs."""
    lat = q.Lattice(group, Ns, Nt, 2.3, flux, FP64_PLAIN, HOT, 7)
    orc = oracle.OracleLattice(group, Ns, Nt, 2.3, flux, 10, 0)
    start = lat.get_links() * scale
    for kind, parity, mu in ((q.QCD_OVERRELAX, 0, 0), (q.QCD_OVERRELAX, 1, 1), (q.QCD_HEATBATH, 0, 3)):
        lat.set_links(start)
        orc.set_links(start)
        err = step(q, lat, orc, kind, parity, mu)
        # (the SU(2) heat-bath replaces the link by a unit one)
        assert err < 1e-10 * (scale if kind == q.QCD_OVERRELAX or group == 3 else 1.0), (kind, parity, mu, err)
    assert lat.exhausted == orc.exhausted
    lat.set_links(start)
    orc.set_links(start)
    (p, l), (op, ol) = lat.measure(), orc.measure()
    assert np.abs(np.array(p) - np.array(op)).max() < 1e-12 * scale ** 4, (p, op)
    assert np.abs(np.array(l) - np.array(ol)).max() < 1e-12 * scale ** Nt, (l, ol)
    lat.phase(q.QCD_OVERRELAX_REUNIT, 1, 2, 5)
    orc.phase(q.QCD_OVERRELAX, 1, 2, 5)
    orc.reunitarize_phase(1, 2)
    assert np.abs(lat.get_links() - orc.get_links()).max() < 1e-10
    lat.close()


@pytest.mark.parametrize("beta", [30.0, 1e3, 1e5])
@pytest.mark.parametrize("group,Ns,Nt", [(2, 4, 4), (2, 20, 6), (3, 4, 4), (3, 18, 4), (3, 20, 6)])
def test_weak_coupling(q, group, Ns, Nt, beta):
    """Heat-bath phases of a cold lattice (blocks of norm 6) up to weak coupling: a link is about ten FP64
    operations on numbers of order 1 in the oracle for each subgroup (2^-53 each), a tenth of it here."""
    lat = q.Lattice(group, Ns, Nt, beta, 0, FP64_PLAIN, COLD, 7)
    orc = oracle.OracleLattice(group, Ns, Nt, beta, 0, 10, 0)
    for parity, mu in ((0, 0), (1, 3)):
        lat.set_links(exact_links("cold", group, Ns ** 3 * Nt, None))
        orc.set_links(lat.get_links())
        assert step(q, lat, orc, q.QCD_HEATBATH, parity, mu) < (4e-15 if group == 2 else 1.2e-14), (parity, mu)
    assert lat.exhausted == orc.exhausted
    lat.close()
