"""The measurement of FP32 SU(3) configurations: (1/3) Re Tr of the products of the
stored links (rows 0 and 1, row 2 rebuilt as conj(row 0 x row 1)), whether or not
the rows are orthonormal.  A product of four FP32 matrices of norm up to n rounds to
about 20 x 2^-24 n^4 (1.2e-6 n^4)."""
import numpy as np
import pytest

from workloads import FP32_COMPRESSED, HOT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def q():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1310_7087_gb300 import build
    build.build()
    import paper_1310_7087_gb300 as q
    return q


def plaquettes(U, B):
    """{P, P_s, P_t} of links U[t, z, y, x, mu], y-links times diag(B[x])."""
    L = [U[..., mu, :, :] for mu in range(4)]
    L[1] = L[1] * B[:, None, :]
    at = lambda f, mu: np.roll(f, -1, 3 - mu)
    P = [0.0, 0.0]
    for mu in range(4):
        for nu in range(mu + 1, 4):
            ab, dc = L[mu] @ at(L[nu], mu), L[nu] @ at(L[mu], nu)
            P[nu == 3] += (ab * dc.conj()).real.sum((-1, -2)).mean() / 3
    return np.array([(P[0] + P[1]) / 6, P[0] / 3, P[1] / 3])


@pytest.mark.parametrize("flux,flux8", [(0, 0), (1, 0), (2, 1)])
@pytest.mark.parametrize("Ns,Nt", [(4, 4), (10, 6)])
@pytest.mark.parametrize("kind", ["unitary", "scaled", "skewed"])
def test_plaquettes(q, kind, Ns, Nt, flux, flux8):
    rng = np.random.default_rng(1)
    lat = q.Lattice(3, Ns, Nt, 5.7, flux, FP32_COMPRESSED, HOT, 7, flux8=flux8)
    U = lat.get_links()
    if kind == "scaled":
        U *= rng.uniform(0.5, 1.5, U.shape[:2])[:, :, None, None]
    elif kind == "skewed":  # row 1 no longer orthogonal to row 0
        U[:, :, 1] += 0.3 * U[:, :, 0]
    lat.set_links(U)
    U = lat.get_links().reshape(Nt, Ns, Ns, Ns, 4, 3, 3)
    x = np.arange(Ns) * 2 * np.pi / Ns ** 2
    B = np.exp(1j * x[:, None] * np.array([flux + flux8, -flux + flux8, -2 * flux8]))
    size = {"unitary": 1.0, "scaled": 2.25 ** 4, "skewed": 1.4 ** 4}[kind]
    got, _ = lat.measure()
    assert np.abs(np.array(got) - plaquettes(U, B)).max() < 1.2e-6 * size, got
    assert np.abs(np.array(lat.measure_bare()) - plaquettes(U, np.ones((Ns, 3)))).max() < 1.2e-6 * size
    lat.close()


@pytest.mark.parametrize("group,Ns", [(2, 4), (2, 10), (3, 4), (3, 10)])
def test_sums_of_exact_terms(q, group, Ns):
    """Links of small integers times powers of two, whose plaquettes are exact in FP32 and spread over 2^50: their
    sums are those of FP64, at most one rounding (2^-53 of the sum of magnitudes) in each of some ten steps."""
    rng = np.random.default_rng(2)
    Nt, V = 2, Ns ** 3 * 2
    k = rng.integers(-1, 2, (V, 4, 4 if group == 2 else 12)).astype(float)
    if group == 2:
        U = np.empty((V, 4, 2, 2), complex)
        U[..., 0, 0], U[..., 0, 1] = k[..., 0] + 1j * k[..., 3], k[..., 2] + 1j * k[..., 1]
        U[..., 1, 0], U[..., 1, 1] = -U[..., 0, 1].conj(), U[..., 0, 0].conj()
    else:
        U = np.zeros((V, 4, 3, 3), complex)
        U[:, :, :2] = (k[..., ::2] + 1j * k[..., 1::2]).reshape(V, 4, 2, 3)
    # SU(3): powers of the second row carry over to the third, so its links have one power for all
    U *= 2.0 ** (rng.integers(-6, 7, (V, 4)) if group == 2 else np.full((V, 4), -1))[:, :, None, None]
    lat = q.Lattice(group, Ns, Nt, 2.3, 0, FP32_COMPRESSED, HOT, 7)
    lat.set_links(U)
    U = lat.get_links().reshape(Nt, Ns, Ns, Ns, 4, group, group)
    L, at, sums, sizes = [U[..., mu, :, :] for mu in range(4)], lambda f, mu: np.roll(f, -1, 3 - mu), [0, 0], [0, 0]
    for mu in range(4):
        for nu in range(mu + 1, 4):
            ab, dc = L[mu] @ at(L[nu], mu), L[nu] @ at(L[mu], nu)
            t = [int(v) for v in np.rint((ab * dc.conj()).real.sum((-1, -2)) * 2.0 ** 60).ravel()]
            sums[nu == 3] += sum(t)
            sizes[nu == 3] += sum(abs(v) for v in t)
    P, S = np.array(sums, float) * 2.0 ** -60 / (3 * V * group), np.array(sizes, float) * 2.0 ** -60 / (3 * V * group)
    poly = np.trace(L[3][0] @ L[3][1], axis1=-2, axis2=-1)
    got, l = lat.measure()
    assert (np.abs(np.array(got[1:]) - P) < 10 * 2.0 ** -53 * S).all(), (got, P)
    assert abs(complex(*l) - poly.mean() / group) < 10 * 2.0 ** -53 * np.abs(poly).mean(), (l, poly.mean())
    lat.close()
