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
