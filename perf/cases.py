"""What is measured: the Monte Carlo work that a run with this package does, through its public entry points.

Five kinds of pass:

  chain    a stored configuration goes to the lattice (pinned host memory), `sweeps` working sweeps run on it
           (1 heat-bath pass, n_or overrelaxation passes, reunitarization, plaquettes and Polyakov loop each), and
           the configuration comes back: the stretch of a production run between two stored configurations.
  scan     one call of the batched SU(2) parameter scan (`sweeps` sweeps of every lattice, measured each).
  on       the O(N) model: `sweeps` Metropolis sweeps, a measurement, and the field.
  stored   analysis of a stored configuration: canonical links to the lattice, the measurements, the links back.

Sizes and couplings are those of the repository's workloads (SU(2) 4^3x4, SU(3) 16^3x4, 32^3x8 and 64^3x16, the
64-lattice scan, O(4) on 32^4), its tests (6^3x4, 20^3, 24^3x6, 48^3x16) and even extents between them.
"""
import math

import numpy as np
import torch

import paper_1310_7087_gb300 as q

FP64, FP32 = 0, 1
MASK = 0xFFFFFFFF


def chain(name, group, Ns, Nt, beta, precision, sweeps, n_or, flux=1, flux8=0, frozen=False):
    return dict(name=name, kind="chain", group=group, Ns=Ns, Nt=Nt, beta=beta, precision=precision, sweeps=sweeps,
                n_or=n_or, flux=flux, flux8=flux8, frozen=frozen)


def listed():
    return [
        # The smallest calls: a test lattice in double precision, each sweep's results read as they come.
        chain("su2_fp64_4x4", 2, 4, 4, 2.3, FP64, 4, 1, flux=0),
        # A small finite-temperature lattice, in both storages, one sweep between stored configurations.
        chain("su3_fp32_16x4", 3, 16, 4, 5.7, FP32, 1, 4),
        chain("su3_fp64_16x4", 3, 16, 4, 5.7, FP64, 1, 4),
        # The lattice of the flux scan: the FP32 production chain, and the double-precision run that checks it.
        chain("su3_fp32_32x8", 3, 32, 8, 6.0, FP32, 10, 4, flux=2),
        chain("su3_fp64_32x8", 3, 32, 8, 6.0, FP64, 1, 4, flux=2),
        # The large production lattices: links far beyond L2.
        chain("su3_fp32_64x16", 3, 64, 16, 6.2, FP32, 10, 4),
        chain("su2_fp32_64x16", 2, 64, 16, 2.4, FP32, 10, 1),
        # The physically visible field: frozen t = 0 links, both flux components, extents that are not powers of two
        # (there the measurement is a pass of its own).
        chain("su3_fp32_frozen_20x6", 3, 20, 6, 5.9, FP32, 5, 4, flux=1, flux8=1, frozen=True),
        # The batched scan of 64 uneven lattices.
        dict(name="scan64_fp32", kind="scan", lattices=64, Ns_max=24, precision=FP32, sweeps=20, n_or=1, draw=11),
        # The second model family: the benchmark lattice in FP32, a smaller one in double precision.
        dict(name="o4_fp32_32", kind="on", N=4, Ns=32, Nt=32, precision=FP32, sweeps=20, nhit=100),
        dict(name="o4_fp64_16", kind="on", N=4, Ns=16, Nt=16, precision=FP64, sweeps=5, nhit=100),
        # A stored configuration read, measured and written back.
        dict(name="su3_fp32_stored_24x6", kind="stored", group=3, Ns=24, Nt=6, beta=5.9, precision=FP32, flux=1),
    ]


def draw(rng):
    """One more case of the same ranges; a chain's size is spread over the logarithm of its volume."""

    def extents(v_max):
        v = math.exp(rng.uniform(math.log(256), math.log(v_max)))
        Nt = 2 * rng.randint(1, max(1, min(8, int(round((v ** 0.25) / 2)))))
        Ns = 2 * max(2, min(32, int((v / Nt) ** (1 / 3) / 2)))
        return Ns, Nt

    kind = rng.choice(["chain"] * 6 + ["scan", "scan", "on", "on", "stored"])
    if kind == "chain":
        group, precision = rng.choice([2, 3]), rng.choice([FP64, FP32])
        Ns, Nt = extents({(2, FP64): 48 ** 3 * 8, (3, FP64): 32 ** 3 * 8, (2, FP32): 60 ** 3 * 16,
                          (3, FP32): 60 ** 3 * 14}[group, precision])
        n_or = rng.choice([1, 2]) if group == 2 else rng.choice([2, 3, 4])
        sweeps = rng.randint(1, 10) if precision == FP32 else 1 if group == 3 else rng.randint(1, 3)
        beta = round(rng.uniform(2.2, 2.5) if group == 2 else rng.uniform(5.5, 6.3), 3)
        c = chain("", group, Ns, Nt, beta, precision, sweeps, n_or, flux=rng.randint(0, 4),
                  flux8=rng.choice([0, 0, 1]) if group == 3 else 0, frozen=rng.random() < 0.2)
    elif kind == "scan":
        precision = rng.choice([FP64, FP32])
        c = dict(kind="scan", lattices=rng.randint(4, 96 if precision == FP32 else 24),
                 Ns_max=rng.choice([8, 12, 16, 24]), precision=precision,
                 sweeps=rng.randint(1, 30) if precision == FP32 else 1, n_or=rng.choice([1, 2]),
                 draw=rng.randint(1, 999))
    elif kind == "on":
        precision = rng.choice([FP64, FP32])
        Ns = 2 * rng.randint(2, 16 if precision == FP32 else 12)
        c = dict(kind="on", N=rng.randint(1, 4), Ns=Ns, Nt=2 * rng.randint(2, 16 if precision == FP32 else 12),
                 precision=precision, sweeps=rng.randint(1, 20 if precision == FP32 else 5),
                 nhit=rng.choice([10, 30, 100]))
    else:
        group = rng.choice([2, 3])
        Ns, Nt = extents(32 ** 3 * 8)
        c = dict(kind="stored", group=group, Ns=Ns, Nt=Nt, beta=5.9 if group == 3 else 2.3,
                 precision=rng.choice([FP64, FP32]), flux=rng.randint(0, 4))
    c.pop("name", None)
    return c


# ---- inputs ----------------------------------------------------------------

def configuration(case, seed, device):
    """Links (t, z, y, x, mu, N, N) of about the plaquette that a thermal run has at these couplings (0.55 to 0.65),
    in a random gauge: matrices near the unit, then a gauge transformation by Haar-random ones."""
    N, Ns, Nt = case["group"], case["Ns"], case["Nt"]
    gen = torch.Generator(device=device).manual_seed(int(seed))
    shape = (Nt, Ns, Ns, Ns)

    def near_unit(eps):
        z = torch.randn(*shape, N, N, 2, generator=gen, device=device, dtype=torch.float64)
        return _group(torch.eye(N, device=device, dtype=torch.complex128) * (1.0 if eps else 0.0)
                      + (eps or 1.0) * torch.view_as_complex(z))

    g = near_unit(0.0)
    U = torch.empty(*shape, 4, N, N, dtype=torch.complex128, device=device)
    for mu in range(4):
        U[..., mu, :, :] = _mm(_mm(g, near_unit(0.2)), _dag(_at(g, mu, 1)))
    return U


def scan_parameters(case):
    rng = np.random.default_rng(case["draw"])
    n = case["lattices"]
    Ns = [int(v) for v in rng.choice([s for s in (8, 12, 16, 24) if s <= case["Ns_max"]], n)]
    Nt = [int(v) for v in rng.choice([4, 6, 8], n)]
    return Ns, Nt, [float(v) for v in rng.uniform(2.2, 2.5, n)], [int(v) for v in rng.integers(0, 4, n)]


def real_view(U):
    return np.ascontiguousarray(torch.view_as_real(U.reshape(-1, *U.shape[4:])).cpu().numpy())


def make_lattice(case, seed):
    return q.Lattice(case["group"], case["Ns"], case["Nt"], case["beta"], case["flux"], case["precision"], q.QCD_COLD,
                     seed, flux8=case.get("flux8", 0),
                     field_mode=q.QCD_FIELD_FROZEN if case.get("frozen") else q.QCD_FIELD_LINKS)


def prepare(case, seed):
    s = dict(case=case, seed=seed)
    if case["kind"] == "scan":
        s["scan"] = q.Batch(*scan_parameters(case), case["precision"], q.QCD_HOT, seed)
    elif case["kind"] == "on":
        s["model"] = q.ONModel(case["N"], case["Ns"], case["Nt"], 0.3, 1.0, 0.8, case["precision"], q.QCD_HOT, seed,
                               nhit=case["nhit"])
    else:
        s["lat"] = lat = make_lattice(case, seed)
        U = configuration(case, seed, "cuda")
        if case.get("frozen"):
            _freeze(case, U)
        s["links"] = real_view(U)
        if case["kind"] == "chain":
            raw = torch.zeros(lat.link_bytes // (8 if case["precision"] == FP64 else 4), pin_memory=True,
                              dtype=torch.float64 if case["precision"] == FP64 else torch.float32)
            q.qcd_copy_links_in(lat.h, raw.data_ptr(), lat.link_bytes)  # zeros in the padding of the planes
            lat.set_links(s.pop("links"))
            q.qcd_copy_links_out(lat.h, raw.data_ptr(), lat.link_bytes)
            s["in"], s["out"] = raw, torch.zeros_like(raw).pin_memory()
            s["rows"] = torch.zeros(case["sweeps"], 5, dtype=torch.float64, pin_memory=True)
    return s


# ---- one pass ----------------------------------------------------------------

def run(s):
    case, seed = s["case"], s["seed"]
    # An FP32 run's measurements are sums over FP32 products: they come back in the type of their links.
    real = np.float64 if case["precision"] == FP64 else np.float32
    if case["kind"] == "scan":
        return s["scan"].sweep(case["sweeps"], case["n_or"], seed).astype(real)
    if case["kind"] == "on":
        m = s["model"]
        m.sweep(case["sweeps"], seed)
        return {"measured": np.array(m.measure(), real), "field": m.get_field()}
    lat = s["lat"]
    if case["kind"] == "stored":
        lat.set_links(s["links"])
        p, l = lat.measure()
        b = lat.measure_bare()
        return {"measured": np.array(p + l + b, real), "links": lat.get_links()}
    q.qcd_copy_links_in(lat.h, s["in"].data_ptr(), lat.link_bytes)
    rows = s["rows"]
    for k in range(case["sweeps"]):
        q.qcd_working_sweep(lat.h, 1, case["n_or"], seed, rows[k].data_ptr(), wait=False)
    q.qcd_copy_links_out(lat.h, s["out"].data_ptr(), lat.link_bytes)
    return {"measured": rows.numpy().astype(real), "links": s["out"]}


def work(case):
    """Bytes: a phase (one parity, one direction) depends on the whole lattice after the phase before it, so it reads
    the 4.5 V links that its V/2 updates need and writes V/2 links; a measurement reads the links once; a stored
    configuration goes in and comes out once.  Flops: the 12 matrix products of the staple, U A and the update."""
    if case["kind"] == "scan":
        Ns, Nt, _, _ = scan_parameters(case)
        V, group = sum(a ** 3 * b for a, b in zip(Ns, Nt)), 2
    else:
        V, group = case["Ns"] ** 3 * case["Nt"], case.get("group", 0)
    word = 8 if case["precision"] == FP64 else 4
    if case["kind"] == "on":
        N = case["N"]
        return {"bytes": float(case["sweeps"] * V * N * word * 2 + V * N * (word + 8)),
                "flops": float(case["sweeps"]) * V * case["nhit"] * (8 * N + 10)}
    link = word * (4 if group == 2 else 18 if case["precision"] == FP64 else 12)
    if case["kind"] == "stored":
        canonical = 4 * V * group * group * 16
        return {"bytes": float(2 * canonical + 4 * 4 * V * link), "flops": 2 * 6.0 * V * (60 if group == 2 else 450)}
    updates = 4.0 * V * case["sweeps"] * (1 + case["n_or"])
    io = 2 * 4 * V * link if case["kind"] == "chain" else 0
    return {"bytes": updates * 9 * link + io, "flops": updates * (430 if group == 2 else 3400)}


# ---- the same numbers in 64 bits, by plain torch ----------------------------

def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


def _at(f, mu, step):
    """The field at x + step mu (dimensions t, z, y, x)."""
    return torch.roll(f, -step, 3 - mu)


def _group(z):
    """Rows by Gram-Schmidt, the last one from the others: a group element."""
    r0 = z[..., 0, :]
    r0 = r0 / r0.abs().square().sum(-1, keepdim=True).sqrt()
    if z.shape[-1] == 2:
        return torch.stack([r0, torch.stack([-r0[..., 1].conj(), r0[..., 0].conj()], -1)], -2)
    r1 = z[..., 1, :] - (r0.conj() * z[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], -2)


def _philox(c0, c1, c2, c3, k0, k1):
    c = [torch.as_tensor(v, dtype=torch.int64, device=c0.device).expand_as(c0) for v in (c0, c1, c2, c3)]
    for r in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & MASK) ^ c[1] ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c[3] ^ k1, p0 & MASK]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in c]


def _quaternion(w, i, j):
    return torch.stack([w[..., i, i].real + w[..., j, j].real, w[..., i, j].imag + w[..., j, i].imag,
                        w[..., i, j].real - w[..., j, i].real, w[..., i, i].imag - w[..., j, j].imag], -1) * 0.5


def _matrix(v):
    a, b, c, d = v.unbind(-1)
    return torch.stack([torch.stack([torch.complex(a, d), torch.complex(c, b)], -1),
                        torch.stack([torch.complex(-c, b), torch.complex(a, -d)], -1)], -2)


class Exact:
    """One gauge lattice in 64 bits; `number` is its place in a batch (it enters the random numbers' key)."""

    def __init__(self, U, group, beta, flux, flux8, frozen, seed, number=0, nhit=10):
        self.U, self.N, self.beta, self.frozen, self.nhit = U, group, beta, frozen, nhit
        self.key = ((seed & MASK) ^ (number * 0x9E3779B9 & MASK), (seed >> 32) & MASK)
        Nt, Ns = U.shape[0], U.shape[1]
        t, z, y, x = torch.meshgrid(*(torch.arange(n, device=U.device) for n in U.shape[:4]), indexing="ij")
        self.parity, self.t, self.site = (x + y + z + t) & 1, t, x + Ns * (y + Ns * (z + Ns * t))
        self.B = _background(group, Ns, flux, flux8, U.device) if not frozen else torch.ones(Ns, group, device=U.device) + 0j

    def eff(self, mu):
        return self.U[..., mu, :, :] * self.B[:, None, :] if mu == 1 else self.U[..., mu, :, :]

    def staple(self, mu):
        A = 0
        um = self.eff(mu)
        for nu in range(4):
            if nu != mu:
                un = self.eff(nu)
                ahead = _at(un, mu, 1)
                A = A + _mm(_mm(ahead, _dag(_at(um, nu, 1))), _dag(un))
                A = A + _at(_mm(_dag(_mm(um, ahead)), un), nu, -1)
        return A

    def draw(self, alpha, site, sweep, tag):
        """Kennedy-Pendleton: the quaternion, and whether a try was accepted."""
        delta, done = torch.ones_like(alpha), torch.zeros_like(alpha, dtype=torch.bool)
        for k in range(self.nhit):
            u = _philox(site, sweep, tag, k, *self.key)
            d = (-u[1].log() - u[0].log() * torch.cos(2 * math.pi * u[2]) ** 2) / alpha
            ok = ~done & (u[3] ** 2 <= 1 - d / 2)
            delta, done = torch.where(ok, d, delta), done | ok
            if bool(done.all()):
                break
        u = _philox(site, sweep, tag | 16, 0, *self.key)
        r, st = (delta * (2 - delta)).sqrt(), 2 * (u[0] * (1 - u[0])).sqrt()
        phi = 2 * math.pi * u[1]
        return torch.stack([1 - delta, r * st * phi.cos(), r * st * phi.sin(), r * (2 * u[0] - 1)], -1), done

    def phase(self, heat, p, mu, sweep):
        m = self.parity == p
        if self.frozen and mu < 3:
            m = m & (self.t != 0)
        A, U, Ut, site = self.staple(mu)[m], self.U[..., mu, :, :][m], self.eff(mu)[m], self.site[m]
        if self.N == 2:
            a = _quaternion(A, 0, 1)
            k = a.square().sum(-1).sqrt()
            V = _dag(_matrix(a / k[:, None]))
            if heat:
                X, ok = self.draw(self.beta * k, site, sweep, mu)
                new = torch.where(ok[:, None, None], _mm(_matrix(X), V), Ut)
            else:
                new = _mm(_mm(V, _dag(Ut)), V)
        else:
            W, new = _mm(Ut, A), Ut
            for sub, (i, j) in enumerate(((0, 1), (1, 2), (0, 2))):
                w = _quaternion(W, i, j)
                k = w.square().sum(-1).sqrt()
                V = _dag(_matrix(w / k[:, None]))
                R = _mm(V, V)
                if heat:
                    X, ok = self.draw(2.0 / 3.0 * self.beta * k, site, sweep, mu | sub << 2)
                    R = torch.where(ok[:, None, None], _mm(_matrix(X), V), torch.eye(2, device=U.device) + 0j)
                E = torch.eye(3, device=U.device, dtype=U.dtype).expand(U.shape).clone()
                E[:, i, i], E[:, i, j], E[:, j, i], E[:, j, j] = R[:, 0, 0], R[:, 0, 1], R[:, 1, 0], R[:, 1, 1]
                W, new = _mm(E, W), _mm(E, new)
        if mu == 1:
            new = new * (self.B[:, None, :].conj().expand(*self.U.shape[:4], self.N, self.N)[m])
        V = self.U[..., mu, :, :].clone()
        V[m] = new
        self.U[..., mu, :, :] = V

    def sweep(self, n, n_or):
        for o in range(1 + n_or):
            for p in (0, 1):
                for mu in range(4):
                    self.phase(o == 0, p, mu, n)
        V = _group(self.U)
        if self.frozen:
            V[0, :, :, :, :3] = self.U[0, :, :, :, :3]
        self.U = V

    def measure(self, bare=False):
        link = (lambda mu: self.U[..., mu, :, :]) if bare else self.eff
        P = [0.0, 0.0]
        for mu in range(4):
            for nu in range(mu + 1, 4):
                ab, dc = _mm(link(mu), _at(link(nu), mu, 1)), _mm(link(nu), _at(link(mu), nu, 1))
                P[nu == 3] += float((ab * dc.conj()).real.sum((-1, -2)).mean()) / self.N
        L = self.U[0, ..., 3, :, :]
        for t in range(1, self.U.shape[0]):
            L = _mm(L, self.U[t, ..., 3, :, :])
        L = torch.diagonal(L, dim1=-2, dim2=-1).sum(-1).mean() / self.N
        return [(P[0] + P[1]) / 6, P[0] / 3, P[1] / 3] + ([] if bare else [float(L.real), float(L.imag)])


def _background(group, Ns, flux, flux8, device):
    theta = 2 * math.pi * torch.arange(Ns, device=device, dtype=torch.float64)[:, None] / Ns ** 2 * torch.tensor(
        [flux, -flux] if group == 2 else [flux + flux8, -flux + flux8, -2 * flux8], device=device, dtype=torch.float64)
    return torch.polar(torch.ones_like(theta), theta)


def _freeze(case, U):
    """The spatial links of t = 0 hold the background."""
    U[0, :, :, :, :3] = torch.eye(case["group"], device=U.device) + 0j
    U[0, :, :, :, 1] = torch.diag_embed(_background(case["group"], case["Ns"], case["flux"], case["flux8"], U.device))


def _stored(case, U):
    """The links as the storage holds them: FP32 keeps rows 0 and 1 of SU(3), the four reals of SU(2)."""
    if case["precision"] == FP64 and case["group"] == 3:
        return U
    if case["group"] == 2:
        v = _quaternion(U, 0, 1)
        return _matrix(v if case["precision"] == FP64 else v.float().double())
    r = torch.view_as_complex(torch.view_as_real(U[..., :2, :].contiguous()).float().double())
    return torch.cat([r, torch.linalg.cross(r[..., 0, :], r[..., 1, :]).conj().unsqueeze(-2)], -2)


def _raw(case, U):
    """The storage's bytes as reals: 16-byte vectors [component][mu][parity][site / 2], planes padded to 64."""
    if case["group"] == 2:
        v = _quaternion(U, 0, 1)
    else:
        v = torch.view_as_real((U if case["precision"] == FP64 else U[..., :2, :]).contiguous()).flatten(-3)
    lanes = 2 if case["precision"] == FP64 else 4
    Ns, Vh = case["Ns"], v.shape[0] * case["Ns"] ** 3 // 2
    v = v.reshape(-1, Ns // 2, 2, 4, v.shape[-1] // lanes, lanes)  # rows of x-pairs
    row = torch.arange(v.shape[0], device=U.device)
    odd = (row % Ns + row // Ns % Ns + row // Ns ** 2) & 1
    v = torch.where(odd.bool()[:, None, None, None, None, None], v.flip(2), v)  # [.., parity, ..]
    out = torch.zeros(v.shape[4], 4, 2, (Vh + 63) // 64 * 64, lanes, device=U.device, dtype=torch.float64)
    out[:, :, :, :Vh] = v.reshape(Vh, 2, 4, v.shape[4], lanes).permute(3, 2, 1, 0, 4)
    return out.flatten()


def _exact_on(case, seed):
    N, Ns, Nt = case["N"], case["Ns"], case["Nt"]
    t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (Nt, Ns, Ns, Ns)), indexing="ij")
    parity, site = (x + y + z + t) & 1, x + Ns * (y + Ns * (z + Ns * t))
    key, kappa, lam, delta = (seed & MASK, (seed >> 32) & MASK), 0.3, 1.0, 0.8
    phi = 2 * torch.stack(_philox(site, MASK, 2 << 4, 0, *key)[:N], -1) - 1
    for n in range(case["sweeps"]):
        for p in (0, 1):
            m = parity == p
            F = sum(_at(phi, mu, d) for mu in range(4) for d in (1, -1))[m]
            f, s = phi[m], site[m]

            def action(v):
                vv = v.square().sum(-1)
                return -2 * kappa * (v * F).sum(-1) + vv + lam * (vv - 1) ** 2

            cur = action(f)
            for h in range(case["nhit"]):
                trial = f + delta * (2 * torch.stack(_philox(s, n, 3 << 4, h, *key)[:N], -1) - 1)
                u = _philox(s, n, 4 << 4, h >> 2, *key)[h & 3]
                new = action(trial)
                ok = (new <= cur) | (u < torch.exp(cur - new))
                f, cur = torch.where(ok[:, None], trial, f), torch.where(ok, new, cur)
            phi[m] = f
    M = phi.reshape(-1, N).mean(0)
    links = sum((phi * _at(phi, mu, 1)).sum() for mu in range(4)) / (4 * phi[..., 0].numel())
    out = [float(phi.square().sum(-1).mean()), float(links), float(M.norm())] + [float(v) for v in M] + [0.0] * (4 - N)
    return {"measured": np.array(out), "field": phi.reshape(-1, N).cpu().numpy()}


def exact(case, seed):
    """None where the rounding decides the numbers, because no 64-bit run stays near: chains of FP32 sweeps with
    overrelaxation (a pass multiplies a difference by about ten), FP32 Metropolis chains; and for lattices too large
    to be done in seconds."""
    chaotic = case["precision"] == FP32 and (case["kind"] in ("scan", "on") or case.get("sweeps", 1) > 1)
    if chaotic:
        return None
    if case["kind"] == "on":
        return _exact_on(case, seed) if case["Ns"] ** 3 * case["Nt"] * case["nhit"] <= 3e7 else None
    if case["kind"] == "scan":
        Ns, Nt, beta, flux = scan_parameters(case)
        if case["lattices"] > 24:
            return None
        rows = []
        for i, (a, b) in enumerate(zip(Ns, Nt)):
            t, z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (b, a, a, a)), indexing="ij")
            site = x + a * (y + a * (z + a * t))
            k = ((seed & MASK) ^ (i * 0x9E3779B9 & MASK), (seed >> 32) & MASK)
            v = []
            for mu in range(4):  # the hot start: Haar quaternions
                u = _philox(site, MASK, mu | 2 << 4, 0, *k)
                r1, r2 = (1 - u[0]).sqrt(), u[0].sqrt()
                v.append(torch.stack([r1 * torch.sin(2 * math.pi * u[1]), r1 * torch.cos(2 * math.pi * u[1]),
                                      r2 * torch.sin(2 * math.pi * u[2]), r2 * torch.cos(2 * math.pi * u[2])], -1))
            e = Exact(_matrix(torch.stack(v, -2)), 2, beta[i], flux[i], 0, False, seed, i)
            got = []
            for n in range(case["sweeps"]):
                e.sweep(n, case["n_or"])
                got.append(e.measure())
            rows.append(got)
        return np.array(rows)
    V = case["Ns"] ** 3 * case["Nt"]
    if V > 4e5 or V * case.get("sweeps", 1) > 6e5:
        return None
    U = configuration(case, seed, "cuda")
    if case.get("frozen"):
        _freeze(case, U)
    U = _stored(case, U)
    e = Exact(U, case["group"], case["beta"], case["flux"], case.get("flux8", 0), case.get("frozen", False), seed)
    if case["kind"] == "stored":
        return {"measured": np.array(e.measure() + e.measure(bare=True)),
                "links": U.reshape(V, *U.shape[4:]).cpu().numpy()}
    rows = []
    for n in range(case["sweeps"]):
        e.sweep(n, case["n_or"])
        rows.append(e.measure())
    return {"measured": np.array(rows), "links": _raw(case, e.U)}
