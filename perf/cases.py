"""The work that a user of this library has it do, as cases that can be timed and compared.

A spectrum is made from: the spectral bounds of H (``KPM.bounds``), the dipole applied to the
ground state (``KPM.apply_dipole``), the Chebyshev recursion (``KPM.moments``, one ``KPM.sigma`` a
step and column; ``moments_batch`` for many small molecules), and the reconstruction of the
intensity (``spectrum``).  Nearly all of the time goes into sigma, so most cases are one H
application at a size and precision in use; the whole calls are the FP64 ones, whose results are
held to FP64 rounding.

Integrals follow the recipe of ``synthetic`` (linspace one-body diagonal, Cholesky-factored
(pq|rs), Gaussian dipoles).  Vectors are normal draws whose weight falls with the rank of the
strings, as that of a low-lying state does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_07430_gb300 import KPM, moments_batch, spectrum

DEV = "cuda"


# ---------------------------------------------------------------- cases

def listed():
    return [
        # the 8-orbital FP64 workload: 256 moments of x, y and z, where launches and latency count
        dict(name="moments_fp64_8o", kind="moments", norb=8, na=4, nb=4, mask=7, nmoments=256),
        # many small molecules in one call, odd sizes and open shells among them
        dict(name="batch_fp64_small", kind="batch", count=12, norb=6, spread=3, mask=7,
             nmoments=128),
        # a, b of a request: 40 Lanczos steps at the served 10-orbital size
        dict(name="bounds_fp64_10o", kind="bounds", norb=10, na=5, nb=5, iters=40),
        # the FP64 H application of the 12-orbital workload: ground states, accuracy reference
        dict(name="sigma_fp64_12o", kind="sigma", prec="fp64", norb=12, na=6, nb=6, ncol=1),
        # the 12-orbital FP32 workload: x, y, z as one block of three columns
        dict(name="sigma_fp32_12o_xyz", kind="sigma", prec="fp32", norb=12, na=6, nb=6, ncol=3),
        # open shell, odd orbital count: 1716 x 1287 strings, ragged in every tile
        dict(name="sigma_fp32_13o_open", kind="sigma", prec="fp32", norb=13, na=7, nb=5, ncol=1),
        # the smallest served size on the default (tensor-core) precision
        dict(name="sigma_mixed_10o_xyz", kind="sigma", prec="mixed", norb=10, na=5, nb=5, ncol=3),
        # BF16 operand pieces, odd orbital count, open shell
        dict(name="sigma_bf16_13o_open", kind="sigma", prec="mixed_bf16", norb=13, na=7, nb=6,
             ncol=1),
        # the largest served size, x, y and z
        dict(name="sigma_mixed_14o_xyz", kind="sigma", prec="mixed", norb=14, na=7, nb=7, ncol=3),
        # the benchmark's 16-orbital / 16-electron H application
        dict(name="sigma_mixed_16o", kind="sigma", prec="mixed", norb=16, na=8, nb=8, ncol=1),
        # mu|0> that starts a recursion, once for each component
        dict(name="dipole_14o", kind="dipole", prec="mixed", norb=14, na=7, nb=7, comp=2),
        # the reconstruction of a finished request: host moments in, host spectrum out
        dict(name="spectrum_2048", kind="spectrum", nmoments=2048, npoints=2048,
             kernel="jackson"),
    ]


def _shell(rng, n):
    """Electrons of each spin: near half filling, open shells among them."""
    lo, hi = max(1, n // 2 - 2), min(n - 1, (n + 1) // 2 + 1)
    return rng.randint(lo, hi), rng.randint(lo, hi)


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "sigma", "sigma", "moments", "batch", "bounds",
                       "dipole", "spectrum"])
    if kind == "sigma":
        prec = rng.choice(["fp64", "fp32", "mixed", "mixed", "mixed_bf16"])
        n = rng.randint(6, {"fp64": 12, "fp32": 14, "mixed": 16, "mixed_bf16": 15}[prec])
        na, nb = _shell(rng, n)
        dim = math.comb(n, na) * math.comb(n, nb)
        ncol = rng.randint(1, 3) if dim <= 4_000_000 else 1
        return dict(kind="sigma", prec=prec, norb=n, na=na, nb=nb, ncol=ncol)
    if kind == "moments":
        n = rng.randint(4, 9)
        na, nb = _shell(rng, n)
        return dict(kind="moments", norb=n, na=na, nb=nb, mask=rng.randint(1, 7),
                    nmoments=2 * int(round(math.exp(rng.uniform(math.log(16), math.log(128))))))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 16), norb=rng.randint(4, 6),
                    spread=rng.randint(1, 3), mask=rng.randint(1, 7),
                    nmoments=2 * int(round(math.exp(rng.uniform(math.log(16), math.log(100))))))
    if kind == "bounds":
        n = rng.randint(8, 11)
        na, nb = _shell(rng, n)
        return dict(kind="bounds", norb=n, na=na, nb=nb, iters=rng.randint(20, 40))
    if kind == "dipole":
        n = rng.randint(8, 15)
        na, nb = _shell(rng, n)
        return dict(kind="dipole", prec=rng.choice(["fp64", "fp32", "mixed"]) if n < 14 else "mixed",
                    norb=n, na=na, nb=nb, comp=rng.randint(0, 2))
    # moment counts up to the tens of thousands of the paper's molecules
    return dict(kind="spectrum",
                nmoments=int(round(math.exp(rng.uniform(math.log(200), math.log(60000))))),
                npoints=int(round(math.exp(rng.uniform(math.log(500), math.log(8192))))),
                kernel=rng.choice(["jackson", "jackson", "lorentz", "none"]))


# ---------------------------------------------------------------- inputs

def _mirror(m, k):
    return np.triu(m, k) + np.triu(m, 1).T


def _integrals(n, seed):
    rng = np.random.default_rng(seed)
    h1 = _mirror(rng.normal(0.0, 0.05, (n, n)), 1)
    h1[np.diag_indices(n)] = np.linspace(-2.0, 1.0, n)
    L = np.stack([_mirror(rng.normal(0.0, 0.1, (n, n)), 0) for _ in range(2 * n)])
    eri = np.tensordot(L, L, axes=(0, 0))
    # the 8-fold symmetry to the last bit
    eri = 0.5 * (eri + eri.transpose(2, 3, 0, 1))
    dip = np.stack([_mirror(rng.normal(0.0, 0.3, (n, n)), 0) for _ in range(3)])
    return h1, eri, dip


def _vectors(case, seed, ncol, dtype):
    n, na, nb = case["norb"], case["na"], case["nb"]
    sa, sb = math.comb(n, na), math.comb(n, nb)
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + 7)
    x = torch.randn((ncol, sa, sb), generator=g, device=DEV, dtype=dtype)
    wa = torch.exp(-3.0 * torch.arange(sa, device=DEV, dtype=torch.float64) / sa)
    wb = torch.exp(-3.0 * torch.arange(sb, device=DEV, dtype=torch.float64) / sb)
    x *= wa.to(dtype)[None, :, None]
    x *= wb.to(dtype)[None, None, :]
    for c in range(ncol):
        x[c] /= x[c].norm()
    return x.reshape(ncol, sa * sb)


def _molecules(case):
    """(norb, na, nb) of a batch: sizes norb .. norb + spread - 1, open shells in between."""
    out = []
    for i in range(case["count"]):
        n = case["norb"] + i % case["spread"]
        out.append((n, n // 2, (n + 1) // 2 if i % 2 else n // 2))
    return out


def _moments_of(seed, nmoments):
    """Moments as a finished recursion leaves them: a decaying cosine sum, |Omega_n| <= Omega_0."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.98, 0.98, 24)
    w = rng.exponential(1.0, 24)
    n = np.arange(nmoments)
    return (w[:, None] * np.cos(n[None, :] * np.arccos(x)[:, None])).sum(0)


SCALE_A, SCALE_B = 14.25, -3.5      # a, b of the spectrum cases (Hartree)


def _state(n, na, nb, seed):
    """Integrals, a near ground state (the lowest Ritz vector of a short Lanczos run) and a, b."""
    h1, eri, dip = _integrals(n, seed)
    sa, sb = math.comb(n, na), math.comb(n, nb)
    H = _Plain(h1, eri, n, na, nb)
    v = _vectors(dict(norb=n, na=na, nb=nb), seed, 1, torch.float64)[0].reshape(sa, sb)
    k = min(30, sa * sb)
    al, be, vs = [], [], [v]
    for j in range(k):
        w = H.sigma(vs[j])
        al.append(float((w * vs[j]).sum()))
        for _ in range(2):
            for u in vs:
                w = w - (u * w).sum() * u
        b = float(w.norm())
        if j == k - 1 or b < 1e-8:
            break
        be.append(b)
        vs.append(w / b)
    e, s = np.linalg.eigh(np.diag(al) + np.diag(be[: len(al) - 1], 1) + np.diag(be[: len(al) - 1], -1))
    psi = sum(float(s[j, 0]) * vs[j] for j in range(len(al)))
    psi = psi / psi.norm()
    half = 0.5 * (e[-1] - e[0])
    return h1, eri, dip, psi.reshape(-1).contiguous(), round(1.04 * half + 0.1, 3), \
        round(0.5 * float(e[0] + e[-1]), 3)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return dict(case=case, mom=_moments_of(seed, case["nmoments"]))
    if kind == "batch":
        mols = []
        for i, (n, na, nb) in enumerate(_molecules(case)):
            h1, eri, dip, psi, a, b = _state(n, na, nb, seed * 64 + i)
            mols.append((KPM(h1, eri, dip, n, na, nb, precision="fp64"), psi, a, b))
        return dict(case=case, kpms=[m[0] for m in mols], psis=[m[1] for m in mols],
                    a=[m[2] for m in mols], b=[m[3] for m in mols])
    n, na, nb = case["norb"], case["na"], case["nb"]
    if kind == "moments":
        h1, eri, dip, psi, a, b = _state(n, na, nb, seed)
        return dict(case=case, k=KPM(h1, eri, dip, n, na, nb, precision="fp64"), psi=psi, a=a, b=b)
    h1, eri, dip = _integrals(n, seed)
    if kind == "bounds":
        return dict(case=case, k=KPM(h1, eri, dip, n, na, nb, precision="fp64"), seed=seed)
    k = KPM(h1, eri, dip, n, na, nb, precision=case["prec"])
    if kind == "dipole":
        return dict(case=case, k=k, psi=_vectors(case, seed, 1, torch.float64)[0],
                    y=torch.empty(k.dim, dtype=k.vdtype, device=DEV))
    x = _vectors(case, seed, case["ncol"], k.vdtype)
    return dict(case=case, k=k, x=x, y=torch.empty_like(x))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sigma":
        return state["k"].sigma(state["x"], state["y"])
    if kind == "moments":
        return state["k"].moments(state["psi"], case["mask"], state["a"], state["b"],
                                  case["nmoments"])
    if kind == "batch":
        return moments_batch(state["kpms"], state["psis"], case["mask"], state["a"], state["b"],
                             case["nmoments"])
    if kind == "bounds":
        return state["k"].bounds(case["iters"], state["seed"])
    if kind == "dipole":
        return state["k"].apply_dipole(case["comp"], state["psi"], state["y"])
    om, it = spectrum(state["mom"], SCALE_A, SCALE_B, npoints=case["npoints"],
                      kernel=case["kernel"])
    return dict(omega=om, intensity=it)


# ---------------------------------------------------------------- work

def _sigma_flops(n, na, nb):
    """One H application of one column: off-diagonal excitations of a string, plus its diagonal
    ones as one, by those of the other spin; and the same-spin neighbours of both."""
    dim = math.comb(n, na) * math.comb(n, nb)
    ea, eb = na * (n - na), nb * (n - nb)
    nbr = ea + math.comb(na, 2) * math.comb(n - na, 2) + eb + math.comb(nb, 2) * math.comb(n - nb, 2)
    return 2.0 * dim * ((ea + 1) * (eb + 1) + nbr)


def work(case):
    kind = case["kind"]
    if kind == "spectrum":
        N, M = case["nmoments"], case["npoints"]
        # the sum over moments at every point, in the fewest operations known: a fast transform
        L = 2 * max(N, M)
        return dict(bytes=8.0 * (N + 2 * M), flops=2.5 * L * math.log2(L))
    if kind == "batch":
        flops = nbytes = 0.0
        ncol = bin(case["mask"]).count("1")
        for n, na, nb in _molecules(case):
            dim = math.comb(n, na) * math.comb(n, nb)
            flops += ncol * case["nmoments"] // 2 * (_sigma_flops(n, na, nb) + 8.0 * dim)
            nbytes += 8.0 * (dim + n ** 4 + ncol * case["nmoments"])
        return dict(bytes=nbytes, flops=flops)
    n, na, nb = case["norb"], case["na"], case["nb"]
    dim = math.comb(n, na) * math.comb(n, nb)
    sf = _sigma_flops(n, na, nb)
    if kind == "moments":
        ncol = bin(case["mask"]).count("1")
        return dict(bytes=8.0 * (dim + n ** 4 + ncol * case["nmoments"]),
                    flops=ncol * case["nmoments"] // 2 * (sf + 8.0 * dim))
    if kind == "bounds":
        return dict(bytes=8.0 * (n ** 4 + 2), flops=case["iters"] * (sf + 9.0 * dim))
    esz = 8 if case["prec"] == "fp64" else 4
    if kind == "dipole":
        return dict(bytes=float(dim * (8 + esz)),
                    flops=2.0 * dim * (na * (n - na) + nb * (n - nb) + 1))
    return dict(bytes=2.0 * case["ncol"] * dim * esz + 8.0 * n ** 4, flops=case["ncol"] * sf)


# ---------------------------------------------------------------- 64-bit values in plain torch

class _Strings:
    """One spin's strings: for every unordered pair s = {p, q} of orbitals the string that
    E_pq + E_qp (E_pp on the diagonal) connects each string with, and the sign (0: none)."""

    def __init__(self, n, m):
        masks = np.array([k for k in range(1 << n) if bin(k).count("1") == m], dtype=np.int64)
        rank = np.zeros(1 << n, dtype=np.int64)
        rank[masks] = np.arange(len(masks))
        pairs = [(p, q) for q in range(n) for p in range(q + 1)]
        tgt = np.zeros((len(pairs), len(masks)), dtype=np.int64)
        sgn = np.zeros((len(pairs), len(masks)))
        pop = np.array([bin(k).count("1") for k in range(1 << n)], dtype=np.int64)
        for s, (p, q) in enumerate(pairs):
            bp, bq = (masks >> p) & 1, (masks >> q) & 1
            if p == q:
                tgt[s], sgn[s] = np.arange(len(masks)), bp
                continue
            ok = bp != bq
            between = ((1 << q) - 1) & ~((2 << p) - 1)
            tgt[s] = np.where(ok, rank[np.where(ok, masks ^ (1 << p) ^ (1 << q), masks)], 0)
            sgn[s] = np.where(ok, 1 - 2 * (pop[masks & between] & 1), 0)
        self.ns, self.npair, self.pairs = len(masks), len(pairs), pairs
        self.tgt = torch.tensor(tgt, device=DEV)
        self.sgn = torch.tensor(sgn, device=DEV)


class _Plain:
    """H = sum k_pq E_pq + 1/2 sum (pq|rs) E_pq E_rs in 64 bits, with E over unordered pairs."""

    def __init__(self, h1, eri, n, na, nb):
        self.A = _Strings(n, na)
        self.B = self.A if na == nb else _Strings(n, nb)
        P = self.A.pairs
        k = h1 - 0.5 * np.einsum("pttq->pq", eri)
        self.k = torch.tensor([k[p, q] for p, q in P], device=DEV, dtype=torch.float64)
        self.W = torch.tensor([[eri[p, q, r, s] for r, s in P] for p, q in P], device=DEV,
                              dtype=torch.float64)

    def _own(self, T, x, cross):
        """Rows of x [c, ns] under one spin's operators: (k E + 1/2 E W E) x, and W E x if wanted."""
        c = x.shape[0]
        z = x[:, T.tgt.reshape(-1)].reshape(c, T.npair, T.ns) * T.sgn
        u = torch.matmul(self.W, z)
        y = torch.einsum("s,csj->cj", self.k, z)
        y += 0.5 * (torch.gather(u, 2, T.tgt.expand(c, -1, -1)) * T.sgn).sum(1)
        return y, (u if cross else None)

    def sigma(self, x):
        """x [Na, Nb]."""
        A, B = self.A, self.B
        y = torch.empty_like(x)
        step = max(1, int(6e7 // (B.npair * B.ns)))
        if step >= A.ns:                   # small: gathers only, the same bits every time
            y, u = self._own(B, x, True)
            for s in range(A.npair):
                y += A.sgn[s][:, None] * u[A.tgt[s], s]
        else:
            y.zero_()
            for r in range(0, A.ns, step):
                rows = slice(r, min(r + step, A.ns))
                own, u = self._own(B, x[rows], True)
                y[rows] += own
                for s in range(A.npair):   # (absent targets add zeros to row 0)
                    y.index_add_(0, A.tgt[s, rows], A.sgn[s, rows][:, None] * u[:, s])
        xt = x.t().contiguous()
        yt = torch.empty_like(xt)
        step = max(1, int(6e7 // (A.npair * A.ns)))
        for r in range(0, B.ns, step):
            yt[r:r + step] = self._own(A, xt[r:r + step], False)[0]
        return y + yt.t()

    def dipole(self, d, psi):
        A, B = self.A, self.B
        y = torch.zeros_like(psi)
        for s, (p, q) in enumerate(A.pairs):
            y += float(d[p, q]) * (A.sgn[s][:, None] * psi[A.tgt[s]])
            y += float(d[p, q]) * (psi[:, B.tgt[s]] * B.sgn[s])
        return -y

    def moments(self, d, psi, a, b, nmoments):
        cur = self.dipole(d, psi)
        nxt = (self.sigma(cur) - b * cur) / a
        out = [float((cur * cur).sum()), float((nxt * cur).sum())]
        for _ in range(1, nmoments // 2):
            cur, nxt = nxt, 2.0 * (self.sigma(nxt) - b * nxt) / a - cur
            out += [2.0 * float((cur * cur).sum()) - out[0], 2.0 * float((nxt * cur).sum()) - out[1]]
        return np.array(out)


def _exact_spectrum(case, seed):
    N, M = case["nmoments"], case["npoints"]
    n = np.arange(N)
    mom = _moments_of(seed, N)
    g = np.ones(N)
    if case["kernel"] == "jackson":
        q = math.pi / (N + 1)
        g = ((N - n + 1) * np.cos(q * n) + np.sin(q * n) / math.tan(q)) / (N + 1)
    elif case["kernel"] == "lorentz":
        g = np.sinh(4.0 * (1.0 - n / N)) / math.sinh(4.0)
    w = torch.tensor(g * mom * np.where(n == 0, 1.0, 2.0), device=DEV)
    k = torch.arange(M, device=DEV, dtype=torch.int64)
    acc = torch.zeros(M, device=DEV, dtype=torch.float64)
    step = max(1, int(3e7 // M))
    for lo in range(0, N, step):           # angles reduced in whole numbers: n (2k + 1) mod 4M
        nn = torch.arange(lo, min(lo + step, N), device=DEV, dtype=torch.int64)
        ang = (nn[:, None] * (2 * k + 1)[None, :]) % (4 * M)
        acc += (w[lo:lo + step, None] * torch.cos(ang.double() * (math.pi / (2 * M)))).sum(0)
    th = (k.double() + 0.5) * (math.pi / M)
    om = SCALE_A * torch.cos(th) + SCALE_B
    it = acc / (math.pi * torch.sin(th)) / SCALE_A
    return dict(omega=om.flip(0).cpu().numpy(), intensity=it.flip(0).cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return _exact_spectrum(case, seed)
    if kind == "bounds":
        return None                        # Ritz values of a start vector of the library's own
    if kind in ("moments", "batch"):
        mols = _molecules(case) if kind == "batch" else [(case["norb"], case["na"], case["nb"])]
        out = []
        for i, (n, na, nb) in enumerate(mols):
            h1, eri, dip, psi, a, b = _state(n, na, nb, seed * 64 + i if kind == "batch" else seed)
            H = _Plain(h1, eri, n, na, nb)
            out.append(np.stack([H.moments(dip[c], psi.reshape(H.A.ns, H.B.ns), a, b, case["nmoments"])
                                 for c in range(3) if case["mask"] >> c & 1]))
        return np.stack(out) if kind == "batch" else out[0]
    n, na, nb = case["norb"], case["na"], case["nb"]
    h1, eri, dip = _integrals(n, seed)
    H = _Plain(h1, eri, n, na, nb)
    if kind == "dipole":
        psi = _vectors(case, seed, 1, torch.float64)[0].reshape(H.A.ns, H.B.ns)
        return H.dipole(dip[case["comp"]], psi).reshape(-1)
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    x = _vectors(case, seed, case["ncol"], dt)
    return torch.stack([H.sigma(v.double().reshape(H.A.ns, H.B.ns)).reshape(-1) for v in x])
