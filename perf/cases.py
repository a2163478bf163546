"""The work that users of this framework have it do, as timed cases.

Each case is one call of a public entry point on a seeded synthetic system of
the repository's own recipe (paper_1607_02859_gb300.inputs): orthonormal
orbitals over the lowest n_b plane waves of an n^3 grid, eigenvalues uniform in
an occupied and an unoccupied window with the gap pinned, and the optimised
time / frequency grids with their transform matrices.  The kinds are the stages
of a calculation:

  chi0       chi0(G,G',i omega) from orbitals (gw.chi0_omega)
  chi0_pw    the same with G through its plane-wave form (gw.chi0_omega_pw)
  chi0_k     chi0_q on a k mesh (gw.chi0_omega_kmesh)
  screen     W~(i omega) from chi0(i omega), optionally refined (gw.screen_W)
  tau        W~(i omega) -> W~(i tau) (gw.tau_to_omega with the inverse matrix)
  sigma      Sigma_nn(i omega) from W~(i tau) (gw.sigma_diag)

Orbitals, tables and the output buffer are what a program has in hand; the
library context (scratch arena) is one per process, as in a program.
"""
import functools
import math

import numpy as np
import torch

from paper_1607_02859_gb300 import gw

DEV = "cuda:0"


def listed():
    return [
        # the smallest system: a 12^3 cell with 128 real orbitals in single precision, where launches count
        dict(name="chi0_toy", kind="chi0", n=12, n_b=128, n_occ=16, n_tau=8, n_chi=1728, real=True, prec="fp32"),
        # the same cell in the double precision that a user checks results with
        dict(name="chi0_toy_fp64", kind="chi0", n=12, n_b=128, n_occ=16, n_tau=8, n_chi=1728, real=True, prec="fp64"),
        # an ordinary request to the server: a 20^3 cell, 512 bands, 12 times
        dict(name="chi0_mix", kind="chi0", n=20, n_b=512, n_occ=64, n_tau=12, n_chi=1536, real=False, prec="f16x3"),
        # an eight-atom cell at full band count, ragged G set, few times
        dict(name="chi0_si8", kind="chi0", n=24, n_b=1024, n_occ=16, n_tau=8, n_chi=4097, real=False, prec="f16x3"),
        # the 64-atom cell (36^3, 4224 bands): the size the framework is built for, two of its times
        dict(name="chi0_si64", kind="chi0", n=36, n_b=4224, n_occ=128, n_tau=2, n_chi=8192, real=False, prec="f16x3"),
        # the 64-atom cell through the plane-wave form of G
        dict(name="chi0_pw_si64", kind="chi0_pw", n=36, n_b=4224, n_occ=128, n_tau=2, n_chi=8192, real=False,
             prec="f16x3"),
        # a small cell on a 2x2x2 k mesh (24^3 supercell)
        dict(name="chi0_kmesh", kind="chi0_k", n=12, nk=2, n_b=96, n_occ=12, n_tau=6, n_chi=509, real=False,
             prec="f16x3"),
        # screening of the server's systems: many small frequencies
        dict(name="screen_mix", kind="screen", n=20, n_chi=1536, n_tau=12, refine=0, prec="f16x3"),
        # screening of the 64-atom cell with one refinement step, two of its frequencies
        dict(name="screen_si64", kind="screen", n=36, n_chi=8192, n_tau=2, refine=1, prec="f16x3"),
        # back to imaginary time at 20 points
        dict(name="tau_20", kind="tau", n=24, n_chi=2048, n_tau=20, prec="f16x3"),
        # the self-energy of an ordinary request: 4 bands around the gap
        dict(name="sigma_mix", kind="sigma", n=20, n_b=512, n_occ=64, n_tau=12, n_chi=1536, n_n=4, real=False,
             prec="f16x3"),
        # the self-energy of the 64-atom cell: 32 bands, two of its times
        dict(name="sigma_si64", kind="sigma", n=36, n_b=4224, n_occ=128, n_tau=2, n_chi=8192, n_n=32, real=False,
             prec="f16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chi0", "chi0", "chi0", "chi0_pw", "chi0_k", "screen", "screen", "tau", "sigma", "sigma"])
    if kind == "screen":
        refine = rng.choice([0, 0, 1])
        n_chi = _log(rng, 256, 6000)
        return dict(kind=kind, n=24, n_chi=n_chi, n_tau=rng.randint(1, 2) if n_chi > 3000 else rng.randint(2, 16),
                    refine=refine, prec=rng.choice(["f16x3", "f16x3", "f16x3", "fp32"]) if n_chi < 2000 and not refine
                    else "f16x3")
    if kind == "tau":
        return dict(kind=kind, n=20, n_chi=_log(rng, 200, 2100), n_tau=rng.randint(4, 24),
                    prec=rng.choice(["f16x3", "f16x3", "fp32"]))
    if kind == "chi0_k":
        n, nk = rng.choice([(6, 2), (8, 2), (12, 2), (4, 3)])
        n_b = rng.randint(24, min(120, n ** 3))
        return dict(kind=kind, n=n, nk=nk, n_b=n_b, n_occ=max(2, n_b // 8), n_tau=rng.randint(4, 8),
                    n_chi=rng.randint(min(40, n ** 3), min(n ** 3, 600)), real=False,
                    prec=rng.choice(["f16x3", "f16x3", "fp32"]))
    n = rng.choice([12, 16, 20, 24, 36] if kind != "chi0_pw" else [16, 20, 24, 36])
    prec = rng.choice(["f16x3", "f16x3", "f16x3", "fp32"]) if n < 24 else "f16x3"
    n_b = _log(rng, 100, {12: 512, 16: 768, 20: 1024, 24: 1100, 36: 4300}[n])
    c = dict(kind=kind, n=n, n_b=n_b, n_occ=max(4, n_b // rng.choice([8, 16, 32])),
             n_tau=rng.randint(1, 2) if n == 36 else rng.randint(4, 9) if n == 24 else rng.randint(6, 16),
             n_chi=_log(rng, 400, min(n ** 3, 2000 if n < 24 else 5000)), real=kind == "chi0" and n == 12 and rng.random() < 0.5,
             prec=prec)
    if kind == "sigma":
        c["n_n"] = rng.randint(1, 32)
    return c


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=1)
def _ctx():
    return gw.Context(0)


def _seed(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + case["n"])
    return g, np.random.default_rng([int(seed), case["n"], case["n_chi"]])


def _triples(n):
    """Integer triples in [-n/2, n/2)^3 ordered by (|g|^2, g1, g2, g3), and their FFT positions."""
    ax = np.arange(-(n // 2), n - n // 2)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    g = g[np.lexsort((g[:, 2], g[:, 1], g[:, 0], (g ** 2).sum(1)))]
    m = g % n
    return g, (m[:, 0] * n + m[:, 1]) * n + m[:, 2]


def _cell(case):
    return case["n"] * 10.26 / 18 if case["n"] == 36 else case["n"] * 10.26 / 24 if case["n"] == 24 else case["n"] * 10.26 / 12


def _cdt(case):
    return torch.complex128 if case["prec"] == "fp64" else torch.complex64


def _orthonormal(m, gen, dt):
    z = torch.randn((m, m), generator=gen, device=DEV, dtype=dt)
    return torch.linalg.qr(z)[0]


def _orbitals(case, gen):
    """psi [n_b][N_r], orthonormal over the lowest plane waves (or their cos / sin pairs)."""
    n, n_b, dt = case["n"], case["n_b"], _cdt(case)
    nr, vol = n ** 3, _cell(case) ** 3
    g, pos = _triples(n)
    if case["real"]:
        u = _orthonormal(n_b, gen, torch.float64).T.contiguous().to(torch.complex128)
        spec = torch.zeros((n_b, nr), dtype=torch.complex128, device=DEV)
        seen, col = set(), 0
        for t in map(tuple, g.tolist()):
            if col >= n_b:
                break
            if t in seen or any(2 * x == -n for x in t):
                continue
            neg = tuple(-x for x in t)
            seen.update((t, neg))
            p = [((x[0] % n) * n + x[1] % n) * n + x[2] % n for x in (t, neg)]
            if t == neg:
                spec[:, p[0]] += u[:, col]
                col += 1
                continue
            for f in (1.0, -1j):             # sqrt2 cos(G.r), sqrt2 sin(G.r)
                if col < n_b:
                    a = u[:, col] * (f / math.sqrt(2.0))
                    spec[:, p[0]] += a
                    spec[:, p[1]] += a.conj()
                    col += 1
        psi = torch.fft.ifftn(spec.reshape(n_b, n, n, n), dim=(1, 2, 3)).real * (nr / math.sqrt(vol))
        return psi.reshape(n_b, nr).to(dt).contiguous()
    u = _orthonormal(n_b, gen, dt)
    psi = torch.empty((n_b, nr), dtype=dt, device=DEV)
    ix = torch.from_numpy(pos[:n_b].copy()).to(DEV)
    for b in range(0, n_b, 512):
        e = min(n_b, b + 512)
        spec = torch.zeros((e - b, nr), dtype=dt, device=DEV)
        spec[:, ix] = u[b:e]
        psi[b:e] = torch.fft.ifftn(spec.reshape(e - b, n, n, n), dim=(1, 2, 3)).reshape(e - b, nr) * (nr / math.sqrt(vol))
    return psi


MU = 0.015


def _energies(case, rng, n_k=1):
    """Eigenvalues [n_k][n_b] with the gap [0, 0.03] Ha pinned at every k."""
    o, u = case["n_occ"], case["n_b"] - case["n_occ"]
    eo, eu = np.sort(rng.uniform(-0.5, 0.0, (n_k, o)), 1), np.sort(rng.uniform(0.03, 5.0, (n_k, u)), 1)
    eo[:, -1], eu[:, 0] = 0.0, 0.03
    return np.concatenate([eo, eu], 1)


def _grids(case):
    """Optimised time / frequency grids and transform matrices of the window the energies are drawn from."""
    return _grids_of(case["n_tau"])


@functools.lru_cache(maxsize=64)
def _grids_of(n_tau):
    x_min, x_max = MU, 5.5 + 5.0
    g = gw.mp2_grids(n_tau, x_min, x_max)
    return g["tau"], g["omega"], gw.fit_transform(g["tau"], g["omega"], x_min, x_max, 4000, 0.0)


def _grid(case):
    return gw.make_grid((case["n"],) * 3, np.diag([_cell(case)] * 3))


def _vhalf(case, n_chi):
    """sqrt(4 pi)/|G| over the G set, 0 at G = 0."""
    g = 2 * np.pi / _cell(case) * np.linalg.norm(_triples(case["n"])[0][:n_chi], axis=1)
    return np.where(g > 0, math.sqrt(4 * math.pi) / np.where(g > 0, g, 1.0), 0.0)


def _hermitian_sums(case, gen, weights):
    """[len(weights)][n_chi][n_chi] Hermitian -B diag(w_j) B^H with rows damped along the G set as pair
    densities are, scaled to unit largest diagonal element at the first weight vector."""
    m, rank = case["n_chi"], weights.shape[1]
    b = torch.randn((m, rank), generator=gen, device=DEV, dtype=torch.complex64)
    b *= (1.0 / (1.0 + torch.arange(m, device=DEV) / 64.0))[:, None]
    out = torch.empty((len(weights), m, m), dtype=torch.complex64, device=DEV)
    s = 0.0
    for j, w in enumerate(weights):
        x = -(b * torch.from_numpy(w).to(DEV, torch.float32)) @ b.mH
        s = s or 1.0 / float(x.diagonal().real.abs().max())
        out[j] = (x + x.mH) * (0.5 * s)
    return out


def _screened(case, gen, grid_points, of):
    """Hermitian matrices with poles at rank/8 energies Omega_p in [0.2, 3] Ha: of(Omega, point) gives the weights."""
    om = np.geomspace(0.2, 3.0, max(16, case["n_chi"] // 8))
    return _hermitian_sums(case, gen, np.array([of(om, x) for x in grid_points]))


def _inputs(case, seed):
    """The tensors and tables of a case, from the seed alone."""
    gen, rng = _seed(case, seed)
    tau, omega, mats = _grids(case)
    s = dict(case=case, tau=tau, omega=omega, mats=mats, prec=case["prec"])
    kind = case["kind"]
    if kind == "screen":
        chi = _screened(case, gen, omega, lambda o, w: o / (o * o + w * w))
        vh = torch.from_numpy(_vhalf(case, case["n_chi"])).to(DEV, torch.float32)
        v = torch.randn(case["n_chi"], generator=gen, device=DEV, dtype=torch.complex64)
        for _ in range(8):                   # largest eigenvalue of v^1/2 chi v^1/2 to about 8
            v = vh * (chi[0] @ (vh * v))
            lam = float(v.norm())
            v /= lam
        s["chi"] = chi * (8.0 / lam)
    elif kind == "tau":
        s["w"] = _screened(case, gen, omega, lambda o, w: o / (o * o + w * w))
    elif kind == "chi0_k":
        nk, n, n_b = case["nk"], case["n"], case["n_b"]
        x = torch.arange(n, device=DEV, dtype=torch.float64) / n
        psi = []
        for k in range(nk ** 3):
            kk = (k // (nk * nk), k // nk % nk, k % nk)
            e = [torch.exp(2j * math.pi * kk[d] / nk * x) for d in range(3)]
            ph = (e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]).reshape(-1)
            psi.append((_orbitals(case, gen) * ph).to(_cdt(case)))
        s["psi"], s["eps"] = torch.stack(psi), _energies(case, rng, nk ** 3)
    else:
        s["psi"], s["eps"] = _orbitals(case, gen), _energies(case, rng)[0]
        if kind == "sigma":
            s["w"] = _screened(case, gen, tau, lambda o, t: o * np.exp(-o * t))
            h = max(0, case["n_occ"] - case["n_n"] // 2)
            s["bands"] = np.arange(h, h + case["n_n"])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["ctx"], s["grid"] = _ctx(), _grid(case)
    s["gvec"], s["idx"] = gw.g_set(s["grid"], case["n_chi"])
    m, nw, kind = case["n_chi"], case["n_tau"], case["kind"]
    if kind == "chi0_pw":
        s["pw"] = gw.g_set(s["grid"], case["n_b"])[1]
    shape = (case["nk"] ** 3, nw, m, m) if kind == "chi0_k" else (nw, m, m)
    if kind != "sigma":
        s["out"] = torch.empty(shape, dtype=_cdt(case), device=DEV)
    return s


def run(s):
    c, k, p = s["case"], s["case"]["kind"], s["prec"]
    if k == "chi0":
        gw.chi0_omega(s["ctx"], s["grid"], s["psi"], s["eps"], c["n_occ"], MU, s["tau"], s["mats"]["C"], s["idx"], p,
                      s["out"])
    elif k == "chi0_pw":
        gw.chi0_omega_pw(s["ctx"], s["grid"], s["psi"], s["eps"], c["n_occ"], MU, s["tau"], s["mats"]["C"], s["idx"],
                         s["pw"], p, s["out"])
    elif k == "chi0_k":
        gw.chi0_omega_kmesh(s["ctx"], s["grid"], (c["nk"],) * 3, s["psi"], s["eps"], c["n_occ"], MU, s["tau"],
                            s["mats"]["C"], s["gvec"], p, s["out"])
    elif k == "screen":
        gw.screen_W(s["ctx"], s["grid"], s["gvec"], p, s["chi"], s["out"], resid=False, refine=c["refine"])
    elif k == "tau":
        gw.tau_to_omega(s["ctx"], gw.CT, s["mats"]["Cinv"], s["w"], s["out"], p)
    else:
        return gw.sigma_diag(s["ctx"], s["grid"], s["psi"], s["eps"], c["n_occ"], MU, s["bands"], s["tau"], s["omega"],
                             s["mats"]["C"], s["mats"]["S"], s["w"], s["idx"], p)
    return s["out"]


def work(case):
    """Inputs and outputs once; the flops of the method with what its Hermitian results allow (half of G)."""
    m, nw, kind = case["n_chi"], case["n_tau"], case["kind"]
    es = 16 if case["prec"] == "fp64" else 8
    mats = nw * m * m * es
    if kind == "screen":
        return dict(bytes=2 * mats, flops=nw * (4.0 + 8.0 * case["refine"]) * m ** 3)
    if kind == "tau":
        return dict(bytes=2 * mats, flops=4.0 * nw * nw * m * m)
    nr, nb = case["n"] ** 3, case["n_b"]
    fft = nw * (nr + m) * 5.0 * nr * math.log2(nr)
    psi = nb * nr * es
    if kind == "chi0_k":
        q = case["nk"] ** 3
        ns = nr * q                          # points of the supercell
        return dict(bytes=q * (psi + mats),
                    flops=nw * (8.0 * nr * nr * nb * q + (nr + m) * 5.0 * ns * math.log2(ns)))
    if kind == "chi0_pw":
        return dict(bytes=psi + mats, flops=nw * (4.0 * nb ** 3 + (2 * nr + 2 * nb) * 5.0 * nr * math.log2(nr)) + fft)
    if kind == "chi0":
        return dict(bytes=psi + mats, flops=nw * 4.0 * nr * nr * nb + fft)
    return dict(bytes=psi + mats, flops=nw * (4.0 * nr * nr * nb + 8.0 * nr * nr * case["n_n"]) + fft)


# ------------------------------------------------------------------ 64-bit values

def _rows(n, spectrum, sign):
    """sum_g x(g) exp(sign i g.r) over the last axis [.., n^3] of a full-grid spectrum."""
    x = spectrum.reshape(-1, n, n, n)
    x = torch.fft.fftn(x, dim=(1, 2, 3)) if sign < 0 else torch.fft.ifftn(x, dim=(1, 2, 3)) * float(n ** 3)
    return x.reshape(len(spectrum), n ** 3)


def _columns(n, a, pos, sign):
    """[N_r][cols] of sum_g exp(sign i g.r) a(g, col), the rows g of `a` sitting at FFT positions `pos`."""
    out = torch.empty((n ** 3, a.shape[1]), dtype=torch.complex128, device=DEV)
    for b in range(0, a.shape[1], 1024):
        x = torch.zeros((min(1024, a.shape[1] - b), n ** 3), dtype=torch.complex128, device=DEV)
        x[:, pos] = a[:, b:b + 1024].T
        out[:, b:b + 1024] = _rows(n, x, sign).T
    return out


def _expand(n, t, pos, sign):
    """Rows t(r, g') -> sum_g' t(r, g') exp(sign i g'.R') for a block of rows."""
    x = torch.zeros((t.shape[0], n ** 3), dtype=torch.complex128, device=DEV)
    x[:, pos] = t
    return _rows(n, x, sign)


def _green_factors(s, psi, eps, pos):
    """Per tau: the column-transformed plane-wave matrices T(r, g') of G_occ and G_unocc."""
    n, o = s["case"]["n"], s["case"]["n_occ"]
    c = torch.empty((len(psi), len(pos)), dtype=torch.complex128, device=DEV)
    for b in range(0, len(psi), 512):
        x = torch.fft.fftn(psi[b:b + 512].to(torch.complex128).reshape(-1, n, n, n), dim=(1, 2, 3))
        c[b:b + 512] = x.reshape(-1, n ** 3)[:, pos] / n ** 3
    e = torch.from_numpy(eps - MU).to(DEV)
    for tau in s["tau"]:
        f = torch.exp(torch.where(torch.arange(len(eps), device=DEV) < o, e * tau, -e * tau))
        yield [_columns(n, (c[sl].T * f[sl]) @ c[sl].conj(), pos, +1) for sl in (slice(0, o), slice(o, None))]


def _basis(case):
    """FFT positions of the plane waves that span the orbitals."""
    g, pos = _triples(case["n"])
    return torch.from_numpy(pos[:case["n_b"] * (2 if case["real"] else 1) + 64].copy()).to(DEV) if case["real"] \
        else torch.from_numpy(pos[:case["n_b"]].copy()).to(DEV)


def exact(case, seed):
    s, kind, n, m = _inputs(case, seed), case["kind"], case["n"], case["n_chi"]
    c128, chunk = torch.complex128, 1024
    if kind == "tau":
        mat = torch.from_numpy(s["mats"]["Cinv"]).to(DEV, c128)
        x = s["w"].reshape(case["n_tau"], -1)
        return torch.cat([mat @ p.to(c128) for p in x.split(1 << 22, 1)], 1).reshape(s["w"].shape)
    if kind == "screen":
        vh = torch.from_numpy(_vhalf(case, m)).to(DEV)
        out = torch.empty(s["chi"].shape, dtype=c128, device=DEV)
        eye = torch.eye(m, dtype=c128, device=DEV)
        for j, x in enumerate(s["chi"]):
            low = torch.tril(x.to(c128), -1)
            x = vh[:, None] * (low + low.mH + torch.diag(x.diagonal().real.to(c128))) * vh
            out[j] = vh[:, None] * (torch.linalg.solve(eye - x, x)) * vh
        return out
    idx = torch.from_numpy(_triples(n)[1][:m].copy()).to(DEV)
    nr, vol = n ** 3, _cell(case) ** 3
    dv, mats = vol / nr, {k: torch.from_numpy(np.asarray(v)).to(DEV) for k, v in s["mats"].items() if k in "CS"}
    if kind == "chi0_k":
        return _exact_kmesh(s, idx, mats["C"], dv, vol)
    pos = _basis(case)
    if kind == "sigma":
        psi = s["psi"][torch.from_numpy(s["bands"]).to(DEV)].to(c128)
        su, so = (torch.zeros((case["n_n"], case["n_tau"]), dtype=torch.float64, device=DEV) for _ in range(2))
        for j, (to, tu) in enumerate(_green_factors(s, s["psi"], s["eps"], pos)):
            tw = _columns(n, s["w"][j].to(c128), idx, +1)
            for r in range(0, nr, chunk):
                w = _expand(n, tw[r:r + chunk], idx, -1) * (dv * dv / vol)
                for t, acc, sign in ((tu, su, 1.0), (to, so, -1.0)):
                    v = (_expand(n, t[r:r + chunk], pos, -1) * w) @ psi.T
                    acc[:, j] += sign * (psi[:, r:r + chunk].T.conj() * v).real.sum(0)
            del tw, to, tu
        iw = ((su + so) / 2) @ mats["C"].T + 1j * (((su - so) / 2) @ mats["S"].T)
        return {"sigma_unocc": su, "sigma_occ": so, "sigma_iw": iw}
    out = torch.zeros((case["n_tau"], m, m), dtype=c128, device=DEV)
    for j, (to, tu) in enumerate(_green_factors(s, s["psi"], s["eps"], pos)):
        x = torch.empty((nr, m), dtype=c128, device=DEV)
        for r in range(0, nr, chunk):
            chi = -2.0 * _expand(n, to[r:r + chunk], pos, -1) * _expand(n, tu[r:r + chunk], pos, -1).conj()
            x[r:r + chunk] = _rows(n, chi, +1)[:, idx]
        _to_omega(out, x, n, idx, mats["C"][:, j], dv * dv / vol)
    return out


def _to_omega(out, x, n, idx, weights, scale):
    """out[k] += weights[k] scale sum_r exp(-i G.r) x(r, G')."""
    for b in range(0, x.shape[1], 512):
        y = _rows(n, x[:, b:b + 512].T.contiguous(), -1)[:, idx].T * scale
        for k in range(len(out)):
            out[k][:, b:b + 512] += weights[k] * y


def _exact_kmesh(s, idx, C, dv, vol):
    case, c128 = s["case"], torch.complex128
    n, nk, o, m = case["n"], case["nk"], case["n_occ"], case["n_chi"]
    nr, q3, big = n ** 3, nk ** 3, n * nk
    ks = [(k // (nk * nk), k // nk % nk, k % nk) for k in range(q3)]
    gv = _triples(n)[0][:m]
    x1 = torch.arange(n, device=DEV, dtype=torch.float64) / n
    out = torch.zeros((q3, case["n_tau"], m, m), dtype=c128, device=DEV)
    psi, eps = s["psi"].to(c128), torch.from_numpy(s["eps"] - MU).to(DEV)
    for j, tau in enumerate(s["tau"]):
        g = []
        for sl, sg in ((slice(0, o), 1.0), (slice(o, None), -1.0)):
            st = torch.zeros((nr, nk, n, nk, n, nk, n), dtype=c128, device=DEV)
            for k, kk in enumerate(ks):
                a = psi[k][sl]
                gk = ((a.T * torch.exp(sg * eps[k][sl] * tau)) @ a.conj()).reshape(nr, n, n, n) / q3
                for L in ks:
                    ph = np.exp(-2j * np.pi * sum(kk[d] * L[d] for d in range(3)) / nk)
                    st[:, L[0], :, L[1], :, L[2], :] += complex(ph) * gk
            g.append(st.reshape(nr, -1))
        chi = -2.0 * g[0] * g[1].conj()
        x = torch.cat([_rows(big, p, +1) for p in chi.split(256)])
        for k, kk in enumerate(ks):
            p = [torch.from_numpy((kk[d] + nk * gv[:, d]) % big).to(DEV) for d in range(3)]
            e = [torch.exp(-2j * math.pi * kk[d] / nk * x1) for d in range(3)]
            ph = (e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]).reshape(-1)
            _to_omega(out[k], ph[:, None] * x[:, (p[0] * big + p[1]) * big + p[2]], n, idx, C[:, j], dv * dv / vol)
    return out
