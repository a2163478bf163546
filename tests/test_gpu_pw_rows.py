"""Plane-wave chi rows on both sides of the one-CTA form (two rows in 72 KB: up to 16^3
in FP32, 12^3 in FP64) for G sets and plane-wave sets that touch few, many or all
columns, against dense sums."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {"fp64": 1e-12, "fp32": 1e-6, "f16x3": 5e-6}


def sets(n):
    nr = int(np.prod(n))
    rng = np.random.default_rng(5)
    sphere = gw.g_set(gw.make_grid(n, np.eye(3) * 8.0), min(150, nr // 5))[1]
    return {"sphere": sphere, "one": np.array([nr - 1]), "scattered": rng.permutation(nr)[:min(131, nr // 3)],
            "plane": np.arange(n[2] * 2) + (n[0] - 1) * n[1] * n[2], "many": rng.permutation(nr)[:min(nr, 600)]}


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
@pytest.mark.parametrize("n", [(4, 4, 4), (6, 4, 6), (8, 6, 10), (12, 12, 12), (16, 16, 16), (20, 20, 20)])
def test_pw_chi0_of_any_set(n, prec):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    if n[0] == 20 and prec == "fp64":
        pytest.skip("dense sums of the other precisions are enough at 20^3")
    ctx = gw.Context(0)
    p = inputs.tiny(seed=37, n=n, n_occ=3, n_unocc=12, n_tau=2)
    grid = gw.make_grid(p.n, p.lattice)
    nr, dt = p.n_r, gw.cdtype(prec)
    psi = torch.from_numpy(p.psi).to("cuda", dtype=dt)
    C = np.random.default_rng(3).uniform(-1, 1, (2, 2))
    c = psi.to(torch.complex128)
    e = torch.from_numpy(p.eps - p.mu).to("cuda")
    i = np.indices(n).reshape(3, -1)
    support = np.abs(np.fft.fftn(p.psi.reshape((-1,) + n), axes=(1, 2, 3))).reshape(len(p.psi), -1).max(0)
    lowest = np.flatnonzero(support > 1e-10 * support.max()).astype(np.int32)
    chi = []
    for t in p.tau:
        go = (c[:p.n_occ].T * torch.exp(e[:p.n_occ] * t)) @ c[:p.n_occ].conj()
        gu = (c[p.n_occ:].T * torch.exp(-e[p.n_occ:] * t)) @ c[p.n_occ:].conj()
        chi.append(-2 * go * gu.conj() * ((p.volume / nr) ** 2 / p.volume))
    for name, idx in sets(n).items():
        g = np.stack([idx // (n[1] * n[2]), idx // n[2] % n[1], idx % n[2]])
        ph = torch.from_numpy(np.exp(2j * np.pi * sum(np.outer(g[d], i[d]) / n[d] for d in range(3)))).to("cuda")
        per = torch.stack([ph.conj() @ x @ ph.T for x in chi]).cpu().numpy()
        ref = np.einsum("kj,jab->kab", C, per)
        for pw in (lowest, np.random.default_rng(8).permutation(nr).astype(np.int32)) if nr <= 480 else (lowest,):
            out = torch.full((2, len(idx), len(idx)), float("nan"), dtype=dt, device="cuda")
            gw.chi0_omega_pw(ctx, grid, psi, p.eps, p.n_occ, p.mu, p.tau, C, idx, pw, prec, out)
            err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
            assert err < TOL[prec], (name, len(pw), err)
    ctx.close()
