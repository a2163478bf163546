"""The rows that are formed and transformed only for R' <= r, and the pencils that
the passes skip because the G set does not touch them: chi0 (every precision) and
the fused self-energy against the FP64 library path and the oracle's definition,
for G sets that are spheres, ragged, one-sided and single points."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {"fp64": 1e-12, "fp32": 1e-6, "f16x3": 5e-6}


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = gw.Context(0)
    yield c
    c.close()


def sets(n):
    nr = int(np.prod(n))
    rng = np.random.default_rng(5)
    sphere = gw.g_set(gw.make_grid(n, np.eye(3) * 8.0), max(1, nr // 5))[1]
    return {"sphere": sphere, "odd": sphere[:max(1, len(sphere) // 2 * 2 - 1)], "one": np.array([nr - 1]),
            "scattered": rng.permutation(nr)[:nr // 3], "plane": np.arange(n[1] * n[2]) + (n[0] - 1) * n[1] * n[2],
            "whole": rng.permutation(nr)}


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
@pytest.mark.parametrize("n", [(4, 4, 4), (6, 4, 6), (8, 6, 10), (12, 12, 12)])
@pytest.mark.parametrize("r_block", [0, 1, 37])
def test_chi0_of_any_set(ctx, n, prec, r_block):
    p = inputs.tiny(seed=31, n=n, n_occ=3, n_unocc=12, n_tau=3)
    grid = gw.make_grid(p.n, p.lattice)
    nr, dt = p.n_r, gw.cdtype(prec)
    psi = torch.from_numpy(p.psi).to("cuda", dtype=dt)
    if r_block == 1 and nr > 200:
        pytest.skip("one launch per row: small grids only")
    C = np.random.default_rng(3).uniform(-1, 1, (3, 3))
    c = psi.cpu().numpy().astype(np.complex128)
    e = p.eps - p.mu
    i = np.indices(n).reshape(3, -1)
    for name, idx in sets(n).items():
        out = torch.full((3, len(idx), len(idx)), float("nan"), dtype=dt, device="cuda")
        gw.chi0_omega(ctx, grid, psi, p.eps, p.n_occ, p.mu, p.tau, C, idx, prec, out, r_block=r_block)
        g = np.stack([idx // (n[1] * n[2]), idx // n[2] % n[1], idx % n[2]])
        ph = np.exp(2j * np.pi * sum(np.outer(g[d], i[d]) / n[d] for d in range(3)))      # [G][r]
        per = []
        for t in p.tau:
            go = (c[:p.n_occ].T * np.exp(e[:p.n_occ] * t)) @ c[:p.n_occ].conj()
            gu = (c[p.n_occ:].T * np.exp(-e[p.n_occ:] * t)) @ c[p.n_occ:].conj()
            per.append((p.volume / nr) ** 2 / p.volume * ph.conj() @ (-2 * go * gu.conj()) @ ph.T)
        ref = np.einsum("kj,jab->kab", C, np.array(per))
        err = np.linalg.norm(out.cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err < TOL[prec], (name, err)


@pytest.mark.parametrize("n,n_chi", [((12, 12, 12), 301), ((16, 16, 16), 700), ((20, 20, 20), 901)])
def test_fused_sigma_reads_only_what_is_written(ctx, n, n_chi):
    """The fused self-energy reads W~(r, R') as far as its tiles reach; the rest of
    the rows is not written, so what an earlier call left there must not show."""
    p = inputs.tiny(seed=33, n=n, a=(9.0, 9.5, 10.0), n_occ=5, n_unocc=60, n_tau=3, n_chi=n_chi)
    grid = gw.make_grid(p.n, p.lattice)
    idx = gw.g_set(grid, n_chi)[1]
    rng = np.random.default_rng(9)
    b = rng.standard_normal((n_chi, 20)) + 1j * rng.standard_normal((n_chi, 20))
    w = -np.stack([(b * np.exp(-k)) @ b.conj().T for k in range(3)]) / n_chi
    C, S = np.eye(3), np.eye(3)
    out = {}
    for prec in ("fp64", "f16x3"):
        dt = gw.cdtype(prec)
        psi = torch.from_numpy(p.psi).to("cuda", dtype=dt)
        c2 = gw.Context(0)
        bad = torch.full((3, n_chi, n_chi), float("nan"), dtype=dt, device="cuda")
        try:                                       # leaves NaN rows of W~ in the context's scratch
            gw.sigma_diag(c2, grid, psi, p.eps, p.n_occ, p.mu, p.bands, p.tau, p.omega, C, S, bad, idx, prec)
        except gw.GwError:
            pass
        out[prec] = gw.sigma_diag(c2, grid, psi, p.eps, p.n_occ, p.mu, p.bands, p.tau, p.omega, C, S,
                                  torch.from_numpy(w).to("cuda", dtype=dt), idx, prec)["sigma_iw"]
        c2.close()
    scale = np.abs(out["fp64"]).max()
    assert np.abs(out["f16x3"] - out["fp64"]).max() < 1e-5 * scale
