"""Sizes at the edges of the tiles: the sliced product on pairs of 128-row tiles, the
band groups of the fused self-energy, and rows longer than a CTA's shared memory for
G sets that leave out or scatter over pencils and planes."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = gw.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 128, 31), (128, 127, 32), (129, 64, 33), (255, 65, 64),
                                   (256, 129, 65), (257, 63, 127), (384, 257, 129), (513, 1, 1000)])
def test_sliced_product_edges(ctx, m, n, k):
    """Integer components below 64 are one slice each: the result is exact."""
    rng = np.random.default_rng(m + n + k)
    a, b = (rng.integers(-50, 51, s + (2,)) for s in ((m, k), (k, n)))
    ref = (a[..., 0] @ b[..., 0] - a[..., 1] @ b[..., 1]) + 1j * (a[..., 0] @ b[..., 1] + a[..., 1] @ b[..., 0])
    A, B = (torch.from_numpy(x[..., 0] + 1j * x[..., 1]).to("cuda") for x in (a, b))
    C = torch.full((m, n + 3), 7.0 + 0j, dtype=torch.complex128, device="cuda")
    gw.zgemm_sliced(ctx, A, B, C[:, :n], levels=1)
    assert np.array_equal(C[:, :n].cpu().numpy(), ref)
    assert bool((C[:, n:] == 7).all())


@pytest.mark.parametrize("n_bands", [1, 4, 5, 8, 9, 16, 17, 32])
def test_fused_sigma_band_groups(ctx, n_bands):
    """Split products of 22 bits over 48 bands and 1728 points: well inside 1e-5 of the FP64 path."""
    n, n_chi = (12, 12, 12), 257
    p = inputs.tiny(seed=35, n=n, a=(9.0, 9.5, 10.0), n_occ=6, n_unocc=42, n_tau=3, n_chi=n_chi)
    grid = gw.make_grid(p.n, p.lattice)
    idx = gw.g_set(grid, n_chi)[1]
    rng = np.random.default_rng(9)
    b = rng.standard_normal((n_chi, 20)) + 1j * rng.standard_normal((n_chi, 20))
    w = -np.stack([(b * np.exp(-k)) @ b.conj().T for k in range(3)]) / n_chi
    bands = rng.permutation(48)[:n_bands]
    out = {}
    for prec in ("fp64", "f16x3"):
        dt = gw.cdtype(prec)
        out[prec] = gw.sigma_diag(ctx, grid, torch.from_numpy(p.psi).to("cuda", dtype=dt), p.eps, p.n_occ, p.mu,
                                  bands, p.tau, p.omega, np.eye(3), np.eye(3),
                                  torch.from_numpy(w).to("cuda", dtype=dt), idx, prec)["sigma_iw"]
    assert np.abs(out["f16x3"] - out["fp64"]).max() < 1e-5 * np.abs(out["fp64"]).max()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("which", ["one", "plane", "scattered", "odd"])
def test_long_rows_of_any_set(ctx, which, prec):
    n = (36, 36, 36)
    nr, rows = 36 ** 3, 3
    rng = np.random.default_rng(11)
    idx = {"one": np.array([nr - 1]), "plane": np.arange(36 * 36) + 17 * 36 * 36,
           "scattered": rng.permutation(nr)[:3000], "odd": np.arange(0, nr, 37)[:-1]}[which].astype(np.int32)
    grid = gw.make_grid(n, np.eye(3) * 20.0)
    dt = gw.cdtype(prec)
    tol = 1e-6 if prec == "fp32" else 1e-13
    x = rng.standard_normal((rows, nr)) + 1j * rng.standard_normal((rows, nr))
    out = torch.full((rows, len(idx)), float("nan"), dtype=dt, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, 1, 1, idx, prec, 0, rows, torch.from_numpy(x).to("cuda", dtype=dt), out)
    ref = nr * np.fft.ifftn(x.reshape((rows,) + n), axes=(1, 2, 3)).reshape(rows, -1)[:, idx]
    assert np.linalg.norm(out.cpu().numpy() - ref) < tol * np.linalg.norm(ref)
    w = rng.standard_normal((rows, len(idx))) + 1j * rng.standard_normal((rows, len(idx)))
    out = torch.full((rows, nr), float("nan"), dtype=dt, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, -1, 1, idx, prec, 0, rows, torch.from_numpy(w).to("cuda", dtype=dt), out)
    y = np.zeros((rows, nr), dtype=np.complex128)
    y[:, idx] = w
    ref = np.fft.fftn(y.reshape((rows,) + n), axes=(1, 2, 3)).reshape(rows, -1) / 8000.0
    assert np.linalg.norm(out.cpu().numpy() - ref) < tol * np.linalg.norm(ref)


@pytest.mark.parametrize("direction", [1, -1])
def test_long_rows_beyond_one_chunk(ctx, direction):
    """Forward, the workspace holds 1024 rows at a time."""
    n, rows = (36, 36, 36), 1030
    nr = 36 ** 3
    grid = gw.make_grid(n, np.eye(3) * 20.0)
    idx = gw.g_set(grid, 501)[1]
    gen = torch.Generator(device="cuda").manual_seed(3)
    shape = (rows, nr) if direction > 0 else (rows, 501)
    x = torch.randn(shape, dtype=torch.complex64, device="cuda", generator=gen)
    out = torch.full((rows, 501) if direction > 0 else (rows, nr), float("nan"), dtype=torch.complex64, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, direction, 1, idx, "fp32", 0, rows, x, out)
    for r in (0, 1023, 1024, 1029):
        v = x[r].cpu().numpy().astype(np.complex128)
        if direction > 0:
            ref = nr * np.fft.ifftn(v.reshape(n)).reshape(-1)[idx]
        else:
            y = np.zeros(nr, dtype=np.complex128)
            y[idx] = v
            ref = np.fft.fftn(y.reshape(n)).reshape(-1) / 8000.0
        assert np.linalg.norm(out[r].cpu().numpy() - ref) < 1e-6 * np.linalg.norm(ref)
    assert not bool(torch.isnan(torch.view_as_real(out)).any())
