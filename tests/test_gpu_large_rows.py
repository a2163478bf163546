"""Row transforms past the sizes of one launch or one CTA's shared memory: G-set rows
too long to be staged, more rows than one launch takes, more tiles per CTA than the
G formation looks up in advance, and the column passes of the 48^3 grid."""
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


def rel(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("n,prec,n_chi", [(36, "fp32", 14080), (36, "fp32", 14081), (36, "fp32", 20001),
                                          (36, "fp32", 46656), (48, "fp32", 14083), (36, "fp64", 7040),
                                          (36, "fp64", 7041)])
def test_rows_on_either_side_of_the_staged_set(ctx, n, prec, n_chi):
    nr, rows = n ** 3, 3
    rng = np.random.default_rng(n_chi)
    idx = rng.permutation(nr)[:n_chi].astype(np.int32)
    grid, dt = gw.make_grid((n,) * 3, np.eye(3) * 20.0), gw.cdtype(prec)
    tol = 1e-6 if prec == "fp32" else 1e-13
    x = rng.standard_normal((rows, nr)) + 1j * rng.standard_normal((rows, nr))
    out = torch.full((rows, n_chi), float("nan"), dtype=dt, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, 1, 1, idx, prec, 0, rows, torch.from_numpy(x).to("cuda", dtype=dt), out)
    assert rel(out.cpu().numpy(), nr * np.fft.ifftn(x.reshape((rows,) + (n,) * 3), axes=(1, 2, 3)).reshape(rows, -1)[:, idx]) < tol
    w = rng.standard_normal((rows, n_chi)) + 1j * rng.standard_normal((rows, n_chi))
    out = torch.full((rows, nr), float("nan"), dtype=dt, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, -1, 1, idx, prec, 0, rows, torch.from_numpy(w).to("cuda", dtype=dt), out)
    y = np.zeros((rows, nr), dtype=np.complex128)
    y[:, idx] = w
    assert rel(out.cpu().numpy(), np.fft.fftn(y.reshape((rows,) + (n,) * 3), axes=(1, 2, 3)).reshape(rows, -1) / 8000.0) < tol


def test_more_rows_than_one_launch(ctx):
    """Long rows go 32768 at a time (backward; forward the workspace holds fewer)."""
    n, rows = (36, 36, 36), 32768 + 130
    grid = gw.make_grid(n, np.eye(3) * 20.0)
    idx = gw.g_set(grid, 33)[1]
    x = torch.randn((rows, 33), dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    out = torch.full((rows, 36 ** 3), float("nan"), dtype=torch.complex64, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, -1, 1, idx, "fp32", 0, rows, x, out)
    for r in (0, 32767, 32768, rows - 1):
        y = np.zeros(36 ** 3, dtype=np.complex128)
        y[idx] = x[r].cpu().numpy()
        assert rel(out[r].cpu().numpy(), np.fft.fftn(y.reshape(n)).reshape(-1) / 8000.0) < 1e-6


@pytest.mark.parametrize("prec", ["f16x3", "fp32"])
def test_chi0_with_every_row_in_one_block(ctx, prec):
    """r_block = N_r at 36^3: 439 tiles per CTA, the row transform of the triangle in two pieces, in
    place.  The same sums as in blocks of the default size."""
    p = inputs.tiny(seed=51, n=(36, 36, 36), a=(20.0, 20.5, 21.0), n_occ=5, n_unocc=27, n_tau=1, n_chi=301)
    grid = gw.make_grid(p.n, p.lattice)
    idx = gw.g_set(grid, p.n_chi)[1]
    psi = torch.from_numpy(p.psi).to("cuda", dtype=torch.complex64)
    got = []
    for r_block in (0, p.n_r):
        chi = torch.full((1, p.n_chi, p.n_chi), float("nan"), dtype=torch.complex64, device="cuda")
        gw.chi0_omega(ctx, grid, psi, p.eps, p.n_occ, p.mu, p.tau, np.eye(1), idx, prec, chi, r_block=r_block)
        got.append(chi.cpu().numpy())
    assert rel(got[1], got[0]) < 1e-6


def test_green_rows_of_a_whole_grid(ctx):
    """All 46656 rows of G_occ at 36^3 in one call: 877 tiles per CTA."""
    p = inputs.tiny(seed=52, n=(36, 36, 36), a=(20.0, 20.5, 21.0), n_occ=5, n_unocc=7, n_tau=1, n_chi=8)
    grid = gw.make_grid(p.n, p.lattice)
    psi = torch.from_numpy(p.psi).to("cuda", dtype=torch.complex64)
    g = torch.empty((p.n_r, p.n_r), dtype=torch.complex64, device="cuda")
    t = float(p.tau[0])
    gw.green_tau(ctx, grid, psi, p.eps, p.n_occ, p.mu, t, 0, p.n_r, "f16x3", g, None)
    c = psi[:p.n_occ].cpu().numpy().astype(np.complex128)
    f = np.exp((p.eps[:p.n_occ] - p.mu) * t)
    for r in (0, 127, 128, 20011, 46463, 46655):
        assert rel(g[r].cpu().numpy(), (c[:, r] * f) @ c.conj()) < 5e-6


def test_columns_of_48cube(ctx):
    n, n_chi = (48, 48, 48), 37
    nr, vol = 48 ** 3, 8000.0
    rng = np.random.default_rng(6)
    idx = rng.permutation(nr)[:n_chi].astype(np.int32)
    grid = gw.make_grid(n, np.eye(3) * 20.0)
    x = (rng.standard_normal((nr, n_chi)) + 1j * rng.standard_normal((nr, n_chi))).astype(np.complex64)
    out = torch.full((n_chi, n_chi), float("nan"), dtype=torch.complex64, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, 1, 2, idx, "fp32", 0, 0, torch.from_numpy(x).to("cuda"), out)
    ref = np.fft.fftn(x.astype(np.complex128).reshape(n + (n_chi,)), axes=(0, 1, 2)).reshape(nr, n_chi)[idx]
    assert rel(out.cpu().numpy(), ref * (vol / nr) ** 2 / vol) < 1e-6
    w = (rng.standard_normal((n_chi, n_chi)) + 1j * rng.standard_normal((n_chi, n_chi))).astype(np.complex64)
    out = torch.full((nr, n_chi), float("nan"), dtype=torch.complex64, device="cuda")
    gw.rr_to_GG_fft(ctx, grid, -1, 2, idx, "fp32", 0, 0, torch.from_numpy(w).to("cuda"), out)
    y = np.zeros((nr, n_chi), dtype=np.complex128)
    y[idx] = w
    ref = nr * np.fft.ifftn(y.reshape(n + (n_chi,)), axes=(0, 1, 2)).reshape(nr, n_chi)
    assert rel(out.cpu().numpy(), ref) < 1e-6
