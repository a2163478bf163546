"""The fused self-energy reads no element of its W~ rows that its own row transform has
not written: the same figures after calls that left NaN in all of the scratch."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,n_chi", [((12, 12, 12), 301), ((16, 16, 16), 700), ((20, 20, 20), 901)])
def test_fused_sigma_over_poisoned_rows(n, n_chi):
    """The matrix self-energy writes whole rows of G and W~ where the fused one keeps its W~ rows."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = inputs.tiny(seed=33, n=n, a=(9.0, 9.5, 10.0), n_occ=5, n_unocc=60, n_tau=3, n_chi=n_chi)
    grid = gw.make_grid(p.n, p.lattice)
    idx = gw.g_set(grid, n_chi)[1]
    rng = np.random.default_rng(9)
    b = rng.standard_normal((n_chi, 20)) + 1j * rng.standard_normal((n_chi, 20))
    w = torch.from_numpy(-np.stack([(b * np.exp(-k)) @ b.conj().T for k in range(3)]) / n_chi).to("cuda", torch.complex64)
    psi = torch.from_numpy(p.psi).to("cuda", dtype=torch.complex64)
    args = (p.eps, p.n_occ, p.mu, p.bands, p.tau, p.omega, np.eye(3), np.eye(3))

    def fused(c):
        return gw.sigma_diag(c, grid, psi, *args, w, idx, "f16x3")["sigma_iw"]

    c = gw.Context(0)
    clean = fused(c)
    bad = gw.sigma_matrix(c, grid, torch.full_like(psi, float("nan")), *args, torch.full_like(w, float("nan")), idx, "f16x3")
    assert np.isnan(bad["sigma_iw"]).all()
    got = fused(c)
    c.close()
    # sums of the same numbers; the order of the tiles' additions in FP64 is free
    assert np.abs(got - clean).max() < 1e-12 * np.abs(clean).max()
