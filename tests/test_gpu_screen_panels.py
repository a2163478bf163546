"""Screening at the edges of its panels: the 64-column CUDA-core panels (their
factor-and-invert kernel and the two panel products) and the 512-column panels
of the tensor-core precisions, against a dense FP64 solve."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
# FP64: ~n u cond; FP32: ~30 u with eps~ in [1, 9]; split products: the FP32-accumulated
# sums over K blocks of 512 truncate up to ~200 times at 2^-24 each
TOL = {"fp64": 1e-13, "fp32": 2e-6, "f16x3": 2e-5}


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = gw.Context(0)
    yield c
    c.close()


def problem(n_chi, n_w):
    grid = gw.make_grid((12, 12, 12), np.diag([10.26, 10.0, 9.5]))
    gv, _ = gw.g_set(grid, n_chi)
    vh = gw.coulomb_sqrt(grid, gv)
    chi = inputs.screening_chi(n_chi, n_w, rank=max(1, n_chi // 2), seed=7 + n_chi)
    for w in range(n_w):
        x = vh[:, None] * chi[w] * vh
        lam = np.abs(np.linalg.eigvalsh(x)).max()
        chi[w] *= (8.0 if w == 0 else 0.5) / lam if lam > 0 else 1.0
    return grid, gv, vh, chi


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
@pytest.mark.parametrize("n_chi", [1, 2, 17, 63, 64, 65, 127, 130, 511, 513, 577])
def test_panel_edges(ctx, n_chi, prec):
    grid, gv, vh, chi = problem(n_chi, 3)
    d = torch.from_numpy(chi).to("cuda", dtype=gw.cdtype(prec))
    out = torch.full_like(d, float("nan"))
    gw.screen_W(ctx, grid, gv, prec, d, out, resid=False)
    got = out.cpu().numpy().astype(np.complex128)
    eye = np.eye(n_chi)
    for w in range(len(chi)):
        x = vh[:, None] * d[w].cpu().numpy().astype(np.complex128) * vh
        ref = vh[:, None] * np.linalg.solve(eye - x, x) * vh
        norm = np.linalg.norm(ref)
        assert np.linalg.norm(got[w] - ref) <= TOL[prec] * norm if norm else not got[w].any()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "f16x3"])
@pytest.mark.parametrize("col", [5, 64, 100])
def test_bad_pivot_is_named(ctx, col, prec):
    n_chi = 130
    grid, gv, vh, _ = problem(n_chi, 1)
    chi = np.zeros((2, n_chi, n_chi), dtype=np.complex128)
    chi[1, col, col] = 3.0 / vh[col] ** 2              # eps~ = 1 - 3 at that column of the second frequency
    d = torch.from_numpy(chi).to("cuda", dtype=gw.cdtype(prec))
    with pytest.raises(gw.GwError) as e:
        gw.screen_W(ctx, grid, gv, prec, d, torch.empty_like(d), resid=False)
    assert e.value.status == 5 and "column %d of frequency 1" % col in e.value.message
