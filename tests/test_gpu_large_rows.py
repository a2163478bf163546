"""Row transforms with G-set rows too long to be staged in one CTA's shared memory."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw

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
