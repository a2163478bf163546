"""The tensor-core G formation on a k mesh takes the k points in groups where their
operands would outgrow the rest of the call's scratch: the same chi_q with any
group, and no more than twice the scratch of the CUDA-core call, which has none."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


def chi(ctx, p, psi, gv, prec, r_block):
    n = len(p.tau)
    out = torch.full((p.n_k, n, len(gv), len(gv)), float("nan"), dtype=torch.complex64, device="cuda")
    gw.chi0_omega_kmesh(ctx, gw.make_grid(p.n, p.lattice), p.nk, psi, p.eps_k, p.n_occ, p.mu, p.tau, np.eye(n), gv,
                        prec, out, r_block=r_block)
    return out.cpu().numpy()


@pytest.mark.parametrize("r_block", [1, 5, 16, 30])
def test_same_chi_with_any_group(r_block):
    """Split products of the same operands, with the scaling of each k: equal up to FP32 sums."""
    p = inputs.kmesh_problem(n=(6, 6, 6), a=(6.0, 6.5, 7.0), nk=(2, 2, 2), n_occ=4, n_unocc=20, n_tau=2, seed=81)
    gv = gw.g_set(gw.make_grid(p.n, p.lattice), 9)[0]
    psi = torch.from_numpy(p.psi_k).to("cuda", dtype=torch.complex64)
    ctx = gw.Context(0)
    ref = chi(ctx, p, psi, gv, "f16x3", 0)
    got = chi(ctx, p, psi, gv, "f16x3", r_block)
    ctx.close()
    assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref)


def test_scratch_stays_within_twice_the_rest():
    p = inputs.kmesh_problem(n=(12, 12, 12), a=(10.0, 10.0, 10.0), nk=(4, 4, 4), n_occ=8, n_unocc=192, n_tau=1, seed=82)
    gv = gw.g_set(gw.make_grid(p.n, p.lattice), 27)[0]
    psi = torch.from_numpy(p.psi_k).to("cuda", dtype=torch.complex64)
    got, size = {}, {}
    for prec in ("fp32", "f16x3"):
        ctx = gw.Context(0)
        got[prec] = chi(ctx, p, psi, gv, prec, 32)
        size[prec] = ctx.scratch_bytes
        ctx.close()
    assert size["f16x3"] < 2.05 * size["fp32"], size
    assert np.linalg.norm(got["f16x3"] - got["fp32"]) < 5e-6 * np.linalg.norm(got["fp32"])
