"""A time-out that any tensor-core G formation of a call records is reported at the
end of the call, also when more operands were prepared after it, and the next call
starts clean.  The time-out is set on the host (gw_ctx_inject_timeout)."""
import numpy as np
import pytest

from paper_1607_02859_gb300 import gw, inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
N = (6, 6, 6)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = gw.Context(0)
    yield c
    c.close()


def dev(a, dt=torch.complex64):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype=dt)


def calls(ctx):
    """name -> (call, G formations in it)"""
    p = inputs.tiny(seed=61, n=N, n_occ=4, n_unocc=20, n_tau=3, n_chi=40)
    grid = gw.make_grid(p.n, p.lattice)
    gv, idx = gw.g_set(grid, p.n_chi)
    pw = np.arange(p.n_r, dtype=np.int32)
    psi, nt = dev(p.psi), len(p.tau)
    C, S, om = np.eye(nt), np.eye(nt), np.asarray(p.omega)
    chi = torch.empty((nt, p.n_chi, p.n_chi), dtype=torch.complex64, device="cuda")
    w = -torch.eye(p.n_chi, dtype=torch.complex64, device="cuda").repeat(nt, 1, 1)
    row = torch.empty((p.n_r, p.n_r), dtype=torch.complex64, device="cuda")
    a = (ctx, grid, psi, p.eps, p.n_occ, p.mu)
    many = np.arange(34) % p.n_b
    plan = gw.Chi0Plan(ctx, grid, p.n_b, p.eps, p.n_occ, p.mu, p.tau, C, idx, "f16x3", r_block=100)

    def planned():
        plan.launch(psi, chi)
        plan.status()

    q = inputs.kmesh_problem(n=N, a=(6.0, 6.5, 7.0), nk=(2, 2, 2), n_occ=3, n_unocc=9, n_tau=2, seed=62, n_chi=30)
    qgrid = gw.make_grid(q.n, q.lattice)
    qgv = gw.g_set(qgrid, 30)[0]
    psi_k, nq = dev(q.psi_k), len(q.tau)
    D = np.eye(nq)
    chi_k = torch.empty((q.n_k, nq, 30, 30), dtype=torch.complex64, device="cuda")
    w_k = -torch.eye(30, dtype=torch.complex64, device="cuda").repeat(q.n_k, nq, 1, 1)
    b = (ctx, qgrid, q.nk, psi_k, q.eps_k, q.n_occ, q.mu)
    all_k = np.arange(int(np.prod(N)), dtype=np.int32)
    return {
        "green_tau": (lambda: gw.green_tau(*a, float(p.tau[0]), 0, p.n_r, "f16x3", row, None), 1),
        "chi0_rtau_fused": (lambda: gw.chi0_rtau_fused(*a, float(p.tau[0]), 0, p.n_r, "f16x3", row), 1),
        "chi0_omega": (lambda: gw.chi0_omega(*a, p.tau, C, idx, "f16x3", chi, r_block=100), 3),
        "chi0_plan": (planned, 3),
        "chi0_omega_pw": (lambda: gw.chi0_omega_pw(*a, p.tau, C, idx, pw, "f16x3", chi), 3),
        "sigma_diag": (lambda: gw.sigma_diag(*a, [2, 3], p.tau, om, C, S, w, idx, "f16x3"), 3),
        "sigma_diag_unfused": (lambda: gw.sigma_diag(*a, many, p.tau, om, C, S, w, idx, "f16x3"), 3),
        "sigma_matrix": (lambda: gw.sigma_matrix(*a, [2, 3], p.tau, om, C, S, w, idx, "f16x3"), 3),
        "sigma_diag_pw": (lambda: gw.sigma_diag_pw(*a, [2, 3], p.tau, om, C, S, w, idx, pw, "f16x3"), 3),
        "chi0_kmesh": (lambda: gw.chi0_omega_kmesh(*b, q.tau, D, qgv, "f16x3", chi_k, r_block=100), 6),
        "chi0_kmesh_pw": (lambda: gw.chi0_omega_kmesh_pw(*b, q.tau, D, qgv, all_k, "f16x3", chi_k), 16),
        "sigma_kmesh": (lambda: gw.sigma_diag_kmesh(*b, [(2, 0), (3, 1)], q.tau, q.omega, D, D, w_k, qgv, "f16x3"), 2),
    }


NAMES = ["green_tau", "chi0_rtau_fused", "chi0_omega", "chi0_plan", "chi0_omega_pw", "sigma_diag",
         "sigma_diag_unfused", "sigma_matrix", "sigma_diag_pw", "chi0_kmesh", "chi0_kmesh_pw", "sigma_kmesh"]


@pytest.fixture(scope="module")
def table(ctx):
    return calls(ctx)


@pytest.mark.parametrize("name", NAMES)
def test_a_time_out_in_any_product_is_reported(ctx, table, name):
    call, products = table[name]
    for product in range(1, products + 1):
        ctx.inject_timeout(product)
        with pytest.raises(gw.GwError) as e:
            call()
        assert e.value.status == 6, (name, product)
        ctx.inject_timeout(0)
        call()
