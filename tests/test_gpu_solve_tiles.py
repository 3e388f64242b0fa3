"""Regularised solves in one launch (257 to 12287 unknowns; sizes below are the other form's, at the line between them): sizes around the
tiles of 128, few and many right-hand sides, columns in groups of one, two and four, the widest system, against 64 bits."""
import pytest
import torch

from paper_2510_03246_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _system(n, m, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    B = torch.randn(2 * n, n, generator=g, device=DEV, dtype=torch.float64) / (2 * n) ** 0.5
    G = (B.T @ B).float()                       # condition number about 34: (1 + 2^-1/2)^2 / (1 - 2^-1/2)^2
    return G, torch.randn(m, n, generator=g, device=DEV)


@pytest.mark.parametrize("n,m", [(1, 1), (256, 129), (257, 1), (383, 128), (640, 127), (767, 300), (1024, 129), (1153, 130), (2304, 40),
                                 (5100, 300), (5340, 129), (7680, 300), (8069, 513), (12287, 3)])
def test_solve_around_the_tiles(n, m):
    G, R = _system(n, m, n + m)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    W = api.sp_ridge_solve(R, G, 1e-3, rho_relative=False, status=status)
    assert status.tolist() == [0, 0, 0, 0]
    G64 = G.double().tril() + G.double().tril(-1).T + 1e-3 * torch.eye(n, device=DEV, dtype=torch.float64)
    ref = torch.cholesky_solve(R.double().T, torch.linalg.cholesky(G64)).T
    # roundings of fp32 size, magnified by the condition number: ten of them, or as many as add up at random over n terms
    assert float((W.double() - ref).norm() / ref.norm()) <= max(10.0, n ** 0.5) * 34 * 2.0 ** -24
    assert torch.equal(W, api.sp_ridge_solve(R, G, 1e-3, rho_relative=False))       # a fixed order, whatever the timing


@pytest.mark.parametrize("n,k", [(256, 128), (264, 64), (600, 128), (768, 385), (1160, 577), (5240, 1901), (7928, 3137)])
def test_solution_on_the_kept_support_comes_with_the_factor(n, k):
    """The second of two steps whose mask stays takes the restricted solution from the unrestricted solve: the same as the solve of
    the restricted system by itself."""
    d, N = 136, 2 * n
    g = torch.Generator(device=DEV).manual_seed(n + k)
    rand = lambda *s: torch.randn(*s, generator=g, device=DEV)
    mod = api.FfnModule(rand(N, d).bfloat16(), rand(n, d) * 0.1, rand(d, n) * 0.1)
    mod.sp_ffn_init()
    mod.sp_admm_step(api.AdmmParams(k_keep=k, rho=0.1))
    G, R2 = mod.G_A.clone(), mod.R2.clone()
    mod.sp_admm_step(api.AdmmParams(k_keep=k, rho=0.1, reselect_mask=False))
    mod.check_status()
    assert mod.read_report()["factor_reused"] == 1.0
    W = api.sp_linear_refit(R2, G, mod.mask, k, 0.1, rho_relative=True)
    assert torch.equal(W != 0, mod.W2 != 0)
    # two solves of one system: fp32 roundings magnified by its condition number, at most 1 + n / rho
    assert float((W - mod.W2).norm() / W.norm()) <= 10 * (1 + n / 0.1) * 2.0 ** -24


@pytest.mark.parametrize("n,m", [(300, 40), (1024, 129), (1153, 64)])
@pytest.mark.parametrize("scale", [-112, -116])
def test_systems_of_tiny_entries(n, m, scale):
    """G and R times 2^scale have the solution of G and R, with the same bound: no part of an operand is cut off."""
    G, R = _system(n, m, n + m)
    c = 2.0 ** scale
    W = api.sp_ridge_solve(R * c, G * c, 1e-3 * c, rho_relative=False)
    G64 = G.double().tril() + G.double().tril(-1).T + 1e-3 * torch.eye(n, device=DEV, dtype=torch.float64)
    ref = torch.cholesky_solve(R.double().T, torch.linalg.cholesky(G64)).T
    assert float((W.double() - ref).norm() / ref.norm()) <= max(10.0, n ** 0.5) * 34 * 2.0 ** -24


@pytest.mark.parametrize("n,m,budget", [(1024, 300, 1), (2304, 128, 20000)])
def test_waits_that_run_out_end_the_solve(n, m, budget):
    """With a budget of a few cycles ordinary waits run out (nothing is withheld): the solve reports SP_ERR_TIMEOUT and returns, and the
    next one is the same as the one before."""
    G, R = _system(n, m, n)
    status = torch.zeros(4, dtype=torch.int32, device=DEV)
    W = api.sp_ridge_solve(R, G, 1e-3, rho_relative=False)
    torch.cuda.synchronize()
    assert api.lib().sp_set_wait_budget(budget) == 0
    try:
        for _ in range(4):
            status.zero_()
            api.sp_ridge_solve(R, G, 1e-3, rho_relative=False, status=status)
            torch.cuda.synchronize()
            assert status.tolist()[0] == 7 and status.tolist()[2] == 13
    finally:
        api.lib().sp_set_wait_budget(0)
    status.zero_()
    assert torch.equal(W, api.sp_ridge_solve(R, G, 1e-3, rho_relative=False, status=status))
    assert status.tolist() == [0, 0, 0, 0]
