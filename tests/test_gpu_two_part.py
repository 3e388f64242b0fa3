"""The unrestricted recovery with fp16 hi + lo parts: badly scaled systems and right-hand sides (a power of two per channel and per
row is taken out before the split), rows of zeros, sizes around the blocks of 128 and on both sides of the two-level blocking."""
import pytest
import torch

from paper_2510_03246_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n,d", [(96, 40), (130, 72), (256, 8), (641, 136), (1000, 264), (6272, 72)])
@pytest.mark.parametrize("spread", [0, 9])
def test_unrestricted_recovery_of_scaled_systems(n, d, spread):
    g = torch.Generator(device=DEV).manual_seed(n + d + spread)
    rand = lambda *s: torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)
    powers = lambda k: torch.exp2(torch.randint(-spread, spread + 1, (k,), generator=g, device=DEV).double())
    mod = api.FfnModule(rand(2 * d, d).bfloat16(), rand(n, d).float(), rand(d, n).float())
    mod.sp_ffn_init()
    # channels and right-hand sides that differ by 2^(2 spread); condition number of the scaled system about 34
    s, r = powers(n), powers(d)
    B = rand(2 * n, n) / (2 * n) ** 0.5
    G = ((B.T @ B) * s[:, None] * s[None, :]).float()
    R = (rand(d, n) * s[None, :] * r[:, None]).float()
    R[d // 2] = 0.0
    mod.G_A.copy_(G)
    mod.R2.copy_(R)
    rho = 1e-9 * float(s.min()) ** 2
    mod.sp_admm_scores(api.AdmmParams(rho=rho, rho_relative=False, k_keep=n))
    mod.check_status()
    G64 = G.double().tril() + G.double().tril(-1).T
    L = torch.linalg.cholesky(G64 / s[:, None] / s[None, :] + torch.diag(rho / s.square()))
    W = torch.cholesky_solve((R.double() / s[None, :]).T, L).T / s[None, :]
    ref = W.square().sum(0).sqrt() * G64.diagonal().sqrt()
    # roundings of fp32 size (2^-24), magnified by the condition number: about ten of them in a small system; in a large one
    # they add up at random over the n terms of a sum, as the root of n
    assert float(((mod.scores.double() - ref).abs() / ref).max()) <= max(10.0, n ** 0.5) * 34 * 2.0 ** -24
