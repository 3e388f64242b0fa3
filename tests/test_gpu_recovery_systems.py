"""The recoveries on planted systems: channels and right-hand sides that differ by powers of two, rows of zeros, sizes around the
blocks of 128, and systems whose solution shows the rounding of the factor's products magnified a thousand times."""
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


def _pairs(n, d, gap):
    """Channels i and i + n/2 coupled by l, every pair for itself: the factor has l below its diagonal blocks, and what the second
    channel's pivot keeps is gap out of l^2 + gap.  l = 1 + 2^-12 + 2^-23 has bits at both ends of a fp32 mantissa.  The right-hand
    sides are small enough that W W^T, the a-update's system, is far below the identity that is added to it."""
    l = 1.0 + 2.0 ** -12 + 2.0 ** -23
    h = n // 2
    G = torch.eye(n, dtype=torch.float64, device=DEV)
    i = torch.arange(h, device=DEV)
    G[i, i + h] = G[i + h, i] = l
    G[i + h, i + h] = float(torch.tensor(l * l + gap).float())
    R = torch.zeros(d, n, dtype=torch.float64, device=DEV)
    R[:, h:] = torch.exp2(((torch.arange(d, device=DEV)[:, None] + i[None, :]) % 3 - 16).double())
    W = torch.empty_like(R)                     # R G^-1: the first channel's right-hand sides are zero
    W[:, h:] = R[:, h:] / (G[-1, -1] - l * l)
    W[:, :h] = -l * W[:, h:]
    return G, R, W


@pytest.mark.parametrize("scores_only", [True, False])
def test_products_of_the_factor_keep_all_bits_of_fp32(scores_only):
    """The unrestricted recovery, and the recovery on the kept support from its factor: l^2 within three roundings of 2^-24 (the
    product, its last part, the difference), magnified by 1 / gap.  Operands cut to 22 bits are off by 5 * 2^-24."""
    n, d, gap = 1024, 24, 2.0 ** -10
    G, R, W = _pairs(n, d, gap)
    g = torch.Generator(device=DEV).manual_seed(7)
    rand = lambda *s: torch.randn(*s, generator=g, device=DEV)
    mod = api.FfnModule(rand(64, d).bfloat16(), rand(n, d), rand(d, n))
    mod.sp_ffn_init()
    mod.G_A.copy_(G)
    mod.R2.copy_(R)
    # whole pairs are kept; with the kept channels in front the two of a pair are still two blocks of 128 apart
    keep = torch.arange(n, device=DEV) % 2 == 0
    mod.mask.copy_(keep)
    prm = api.AdmmParams(rho=2.0 ** -60, rho_relative=False, k_keep=n // 2, reselect_mask=False)
    bound = 3 * 2.0 ** -24 / gap
    if scores_only:
        mod.sp_admm_scores(api.AdmmParams(rho=2.0 ** -60, rho_relative=False, k_keep=n))
    else:
        mod.sp_admm_step(prm)
    mod.check_status()
    ref = W.square().sum(0).sqrt() * G.diagonal().sqrt()
    assert float(((mod.scores.double() - ref).abs() / ref).max()) <= bound
    if not scores_only:
        assert int(mod.read_report()["factor_reused"]) == 1
        assert float(((mod.W2.double() - W).abs()[:, keep] / W.abs()[:, keep]).max()) <= bound
        assert torch.all(mod.W2[:, ~keep] == 0)
