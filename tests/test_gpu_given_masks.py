"""Given masks that do not keep the announced number of units: reported, nothing is read or written out of place, and the weights are
those of the units that the mask keeps."""
import pytest
import torch

from paper_2510_03246_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _spd(n, g):
    B = torch.randn(2 * n, n, generator=g, device=DEV, dtype=torch.float64) / (2 * n) ** 0.5
    return (B.T @ B).float()


@pytest.mark.parametrize("precise", [False, True])
@pytest.mark.parametrize("units,group,k,kept", [(96, 1, 40, 33), (300, 2, 200, 1), (48, 8, 48, 0)])
def test_refit_on_fewer_units_than_announced(units, group, k, kept, precise):
    """The list of kept units is as long as announced and names units throughout, whatever the workspace held before."""
    n, m = units * group, 24
    g = torch.Generator(device=DEV).manual_seed(n + k)
    G, R = _spd(n, g), torch.randn(m, n, generator=g, device=DEV)
    mask = torch.zeros(units, dtype=torch.uint8, device=DEV)
    mask[torch.randperm(units, generator=g, device=DEV)[:kept]] = 1
    ws = api._ws(api.workspace_bytes(api.SP_WS_LINEAR_REFIT, m, n, 0, 0, api.SP_F64 if precise else api.SP_F32), R.device)
    ws.fill_(0x7f)                                   # as a list of units: far out of range
    W = torch.full_like(R, 7.0)
    api.sp_linear_refit(R, G, mask, k, 0.5, group=group, precise=precise, W=W, ws=ws)
    torch.cuda.synchronize()
    assert torch.isfinite(W).all()
    cols = mask.bool().repeat_interleave(group)
    first = torch.arange(n, device=DEV) < group      # what an empty mask's list names
    assert torch.all(W[:, ~(cols | first)] == 0)


@pytest.mark.parametrize("kept", [0, 100, 300, 301, 302, 520])
def test_w1_of_a_mask_of_another_size(kept):
    """W1 is R1 (G_X + rho I)^-1 on the units that the mask keeps and zero elsewhere."""
    d, n, N, k = 136, 520, 768, 301
    g = torch.Generator(device=DEV).manual_seed(kept)
    rand = lambda *s: torch.randn(*s, generator=g, device=DEV)
    mod = api.FfnModule(rand(N, d).bfloat16(), rand(n, d) * 0.1, rand(d, n) * 0.1, overlap_k=k)
    mod.sp_ffn_init()
    mod.mask.zero_()
    mod.mask[torch.randperm(n, generator=g, device=DEV)[:kept]] = 1
    G, R1 = mod.G_X.double(), mod.R1.double()
    mod._workspace(0).fill_(0x7f)
    mod.W1.fill_(7.0)
    mod.sp_admm_step(api.AdmmParams(k_keep=k, rho=0.1, reselect_mask=False, skip_scores=True))
    assert mod.status.tolist()[:2] == ([2, kept] if kept != k else [0, 0])      # SP_ERR_SHAPE, units kept
    G = G.tril() + G.tril(-1).T
    inv = torch.linalg.inv(G + 0.1 * G.diagonal().mean() * torch.eye(d, device=DEV, dtype=torch.float64))
    ref = R1 @ inv
    keep = mod.mask.bool()
    assert torch.all(mod.W1[~keep] == 0)
    # the inverse rounded to fp32, six part products without terms below 2^-23: a few roundings per term, at random over d terms
    bound = 8 * d ** 0.5 * 2.0 ** -24 * (R1.abs() @ inv.abs())
    assert bool(((mod.W1.double() - ref).abs() <= bound)[keep].all())


@pytest.mark.parametrize("kept", [302, 315, 520])
@pytest.mark.parametrize("act", ["relu", "gated", "dual"])
@pytest.mark.parametrize("overlap", [False, True])
def test_step_on_more_units_than_announced(kept, act, overlap):
    """The units beyond the announced number have no column among the kept ones' products: they are updated like pruned ones."""
    d, n, N, k = 136, 520, 768, 301
    g = torch.Generator(device=DEV).manual_seed(kept)
    rand = lambda *s: torch.randn(*s, generator=g, device=DEV)
    mod = api.FfnModule(rand(N, d).bfloat16(), rand(n, d) * 0.1, rand(d, n) * 0.1, dual_mode=act == "dual", overlap_k=k if overlap else 0,
                        Wg_0=rand(n, d) * 0.1 if act == "gated" else None)
    mod.sp_ffn_init()
    mod.mask.zero_()
    mod.mask[torch.randperm(n, generator=g, device=DEV)[:kept]] = 1
    beyond = torch.nonzero(mod.mask).flatten()[k:]
    z = mod.Z.clone()
    mod._workspace(0).fill_(0x7f)
    mod.sp_admm_step(api.AdmmParams(k_keep=k, rho=0.1, reselect_mask=False, skip_scores=True, dual_mode=act == "dual"))
    assert mod.status.tolist()[:2] == [2, kept]      # SP_ERR_SHAPE, units kept
    # z1 = 0 and a = phi(z) there; one product, one sum and one quotient of fp32
    want = torch.where(z < 0, 0.0, z / 2) if act != "gated" else mod.Gate.square() * z / (mod.Gate.square() + 1)
    assert float((mod.Z - want).abs()[:, beyond].max()) <= 4 * 2.0 ** -24 * float(z.abs().max())
    assert torch.isfinite(mod.Z).all() and torch.isfinite(mod.W1).all()
