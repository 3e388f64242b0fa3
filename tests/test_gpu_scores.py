"""Wanda scores at the edges of their grid: column groups of 128 that are partly filled, one to eight row blocks per column group,
units inside and across column groups, rows that are not 16-byte aligned; against the definition in fp64."""
import pytest
import torch

from paper_2510_03246_b200 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("kind", [api.SP_SCORE_WANDA_L2, api.SP_SCORE_WANDA_L1])
@pytest.mark.parametrize("rows,units,group,pad", [
    (1, 1, 1, 0), (7, 130, 1, 0), (9, 127, 1, 1), (64, 128, 1, 4), (65, 257, 1, 3), (530, 43, 3, 0), (96, 12, 64, 0),
    (40, 5, 200, 0), (33, 20000, 1, 0), (12, 80000, 1, 0)])
def test_wanda_scores_at_grid_edges(kind, rows, units, group, pad):
    g = torch.Generator(device=DEV).manual_seed(rows * 1000 + units)
    cols = units * group
    W = torch.randn(rows, cols + pad, generator=g, device=DEV)[:, :cols]
    colsq = torch.rand(cols, generator=g, device=DEV) + 0.5
    colabs = (torch.rand(cols, generator=g, device=DEV) + 0.5).double()
    # twice: the second call follows the first without a host synchronisation between their kernels
    for _ in range(2):
        scores, imp, _ = api.sp_struct_scores(kind, units, group, W=W, colsq=colsq, colabs=colabs, inv_tokens=0.25)
    Wd = W.double()
    if kind == api.SP_SCORE_WANDA_L2:
        ref = (Wd.square().sum(0) * colsq.double()).view(units, group).sum(1).sqrt()
    else:
        ref = (Wd.abs().sum(0) * colabs * 0.25).view(units, group).sum(1)
    # fp64 sums rounded to fp32 once: 2^-24, and the fp64 roundings of a few thousand terms
    assert torch.all((scores.double() - ref).abs() <= ref * (2.0 ** -24 + 1e-12))
    assert abs(float(imp) - float(scores.double().mean())) <= 1e-12 * float(scores.double().mean())
