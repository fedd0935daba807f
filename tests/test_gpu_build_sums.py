"""The sums of squares that Build's epilogue forms, on both sides of the choice
between its FP32 and FP64 additions (by operand width, kernel function and number
of blocks; 13 tile rows of 1024 are enough blocks on 152 SMs).

They show in the precision map of the K-norm rule, u ||K_ik||_F <= eps ||K||_F / NT:
with eps halfway between the two middle tiles of the order by norm, half of the tiles
are FP16 and half FP32, and a sum off by as little as the gap between those two
(1e-5 of the norm or less) swaps them.  The expected norms are FP64 sums over the
kernel that the library stored (padding rows count as identity rows).
"""
import pytest
import torch

from paper_2409_01712_gb300 import KRR, inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("n,m,tile,kernel,nc", [(1500, 300, 256, "gaussian", 0), (12795, 12160, 1024, "gaussian", 0),
                                                (12795, 12288, 1024, "gaussian", 0), (12795, 16384, 1024, "gaussian", 3),
                                                (12795, 8192, 1024, "ibs", 0)])
def test_tile_norms(n, m, tile, kernel, nc):
    g = inputs.problem(n, m, 1, 1, seed=3 + m, device=DEV)["G"]
    conf = inputs.confounders(n, nc, seed=3, scale=0.1 * m ** 0.5).to(DEV) if nc else None
    # (lambda: FP16 tiles in the first column, which this rule allows, leave the IBS
    # kernel indefinite with 0.1)
    gamma, lam, nt = 1.0 / m, 10.0, (n + tile - 1) // tile
    with KRR(tile=tile, kernel=kernel) as model:
        model.build_kernel(g, gamma, conf=conf)
        k = model.kernel(torch.zeros((n, n), device=DEV))
    sq = torch.zeros((nt, nt), dtype=torch.float64)
    for i in range(nt):
        for j in range(i + 1):
            sq[i, j] = k[i * tile:(i + 1) * tile, j * tile:(j + 1) * tile].double().square().sum()
    total = 2 * torch.tril(sq, -1).sum() + sq.diagonal().sum() + (nt * tile - n)
    low = torch.tril_indices(nt, nt, -1)
    ratio = 2.0 ** -11 * (sq[low[0], low[1]].sqrt() * nt / total.sqrt())
    order = ratio.sort().values
    mid = len(order) // 2
    eps = float((order[mid - 1] + order[mid]) / 2)
    assert order[mid] - order[mid - 1] > 1e-11 * eps
    with KRR(tile=tile, kernel=kernel, prec_rule="knorm", eps=eps) as model:
        model.build_kernel(g, gamma, conf=conf)
        model.factor(lam)
        pmap = torch.as_tensor(model.precision_map())
    got = pmap[low[0], low[1]]
    want = torch.where(ratio <= eps, 2, 1)
    assert torch.equal(got.long(), want), (got.tolist(), want.tolist())
