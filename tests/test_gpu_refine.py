"""The refined solution and the refinement residual against FP64.

Covariates in units of their own: ridge coefficients whose magnitudes lie orders
of magnitude apart, next to each other.  The refined solution's residual stays at
the level of each entry's own rounding: entries off by 1.5 u of themselves
(u = 2^-24), K - c as an FP16 pair (2 u) and FP32 sums of 64 products (8 u, their
random walk) leave 11.5 u || (|K| + |c| + lambda) |beta| ||, and refinement ends
when a step does not halve its residual: twice that.
"""
import pytest
import torch

from paper_2409_01712_gb300 import KRR

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


def test_coefficients_of_very_different_magnitudes():
    n, m, p, lam, tile = 3000, 60, 4, 10.0, 256
    unit = torch.tensor([0.1, 100.0, 1.0])
    gen = torch.Generator().manual_seed(7)
    g = torch.randint(0, 3, (n, m), dtype=torch.int8, generator=gen)
    z = torch.randn((n, 3), generator=gen)
    y = (g.float() @ torch.randn((m, p), generator=gen) * 0.1 + z @ torch.randn((3, p), generator=gen)
         + torch.randn((n, p), generator=gen))
    with KRR(tile=tile) as model:
        model.rr_build(g.to(DEV), conf=(z * unit).to(DEV))
        rhs = model.rr_rhs(y.to(DEV))
        model.factor(lam)
        beta, _ = model.solve(rhs)
        k = torch.as_tensor(model.kernel()).double()
    k = torch.tril(k) + torch.tril(k, -1).T
    beta, rhs = torch.as_tensor(beta).cpu().double(), torch.as_tensor(rhs).cpu().double()
    lam_i = lam * torch.eye(m + 3, dtype=torch.float64)
    # mean off-diagonal entry over the padded rows, the residual's shift
    c = (k.sum() - (m + 3)).abs() / (tile * tile - tile)
    level = 2.0 ** -24 * ((k.abs() + c + lam_i) @ beta.abs()).norm()
    assert (rhs - (k + lam_i) @ beta).norm() <= 23 * level
