"""X^T Y of ridge regression on both sides of the choice between the packed and the
general product (8 and 16 columns, 1000 rows), with and without confounders: FP32
sums of at most 2048 terms added in FP64, so each entry is within 2048 u |X|^T |Y| of
the exact one."""
import pytest
import torch

from paper_2409_01712_gb300 import KRR, inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("n,m,p,nc", [(700, 1003, 9, 0), (2500, 1000, 16, 9), (2500, 999, 16, 12), (700, 1003, 17, 0),
                                      (300, 1100, 32, 2), (130, 70, 12, 16)])
def test_xty_routes(n, m, p, nc):
    gen = torch.Generator().manual_seed(n + m + p)
    g = torch.randint(0, 3, (n, m), dtype=torch.int8, generator=gen).to(DEV)
    y = torch.randn((n, p), generator=gen).to(DEV)
    c = inputs.confounders(n, nc, seed=4, scale=1.0).to(DEV) if nc else None
    with KRR(tile=256) as model:
        model.rr_build(g, conf=c)
        rhs = torch.as_tensor(model.rr_rhs(y)).to(DEV).double()
        k = model.kernel(torch.zeros((m + nc, m + nc), device=DEV)).double()
    x = torch.cat([g.double(), c.double()], 1) if nc else g.double()
    u = 2.0 ** -24
    assert ((rhs - x.T @ y.double()).abs() <= 2049 * u * (x.abs().T @ y.double().abs())).all()
    assert ((torch.tril(k) - torch.tril(x.T @ x)).abs() <= 2049 * u * (x.abs().T @ x.abs())).all()
