"""The refined solution and the refinement residual against FP64.

Covariates in units of their own: ridge coefficients whose magnitudes lie orders
of magnitude apart, next to each other.  The refined solution's residual stays at
the level of each entry's own rounding: entries off by 1.5 u of themselves
(u = 2^-24), K - c as an FP16 pair (2 u) and FP32 sums of 64 products (8 u, their
random walk) leave 11.5 u || (|K| + |c| + lambda) |beta| ||, and refinement ends
when a step does not halve its residual: twice that.

The residual where its items are parts of tiles and where they are groups of
tiles, and in a second chunk of columns.  It is formed from (K - c) a with K - c an
FP16 pair (2 u) and FP32 sums of 64 products (up to 64 u of a sum, if every
addition truncates the same way); rows and chunks are independent, so its error is
at most 66 u || (K - c)_ij a_j ||_F.  A refined solution's own residual is at most
what independent FP32 roundings of A leave, u (||K||_F / sqrt(n) + lambda) ||A||_F,
plus the random walk of that evaluation, 10 u || (K - c)_ij a_j ||_F.

The substitutions with a single tile's inverse, unrefined, against FP64 with the
stored factor, to the 2e-5 that the sweeps over several tiles are held to: the rows
of the inverse, their FP16 split and their transposed use, at every tile edge.
"""
import pytest
import torch

from paper_2409_01712_gb300 import KRR, inputs

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


@pytest.mark.parametrize("n,tile,p", [(1000, 1024, 1), (5000, 1024, 2), (12600, 256, 3), (13100, 256, 33)])
def test_residual_matches_fp64(n, tile, p):
    m, lam, u = 200, 0.1, 2.0 ** -24
    prob = inputs.problem(n, m, p, 1, seed=31 + n, device=DEV)
    with KRR(tile=tile) as model:
        model.build_kernel(prob["G"], 1.0 / m)
        model.factor(lam)
        a, info = model.solve(prob["Y"])
        k = torch.as_tensor(model.kernel()).to(DEV).double()
    k = torch.tril(k) + torch.tril(k, -1).T
    a, y = a.double(), prob["Y"].double()
    pad = (n + tile - 1) // tile * tile
    c = (k.sum() - n) / (pad * pad - pad)
    true = (y - k @ a - lam * a).norm() / y.norm()
    level = u * (k.norm() / n ** 0.5 + lam) * a.norm() / y.norm()
    spread = ((k - c).square() @ a.square()).sum().sqrt() / y.norm()
    assert abs(info["rel_residual"] - true) <= 66 * u * spread
    assert true <= level + 10 * u * spread


@pytest.mark.parametrize("mode", ["mixed", "fp32"])
@pytest.mark.parametrize("tile", [256, 512, 1024, 2048])
def test_substitutions_of_one_tile(tile, mode):
    n, m, lam = tile - 3, 300, 0.1
    prob = inputs.problem(n, m, 4, 1, seed=tile, device=DEV)
    with KRR(tile=tile, mode=mode, ir_max=0) as model:
        model.build_kernel(prob["G"], 1.0 / m)
        model.factor(lam)
        a, _ = model.solve(prob["Y"], raise_on_noconv=False)
        low = torch.tril(torch.as_tensor(model.factor_matrix()).to(DEV).double())
    want = torch.cholesky_solve(prob["Y"].double(), low)
    assert (a.double() - want).norm() <= 2e-5 * want.norm()
