"""Edges of the split residual, the sweeps' column padding, the diagonal step's
chain and the ridge products, against FP64.

Refinement: A of a refined solve against FP64 Cholesky of the kernel the library
stored, to the 1e-4 that mixed-mode solutions are held to.  Sizes: one row, one
tile, a tile split in parts (few items for the SMs), more than 48 tile rows
(several source tiles an item, a short last group), and 1, 16, 17, 32 and 33
right-hand sides (the padded column counts and a second column chunk).

Diagonal step: the factor of a single tile (plain FP32 mode: no other kernel
takes part) reproduces K + lambda I to the FP32 Cholesky bound
||L L^T - A||_F <= (b + 1) u ||L||_F^2, u = 2^-24 (Higham, Theorem 10.3); the two
substitutions, products with the explicit inverse, match FP64 substitution with
the same factor to 8 b u cond(L): each product and each inverse contributes at
most 2 b u cond(L) to first order.

Ridge products: X^T C in the Gram matrix and X^T Y are FP32 sums of at most 2048
terms added in FP64, so each entry is within 2048 u |X|^T |B| of the exact one.
"""
import pytest
import torch

from paper_2409_01712_gb300 import KRR, inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("n,tile,p", [(1, 256, 1), (250, 256, 17), (2048, 256, 16), (5000, 1024, 2), (2500, 1024, 33),
                                      (12600, 256, 3), (13100, 256, 32)])
def test_refined_solution_matches_fp64(n, tile, p):
    m, lam = 200, 0.1
    prob = inputs.problem(n, m, p, 1, seed=77 + n + p, device=DEV)
    with KRR(tile=tile, mode="mixed") as model:
        model.build_kernel(prob["G"], 1.0 / m)
        model.factor(lam)
        a, _ = model.solve(prob["Y"])
        k = torch.as_tensor(model.kernel()).to(DEV).double()
    k = torch.tril(k) + torch.tril(k, -1).T
    k.diagonal().add_(lam)
    want = torch.cholesky_solve(prob["Y"].double(), torch.linalg.cholesky(k))
    assert (a.double() - want).norm() <= 1e-4 * want.norm()


def test_zero_and_late_columns():
    """A column of zeros solves to zeros, and a column that is zero up to some
    row and tiny after it (the scale of a zero block does not suit it) to the
    same accuracy as the others."""
    n, m, lam, tile = 1500, 200, 0.1, 256
    prob = inputs.problem(n, m, 4, 1, seed=9, device=DEV)
    prob["Y"][:, 1] = 0.0
    prob["Y"][:700, 2] = 0.0
    prob["Y"][700:, 2] *= 1e-6
    with KRR(tile=tile, mode="mixed") as model:
        model.build_kernel(prob["G"], 1.0 / m)
        model.factor(lam)
        a, _ = model.solve(prob["Y"])
        k = torch.as_tensor(model.kernel()).to(DEV).double()
    k = torch.tril(k) + torch.tril(k, -1).T
    k.diagonal().add_(lam)
    want = torch.cholesky_solve(prob["Y"].double(), torch.linalg.cholesky(k))
    assert torch.count_nonzero(a[:, 1]) == 0
    for q in (0, 2, 3):
        assert (a[:, q].double() - want[:, q]).norm() <= 1e-4 * want[:, q].norm()


@pytest.mark.parametrize("tile", [256, 512, 1024, 2048])
def test_diagonal_step_of_one_tile(tile):
    n, m, lam = tile - 3, 300, 0.1
    prob = inputs.problem(n, m, 4, 1, seed=tile, device=DEV)
    with KRR(tile=tile, mode="fp32") as model:
        model.build_kernel(prob["G"], 1.0 / m)
        model.factor(lam)
        a, _ = model.solve(prob["Y"])
        k = torch.as_tensor(model.kernel()).to(DEV).double()
        low = torch.tril(torch.as_tensor(model.factor_matrix()).to(DEV).double())
    full = torch.tril(k) + torch.tril(k, -1).T + lam * torch.eye(n, device=DEV, dtype=torch.float64)
    u = 2.0 ** -24
    assert (low @ low.T - full).norm() <= (tile + 1) * u * low.norm() ** 2
    cond = torch.linalg.cond(low)
    x = torch.cholesky_solve(prob["Y"].double(), low)
    assert (a.double() - x).norm() <= 8 * tile * u * cond * x.norm()


@pytest.mark.parametrize("n,m,p,nc,pad", [(1, 1, 1, 0, 0), (130, 65, 8, 3, 1), (513, 300, 9, 16, 0), (3001, 130, 17, 5, 3),
                                          (2050, 64, 33, 0, 4)])
def test_ridge_products(n, m, p, nc, pad):
    """Row edges of the transposing pack (pad: extra columns of the genotype
    rows, so that rows are 4-byte aligned or not) and column edges of the
    packed products."""
    gen = torch.Generator().manual_seed(5 + n + m)
    wide = torch.randint(0, 3, (n, m + pad), dtype=torch.int8, generator=gen).to(DEV)
    g = wide[:, :m]
    yy = torch.randn((n, p), generator=gen).to(DEV)
    c = inputs.confounders(n, nc, seed=3, scale=1.0).to(DEV) if nc else None
    with KRR(tile=256, mode="mixed") as model:
        model.rr_build(g, conf=c)
        rhs = torch.as_tensor(model.rr_rhs(yy)).to(DEV).double()
        k = torch.as_tensor(model.kernel()).to(DEV).double()
    x = g.double()
    if nc:
        x = torch.cat([x, c.double()], 1)
    u = 2.0 ** -24
    y = yy.double()
    assert ((rhs - x.T @ y).abs() <= 2049 * u * (x.abs().T @ y.abs())).all()
    gram = torch.tril(x.T @ x)
    assert (torch.equal(torch.tril(k)[:m, :m], gram[:m, :m]))
    assert ((torch.tril(k) - gram).abs() <= 2049 * u * (x.abs().T @ x.abs())).all()
