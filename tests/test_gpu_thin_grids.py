"""Products of grids with a single plane, row or column, against the CPU oracle.

Tolerances as for the other products: complex128 1e-12, complex64 1e-5."""
import numpy as np
import pytest
import torch

from oracle import mvm as omvm
from oracle import precond as oprecond
from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu

K0 = 2 * np.pi
H = 0.05
DT = {vie.C64: torch.complex64, vie.C128: torch.complex128}
SHAPES = [(1, 1, 1), (17, 1, 1), (1, 40, 1), (40, 30, 1), (130, 9, 1), (9, 130, 1), (70, 140, 1), (300, 7, 1),
          (1, 33, 20), (1, 64, 5), (1, 300, 3), (2, 260, 3), (1, 1, 70)]


def rel(a, b):
    torch.cuda.synchronize()
    return float(np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_product_of_a_thin_grid(precision, n):
    eps_r, _, x = inputs.random_case(n, seed=sum(n))
    g = vie.Grid(eps_r, H)
    y = g.matvec(g.spectrum(K0), torch.from_numpy(x).to(device="cuda", dtype=DT[precision]))
    assert rel(y, omvm.FFTOperator(eps_r, H, K0)(x)) <= (1e-12 if precision == vie.C128 else 1e-5)


@pytest.mark.parametrize("ext", [(20, 18, 1), (1, 18, 20), (1, 40, 1)])
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_thin_blocks_in_the_batched_launches(precision, ext):
    # full layout of the spectrum; both sides stop at tau, ||A_k^-1|| <= 10 for |chi| <= 0.7: they differ by at most
    # 20 tau
    nx, ny, nz = ext[0] + 3, ext[1], ext[2]
    eps_r, _, b = inputs.random_case((nx, ny, nz), seed=9 + sum(ext))
    bid = np.full((nz, ny, nx), -1, np.int32)
    bid[:, :, :ext[0]] = 0
    bid[:, :, ext[0] + 1:ext[0] + 1 + min(2, ext[0])] = 1
    tau = 1e-11 if precision == vie.C128 else 1e-5
    P = oprecond.BlockPreconditioner(eps_r, bid, H, K0, inner_tol=1e-12, inner_maxit=500)
    bb = b.astype(np.complex64).astype(np.complex128) if precision == vie.C64 else b
    g = vie.Grid(eps_r, H, bid, inner=vie.INNER_BATCHED)
    y, st = g.precond(g.spectrum(K0), torch.from_numpy(b).to(device="cuda", dtype=DT[precision]), inner_tol=tau,
                      inner_maxit=500)
    assert st["nblocks"] == 2 and st["not_converged"] == 0 and st["breakdowns"] == 0
    assert rel(y, P(bb)) <= 20 * tau
