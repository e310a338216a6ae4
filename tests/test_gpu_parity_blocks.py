"""Block solves of the parity-split MVM at the edges of its range, against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import precond as oprecond
from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu

K0 = 2 * np.pi
H = 0.05


def dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype)


def host(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy().astype(np.complex128)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# extents of the blocks: every transform length of the parity-split MVM (2, 4, 6, 8, 10, 12, 16) at its smallest
# and largest extent, alone and with a smaller block of another length in the same group
PAR_EXTENTS = [(1, 1, 1), (2, 1, 3), (3, 4, 2), (5, 6, 7), (8, 7, 5), (9, 10, 11), (12, 11, 9), (13, 16, 14), (16, 16, 16)]


@pytest.mark.parametrize("ext", PAR_EXTENTS)
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_precond_block_extents_match_oracle(precision, ext):
    # tolerance: both sides stop at a relative residual of tau, so they differ by at most 2 tau ||A_k^-1||, with
    # ||A_k^-1|| <= 10 for |chi| <= 0.7 (numerical range of A within [1 - |chi|, ...]); FP32 adds its own
    # residual floor of about 1e-6 per iteration, below tau = 1e-5
    nx, ny, nz = ext[0] + 3, ext[1] + 2, ext[2]
    eps_r, _, b = inputs.random_case((nx, ny, nz), seed=100 + sum(ext))
    bid = np.full((nz, ny, nx), -1, np.int32)
    bid[:ext[2], :ext[1], :ext[0]] = 0
    bid[:, :min(ny, ext[1]), ext[0] + 1:ext[0] + 3] = 1      # two voxels wide, apart from the first
    tau = 1e-11 if precision == vie.C128 else 1e-5
    dt = torch.complex128 if precision == vie.C128 else torch.complex64
    P = oprecond.BlockPreconditioner(eps_r, bid, H, K0, inner_tol=1e-12, inner_maxit=500)
    bb = b.astype(np.complex64).astype(np.complex128) if precision == vie.C64 else b
    ref = P(bb)
    g = vie.Grid(eps_r, H, bid)
    sp = g.spectrum(K0)
    y, st = g.precond(sp, dev(b, dt), inner_tol=tau, inner_maxit=500)
    assert st["nblocks"] == 2 and st["not_converged"] == 0 and st["breakdowns"] == 0
    assert rel(host(y), ref) <= 20 * tau


def test_precond_with_another_grids_spectrum():
    # same shape and group box, other blocks within it: the spectrum of the first grid has no lengths for the
    # second one's smaller block, which then runs with those of the group's box
    n, rng = (12, 12, 12), np.random.default_rng(5)
    eps_r, _, b = inputs.random_case(n, seed=3)
    one = np.full(n, -1, np.int32)
    one[:, :11, :11] = 0
    two = np.full(n, -1, np.int32)
    two[:, :11, :11] = 0
    two[:, 2:11, 2:11] = 1                                    # 9 x 9 x 12, inside the first block's box
    ga, gb = vie.Grid(eps_r, H, one), vie.Grid(eps_r, H, two)
    P = oprecond.BlockPreconditioner(eps_r, two, H, K0, inner_tol=1e-12, inner_maxit=500)
    y, st = gb.precond(ga.spectrum(K0), dev(b), inner_tol=1e-11, inner_maxit=500)
    assert st["nblocks"] == 2 and st["not_converged"] == 0
    assert rel(host(y), P(b)) <= 20 * 1e-11
