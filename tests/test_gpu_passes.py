"""The FFT passes at the edges of their dispatch, against the CPU oracle.

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


def host(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy().astype(np.complex128)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# padded lengths 4 .. 1024 on every axis at their smallest and largest extent: planes in one CTA and separate
# passes, columns of 64 .. 512 in two register steps, z passes of 4 .. 32 and 64 .. 512 points and the radix-4
# form (one plane, 1024 points, few complex128 columns)
SHAPES = [(2, 2, 2), (3, 4, 5), (8, 9, 16), (16, 17, 3), (33, 32, 17), (64, 65, 4), (65, 64, 9), (128, 16, 33), (129, 2, 64),
          (3, 128, 65), (2, 129, 5), (130, 140, 8), (257, 3, 2), (3, 258, 2), (5, 6, 129), (4, 3, 256), (2, 3, 257),
          (70, 66, 40)]


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_product_of_every_padded_length(precision, n):
    eps_r, _, x = inputs.random_case(n, seed=sum(n))
    g = vie.Grid(eps_r, H)
    sp = g.spectrum(K0)
    dt = torch.complex128 if precision == vie.C128 else torch.complex64
    y = g.matvec(sp, torch.from_numpy(x).to(device="cuda", dtype=dt))
    assert rel(host(y), omvm.FFTOperator(eps_r, H, K0)(x)) <= (1e-12 if precision == vie.C128 else 1e-5)


@pytest.mark.parametrize("ext", [(17, 20, 3), (20, 12, 17), (18, 5, 33), (33, 18, 6)])
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_batched_blocks_with_the_full_spectrum_layout(precision, ext):
    # two blocks (one smaller, masked voxels) in the batched launches, whose spectra keep the full layout;
    # both sides stop at tau, ||A_k^-1|| <= 10 for |chi| <= 0.7: they differ by at most 20 tau
    nx, ny, nz = ext[0] + 19, ext[1], ext[2]
    eps_r, _, b = inputs.random_case((nx, ny, nz), seed=7 + sum(ext))
    bid = np.full((nz, ny, nx), -1, np.int32)
    bid[:, :, :ext[0]] = 0
    bid[:, :, ext[0] + 1:ext[0] + 18] = 1
    tau = 1e-11 if precision == vie.C128 else 1e-5
    dt = torch.complex128 if precision == vie.C128 else torch.complex64
    P = oprecond.BlockPreconditioner(eps_r, bid, H, K0, inner_tol=1e-12, inner_maxit=500)
    bb = b.astype(np.complex64).astype(np.complex128) if precision == vie.C64 else b
    g = vie.Grid(eps_r, H, bid, inner=vie.INNER_BATCHED)
    y, st = g.precond(g.spectrum(K0), torch.from_numpy(b).to(device="cuda", dtype=dt), inner_tol=tau, inner_maxit=500)
    assert st["nblocks"] == 2 and st["not_converged"] == 0 and st["breakdowns"] == 0
    assert rel(host(y), P(bb)) <= 20 * tau
