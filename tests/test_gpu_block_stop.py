"""When a block solve stops: the same rule in the persistent solver and in the batched launches."""
import numpy as np
import pytest
import torch

from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu

K0 = 2 * np.pi
H = 0.05
DT = {vie.C64: torch.complex64, vie.C128: torch.complex128}


def blocks_of_four(count, contrast, seed):
    """count blocks of 4 x 4 x 4 voxels of permittivity 1 + contrast (0.5 .. 1.5), two voxels apart."""
    rng = np.random.default_rng(seed)
    eps_r = np.ones((4, 4, 6 * count), complex)
    bid = np.full(eps_r.shape, -1, np.int32)
    for k in range(count):
        s = np.s_[:, :, 6 * k:6 * k + 4]
        eps_r[s] += contrast * (0.5 + rng.random((4, 4, 4)))
        bid[s] = k
    return eps_r, bid


@pytest.mark.parametrize("precision,contrast,tau", [(vie.C64, 1e-4, 1e-9), (vie.C64, 3e-4, 1e-10),
                                                    (vie.C128, 1e-8, 1e-18)])
def test_block_stops_on_the_residual_itself(precision, contrast, tau):
    # A = I + E with ||E|| about the contrast c: the residual is c after half an iteration and c^2 after one,
    # above tau, and below it after 1.5. A solver that took ||r||^2 from the difference of ||s||^2 = c^2 and a
    # sum equal to it within rounding would find about zero and stop after one
    eps_r, bid = blocks_of_four(16, contrast, seed=4)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    b = torch.randn((3,) + eps_r.shape, generator=g, dtype=DT[precision], device="cuda")
    for inner in (vie.INNER_BATCHED, vie.INNER_AUTO, vie.INNER_PERSISTENT):
        grid = vie.Grid(eps_r, H, bid, inner=inner)
        _, st = grid.precond(grid.spectrum(K0), b, inner_tol=tau, inner_maxit=50)
        assert st["not_converged"] == 0 and st["breakdowns"] == 0
        assert st["mean_iters"] == 1.5, inner


@pytest.mark.parametrize("inner", [vie.INNER_AUTO, vie.INNER_BATCHED, vie.INNER_PERSISTENT])
@pytest.mark.parametrize("ext", [(6, 5, 4), (18, 17, 4)])
@pytest.mark.parametrize("precision", [vie.C64, vie.C128])
def test_start_that_meets_the_tolerance_is_kept(precision, ext, inner):
    # x = 0 leaves ||b||, within a tolerance of 1 or more: no iteration, whichever solver takes the block
    nx, ny, nz = ext
    eps_r, _, b = inputs.random_case((nx + 1, ny, nz), seed=3)
    bid = np.full((nz, ny, nx + 1), -1, np.int32)
    bid[:, :, :nx] = 0
    b = torch.from_numpy(b).to(device="cuda", dtype=DT[precision])
    grid = vie.Grid(eps_r, H, bid, inner=inner)
    sp = grid.spectrum(K0)
    for tau in (1.0, 1.5):
        y, st = grid.precond(sp, b, inner_tol=tau)
        assert st["max_iters"] == 0 and st["not_converged"] == 0 and st["breakdowns"] == 0
        assert not y[..., :nx].any() and torch.equal(y[..., nx], b[..., nx])
