"""Launches of the persistent block solver beside those of boxes of at most 16 voxels per axis: the
shared-memory passes with the tuner's launch shapes, and grids with blocks of both kinds."""
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


def row_of_blocks(boxes, seed):
    """One box of random permittivity per block, side by side along x."""
    nx, ny, nz = sum(b[0] + 1 for b in boxes), max(b[1] for b in boxes), max(b[2] for b in boxes)
    eps_r, _, b = inputs.random_case((nx, ny, nz), seed=seed)
    bid = np.full((nz, ny, nx), -1, np.int32)
    x = 0
    for k, (ex, ey, ez) in enumerate(boxes):
        bid[:ez, :ey, x:x + ex] = k
        x += ex + 1
    return eps_r, bid, b


def check_every_block(grid, eps_r, bid, b, precision, tau, applies, seen):
    sp = grid.spectrum(K0)
    bd = torch.from_numpy(b).to(device="cuda", dtype=DT[precision])
    bb = bd.cpu().numpy().astype(np.complex128)
    blocks = oprecond.find_blocks(bid)
    ops = [omvm.FFTOperator(eps_r[blk.slices], H, K0, mask=blk.mask) for blk in blocks]
    for apply in range(applies):
        y, st = grid.precond(sp, bd, inner_tol=tau)
        assert st["nblocks"] == len(blocks) and st["not_converged"] == 0 and st["breakdowns"] == 0
        y = y.cpu().numpy().astype(np.complex128)
        for blk, op in zip(blocks, ops):
            sl = (slice(None),) + blk.slices
            bk = np.where(blk.mask[None], bb[sl], 0)
            xk = np.where(blk.mask[None], y[sl], 0)
            # 1 %: rounding of the complex64 iterate against a tolerance of 1e-3 or more
            assert np.linalg.norm(bk - op(xk)) <= 1.01 * tau * np.linalg.norm(bk), (apply, blk.slices)
        seen.append(grid.info()["inner_cluster"][0 if precision == vie.C128 else 1])


@pytest.mark.parametrize("precision,tau", [(vie.C128, 1e-8), (vie.C64, 1e-3)])
def test_tuner_of_larger_blocks(precision, tau):
    # 22 blocks over 16 voxels along x: one apply to warm up, then 2 CTAs a block, 4, and the slowest blocks on 4
    # beside the rest on 2, then the best of the three
    rng = np.random.default_rng(2)
    eps_r, bid, b = row_of_blocks([(17 + k % 4, 1 + int(rng.integers(6)), 1 + int(rng.integers(4))) for k in range(22)], 5)
    grid = vie.Grid(eps_r, H, bid, inner=vie.INNER_PERSISTENT)
    seen = []
    check_every_block(grid, eps_r, bid, b, precision, tau, 6, seen)
    assert seen[:3] == [0, 0, 0] and set(seen[3:]) <= {2, 4, -1}


@pytest.mark.parametrize("precision,tau", [(vie.C128, 1e-8), (vie.C64, 1e-3)])
@pytest.mark.parametrize("inner", [vie.INNER_AUTO, vie.INNER_PERSISTENT, vie.INNER_BATCHED])
def test_blocks_of_both_kinds_in_one_grid(inner, precision, tau):
    boxes = [(17 if k % 3 == 0 else 5, 4 + k % 2, 3) for k in range(40)]
    eps_r, bid, b = row_of_blocks(boxes, 6)
    check_every_block(vie.Grid(eps_r, H, bid, inner=inner), eps_r, bid, b, precision, tau, 5, [])
