"""Which solver takes the blocks of a grid: very many very small boxes, few or flat complex128 ones, and grids that
hold several kinds at once, against the CPU oracle."""
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
TAU = {vie.C64: 1e-4, vie.C128: 1e-9}


def lattice(boxes, per_row, seed):
    """One block per box, per_row side by side along x, rows of blocks along y."""
    px, py = max(b[0] for b in boxes) + 1, max(b[1] for b in boxes) + 1
    rows = -(-len(boxes) // per_row)
    nx, ny, nz = px * per_row, py * rows, max(b[2] for b in boxes)
    eps_r, _, b = inputs.random_case((nx, ny, nz), seed=seed)
    bid = np.full((nz, ny, nx), -1, np.int32)
    for k, (ex, ey, ez) in enumerate(boxes):
        x, y = px * (k % per_row), py * (k // per_row)
        bid[:ez, y:y + ey, x:x + ex] = k
    return eps_r, bid, b


def check(grid, sp, eps_r, bid, b, precision, applies=1):
    tau = TAU[precision]
    bd = torch.from_numpy(b).to(device="cuda", dtype=DT[precision])
    bb = bd.cpu().numpy().astype(np.complex128)
    blocks = oprecond.find_blocks(bid)
    for _ in range(applies):
        y, st = grid.precond(sp, bd, inner_tol=tau, inner_maxit=500)
        assert st["nblocks"] == len(blocks) and st["not_converged"] == 0 and st["breakdowns"] == 0
        y = y.cpu().numpy().astype(np.complex128)
        assert np.array_equal(y[:, bid < 0], bb[:, bid < 0])
        for blk in blocks:
            sl = (slice(None),) + blk.slices
            bk, xk = np.where(blk.mask[None], bb[sl], 0), np.where(blk.mask[None], y[sl], 0)
            r = bk - omvm.FFTOperator(eps_r[blk.slices], H, K0, mask=blk.mask)(xk)
            # complex64: rounding of the iterate, about 1e-6, against a tolerance of 1e-4
            assert np.linalg.norm(r) <= 1.02 * tau * np.linalg.norm(bk), blk.slices


# boxes, blocks per row; inner_cluster of complex128 and complex64 (CTAs per block; 0: batched launches)
CASES = {
    "single voxels": ([(1, 1, 1)] * 160, 40, 1, 1),
    "pairs and rods": ([(2, 2, 1 + k % 2) for k in range(100)] + [(16, 1, 1)] * 60, 20, 1, 1),
    "cubes of 4": ([(4, 4, 4)] * 60, 20, 1, 4),
    "cubes of 4, few": ([(4, 4, 4)] * 8, 4, 4, 4),
    "cubes of 12, few": ([(12, 12, 12), (11, 10, 9)], 2, 0, 4),
    "plates": ([(16, 15, 2)] * 64, 16, 0, 4),
    "cubes of 9 and 10": ([(9 + k % 2, 10, 9) for k in range(40)], 10, 4, 4),
    # the small shape of complex64 with its largest box, and the L2 shape
    "many of 1024 points": ([(16, 16, 4)] * 80, 16, None, 4),
    "many of 2304 points": ([(12, 12, 16)] * 106, 20, None, 4),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_path_of_a_grid(precision, name):
    boxes, per_row, c128, c64 = CASES[name]
    want = c128 if precision == vie.C128 else c64
    if want is None:
        pytest.skip("complex64 only")
    eps_r, bid, b = lattice(boxes, per_row, seed=len(boxes))
    g = vie.Grid(eps_r, H, bid)
    check(g, g.spectrum(K0), eps_r, bid, b, precision)
    assert g.info()["inner_cluster"][0 if precision == vie.C128 else 1] == want


@pytest.mark.parametrize("inner", [vie.INNER_AUTO, vie.INNER_PERSISTENT])
@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_every_kind_in_one_grid(precision, inner):
    # more very small boxes than clusters, boxes of the parity-split solver, and boxes over 16 voxels (tuner)
    boxes = [(2, 2, 2)] * 170 + [(6, 7, 5)] * 4 + [(9, 9, 10)] * 2 + [(17, 6, 4)] * 3
    eps_r, bid, b = lattice(boxes, 20, seed=11)
    g = vie.Grid(eps_r, H, bid, inner=inner)
    check(g, g.spectrum(K0), eps_r, bid, b, precision, applies=5)


@pytest.mark.parametrize("precision", [vie.C128, vie.C64])
def test_spectrum_serves_a_grid_of_another_path(precision):
    # one grid with two boxes, one with many: same shape and group box, other solvers
    many = [(2, 2, 2)] * 200
    eps_r, bid, b = lattice(many, 20, seed=12)
    few = np.where(bid < 2, bid, -1)
    ga, gb = vie.Grid(eps_r, H, few), vie.Grid(eps_r, H, bid)
    check(gb, ga.spectrum(K0), eps_r, bid, b, precision)
    check(ga, gb.spectrum(K0), eps_r, few, b, precision)


@pytest.mark.parametrize("mode", [vie.MODE_MIXED, vie.MODE_PLAIN_C128])
def test_merged_solves_with_every_kind_of_block(mode):
    # two grids in one session, their very small blocks in one launch and the others in another; the solutions are those
    # of the grids alone (both within 1e-8 of the right-hand side in residual, ||A^-1|| <= 10 for |chi| <= 0.7)
    problems, alone = [], []
    for seed in (21, 22):
        eps_r, bid, b = lattice([(2, 2, 2)] * 170 + [(6, 7, 5)] * (2 + seed % 2) + [(9, 9, 10)], 20, seed=seed)
        b = torch.from_numpy(b).cuda()
        grids = [vie.Grid(eps_r, H, bid) for _ in range(2)]
        specs = [g.spectrum(K0) for g in grids]
        alone.append(grids[0].solve(specs[0], b, outer_tol=1e-8, mode=mode))
        problems.append({"grid": grids[1], "spec": specs[1], "einc": b, "outer_tol": 1e-8, "mode": mode})
    res, ms = vie.solve_many(problems)
    assert ms["launches"] >= 1 and ms["max_solves"] == 2
    for (e, st), (e1, st1) in zip(res, alone):
        assert st["status"] == vie.VIE_OK and st1["status"] == vie.VIE_OK
        assert float((e - e1).norm() / e1.norm()) <= 2e-7
