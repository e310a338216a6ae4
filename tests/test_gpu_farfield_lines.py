"""Far field with one and with four directions per CTA, lines along y and along z, cut and whole, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import solve as osolve
from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu


# FP64 sums of n terms: a few 1e-16 of the largest lobe and of the value itself; 1e-12 as for the other far fields
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 1, 3), (40, 3, 200), (300, 9, 2), (64, 33, 16), (2, 200, 40)])
@pytest.mark.parametrize("ndir", [1, 3, 81, 1217])
def test_far_field_of_lines(shape, ndir):
    eps_r, _, x = inputs.random_case(shape, seed=sum(shape))
    k0, h = 2 * np.pi, 0.05
    rng = np.random.default_rng(ndir)
    dirs = rng.normal(size=(ndir, 3))
    dirs /= np.linalg.norm(dirs, axis=1, keepdims=True)
    got = vie.Grid(eps_r, h).far_field_rcs(k0, torch.from_numpy(x).cuda(), dirs)
    ref = osolve.far_field_rcs(x, eps_r, h, k0, dirs[:130])
    assert got.shape == (ndir,)
    assert np.all(np.abs(got[:130] - ref) <= 1e-12 * (np.abs(ref) + np.abs(ref).max()))
    # the same directions one by one and the last ones of the list
    some = [0, ndir // 2, ndir - 1]
    alone = vie.Grid(eps_r, h).far_field_rcs(k0, torch.from_numpy(x).cuda(), dirs[some])
    assert np.all(np.abs(got[some] - alone) <= 1e-12 * (np.abs(alone) + np.abs(ref).max()))
