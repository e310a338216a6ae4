"""What a batch keeps on the device for a wavenumber."""
import numpy as np
import pytest
import torch

from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu


def job(n, count, seed):
    ws = [inputs.blob(n=n, seed=seed + i) for i in range(count)]
    r = np.stack(inputs.voxel_centres(ws[0].n, ws[0].h))
    einc = np.stack([w.pol[:, None, None, None] * np.exp(-1j * w.k0 * np.tensordot(w.khat, r, 1)) for w in ws])
    return {"batch": vie.Batch([w.eps_r for w in ws], ws[0].h), "k0s": [ws[0].k0] * count,
            "einc": torch.from_numpy(einc).cuda(), "outer_tol": 1e-6}


def test_layout_of_merged_launches_is_built_when_one_reads_it():
    # 20^3 voxels pad to 64^3: octants of 33^3 in both precisions; merged launches read the full complex64 layout
    a, b = job(20, 2, 1), job(20, 2, 5)
    before = a["batch"].info()["device_bytes"]
    e1, _ = a["batch"].solve(a["k0s"], a["einc"], outer_tol=1e-6)
    octants = 6 * 33**3 * (16 + 8)
    assert a["batch"].info()["device_bytes"] - before == octants
    res, ms = vie.batch_solve_many([a, b])
    assert ms["max_solves"] == 2
    assert a["batch"].info()["device_bytes"] - before == octants + 6 * 64**3 * 8
    e2 = res[0][0]
    assert float((e2 - e1).norm() / e1.norm()) <= 1e-5
    e3, _ = a["batch"].solve(a["k0s"], a["einc"], outer_tol=1e-6)
    assert torch.equal(e1, e3)
    a["batch"].close()
    b["batch"].close()
