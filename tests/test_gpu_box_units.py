"""FP64 forces and adjoint in boxes whose lengths no float holds: the FP32 records from which
the kernel finds its candidates are then in units of the box."""
import numpy as np
import pytest
import torch

import oracle
from _gpu_helpers import gpu_forces, rel_rms
from paper_2112_01508_gb300 import ShortRange
from paper_2112_01508_gb300._native import P3MError

pytestmark = pytest.mark.gpu

N, TOL = 1500, 1e-12  # the FP64 path's tolerance


def _set(box):
    return np.random.default_rng(5).uniform(size=(3, N)) * box, 0.2 * box, 0.004 * box


@pytest.mark.parametrize("box", [1e39, 2.6e45, 1e100, 1e-42])
def test_forces(box):
    pos, x_r, eps = _set(box)
    ref, pairs = oracle.sr_accel(pos, x_r / 4.5, x_r, 1.0, "bspline", eps, box=box)
    r = gpu_forces(pos, x_r / 4.5, x_r, 1.0, "bspline", eps, precision=64, box=box)
    assert r["pairs"] == pairs and pairs > 0
    scale = box * box  # accelerations ~ 1 / box^2: brought near 1 before they are squared
    assert rel_rms(r["acc"] * scale, ref * scale) <= TOL


@pytest.mark.parametrize("softening", ["none", "plummer", "bspline"])
def test_adjoint(softening):
    box = 2.6e45
    pos, x_r, eps = _set(box)
    eps = 0.0 if softening == "none" else eps
    bar = np.random.default_rng(6).normal(size=(3, N))
    ref = oracle.sr_vjp(pos, bar, x_r / 4.5, x_r, 1.0, softening, eps, box=box)
    r = gpu_forces(pos, x_r / 4.5, x_r, 1.0, softening, eps, precision=64, box=box, return_ctx=True)
    got = np.empty((3, N))
    with r["ctx"] as sr:
        got[:, r["perm"]] = sr.vjp(r["pos_dev"], torch.from_numpy(bar[:, r["perm"]].copy()).cuda(), 64).cpu().numpy()
    scale = box * box * box
    assert rel_rms(got * scale, ref * scale) <= TOL


def test_a_drift_beyond_the_range_of_its_bound_is_refused():
    box = 2.6e45
    pos, x_r, eps = _set(box)
    p = torch.from_numpy(pos).cuda()
    q = torch.empty_like(p)
    with ShortRange(N, x_r / 4.5, x_r, 1.0, eps=eps, box=box) as sr:
        sr.sort_into(p, q)
        sr.drift(q, torch.randn_like(q), 0.01 * box)
        sr.build_pairs()
        with pytest.raises(P3MError):
            sr.forces(q, 64)
            sr.sync()
