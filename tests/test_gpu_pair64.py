"""The FP64 pair kernels at the edges of their work split and of the bracket tables.

Sets are sized around the warp (32), the staged batch (128 suppliers), the supplier list
(128 subtiles) and the split of chunks between work items; x_r / x_s puts the pairs inside
the tables, below their first interval and beyond their last one.  The oracle is the
reference; 1e-12 relative RMS is the tolerance of the FP64 path."""
import numpy as np
import pytest
import torch

import oracle
from _gpu_helpers import gpu_forces, rel_rms

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _positions(n, layout, seed):
    rng = np.random.default_rng(seed)
    if layout == "uniform":
        return rng.uniform(size=(3, n))
    p = 0.995 + 0.02 * rng.normal(size=(3, n))  # a dense blob across the periodic boundary
    p -= np.floor(p)
    if n >= 4:
        p[:, 1] = p[:, 0]  # coincident particles
    return np.where(p >= 1.0, 0.0, p)


@pytest.mark.parametrize("box", [3.1e24, 1.7e-20])
def test_any_unit_of_length(box):
    """The FP32 part of the kernel works in units of the box's binary exponent."""
    n, x_r, eps = 1500, 0.2 * box, 0.004 * box
    pos = _positions(n, "uniform", 5) * box
    ref, pairs = oracle.sr_accel(pos, x_r / 4.5, x_r, 1.0, "bspline", eps, box=box)
    r = gpu_forces(pos, x_r / 4.5, x_r, 1.0, "bspline", eps, precision=64, box=box)
    assert r["pairs"] == pairs and pairs > 0
    scale = box * box  # accelerations ~ 1 / box^2: brought near 1 before they are squared
    assert rel_rms(r["acc"] * scale, ref * scale) <= TOL


@pytest.mark.parametrize("softening", ["none", "plummer", "bspline"])
@pytest.mark.parametrize("n,layout,n_sub,ratio", [
    (1, "blob", 2, 4.5), (2, "blob", 2, 4.5), (33, "blob", 1, 4.5), (129, "blob", 2, 4.5), (700, "blob", 2, 4.5),
    (4000, "uniform", 8, 4.5),   # more than 128 subtiles around a chunk
    (900, "blob", 2, 0.02),      # every pair below the first interval
    (900, "blob", 2, 9.5),       # distant pairs beyond the last interval
    (20000, "uniform", 2, 4.5),  # chunks not split into 32
])
def test_forces_and_vjp_match_the_oracle(n, layout, n_sub, ratio, softening):
    pos = _positions(n, layout, 7 * n)
    x_r = 0.2 if n <= 4000 else 0.06
    x_s = x_r / ratio
    eps = 0.0 if softening == "none" else min(0.004, 0.3 * x_s)
    G_m = 1.0 / n
    ref, pairs = oracle.sr_accel(pos, x_s, x_r, G_m, softening, eps)
    r = gpu_forces(pos, x_s, x_r, G_m, softening, eps, precision=64, n_sub=n_sub, return_ctx=True)
    assert r["pairs"] == pairs
    if pairs == 0:
        assert not r["acc"].any()
    else:
        assert rel_rms(r["acc"], ref) <= TOL
    rng = np.random.default_rng(n)
    bar = rng.normal(size=(3, n))
    xref = oracle.sr_vjp(pos, bar, x_s, x_r, G_m, softening, eps)
    sr, p, perm = r["ctx"], r["pos_dev"], r["perm"]
    got = np.empty((3, n))
    got[:, perm] = sr.vjp(p, torch.from_numpy(bar[:, perm].copy()).cuda(), 64).cpu().numpy()
    again = sr.forces(p, 64)
    assert torch.equal(again, sr.forces(p, 64))  # bitwise reproducible, split or not
    sr.sync()
    sr.close()
    if pairs == 0:
        assert not got.any()
    else:
        assert rel_rms(got, xref) <= TOL
