"""The each-pair-once kernel at the edges of its blocks: chunks of 32 receivers, blocks of 64
staged suppliers with power-of-two tails, chunks split into slices of their suppliers."""
import numpy as np
import pytest
import torch

import oracle
from _gpu_helpers import gpu_forces, rel_rms

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the FP32 path's tolerance


@pytest.mark.parametrize("softening", ["plummer", "bspline"])
@pytest.mark.parametrize("n", [2, 3, 17, 31, 32, 33, 34, 35, 37, 48, 63, 64, 65, 96, 97, 98, 130, 1000, 6000])
def test_forces_and_vjp_match_the_oracle(n, softening):
    rng = np.random.default_rng(n)
    x_r, eps = 0.2, 0.004
    p = 0.1 + 0.03 * rng.normal(size=(3, n))  # within one tile and its neighbours: most pairs interact
    pos = p - np.floor(p)
    pos[:, 1] = pos[:, 0]  # coincident particles
    ref, pairs = oracle.sr_accel(pos, x_r / 4.5, x_r, 1.0 / n, softening, eps)
    r = gpu_forces(pos, x_r / 4.5, x_r, 1.0 / n, softening, eps, precision=32, return_ctx=True)
    assert abs(r["pairs"] - pairs) <= 1e-6 * pairs
    if n > 2:
        assert rel_rms(r["acc"], ref) <= TOL
    else:
        assert not r["acc"].any()  # two coincident particles exert no force
    bar = rng.normal(size=(3, n)).astype(np.float32).astype(np.float64)
    xref = oracle.sr_vjp(pos, bar, x_r / 4.5, x_r, 1.0 / n, softening, eps)
    sr, dev, perm = r["ctx"], r["pos_dev"], r["perm"]
    got = np.empty((3, n))
    got[:, perm] = sr.vjp(dev, torch.from_numpy(np.ascontiguousarray(bar[:, perm], dtype=np.float32)).cuda(), 32).cpu().numpy()
    sr.sync()
    sr.close()
    assert rel_rms(got, xref) <= TOL
