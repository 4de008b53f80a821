"""The mesh kernels' row handling: vector reductions of the FP32 assignment at every row and
cell alignment (n_phi a multiple of 4 or not) and at rows that wrap, and both forms of the
Green's function multiplication (rows that fill their warps or not), against the oracle."""
import numpy as np
import pytest
import torch

from oracle import pm as opm
from paper_2112_01508_gb300 import LongRange

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("p_i", [1, 2, 3, 4])
@pytest.mark.parametrize("n_phi", [8, 10, 30, 60, 66])
def test_assignment_and_accel(n_phi, p_i):
    rng = np.random.default_rng(n_phi * 10 + p_i)
    n = 3000
    pos = rng.uniform(size=(3, n))
    pos[2, :200] = rng.uniform(size=200) * 2.0 / n_phi            # rows that wrap at the box's lower face
    pos[2, 200:400] = 1.0 - rng.uniform(size=200) * 2.0 / n_phi   # and at its upper face
    dev = torch.from_numpy(pos).cuda()
    rho = opm.assign(pos, n_phi, p_i)
    acc = opm.lr_accel(pos, n_phi, 1.25 / n_phi, 1.0 / n, p_i=p_i, p_d=4)
    for precision, tol_rho, tol_acc in ((32, 1e-6, 1e-5), (64, 1e-14, 1e-12)):
        with LongRange(n, n_phi, 1.25 / n_phi, 1.0 / n, p_i=p_i, p_d=4, precision=precision) as lr:
            assert _rel(lr.assign(dev).cpu().numpy().astype(np.float64), rho) <= tol_rho
            assert _rel(lr.accel(dev).cpu().numpy().astype(np.float64), acc) <= tol_acc
            lr.sync()


@pytest.mark.parametrize("p_i", [1, 2, 3, 4])
@pytest.mark.parametrize("n_phi,box", [(8, 1.0), (30, 3.0), (256, 0.7)])
def test_positions_at_cell_faces_and_centres(n_phi, box, p_i):
    # faces and centres of cells and their neighbours in double, both zeros, tiny and the last
    # positions of the box: the cell and the offset come from the bit patterns
    k = np.arange(n_phi + 1)
    at = np.concatenate([k * (box / n_phi), (k[:-1] + 0.5) * (box / n_phi)])
    x = np.concatenate([at, np.nextafter(at, -1.0), np.nextafter(at, 9.0), [0.0, -0.0, 5e-324, 1e-300, 1e-17, np.nextafter(box, 0)]])
    x = x[(x >= 0.0) & (x < box)]
    rng = np.random.default_rng(p_i)
    pos = np.stack([x, rng.permutation(x), rng.permutation(x)])
    dev = torch.from_numpy(pos).cuda()
    n = pos.shape[1]
    rho = opm.assign(pos / box, n_phi, p_i) if box == 1.0 else None
    fx = np.floor(pos * (n_phi / box) - 0.5 + (0.5 if p_i % 2 else 0.0))  # a cell is the oracle's or its neighbour with weight 0
    for precision, tol in ((32, 1e-6), (64, 1e-14)):
        with LongRange(n, n_phi, 1.25 * box / n_phi, 1.0 / n, p_i=p_i, p_d=4, precision=precision, box=box) as lr:
            got = lr.assign(dev).cpu().numpy().astype(np.float64)
            lr.sync()
        assert abs(got.sum() - n) <= tol * n
        if rho is not None:
            assert _rel(got, rho) <= tol
        if p_i == 1:
            want = np.zeros((n_phi,) * 3)
            np.add.at(want, tuple(fx.astype(int) % n_phi), 1.0)
            assert np.array_equal(got, want)
