"""The mesh assignment cell by cell, in boxes of any side, for positions at cell faces and centres
and their neighbours in double: the weights sum to 1 wherever a stencil lands, so a wrong cell
shows only here."""
import numpy as np
import pytest
import torch

from paper_2112_01508_gb300 import LongRange

pytestmark = pytest.mark.gpu


def _weight(p, t):
    t = np.abs(t)
    if p == 2:
        return 1.0 - t
    if p == 3:
        return np.where(t < 0.5, 0.75 - t * t, 0.5 * (1.5 - t) ** 2)
    return np.where(t < 1.0, (4.0 - 6.0 * t ** 2 + 3.0 * t ** 3) / 6.0, (2.0 - t) ** 3 / 6.0)


def _mesh(pos, n_phi, box, p):
    cells, weights = [], []
    for x in pos:
        s = x * (n_phi / box) - 0.5
        first = np.floor(s + 0.5) - 1 if p == 3 else np.floor(s) - (p // 2 - 1)
        m = first[:, None] + np.arange(p)
        cells.append(m.astype(np.int64) % n_phi)
        weights.append(_weight(p, m - s[:, None]))
    rho = np.zeros((n_phi,) * 3)
    w = weights[0][:, :, None, None] * weights[1][:, None, :, None] * weights[2][:, None, None, :]
    np.add.at(rho, (cells[0][:, :, None, None], cells[1][:, None, :, None], cells[2][:, None, None, :]), w)
    return rho


@pytest.mark.parametrize("p_i", [2, 3, 4])
@pytest.mark.parametrize("n_phi,box", [(8, 1.0), (30, 3.0), (256, 0.7)])
def test_every_cell_of_the_mesh(n_phi, box, p_i):
    k = np.arange(n_phi + 1)
    at = np.concatenate([k * (box / n_phi), (k[:-1] + 0.5) * (box / n_phi)])
    rng = np.random.default_rng(p_i)
    x = np.concatenate([at, np.nextafter(at, -1.0), np.nextafter(at, 9.0), rng.uniform(size=200) * box,
                        [0.0, -0.0, 5e-324, 1e-300, 1e-17, np.nextafter(box, 0)]])
    x = x[(x >= 0.0) & (x < box)]
    pos = np.stack([x, rng.permutation(x), rng.permutation(x)])
    want = _mesh(pos, n_phi, box, p_i)
    dev = torch.from_numpy(pos).cuda()
    # s is off by at most 3 n_phi 2^-53 in double, each weight by that (slopes up to 1) and in single
    # precision by 2^-23 more; relative to the weights' RMS, over three dimensions, 5 times that
    for precision, tol in ((32, 1e-6), (64, 16 * n_phi * 2.0 ** -53)):
        with LongRange(pos.shape[1], n_phi, 1.25 * box / n_phi, 1.0, p_i=p_i, p_d=4, precision=precision, box=box) as lr:
            got = lr.assign(dev).cpu().numpy().astype(np.float64)
            lr.sync()
        assert np.sqrt(((got - want) ** 2).sum() / (want ** 2).sum()) <= tol
