"""The context's sort outlives the differentiable force call that made it: later calls of the
autograd functions neither drop it nor write over the array that it describes."""
import pytest
import torch

from paper_2112_01508_gb300 import ShortRange
from paper_2112_01508_gb300.autograd import Drift, Kick, short_range_accel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [500, 60_000])
@pytest.mark.parametrize("backward", [False, True])
def test_the_sort_stays_usable_after_drifts_and_kicks(n, backward):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand(3, n, generator=g, device="cuda", dtype=torch.float64, requires_grad=backward)
    m = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
    with ShortRange(n, 0.02, 0.09, 1.0 / n, eps=0.001) as sr:
        a = short_range_accel(x, sr, 64)
        if backward:
            a.sum().backward()
        kept = []
        for _ in range(3):  # outputs of the size of the sorted copy
            kept.append(Drift.apply(x.detach(), m, sr, 0.01))
            kept.append(Kick.apply(m, a.detach(), sr, 0.01))
        offsets = sr.tile_offsets()
        sr.build_pairs()
        again = sr.unpermute(sr.forces(sr.permute(x.detach()), 64))
        sr.sync()
        n_t = sr.stats_geometry()[0]
        tile = (x.detach() * n_t).floor().long()
        counts = torch.bincount((tile[0] * n_t + tile[1]) * n_t + tile[2], minlength=n_t ** 3)
        assert torch.equal(offsets.diff().long(), counts)
        assert torch.equal(again, a.detach())
