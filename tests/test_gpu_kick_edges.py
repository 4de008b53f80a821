"""Kick and drift are bit-exact in IEEE double for values at the edges of their integer
conversions and of the FP32 kick's rounding test: zeros of both signs, subnormals, the
ends of the float range, ties, momenta that cancel the kick, and ordinary values."""
import numpy as np
import pytest
import torch

from paper_2112_01508_gb300 import ShortRange
from paper_2112_01508_gb300._native import P3MError
from paper_2112_01508_gb300.autograd import Drift, Kick, short_range_accel

pytestmark = pytest.mark.gpu

_F = {32: np.float32, 64: np.float64}


def _values(n, dtype, seed):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=n) * 10.0 ** rng.integers(-12, 6, size=n)
    edge = np.array([0.0, -0.0, 1e-45, -1e-45, 5e-42, 1.1754944e-38, -1.1754942e-38, 1.0, -1.0, 0.5, 3.0, 1e-30, 1e30,
                     3.4e37, 1.0 + 2.0 ** -23, 2.0 ** -24, 1.5, 2.0 ** -126, 7.0e-39, 123456.789])
    v[: len(edge) ** 2] = np.tile(edge, len(edge)) if seed % 2 else np.repeat(edge, len(edge))
    return v.astype(dtype)


@pytest.mark.parametrize("mom_bits,acc_bits", [(32, 32), (32, 64), (64, 32), (64, 64)])
@pytest.mark.parametrize("factor", [1e-3, 1.0 / 3.0, 2.0 ** -24, -0.7, 0.0, 2.0 ** -75, 1e20])
def test_kick_and_drift_bits(mom_bits, acc_bits, factor):
    n = 5000
    q = np.stack([_values(n, _F[mom_bits], s) for s in (1, 3, 5)])
    a = np.stack([_values(n, _F[acc_bits], s) for s in (2, 4, 6)])
    if factor == 2.0 ** -24:  # ties, and sums that cancel
        q[:, 1000:2000] = 1.0 + 2.0 ** -23 * np.arange(1000)
        a[:, 1000:1500] = 1.0
        a[:, 1500:2000] = -(q[:, 1500:2000].astype(np.float64) * 2.0 ** 24).astype(_F[acc_bits])
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        want = (q.astype(np.float64) + a.astype(np.float64) * factor).astype(_F[mom_bits])
    sr = ShortRange(n, 0.02, 0.09, 1.0, eps=0.001)
    dq, da = torch.from_numpy(q.copy()).cuda(), torch.from_numpy(a).cuda()
    sr.kick(dq, da, [factor])
    got = dq.cpu().numpy()
    assert np.array_equal(got.view(np.uint8), want.view(np.uint8))

    x = np.random.default_rng(9).uniform(size=(3, n))
    p = q[:, :].astype(np.float64)
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        v = x + p * (factor * 1e-9)
    inside = (v >= 0.0) & (v < 1.0)
    dx = torch.from_numpy(x.copy()).cuda()
    sr.drift(dx, torch.from_numpy(q).cuda(), factor * 1e-9)
    sr.sync()
    out = dx.cpu().numpy()
    assert np.array_equal(out[inside].view(np.uint64), v[inside].view(np.uint64))
    assert ((out >= 0.0) & (out < 1.0)).all()
    sr.close()


@pytest.mark.parametrize("mom_bits,acc_bits", [(32, 32), (32, 64), (64, 32), (64, 64)])
@pytest.mark.parametrize("n", [1, 255, 5000])
def test_out_of_place_kick_and_drift_equal_the_in_place_ones(n, mom_bits, acc_bits):
    def bits(t):
        return t.contiguous().view(torch.uint8)

    t = {32: torch.float32, 64: torch.float64}
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand(3, n, generator=g, device="cuda", dtype=torch.float64)
    q = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64).to(t[mom_bits])
    a = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64).to(t[acc_bits])
    with ShortRange(n, 0.02, 0.09, 1.0, eps=0.001) as sr:
        for mom in (q, None):
            want = q.clone() if mom is not None else torch.zeros_like(q)
            before, out = q.clone(), torch.full_like(q, 7.0)
            sr.kick(want, a, [0.3])
            sr.kick_into(mom, out, a, 0.3)
            assert torch.equal(bits(out), bits(want)) and torch.equal(q, before)
        want, before, out = x.clone(), x.clone(), torch.full_like(x, 7.0)
        sr.drift(want, q, 0.2)
        sr.drift_into(x, out, q, 0.2)
        assert torch.equal(bits(out), bits(want)) and torch.equal(x, before)
        with pytest.raises(P3MError):
            sr.drift_into(x, x, q, 0.2)
        sr.sort_into(x, out)
        sr.drift_into(x, out, q, 0.2)  # writes over the sorted positions
        with pytest.raises(P3MError):
            sr.build_pairs()


def test_autograd_takes_arrays_whose_elements_lie_apart():
    n = 500
    g = torch.Generator(device="cuda").manual_seed(2)
    wide = torch.rand(3, 2 * n, generator=g, device="cuda", dtype=torch.float64)
    apart, packed = wide[:, ::2], wide[:, ::2].contiguous()
    with ShortRange(n, 0.02, 0.09, 1.0, eps=0.001) as sr:
        a, b = (short_range_accel(p, sr, 64) for p in (apart, packed))
        assert torch.equal(a, b)
        assert torch.equal(Drift.apply(apart, apart, sr, 0.1), Drift.apply(packed, packed, sr, 0.1))
        assert torch.equal(Kick.apply(apart, packed, sr, 0.1), Kick.apply(packed, packed, sr, 0.1))
