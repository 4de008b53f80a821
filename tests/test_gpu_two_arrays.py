"""Force and adjoint calls that alternate between the sorted array and another one: the FP32
subtile-relative records are those of the array at hand in every call, in either precision."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_01508_gb300 import ShortRange

pytestmark = pytest.mark.gpu

N, X_R, EPS, G_M = 3000, 0.1, 0.001, 1.0 / 3000
X_S = X_R / 4.5


def _calls(sr, bar):
    return {"forces32": lambda a: sr.forces(a, 32), "forces64": lambda a: sr.forces(a, 64),
            "tabulated": lambda a: sr.forces_tabulated(a, 12),
            "vjp32": lambda a: sr.vjp(a, bar.float(), 32), "vjp64": lambda a: sr.vjp(a, bar, 64)}


@pytest.mark.parametrize("first", ["forces32", "forces64", "tabulated", "vjp32", "vjp64"])
@pytest.mark.parametrize("drifted", ["sorted", "other"])  # which of the two arrays moves after the sort
def test_calls_on_two_arrays_in_turn(drifted, first):
    g = torch.Generator(device="cuda").manual_seed(11)
    pos = torch.rand(3, N, generator=g, device="cuda", dtype=torch.float64)
    mom = torch.randn(3, N, generator=g, device="cuda", dtype=torch.float64)
    bar = torch.randn(3, N, generator=g, device="cuda", dtype=torch.float64)
    # one-sided FP32 kernels: their results are reproducible bit for bit
    with ShortRange(N, X_S, X_R, G_M, eps=EPS, symmetric=False) as sr:
        a = torch.empty_like(pos)
        sr.sort_into(pos, a)
        b = a.clone()
        sr.drift(a if drifted == "sorted" else b, mom, 0.015)
        sr.build_pairs()
        count = {}
        for name, t in (("a", a), ("b", b)):
            count[name] = oracle.sr_accel(t.cpu().numpy(), X_S, X_R, G_M, "bspline", EPS)[1]
        assert count["a"] != count["b"]
        calls = _calls(sr, bar)

        def pairs(name, want):
            got = sr.stats().pairs_last
            assert got == want if name.endswith("64") else abs(got - want) <= 1e-4 * want, (name, got, want)

        before = calls[first](a)
        pairs(first, count["a"])
        for other in calls:
            calls[other](b)
            if drifted == "sorted":  # the reach covers both arrays
                pairs(other, count["b"])
            assert torch.equal(calls[first](a), before), other
            pairs(first, count["a"])
        want = oracle.sr_accel(a.cpu().numpy(), X_S, X_R, G_M, "bspline", EPS)[0]
        err = np.linalg.norm(sr.forces(a, 64).cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= 1e-12
