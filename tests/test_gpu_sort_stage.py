"""The out-of-place sort's staged gather against a stable CPU sort of the oracle's subtile
ids: inputs in random order, nearly sorted, and mixed tile by tile, with carried arrays of
one word of each width, of several words and of odd sizes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_01508_gb300 import ShortRange

pytestmark = pytest.mark.gpu

N = 1_700_003  # 24 and more bytes of arrays per particle: past half of L2 with 17 carried


@pytest.mark.parametrize("order", ["random", "sorted", "mixed"])
@pytest.mark.parametrize("carried", ["f64x3 f32x3 i8 i64", "f32x3", "f32", "i8 i8 i8 f16", "f64x4 f32x3 f32x3", "rows20"])
def test_sort_into_matches_a_stable_cpu_sort(order, carried):
    rng = np.random.default_rng(3)
    x_r, n_sub = 0.03, 2
    pos = rng.uniform(size=(3, N))
    n_t = int(np.floor(1.0 / x_r))
    ids = oracle.subtile_ids(pos, n_t, n_sub)
    if order != "random":
        pos = np.ascontiguousarray(pos[:, np.argsort(ids, kind="stable")])
        if order == "mixed":  # shuffle the second half
            half = N // 2 + 777
            pos[:, half:] = pos[:, half:][:, rng.permutation(N - half)]
        ids = oracle.subtile_ids(pos, n_t, n_sub)
    perm = np.argsort(ids, kind="stable")
    dev = torch.device("cuda")
    arrays = []
    for word in carried.split():
        if word == "rows20":  # 20 bytes per particle
            arrays.append(torch.from_numpy(rng.integers(0, 255, size=(N, 20), dtype=np.uint8)).to(dev))
            continue
        kind, _, rows = word.partition("x")
        dt = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "i8": torch.int8, "i64": torch.int64}[kind]
        for _ in range(int(rows or 1)):
            arrays.append((torch.rand(N, device=dev) * 100).to(dt))
    arrays = arrays[:8]
    out = [torch.empty_like(a) for a in arrays]
    p = torch.from_numpy(pos).to(dev)
    q = torch.empty_like(p)
    got = torch.empty(N, dtype=torch.int32, device=dev)
    with ShortRange(N, x_r / 4.5, x_r, 1.0, eps=0.0005, n_sub=n_sub) as sr:
        sr.sort_into(p, q, arrays, out, perm_out=got)
        sr.sync()
        order_gpu = torch.from_numpy(perm).to(dev)
        assert torch.equal(got.long(), order_gpu)
        assert torch.equal(q, p[:, order_gpu])
        for a, b in zip(arrays, out):
            assert torch.equal(b, a[order_gpu])
        sr.sort(p, carry=arrays)  # in place: every position staged
        sr.sync()
    assert torch.equal(p, q)
    for a, b in zip(arrays, out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n, x_r, n_sub", [(1, 0.2, 1), (511, 0.2, 2), (512, 0.2, 2), (513, 0.05, 1), (40_001, 0.05, 3),
                                           (311_296, 0.03, 2), (311_297, 0.03, 2),  # the last short and the first long tile
                                           (70_001, 0.01, 2),    # 2^23 subtiles: three radix passes
                                           (70_001, 0.0099, 3)])  # 2.8e7 subtiles: the scans run by themselves
def test_sort_at_the_edges_of_the_radix_tiles(n, x_r, n_sub):
    rng = np.random.default_rng(n)
    pos = rng.uniform(size=(3, n))
    perm = np.argsort(oracle.subtile_ids(pos, int(np.floor(1.0 / x_r)), n_sub), kind="stable")
    p = torch.from_numpy(pos).cuda()
    q, got = torch.empty_like(p), torch.empty(n, dtype=torch.int32, device="cuda")
    with ShortRange(n, x_r / 4.5, x_r, 1.0, eps=0.01 * x_r, n_sub=n_sub) as sr:
        for _ in range(2):  # the second finds the first one's counts in its workspaces
            sr.sort_into(p, q, perm_out=got)
        sr.sync()
    order = torch.from_numpy(perm).cuda()
    assert torch.equal(got.long(), order)
    assert torch.equal(q, p[:, order])
