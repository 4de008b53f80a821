"""Staged records that hold 4-byte words: sort_into with one, two and more float32 arrays and no
8-byte one, at a size whose arrays exceed half of L2 (64 MiB = 33.6 bytes per particle), as float32
momenta of 2 M unordered particles are carried."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_01508_gb300 import ShortRange

pytestmark = pytest.mark.gpu

N = 2_000_003


@pytest.mark.parametrize("order", ["random", "sorted", "mixed"])
@pytest.mark.parametrize("rows4,rows20,i8", [(3, 0, 0), (1, 1, 0), (2, 1, 1), (4, 0, 2)])
def test_four_byte_words_of_staged_records(order, rows4, rows20, i8):
    assert N * (24 + 4 * rows4 + 20 * rows20 + i8) > 64 << 20  # staged where a tile is unordered
    rng = np.random.default_rng(7)
    x_r, n_sub = 0.03, 2
    n_t = int(np.floor(1.0 / x_r))
    pos = rng.uniform(size=(3, N))
    if order != "random":
        pos = np.ascontiguousarray(pos[:, np.argsort(oracle.subtile_ids(pos, n_t, n_sub), kind="stable")])
        if order == "mixed":  # shuffle the second half
            half = N // 2 + 777
            pos[:, half:] = pos[:, half:][:, rng.permutation(N - half)]
    perm = torch.from_numpy(np.argsort(oracle.subtile_ids(pos, n_t, n_sub), kind="stable")).cuda()
    index = torch.arange(N, device="cuda", dtype=torch.float32)  # exact below 2^24: no two words alike
    arrays = [index + 4_000_000 * r for r in range(rows4)]
    arrays += [torch.randint(0, 256, (N, 20), device="cuda", dtype=torch.uint8) for _ in range(rows20)]
    arrays += [torch.randint(0, 128, (N,), device="cuda", dtype=torch.int8) for _ in range(i8)]
    out = [torch.empty_like(a) for a in arrays]
    p = torch.from_numpy(pos).cuda()
    q = torch.empty_like(p)
    with ShortRange(N, x_r / 4.5, x_r, 1.0, eps=0.0005, n_sub=n_sub) as sr:
        sr.sort_into(p, q, arrays, out)
        sr.sync()
    assert torch.equal(q, p[:, perm])
    for a, b in zip(arrays, out):
        assert torch.equal(b, a[perm])
