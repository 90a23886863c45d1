"""ss_dedup_paths at path lengths around what a warp reads in a round, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_39334_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# the three forms: one cluster (96 paths), shared memory (4096), a table in the workspace
@pytest.mark.parametrize("n", [90, 700, 4500])
@pytest.mark.parametrize("weak", [False, True])
def test_lengths_around_a_round(n, weak):
    """Lengths around a warp, four and eight ids a lane and their multiples, none at all; every third path repeats an earlier one,
    every seventh does but for its first, its last or one id between."""
    if weak and n > 1000:
        n = 4100                                                # (every path of the table form is compared with many: a few suffice)
    rng = np.random.default_rng(n)
    lengths = np.asarray([0, 1, 31, 32, 33, 127, 128, 129, 159, 160, 255, 256, 257, 300, 511, 512, 513, 640])
    paths = []
    for i in range(n):
        if i > 20 and i % 3 == 0:
            p = paths[rng.integers(0, i)].copy()
        elif i > 20 and i % 7 == 0:
            p = paths[rng.integers(0, i)].copy()
            if len(p):
                p[(0, len(p) - 1, len(p) // 2)[i % 3]] ^= 1
        else:
            p = rng.integers(0, 1000, size=lengths[i % len(lengths)]).astype(np.int32)
        paths.append(p)
    off = np.concatenate([[0], np.cumsum([len(p) for p in paths])]).astype(np.int64)
    ids = np.concatenate(paths).astype(np.int32)
    want = oracle.dedup(ids, off)
    i32 = dict(dtype=torch.int32, device=DEV)
    outs = [torch.empty(n, **i32) for _ in range(4)]
    num = torch.zeros(1, **i32)
    ws = B.alloc_workspace(B.ss_dedup_workspace_bytes(n), DEV)
    B.ss_dedup_paths(torch.from_numpy(ids).to(DEV), torch.from_numpy(off).to(DEV), None, None, n, B.SS_FLAG_WEAK_HASH if weak else 0,
                     *outs, None, num, ws)
    U = int(num.item())
    assert U == want["num_unique"]
    for t, key in zip(outs, ("canon", "path_to_unique", "unique_paths", "multiplicity")):
        m = n if key in ("canon", "path_to_unique") else U
        assert np.array_equal(t[:m].cpu().numpy(), want[key][:m]), key
