"""Decode leaves around the ends of a leaf item (256 keys, or 512 where the leaves are enough for a warp each) against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_39334_b200 import synth
from paper_2609_39334_b200.pipeline import DevicePipeline

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("lo,hi", [(0, 20), (250, 262), (505, 520), (1018, 1030)])
@pytest.mark.parametrize("more", [-1, 0])
def test_leaf_items_at_their_ends(lo, hi, more):
    """One path fewer than the longer items are taken for, and just as many."""
    n = torch.cuda.get_device_properties(0).multi_processor_count * 12 // 2 + more
    w = synth.build_tree_workload("leaves", lo + n, 8, 2, [32], [n], 1, (lo, hi), lambda i, m, rng: 1, device=DEV)
    pipe = DevicePipeline(w, DEV)
    pipe.step()
    r = pipe.results()
    paths = r["unique_paths"]
    sample = np.unique(np.concatenate([np.arange(0, len(paths), max(1, len(paths) // 60)), [len(paths) - 1]]))
    want, want_lse = oracle.tree_attention_workload(w, paths=paths[sample])
    got, lse = r["out"][sample], r["lse"][sample]
    # the rows are rounded to bf16 (2^-9 of them), the probabilities too before they multiply V: at most 2^-9 of the largest |v|, below
    # 4.6 for these inputs.  A key too many or too few moves the log-sum by 1e-3 on average.
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -9 * 4.6).all()
    assert np.abs(lse - want_lse).max() <= 2e-5
    assert np.isfinite(r["out"]).all()
