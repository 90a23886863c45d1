"""Decode leaves around the ends of a leaf item (256 keys, or 512 where the leaves are enough for a warp each) against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_39334_b200 import binding as B
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


@pytest.mark.parametrize("heads", [(8, 2), (24, 2), (8, 4)])
@pytest.mark.parametrize("dup", [0.0, 0.9])
@pytest.mark.parametrize("fan", [64, 300])
def test_leaf_items_follow_the_live_leaves(heads, dup, fan):
    """The length of a leaf item depends on the leaves that are there, not on how many candidates there may be: 256 keys until those
    make an item for every warp of the leaf kernel (12 an SM, 8 with groups of more than 8 query heads); both planners."""
    w = synth.build_tree_workload("leaves", fan, heads[0], heads[1], [32], [fan], 8, (200, 700), lambda i, m, rng: 1, dup_frac=dup,
                                  device=DEV)
    pipe = DevicePipeline(w, DEV)
    pipe.step()
    r = pipe.results()
    lens = w.node_kv_len[w.path_leaf_node[r["unique_paths"]]].astype(np.int64)
    warps = torch.cuda.get_device_properties(0).multi_processor_count * (8 if heads[0] > 8 * heads[1] else 12)
    short = int(np.ceil(lens / 256).sum()) * heads[1]
    want_items = short if short < warps else int(np.ceil(lens / 512).sum()) * heads[1]
    assert int(pipe.attn_ws[:64].view(torch.int32)[4]) == want_items
    paths = r["unique_paths"]
    sample = np.unique(np.concatenate([np.arange(0, len(paths), max(1, len(paths) // 40)), [len(paths) - 1]]))
    want, want_lse = oracle.tree_attention_workload(w, paths=paths[sample])
    got, lse = r["out"][sample], r["lse"][sample]
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -9 * 4.6).all()      # (as above)
    assert np.abs(lse - want_lse).max() <= 2e-5


@pytest.mark.parametrize("heads", [(8, 2), (24, 2)])
def test_long_leaf_items_in_the_register_staged_kernel(heads):
    """A pool whose blocks are 17 rows apart, which the streaming kernel does not take: items of 512 keys, groups of up to 8 query
    heads and of more."""
    w = synth.build_tree_workload("staged", sum(heads), heads[0], heads[1], [32], [150], 8, (200, 1100), lambda i, m, rng: 1, device=DEV)
    pipe = DevicePipeline(w, DEV)
    pool = pipe.kv_pool                                          # [page][2][Hkv][16][128]
    padded = torch.full((pool.shape[0], 2, heads[1], 17, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    padded[:, :, :, :16] = pool
    d, blk = pipe.desc, heads[1] * 17 * 128
    d.k_pool, d.v_pool = padded.data_ptr(), padded.data_ptr() + blk * 2
    d.kv_page_stride, d.kv_head_stride, d.kv_token_stride = 2 * blk, 17 * 128, 128
    pipe.attn_ws = B.alloc_workspace(B.ss_tree_attention_workspace_bytes(d), pool.device)
    pipe.step()
    r = pipe.results()
    lens = w.node_kv_len[w.path_leaf_node].astype(np.int64)
    assert int(pipe.attn_ws[:64].view(torch.int32)[4]) == int(np.ceil(lens / 512).sum()) * heads[1]
    sample = np.arange(0, len(lens), 29)
    want, want_lse = oracle.tree_attention_workload(w, paths=r["unique_paths"][sample])
    assert (np.abs(r["out"][sample] - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -9 * 4.6).all()   # (as above)
    assert np.abs(r["lse"][sample] - want_lse).max() <= 2e-5
