"""ss_candidate_step (shared launches up to 4096 candidates) against the four calls it stands for."""
import numpy as np
import pytest
import torch

from paper_2609_39334_b200 import binding as B
from paper_2609_39334_b200 import synth
from paper_2609_39334_b200.pipeline import DevicePipeline

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NAMES = ("canon", "path_to_unique", "unique_paths", "multiplicity", "slot_out", "num_unique", "u_leaf", "u_q_len",
         "u_q_offsets", "u_q_src", "survivors", "keep", "out", "lse")


def both(w, dedup_flags, seg_offsets=None):
    got = []
    for whole in (False, True):
        pipe = DevicePipeline(w, DEV, dedup_flags=dedup_flags)
        if seg_offsets is not None:
            pipe.seg_offsets = torch.tensor(seg_offsets, dtype=torch.int32, device=DEV)
            pipe.P = len(seg_offsets) - 1
            pipe.survivors = torch.empty((pipe.P, w.top_k), dtype=torch.int32, device=DEV)
        for name in NAMES:
            getattr(pipe, name).fill_(0)
        pipe.multiplicity.fill_(-5)
        if whole:
            pipe.step()
        else:
            pipe.dedup()
            pipe.compact_unique()
            pipe.attention()
            pipe.topk()
        torch.cuda.synchronize()
        assert B.ss_last_device_status(pipe.attn_ws) == B.SS_OK
        got.append(({n: getattr(pipe, n).cpu() for n in NAMES}, B.ss_last_device_status(pipe.topk_ws)))
    return got


# sizes around a warp, the cluster form (96), a thread's paths (1024), the shared-memory form (4096); segments of which the
# selection has as many threads as it would have by itself, and ones (1 x 600, 1 x 4096) that take its own launch
@pytest.mark.parametrize("problems,fanout,flags", [
    (1, 1, 0), (1, 31, 0), (3, 32, 0), (96, 1, 0), (97, 1, 0), (33, 3, B.SS_FLAG_WEAK_HASH), (1, 600, 0), (1, 1023, 0),
    (16, 64, 0), (16, 64, B.SS_FLAG_WEAK_HASH), (205, 5, 0), (1000, 3, 0), (1, 4096, 0), (64, 64, 0), (17, 241, 0)])
def test_step_equals_the_four_calls(problems, fanout, flags):
    w = synth.build_tree_workload("step", problems * 7 + fanout, 4, 2, [32], [fanout], problems, (0, 40),
                                  lambda i, n, rng: int(rng.integers(1, 4)), dup_frac=0.3 if fanout > 1 else 0.0)
    (a, st_a), (b, st_b) = both(w, flags)
    for n in NAMES:
        assert torch.equal(a[n], b[n]), n
    assert st_a == st_b == B.SS_OK


@pytest.mark.parametrize("n", [40, 300])
def test_step_with_uneven_and_bad_segments(n):
    """Segments that leave candidates out in front and behind, empty ones, and one that runs backwards."""
    w = synth.build_tree_workload("step", n, 4, 2, [16], [n], 1, (0, 30), lambda i, m, rng: 1, dup_frac=0.2)
    for seg in ([3, 3, n // 2, n - 5], [0, n // 4, n // 8, n]):
        (a, st_a), (b, st_b) = both(w, 0, seg)
        for name in NAMES:
            assert torch.equal(a[name], b[name]), name
        assert st_a == st_b == (B.SS_OK if list(seg) == sorted(seg) else B.SS_ERR_BAD_INPUT)
