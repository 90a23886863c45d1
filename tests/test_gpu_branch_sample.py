"""ss_branch_sample (+ grouping with ss_dedup_paths) on the GPU against the oracle."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2609_39334_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GOLDEN = os.path.join(os.path.dirname(__file__), "golden")


def run(logits, off, u, T):
    dev = torch.device(DEV)
    n = int(off[-1])
    lg = torch.from_numpy(np.ascontiguousarray(logits, dtype=np.float32)).to(dev)
    of = torch.from_numpy(np.ascontiguousarray(off, dtype=np.int64)).to(dev)
    un = torch.from_numpy(np.ascontiguousarray(u if n else np.zeros(1, np.float32), dtype=np.float32)).to(dev)
    tok = torch.full((max(n, 1),), -3, dtype=torch.int32, device=dev)
    seq = torch.full((max(n, 1),), -3, dtype=torch.int64, device=dev)
    B.ss_branch_sample(lg, of, un, logits.shape[0], logits.shape[1], T, tok, seq)
    torch.cuda.synchronize()
    return tok[:n], seq[:n]


def group(tok, seq):
    """Grouping of the draws with the library's own dedup: children and their potential sizes."""
    n = tok.numel()
    dev = tok.device
    i32 = dict(dtype=torch.int32, device=dev)
    outs = [torch.empty(n, **i32) for _ in range(4)]
    nu = torch.zeros(1, **i32)
    ws = B.alloc_workspace(B.ss_dedup_workspace_bytes(n), dev)
    B.ss_dedup_paths(tok.contiguous(), torch.arange(n + 1, dtype=torch.int64, device=dev), seq.contiguous(), None, n, 0,
                     outs[0], outs[1], outs[2], outs[3], None, nu, ws)
    torch.cuda.synchronize()
    U = int(nu.item())
    return outs[2][:U].cpu().numpy(), outs[3][:U].cpu().numpy()


def test_paper_worked_example_on_gpu():
    kv = {}
    for l in open(os.path.join(GOLDEN, "branch_sampling_example.txt")):
        if l.strip() and not l.startswith("#"):
            k, *v = l.split()
            kv[k] = v
    with np.errstate(divide="ignore"):
        logits = np.log(np.asarray([float(x) for x in kv["probs"]])).astype(np.float32)[None, :]
    u = np.asarray([float(x) for x in kv["uniforms"]], np.float32)
    tok, seq = run(logits, [0, len(u)], u, float(kv["temperature"][0]))
    assert tok.cpu().tolist() == [int(x) for x in kv["tokens"]]
    uniq, mult = group(tok, seq)
    assert mult.tolist() == [int(x) for x in kv["potentials"]]


@pytest.mark.parametrize("S,V,T,maxpot", [(3, 6, 1.0, 5), (16, 1000, 0.8, 40), (8, 4097, 1.3, 8), (4, 151936, 0.8, 32),
                                          (2, 151936, 0.8, 3000), (64, 32000, 0.5, 16)])
def test_branch_sample_vs_oracle(S, V, T, maxpot):
    rng = np.random.default_rng(S * 1000 + V)
    logits = (rng.normal(size=(S, V)) * 3).astype(np.float32)
    logits[rng.random((S, V)) < 0.01] = -np.inf                 # masked tokens
    pot = rng.integers(0, maxpot + 1, size=S)
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    u = rng.random(int(off[-1])).astype(np.float32)
    tok, seq = run(logits, off, u, T)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, T)
    got = tok.cpu().numpy()
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    sure = margin > 1e-12                                       # both sides decide in fp64
    assert np.array_equal(got[sure], want_tok[sure])
    # grouping: children and potential sizes equal the oracle's dedup of the oracle's draws
    if len(got) and sure.all():
        uniq, mult = group(tok, seq)
        r = oracle.dedup(want_tok, np.arange(len(want_tok) + 1), ctx_key=want_seq)
        assert np.array_equal(uniq, r["unique_paths"]) and np.array_equal(mult, r["multiplicity"])
        assert int(mult.sum()) == int(off[-1])


@pytest.mark.parametrize("V", [1, 3, 127, 511, 512, 513, 32767, 32772, 65537])
@pytest.mark.parametrize("kind", ["plain", "offset_up", "offset_down", "cold", "hot", "masked"])
def test_branch_sample_slices_segments_and_ranges(V, kind):
    """Vocabularies at the edges of a warp's slice and its segments, rows inside and outside the table path's range of
    exponents, masks of -inf and of a large negative number, uniforms of exactly 0 and just below 1.  Draws are compared
    where the oracle's distance to a boundary is above 1e-12 of the sum (both sides round at 1e-15)."""
    rng = np.random.default_rng(V)
    S, T = 5, {"cold": 2e-4, "hot": 3e6}.get(kind, 0.8)
    logits = (rng.normal(size=(S, V)) * 3).astype(np.float32)
    logits += np.float32({"offset_up": 3000.0, "offset_down": -700.0}.get(kind, 0.0))
    if kind == "masked":
        logits[:, : V // 3] = -np.inf
        logits[rng.random((S, V)) < 0.2] = -1e9
        logits[:, V - 1] = 1.0                                     # (something to draw)
    pot = np.asarray([1, 33, 0, 70, 4])
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    u = rng.random(int(off[-1])).astype(np.float32)
    u[:40:7] = 0.0
    u[3:60:9] = np.float32(1.0) - np.float32(2.0 ** -24)
    tok, seq = run(logits, off, u, T)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, T)
    got = tok.cpu().numpy()
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    sure = margin > 1e-12
    assert np.array_equal(got[sure], want_tok[sure])
    assert np.array_equal(got[u == 0.0], want_tok[u == 0.0])


@pytest.mark.parametrize("V", [5, 700, 9000, 151936])
@pytest.mark.parametrize("masked", [False, True])
def test_a_row_with_a_nan_draws_its_last_token(V, masked):
    """No cumulative sum exceeds a target that is NaN, wherever the NaN lies: beside ordinary tokens, beside masked ones, in a
    segment that ends with the row, or alone.  The rows around it are not touched."""
    rng = np.random.default_rng(V)
    S = 9
    logits = (rng.normal(size=(S, V)) * 3).astype(np.float32)
    if masked:
        logits[rng.random((S, V)) < 0.3] = -np.inf
        logits[:, 1] = 0.5
    for s, at in ((1, 0), (3, V - 1), (5, V // 2), (6, slice(None))):
        logits[s, at] = np.nan
    off = np.arange(S + 1, dtype=np.int64) * 6
    u = rng.random(6 * S).astype(np.float32)
    u[::6] = 0.0
    tok, _ = run(logits, off, u, 0.8)
    got = tok.cpu().numpy().reshape(S, 6)
    want, _, margin = oracle.branch_sample(logits, off, u, 0.8)
    want, sure = want.reshape(S, 6), margin.reshape(S, 6) > 1e-12
    for s in range(S):
        if np.isnan(logits[s]).any():
            assert (got[s] == V - 1).all() and (want[s] == V - 1).all()
        else:
            assert np.array_equal(got[s][sure[s]], want[s][sure[s]])


def test_targets_between_two_roundings_of_a_slice_end():
    """The end of a warp's slice is rounded one way when the slice is chosen and another when its segment is.  Rows are made whose
    target (u = 1/2) lies between the two: three terms S, f, x in three slices with fl(S + fl(f + x)) above fl(fl(S + f) + x) = a,
    the rest of x's slice masked, and a tail that makes the total 2 a (64 rows scan the rounding of the table's exponentials).
    The draw is x or the tail's first token, never a masked one.  Slices of 1024 tokens, 32 of them over a cluster of two blocks."""
    V, S_rows = 32768, 64
    dev = torch.device(DEV)
    rng = np.random.default_rng(7)
    at_s, at_f, at_x, at_y = 10, 16 * 1024 + 3, 17 * 1024 + 5, [20 * 1024 + i for i in range(3)]
    off = torch.arange(S_rows + 1, dtype=torch.int64, device=dev)
    u = torch.full((S_rows,), 0.5, device=dev)
    tok = torch.empty(S_rows, dtype=torch.int32, device=dev)
    seq = torch.empty(S_rows, dtype=torch.int64, device=dev)
    tried = 0
    while tried < 60:
        l = rng.normal(size=3).astype(np.float32)
        s, f, x = (float(v) for v in np.exp(l.astype(np.float64)))
        a = (s + f) + x
        if not s + (f + x) > a:
            continue
        tried += 1
        logits = torch.full((S_rows, V), -float("inf"), device=dev)
        cols = np.empty((S_rows, 6), np.float32)
        for r in range(S_rows):
            left = a + (r - S_rows // 2) * a * 2.0 ** -53          # the tail's sum, about a
            cols[r, :3] = l
            for i, share in enumerate((1.0 - 2.0 ** -20, 1.0 - 2.0 ** -14, 1.0)):
                y = np.float32(np.log(left * share))
                left -= float(np.exp(np.float64(y)))
                cols[r, 3 + i] = y
        logits[:, [at_s, at_f, at_x] + at_y] = torch.from_numpy(cols).to(dev)
        B.ss_branch_sample(logits, off, u, S_rows, V, 1.0, tok, seq)
        assert set(tok.tolist()) <= {at_x, at_y[0]}


@pytest.mark.parametrize("S", [2, 40, 160])
@pytest.mark.parametrize("V,live", [(151936, 10), (32001, 1), (9000, 8500)])
def test_uniform_zero_draws_the_first_token_with_any_probability(S, V, live):
    """u = 0: the first token whose term is not 0 in fp64, behind masked ones and ones that underflow to 0 (1000 below the
    maximum at T = 0.8); one that is merely tiny (590 below: 1e-320) counts.  Rows on clusters of 8, 2 and 1 blocks."""
    rng = np.random.default_rng(V)
    logits = np.full((S, V), -np.inf, np.float32)
    logits[:, V - live:] = (rng.normal(size=(S, live)) * 3).astype(np.float32)
    logits[1::2, : V // 2] = -900.0
    logits[::4, (V - live) // 2] = logits[::4].max(axis=1) - 590.0
    off = np.arange(S + 1, dtype=np.int64) * 2
    u = np.tile(np.asarray([0.0, 0.5], np.float32), S)
    tok, _ = run(logits, off, u, 0.8)
    want, _, _ = oracle.branch_sample(logits, off, u, 0.8)
    assert np.array_equal(tok.cpu().numpy()[::2], want[::2])


@pytest.mark.parametrize("S", [3, 30, 70, 160])
@pytest.mark.parametrize("V", [700, 9001, 70000])
@pytest.mark.parametrize("kind,T", [("up", 0.8), ("up", 1.1e-3), ("down", 0.8), ("cold", 9e-4), ("cold", 1e-12), ("cold", 2e-30), ("hot", 5e6),
                                    ("hot", 9e29), ("tiny", 1e-32), ("huge", 1e32)])
def test_rows_outside_the_table_path(S, V, kind, T):
    """Rows whose largest exponent is out of range are summed again relative to their maximum: by the table (up, down, cold,
    hot) or by CUDA's exp (temperatures beyond 1e-30 and 1e30), on blocks and on clusters of 2, 4 and 8.  Scores are scaled so
    that there is something to choose from; every third row is an ordinary one, every fourth is partly masked."""
    rng = np.random.default_rng(S + V)
    logits = (rng.normal(size=(S, V)) * 3).astype(np.float32)
    if kind in ("cold", "tiny"):
        logits = (logits * T).astype(np.float32)
    elif kind in ("hot", "huge"):
        logits = (logits.astype(np.float64) * T / 4).astype(np.float32)
    else:
        rows = np.arange(S) % 3 != 1
        logits[rows] += np.float32({"up": 3000.0, "down": -900.0}[kind])
    logits[::4][rng.random(logits[::4].shape) < 0.3] = -np.inf
    logits[::4, V // 2] = logits[::4].max(axis=1)
    pot = rng.integers(0, 6, size=S)
    pot[0] = 70
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    u = rng.random(int(off[-1])).astype(np.float32)
    u[:60:9] = 0.0
    tok, seq = run(logits, off, u, T)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, float(np.float32(T)))
    got, sure = tok.cpu().numpy(), margin > 1e-12
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    assert np.array_equal(got[sure], want_tok[sure]) and np.array_equal(got[u == 0.0], want_tok[u == 0.0])


@pytest.mark.parametrize("S,V,most", [(150, 300, 900), (150, 5000, 700), (151, 32001, 900), (70, 32000, 1200), (40, 700, 3000), (3, 600, 5000)])
@pytest.mark.parametrize("peak", [0.0, 12.0])
def test_many_draws_of_a_row(S, V, most, peak):
    """Rows with more draws than are looked up one by one, beside rows with few, none and just as many as a queue holds; flat
    rows and rows with nearly all of their probability on one token."""
    rng = np.random.default_rng(S + V)
    logits = (rng.normal(size=(S, V)) * 2).astype(np.float32)
    logits[:, V // 3] += np.float32(peak)
    logits[::5, : V // 4] = -np.inf
    pot = rng.integers(0, most + 1, size=S)
    pot[1::7] = rng.integers(0, 70, size=len(pot[1::7]))
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    u = rng.random(int(off[-1])).astype(np.float32)
    u[::97] = 0.0
    tok, seq = run(logits, off, u, 0.9)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, float(np.float32(0.9)))
    got, sure = tok.cpu().numpy(), margin > 1e-12
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    assert np.array_equal(got[sure], want_tok[sure]) and np.array_equal(got[u == 0.0], want_tok[u == 0.0])


@pytest.mark.parametrize("S,V", [(148, 16384), (149, 40961), (222, 151936), (330, 128256)])
@pytest.mark.parametrize("kind", ["flat", "peaked", "masked"])
def test_draws_at_the_boundaries_between_tokens(S, V, kind):
    """Rows that blocks take by themselves (with fp32 sums: test_few_draws_of_many_rows): uniforms that lie on a token's end (to fp32),
    between two ends, at 0 and just below 1; flat rows, rows with all of their
    probability on a few tokens, rows that begin and end with masked ones.  Few and many draws of a row."""
    rng = np.random.default_rng(S + V)
    logits = (rng.normal(size=(S, V)) * (0.0 if kind == "flat" else 3.0)).astype(np.float32)
    if kind == "peaked":
        logits[np.arange(S), rng.integers(0, V, size=S)] = 60.0
    if kind == "masked":
        logits[:, : V // 5] = -np.inf
        logits[:, V - 700:] = -np.inf
    pot = rng.integers(1, 12, size=S)
    pot[::50] = 2500000 // V + 5
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    u = rng.random(int(off[-1])).astype(np.float32)
    for s in range(0, S, 3):
        e = np.exp((logits[s].astype(np.float64) - logits[s].max()) / 0.8)
        c = np.cumsum(e) / e.sum()
        u[off[s]: off[s + 1]] = np.minimum(c[rng.integers(0, V, size=pot[s])], 1.0 - 2.0 ** -24).astype(np.float32)
    u[5::31] = 0.0
    u[7::37] = np.float32(1.0) - np.float32(2.0 ** -24)
    tok, seq = run(logits, off, u, 0.8)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, float(np.float32(0.8)))
    got, sure = tok.cpu().numpy(), margin > 1e-12
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    # (a third of the rows have their targets on the ends: exactly, where 16384 equal logits make those fp32 numbers)
    assert np.array_equal(got[sure], want_tok[sure]) and sure.mean() > 0.5


SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


@pytest.mark.parametrize("rounds,more,V", [(4, 0, 125000), (4, 16, 131072), (5, 9, 100000), (5, 40, 100001), (16, 1, 32000)])
@pytest.mark.parametrize("kind,T", [("plain", 0.8), ("flat", 0.8), ("masked", 0.8), ("nan", 0.8), ("rising", 0.8), ("top", 1.1e-3), ("bottom", 9e5)])
def test_few_draws_of_many_rows(rounds, more, V, kind, T):
    """Whole rounds of rows on single blocks, whose sums are first made in fp32, and none, few and more rows left over: targets on
    the ends of tokens, at 0 and just below 1; rows with none, one, 20 and 130 draws (beyond the quick sums, beyond what is drawn one
    by one); flat rows, masked ones, rows with a NaN, rows whose logits rise by 2^60 and more within a warp's slice, rows whose
    largest exponent is just inside and just outside the range of the sums, at temperatures near the ends of theirs."""
    S = rounds * SMS + more
    rng = np.random.default_rng(rounds + V)
    logits = rng.standard_normal((S, V), dtype=np.float32)
    nat = T / 1.4426950408889634                                # a logit of this is an exponent of 1
    logits *= np.float32(0.0 if kind == "flat" else 2.0 * T)
    if kind == "masked":
        logits[:, : V // 5] = -np.inf
        logits[1::2, V - 700:] = -np.inf
    elif kind == "nan":
        for s, at in ((1, 0), (5, V - 1), (S // 2, V // 2), (S - 1, 7), (9, slice(None))):
            logits[s, at] = np.nan
        logits[S // 2, V // 2 + 64] = 900.0 * nat               # (beside the NaN, in the same lane: the row's largest)
    elif kind == "rising":
        logits += (np.arange(V, dtype=np.float32) / V * 700.0 * nat)[None, :]
    elif kind in ("top", "bottom"):
        edge = {"top": 880.0, "bottom": -190.0}[kind] * nat
        logits[::2] += np.float32(edge)
        logits[::8] += np.float32(edge / 2)                     # (outside)
    pot = np.ones(S, np.int64)
    pot[3::40] = 0
    pot[::50] = 20
    pot[S // 3] = 130
    off = np.concatenate([[0], np.cumsum(pot)]).astype(np.int64)
    assert off[-1] <= 2 * S
    u = rng.random(int(off[-1])).astype(np.float32)
    for s in range(0, S, 9):
        row = logits[s].astype(np.float64)
        if np.isnan(row).any():
            continue
        e = np.exp((row - row.max()) / float(np.float32(T)))
        c = np.cumsum(e) / e.sum()
        u[off[s]: off[s + 1]] = np.minimum(c[rng.integers(0, V, size=pot[s])], 1.0 - 2.0 ** -24).astype(np.float32)
    u[5::31] = 0.0
    u[7::37] = np.float32(1.0) - np.float32(2.0 ** -24)
    tok, seq = run(logits, off, u, T)
    want_tok, want_seq, margin = oracle.branch_sample(logits, off, u, float(np.float32(T)))
    got, bad = tok.cpu().numpy(), np.isnan(logits).any(axis=1)[want_seq]
    sure = (margin > 1e-12) & ~bad
    assert np.array_equal(seq.cpu().numpy(), want_seq)
    assert np.array_equal(got[sure], want_tok[sure]) and sure.mean() > 0.5
    assert np.array_equal(got[(u == 0.0) & ~bad], want_tok[(u == 0.0) & ~bad])
    assert (got[bad] == V - 1).all()


def test_calls_with_few_rows_or_many_draws_are_one_launch():
    """Blocks add up in fp32, with a second launch for the draws that this leaves open, only where both are worth it: many rows of a
    large vocabulary with few draws each (148 rows of 16384, one draw each: 8.2 us in one launch, 20 in two)."""
    def launches(S, V, draws, bound=True):
        lg = torch.zeros((S, V), device=DEV)
        off = torch.arange(S + 1, dtype=torch.int64, device=DEV) * draws
        u = torch.full((S * draws,), 0.5, device=DEV)
        tok = torch.empty(S * draws, dtype=torch.int32, device=DEV)
        seq = torch.empty(S * draws, dtype=torch.int64, device=DEV)
        before = B.ss_launch_count()
        if bound:
            B.ss_branch_sample(lg, off, u, S, V, 0.8, tok, seq)
        else:
            args = [t.data_ptr() for t in (lg, off, u)] + [S, V, 0.8, tok.data_ptr(), seq.data_ptr(), None]
            assert B.lib().ss_branch_sample(*args) == B.SS_OK
        torch.cuda.synchronize()
        return B.ss_launch_count() - before

    assert [launches(SMS, 16384, 1), launches(SMS, 151936, 1), launches(4 * SMS, 131072, 8)] == [1, 1, 1]
    assert launches(4 * SMS, 131072, 2) == 2 and launches(4 * SMS, 131072, 2, bound=False) == 1
