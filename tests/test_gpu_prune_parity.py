"""GPU parity of esp_metric_prune against the CPU oracle, through the C ABI.

Bars: integer outputs (histogram counts, permutation, metadata, kept values as bit patterns, swap and near-tie counts)
bit-exact; fp64 channel statistics within 1e-12 relative (the GPU adds the same exact squares in a different order and
uses a different log implementation).

Everything after the score is integer or exactly rounded fp64 work, so it is compared without any tolerance and without
any excuse: the GPU's score is first held to the oracle's at 1e-12, then the oracle is run on the GPU's OWN score and the
permutation, metadata, kept values, swap count, the three near-tie counts and the three objectives must all be identical.
"""
import math

import numpy as np
import pytest

from oracle import esparse_oracle as orc
from paper_2310_15929_b200 import inputs

pytestmark = pytest.mark.gpu

STAT_RTOL = 1e-12


def layer(seed, No, C, T, outliers=3):
    g = np.random.default_rng(seed)
    W = (g.standard_normal((No, C)) * 0.02).astype(np.float16)
    X = g.standard_normal((T, C))
    X[:, g.choice(C, outliers, replace=False)] *= 25
    return W, X.astype(np.float16)


def assert_identical_to_oracle(g, ref, check_stats=True):
    """Every discrete output and every exactly-rounded fp64 output of one esp_metric_prune call against the oracle's
    result for the same score: no tolerance, no excuse."""
    vals, meta, perm = g.host()
    assert np.array_equal(perm, ref.theta)
    assert np.array_equal(meta, ref.meta)
    assert np.array_equal(vals.view(np.uint16), ref.vals.view(np.uint16))
    if check_stats:
        assert g.stats.near_tie_groups == int(ref.near_tie_groups.sum())
        assert g.stats.near_tie_sort == ref.near_tie_sort
        assert g.stats.near_tie_swaps == ref.lbs.near_tie_swaps
        assert g.stats.lbs_swaps_total == ref.lbs.swaps_total
        assert g.stats.obj_identity == ref.obj_identity           # same exact sums, same order of additions
        assert g.stats.obj_after_gns == ref.obj_after_gns
        assert g.stats.obj_after_lbs == ref.obj_after_lbs


def assert_statistics(g, X, alpha, **score_kw):
    """AM_c, IR_c, s_c of the GPU against the oracle's at the statistics bar; returns the GPU's score."""
    am, ir = orc.channel_norm(X), orc.channel_entropy(X, global_range=bool(score_kw.pop("global_range", False)))
    s = orc.channel_score(ir, am, alpha, **score_kw)
    assert np.allclose(g.norm.cpu().numpy(), am, rtol=STAT_RTOL, atol=0)
    assert np.allclose(g.entropy.cpu().numpy(), ir, rtol=STAT_RTOL, atol=1e-14)
    gs = g.score.cpu().numpy()
    assert np.allclose(gs, s, rtol=STAT_RTOL, atol=1e-14)
    return gs


@pytest.mark.parametrize("No,C,T", [(512, 512, 128), (200, 264, 333), (96, 1024, 77)])
def test_channel_statistics(No, C, T):
    from tests.gpu_util import GpuPrune
    W, X = layer(100 + C, No, C, T)
    X[:, 5] = 3.0                                              # a constant channel: entropy exactly 0
    X[: T // 2, 6] = -1.0; X[T // 2:, 6] = 1.0                 # two values
    alpha = 1.0 / math.sqrt(T)
    g = GpuPrune(W, X, alpha, use_lbs=0)
    assert_statistics(g, X, alpha)
    assert g.entropy[5].item() == 0.0
    if T % 2 == 0:
        assert abs(g.entropy[6].item() - math.log(2)) < 1e-14


@pytest.mark.parametrize("No,C,T,block", [(512, 512, 128, 256), (200, 264, 90, 256), (130, 520, 64, 128), (64, 64, 50, 16)])
def test_shuffle_select_compress_bit_exact_given_oracle_scores(No, C, T, block):
    """With the oracle's s_c handed in, everything downstream must be identical bit for bit."""
    from tests.gpu_util import GpuPrune
    W, X = layer(200 + C, No, C, T)
    alpha = 1.0 / math.sqrt(T)
    ref = orc.metric_prune(W, X, alpha, lbs_block=block)
    g = GpuPrune(W, None, alpha, score=ref.score, lbs_block=block)
    assert_identical_to_oracle(g, ref)
    assert ref.lbs.swaps_total > 0


@pytest.mark.parametrize("No,C,block,cap", [(1100, 520, 256, 0), (1024, 256, 256, 12), (2100, 264, 256, 6)])
def test_block_shuffle_tall_weights_bit_exact(No, C, block, cap):
    """Several chunks of the bounds' table (256 rows each), with a ragged last block of channels and slices of the clusters that end in a
    ragged eight rows.  (The exact kernels' chunks: test_block_shuffle_exact_kernels_on_tall_weights.)"""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(7000 + No)
    W = (g0.standard_normal((No, C)) * 0.02 * np.sqrt(4.0 / g0.chisquare(4.0, size=(No, 1)))).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_block=block, lbs_max_swaps=cap)
    g = GpuPrune(W, None, 1.0, score=s, lbs_block=block, lbs_max_swaps=cap)
    assert_identical_to_oracle(g, ref)
    assert ref.lbs.swaps_total > 0


@pytest.mark.parametrize("kind", ["equal_scores", "zero_scores", "negative_scores", "large_weights", "ties_in_some_rows"])
@pytest.mark.parametrize("No,C,block,cap", [(40, 264, 256, 0), (1100, 256, 256, 5), (67, 48, 12, 0)])
def test_block_shuffle_rows_that_fp32_cannot_decide(kind, No, C, block, cap):
    """Rows with equal products (settled by position), rows with |w| >= 0.5, blocks with scores that are zero or negative -- all rows of a
    weight or a few among regular ones, in short and long slices: whichever kernels decide them."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8100 + No)
    W = (g0.standard_normal((No, C)) * (1.5 if kind == "large_weights" else 0.02)).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    if kind == "equal_scores":
        s[:] = 2.5
    elif kind == "zero_scores":
        s[::5] = 0.0
    elif kind == "negative_scores":
        s[::7] *= -1.0
    elif kind == "ties_in_some_rows":
        s[1::2] = s[::2]
        W[::6, 1::2] = W[::6, ::2]
        W[3::6, ::3] = 0.0
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_block=block, lbs_max_swaps=cap)
    g = GpuPrune(W, None, 1.0, score=s, lbs_block=block, lbs_max_swaps=cap)
    assert_identical_to_oracle(g, ref)


@pytest.mark.parametrize("No", [1, 3, 192 * 16, 192 * 16 + 1, 1024 * 16 + 5])
def test_block_shuffle_row_slices(No):
    """Rows dealt to the CTAs of one block's cluster: fewer rows than CTAs, slices of a chunk and of more than one."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8200 + No)
    W = (g0.standard_normal((No, 64)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(64)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_max_swaps=6)
    g = GpuPrune(W, None, 1.0, score=s, lbs_max_swaps=6)
    assert_identical_to_oracle(g, ref)


@pytest.mark.parametrize("block", [4, 8, 60, 64])
@pytest.mark.parametrize("No,C", [(33, 8), (48, 64), (300, 264)])
def test_block_shuffle_narrow_blocks(No, C, block):
    """Narrow blocks, whose clusters come to their first exchange of winners with next to no set-up: a single group (no pair
    at all), two groups, a width that is no power of two, a ragged last block."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8300 + No)
    W = (g0.standard_normal((No, C)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_block=block)
    g = GpuPrune(W, None, 1.0, score=s, lbs_block=block)
    assert_identical_to_oracle(g, ref)


@pytest.mark.parametrize("block", [12, 28, 32, 36, 128])
def test_block_shuffle_rows_told_apart_in_blocks_of_every_width(block):
    """Two channels of a block that tie in every third row, at the widths where kernels and layouts change.  (The sort that finds such rows
    for the exact kernels: test_block_shuffle_exact_kernels_in_blocks_of_every_width.)"""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8400 + block)
    No, C = 90, 264
    W = (g0.standard_normal((No, C)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    perm = g0.permutation(C).astype(np.int32)                 # the order the shuffle starts from
    for b0 in range(0, C, block):
        first, last = perm[b0], perm[min(C, b0 + block) - 1]
        s[last] = s[first]
        W[::3, last] = W[::3, first]
    theta, info = orc.local_block_shuffle(W, s, perm, block)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=block)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps


@pytest.mark.parametrize("No", [16 * 512, 16 * 512 + 1, 16 * 1024 + 8 * 16 + 1])
def test_block_shuffle_bound_sums_at_the_edges_of_folds_and_chunks(No):
    """Slices of one fold (512 rows of a CTA), of a row more, of a chunk (1024) and some rows."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8500 + No)
    W = (g0.standard_normal((No, 64)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(64)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_max_swaps=6)
    g = GpuPrune(W, None, 1.0, score=s, lbs_max_swaps=6)
    assert_identical_to_oracle(g, ref)
    assert ref.lbs.swaps_total == 6


@pytest.mark.parametrize("kind", ["tied_from_the_start", "tied_later", "few_ties", "far_apart", "negative", "very_far_apart", "not_finite"])
@pytest.mark.parametrize("cap", [0, 9])
def test_block_shuffle_handed_to_the_exact_kernels(kind, cap):
    """Blocks that bounds cannot decide: dozens of tied pairs at the first swap, or only once the wide channels have found their places; scores
    too far apart, a weight that is not finite.  One block among others that need no help.  And what needs none: a tie that is settled by
    itself (two equal channels), one score far below the others, a negative one."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8600)
    No, C, block = 120, 264, 64
    W = (g0.standard_normal((No, C)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    perm = g0.permutation(C).astype(np.int32)
    first = perm[:block]                                      # the channels of the first block
    if kind == "tied_from_the_start":
        W[:, first] = W[:, first[np.arange(block) % 6]]
        s[first] = 2.0
    elif kind == "tied_later":
        small = first[block // 2:]
        W[:, small] = (W[:, small[np.arange(block // 2) % 5]].astype(np.float32) / 64).astype(np.float16)
        s[small] = 1.0
    elif kind == "few_ties":
        W[:, first[9]], s[first[9]] = W[:, first[40]], s[first[40]]
    elif kind == "not_finite":
        W[17, first[23]] = np.inf
    else:
        s[first[7]] = {"far_apart": 2.0 ** -70, "negative": -3.0, "very_far_apart": 2.0 ** -220}[kind]
    theta, info = orc.local_block_shuffle(W, s, perm, block, cap)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=block, lbs_max_swaps=cap)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps
    assert g.stats.obj_after_lbs == orc.objective(W, s, theta)
    handed, swaps = g.handed()
    assert handed[1:] == [0, 0, 0, 0]
    assert bool(handed[0]) == (kind not in ("few_ties", "far_apart", "negative") and not (kind == "tied_later" and cap))
    assert (swaps[0] > 0) == (kind == "tied_later" and cap == 0)


@pytest.mark.parametrize("number", [1, 9, 64])
def test_block_shuffle_number_of_blocks_handed_over(number):
    """One block of 64, nine (more than there is room for clusters of 16), all: in large clusters, or in the size for all blocks."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8630)
    No, C, block = 300, 2048, 32
    W = (g0.standard_normal((No, C)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    perm = g0.permutation(C).astype(np.int32)
    chosen = g0.choice(C // block, number, replace=False)
    W[17, perm[chosen * block]] = np.inf
    theta, info = orc.local_block_shuffle(W, s, perm, block)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=block)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps
    assert np.flatnonzero(g.handed()[0]).tolist() == sorted(chosen.tolist())


@pytest.mark.parametrize("No", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("block,equal", [(12, False), (256, False), (256, True)])
def test_block_shuffle_few_rows(No, block, equal):
    """One to three rows are shuffled by the exact kernels from the start, more by bounds first."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8640 + No)
    W = (g0.standard_normal((No, 520)) * 0.02).astype(np.float16)
    s = np.full(520, 2.5) if equal else 1.0 + 3.0 * g0.random(520)
    g = GpuPrune(W, None, 1.0, score=s, lbs_block=block)
    assert_identical_to_oracle(g, orc.metric_prune(W, None, 1.0, score=s, lbs_block=block))
    handed, swaps = g.handed()
    if No < 4:
        assert all(handed) and not any(swaps)


@pytest.mark.parametrize("block", [12, 64, 256])
@pytest.mark.parametrize("every", [1, 4, 10])
def test_block_shuffle_zero_columns_are_decided_by_bounds(every, block):
    """Columns of zeros (a weight that was pruned before) exchange for exactly nothing: no block needs the exact kernels for them.
    (Every second one would: groups that keep both of their other channels in every row tie with each other.)"""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8650 + every)
    W = (g0.standard_normal((150, 264)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(264)
    W[:, ::every] = 0.0
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_block=block)
    g = GpuPrune(W, None, 1.0, score=s, lbs_block=block)
    assert_identical_to_oracle(g, ref)
    assert not any(g.handed()[0])


@pytest.mark.parametrize("kind", ["ordinary", "zero_scores", "negative_scores", "far_apart", "zero_columns", "equal"])
@pytest.mark.parametrize("No,cap", [(100, 1), (700, 7), (17 * 1024, 3)])
def test_block_shuffle_bounds_hold(kind, No, cap):
    """Every entry of the bounds' table, as `cap` swaps have left it (untouched, formed anew, shifted): its distance from the exact gain is at
    most the bound that it carries, and the bound is small against the sums of the block's products."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8690 + No)
    m = 64
    W = (g0.standard_normal((No, m)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(m)
    if kind == "zero_scores":
        s[::7] = 0.0
    elif kind == "negative_scores":
        s[::3] *= -1.0
    elif kind == "far_apart":
        s[::9] *= 2.0 ** -70
    elif kind == "zero_columns":
        W[:, ::7] = 0.0
    elif kind == "equal":
        s[:] = 2.5
    perm = g0.permutation(m).astype(np.int32)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=m, lbs_max_swaps=cap)
    assert g.stats.lbs_swaps_total == cap and g.handed()[0] == [0]
    theta = g.host()[2]
    bits = g.ws[g.ws.numel() - 256 * 256 * 8:].cpu().numpy().view(np.uint64).reshape(256, 256)[:m, :m]
    value = (bits & ~np.uint64(0xFFFF)).view(np.float64)
    error = (bits.astype(np.uint32) << np.uint32(16)).view(np.float32).astype(np.float64)
    # products scaled to 1/2 by a power of two
    a = np.abs(W.astype(np.float64))
    p = a * s * 2.0 ** -(np.frexp(np.abs(s).max())[1] - 1 + 3 + np.frexp(a.max())[1] - 1)
    for pos in range(m):
        mine = theta[pos // 4 * 4: pos // 4 * 4 + 4]
        f2 = np.sort(p[:, [c for c in mine if c != theta[pos]]], axis=1)[:, 1]
        exact = np.maximum(p[:, perm] - f2[:, None], 0.0).sum(0) - np.maximum(p[:, theta[pos]] - f2, 0.0).sum()
        others = ~np.isin(perm, mine)
        assert np.all(np.abs(value[pos] - exact)[others] <= error[pos, others] + 1e-13 * No * (error[pos, others] > 0))
        # (an entry's R, D and S are column sums at most; below 100 additions and 4 S; shifted once per swap)
        assert error[pos, others].max() <= (1 + cap) * 2.0 ** -16 * np.abs(p).sum(0).max()


def handed_over(kind, No, C, block, seed):
    """A weight whose first block the exact kernels take: from the start, by an infinite weight (all rows but that one have products that fp32
    can order), or after some swaps, by ties among narrow channels."""
    g0 = np.random.default_rng(seed)
    W = (g0.standard_normal((No, C)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(C)
    perm = g0.permutation(C).astype(np.int32)
    if kind == "not_finite":
        W[No // 2, perm[min(block, C) - 1]] = np.inf
    else:
        small = perm[block // 2: block]
        W[:, small] = (W[:, small[np.arange(len(small)) % 5]].astype(np.float32) / 64).astype(np.float16)
        s[small] = 1.0
    return W, s, perm


@pytest.mark.parametrize("kind", ["not_finite", "tied_later"])
@pytest.mark.parametrize("No", [192, 193, 1100, 2100, 192 * 16, 192 * 16 + 1, 1024 * 16 + 5])
def test_block_shuffle_exact_kernels_on_tall_weights(kind, No):
    """The exact kernels on the edge between their two row loops (192 rows of the table kernel, of a CTA of the cluster), on one to
    eighteen chunks of the table kernel (928 rows at most) and on slices of more than one chunk; from the start and from where bounds stopped."""
    from tests.gpu_util import GpuPrune
    W, s, perm = handed_over(kind, No, 128, 64, 8670 + No)
    cap = 6 if kind == "not_finite" else 0
    theta, info = orc.local_block_shuffle(W, s, perm, 64, cap)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=64, lbs_max_swaps=cap)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps
    assert g.stats.obj_after_lbs == orc.objective(W, s, theta)
    handed, swaps = g.handed()
    assert [bool(h) for h in handed] == [True, False]
    assert (swaps[0] > 0) == (kind == "tied_later")


@pytest.mark.parametrize("block", [8, 12, 28, 32, 36, 64, 128, 256])
@pytest.mark.parametrize("ties", [False, True])
def test_block_shuffle_exact_kernels_in_blocks_of_every_width(block, ties):
    """Rows whose products fp32 cannot order are found by a sort as wide as the block: none (but the infinite one), or ties between the
    first and the last channels of the block in every third row, at the widths where the sort changes."""
    from tests.gpu_util import GpuPrune
    W, s, perm = handed_over("not_finite", 250, 264, block, 8680 + block)
    if ties:
        first, last = perm[0], perm[block - 2]
        s[last] = s[first]
        W[::3, last] = W[::3, first]
    theta, info = orc.local_block_shuffle(W, s, perm, block)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=block)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps
    assert g.handed()[0][0] == 1


def test_block_shuffle_settles_only_pairs_that_may_gain():
    """Nine channels of score zero in nine groups (36 pairs that exchange for exactly nothing) and two equal channels, whose exchange
    bounds cannot tell from a gain: the last question is about one pair, and is settled without the exact kernels."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8660)
    W = (g0.standard_normal((150, 64)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(64)
    s[0:36:4] = 0.0
    W[:, 41], s[41] = W[:, 50], s[50]
    perm = np.arange(64, dtype=np.int32)
    theta, info = orc.local_block_shuffle(W, s, perm, 64)
    g = GpuPrune(W, None, 1.0, score=s, perm=perm, lbs_block=64)
    assert np.array_equal(g.host()[2], theta)
    assert g.stats.lbs_swaps_total == info.swaps_total and g.stats.near_tie_swaps == info.near_tie_swaps
    assert g.handed()[0] == [0]


@pytest.mark.parametrize("No", [1, 255, 256, 257, 2048, 2049])
def test_objectives_at_the_edges_of_a_warps_rows(No):
    """Group values of both orders: a warp's lanes take 256 rows at a time, a CTA has up to eight warps (2048 rows)."""
    from tests.gpu_util import GpuPrune
    g0 = np.random.default_rng(8700 + No)
    W = (g0.standard_normal((No, 40)) * 0.02).astype(np.float16)
    s = 1.0 + 3.0 * g0.random(40)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_block=16, lbs_max_swaps=2)
    assert_identical_to_oracle(GpuPrune(W, None, 1.0, score=s, lbs_block=16, lbs_max_swaps=2), ref)


def test_llama7b_q_projection_full_size_block_shuffle():
    """Workload 1's q projection whole (4096 x 4096, 16 shuffle blocks, Student-t rows): global shuffle, block shuffle
    capped at 4 swaps per block on both sides (the oracle's table alone is 4.3e9 row evaluations), selection and
    compression, all bit-exact given the same score."""
    from tests.gpu_util import GpuPrune
    wl = inputs.WORKLOADS[1]
    W = inputs.make_weight(wl, "q")
    s = 1.0 + 3.0 * np.random.default_rng(11).random(W.shape[1])
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_max_swaps=4)
    g = GpuPrune(W, None, 1.0, score=s, lbs_max_swaps=4)
    assert_identical_to_oracle(g, ref)
    assert ref.lbs.swaps_total == 4 * 16


@pytest.mark.parametrize("wl_index,lin", [(3, "gate"), (4, "fc1")])
def test_block_shuffle_all_rows_of_the_widest_layers(wl_index, lin):
    """All 22016 / 36864 output rows of the widest LLaMA-65B / OPT-66B linears on one block of 256 input channels: 86 and
    144 chunks of the bounds' table, slices of several chunks in the clusters; two swaps, bit-exact."""
    from tests.gpu_util import GpuPrune
    wl = inputs.WORKLOADS[wl_index]
    W = inputs.make_weight(wl, lin, C=256)
    s = 1.0 + 3.0 * np.random.default_rng(12 + wl_index).random(256)
    ref = orc.metric_prune(W, None, 1.0, score=s, lbs_max_swaps=2)
    g = GpuPrune(W, None, 1.0, score=s, lbs_max_swaps=2)
    assert_identical_to_oracle(g, ref)
    assert ref.lbs.swaps_total == 2


@pytest.mark.parametrize("toggles", [dict(use_gns=0, use_lbs=0), dict(use_gns=1, use_lbs=0), dict(use_gns=0, use_lbs=1),
                                     dict(use_entropy=0), dict(use_norm=0), dict(lbs_max_swaps=5)])
def test_ablation_toggles(toggles):
    from tests.gpu_util import GpuPrune
    W, X = layer(300, 128, 256, 100)
    alpha = 0.25
    kw = dict(use_entropy=True, use_norm=True, use_gns=True, use_lbs=True, lbs_max_swaps=0)
    kw.update({k: (bool(v) if k.startswith("use") else v) for k, v in toggles.items()})
    g = GpuPrune(W, X, alpha, **toggles)
    gs = assert_statistics(g, X, alpha, use_entropy=kw["use_entropy"], use_norm=kw["use_norm"])
    ref = orc.metric_prune(W, X, alpha, score=gs, **kw)       # the oracle on the GPU's own score
    assert_identical_to_oracle(g, ref)
    if not kw["use_lbs"]:
        assert g.stats.lbs_swaps_total == 0 and g.stats.obj_after_lbs == g.stats.obj_after_gns
    if not kw["use_gns"]:                                     # the block shuffle then starts from the identity order
        assert g.stats.near_tie_sort == 0 and g.stats.obj_after_gns == g.stats.obj_identity


def test_config0_end_to_end():
    """Workload 0: 512x512 layer, 128 calibration tokens, 8 outlier channels x20, both values of alpha."""
    from tests.gpu_util import GpuPrune
    wl = inputs.WORKLOADS[0]
    W, X = inputs.make_weight(wl, "fc"), inputs.make_calibration(wl, "fc")
    for alpha in (1.0, 1.0 / math.sqrt(X.shape[0])):
        g = GpuPrune(W, X, alpha)
        gs = assert_statistics(g, X, alpha)
        ref = orc.metric_prune(W, X, alpha, score=gs)
        assert_identical_to_oracle(g, ref)
        assert g.stats.obj_after_lbs >= g.stats.obj_after_gns > 0.0
        # run-to-run determinism
        g2 = GpuPrune(W, X, alpha)
        for a, c in zip(g.host(), g2.host()):
            assert np.array_equal(a.view(np.uint8), c.view(np.uint8))


def test_llama7b_shaped_slice():
    """Config 1 distributions (Student-t rows, 1 % outlier channels x30) on a reduced q-projection:
    all 4096 input channels (16 shuffle blocks), 256 output rows, 2048 calibration tokens."""
    from tests.gpu_util import GpuPrune
    wl = inputs.WORKLOADS[1]
    W = inputs.make_weight(wl, "q", No=256)
    X = inputs.make_calibration(wl, "q", T=2048)
    alpha = 1.0 / math.sqrt(X.shape[0])
    g = GpuPrune(W, X, alpha, lbs_max_swaps=24)
    gs = assert_statistics(g, X, alpha)
    ref = orc.metric_prune(W, X, alpha, score=gs, lbs_max_swaps=24)
    assert_identical_to_oracle(g, ref)


def test_decompress_and_pack_roundtrip():
    import torch
    from paper_2310_15929_b200 import binding as b
    from tests.gpu_util import GpuPrune, DEV
    W, X = layer(400, 136, 264, 60)
    ref = orc.metric_prune(W, X, 0.3)
    g = GpuPrune(W, None, 0.3, score=ref.score)
    out = torch.empty(136, 264, dtype=torch.float16, device=DEV)
    b.esp_decompress(g.vals, g.meta, g.perm, 136, 264, out)
    assert np.array_equal(out.cpu().numpy().view(np.uint16), orc.decompress(ref.vals, ref.meta, ref.theta).view(np.uint16))
    # the packed copy holds exactly the kept values (as a multiset per tile) plus legal metadata
    packed = g.packed.cpu().numpy().reshape(2, 3, 18432)
    tile = packed[0, 0, :16384].view(np.float16).reshape(128, 64)
    unsw = np.empty_like(tile)
    for r in range(128):
        for q in range(8):
            unsw[r, q * 8:(q + 1) * 8] = tile[r, (q ^ (r & 7)) * 8:(q ^ (r & 7)) * 8 + 8]
    assert np.array_equal(unsw.view(np.uint16), ref.vals[:128, :64].view(np.uint16))
    nibbles = packed[:, :, 16384:]
    assert set(np.unique(nibbles & 0xF).tolist()) | set(np.unique(nibbles >> 4).tolist()) <= set(orc.LEGAL_NIBBLES)


@pytest.mark.parametrize("No,C,T", [(96, 256, 200), (200, 1024, 130)])
def test_four_of_eight_pattern(No, C, T):
    """4:8 (Table 1's second pattern): statistics, score, global shuffle in groups of 8, 4-of-8 selection and compression
    against the oracle run on the GPU's own score, bit-exact; the library refuses what 4:8 has no form for."""
    from paper_2310_15929_b200 import binding as b
    from tests.gpu_util import GpuPrune
    W, X = layer(70 + C, No, C, T)
    alpha = 1.0 / math.sqrt(T)
    gp = GpuPrune(W, X, alpha, stats=True, pack=False, n_keep=4, m_group=8, use_lbs=0)
    gs = assert_statistics(gp, X, alpha)
    theta0, near_sort = orc.global_naive_shuffle(orc.channel_mean_metric(W, gs), m_group=8)
    vals_ref, mask_ref, near = orc.select_compress_nm(W, gs, theta0, 4, 8)
    vals, mask, perm = gp.host()
    assert np.array_equal(perm, theta0)
    assert np.array_equal(mask, mask_ref)
    assert np.array_equal(vals.view(np.uint16), vals_ref.view(np.uint16))
    assert gp.stats.near_tie_groups == int(near.sum())
    assert gp.stats.near_tie_sort == near_sort
    with pytest.raises(b.EsparseError) as e:
        GpuPrune(W, X, alpha, stats=False, pack=False, n_keep=4, m_group=8, use_lbs=1)
    assert e.value.status == b.ESP_ERR_UNSUPPORTED
    with pytest.raises(b.EsparseError) as e:
        GpuPrune(W, X, alpha, stats=False, pack=True, n_keep=4, m_group=8, use_lbs=0)
    assert e.value.status == b.ESP_ERR_UNSUPPORTED


@pytest.mark.parametrize("C,splits", [(264, (100, 37, 256, 3)), (1024, (77,)), (512, (1, 1, 700, 5000))])
def test_streaming_calibration_equals_one_shot(C, splits):
    """Chunked statistics (two passes over the chunks) against the oracle on the concatenation: counts bit-exact,
    norm / entropy / score to the statistics bar; then the streamed score drives the same pruning decisions."""
    from tests.gpu_util import GpuPrune, calibrate_in_chunks
    T = sum(splits)
    W, X = layer(900 + C, 128, C, T)
    X[:, 5] = 3.0
    X[-1, 7] = 1000.0                                           # the range of channel 7 is set by the last chunk
    alpha = 1.0 / math.sqrt(T)
    chunks, r = [], 0
    for n in splits:
        chunks.append(X[r: r + n]); r += n
    norm, ent, score, counts, score_d = calibrate_in_chunks(chunks, alpha)
    assert np.array_equal(counts, orc.channel_histogram(X))
    assert counts.sum(axis=1).tolist() == [T] * C
    am, ir = orc.channel_norm(X), orc.channel_entropy(X)
    assert np.allclose(norm, am, rtol=STAT_RTOL, atol=0)
    assert np.allclose(ent, ir, rtol=STAT_RTOL, atol=1e-14)
    assert np.allclose(score, orc.channel_score(ir, am, alpha), rtol=STAT_RTOL, atol=0)
    assert ent[5] == 0.0
    # ablation switches reach the streamed score too
    _, _, s_norm_only, _, _ = calibrate_in_chunks(chunks, alpha, use_entropy=0)
    assert np.allclose(s_norm_only, alpha * am, rtol=STAT_RTOL, atol=0)
    # the streamed score feeds the pruner without the calibration matrix
    ref = orc.metric_prune(W, None, alpha, use_lbs=False, score=score)
    g = GpuPrune(W, None, alpha, score=score, use_lbs=0)
    assert_identical_to_oracle(g, ref)


@pytest.mark.parametrize("T", [300, 6600])
@pytest.mark.parametrize("bins", [2, 54, 55, 108, 109, 110, 512])
def test_histogram_counter_replicas(T, bins):
    """Counts at the bin counts where the number of counter replicas changes, with few and with more than 512 rows per CTA (4096
    channels are dealt to six row slices)."""
    from tests.gpu_util import calibrate_in_chunks
    g0 = np.random.default_rng(1000 + bins)
    C = 4096
    X = (g0.standard_normal((T, C), dtype=np.float32) * np.where(np.arange(C) % 7, 1.0, 20.0).astype(np.float32)).astype(np.float16)
    counts = calibrate_in_chunks([X], 0.1, bins=bins)[3]
    cols = np.unique(np.concatenate([[0, 7, 63, 64, C - 1], g0.choice(C, 60, replace=False)]))
    assert np.array_equal(counts[cols], orc.channel_histogram(np.ascontiguousarray(X[:, cols]), bins))
    assert counts.sum(axis=1).tolist() == [T] * C


@pytest.mark.parametrize("No,C,T", [(128, 264, 333), (96, 1024, 200)])
def test_global_bin_range_variant(No, C, T):
    """Layer-wide bin range (the other reading of Eq. 1): entropy and score to the statistics bar, everything downstream
    identical to the oracle on the GPU's own score, and different from the per-channel reading on this input."""
    from tests.gpu_util import GpuPrune
    W, X = layer(300 + C, No, C, T)
    X[:, 9] = (X[:, 9].astype(np.float32) / 64).astype(np.float16)          # a narrow channel
    alpha = 1.0 / math.sqrt(T)
    g = GpuPrune(W, X, alpha, use_lbs=0, global_bin_range=1)
    gs = assert_statistics(g, X, alpha, global_range=True)
    assert g.entropy[9].item() < 0.5 * orc.channel_entropy(X)[9]
    ref = orc.metric_prune(W, X, alpha, use_lbs=False, global_bin_range=True, score=gs)
    assert_identical_to_oracle(g, ref)


@pytest.mark.parametrize("what", ["histogram", "product"])
def test_shared_memory_size_is_not_lowered_by_another_thread(what):
    """The size of dynamic shared memory that a kernel may be launched with belongs to the process: a thread that launches a kernel
    with much, another that launches it with little, and the first one again."""
    import threading
    from tests.gpu_util import calibrate_in_chunks, pack_on_gpu, spgemm
    g0 = np.random.default_rng(31)
    X = g0.standard_normal((100, 512)).astype(np.float16)
    if what == "histogram":
        def call(much):
            bins = 512 if much else 300
            assert np.array_equal(calibrate_in_chunks([X], 0.1, bins=bins)[3], orc.channel_histogram(X, bins))
    else:
        W = (g0.standard_normal((128, 512)) * 0.02).astype(np.float16)
        ref = orc.metric_prune(W, None, 1.0, score=np.ones(512), use_lbs=False)
        packed = pack_on_gpu(ref.vals, ref.meta)
        want = orc.product(X, ref.vals, ref.meta, ref.theta)
        def call(much):
            Y = spgemm(X, packed, ref.theta, 128, channel_major=True, kernel=4, token_tile=64, split_k=1, pipeline_stages=4 if much else 2)
            assert np.linalg.norm(Y - want) < 1e-3 * np.linalg.norm(want)
    errors, turn = [], [threading.Event() for _ in range(4)]

    def steps(mine):
        for i in mine:
            turn[i].wait(60)
            try:
                call(i != 1)
            except Exception as e:                            # (a failed assertion is reported below, by the test's own thread)
                errors.append((i, repr(e)))
            turn[i + 1].set()
    threads = [threading.Thread(target=steps, args=(m,)) for m in ((0, 2), (1,))]
    for t in threads:
        t.start()
    turn[0].set()
    for t in threads:
        t.join()
    assert errors == []


# --------------------------------------------------------------------------- full width: workloads 2, 3, 4
@pytest.mark.parametrize("wl_index,lin", [(2, "q"), (2, "down"), (3, "down"), (4, "fc2")])
def test_channel_statistics_full_width_full_calibration(wl_index, lin):
    """Norm, entropy and score over all C input channels and all 16 x 2048 calibration tokens of the LLaMA-13B, LLaMA-65B
    and OPT-66B shaped layers (C = 5120, 13824, 22016, 36864).  The GPU processes the whole [T, C] matrix, once through
    esp_metric_prune and once as two uneven chunks through the streaming-calibration calls; the oracle, whose statistics
    are per channel, is applied to a seeded sample of channels: all outlier channels, the channels at the kernels' 64- and
    256-wide boundaries, and random ones.  Counts bit-exact, fp64 statistics to 1e-12."""
    import torch
    from tests.gpu_util import GpuPrune, calibrate_in_chunks, DEV
    wl = inputs.WORKLOADS[wl_index]
    C = wl.linears[lin][1]
    X = inputs.make_calibration(wl, lin)
    T = X.shape[0]
    assert T == 16 * 2048
    g0 = np.random.default_rng(500 + wl_index)
    out = inputs.outlier_channels(wl, lin)
    cols = np.unique(np.concatenate([out[:64], g0.choice(C, 160, replace=False),
                                     [0, 63, 64, 255, 256, C - 257, C - 256, C - 65, C - 64, C - 1]]))
    Xs = np.ascontiguousarray(X[:, cols])
    am, cnt = orc.channel_norm(Xs), orc.channel_histogram(Xs)
    ir = orc.entropy_from_counts(cnt, T)
    alpha = 1.0 / math.sqrt(T)
    s = orc.channel_score(ir, am, alpha)
    # one-shot path (what the benchmark's producer runs); the weight is a thin slice, the statistics do not read it
    W = inputs.make_weight(wl, lin, No=128)
    g = GpuPrune(W, X, alpha, use_lbs=0, stats=False, pack=False)
    assert np.allclose(g.norm.cpu().numpy()[cols], am, rtol=STAT_RTOL, atol=0)
    assert np.allclose(g.entropy.cpu().numpy()[cols], ir, rtol=STAT_RTOL, atol=1e-14)
    assert np.allclose(g.score.cpu().numpy()[cols], s, rtol=STAT_RTOL, atol=0)
    del g
    torch.cuda.empty_cache()
    # streaming path: exposes the counts themselves
    cut = 20000
    norm, ent, score, counts, _ = calibrate_in_chunks([X[:cut], X[cut:]], alpha)
    assert np.array_equal(counts[cols], cnt)
    assert counts.sum(axis=1).tolist() == [T] * C
    assert np.allclose(norm[cols], am, rtol=STAT_RTOL, atol=0)
    assert np.allclose(ent[cols], ir, rtol=STAT_RTOL, atol=1e-14)
    assert np.allclose(score[cols], s, rtol=STAT_RTOL, atol=0)
