"""Exact search-space pruning on the device (section 6: search only the
partitions where an optimal alignment can lie) against the oracle:

* the device's tile bounds equal oracle_tile_bounds element by element, for
  several extents and k = 2 .. 5;
* the pruned fill gives the full oracle's score and alignment (the same tie
  rule), with the device's own lower bound, with the optimum itself as the
  bound, and with a bound too low to leave anything out;
* the tiles it leaves out are those whose bound is below L, and the oracle's DP
  with exactly those cells left out gives the same result;
* the device's lower bound never exceeds the optimum, and related sequences get
  tiles left out;
* a bound above the optimum is reported, not answered."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2311_17530_gb300 as msa
from paper_2311_17530_gb300 import msadp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PAPER_TABLE = np.eye(4, dtype=np.int32)  # section 5.2: +1 match, 0 mismatch, gap -1


def _problems():
    out = []
    shapes = [(40, 37), (150, 170), (20, 24, 22), (45, 40, 50), (9, 11, 10, 12), (14, 13, 15, 12), (6, 7, 5, 6, 7)]
    for i, lens in enumerate(shapes):
        out.append(inputs.random_problem(9000 + i, len(lens), list(lens), alphabet=inputs.PROTEIN, related=True))
        out.append(inputs.random_problem(9100 + i, len(lens), list(lens), alphabet=inputs.DNA, related=False))
    out.append(inputs.random_problem(9200, 3, [30, 28, 33], table=PAPER_TABLE, gap=-1))
    return out


def plan_extents(k, lens):
    """Tile extents of the generic tile kernel for this shape (the pruned fill's tiles)."""
    msa.msa_config("fill_kernel", 1)
    try:
        ext, grid = msa.msa_tile_shape(lens)
    finally:
        msa.msa_config("fill_kernel", 0)
    return ext, grid


@pytest.mark.parametrize("p", _problems(), ids=lambda p: p.name)
def test_tile_bounds_match_oracle(p):
    for ext in ([3] * p.k, [5] * p.k, [1] + [4] * (p.k - 1), plan_extents(p.k, p.lens)[0]):
        got = msadp.msa_tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext)
        want = oracle.tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext).reshape(-1)
        np.testing.assert_array_equal(got, want, err_msg=f"{p.name} {ext}")


@pytest.mark.parametrize("p", _problems(), ids=lambda p: p.name)
def test_pruned_fill_matches_full_oracle(p):
    want = oracle.align_problem(p)
    score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap)
    assert (score, rows) == (want.score, want.rows), p.name
    assert st["lower_bound"] <= want.score
    assert 0 <= st["tiles_skipped"] <= st["tiles"] and 0 <= st["cells_skipped"] <= st["cells"]
    # the same with the optimum as the bound (the tightest exact bound)
    score2, rows2, st2 = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=want.score)
    assert (score2, rows2) == (want.score, want.rows)
    assert st2["tiles_skipped"] >= st["tiles_skipped"]
    # a bound below every tile's: nothing left out
    score3, rows3, st3 = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=-(1 << 40))
    assert (score3, rows3) == (want.score, want.rows) and st3["tiles_skipped"] == 0


@pytest.mark.parametrize("p", _problems()[::3], ids=lambda p: p.name)
def test_left_out_tiles_are_those_below_the_bound(p):
    """Rebuild the set of left-out cells from the device bounds and L, and run the
    oracle's DP without them: the same score and alignment, and the same count."""
    want = oracle.align_problem(p)
    score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=want.score)
    ext, grid = plan_extents(p.k, p.lens)
    bounds = msadp.msa_tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext).reshape(grid)
    out_tiles = bounds < want.score
    assert int(out_tiles.sum()) == st["tiles_skipped"]
    ex = np.zeros([n + 1 for n in p.lens], dtype=np.uint8)
    for t in zip(*np.nonzero(out_tiles)):
        ex[tuple(slice(c * e, (c + 1) * e) for c, e in zip(t, ext))] = 1
    assert int(ex.sum()) == st["cells_skipped"]
    got = oracle.align_excluding(p.seqs, p.alphabet, p.subst, p.gap, ex)
    assert (got.score, got.rows) == (want.score, want.rows) == (score, rows)


def test_related_sequences_leave_tiles_out():
    """Related sequences: the device's feasible alignment is close to the optimum
    and most of the tensor lies below it."""
    for seed, lens in [(9300, [120, 110, 130]), (9301, [40, 42, 38, 41])]:
        p = inputs.random_problem(seed, len(lens), lens, alphabet=inputs.PROTEIN, related=True)
        want = oracle.align_problem(p)
        score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap)
        assert (score, rows) == (want.score, want.rows)
        assert st["cells_skipped"] > st["cells"] // 4, st


def test_bound_above_the_optimum_is_reported():
    p = inputs.random_problem(9400, 3, [25, 22, 27], alphabet=inputs.PROTEIN, related=True)
    want = oracle.align_problem(p)
    with pytest.raises(msa.MsaError) as ei:
        msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=want.score + 1000)
    assert ei.value.code == msa.MSA_EINVAL


@pytest.mark.parametrize("lens", [(1024, 33), (1023, 31), (1100, 1090), (64, 63), (127, 130), (130, 150, 140), (65, 20, 90, 22),
                                  (8, 9, 7, 8, 9, 8), (6, 5, 6, 7, 5, 6, 6), (4, 5, 4, 3, 4, 5, 4, 4)])
def test_passes_boxes_and_mask_rounds(lens):
    """The edges of the pair tables' passes (1024 rows), warps (128 rows) and chunks
    (32 columns), of the greedy walk's boxes and of its rounds of 32 masks (k >= 6)."""
    for seed, related in ((9300, True), (9301, False)):
        p = inputs.random_problem(seed + len(lens), len(lens), list(lens), alphabet=inputs.PROTEIN, related=related)
        ext = plan_extents(p.k, p.lens)[0]
        np.testing.assert_array_equal(msadp.msa_tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext),
                                      oracle.tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext).reshape(-1))
        want = oracle.align_problem(p)
        score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap)
        assert (score, rows) == (want.score, want.rows), p.name
        assert st["lower_bound"] <= want.score
        # the walk takes the largest U at every step: its score is the oracle's lower-bound walk's, cell by cell
        assert st["lower_bound"] == greedy_score(p)


def greedy_score(p):
    """The greedy feasible alignment's score from the oracle's pairwise tables."""
    import itertools
    k, lens = p.k, p.lens
    fb = {(i, j): np.add(*oracle.pair_tables(p.seqs[i], p.seqs[j], p.alphabet, p.subst, p.gap)[:2])
          for i, j in itertools.combinations(range(k), 2)}
    x, score = [0] * k, 0
    while x != list(lens):
        best = None
        for m in range(1, 1 << k):
            y = [v + (m >> i & 1) for i, v in enumerate(x)]
            if any(v > n for v, n in zip(y, lens)):
                continue
            u = sum(int(t[y[i], y[j]]) for (i, j), t in fb.items())
            if best is None or u > best[0]:
                best = (u, m, y)
        _, m, x = best
        for i, j in fb:
            a, b = m >> i & 1, m >> j & 1
            score += (int(p.subst[p.alphabet.index(p.seqs[i][x[i] - 1]), p.alphabet.index(p.seqs[j][x[j] - 1])])
                      if a and b else p.gap if a or b else 0)
    return score


@pytest.mark.parametrize("k,lens", [(6, [20, 20, 21, 22, 20, 21]), (5, [40, 39, 41, 40, 38])])
def test_large_tensors_with_most_tiles_left_out(k, lens):
    """Beyond 8e7 cells with most of them left out the generic tile kernel fills the rest: the same
    score and alignment as the fill of every cell."""
    p = inputs.random_problem(9950 + k, k, lens, alphabet=inputs.PROTEIN, related=True)
    score, rows, stats = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap)
    assert stats["cells"] >= 8e7 and stats["cells_skipped"] > 0.8 * stats["cells"]
    assert (score, rows) == msa.msa_align(p.seqs, p.alphabet, p.subst, p.gap)


SKIPPING = [(150, 170), (300, 40), (45, 40, 50), (60, 64, 58), (20, 22, 19, 24), (9, 11, 10, 12, 8), (7, 8, 6, 7, 8, 6),
            (5, 6, 4, 5, 6, 5, 4), (3, 4, 3, 4, 3, 4, 3, 2)]


@pytest.mark.parametrize("related", [True, False])
@pytest.mark.parametrize("lens", SKIPPING)
def test_fill_that_leaves_tiles_out(lens, related):
    """The tile kernel's fill without the tiles the bound rules out, for every k: the device's bound, the
    optimum, a bound that rules out nothing, and bounds above the optimum, which leave the corner
    unreachable or its best remaining path below the bound."""
    p = inputs.random_problem(9500 + sum(lens) + related, len(lens), list(lens), alphabet=inputs.PROTEIN, related=related)
    want = oracle.align_problem(p)
    msa.msa_config("fill_kernel", 1)
    try:
        for bound in (None, want.score, -(1 << 40)):
            score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=bound)
            assert (score, rows) == (want.score, want.rows), bound
        assert st["tiles_skipped"] == 0
        for above in (1, 50, 1 << 40):
            with pytest.raises(msa.MsaError) as ei:
                msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap, lower_bound=want.score + above)
            assert ei.value.code == msa.MSA_EINVAL
    finally:
        msa.msa_config("fill_kernel", 0)
