"""Optimal and near-optimal alignment enumeration on the device (section 6:
further solutions by forking at equally ranked paths or within a user
threshold) against the oracle's enumeration, item by item: the same alignments
(move masks), in the same order, with the same scores, the same count and the
same "more left" flag, for thresholds 0, 1 and 3 and several caps; k = 2 .. 5
(row-major kept scores for k <= 3, tile-major for k >= 4), the paper's
ties-heavy +1/0/-1/0 scheme and random tables."""
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
    for i, lens in enumerate([(5, 6), (12, 9), (4, 5, 4), (7, 6, 8), (3, 4, 3, 4), (6, 5, 7, 6), (3, 2, 3, 3, 2)]):
        out.append(inputs.random_problem(8000 + i, len(lens), list(lens), table=PAPER_TABLE, gap=-1))
        out.append(inputs.random_problem(8100 + i, len(lens), list(lens), alphabet=inputs.PROTEIN, related=True))
    return out


def check(p, delta, max_count):
    got, more = msadp.msa_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, delta, max_count)
    want, wmore = oracle.align_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, delta, max_count)
    assert more == wmore, (p.name, delta, max_count)
    assert len(got) == len(want), (p.name, delta, max_count, len(got), len(want))
    for a, (g, w) in enumerate(zip(got, want)):
        assert g[1] == w.masks, (p.name, delta, a)
        assert g[0] == w.score, (p.name, delta, a)
        assert g[2] == w.rows, (p.name, delta, a)
    return got


@pytest.mark.parametrize("p", _problems(), ids=lambda p: p.name)
@pytest.mark.parametrize("delta,max_count", [(0, 200), (1, 200), (3, 7), (0, 1)])
def test_enumeration_matches_oracle(p, delta, max_count):
    got = check(p, delta, max_count)
    if delta == 0:  # the first optimal alignment is the single-alignment traceback's
        score, rows = msa.msa_align(p.seqs, p.alphabet, p.subst, p.gap)
        assert (got[0][0], got[0][2]) == (score, rows)


def test_larger_problems_and_caps():
    """Longer sequences: the walk's depth spans hundreds of columns; the cap stops
    it with alignments left."""
    for seed, lens in [(8200, [60, 55, 58]), (8201, [14, 12, 15, 13]), (8202, [300, 280])]:
        p = inputs.random_problem(seed, len(lens), lens, table=PAPER_TABLE, gap=-1)
        check(p, 2, 50)


def test_empty_and_degenerate_shapes():
    for lens in [(0, 0), (0, 5), (3, 0, 2), (1, 1, 1, 1)]:
        p = inputs.random_problem(8300 + sum(lens), len(lens), list(lens), table=PAPER_TABLE, gap=-1)
        check(p, 1, 100)


def test_bad_arguments():
    p = inputs.random_problem(8400, 3, [4, 4, 4])
    with pytest.raises(msa.MsaError) as ei:
        msadp.msa_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, -1, 10)
    assert ei.value.code == msa.MSA_EINVAL
    with pytest.raises(msa.MsaError) as ei:
        msadp.msa_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, 0, 0)
    assert ei.value.code == msa.MSA_EINVAL


@pytest.mark.parametrize("lens", [(3, 2, 2, 3, 2, 3), (2, 2, 1, 2, 2, 1, 2), (1, 2, 1, 1, 2, 1, 1, 2)])
def test_more_masks_than_lanes(lens):
    """k = 6 .. 8: a node's masks take two, four and eight rounds of 32."""
    for seed, delta, count in [(8500, 0, 60), (8501, 3, 200)]:
        check(inputs.random_problem(seed + len(lens), len(lens), list(lens), table=PAPER_TABLE, gap=-1), delta, count)


def test_stack_beyond_shared_memory():
    """Sequences whose tables and stack do not fit in shared memory (kept in global memory)."""
    check(inputs.random_problem(8600, 2, [4700, 4650], alphabet=inputs.PROTEIN, related=True), 2, 40)


@pytest.mark.parametrize("max_count", [1, 4, 5, 127, 128, 129, 2047, 2048, 2049])
def test_level_by_level_and_walk_caps(max_count):
    """k = 3: one below, at and above the slots of a warp, of a round of the CTA's lanes and of the most
    rounds a level takes (the depth-first walk beyond)."""
    check(inputs.random_problem(8700, 3, [9, 8, 10], table=PAPER_TABLE, gap=-1), 5, max_count)


@pytest.mark.parametrize("lens", [(512, 512), (512, 513), (1020, 4), (0, 1024)])
def test_level_by_level_longest(lens):
    """The longest sequences that go level by level, and one residue more."""
    check(inputs.random_problem(8800, 2, list(lens), alphabet=inputs.PROTEIN, related=True), 1, 20)


@pytest.mark.parametrize("lens", [(127, 15), (128, 16), (129, 33), (31, 31, 7), (32, 32, 8), (33, 31, 40), (31, 33, 70),
                                  (3, 3, 100), (64, 2, 3)])
def test_scores_kept_by_the_band_and_column_kernels(lens):
    """Edges of the bands, the groups of columns and the 32 x 32 columns the kept scores are laid out by."""
    for delta in (0, 2):
        check(inputs.random_problem(8900 + sum(lens), len(lens), list(lens), alphabet=inputs.PROTEIN, related=True),
              delta, 60)


@pytest.mark.parametrize("k", range(2, 9))
def test_every_sequence_empty(k):
    """No residue at all: one alignment of no columns, level by level (its only slot stands at the
    origin, where there is no residue code to read) and by the depth-first walk (max_count = 2049)."""
    for max_count in (1, 4, 2049):
        p = inputs.random_problem(9000 + k, k, [0] * k, alphabet=inputs.PROTEIN)
        assert check(p, 3, max_count) == [(0, [], [""] * k)]
