"""The library's limits, bit-exact against the oracle: the column kernel's
largest last axis (4096 positions) and largest alphabet (24 letters; 25 falls
back to the generic kernel), the largest alphabet the ABI takes (32 letters,
through the generic tile kernel and both line kernels),
and a long two-sequence problem over several tile waves."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2311_17530_gb300 as msa
from paper_2311_17530_gb300 import msadp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LETTERS = "ABCDEFGHIJKLMNOPQRSTUVWXYZabcdef"


def run_full(p, want_kernel=None):
    want = oracle.align(p.seqs, p.alphabet, p.subst, p.gap, want_tb=True)
    plan = msa.Plan(p.k, p.lens, p.alphabet)
    try:
        if want_kernel is not None:
            assert plan.info().fill_kernel == want_kernel
        d_res, d_sub = msadp.device_inputs(p)
        d_result, d_masks = msadp.device_outputs(sum(p.lens))
        plan.execute(d_res.data_ptr(), d_sub.data_ptr(), p.gap, d_result.data_ptr(), d_masks.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        score, rows, status = msadp.decode_device_result(d_result, d_masks, p.seqs)
        assert status == 0
        assert (score, rows) == (want.score, want.rows)
        tb = plan.read_tb()
        np.testing.assert_array_equal(tb, np.asarray(want.tb).reshape(tb.shape))
    finally:
        plan.close()


def alphabet_problem(seed, k, lens, size):
    rng = np.random.default_rng(seed)
    table = inputs.protein_table(rng, size)
    return inputs.random_problem(seed, k, lens, alphabet=LETTERS[:size], table=table, gap=-6, related=True)


def test_column_kernel_longest_last_axis():
    p = inputs.random_problem(5000, 3, [20, 40, 4095], alphabet=inputs.PROTEIN, related=True)
    run_full(p, want_kernel=2)


@pytest.mark.parametrize("size,kernel", [(24, 2), (25, 1)])
def test_column_kernel_largest_alphabet(size, kernel):
    run_full(alphabet_problem(5100 + size, 3, [45, 37, 52], size), want_kernel=kernel)


@pytest.mark.parametrize("kernel,k,lens", [(1, 4, [13, 11, 14, 40]), (4, 4, [13, 11, 14, 40]),
                                           (5, 4, [13, 11, 14, 40]), (5, 6, [5, 4, 3, 4, 3, 24])])
def test_largest_alphabet_generic_and_line_kernels(kernel, k, lens):
    """32 letters through the generic tile kernel (1), the line kernel (4) and the
    streamed line kernel (5)."""
    msa.msa_config("fill_kernel", kernel)
    try:
        run_full(alphabet_problem(5200 if k == 4 else 5200 + k, k, lens, 32), want_kernel=kernel)
    finally:
        msa.msa_config("fill_kernel", 0)


def test_long_pair():
    run_full(inputs.random_problem(5300, 2, [3000, 2500], related=True))


def near_limit_problem(lens, sign):
    """Scores at the int32 limit: the gap as large as the device's range check lets it be (the pair
    scores near 2 gap, so that a pair's share beside the gaps stays small), all scores near sign * 2^31."""
    k, pair_min = len(lens), sum(min(a, b) for i, a in enumerate(lens) for b in lens[i + 1:])
    table = np.where(np.eye(4, dtype=bool), 5, -4)
    gap = sign * ((2**31 - 2 - 5 * pair_min) // ((k - 1) * sum(lens)))
    p = inputs.random_problem(5400 + sum(lens), k, lens, table=table, gap=gap, related=True)
    p.subst = (table + 2 * gap).astype(np.int32)
    return p


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("lens", [[60, 57], [700, 650], [30, 28, 33], [14, 12, 15, 13], [6, 5, 7, 6, 5, 6]])
def test_scores_at_the_int32_limit(lens, sign):
    """The enumeration (level by level, and depth first beyond 1024 residues or 2048 alignments) and the
    pruned call with its greedy bound keep scores and bounds in 32 bits: exact up to the range check."""
    p = near_limit_problem(lens, sign)
    want = oracle.align_problem(p)
    assert abs(want.score) > 2**31 - 2**17
    for delta, count in ((0, 30), (3, 30), (1 << 40, 30), (2, 2049)):
        got, more = msadp.msa_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, delta, count)
        exp, emore = oracle.align_near_optimal(p.seqs, p.alphabet, p.subst, p.gap, delta, count)
        assert more == emore and [g[:2] for g in got] == [(e.score, e.masks) for e in exp], (delta, count)
    score, rows, st = msadp.msa_align_pruned(p.seqs, p.alphabet, p.subst, p.gap)
    assert (score, rows) == (want.score, want.rows) and want.score - 2**20 < st["lower_bound"] <= want.score
    ext = [4] * p.k
    np.testing.assert_array_equal(msadp.msa_tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext),
                                  oracle.tile_bounds(p.seqs, p.alphabet, p.subst, p.gap, ext).reshape(-1))
