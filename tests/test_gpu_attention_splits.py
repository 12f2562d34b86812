"""The attention kernel at the edges of its splits: queries per kv head on both
sides of every softmax-set configuration, reference maxima that move in the
middle of a job, merges of many pieces, blocks with several small jobs, and
extreme calls (suffix lengths left in global memory, a job of thousands of
pieces).  Against the fp64 oracle with the
bounds of the other attention tests."""
import numpy as np
import pytest

from paper_2607_20791_gb300 import workloads
from test_gpu_attention import _check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("nq", [1, 8, 9, 16, 17, 24, 25, 32, 33, 48, 49, 64, 65, 72, 73, 96, 97, 128])
def test_query_counts(gpu_lib, nq, D):
    # nq queries per kv head as rows x heads; ragged lengths, an empty suffix, and
    # split and whole jobs (17 blocks for 6 jobs)
    rpg = next(r for r in (16, 12, 11, 9, 8, 7, 5, 4, 3, 2, 1) if nq % r == 0)
    rng = np.random.default_rng(nq * 1000 + D)
    G = 3
    case = workloads.make_attn_case("nq", G, rpg, 2 * (nq // rpg), 2, D, [130, 777, 16],
                                    rng.integers(0, 70, G * rpg), seed=nq + D,
                                    row_active=(rng.random(G * rpg) > 0.1).astype(np.uint8))
    _check(case, _run(case, num_ctas=17))
    _check(case, _run(case))


@pytest.mark.parametrize("nq_rows,heads", [(2, 4), (5, 4), (9, 4), (9, 8), (16, 8)])
def test_moving_maxima(gpu_lib, nq_rows, heads):
    # scores of standard deviation ~20: a query's maximum moves by more than 2^8
    # again and again along a job, in every configuration's rescale path
    case = workloads.make_attn_case("moving", 2, nq_rows, heads, 1, 128, [900, 1500],
                                    np.arange(2 * nq_rows) * 9 % 100, seed=nq_rows * heads)
    case.softmax_scale = 2.0
    _check(case, _run(case, num_ctas=5))
    _check(case, _run(case))


@pytest.mark.parametrize("D,rpg,heads", [(128, 5, 32), (64, 3, 8), (128, 16, 64)])
def test_merge_of_many_pieces(gpu_lib, D, rpg, heads):
    # one prompt over the whole chip: every job is merged from about 19 pieces
    case = workloads.make_attn_case("single", 1, rpg, heads, 8, D, [2500], np.arange(rpg) * 13, seed=D + rpg)
    _check(case, _run(case))


@pytest.mark.parametrize("D,rpg,heads", [(128, 5, 4), (64, 1, 1), (64, 15, 4), (128, 9, 8), (128, 16, 8)])
@pytest.mark.parametrize("pieces", [2, 3, 5, 6])
def test_fold_of_few_pieces(gpu_lib, D, rpg, heads, pieces):
    # one job in exactly `pieces` blocks, on both sides of the most that is folded
    # in the K ring (4 others, fewer where the partials are large), and the same
    # with whole jobs before the split ones; some pieces hold suffix pages only
    rng = np.random.default_rng(pieces)
    act = np.ones(rpg, np.uint8)
    act[rpg // 2] = rpg < 2
    case = workloads.make_attn_case("fold", 1, rpg, heads, 1, D, [330], rng.integers(0, 60, rpg), seed=pieces,
                                    row_active=act)
    _check(case, _run(case, num_ctas=pieces))
    case = workloads.make_attn_case("fold2", 6, rpg, heads, 1, D, [20, 1, 900, 33, 0, 700],
                                    rng.integers(0, 60, 6 * rpg), seed=pieces)
    _check(case, _run(case, num_ctas=pieces + 2))


@pytest.mark.parametrize("G", [1, 2, 31, 32, 33])
@pytest.mark.parametrize("ctas", [2, 7, 40, 0])
def test_pages_dealt_to_blocks(gpu_lib, G, ctas):
    # both sides of the 32 groups up to which a job's end counts as pages, with
    # empty and inactive groups, jobs of a page, and ends on both sides of a block's
    # bounds (2 to about 150 blocks)
    rng = np.random.default_rng(G * 100 + ctas)
    plen = rng.integers(1, 400, G)
    plen[G // 3::5] = 0
    plen[G // 2] = 16
    act = (rng.random(2 * G) > 0.15).astype(np.uint8)
    act[2 * (G // 4):2 * (G // 4) + 2] = G < 2
    case = workloads.make_attn_case("dealt", G, 2, 6, 3, 64 if G % 2 else 128, plen, rng.integers(0, 40, 2 * G),
                                    seed=G + ctas, row_active=act)
    _check(case, _run(case, num_ctas=ctas))


def test_blocks_with_several_small_jobs(gpu_lib):
    # three blocks for 40 jobs of 1-4 pages: pieces follow one another with one group each
    rng = np.random.default_rng(3)
    case = workloads.make_attn_case("smalljobs", 20, 2, 4, 2, 128, rng.integers(1, 50, 20), rng.integers(0, 10, 40),
                                    seed=3)
    _check(case, _run(case, num_ctas=3))


def test_suffix_lengths_in_global_memory(gpu_lib):
    # 48000 rows: their suffix lengths do not fit shared memory
    rng = np.random.default_rng(11)
    G, rpg = 3000, 16
    case = workloads.make_attn_case("rows", G, rpg, 1, 1, 64, rng.integers(0, 20, G), rng.integers(0, 16, G * rpg),
                                    seed=11)
    rows = [r for g in (0, 1, 777, 1500, 2999) for r in range(g * rpg, g * rpg + rpg)]
    _check(case, _run(case), rows=rows)


def test_job_of_thousands_of_pieces(gpu_lib):
    # a page per block: a merge of hundreds of rounds
    case = workloads.make_attn_case("pieces", 1, 2, 2, 1, 64, [330000], [5, 20], seed=12)
    _check(case, _run(case, num_ctas=40000))
