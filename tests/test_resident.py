"""The kernel that keeps the state between layers in shared memory: matrices with classes of equal rows and columns.

Tables, optima and plans against the CPU oracle, exact: everything is integers.
"""
import numpy as np
import pytest

from paper_2504_03662_b200 import inputs
from tests.test_gpu_parity import check_batch, galv, oracle_search_many  # noqa: F401  (galv is a fixture)

pytestmark = pytest.mark.gpu


def classed(seed, B, Lmax, S, M, rows, cols, **kw):
    """Random tables whose transition matrices have `rows` distinct rows and `cols` distinct columns, members scattered."""
    w = inputs.random_tables(seed, B, Lmax, S, M, **kw)
    rng = np.random.default_rng(seed)
    for i in range(B):
        r, c = rng.integers(0, rows, S), rng.integers(0, cols, S)
        w.trans_q[i] = rng.integers(0, 2000, (rows, cols), np.int32)[r][:, c]
    return w


# S and classes at the edges: one class, the accumulator widths 4 / 8 / 16, one more than 16 (unstructured), a word more than a warp
@pytest.mark.parametrize("S,rows,cols", [(5, 1, 1), (24, 4, 4), (24, 5, 3), (33, 8, 7), (64, 9, 16), (64, 16, 9), (40, 17, 5), (128, 8, 8)])
@pytest.mark.parametrize("flags", [1, 0, 3, 2])
def test_classes_of_equal_rows_and_columns(orc, galv, S, rows, cols, flags):
    M = 700
    w = classed(900 + S + rows, 6, 7, S, M, rows, cols, ragged=True, mem_lo=0, mem_hi=M // 5, time_hi=4000)
    w.mem_q[1, 2, : S // 2] = M + 3                              # rows that never fit
    w.time_q[2, 1, :] = 9                                        # ties: the lowest strategy must win
    w.mem_q[3, 0, :] = M // 2                                    # the lower half of every later column is +inf
    check_batch(orc, galv, w, flags)


# columns per CTA against shifts: inside the CTA, into the halo, beyond it (read from the owner), from the last column
@pytest.mark.parametrize("n,M,mem_hi", [(1, 500, 90), (2, 1000, 40), (3, 1000, 990), (5, 2880, 700), (8, 2879, 2879), (16, 2880, 1500)])
@pytest.mark.parametrize("S,classes", [(24, 4), (24, 0)])
def test_shifts_across_the_cluster(orc, galv, n, M, mem_hi, S, classes):
    from paper_2504_03662_b200 import binding as gb
    kw = dict(ragged=True, mem_lo=0, mem_hi=mem_hi)
    w = classed(40 + n, 3, 5, S, M, classes, classes, **kw) if classes else inputs.random_tables(40 + n, 3, 5, S, M, **kw)
    w.mem_q[0, 1, 0] = M
    for flags in (gb.STORE_C_FULL, 0, gb.STORE_ARGMIN):
        check_batch(orc, galv, w, flags | gb.CLUSTER_SIZE(n))


def test_some_instances_left_to_the_other_kernels(orc, galv):
    """One batch with structured, unstructured and flagged matrices, too many strategies for an unstructured state."""
    w = classed(7, 9, 6, 60, 3000, 6, 6, mem_lo=0, mem_hi=300, ragged=True)
    rng = np.random.default_rng(1)
    for i in (1, 4, 5):
        w.trans_q[i] = rng.integers(0, 3000, (60, 60), np.int32)
    w.trans_q[3, 2, 2] = -1
    w.L[7] = 0
    for flags in (1, 0, 3):
        sb, res = check_batch(orc, galv, w, flags, idx=[0, 1, 2, 4, 5, 6, 8])
        assert res["status"][[3, 7]].tolist() == [2, 2]


@pytest.mark.parametrize("B,S,rows", [(1, 24, 4), (40, 48, 8), (3, 64, 64), (5, 7, 7)])
def test_host_plans_from_states(orc, galv, B, S, rows):
    """The host entry point keeps the states between the layers where a table would be kept: same optima and plans."""
    from paper_2504_03662_b200.search import HostSearch
    w = classed(60 + B, B, 8, S, 900, rows, rows, mem_lo=0, mem_hi=200, ragged=True)
    hs = HostSearch(galv, w, 1)
    for _ in range(2):
        res = {k: v.copy() for k, v in hs.run().items()}
        ref = oracle_search_many(orc, w, w.time_q, w.mem_q, w.trans_q, list(range(B)))
        for i in range(B):
            Li = int(w.L[i])
            assert res["opt_cost"][i] == ref[i]["opt_cost"] and res["status"][i] == ref[i]["status"], i
            assert (res["plan"][i, :Li] == ref[i]["plan"]).all() and res["mem_used"][i] == ref[i]["mem_used"], i


@pytest.mark.parametrize("twins", [None, (0, 1), (15, 16), (0, 16), (0, 17), (38, 39)])
def test_probe_of_the_first_rows(orc, galv, twins):
    """Which of a matrix's first 17 rows are equal decides who searches the instance, never what is found: no pair, pairs
    at both ends of the 17, pairs the probe does not look at.  (Its warps leave their loops at different pairs.)"""
    w = inputs.random_tables(71, 4, 18, 40, 1100, ragged=True, mem_lo=0, mem_hi=150)
    if twins:
        w.trans_q[1::2, twins[1]] = w.trans_q[1::2, twins[0]]
    for flags in (1, 0):
        check_batch(orc, galv, w, flags)
