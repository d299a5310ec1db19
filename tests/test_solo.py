"""The kernel that keeps an instance's state on one SM: every table, optimum and plan against the one-thread-per-cell kernel,
which other tests tie to the CPU oracle, and against the oracle itself.  Whole numbers: exact.
"""
import numpy as np
import pytest

from paper_2504_03662_b200 import inputs
from tests.test_gpu_parity import INF, check_batch, galv, oracle_search_many  # noqa: F401  (galv is a fixture)
from tests.test_resident import classed

pytestmark = pytest.mark.gpu


def against_reference(galv, w, flags):
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    ref = SearchBuffers(galv, w, flags | gb.KERNEL_REFERENCE)
    ref.dp_search(); ref.backtrack()
    one = SearchBuffers(galv, w, flags | (0 if flags & (gb.STORE_C_FULL | gb.STORE_ARGMIN) else gb.KERNEL_SOLO))
    for t in (one.C, one.A, one.C_last):
        if t is not None:
            t.fill_(77)
    for _ in range(2):
        one.dp_search(); one.backtrack()
        torch.cuda.synchronize()
        assert torch.equal(one.status, ref.status)
        assert torch.equal(one.opt_cost, ref.opt_cost)
        assert torch.equal(one.plan, ref.plan) and torch.equal(one.mem_used, ref.mem_used)
        ok = [i for i in range(w.B) if int(ref.status[i]) in (0, 1)]
        for i in ok:
            Li = int(w.L[i])
            assert torch.equal(one.C_last[i], ref.C_last[i]), i
            if ref.C is not None:
                assert torch.equal(one.C[i, :Li], ref.C[i, :Li]), i
                assert Li == w.Lmax or bool((one.C[i, Li:] == 77).all())          # layers that are not there are not touched
            if ref.A is not None:
                assert torch.equal(one.A[i, :Li], ref.A[i, :Li]), i
    return one


# S and classes at the edges of the accumulator widths (8 / 16 / 32 / 64 rows), of a warp's lanes and of the boxes of collected rows
@pytest.mark.parametrize("S,rows,cols", [(1, 1, 1), (5, 1, 1), (7, 0, 0), (8, 0, 0), (9, 0, 0), (16, 0, 0), (17, 0, 0), (24, 4, 4), (24, 5, 9), (31, 0, 0),
                                         (32, 0, 0), (33, 8, 7), (33, 0, 0), (44, 0, 0), (64, 9, 16), (64, 16, 9), (64, 0, 0), (65, 3, 3), (128, 8, 8)])
@pytest.mark.parametrize("flags", [0])
def test_rows_of_the_state(galv, S, rows, cols, flags):
    M = 700
    kw = dict(ragged=True, mem_lo=0, mem_hi=M // 5, time_hi=4000)
    w = classed(300 + S + rows, 6, 7, S, M, rows, cols, **kw) if rows else inputs.random_tables(300 + S, 6, 7, S, M, **kw)
    w.mem_q[1, 2, : S // 2] = M + 3                              # rows that never fit
    w.time_q[2, 1, :] = 9                                        # ties: the lowest strategy must win
    w.time_q[4, :, :] = 3
    w.mem_q[3, 0, :] = M // 2                                    # the lower half of every later column is +inf
    w.L[5] = 1
    against_reference(galv, w, flags)


# columns: less than a group, one more than a group, a step of tiles and one more, several steps; largest shifts from none to the budget
@pytest.mark.parametrize("M,mem_hi", [(0, 0), (5, 2), (31, 9), (32, 32), (607, 40), (608, 700), (2880, 300), (3040, 3040), (8191, 700)])
@pytest.mark.parametrize("S,K", [(24, 4), (12, 0), (20, 0)])
def test_columns_and_shifts(galv, M, mem_hi, S, K):
    kw = dict(ragged=True, mem_lo=0, mem_hi=mem_hi, time_hi=10 ** 6)
    for B in (1, 3):
        w = classed(M + 40, B, 5, S, M, K, K, **kw) if K else inputs.random_tables(M + 41, B, 5, S, M, **kw)
        w.mem_q[0, min(1, w.Lmax - 1), 0] = M
        for flags in (0,):
            against_reference(galv, w, flags)


# largest transition entry: differences of 16 and of 32 bits, packed relaxations or not, keys of the argmin
@pytest.mark.parametrize("top", [0, 1, 32767, 32768, 65535, 65536, (1 << 23) - 1, 1 << 23])
@pytest.mark.parametrize("S,K", [(24, 6), (16, 0), (40, 0), (64, 0)])
def test_largest_transition_entry(galv, top, S, K):
    for time_hi in (50, 60_000_000):
        w = inputs.random_tables(S + top % 97, 4, 6, S, 900, ragged=True, mem_lo=0, mem_hi=150, time_hi=time_hi, trans_hi=top)
        if K:
            rng = np.random.default_rng(S)
            for i in range(w.B):
                w.trans_q[i] = rng.integers(0, top + 1, (K, K), np.int32)[rng.integers(0, K, S)][:, rng.integers(0, K, S)]
        w.trans_q[:, 0, S - 1] = top
        for flags in (0,):
            against_reference(galv, w, flags)


@pytest.mark.parametrize("block", range(6))
def test_against_reference_kernel_on_many_shapes(galv, block):
    rng = np.random.default_rng(7700 + block)
    for case in range(14):
        S = int(rng.choice([1, 3, 8, 13, 16, 17, 24, 32, 40, 64, 100, 128]))
        Lmax, M, B = int(rng.integers(1, 14)), int(rng.integers(0, 4000)), int(rng.choice([1, 2, 5, 16, 40, 130, 200]))
        kw = dict(ragged=bool(rng.integers(0, 2)), mem_lo=0, mem_hi=int(rng.choice([0, 5, M // 30 + 1, M // 4 + 1, M + 50, 3 * M + 1])),
                  time_hi=int(rng.choice([5, 10 ** 4, 10 ** 6])))
        K = int(rng.choice([0, 1, 4, 8, 16]))
        w = classed(91000 + 100 * block + case, B, Lmax, S, M, K, max(1, K - 1), **kw) if K else \
            inputs.random_tables(91000 + 100 * block + case, B, Lmax, S, M, trans_hi=int(rng.choice([0, 9, 40000, 200000])), **kw)
        if Lmax > 2 and rng.integers(0, 2):
            w.time_q[:, 2] = w.time_q[:, 1]; w.mem_q[:, 2] = w.mem_q[:, 1]         # layers with the same rows share their records
        if rng.integers(0, 4) == 0 and B * Lmax * S * S < 4_000_000:
            w.trans_q = np.ascontiguousarray(rng.integers(0, 3000, (B, Lmax, S, S), np.int32))
        against_reference(galv, w, 0)


@pytest.mark.parametrize("S,K,top", [(64, 7, 2000), (24, 4, 50000), (40, 0, 900), (30, 0, 60000), (12, 0, 90000), (48, 8, 300000), (2, 0, 9), (1, 0, 9)])
def test_host_plans_from_states(galv, S, K, top):
    """The host entry point, whose table nobody sees: states of 16- and 32-bit differences, odd numbers of rows, +inf regions."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import HostSearch, SearchBuffers
    for M, B in ((1100, 5), (95, 3)):
        w = inputs.random_tables(17 + S, B, 20, S, M, ragged=True, mem_lo=0, mem_hi=max(1, M // 12), trans_hi=top, time_hi=4 * top)
        if K:
            rng = np.random.default_rng(S)
            for i in range(B):
                w.trans_q[i] = rng.integers(0, top + 1, (K, K), np.int32)[rng.integers(0, K, S)][:, rng.integers(0, K, S)]
        w.mem_q[1, 3, : S // 2] = M + 3
        w.mem_q[2, 0, :] = M // 2
        w.time_q[0, ::2] = 5                                     # ties: the lowest strategy must win
        ref = SearchBuffers(galv, w, gb.STORE_C_FULL | gb.KERNEL_REFERENCE)
        ref.dp_search(); ref.backtrack()
        want = ref.results()
        hs = HostSearch(galv, w, gb.STORE_C_FULL | gb.KERNEL_SOLO)
        for _ in range(2):
            res = hs.run()
            for k in ("status", "opt_cost", "plan", "mem_used"):
                assert (res[k] == want[k]).all(), (k, M)


@pytest.mark.parametrize("S,M", [(11, 8191), (12, 8191), (13, 7400), (14, 7400), (15, 6500), (16, 6500), (16, 8191)])
def test_what_lies_behind_the_matrices(galv, S, M):
    """Too many columns for an unstructured state of 32-bit rows, fewer rows than a look at the first 17 would read: what follows
    the last matrix is not looked at, and whatever it holds the results are the same."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    B = 160                                                      # more instances than SMs
    for cols in (S, 4):                                          # no two rows alike; with few kinds of columns the state fits all the same
        w = inputs.random_tables(500 + S, B, 3, S, M, ragged=True, mem_lo=0, mem_hi=M // 3, trans_hi=900)
        if cols < S:
            w.trans_q[:] = np.ascontiguousarray(w.trans_q[:, :, np.random.default_rng(S).integers(0, cols, S)])
        ref = SearchBuffers(galv, w, gb.STORE_C_FULL | gb.KERNEL_REFERENCE)
        ref.dp_search(); ref.backtrack()
        ref.C = None
        for flags in (0, gb.KERNEL_SOLO):
            for behind in ("rows of it", "others"):
                one = SearchBuffers(galv, w, flags)
                n = one.trans_q.numel()
                room = torch.full((n + 17 * S,), 7, dtype=torch.int32, device=one.dev)
                room[:n] = one.trans_q.flatten()
                room[n:] = one.trans_q[-1, 0].repeat(17) if behind == "rows of it" else torch.arange(-17 * S, 0, dtype=torch.int32, device=one.dev)
                one.trans_q = room[:n].view(B, S, S)
                one.dp_search(); one.backtrack()
                torch.cuda.synchronize()
                assert torch.equal(one.status, ref.status) and torch.equal(one.opt_cost, ref.opt_cost) and torch.equal(one.C_last, ref.C_last), (flags, behind)
                assert not flags or cols == S or galv.galv_dp_search_path(one.shape, one.workspace) == gb.PATH_SOLO


def milliseconds(sb):
    import torch
    sb.dp_search()
    best = 1e9
    for _ in range(5):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        sb.dp_search()
        t1.record()
        torch.cuda.synchronize()
        best = min(best, t0.elapsed_time(t1))
    return best


# (instances, layers, strategies, budget, classes or 0, largest transition entry over the median time, by the kernel that suits it)
@pytest.mark.parametrize("B,Lmax,S,M,K,share,kernel", [(6, 40, 64, 4000, 8, 2.0, "KERNEL_RESIDENT"), (40, 48, 64, 4000, 7, 1.0, "KERNEL_RESIDENT"),
                                                       (200, 40, 64, 4000, 4, 2.0, "KERNEL_RESIDENT"), (6, 48, 48, 1500, 0, 0.03, "KERNEL_CLUSTER"),
                                                       (200, 24, 16, 2880, 0, 1.0, "KERNEL_NO_CLUSTER")])
def test_batches_that_nothing_can_be_ruled_out_in(galv, B, Lmax, S, M, K, share, kernel):
    """Without a flag a batch that most strategies matter in goes where all of them are relaxed fast: on the solo kernel these
    take 2.2 to 5 times as long.  Twice as long as the kernel that suits them leaves room for the look and for the clock."""
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    rng = np.random.default_rng(S + B)
    w = inputs.random_tables(800 + B, B, Lmax, S, M, mem_lo=M // (6 * Lmax), mem_hi=3 * M // Lmax)
    w.time_q[:] = np.sort(np.rint(5e5 * np.exp(0.5 * rng.standard_normal(w.time_q.shape))).astype(np.int32), axis=2)
    w.mem_q[:] = -np.sort(-w.mem_q, axis=2)                      # less memory costs time
    top = int(5e5 * share) + 1
    w.trans_q[:] = rng.integers(0, top, w.trans_q.shape, np.int32)
    if K:
        for i in range(B):
            w.trans_q[i] = rng.integers(0, top, (K, K), np.int32)[rng.integers(0, K, S)][:, rng.integers(0, K, S)]
    plain, suited = SearchBuffers(galv, w, 0), SearchBuffers(galv, w, getattr(gb, kernel))
    assert milliseconds(plain) < 2 * milliseconds(suited)
    plain.backtrack(); suited.backtrack()
    import torch
    assert torch.equal(plain.status, suited.status) and torch.equal(plain.opt_cost, suited.opt_cost) and torch.equal(plain.C_last, suited.C_last)


def path_of(galv, w, flags):
    import torch
    from paper_2504_03662_b200.search import SearchBuffers
    sb = SearchBuffers(galv, w, flags)
    sb.dp_search()
    torch.cuda.synchronize()
    return galv.galv_dp_search_path(sb.shape, sb.workspace)


def test_path_word(galv):
    """What galv_dp_search_path says is what ran: the solo kernel alone (structured and unstructured matrices, also more instances
    than SMs), or who took the instances it has no room for, or the batches it is not worth its while for."""
    from paper_2504_03662_b200 import binding as gb
    kw = dict(mem_lo=0, mem_hi=90)
    for B in (5, 160):
        for S in (24, 30):
            for w in (inputs.random_tables(50 + S, B, 6, S, 900, trans_hi=900, **kw), inputs.random_tables(50 + S, B, 6, S, 900, trans_hi=90000, **kw),
                      classed(50 + S, B, 6, S, 900, 4, 5, **kw)):
                assert path_of(galv, w, gb.KERNEL_SOLO) == gb.PATH_SOLO, (B, S)
    w = classed(60, 5, 6, 100, 900, 4, 5, **kw)
    assert path_of(galv, w, gb.KERNEL_SOLO) == gb.PATH_SOLO
    w.trans_q[2] = np.random.default_rng(1).integers(0, 3000, (100, 100), np.int32)      # no room for 100 rows
    assert path_of(galv, w, gb.KERNEL_SOLO) == gb.PATH_CLUSTER
    big = classed(61, 160, 4, 64, 2500, 4, 5, **kw)
    assert path_of(galv, big, gb.KERNEL_SOLO) == gb.PATH_SOLO
    for top, want in ((3000, gb.PATH_TILED_PACKED), (40000, gb.PATH_TILED_32)):          # ... nor for 64 of 2500 columns
        big.trans_q[7] = np.random.default_rng(1).integers(0, top + 1, (64, 64), np.int32)
        big.trans_q[7, 0, 1] = top
        assert path_of(galv, big, gb.KERNEL_SOLO) == want
    # without a flag: times far apart, and times that lie close together
    for S, K in ((24, 0), (64, 7)):
        w = classed(63, 300, 30, S, 3000, K, K, mem_lo=16, mem_hi=300) if K else inputs.random_tables(63, 300, 30, S, 3000, mem_lo=16, mem_hi=300, trans_hi=2000)
        w.time_q[:] = np.rint(5e5 * np.exp(0.5 * np.random.default_rng(S).standard_normal(w.time_q.shape))).astype(np.int32)
        assert path_of(galv, w, 0) == gb.PATH_SOLO
        w.time_q[:] = 500000 + w.time_q // 1000
        assert path_of(galv, w, 0) == (gb.PATH_CLUSTER if K else gb.PATH_TILED_PACKED)
    # with another kernel asked for, or a table to write, the word is that kernel's
    w = classed(62, 5, 40, 24, 900, 4, 5, **kw)
    assert path_of(galv, w, gb.KERNEL_RESIDENT) == gb.PATH_CLUSTER and path_of(galv, w, gb.KERNEL_CLUSTER) == gb.PATH_CLUSTER
    assert path_of(galv, w, gb.KERNEL_NO_CLUSTER) == gb.PATH_TILED_PACKED and path_of(galv, w, gb.STORE_C_FULL | gb.KERNEL_SOLO) == gb.PATH_CLUSTER
