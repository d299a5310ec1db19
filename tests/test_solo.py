"""The kernel that keeps an instance's state on one SM: the last layer's table and the optimum against the one-thread-per-cell
kernel, which other tests tie to the CPU oracle.  Whole numbers: exact.  It writes no table and walks no plan; the host entry
point's plans come from its states.
"""
import numpy as np
import pytest

from paper_2504_03662_b200 import inputs
from tests.test_gpu_parity import galv  # noqa: F401  (a fixture)
from tests.test_resident import classed

pytestmark = pytest.mark.gpu


def reference(galv, w):
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    ref = SearchBuffers(galv, w, gb.KERNEL_REFERENCE)
    ref.dp_search(); ref.backtrack()
    return ref


def same(one, ref, what=""):
    import torch
    torch.cuda.synchronize()
    assert torch.equal(one.status, ref.status) and torch.equal(one.opt_cost, ref.opt_cost), what
    ok = (ref.status & ~1) == 0                                  # tables of flagged instances are left untouched
    assert torch.equal(one.C_last[ok], ref.C_last[ok]), what
    assert bool((one.C_last[~ok] == 77).all()), what


def against_reference(galv, w, path=True):
    """On the solo kernel.  path: it must take every instance; else whether it did is returned."""
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    ref = reference(galv, w)
    one = SearchBuffers(galv, w, gb.KERNEL_SOLO)
    for _ in range(2):
        one.C_last.fill_(77)
        one.dp_search(); one.backtrack()
        same(one, ref)
    ran = galv.galv_dp_search_path(one.shape, one.workspace) == gb.PATH_SOLO
    assert ran or not path
    return ran


# S and classes at the edges of the accumulator widths (8 / 16 / 32 / 64 rows) and of a warp's lanes, odd numbers of packed rows
@pytest.mark.parametrize("S,rows,cols", [(1, 1, 1), (5, 1, 1), (7, 0, 0), (8, 0, 0), (9, 0, 0), (16, 0, 0), (17, 0, 0), (24, 4, 4), (24, 5, 9), (30, 0, 0), (31, 0, 0),
                                         (32, 0, 0), (33, 8, 7), (33, 0, 0), (44, 0, 0), (64, 9, 16), (64, 16, 9), (64, 0, 0), (65, 3, 3), (128, 8, 8)])
def test_rows_of_the_state(galv, S, rows, cols):
    M = 700
    kw = dict(ragged=True, mem_lo=0, mem_hi=M // 5, time_hi=4000)
    w = classed(300 + S + rows, 6, 7, S, M, rows, cols, **kw) if rows else inputs.random_tables(300 + S, 6, 7, S, M, **kw)
    w.mem_q[1, 2, : S // 2] = M + 3                              # rows that never fit
    w.time_q[2, 1, :] = 9                                        # ties
    w.time_q[4, :, :] = 3
    w.mem_q[3, 0, :] = M // 2                                    # the lower half of every later column is +inf
    w.L[5] = 1
    against_reference(galv, w)


# columns: less than a group, one more than a group, a step of tiles and one more, several steps; largest shifts from none to the budget
@pytest.mark.parametrize("M,mem_hi", [(0, 0), (5, 2), (31, 9), (32, 32), (607, 40), (608, 700), (2880, 300), (3040, 3040), (8191, 700)])
@pytest.mark.parametrize("S,K", [(24, 4), (12, 0), (20, 0)])
def test_columns_and_shifts(galv, M, mem_hi, S, K):
    kw = dict(ragged=True, mem_lo=0, mem_hi=mem_hi, time_hi=10 ** 6)
    for B in (1, 3):
        w = classed(M + 40, B, 5, S, M, K, K, **kw) if K else inputs.random_tables(M + 41, B, 5, S, M, **kw)
        w.mem_q[0, min(1, w.Lmax - 1), 0] = M
        against_reference(galv, w, path=bool(K) or M <= 2880)    # a budget's worth of guard columns, or 8192 columns, beside 12 rows: no room


# largest transition entry: differences of 16 and of 32 bits, packed relaxations or not
@pytest.mark.parametrize("top", [0, 1, 32767, 32768, 65535, 65536, (1 << 23) - 1, 1 << 23])
@pytest.mark.parametrize("S,K", [(24, 6), (16, 0), (40, 0), (30, 0), (64, 0)])
def test_largest_transition_entry(galv, top, S, K):
    for time_hi in (50, 60_000_000):
        w = inputs.random_tables(S + top % 97, 4, 6, S, 900, ragged=True, mem_lo=0, mem_hi=150, time_hi=time_hi, trans_hi=top)
        if K:
            rng = np.random.default_rng(S)
            for i in range(w.B):
                w.trans_q[i] = rng.integers(0, top + 1, (K, K), np.int32)[rng.integers(0, K, S)][:, rng.integers(0, K, S)]
        w.trans_q[:, 0, S - 1] = top
        against_reference(galv, w, path=S < 64 or top <= 65535)  # 64 rows of 32-bit differences: no room


@pytest.mark.parametrize("block", range(6))
def test_against_reference_kernel_on_many_shapes(galv, block):
    rng = np.random.default_rng(7700 + block)
    ran = 0
    for case in range(14):
        S = int(rng.choice([1, 3, 8, 13, 16, 17, 24, 32, 40, 64, 100, 128]))
        Lmax, M, B = int(rng.choice([1, 2, 5, 9, 13, 40])), int(rng.integers(0, 4000)), int(rng.choice([1, 2, 5, 16, 40, 130, 200]))
        kw = dict(ragged=bool(rng.integers(0, 2)), mem_lo=0, mem_hi=int(rng.choice([0, 5, M // 30 + 1, M // 4 + 1, M + 50, 3 * M + 1])),
                  time_hi=int(rng.choice([5, 10 ** 4, 10 ** 6])))
        K = int(rng.choice([0, 1, 4, 8, 16]))
        w = classed(91000 + 100 * block + case, B, Lmax, S, M, K, max(1, K - 1), **kw) if K else \
            inputs.random_tables(91000 + 100 * block + case, B, Lmax, S, M, trans_hi=int(rng.choice([0, 9, 40000, 200000])), **kw)
        if Lmax > 2 and rng.integers(0, 2):
            w.time_q[:, 2] = w.time_q[:, 1]; w.mem_q[:, 2] = w.mem_q[:, 1]         # layers with the same rows share their records
        if rng.integers(0, 4) == 0 and B * Lmax * S * S < 4_000_000:
            w.trans_q = np.ascontiguousarray(rng.integers(0, 3000, (B, Lmax, S, S), np.int32))
        ran += against_reference(galv, w, path=False)
    assert ran >= 7                                              # most of the shapes were searched by this kernel alone


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


@pytest.mark.parametrize("S,M,B,Lmax,path", [(40, 1500, 9, 20, "PATH_SOLO"),        # everything fits
                                             (100, 1100, 9, 20, "PATH_CLUSTER"),   # unstructured ones do not: the pushing kernel beside the resident one
                                             (32, 3600, 12, 20, "PATH_CLUSTER"),   # ... the resident one, which has room for them
                                             (64, 2500, 160, 6, "PATH_TILED_PACKED"), (72, 2500, 160, 6, "PATH_TILED_32")])    # ... the tiled ones
def test_one_batch_for_several_kernels(galv, S, M, B, Lmax, path):
    """Structured, unstructured and flagged instances in one batch; the solo kernel takes what fits, the kernels behind the rest
    and nothing else.  The same buffers again and again without a pause, the matrices changing places."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    rng = np.random.default_rng(S)
    sets = []
    for k in range(2):
        w = classed(40 + S + k, B, Lmax, S, M, 5, 6, ragged=True, mem_lo=0, mem_hi=M // 20)
        for i in range(k, B, 3):
            w.trans_q[i] = rng.integers(0, 3000, (S, S), np.int32)
        w.time_q[2, 0, 0] = -1
        w.L[4], w.L[5] = 0, Lmax + 1
        w.L[0] = w.L[1] = w.L[7] = Lmax
        ref = reference(galv, w)
        assert ref.status.cpu().numpy()[[2, 4, 5]].tolist() == [2, 2, 2]
        sets.append((w, ref))
    one = SearchBuffers(galv, sets[0][0], gb.KERNEL_SOLO)
    got = []
    for n in range(8):
        w, ref = sets[n % 2]
        for name in ("time_q", "mem_q", "trans_q", "L"):
            getattr(one, name).copy_(getattr(ref, name))
        one.C_last.fill_(77)
        one.dp_search(); one.backtrack()
        got.append([t.clone() for t in (one.status, one.opt_cost, one.C_last)])
    torch.cuda.synchronize()
    assert galv.galv_dp_search_path(one.shape, one.workspace) == getattr(gb, path)
    for n, (status, opt, last) in enumerate(got):
        one.status, one.opt_cost, one.C_last = status, opt, last
        same(one, sets[n % 2][1], n)


def spread(w, seed, near=False):
    """Measured layer times: half a millisecond, half of it a standard deviation, or all of them within a thousandth."""
    w.time_q[:] = np.rint(5e5 * np.exp(0.5 * np.random.default_rng(seed).standard_normal(w.time_q.shape))).astype(np.int32)
    if near:
        w.time_q[:] = 500000 + w.time_q // 1000
    return w


@pytest.mark.parametrize("S,K,B,Lmax,M", [(24, 0, 300, 30, 3000), (64, 7, 160, 40, 4000), (64, 5, 600, 24, 2880), (12, 0, 200, 40, 3000)])
def test_unasked(galv, S, K, B, Lmax, M):
    """Without a flag, more instances than SMs (600: more than are sorted by length), stacks of 24 to 40 layers: batches whose times
    are far apart are taken, batches whose times lie close together are not, flagged instances or not; the results are the same."""
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    for near in (False, True):
        kw = dict(ragged=B == 600, mem_lo=M // (6 * Lmax), mem_hi=3 * M // Lmax)
        w = spread(classed(S, B, Lmax, S, M, K, K, **kw) if K else inputs.random_tables(S, B, Lmax, S, M, trans_hi=2000, **kw), S, near)
        w.mem_q[1, 2, :] = M + 1                                 # nothing fits
        w.L[0], w.L[B - 1] = 0, Lmax + 1
        w.time_q[B // 2, 0, 0] = -1
        one = SearchBuffers(galv, w, 0)
        one.C_last.fill_(77)
        one.dp_search(); one.backtrack()
        same(one, reference(galv, w), near)
        assert (galv.galv_dp_search_path(one.shape, one.workspace) == gb.PATH_SOLO) == (not near), near


def test_host_plans_unasked(galv):
    """The host entry point without a flag, where it takes the solo kernel's states, and where it does not."""
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import HostSearch, SearchBuffers
    for B, Lmax, near in ((130, 60, False), (130, 60, True), (200, 14, False)):
        w = spread(classed(B, B, Lmax, 32, 8000, 6, 7, ragged=True, mem_lo=8000 // (6 * Lmax), mem_hi=24000 // Lmax), B, near)
        w.L[3] = 0
        ref = SearchBuffers(galv, w, gb.STORE_ARGMIN | gb.KERNEL_NO_CLUSTER)
        ref.dp_search(); ref.backtrack()
        want = ref.results()
        del ref
        hs = HostSearch(galv, w, gb.STORE_C_FULL)
        res = hs.run()
        for k in ("status", "opt_cost", "plan", "mem_used"):
            assert (res[k] == want[k]).all(), (k, B, near)


@pytest.mark.parametrize("flags", ["KERNEL_SOLO", None])
def test_in_a_graph(galv, flags):
    """Captured with what stands behind it: replays with changing matrices and times equal plain calls, whoever takes them."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    f = getattr(gb, flags) if flags else 0
    w = spread(classed(77, 200, 24, 40, 2000, 4, 4, mem_lo=14, mem_hi=250), 3)
    plain, one = SearchBuffers(galv, w, f), SearchBuffers(galv, w, f)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        one.dp_search(); one.backtrack()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            one.dp_search(); one.backtrack()
    rng = np.random.default_rng(3)
    near, far = (torch.from_numpy(spread(w, 3, n).time_q.copy()) for n in (True, False))
    paths = set()
    for k in range(6):
        x = torch.from_numpy(np.ascontiguousarray(w.trans_q if k % 2 else rng.integers(0, 3000, w.trans_q.shape, np.int32)))
        for sb in (plain, one):
            sb.trans_q.copy_(x)
            sb.time_q.copy_(near if k // 2 == 1 else far)
        torch.cuda.synchronize()
        plain.dp_search(); plain.backtrack()
        g.replay()
        torch.cuda.synchronize()
        path = galv.galv_dp_search_path(one.shape, one.workspace)
        assert path == galv.galv_dp_search_path(plain.shape, plain.workspace)
        paths.add(path)
        assert torch.equal(plain.C_last, one.C_last) and torch.equal(plain.opt_cost, one.opt_cost) and torch.equal(plain.status, one.status), k
    assert gb.PATH_SOLO in paths and len(paths) > 1 - bool(flags)
    del g


def test_in_the_library_s_own_scratch(galv):
    """galv_dp_search_static: no table, so the scratch has to hold two layers whichever kernel runs; flagged instances among them."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    for seed in (1, 2):
        w = classed(seed, 7, 12, 9, 900, 4, 4, ragged=True, mem_lo=0, mem_hi=80)
        w.time_q[seed, 0, 0] = -3
        one = SearchBuffers(galv, w, gb.KERNEL_SOLO)
        one.workspace = None
        one.C_last.fill_(77)
        galv.galv_dp_search_static(one.shape, one.L, one.time_q, one.mem_q, one.trans_q, one.C, one.A, one.C_last, one.status)
        one.backtrack()
        same(one, reference(galv, w), seed)
