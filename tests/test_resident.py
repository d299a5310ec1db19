"""The kernel that keeps the state between layers in shared memory: matrices with classes of equal rows and columns.

Tables, optima and plans against the CPU oracle, exact: everything is integers.  RES asks for this kernel at any size, and
without the pushing cluster kernel behind it: the path is then 2 only if this kernel took every instance (with an argmin
table it is 0 whichever kernel ran).
"""
import numpy as np
import pytest

from paper_2504_03662_b200 import inputs
from tests.test_gpu_parity import check_batch, galv, oracle_search_many  # noqa: F401  (galv is a fixture)

pytestmark = pytest.mark.gpu

RES = 1 << 21                 # GALV_KERNEL_RESIDENT


def check_resident(orc, galv, w, flags, **kw):
    sb, res = check_batch(orc, galv, w, flags | RES, **kw)
    assert galv.galv_dp_search_path(sb.shape, sb.workspace) == (0 if flags & 2 else 2)
    return sb, res


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
    check_resident(orc, galv, w, flags)


# columns per CTA against shifts: inside the CTA, into the halo, beyond it (read from the owner), from the last column
@pytest.mark.parametrize("n,M,mem_hi", [(1, 500, 90), (2, 1000, 40), (3, 1000, 990), (5, 2880, 700), (8, 2879, 2879), (16, 2880, 1500)])
@pytest.mark.parametrize("S,classes", [(24, 4), (24, 0)])
def test_shifts_across_the_cluster(orc, galv, n, M, mem_hi, S, classes):
    from paper_2504_03662_b200 import binding as gb
    kw = dict(ragged=True, mem_lo=0, mem_hi=mem_hi)
    w = classed(40 + n, 3, 5, S, M, classes, classes, **kw) if classes else inputs.random_tables(40 + n, 3, 5, S, M, **kw)
    w.mem_q[0, 1, 0] = M
    for flags in (gb.STORE_C_FULL, 0, gb.STORE_ARGMIN):
        check_resident(orc, galv, w, flags | gb.CLUSTER_SIZE(n))


@pytest.mark.parametrize("S,M,path", [(40, 1100, 2),            # the pushing cluster kernel takes the rest
                                      (64, 8200, 1)])           # ... has no room: the tiled kernels (packed loop) do
def test_some_instances_left_to_the_other_kernels(orc, galv, S, M, path):
    """One batch with structured, unstructured and flagged matrices, too many strategies for an unstructured state."""
    w = classed(7, 7, 18, S, M, 6, 6, mem_lo=0, mem_hi=M // 10, ragged=True)
    rng = np.random.default_rng(1)
    for i in (1, 4):
        w.trans_q[i] = rng.integers(0, 3000, (S, S), np.int32)
    w.trans_q[3, 2, 2] = -1
    w.L[5] = 0
    w.L[[0, 1]] = 18                                             # both kinds at full length
    for flags in (1, 0, 3):
        sb, res = check_batch(orc, galv, w, flags, idx=[0, 1, 2, 4, 6])
        assert res["status"][[3, 5]].tolist() == [2, 2]
        if not flags & 2:
            assert galv.galv_dp_search_path(sb.shape, sb.workspace) == path


@pytest.mark.parametrize("B,S,rows", [(1, 24, 4), (40, 48, 8), (3, 64, 64), (5, 7, 7)])
def test_host_plans_from_states(orc, galv, B, S, rows):
    """The host entry point keeps the states between the layers where a table would be kept: same optima and plans."""
    from paper_2504_03662_b200.search import HostSearch
    w = classed(60 + B, B, 8, S, 900, rows, rows, mem_lo=0, mem_hi=200, ragged=True)
    check_resident(orc, galv, w, 0, idx=[0])                     # without a table, as the host entry point runs it: all by this kernel
    hs = HostSearch(galv, w, 1 | RES)
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


@pytest.mark.parametrize("block", range(6))
def test_against_reference_kernel_on_many_shapes(galv, block):
    """Random shapes, cluster sizes, classes (or none), memory distributions and per-layer matrices against the
    one-thread-per-cell kernel, which other tests tie to the oracle.  Two runs per shape on the same buffers."""
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    rng = np.random.default_rng(5200 + block)
    ran = 0
    for case in range(12):
        S = int(rng.choice([1, 3, 8, 13, 16, 17, 24, 32, 40, 64, 100, 128]))
        Lmax, M, B = int(rng.integers(1, 14)), int(rng.integers(31, 4000)), int(rng.choice([1, 2, 5, 16, 40, 130]))
        kw = dict(ragged=bool(rng.integers(0, 2)), mem_lo=0, mem_hi=int(rng.choice([0, 5, M // 30 + 1, M // 4 + 1, M + 50, 3 * M])),
                  time_hi=int(rng.choice([5, 10 ** 4, 10 ** 6])))
        K = int(rng.choice([0, 1, 4, 8, 16]))
        w = classed(71000 + 100 * block + case, B, Lmax, S, M, K, max(1, K - 1), **kw) if K else \
            inputs.random_tables(71000 + 100 * block + case, B, Lmax, S, M, trans_hi=int(rng.choice([0, 9, 40000])), **kw)
        if Lmax > 2 and rng.integers(0, 2):
            w.mem_q[:, int(rng.integers(1, Lmax)), :] += M // 2                          # one heavy layer
        per_layer = case % 4 == 3 and Lmax > 1
        if per_layer:
            w.trans_q = np.ascontiguousarray(np.repeat(w.trans_q[:, None], Lmax, 1))
            w.trans_q[:, 1:] += rng.integers(0, 50, size=(B, Lmax - 1, S, S), dtype=np.int32)
        size = int(rng.choice([0, 0, 1, 2, 3, 4, 6, 8, 11, 16]))
        table = (gb.STORE_C_FULL, gb.STORE_C_FULL | gb.STORE_ARGMIN, 0, gb.STORE_C_FULL)[case % 4 if not per_layer else 0]
        ref = SearchBuffers(galv, w, gb.STORE_C_FULL | gb.KERNEL_REFERENCE)
        ref.dp_search(); ref.backtrack()
        one = SearchBuffers(galv, w, table | RES | gb.CLUSTER_SIZE(size))
        for _ in range(2):
            one.C_last.fill_(-7)
            if table:
                one.C.fill_(-7)
            one.dp_search(); one.backtrack()
            torch.cuda.synchronize()
            ran += not table & 2 and galv.galv_dp_search_path(one.shape, one.workspace) == 2
            st = ref.status.cpu().numpy()
            assert (one.status.cpu().numpy() == st).all() and torch.equal(one.opt_cost, ref.opt_cost), (block, case)
            assert not table or torch.equal(one.plan, ref.plan), (block, case)
            for i in np.flatnonzero((st & ~1) == 0) if table else ():
                Li = int(w.L[i])
                assert torch.equal(one.C[i, :Li], ref.C[i, :Li]), (block, case, int(i), S, Lmax, M, B, size)
            ok = torch.from_numpy((st & ~1) == 0).to(one.C_last.device)
            assert torch.equal(one.C_last[ok], ref.C_last[ok]), (block, case)
        del ref, one
        torch.cuda.empty_cache()
    assert ran >= 10                                             # most of the shapes without an argmin table were searched by this kernel alone


# a halo within the neighbours' columns; shifts beyond the halo (every layer then ends with the full barrier); argmin states
@pytest.mark.parametrize("S,M,n,mem_hi,flags", [(24, 1000, 4, 60, 1), (24, 1000, 4, 60, 2), (64, 2880, 16, 1500, 1), (24, 1000, 5, 700, 0)])
def test_a_halo_that_never_comes(orc, galv, S, M, n, mem_hi, flags):
    """The wait for a halo gives up: the kernel returns, the status says TIMEOUT, the plan step walks nothing, the context
    keeps working."""
    import time
    import torch
    from paper_2504_03662_b200 import binding as gb
    from paper_2504_03662_b200.search import SearchBuffers
    w = inputs.random_tables(3, 3, 6, S, M, mem_lo=1, mem_hi=mem_hi)
    flags |= RES | gb.CLUSTER_SIZE(n)
    bad = SearchBuffers(galv, w, flags | gb.DEBUG_WITHHOLD_LOAD)
    t0 = time.time()
    bad.dp_search()
    torch.cuda.synchronize()
    assert time.time() - t0 < 60
    assert (bad.status.cpu().numpy() == gb.STATUS_TIMEOUT).all()
    bad.backtrack()
    r = bad.results()
    assert (r["status"] & gb.STATUS_TIMEOUT).all() and (r["opt_cost"] == 2 ** 30 - 1).all() and (r["plan"] == -1).all()
    check_resident(orc, galv, w, flags)


# S <= 16: classes whatever the matrix holds; 24, 40: unstructured ones are told by their first rows; 130 columns a CTA with
# shifts over many CTAs and beyond the halo
@pytest.mark.parametrize("S,M,mem_hi", [(12, 1100, 90), (16, 1100, 90), (24, 1500, 1500), (40, 1500, 700), (48, 1500, 1500)])
def test_two_cluster_kernels_beside_one_another(orc, galv, S, M, mem_hi):
    """Small batches: the pushing kernel starts beside the resident one, searches what that one leaves to it (no equal rows,
    many classes, long halos) and nothing else.  The same buffers again and again without a pause, the matrices changing."""
    import torch
    from paper_2504_03662_b200.search import SearchBuffers
    w = classed(300 + S, 5, 18, S, M, 4, 4, ragged=True, mem_lo=0, mem_hi=mem_hi)
    other = classed(301 + S, 5, 18, S, M, 4, 4, ragged=True, mem_lo=0, mem_hi=60)
    rng = np.random.default_rng(S)
    w.trans_q[1] = rng.integers(0, 3000, (S, S), np.int32)
    w.trans_q[2] = rng.integers(0, 2000, (12, 12), np.int32)[np.arange(S) % 12][:, np.arange(S) % 12]
    w.mem_q[3] //= 20                                            # short shifts
    w.time_q[4, 0, 0] = -1
    other.trans_q[[0, 3]] = rng.integers(0, 3000, (2, S, S), np.int32)
    for flags in (1, 0):
        sets = []
        for x in (w, other):
            sb, res = check_batch(orc, galv, x, flags, idx=[0, 1, 2, 3])
            assert galv.galv_dp_search_path(sb.shape, sb.workspace) == 2
            sets.append((sb, {k: getattr(sb, k).clone() for k in ("opt_cost", "plan", "status", "C_last")}))
        assert sets[0][1]["status"][4] == 2
        one = SearchBuffers(galv, w, flags)
        got = []
        for _ in range(10):
            for sb, _r in sets:
                for k in ("time_q", "mem_q", "trans_q", "L"):
                    getattr(one, k).copy_(getattr(sb, k))
                one.dp_search(); one.backtrack()
                got.append({k: getattr(one, k).clone() for k in ("opt_cost", "plan", "status", "C_last")})
        torch.cuda.synchronize()
        for n, g in enumerate(got):
            ref = sets[n % 2][1]
            ok = ref["status"] & ~1 == 0
            for k in ("opt_cost", "plan", "status"):
                assert torch.equal(g[k], ref[k]), (n, k)
            assert torch.equal(g["C_last"][ok], ref["C_last"][ok]), n


def test_both_cluster_kernels_in_a_graph(galv):
    """The launch that may start early is captured as such: replays with changing matrices equal plain calls."""
    import torch
    from paper_2504_03662_b200.search import SearchBuffers
    w = classed(77, 3, 18, 40, 1500, 4, 4, mem_lo=0, mem_hi=200)
    plain, one = SearchBuffers(galv, w, 1), SearchBuffers(galv, w, 1)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        one.dp_search(); one.backtrack()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            one.dp_search(); one.backtrack()
    rng = np.random.default_rng(3)
    for k in range(6):
        x = w.trans_q if k % 2 else rng.integers(0, 3000, w.trans_q.shape, np.int32)
        for sb in (plain, one):
            sb.trans_q.copy_(torch.from_numpy(np.ascontiguousarray(x)))
        torch.cuda.synchronize()
        plain.dp_search(); plain.backtrack()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(plain.C, one.C) and torch.equal(plain.plan, one.plan) and torch.equal(plain.opt_cost, one.opt_cost), k
    del g
