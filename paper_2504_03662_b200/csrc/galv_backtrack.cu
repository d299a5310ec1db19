// Optimum extraction and plan backtrack: one warp per search instance.
//
// (Section 3 of the paper: the selector's result is a per-layer parallelism plan.)
// opt = min_s C_last[s][budget] with the lowest s on ties, found by a warp
// shuffle min over packed (cost << 32 | index) keys.  The walk then goes from
// the last layer to the first; the predecessor is read from the argmin table
// when there is one, otherwise it is the lowest s' whose candidate
// C[l-1][m'][s'] + trans(s',s) equals the cell's value minus time(l,s).

#include "galv_internal.h"

namespace {

constexpr int kInf = GALV_INF;

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w < v ? w : v;
    }
    return v;
}

// The walk from cell (Li - 1, s, m) of value cur down to layer 0: writes the plan, returns the memory it takes; *bad on
// tables that are not consistent.  NJ: strategies per lane (S <= 32 * NJ): the chain of selects, loads and ballots is as long
// as it has to be.  One dependent memory round trip per layer: the cell's value is carried along (it is the chosen candidate
// of the step before), and the mem / time rows of the next layer down are fetched, whole, while this layer's candidates are
// in flight; lane k%32 keeps entries k, k+32, ... (S <= 256).  mrow, trow: the rows of layer Li - 1 on entry.
template <int NJ, bool ARGMIN>
__device__ __forceinline__ long long walk_table(int Li, int S, int m_pitch, const int32_t* __restrict__ tq, const int32_t* __restrict__ mq,
                                                const int32_t* __restrict__ T0, long long trans_layer, const int32_t* __restrict__ C,
                                                const uint8_t* __restrict__ A, int (&mrow)[NJ], int (&trow)[NJ], int s, int m, int cur,
                                                int32_t* __restrict__ pl, bool* bad)
{
    const int lane = threadIdx.x;
    const size_t slice = (size_t)S * m_pitch;
    long long used = 0;
    for (int l = Li - 1; l >= 0; --l) {
        if (lane == 0) pl[l] = s;
        int msel = mrow[0], tsel = trow[0];
#pragma unroll
        for (int j = 1; j < NJ; ++j) {
            msel = (s >> 5) == j ? mrow[j] : msel;
            tsel = (s >> 5) == j ? trow[j] : tsel;
        }
        const int mm = __shfl_sync(0xffffffffu, msel, s & 31);
        const int tt = __shfl_sync(0xffffffffu, tsel, s & 31);
        used += mm;
        if (mm > m) { *bad = true; break; }                      // cannot happen on consistent tables: the cell would be +inf; never index below column 0
        if (l == 0) break;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {                          // rows of layer l-1, needed one step from now
            const int k = lane + 32 * j;
            mrow[j] = k < S ? mq[(l - 1) * S + k] : 0;
            trow[j] = k < S ? tq[(l - 1) * S + k] : 0;
        }
        int sp = 255;
        if (ARGMIN) {
            sp = A[(size_t)l * slice + (size_t)s * m_pitch + m];
        } else {
            const int target = cur - tt;
            const int32_t* prev = C + (size_t)(l - 1) * slice + (m - mm);
            const int32_t* T = T0 + (size_t)l * trans_layer;       // paid between layers l-1 and l
            // every row's candidate is asked for before the first is looked at: one round trip to memory, not one per 32 rows
            int cv[NJ], tv[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = lane + 32 * j;
                cv[j] = k < S ? prev[(size_t)k * m_pitch] : kInf;
                tv[j] = k < S ? T[k * S + s] : 0;
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                if (32 * j >= S) break;
                const unsigned b = __ballot_sync(0xffffffffu, cv[j] < kInf && cv[j] + tv[j] == target);
                if (b) {
                    const int src = __ffs(b) - 1;
                    sp = 32 * j + src;
                    cur = __shfl_sync(0xffffffffu, cv[j], src);
                    break;
                }
            }
        }
        if (sp >= S) { *bad = true; break; }                     // cannot happen on consistent tables; stop instead of walking off
        m -= mm;
        s = sp;
    }
    return used;
}

// The same on the resident kernel's states, [layer][rows][m_pitch], in place of the table: strategy k's value in layer l-1 is
// its time on top of its state row at the column its memory leaves, so rows are fetched two layers ahead.  (A walk of its own:
// the choice inside one loop stood between a candidate's load and its transition entry's, a round trip each, and cost the
// table's walk a fifth: 48 layers of S = 40 20.7 -> 28.9 us.)  s_trans: the transition matrix, or NULL.
template <int NJ, bool STAGED, int FORM>
__device__ __forceinline__ long long walk_states(int Li, int S, int m_pitch, const int32_t* __restrict__ tq, const int32_t* __restrict__ mq,
                                                 const int32_t* __restrict__ T0, long long trans_layer, const int32_t* __restrict__ C,
                                                 const int32_t* __restrict__ row_of, const int32_t* s_trans, int (&mrow)[NJ], int (&trow)[NJ],
                                                 int s, int m, int cur, int32_t* __restrict__ pl, bool* bad)
{
    const int lane = threadIdx.x;
    long long used = 0;
    // FORM: the solo kernel's states are a row of bases and rows of differences' words, two rows to a word if 16 bits do.
    int mnext[NJ], tnext[NJ];                                  // rows of layer l-1
    int crow[NJ], rows = 0;                                    // state row of each of this lane's strategies, rows a layer
    int half[NJ];                                              // ... where its bits begin in the row's words
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        crow[j] = k < S ? row_of[k] & 0xffff : 0;
        half[j] = FORM == kStateHalf ? 16 * (crow[j] & 1) : 0;
        if (FORM) crow[j] = 1 + (FORM == kStateHalf ? crow[j] >> 1 : crow[j]);
        rows = max(rows, crow[j] + 1);
        mnext[j] = k < S && Li > 1 ? mq[(Li - 2) * S + k] : 0;
        tnext[j] = k < S && Li > 1 ? tq[(Li - 2) * S + k] : 0;
    }
    rows = __reduce_max_sync(0xffffffffu, rows);
    // mem and time of the strategy the walk stands on: from here on they come along with the winner of each step
    int mm, tt;
    {
        int msel = mrow[0], tsel = trow[0];
#pragma unroll
        for (int j = 1; j < NJ; ++j) {
            msel = (s >> 5) == j ? mrow[j] : msel;
            tsel = (s >> 5) == j ? trow[j] : tsel;
        }
        mm = __shfl_sync(0xffffffffu, msel, s & 31);
        tt = __shfl_sync(0xffffffffu, tsel, s & 31);
    }
    for (int l = Li - 1; l >= 0; --l) {
        if (lane == 0) pl[l] = s;
        used += mm;
        if (mm > m) { *bad = true; break; }
        if (l == 0) break;
        const int32_t* prev = C + (size_t)(l - 1) * rows * m_pitch;
        const int32_t* T = T0 + (size_t)l * trans_layer;
        int cv[NJ], tv[NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int k = lane + 32 * j, src = m - mm - mnext[j];
            int g;
            if (FORM == 0) {
                g = k < S && src >= 0 ? (l > 1 ? prev[(size_t)crow[j] * m_pitch + src] : 0) : kInf;
            } else {
                const bool in = k < S && src >= 0;
                const int base = in ? (l > 1 ? prev[src] : 0) : kInf;
                const uint32_t word = in && l > 1 ? (uint32_t)prev[(size_t)crow[j] * m_pitch + src] : 0u;
                g = base < kInf ? base + (int)(FORM == kStateHalf ? (word >> half[j]) & 0xffffu : word) : kInf;     // where nothing is finite the words are not there
            }
            cv[j] = g < kInf ? g + tnext[j] : kInf;
            tv[j] = k < S ? (STAGED ? s_trans[k * S + s] : T[k * S + s]) : 0;
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {                          // rows of layer l-2 asked for, a step before the walk gets there
            const int k = lane + 32 * j;
            mrow[j] = mnext[j]; trow[j] = tnext[j];
            mnext[j] = k < S && l > 1 ? mq[(l - 2) * S + k] : 0;
            tnext[j] = k < S && l > 1 ? tq[(l - 2) * S + k] : 0;
        }
        m -= mm;
        int sp = 255;
        const int target = cur - tt;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            if (32 * j >= S) break;
            const unsigned b = __ballot_sync(0xffffffffu, cv[j] < kInf && cv[j] + tv[j] == target);
            if (b) {
                const int src = __ffs(b) - 1;
                sp = 32 * j + src;
                cur = __shfl_sync(0xffffffffu, cv[j], src);
                mm = __shfl_sync(0xffffffffu, mrow[j], src);
                tt = __shfl_sync(0xffffffffu, trow[j], src);
                break;
            }
        }
        if (sp >= S) { *bad = true; break; }
        s = sp;
    }
    return used;
}

enum Source { kTable, kArgmin, kStates };                      // kStates: of some instances; of the others the table
template <int NJ, int SRC, bool STAGED>
__global__ void backtrack_kernel(int B, int Lmax, int S, int M, int m_pitch, long long trans_inst, long long trans_layer,
                                 const int32_t* __restrict__ L, const int32_t* __restrict__ time_q,
                                 const int32_t* __restrict__ mem_q, const int32_t* __restrict__ trans_q,
                                 const int32_t* __restrict__ C, const uint8_t* __restrict__ A,
                                 const int32_t* __restrict__ C_last, const int32_t* __restrict__ lean_map, const int32_t* __restrict__ budget,
                                 int32_t* __restrict__ opt_cost, int32_t* __restrict__ plan,
                                 int32_t* __restrict__ mem_used, int32_t* __restrict__ status)
{
    extern __shared__ int32_t s_trans[];                       // the instance's transition matrix, where it has one that fits
    const int lane = threadIdx.x;
    const int i = blockIdx.x;
    // what does not depend on anything is asked for at once: every round trip to memory counts in a walk of a few dozen
    const int Li = L[i], st_in = status[i], bud = budget ? budget[i] : M;
    const size_t slice = (size_t)S * m_pitch;
    const int32_t* const T0 = trans_q + (size_t)i * trans_inst;
    if (STAGED) {
        for (int k = lane; k < S * S; k += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(s_trans + k)), "l"(T0 + k) : "memory");
    }
    const int32_t* tq = time_q + (size_t)i * Lmax * S;
    const int32_t* mq = mem_q + (size_t)i * Lmax * S;
    int mrow[NJ], trow[NJ];                                    // rows of the last layer (of one that exists, whatever L says)
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j, top = min(max(Li, 1), Lmax) - 1;
        mrow[j] = plan && k < S ? mq[top * S + k] : 0;
        trow[j] = plan && k < S ? tq[top * S + k] : 0;
    }
    unsigned long long key = ~0ull;                            // optimum at the budget: lowest s among the minima
    for (int s = lane; s < S; s += 32) {
        const unsigned long long k = ((unsigned long long)(unsigned)C_last[(size_t)i * slice + (size_t)s * m_pitch + min(max(bud, 0), M)] << 32) | (unsigned)s;
        key = k < key ? k : key;
    }
    if (STAGED) asm volatile("cp.async.wait_all;" ::: "memory");           // the matrix
    const int st0 = st_in & ~GALV_STATUS_INFEASIBLE;
    int32_t* pl = plan ? plan + (size_t)i * Lmax : nullptr;
    if (pl)
        for (int l = lane; l < Lmax; l += 32) pl[l] = -1;
    __syncwarp();          // lane 0 overwrites entries other lanes have just cleared
    // a search whose bounded waits ran out left void tables: not walked either
    const bool skip = (st0 & (GALV_STATUS_BAD_INPUT | GALV_STATUS_OVERFLOW_RISK | GALV_STATUS_TIMEOUT)) != 0 || bud < 0 || bud > M;
    if (skip) {
        if (lane == 0) {
            opt_cost[i] = kInf;
            if (mem_used) mem_used[i] = 0;
            status[i] = st0 | ((bud < 0 || bud > M) ? GALV_STATUS_BAD_INPUT : 0);
        }
        return;
    }
    key = warp_min_u64(key);
    const int opt = (int)(key >> 32);
    int s = (int)(key & 0xffffffffu);
    if (opt >= kInf) {
        if (lane == 0) {
            opt_cost[i] = kInf;
            if (mem_used) mem_used[i] = 0;
            status[i] = st0 | GALV_STATUS_INFEASIBLE;
        }
        return;
    }
    if (lane == 0) { opt_cost[i] = opt; status[i] = st0; }
    if (!pl) return;

    const int32_t* Ci = SRC == kArgmin ? nullptr : C + (size_t)i * Lmax * slice;
    bool bad = false;
    long long used;
    const int form = SRC == kStates ? lean_map[(size_t)i * S] : -1;
#define GALV_WALK_STATES(FORM) walk_states<NJ, STAGED, FORM>(Li, S, m_pitch, tq, mq, T0, trans_layer, Ci, lean_map + (size_t)i * S, s_trans, mrow, trow, s, bud, opt, pl, &bad)
    if (SRC == kStates && form >= 0)
        used = form & kStateHalf ? GALV_WALK_STATES(kStateHalf) : form & kStateWord ? GALV_WALK_STATES(kStateWord) : GALV_WALK_STATES(0);
    else
        used = walk_table<NJ, SRC == kArgmin>(Li, S, m_pitch, tq, mq, T0, trans_layer, Ci, SRC == kArgmin ? A + (size_t)i * Lmax * slice : nullptr, mrow, trow, s, bud, opt, pl, &bad);
#undef GALV_WALK_STATES
    if (bad && lane == 0) status[i] = st0 | GALV_STATUS_BAD_INPUT;
    if (lane == 0 && mem_used) mem_used[i] = (int32_t)used;
}

}  // namespace

cudaError_t galv_backtrack_launch(const galv_shape* sh, const int32_t* L, const int32_t* time_q,
                                  const int32_t* mem_q, const int32_t* trans_q, const int32_t* C,
                                  const uint8_t* A, const int32_t* C_last, const int32_t* lean_map, const int32_t* budget,
                                  int32_t* opt_cost, int32_t* plan, int32_t* mem_used, int32_t* status,
                                  cudaStream_t st)
{
    // a warp per instance, a CTA of its own; beside states one matrix per instance is kept in shared memory (48 KB: S <= 110)
    const bool staged = lean_map && sh->S > 32 && !(sh->flags & GALV_TRANS_PER_LAYER) && (size_t)sh->S * sh->S * 4 <= 48 * 1024;
    const size_t smem = staged ? (size_t)sh->S * sh->S * 4 : 0;
#define GALV_WALK_AS(NJ, SRC, STAGED) backtrack_kernel<NJ, SRC, STAGED><<<sh->B, 32, smem, st>>>( \
        sh->B, sh->Lmax, sh->S, sh->M, sh->m_pitch, galv_trans_inst(sh), galv_trans_layer(sh), L, time_q, mem_q, trans_q, C, A, C_last, lean_map, budget, \
        opt_cost, plan, mem_used, status)
#define GALV_WALK(NJ) do { \
        if (A) GALV_WALK_AS(NJ, kArgmin, false); \
        else if (!lean_map) GALV_WALK_AS(NJ, kTable, false); \
        else if (staged) GALV_WALK_AS(NJ, kStates, true); \
        else GALV_WALK_AS(NJ, kStates, false); } while (0)
    if (sh->S <= 32) GALV_WALK(1);
    else if (sh->S <= 64) GALV_WALK(2);
    else if (sh->S <= 128) GALV_WALK(4);
    else GALV_WALK(8);
#undef GALV_WALK
#undef GALV_WALK_AS
    return cudaGetLastError();
}
