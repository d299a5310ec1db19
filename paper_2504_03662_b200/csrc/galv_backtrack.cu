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

// NJ: strategies per lane (S <= 32 * NJ): the walk's chain of selects, loads and ballots is as long as it has to be.
template <int NJ>
__global__ void backtrack_kernel(int B, int Lmax, int S, int M, int m_pitch, long long trans_inst, long long trans_layer,
                                 const int32_t* __restrict__ L, const int32_t* __restrict__ time_q,
                                 const int32_t* __restrict__ mem_q, const int32_t* __restrict__ trans_q,
                                 const int32_t* __restrict__ C, const uint8_t* __restrict__ A,
                                 const int32_t* __restrict__ C_last, const int32_t* __restrict__ lean_map, const int32_t* __restrict__ budget,
                                 int32_t* __restrict__ opt_cost, int32_t* __restrict__ plan,
                                 int32_t* __restrict__ mem_used, int32_t* __restrict__ status, const bool staged)
{
    extern __shared__ int32_t s_trans[];                       // the instance's transition matrix, where it has one that fits
    const int lane = threadIdx.x;
    const int i = blockIdx.x;
    // what does not depend on anything is asked for at once: every round trip to memory counts in a walk of a few dozen
    const int Li = L[i], st_in = status[i], bud = budget ? budget[i] : M;
    const size_t slice = (size_t)S * m_pitch;
    const int32_t* const T0 = trans_q + (size_t)i * trans_inst;
    if (staged) {
        for (int k = lane; k < S * S; k += 32)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(s_trans + k)), "l"(T0 + k) : "memory");
    }
    unsigned long long key = ~0ull;                            // optimum at the budget: lowest s among the minima
    for (int s = lane; s < S; s += 32) {
        const unsigned long long k = ((unsigned long long)(unsigned)C_last[(size_t)i * slice + (size_t)s * m_pitch + min(max(bud, 0), M)] << 32) | (unsigned)s;
        key = k < key ? k : key;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");           // the matrix
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

    const int32_t* tq = time_q + (size_t)i * Lmax * S;
    const int32_t* mq = mem_q + (size_t)i * Lmax * S;
    int m = bud;
    long long used = 0;
    // One dependent memory round trip per layer: the cell's value is carried along (it is the chosen
    // candidate of the step before), and the mem / time rows of the next layer down are fetched, whole,
    // while this layer's candidates are in flight; lane k%32 keeps entries k, k+32, ... (S <= 256).
    int cur = opt;                                             // C[l][m][s] of the cell the walk stands on
    int mrow[NJ], trow[NJ], mnext[NJ], tnext[NJ];              // rows of layers l and l-1
    // the resident kernel's states in place of the table: state row of each of this lane's strategies, rows a layer
    const bool lean = !A && lean_map && lean_map[(size_t)i * S] >= 0;
    int crow[NJ], rows = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        crow[j] = lean && lane + 32 * j < S ? lean_map[(size_t)i * S + lane + 32 * j] : 0;
        rows = max(rows, crow[j] + 1);
    }
    rows = __reduce_max_sync(0xffffffffu, rows);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        mrow[j] = k < S ? mq[(Li - 1) * S + k] : 0;
        trow[j] = k < S ? tq[(Li - 1) * S + k] : 0;
        mnext[j] = k < S && Li > 1 ? mq[(Li - 2) * S + k] : 0;
        tnext[j] = k < S && Li > 1 ? tq[(Li - 2) * S + k] : 0;
    }
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
        if (mm > m) {                  // cannot happen on consistent tables: the cell would be +inf; never index below column 0
            if (lane == 0) status[i] = st0 | GALV_STATUS_BAD_INPUT;
            break;
        }
        if (l == 0) break;
        int sp = 255;
        int cv[NJ], tv[NJ];
        if (A) {
            sp = A[((size_t)i * Lmax + l) * slice + (size_t)s * m_pitch + m];
        } else {
            // every row's candidate is asked for before the first is looked at: one round trip to memory, not one per 32 rows
            const int32_t* prev = C + ((size_t)i * Lmax + (l - 1)) * slice + (m - mm);
            const int32_t* T = T0 + (size_t)l * trans_layer;       // paid between layers l-1 and l
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const int k = lane + 32 * j;
                if (lean) {
                    // value of strategy k in layer l-1: its time on top of the state at the column its memory leaves
                    const int src = m - mm - mnext[j];
                    const int g = k < S && src >= 0 ? (l > 1 ? C[(size_t)i * Lmax * slice + ((size_t)(l - 1) * rows + crow[j]) * m_pitch + src] : 0) : kInf;
                    cv[j] = g < kInf ? g + tnext[j] : kInf;
                } else {
                    cv[j] = k < S ? prev[(size_t)k * m_pitch] : kInf;
                }
                tv[j] = k < S ? (staged ? s_trans[k * S + s] : T[k * S + s]) : 0;
            }
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {                          // rows of layer l-2 asked for, a step before the walk gets there
            const int k = lane + 32 * j;
            mrow[j] = mnext[j]; trow[j] = tnext[j];
            mnext[j] = k < S && l > 1 ? mq[(l - 2) * S + k] : 0;
            tnext[j] = k < S && l > 1 ? tq[(l - 2) * S + k] : 0;
        }
        m -= mm;
        if (A) {
            int msel = mrow[0], tsel = trow[0];
#pragma unroll
            for (int j = 1; j < NJ; ++j) {
                msel = (sp >> 5) == j ? mrow[j] : msel;
                tsel = (sp >> 5) == j ? trow[j] : tsel;
            }
            mm = __shfl_sync(0xffffffffu, msel, sp & 31);
            tt = __shfl_sync(0xffffffffu, tsel, sp & 31);
        } else {
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
        }
        if (sp >= S) {                 // cannot happen on consistent tables; stop instead of walking off
            if (lane == 0) status[i] = st0 | GALV_STATUS_BAD_INPUT;
            break;
        }
        s = sp;
    }
    if (lane == 0 && mem_used) mem_used[i] = (int32_t)used;
}

}  // namespace

cudaError_t galv_backtrack_launch(const galv_shape* sh, const int32_t* L, const int32_t* time_q,
                                  const int32_t* mem_q, const int32_t* trans_q, const int32_t* C,
                                  const uint8_t* A, const int32_t* C_last, const int32_t* lean_map, const int32_t* budget,
                                  int32_t* opt_cost, int32_t* plan, int32_t* mem_used, int32_t* status,
                                  cudaStream_t st)
{
    // a warp per instance, a CTA of its own; one matrix per instance is kept in shared memory (48 KB: S <= 110; 48 layers of
    // S = 48 69 -> 56 us), a small one stays in L1 anyway (24 layers of S = 24: 22.5 us so, 24 with the copy)
    const bool staged = plan && !A && sh->S > 32 && !(sh->flags & GALV_TRANS_PER_LAYER) && (size_t)sh->S * sh->S * 4 <= 48 * 1024;
    const size_t smem = staged ? (size_t)sh->S * sh->S * 4 : 0;
#define GALV_WALK(NJ) backtrack_kernel<NJ><<<sh->B, 32, smem, st>>>( \
        sh->B, sh->Lmax, sh->S, sh->M, sh->m_pitch, galv_trans_inst(sh), galv_trans_layer(sh), L, time_q, mem_q, trans_q, C, A, C_last, lean_map, budget, \
        opt_cost, plan, mem_used, status, staged)
    if (sh->S <= 32) GALV_WALK(1);
    else if (sh->S <= 64) GALV_WALK(2);
    else if (sh->S <= 128) GALV_WALK(4);
    else GALV_WALK(8);
#undef GALV_WALK
    return cudaGetLastError();
}
