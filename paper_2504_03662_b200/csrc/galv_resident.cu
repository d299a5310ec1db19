// The whole recurrence of one instance on the SMs of one thread-block cluster, its state kept in shared memory.
//
//   C[l][m][s] = time(l,s) + G[l][m - mem(l,s)][s],   G[l][m][s] = min_{s'} ( C[l-1][m][s'] + trans(s',s) )
//
// (Section 3 of the paper: dynamic-programming search over a performance model; Sections 3-4: it runs again while
// the job runs.)
//
// What a layer hands to the next one is G, and G has one row per DISTINCT COLUMN of the transition matrix: strategies
// with equal columns have equal G.  Strategies with equal ROWS enter the minimum with the same offset, so only the
// smallest of them matters.  A matrix that prices a move between layouts (tensor-parallel degree, sequence
// parallelism) has a handful of distinct rows and columns however many strategies there are (8 among 64, 4 among 24):
// a cell then costs one addition, one minimum over its class and its store instead of S add-mins, and the state of an
// instance shrinks from S to 8 rows.  The kernel finds the classes itself, by comparing the matrix's rows and columns
// word by word, so nothing is assumed about where a matrix comes from.
// A matrix without such structure keeps all S rows.  Then a candidate C[l-1][m][s'] that lies more than the largest
// transition entry above its column's best can neither win nor tie (the best row gives a candidate at most that entry
// above itself), so a warp relaxes only the rows that are alive in one of its columns.
//
// The budget columns are split over the CTAs of the cluster: CTA r owns columns r*W .. r*W+W-1 and keeps their G in two
// buffers (this layer's, the next one's), with a halo of H columns to their left: C is produced by GATHERING G at
// m - mem(l,s), from this CTA's own shared memory as long as the shift stays within the halo, else from its owner's.  After
// a layer the service warp sends each row's last columns to the CTAs further up as bulk copies counted on their mbarriers (a
// store through the cluster window took 100 cycles a warp, reading the cells from their owner a round trip on every gather's
// chain: 8.4 us a layer on one instance of 24 strategies over 16 CTAs).  Each CTA waits for its halo with a limit (GALV_STATUS_TIMEOUT);
// the cluster barrier's arrival of one layer is waited for in the next.  No cooperative launch, no cluster multicast, no
// workspace but a word per instance and the path flag; the tables go out as full 128-byte lines and are never read back.
//
// Validation is the kernel's own (same rules and status bits as everywhere).  An instance whose state does not fit this
// launch's shared memory is left alone and marked in done[]; a second launch with larger clusters or the tiled kernels
// take it.

#include <cuda.h>

#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>

#include "galv_internal.h"

namespace {

constexpr int kInf = GALV_INF;
constexpr int kMaxSortedB = 512;          // instances whose lengths fit the ranking scratch below
constexpr int kMaxS = 128;
constexpr int kMaxWarps = 15;             // compute warps per CTA (with the service warp 512 threads: 128 registers each)
constexpr int kStaticSmem = 5632;         // the kernel's static shared memory, rounded up
constexpr int kClassMax = kResidentClassMax;

struct RsArgs {
    int B, Lmax, S, M, m_pitch;
    int CL;            // CTAs per cluster
    int W;             // budget columns per CTA (multiple of 32)
    int gints;         // words of one state buffer: rows of W columns and their halo
    int stage_at;      // word offset of the collected rows
    int SP;            // row pitch of the full transition matrix in shared memory; 0: no room for unstructured matrices
    int sorted;        // clusters take the instances longest first
    int second;        // only the instances earlier launches left alone
    int probed;        // done[] says which matrices are unstructured
    int follow, k_max;             // see RsPlan
    int withhold;      // test hook: a cluster's first CTA keeps the halo of layer 0 to itself, so that the waits for it run out
    const int32_t* L;
    const int32_t* time_q;
    const int32_t* mem_q;
    const int32_t* trans_q;
    long long trans_inst, trans_layer;
    int32_t* C;        // full table or NULL
    int32_t* states;   // in place of the table, when nobody sees it: the states between the layers, [Lmax][rows][m_pitch] per instance; or NULL
    int32_t* map;      // [B][S] state row of each strategy, with `states`
    uint8_t* A;        // argmin table or NULL
    int32_t* C_last;
    int32_t* status;
    int32_t* path;     // [4] device flags of the search; [3]: kernel that ran
    int32_t* done;     // [B] 1: this instance needs nothing more
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ int ld_cluster(uint32_t addr) {
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, int v) { asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void red_min_cluster(uint32_t addr, int v) { asm volatile("red.relaxed.cluster.shared::cluster.min.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ int ld_cluster_u8(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u8 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return (int)v;
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// barrier of the CTA whose parties stand at different places in the code
__device__ __forceinline__ void cta_barrier() {
    __syncwarp();                                              // the aligned forms want the whole warp together
    asm volatile("bar.sync 0;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void fence_cluster() { asm volatile("fence.acq_rel.cluster;" ::: "memory"); }
// an arrival that orders nothing
__device__ __forceinline__ void cluster_arrive_relaxed() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void whole_barrier(int CL) {
    if (CL == 1) cta_barrier();
    else { cluster_arrive(); cluster_wait(); }
}
// One box [S][W / 32][32] from shared memory to element coordinates (0, g0, row0) of the table behind `map`, seen as
// [rows][m_pitch / 32][32]; what lies beyond the tensor's edge (the last CTA's columns past m_pitch) is not written.
__device__ __forceinline__ void tensor_store_3d(const CUtensorMap* map, const void* src, int g0, int row0) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(map), "r"(0), "r"(g0), "r"(row0), "r"(smem_addr(src)) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// bytes of this CTA's shared memory to the same cluster's CTA that `dst` and `bar` lie in; counted on its mbarrier
__device__ __forceinline__ void bulk_to_cta(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar) { asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void cp_async_4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Everything the layer loop needs; lives in registers (all members are uniform over the CTA).
struct Ctx {
    int S, M, W, H, P, G, CL, rank, Li, m_pitch, Kr, Kc, tmax, SP, NW, gints;
    int32_t* g0;               // [2][gints] state of this layer / the next: rows of P = H + W columns
    uint8_t* a0;               // [2][gints] its argmin (argmin table only)
    uint32_t rec;              // address of the per-layer records: four slots of 24 * S2 bytes
    const int* slot;           // [4] the slot of layer l is slot[l & 3] (layers with the same rows share one)
    int S2;                    // record entries a slot
    int n_all;                 // strategies of a slot's records, pads included
    const int* front;          // [4] no column below front[l & 3] holds a finite value in layer l
    const int* reach;          // [4] largest shift of a slot's layer
    const int32_t* tsm;        // transition entries: [16][16] by class, or [S][SP] (two of them with one matrix per layer)
    int tmat;                  // entries of one full matrix when there is one per layer, else 0
    const int* cs;             // [kClassMax + 1] first record of each class
    const int* csp;            // [4][kClassMax + 1] the same in the list of the records that can matter
    const int* cdelta;         // [16] cluster-window address of CTA d minus this CTA's own shared address
    int32_t* stage;            // [2][S][W] collected rows
    int32_t* C;                // this instance's table
    int32_t* states;           // ... or the states between its layers, or NULL
    uint8_t* A;
    int32_t* C_last;
    size_t slice;
    uint32_t bars;             // address of the two mbarriers the halo's bytes are counted on (even, odd layers)
    uint32_t halo_bytes;       // bytes of halo that arrive a layer
    bool strict;               // some shift reaches beyond the halo: layers end with the full cluster barrier
    int* late;                 // [0] set when a bounded wait ran out; [1] the layer from whose halo on they do not go round any more
};
constexpr int kNever = 0x7fffffff;

// End of a layer, by every warp of the CTA.  The state of layer l+1 is complete in this CTA; its last columns go to the
// halo of the CTAs further up that hold them, one bulk copy (through the TMA unit) a row and CTA, issued by the
// service warp: plain stores through the cluster window took about 100 cycles a warp store, 13 thousand a layer for 7 rows of
// 608 columns.  Then the wait for this CTA's own halo.
// The cluster barrier only keeps the buffers apart: an arrival says that this CTA has gathered from the older buffer
// and received its halo, and it is waited for a layer later, before the copies that overwrite that buffer are issued.
// With shifts beyond the halo other CTAs' state is read as well, and the barrier is waited for at once.
// Of the arrivals only one warp's is a release: the other warps' reads of the older buffer come before its own by the CTA's
// barrier at the start of the hand-over, and a release covers what its warp has so observed.  It waits for what its warp has
// in flight, so it is the service warp's where the compute warps store to the table themselves.  Where the service warp has
// just sent a layer of collected rows (48 layers on clusters of 5: 219 us with its release, 165 with none) it is a compute
// warp's fence, set before the wait for the halo, which hides it, and a relaxed arrival.
//
// A wait that runs out sets late[0], at which the CTA's other waits give up too.  If it is the service warp's, it also
// writes its layer v into late[1] of every CTA (the smallest stays) before it arrives at the barrier of layer v.  All service
// warps have waited for that barrier when they look at the word in layer v + 2: from there on no halo is sent or expected
// anywhere in the cluster, and the layers run out with their barriers alone.  (Bytes of layer v + 2 would be counted on the
// mbarrier whose phase of layer v is still open.)  Before anybody leaves, each CTA waits once more, with the same limit, for
// what of layers v and v + 1 may still be under way to it.
template <bool ARG>
__device__ __forceinline__ void send_halo(const Ctx& c, int l, int warp, int lane, bool on = true)
{
    cta_barrier();
    if (c.CL == 1) return;
    if (!c.strict) cluster_wait();
    const uint32_t bar = c.bars + 8u * (l & 1);
    if (warp == c.NW && on) {
        const uint32_t gn = smem_addr(c.g0 + ((l + 1) & 1) * c.gints), an = ARG ? smem_addr(c.a0 + ((l + 1) & 1) * c.gints) : 0u;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");        // plain stores of the state, read next by bulk copies
        for (int d = c.rank + 1, low = c.W - c.H; d < c.CL && low < c.W; ++d, low += c.W) {
            // CTA d holds the columns from d*W - H on: this CTA's local columns from `low` on
            const int from = max(low, 0), n = c.W - from, delta = c.cdelta[d];
            const int at = c.H + from, to = at - (d - c.rank) * c.W;
            for (int k = lane; k < c.Kc; k += 32) {
                bulk_to_cta(gn + (uint32_t)(delta + (k * c.P + to) * 4), gn + (uint32_t)(k * c.P + at) * 4u, (uint32_t)n * 4u, bar + (uint32_t)delta);
                if (ARG) bulk_to_cta(an + (uint32_t)(delta + k * c.P + to), an + (uint32_t)(k * c.P + at), (uint32_t)n, bar + (uint32_t)delta);
            }
        }
    }
}
constexpr int kWaitPolls = 1 << 18;                            // try_wait sleeps in hardware between polls: one second (2^20: four)
__device__ __forceinline__ bool halo_came(const Ctx& c, int l)
{
    const uint32_t bar = c.bars + 8u * (l & 1), parity = (uint32_t)(l >> 1) & 1u;
    int polls = 0;
    while (!mbar_try(bar, parity))
        if (++polls > kWaitPolls || *(volatile int*)c.late) { *(volatile int*)c.late = 1; return false; }
    return true;
}
template <bool STAGE>
__device__ __forceinline__ void await_halo(const Ctx& c, int l, int warp)
{
    if (c.CL == 1) return;
    if (STAGE && warp == 0) fence_cluster();                     // while the halo is on its way
    if (c.halo_bytes) halo_came(c, l);
    if (c.strict) { cluster_arrive(); cluster_wait(); }
    else cluster_arrive_relaxed();
}
__device__ __noinline__ void raise_stop(uint32_t late, const int* cdelta, int CL, int l)
{
    for (int d = 0; d < CL; ++d) {
        st_cluster(late + (uint32_t)cdelta[d], 1);
        red_min_cluster(late + 4u + (uint32_t)cdelta[d], l);
    }
    fence_cluster();
}
// ... by the service warp
template <bool STAGE>
__device__ __forceinline__ void await_halo_service(const Ctx& c, int l, int lane, bool on)
{
    if (c.CL == 1) return;
    if (c.halo_bytes && on) {
        if (lane == 0) mbar_expect(c.bars + 8u * (l & 1), c.halo_bytes);
        if (!halo_came(c, l)) raise_stop(smem_addr(c.late), c.cdelta, c.CL, l);
    }
    if (c.strict || !STAGE) cluster_arrive();
    else cluster_arrive_relaxed();
    if (c.strict) cluster_wait();
}

// Records of a layer, one entry per strategy in class order, three arrays of S2 entries each (a slot of the ring):
//   int2 (x, time)  x = byte offset, from the start of the state, of the cell that column 0 of this CTA reads (the row of
//                   the strategy's column class, shifted by mem); time = kInf where mem exceeds the budget (+inf row)
//   int  row        byte offset of the strategy's row in the table
//   int  who        mem | strategy << 24
//   int2 (x, time)  of the strategies that can be the smallest of their class in some column: a strategy whose column
//                   class, too, has a member that needs no more memory and no more time never is (G does not rise
//                   with the budget).  ZeRO stages and checkpointing mostly differ in memory alone: about half drop out.
// A class has an even number of entries (the last one may stand twice: it stores the same values again, and a minimum
// does not change), so entries are read two to a 128-bit load, and four at a time from one address.
// Shared-memory accesses of the layer loop go through 32-bit addresses and are written in batches, loads first: the table
// stores between two strategies would otherwise hold the next strategy's loads back (they could alias for all the
// compiler knows), and a strategy would cost the latency of its whole chain (220 cycles) instead of a share of it.
__device__ __forceinline__ int lds(uint32_t a) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
template <int OFF>
__device__ __forceinline__ int lds_at(uint32_t a) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
__device__ __forceinline__ int lds_u8(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return (int)v;
}
__device__ __forceinline__ int4 lds4(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, int v) { asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts_u8(uint32_t a, int v) { asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

template <int OFF>
__device__ __forceinline__ int4 lds4_at(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4+%5];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a), "n"(OFF));
    return v;
}
template <int TM, int J = 0>
__device__ __forceinline__ void lds_row(uint32_t a, int (&g)[TM]) {
    g[J] = lds_at<128 * J>(a);
    if constexpr (J + 1 < TM) lds_row<TM, J + 1>(a, g);
}

// Where the cell lies that column `col` of this CTA reads at a shift of mem: the CTA that owns it and its column there.  The
// 32 columns of a warp start in one CTA and end in it or in the next, so the division is the warp's.
struct Owner { int at, delta; bool in; };
__device__ __forceinline__ Owner owner_of(const Ctx& c, int col, int mem)
{
    const int first = c.rank * c.W + (col & ~31) - mem;        // may lie below column 0, by less than the cluster's columns
    int o = (first + c.CL * c.W) / c.W - c.CL;
    int at = first + (col & 31) - o * c.W;
    if (at >= c.W) { at -= c.W; ++o; }
    const bool in = o >= 0;
    return {at, c.cdelta[in ? o : 0], in};
}

// G at the columns that column `col` of this CTA (and those 32, 64, ... after it) reads; ga: the state's address plus
// 4 * col.  FAR: the layer has shifts beyond the halo, whose cells are read from the CTA that owns them.
template <int TM, bool FAR>
__device__ __forceinline__ void gather(const Ctx& c, uint32_t ga, int x, int who, int col, int (&g)[TM])
{
    const int mem = who & 0xffffff;
    if (!FAR || mem <= c.H) {
        lds_row<TM>(ga + (uint32_t)x, g);
    } else {
        static_assert(!FAR || TM == 1, "a run of 32 columns has two owners at most");
        const Owner o = owner_of(c, col, mem);
        g[0] = kInf;
        if (o.in) g[0] = ld_cluster(ga - 4u * (uint32_t)col + (uint32_t)x + (uint32_t)mem * 4u + (uint32_t)(o.at * 4 + o.delta));
    }
}
// ... and their argmin entries; aa: the argmin state's address plus col
template <int TM, bool FAR>
__device__ __forceinline__ void gather_arg(const Ctx& c, uint32_t aa, int x, int who, int col, int (&a)[TM])
{
    const int mem = who & 0xffffff, off = x >> 2;
    if (!FAR || mem <= c.H) {
#pragma unroll
        for (int j = 0; j < TM; ++j) a[j] = lds_u8(aa + (uint32_t)(off + 32 * j));
    } else {
        const Owner o = owner_of(c, col, mem);
        a[0] = 255;
        if (o.in) a[0] = ld_cluster_u8(aa - (uint32_t)col + (uint32_t)(off + mem) + (uint32_t)(o.at + o.delta));
    }
}

// Values of one state row for the tile.
template <int TM, bool ARG, bool KEEP>
__device__ __forceinline__ void emit(const Ctx& c, int l, uint32_t gn, uint32_t an, int k, int colb, int lane, const int (&v)[TM], const int (&a)[TM])
{
    const int at = k * c.P + c.H + colb + lane;
#pragma unroll
    for (int j = 0; j < TM; ++j) {
        sts(gn + (uint32_t)(at + 32 * j) * 4u, v[j]);
        if (ARG) sts_u8(an + (uint32_t)(at + 32 * j), a[j]);
    }
    if (KEEP && c.states) {
        const int m = c.rank * c.W + colb + lane;
        int32_t* const p = c.states + ((size_t)(l + 1) * c.Kc + k) * c.m_pitch + m;
#pragma unroll
        for (int j = 0; j < TM; ++j)
            if (m + 32 * j < c.m_pitch) p[32 * j] = v[j];
    }
}

// Where a tile's values go in the table.
// STAGE: the rows of a layer are collected in shared memory ([S][W], two layers in turn) and leave with one bulk tensor
// store the service warp issues.  A table store of a warp holds the load / store unit for four cycles and more, and the
// loads of the next strategies, which the layer's chain of latencies consists of, queue up behind it.
template <bool STORE, bool ARG, bool STAGE>
struct Out {
    uint32_t stage;        // the tile's first column plus this lane, strategy 0, in the collected rows
    char* C;               // ... in the table
    uint8_t* A;
    bool whole;            // every column of the tile is a budget column
    int cols;              // columns of the tile that exist in the table, less this lane
    int budget;            // ... that are budget columns, less this lane
    template <int TM>
    __device__ __forceinline__ void put(uint32_t row, const int (&v)[TM], const int (&a)[TM]) const
    {
        if (STAGE) {
#pragma unroll
            for (int j = 0; j < TM; ++j) sts(stage + row + 128u * j, whole || 32 * j < budget ? v[j] : kInf);
        } else if (STORE) {
            int32_t* const p = reinterpret_cast<int32_t*>(C + row);
            if (whole) {
#pragma unroll
                for (int j = 0; j < TM; ++j) p[32 * j] = v[j];
            } else {                                           // +inf in the pad columns beyond the budget
#pragma unroll
                for (int j = 0; j < TM; ++j)
                    if (32 * j < cols) p[32 * j] = 32 * j < budget ? v[j] : kInf;
            }
        }
        if (ARG) {
            uint8_t* const p = A + (row >> 2);
#pragma unroll
            for (int j = 0; j < TM; ++j)
                if (whole || 32 * j < cols) p[32 * j] = (uint8_t)((whole || 32 * j < budget) && v[j] < kInf ? a[j] : 255);
        }
    }
};

// U entries' records, from entry address ra (of the (x, time) array) on.
template <int U>
struct Recs { int x[U], t[U], row[U], who[U]; };
template <int U, bool ROW, bool WHO>
__device__ __forceinline__ void fetch_recs(const Ctx& c, uint32_t ra, uint32_t rowa, Recs<U>& r)
{
    if constexpr (U >= 2) {
        const int4 p = lds4_at<0>(ra);
        r.x[0] = p.x; r.t[0] = p.y; r.x[1] = p.z; r.t[1] = p.w;
        if constexpr (U == 4) {
            const int4 q = lds4_at<16>(ra);
            r.x[2 % U] = q.x; r.t[2 % U] = q.y; r.x[3 % U] = q.z; r.t[3 % U] = q.w;
        }
    } else {
        r.x[0] = lds_at<0>(ra); r.t[0] = lds_at<4>(ra);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) { r.row[u] = 0; r.who[u] = 0; }
    if (ROW) {
        r.row[0] = lds_at<0>(rowa);
        if constexpr (U >= 2) r.row[1 % U] = lds_at<4>(rowa);
        if constexpr (U == 4) { r.row[2 % U] = lds_at<8>(rowa); r.row[3 % U] = lds_at<12>(rowa); }
    }
    if (WHO) {
        const uint32_t w = rowa + 4u * c.S2;
        r.who[0] = lds_at<0>(w);
        if constexpr (U >= 2) r.who[1 % U] = lds_at<4>(w);
        if constexpr (U == 4) { r.who[2 % U] = lds_at<8>(w); r.who[3 % U] = lds_at<12>(w); }
    }
}

// U strategies: their C values to the table, their smallest into h (with ARG: whose it is).
template <int U, int TM, bool STORE, bool ARG, bool STAGE, bool FAR>
__device__ __forceinline__ void scan(const Ctx& c, const Out<STORE, ARG, STAGE>& out, uint32_t ra, uint32_t rowa, uint32_t ga, uint32_t aa, int col, int (&h)[TM], int (&hs)[TM])
{
    Recs<U> r;
    int v[U][TM], a[ARG ? U : 1][TM];
    fetch_recs<U, STORE || ARG, ARG || FAR>(c, ra, rowa, r);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        gather<TM, FAR>(c, ga, r.x[u], r.who[u], col, v[u]);
        if (ARG) gather_arg<TM, FAR>(c, aa, r.x[u], r.who[u], col, a[ARG ? u : 0]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
        for (int j = 0; j < TM; ++j) {
            if (STORE || ARG) {
                v[u][j] = __viaddmin_s32(v[u][j], r.t[u], kInf);
                if (ARG) hs[j] = v[u][j] < h[j] ? r.who[u] >> 24 : hs[j];  // ascending strategies: the lowest keeps a tie
                h[j] = min(h[j], v[u][j]);
            } else {
                h[j] = __viaddmin_s32(v[u][j], r.t[u], h[j]);
            }
        }
        if (STORE || ARG) out.template put<TM>((uint32_t)r.row[u], v[u], a[ARG ? u : 0]);
    }
}

// Which of U strategies are alive in some column of the tile, as bits.
template <int U, int TM, bool FAR>
__device__ __forceinline__ uint32_t alive(const Ctx& c, uint32_t ra, uint32_t rowa, uint32_t ga, int col, const int (&thr)[TM])
{
    Recs<U> r;
    int v[U][TM];
    uint32_t bits = 0;
    fetch_recs<U, false, FAR>(c, ra, rowa, r);
#pragma unroll
    for (int u = 0; u < U; ++u) gather<TM, FAR>(c, ga, r.x[u], r.who[u], col, v[u]);
#pragma unroll
    for (int u = 0; u < U; ++u) {
        bool live = false;
#pragma unroll
        for (int j = 0; j < TM; ++j) live = live || __viaddmin_s32(v[u][j], r.t[u], kInf) <= thr[j];
        if (__any_sync(0xffffffffu, live)) bits |= 1u << u;
    }
    return bits;
}

// One layer of one tile of TM x 32 columns.  KC: rows of the next state held in accumulators (PRUNE: per block of rows).
template <int KC, int TM, bool PRUNE, bool STORE, bool ARG, bool STAGE, bool FAR>
__device__ __forceinline__ void tile(const Ctx& c, int l, int colb, int lane)
{
    const int slot = c.slot[l & 3], col = colb + lane;
    const uint32_t ra = c.rec + (uint32_t)(slot * c.S2) * 24u, rowa = ra + (uint32_t)c.S2 * 8u;
    const uint32_t ga = smem_addr(c.g0 + (l & 1) * c.gints + col), gn = smem_addr(c.g0 + ((l + 1) & 1) * c.gints);
    const uint32_t aa = ARG ? smem_addr(c.a0 + (l & 1) * c.gints + col) : 0u, an = ARG ? smem_addr(c.a0 + ((l + 1) & 1) * c.gints) : 0u;
    const int colg = c.rank * c.W + colb;                      // the tile's first budget column
    Out<STORE, ARG, STAGE> out;
    out.stage = STAGE ? smem_addr(c.stage + (l & 1) * c.S * c.W + col) : 0u;
    out.C = STORE ? reinterpret_cast<char*>(c.C + (size_t)l * c.slice + colg + lane) : nullptr;
    out.A = ARG ? c.A + (size_t)l * c.slice + colg + lane : nullptr;
    out.whole = colg + 32 * TM - 1 <= c.M;
    out.cols = c.m_pitch - colg - lane;
    out.budget = c.M + 1 - colg - lane;

    if (colg + 32 * TM - 1 < c.front[l & 3]) {                  // nothing finite in the tile
        int inf[TM], none[TM];
#pragma unroll
        for (int j = 0; j < TM; ++j) { inf[j] = kInf; none[j] = 255; }
        if (STORE || ARG)
#pragma unroll 4
            for (int e = 0; e < c.S; ++e) out.template put<TM>((uint32_t)(e * (STAGE ? c.W : c.m_pitch)) * 4u, inf, none);
        for (int k = 0; k < c.Kc; ++k) emit<TM, ARG, !STORE && !ARG>(c, l, gn, an, k, colb, lane, inf, none);
        return;
    }

    if (!PRUNE) {
        int acc[KC][TM], arg[ARG ? KC : 1][TM];
#pragma unroll
        for (int k = 0; k < KC; ++k)
#pragma unroll
            for (int j = 0; j < TM; ++j) { acc[k][j] = kInf; if (ARG) arg[k][j] = 255; }
        int e = 0;
        // without a table to write, only the strategies that can matter
        constexpr bool kAll = STORE || ARG || FAR;
        const int* const cs = kAll ? c.cs : c.csp + slot * (kClassMax + 1);
        const uint32_t la = kAll ? ra : ra + (uint32_t)c.S2 * 16u;
        const uint32_t ta = smem_addr(c.tsm);
        if constexpr (!STORE && !ARG && !FAR) {
            // The classes as one run of entries, four at a time: the records of the next four are asked for before this
            // four are worked on, their cells half-way through, so that a warp on its own waits for neither (128 instances
            // of the heterogeneous stack, optima only: 3.03 -> 2.80 ms; with stores in the loop it is the other way round).
            const int n = cs[c.Kr];
            int end = cs[1], next_end = cs[min(2, c.Kr)], k = 0;
            int h[TM];
#pragma unroll
            for (int j = 0; j < TM; ++j) h[j] = kInf;
            int4 t4[KC / 4];
#pragma unroll
            for (int q = 0; q < KC / 4; ++q) t4[q] = lds4(ta + 16u * q);
            auto close = [&]() {                               // a class is complete: its smallest goes on to every row of the next state
#pragma unroll
                for (int q = 0; q < KC / 4; ++q) {
                    const int t[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
#pragma unroll
                    for (int j = 0; j < TM; ++j)
#pragma unroll
                        for (int u = 0; u < 4; ++u) acc[4 * q + u][j] = __viaddmin_s32(h[j], t[u], acc[4 * q + u][j]);
                }
#pragma unroll
                for (int j = 0; j < TM; ++j) h[j] = kInf;
                ++k;
                end = next_end;
                next_end = cs[min(k + 2, c.Kr)];
#pragma unroll
                for (int q = 0; q < KC / 4; ++q) t4[q] = lds4(ta + (uint32_t)(min(k, kClassMax - 1) * kClassMax + 4 * q) * 4u);
            };
            auto two = [&](const Recs<4>& r, const int (&g)[4][TM], auto first, int at) {
                constexpr int F = decltype(first)::value;
                while (at >= end && k < c.Kr) close();          // classes without an entry that can matter
#pragma unroll
                for (int u = F; u < F + 2; ++u)
#pragma unroll
                    for (int j = 0; j < TM; ++j) h[j] = __viaddmin_s32(g[u][j], r.t[u], h[j]);
            };
            auto cells = [&](const Recs<4>& r, int (&g)[4][TM]) {
#pragma unroll
                for (int u = 0; u < 4; ++u) gather<TM, false>(c, ga, r.x[u], 0, col, g[u]);
            };
            Recs<4> r0, r1;
            int g0[4][TM], g1[4][TM];
            fetch_recs<4, false, false>(c, la, rowa, r0);
            cells(r0, g0);
            while (e < n) {
                fetch_recs<4, false, false>(c, la + 8u * (e + 4), rowa + 4u * (e + 4), r1);
                two(r0, g0, std::integral_constant<int, 0>(), e);
                cells(r1, g1);
                if (e + 2 < n) two(r0, g0, std::integral_constant<int, 2>(), e + 2);
                e += 4;
                if (e >= n) break;
                fetch_recs<4, false, false>(c, la + 8u * (e + 4), rowa + 4u * (e + 4), r0);
                two(r1, g1, std::integral_constant<int, 0>(), e);
                cells(r0, g0);
                if (e + 2 < n) two(r1, g1, std::integral_constant<int, 2>(), e + 2);
                e += 4;
            }
            while (k < c.Kr) close();
        } else {
            for (int k = 0; k < c.Kr; ++k) {
                const int end = cs[k + 1];
                int h[TM], hs[TM];
#pragma unroll
                for (int j = 0; j < TM; ++j) { h[j] = kInf; hs[j] = 255; }
                int4 t4[KC / 4];
#pragma unroll
                for (int q = 0; q < KC / 4; ++q) t4[q] = lds4(ta + (uint32_t)(k * kClassMax + 4 * q) * 4u);
                constexpr int U = TM > 4 && STORE ? 2 : 4;
                for (; e + U <= end; e += U) scan<U, TM, STORE, ARG, STAGE, FAR>(c, out, la + 8u * e, rowa + 4u * e, ga, aa, col, h, hs);
                if (U == 4 && e < end) { scan<2, TM, STORE, ARG, STAGE, FAR>(c, out, la + 8u * e, rowa + 4u * e, ga, aa, col, h, hs); e += 2; }
#pragma unroll
                for (int q = 0; q < KC / 4; ++q) {
                    const int t[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
#pragma unroll
                    for (int j = 0; j < TM; ++j)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (ARG) {
                                const int cand = h[j] + t[u], old = acc[4 * q + u][j], oa = arg[ARG ? 4 * q + u : 0][j];
                                const bool better = cand < old || (cand == old && hs[j] < oa);
                                if (better && h[j] < kInf) { acc[4 * q + u][j] = cand; arg[ARG ? 4 * q + u : 0][j] = hs[j]; }
                            } else {
                                acc[4 * q + u][j] = __viaddmin_s32(h[j], t[u], acc[4 * q + u][j]);
                            }
                        }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (k < c.Kc) emit<TM, ARG, !STORE && !ARG>(c, l, gn, an, k, colb, lane, acc[k], arg[ARG ? k : 0]);
    } else {
        int thr[TM], dummy[TM];
#pragma unroll
        for (int j = 0; j < TM; ++j) { thr[j] = kInf; dummy[j] = 255; }
        int s = 0;
        for (; s + 4 <= c.S; s += 4) scan<4, TM, STORE, ARG, STAGE, FAR>(c, out, ra + 8u * s, rowa + 4u * s, ga, aa, col, thr, dummy);
        for (; s < c.S; ++s) scan<1, TM, STORE, ARG, STAGE, FAR>(c, out, ra + 8u * s, rowa + 4u * s, ga, aa, col, thr, dummy);
        // a candidate beyond the column's best plus the largest entry cannot win; a column without a finite value
        // keeps nothing alive
#pragma unroll
        for (int j = 0; j < TM; ++j) thr[j] = thr[j] < kInf ? thr[j] + c.tmax : -1;
        uint32_t live[kMaxS / 32];
#pragma unroll
        for (int b = 0; b < kMaxS / 32; ++b) {
            live[b] = 0;
            if (32 * b < c.S) {
                const int n = min(32, c.S - 32 * b);
                int q = 0;
                for (; q + 4 <= n; q += 4) live[b] |= alive<4, TM, FAR>(c, ra + 8u * (32 * b + q), rowa + 4u * (32 * b + q), ga, col, thr) << q;
                for (; q < n; ++q) live[b] |= alive<1, TM, FAR>(c, ra + 8u * (32 * b + q), rowa + 4u * (32 * b + q), ga, col, thr) << q;
            }
        }
        const uint32_t ta = smem_addr(c.tsm + (((l + 1) & 1) ? c.tmat : 0));
        for (int cb = 0; cb < c.S; cb += KC) {
            int acc[KC][TM], arg[ARG ? KC : 1][TM];
#pragma unroll
            for (int k = 0; k < KC; ++k)
#pragma unroll
                for (int j = 0; j < TM; ++j) { acc[k][j] = kInf; if (ARG) arg[k][j] = 255; }
#pragma unroll
            for (int b = 0; b < kMaxS / 32; ++b)
                for (uint32_t m = live[b]; m; m &= m - 1) {
                    const int q = 32 * b + __ffs(m) - 1;
                    Recs<1> r;
                    fetch_recs<1, false, FAR>(c, ra + 8u * q, rowa + 4u * q, r);
                    const uint32_t t0 = ta + (uint32_t)(q * c.SP + cb) * 4u;
                    int v[TM];
                    gather<TM, FAR>(c, ga, r.x[0], r.who[0], col, v);
#pragma unroll
                    for (int j = 0; j < TM; ++j) v[j] = __viaddmin_s32(v[j], r.t[0], kInf);
#pragma unroll
                    for (int w = 0; w < KC / 4; ++w) {
                        const int4 t4 = lds4(t0 + 16u * w);
                        const int t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                        for (int j = 0; j < TM; ++j)
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (ARG) {
                                    const int cand = v[j] + t[u];
                                    if (v[j] < kInf && cand < acc[4 * w + u][j]) { acc[4 * w + u][j] = cand; arg[ARG ? 4 * w + u : 0][j] = q; }
                                } else {
                                    acc[4 * w + u][j] = __viaddmin_s32(v[j], t[u], acc[4 * w + u][j]);
                                }
                            }
                    }
                }
#pragma unroll
            for (int k = 0; k < KC; ++k)
                if (cb + k < c.S) emit<TM, ARG, !STORE && !ARG>(c, l, gn, an, cb + k, colb, lane, acc[k], arg[ARG ? k : 0]);
        }
    }
}

// The last layer hands nothing on: its values go to the table and to C_last.
template <bool STORE, bool ARG, bool STAGE, bool FAR>
__device__ __forceinline__ void last_tile(const Ctx& c, int l, int colb, int lane)
{
    const uint32_t sa = STAGE ? smem_addr(c.stage + (l & 1) * c.S * c.W + colb + lane) : 0u;
    const int slot = c.slot[l & 3], col = colb + lane;
    const uint32_t ra = c.rec + (uint32_t)(slot * c.S2) * 24u, rowa = ra + (uint32_t)c.S2 * 8u, ga = smem_addr(c.g0 + (l & 1) * c.gints + col);
    const uint32_t aa = ARG ? smem_addr(c.a0 + (l & 1) * c.gints + col) : 0u;
    const int colg = c.rank * c.W + colb, m = colg + lane;
    if (colg >= c.m_pitch) return;                             // m_pitch is a multiple of 32: a group exists whole or not at all
    const bool pad = m > c.M;
    auto steps = [&](auto count, int e) {
        constexpr int U = decltype(count)::value;
        Recs<U> r;
        int g[U][1], a[U][1];
        fetch_recs<U, true, ARG || FAR>(c, ra + 8u * e, rowa + 4u * e, r);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            gather<1, FAR>(c, ga, r.x[u], r.who[u], col, g[u]);
            if (ARG) gather_arg<1, FAR>(c, aa, r.x[u], r.who[u], col, a[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int v = pad ? kInf : __viaddmin_s32(g[u][0], r.t[u], kInf);
            if (STAGE) { sts(sa + (uint32_t)r.row[u], v); continue; }
            const size_t row = ((uint32_t)r.row[u] >> 2) + (size_t)m;
            if (STORE) c.C[(size_t)l * c.slice + row] = v;
            c.C_last[row] = v;
            if (ARG) c.A[(size_t)l * c.slice + row] = (uint8_t)(v < kInf ? a[u][0] : 255);
        }
    };
    int e = 0;
    for (; e + 4 <= c.n_all; e += 4) steps(std::integral_constant<int, 4>(), e);
    for (; e < c.n_all; ++e) steps(std::integral_constant<int, 1>(), e);
}

// `n` column groups from group g on, as one tile.
template <int KC, int MAX, bool PRUNE, bool STORE, bool ARG, bool STAGE>
__device__ __forceinline__ void tile_of(const Ctx& c, int l, int g, int n, int lane)
{
    if constexpr (MAX > 1) {
        if (n < MAX) { tile_of<KC, MAX - 1, PRUNE, STORE, ARG, STAGE>(c, l, g, n, lane); return; }
    }
    tile<KC, MAX, PRUNE, STORE, ARG, STAGE, false>(c, l, g * 32, lane);
}

// A warp owns a run of column groups (the warps' runs differ by one group at most) and takes it as one tile, or as
// several of about the same width when it is wider than MAX groups: a record fetched once serves them all.
template <int KC, int MAX, bool PRUNE, bool STORE, bool ARG, bool STAGE>
__device__ __forceinline__ void run_layers(const Ctx& c, int warp, int lane)
{
    const int g0 = c.G * warp / c.NW, g1 = c.G * (warp + 1) / c.NW;
    for (int l = 0; l + 1 < c.Li; ++l) {
        int g = g0;
        if (c.reach[c.slot[l & 3]] <= c.H) {
            for (int left = (g1 - g0 + MAX - 1) / MAX; left > 0; --left) {
                const int n = (g1 - g + left - 1) / left;
                tile_of<KC, MAX, PRUNE, STORE, ARG, STAGE>(c, l, g, n, lane);
                g += n;
            }
        } else {
            for (; g < g1; ++g) tile<KC, 1, PRUNE, STORE, ARG, STAGE, true>(c, l, g * 32, lane);
        }
        send_halo<ARG>(c, l, warp, lane);
        await_halo<STAGE>(c, l, warp);
    }
    if (c.reach[c.slot[(c.Li - 1) & 3]] <= c.H) {
        for (int g = g0; g < g1; ++g) last_tile<STORE, ARG, STAGE, false>(c, c.Li - 1, g * 32, lane);
    } else {
        for (int g = g0; g < g1; ++g) last_tile<STORE, ARG, STAGE, true>(c, c.Li - 1, g * 32, lane);
    }
}

// Cluster c takes instance c (the c-th longest when `sorted`).  Warps 0..NW-1 compute, the last warp fetches the
// layers' mem / time rows (and with one matrix per layer the matrices) ahead and turns them into records.
template <bool STORE, bool ARG, bool STAGE>
__global__ void __launch_bounds__((kMaxWarps + 1) * 32, 1) resident_kernel(const RsArgs a, const __grid_constant__ CUtensorMap map_c,
                                                                           const __grid_constant__ CUtensorMap map_last)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_len[kMaxSortedB], s_twin[2 * kMaxS], s_root[2 * kClassMax];
    __shared__ int s_ccls[kMaxS], s_order[kMaxS + kClassMax], s_csp[4 * (kClassMax + 1)], s_first[kClassMax + 1], s_cnt[kClassMax];
    __shared__ int s_cdelta[16], s_front[4], s_reach[4], s_slot[4], s_inst, s_K[2];
    __shared__ struct { long long sum; int tmax, bad, mmax; } s_part, s_all;
    __shared__ __align__(8) unsigned long long s_bar[2];
    __shared__ int s_late[2];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = (NT >> 5) - 1;
    const int CL = a.CL, rank = CL > 1 ? (int)cluster_rank() : 0, cid = blockIdx.x / CL;
    const int S = a.S, M = a.M, W = a.W, Lmax = a.Lmax, gints = a.gints;

    // ---- shared memory
    int32_t* const g0 = reinterpret_cast<int32_t*>(smem_raw);                              // [2][gints]
    const int tfull = S * a.SP;
    int32_t* const tsm = g0 + 2 * gints;                                                   // [16][16] or [1|2][S][SP]
    const int tints = max(kClassMax * kClassMax, (a.trans_layer ? 2 : 1) * tfull);
    const int S2 = (S + kClassMax + 11) & ~3;                  // a fetch runs up to eight entries ahead
    int32_t* const rec = tsm + tints;                                                      // [4] slots of S2 x (int2, int, int, int2)
    int32_t* const raw = rec + 4 * 6 * S2;                                                 // [4][2][S] mem, time rows as they come
    int32_t* const stage_rows = reinterpret_cast<int32_t*>(smem_raw) + a.stage_at;         // [2][S][W] rows on their way to the table
    uint8_t* const a0 = reinterpret_cast<uint8_t*>(raw + 8 * ((S + 3) & ~3));                           // [2][gints] argmin of the state

    if (blockIdx.x == 0 && tid == 0 && !a.second) a.path[3] = ARG ? 0 : kPathCluster;
    if (a.follow) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");    // the pushing kernel may start beside this one

    // ---- which instance: clusters are dispatched in order, so the longest instances go first
    int i = cid;
    if (a.sorted) {
        for (int j = tid; j < a.B; j += NT) {
            const int v = a.L[j];
            s_len[j] = (v < 1 || v > Lmax) ? 0 : v;
        }
        __syncthreads();
        for (int j = tid; j < a.B; j += NT) {
            const int Lj = s_len[j];
            int before = 0;
            for (int k = 0; k < a.B; ++k) {
                const int Lk = s_len[k];
                before += (Lk > Lj) || (Lk == Lj && k < j);
            }
            if (before == cid) s_inst = j;
        }
        __syncthreads();
        i = s_inst;
    }
    // finished before, or (no room here for an unstructured matrix) found to be one by the probe: nobody in the cluster
    // writes the word before all have read it
    if ((a.second && (a.done[i] & 1)) || (a.probed && a.done[i] == 2)) return;
    const int Li = a.L[i];
    if (Li < 1 || Li > Lmax) {
        if (rank == 0 && tid == 0) { a.status[i] = GALV_STATUS_BAD_INPUT; a.done[i] = 1; }
        return;
    }
    const int32_t* const tq = a.time_q + (size_t)i * Lmax * S;
    const int32_t* const mq = a.mem_q + (size_t)i * Lmax * S;
    const int32_t* const T0 = a.trans_q + (size_t)i * a.trans_inst;

    // ---- validation: the CTAs of the cluster share the layers (and matrices); one matrix per instance is staged whole
    int32_t* const stage = g0;                                 // the state is not in use yet
    const int TP = S | 1;                                       // odd pitch: columns are read without bank conflicts too
    const bool staged = !a.trans_layer && (long long)S * TP <= (long long)2 * gints;
    auto fetch = [&](int l) {
        int32_t* const rm = raw + (l & 3) * 2 * S;
        for (int s = lane; s < S; s += 32) {
            cp_async_4(rm + s, mq + (size_t)l * S + s);
            cp_async_4(rm + S + s, tq + (size_t)l * S + s);
        }
    };
    if (warp == NW) {                                           // the first layers' rows are under way while the rest is looked at
        fetch(0);
        if (Li > 1) fetch(1);
        cp_async_commit();
        if (Li > 2) fetch(2);
        cp_async_commit();
    }
    if (tid == 0) { s_part.sum = 0; s_part.tmax = 0; s_part.bad = 0; s_part.mmax = 0; }
    if (tid == 0) {
        s_late[0] = 0; s_late[1] = kNever;
        mbar_init(smem_addr(&s_bar[0])); mbar_init(smem_addr(&s_bar[1]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 16) s_cdelta[tid] = CL > 1 ? (int)(map_to_rank(smem_addr(g0), (uint32_t)min(tid, CL - 1)) - smem_addr(g0)) : 0;
    __syncthreads();
    {
        long long sum = 0;
        int bad = 0, tmax = 0, mmax = 0;                        // mmax: the largest shift that stays inside the budget
        for (int l = rank * (NW + 1) + warp; l < Li; l += CL * (NW + 1)) {      // a warp per layer: largest time of the layer
            int mx = 0;
            for (int s = lane; s < S; s += 32) {
                const int tv = tq[l * S + s], mv = mq[l * S + s];
                bad |= (tv < 0) | (mv < 0);
                mx = max(mx, tv);
                mmax = max(mmax, mv <= M ? mv : 0);
            }
            mx = __reduce_max_sync(0xffffffffu, mx);
            if (lane == 0) sum += mx;
        }
        if (a.trans_layer) {
            const long long nx = (long long)(Li - 1) * S * S;                     // matrix 0 is unused
            const int32_t* const x = T0 + (size_t)S * S;
#pragma unroll 4
            for (long long k = (long long)rank * NT + tid; k < nx; k += (long long)CL * NT) {
                const int v = x[k];
                bad |= v < 0;
                tmax = max(tmax, v);
            }
        } else {
#pragma unroll 4
            for (int k = tid; k < S * S; k += NT) {
                const int v = T0[k];
                bad |= v < 0;
                tmax = max(tmax, v);
                if (staged) { const int q = k / S; stage[q * TP + k - q * S] = v; }
            }
        }
        tmax = __reduce_max_sync(0xffffffffu, tmax);
        mmax = __reduce_max_sync(0xffffffffu, mmax);
        bad = __any_sync(0xffffffffu, bad != 0);
        if (lane == 0) {
            if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(&s_part.sum), static_cast<unsigned long long>(sum));
            atomicMax(&s_part.tmax, tmax);
            atomicMax(&s_part.mmax, mmax);
            if (bad) atomicOr(&s_part.bad, 1);
        }
    }
    __syncthreads();                                            // the partial results and the staged matrix
    if (CL > 1) cluster_arrive();

    // ---- classes of equal rows and equal columns
    int K = S;                                                  // unstructured unless found otherwise
    if (staged) {
        // the nearest earlier twin of every row (0 .. S-1) and column (S .. 2S-1), compared word by word, a warp each.
        // With the pushing kernel behind this one the first kClassMax + 1 rows first: two of them are equal if there are at
        // most kClassMax classes.  It makes the same test and has started on the instance already if none are.
        // (One copy of the loop: code that runs once is fetched from L2, and its length is what the start takes.)
        auto twins = [&](auto words) -> bool {
            constexpr int N = decltype(words)::value;
            const int probe = a.follow && S > kClassMax ? kClassMax + 1 : 0;
            int x = warp, found = 0;
#pragma unroll 1
            for (int to = probe; ; to = 2 * S) {
#pragma unroll 1
                for (; x < to; x += NW + 1) {
                    const bool row = x < S;
                    const int me = row ? x : x - S, step = row ? TP : 1, word = row ? 1 : TP;      // from one row / column, or word, to the next
                    int w[N];
#pragma unroll
                    for (int j = 0; j < N; ++j) w[j] = lane + 32 * j < S ? stage[me * step + (lane + 32 * j) * word] : 0;
                    int twin = me;
                    for (int o = me - 1; o >= 0; --o) {
                        bool diff = false;
#pragma unroll
                        for (int j = 0; j < N; ++j)
                            if (lane + 32 * j < S) diff |= stage[o * step + (lane + 32 * j) * word] != w[j];
                        if (!__any_sync(0xffffffffu, diff)) { twin = o; break; }
                    }
                    if (lane == 0) s_twin[x] = twin;
                    found |= twin != me;
                }
                if (to == 2 * S) return true;
                if (to && !__syncthreads_or(found)) return false;
            }
        };
        const bool some = S <= 32 ? twins(std::integral_constant<int, 1>()) :
                          S <= 64 ? twins(std::integral_constant<int, 2>()) : twins(std::integral_constant<int, kMaxS / 32>());
        if (!some) {
            if (rank == 0 && tid == 0) a.done[i] = 0;
            if (warp == NW) cp_async_wait<0>();                  // nothing may land in shared memory that is no longer ours
            if (CL > 1) cluster_wait();
            return;
        }
        __syncthreads();
        // a class is the twins that lead back to the same first; classes are numbered in the order of their firsts, and
        // the strategies put into the order of their rows' classes: one warp for the rows, one for the columns
        if (warp < 2) {
            volatile int* const tw = s_twin + (warp == 0 ? 0 : S);
            for (int span = 1; span < S; span <<= 1) {          // pointer jumping: any value read is an ancestor
                for (int s = lane; s < S; s += 32) tw[s] = tw[tw[s]];
                __syncwarp();
            }
            unsigned first[kMaxS / 32];                         // which strategies open a class
            int k = 0, cls[kMaxS / 32];
#pragma unroll
            for (int j = 0; j < kMaxS / 32; ++j) {
                const int s = lane + 32 * j;
                first[j] = __ballot_sync(0xffffffffu, s < S && tw[s] == s);
                k += __popc(first[j]);
            }
#pragma unroll
            for (int j = 0; j < kMaxS / 32; ++j) {
                const int s = lane + 32 * j, root = s < S ? tw[s] : 0;
                int n = 0;
#pragma unroll
                for (int q = 0; q < kMaxS / 32; ++q) n += __popc(first[q] & (q < (root >> 5) ? ~0u : q == (root >> 5) ? (1u << (root & 31)) - 1u : 0u));
                cls[j] = s < S ? n : -1;
                if (s < S && warp == 1) s_ccls[s] = n;
                if (s < S && root == s && n < kClassMax) s_root[warp * kClassMax + n] = s;
            }
            if (lane == 0) s_K[warp] = k;
            if (warp == 0 && k <= kClassMax) {
                // ascending inside a class; a class of an odd number has its last one twice
                int at = 0;
                for (int q = 0; q < k; ++q) {
                    int n = 0;
#pragma unroll
                    for (int j = 0; j < kMaxS / 32; ++j) {
                        const unsigned in = __ballot_sync(0xffffffffu, cls[j] == q);
                        const int pos = at + n + __popc(in & ((1u << lane) - 1u));
                        if (cls[j] == q) s_order[pos + 1] = lane + 32 * j;             // the next entry's owner overwrites it, if there is one
                        __syncwarp();
                        if (cls[j] == q) s_order[pos] = lane + 32 * j;
                        __syncwarp();
                        n += __popc(in);
                    }
                    if (lane == 0) { s_first[q] = at; s_cnt[q] = n; }
                    at += (n + 1) & ~1;
                }
                if (lane == 0) s_first[k] = at;
            }
        }
    }
    if (CL > 1) cluster_wait();                                 // everybody's partial results
    if (warp == 0) {
        long long sum = 0;
        int tmax = 0, bad = 0, mmax = 0;
        if (CL == 1) {
            sum = s_part.sum; tmax = s_part.tmax; bad = s_part.bad; mmax = s_part.mmax;
        } else {
            if (lane < CL) {
                const uint32_t p = map_to_rank(smem_addr(&s_part), (uint32_t)lane);
                sum = (long long)(((unsigned long long)(uint32_t)ld_cluster(p + 4) << 32) | (uint32_t)ld_cluster(p));
                tmax = ld_cluster(p + 8);
                bad = ld_cluster(p + 12);
                mmax = ld_cluster(p + 16);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            tmax = __reduce_max_sync(0xffffffffu, tmax);
            mmax = __reduce_max_sync(0xffffffffu, mmax);
            bad = __any_sync(0xffffffffu, bad != 0);
        }
        if (lane == 0) { s_all.sum = sum; s_all.tmax = tmax; s_all.bad = bad; s_all.mmax = mmax; }
    }
    __syncthreads();
    if (staged) K = max(s_K[0], s_K[1]);
    const bool classes = staged && K <= kClassMax && s_K[1] * W <= gints;
    const bool dense = !classes && a.SP > 0 && S * W <= gints;
    const int Kr = classes ? s_K[0] : S, Kc = classes ? s_K[1] : S;
    if (classes) {
        for (int x = tid; x < kClassMax * kClassMax; x += NT) {
            const int k = x / kClassMax, q = x - k * kClassMax;
            tsm[x] = k < Kr && q < Kc ? stage[s_root[k] * TP + s_root[kClassMax + q]] : 0;
        }
    } else if (dense) {
        for (int s = tid; s < S; s += NT) { s_order[s] = s; s_ccls[s] = s; }
        // the matrix paid between layers 0 and 1; with one matrix per layer, matrix l sits in buffer l & 1
        const int32_t* const T = T0 + (a.trans_layer ? a.trans_layer : 0);
        int32_t* const dst = tsm + (a.trans_layer ? tfull : 0);
        for (int x = tid; x < tfull; x += NT) {
            const int r = x / a.SP, s = x - r * a.SP;
            const int v = (s < S && Li > 1) ? (staged ? stage[r * TP + s] : T[r * S + s]) : 0;
            dst[x] = v;
            if (a.trans_layer) tsm[x] = 0;                      // pad columns of the other buffer stay 0
        }
    }
    int st = 0;
    __syncthreads();                                            // s_all, classes; the staged matrix is no longer read
    if (s_all.bad) st = GALV_STATUS_BAD_INPUT;
    else if (s_all.sum + (long long)(Li - 1) * s_all.tmax >= (long long)kInf) st = GALV_STATUS_OVERFLOW_RISK;
    const bool run = st == 0 && (classes || dense) && !(a.follow && K > a.k_max);

    // The halo: columns left of this CTA's own that its gathers reach, as many as the largest shift asks for or as fit;
    // a multiple of 32.  Below column 0 it holds +inf.
    const int H = max(0, min((s_all.mmax + 31) & ~31, (gints / Kc - W) & ~31)), P = W + H;

    if (rank == 0 && tid == 0) { a.status[i] = st; a.done[i] = st != 0 || run; }

    const int n_all = classes ? s_first[Kr] : S;
    const bool strict = s_all.mmax > H;                         // some shift reaches beyond the halo
    // ---- layer 0 gathers from an all-zero state: C[0] = time where mem fits
    auto prepare = [&](int l, int base) -> int {                // records of layer l by one warp; returns the new frontier
        const int32_t* const rm = raw + (l & 3) * 2 * S;
        // a layer with the rows of one of the two before it takes that one's records
        int slot = -1, least = M + 1;
        for (int back = 1; back <= 2 && back <= l && slot < 0; ++back) {
            const int32_t* const ro = raw + ((l - back) & 3) * 2 * S;
            int diff = 0;
            for (int x = lane; x < 2 * S; x += 32) diff |= rm[x] != ro[x];
            if (!__any_sync(0xffffffffu, diff)) slot = s_slot[(l - back) & 3];
        }
        if (slot < 0) {
            // not one of the three layers before: the oldest may still be on its way to the table
            unsigned used = 0;
            for (int back = 1; back <= 3 && back <= l; ++back) used |= 1u << s_slot[(l - back) & 3];
            slot = __ffs(~used) - 1;
            int32_t* const rs = rec + slot * 6 * S2;
            int most = 0;
            for (int e = lane; e < n_all; e += 32) {
                const int s = s_order[e];
                const int mem = rm[s];
                const bool fits = mem <= M;                     // else +inf everywhere: no shift, time +inf
                const int shift = fits ? mem : 0;
                reinterpret_cast<int2*>(rs)[e] = make_int2((s_ccls[s] * P + H - shift) * 4, fits ? rm[S + s] : kInf);
                rs[2 * S2 + e] = s * (STAGE ? W : a.m_pitch) * 4;
                rs[3 * S2 + e] = shift | (s << 24);
                most = max(most, shift);
            }
            if (lane < 8) {                                     // what a fetch ahead of the end finds: a cell that exists
                reinterpret_cast<int2*>(rs)[n_all + lane] = make_int2(0, kInf);
                rs[2 * S2 + n_all + lane] = 0;
            }
            most = __reduce_max_sync(0xffffffffu, most);
            if (lane == 0) s_reach[slot] = most;
            if (classes && !STORE && !ARG) {
                // the strategies that can matter, class by class
                __syncwarp();
                int2* const keep = reinterpret_cast<int2*>(rs + 4 * S2);
                const int2* const all = reinterpret_cast<const int2*>(rs);
                int at = 0;
                for (int k = 0; k < Kr; ++k) {
                    if (lane == 0) s_csp[slot * (kClassMax + 1) + k] = at;
                    const int first = s_first[k], n = s_cnt[k];
                    int2 lastkept = make_int2(0, 0);
                    int kept = 0;
                    for (int b = 0; b < n; b += 32) {
                        const int p = b + lane;
                        bool in = p < n;
                        int2 me = make_int2(0, kInf);
                        if (in) {
                            me = all[first + p];
                            in = me.y < kInf;
                            const int mm = rm[s_order[first + p]], mc = s_ccls[s_order[first + p]];
                            for (int q = 0; q < n && in; ++q) {
                                const int so = s_order[first + q];
                                const int om = rm[so], ot = rm[S + so];
                                if (s_ccls[so] == mc && om <= mm && ot <= me.y && (om < mm || ot < me.y || q < p)) in = false;
                            }
                        }
                        const unsigned b1 = __ballot_sync(0xffffffffu, in);
                        if (in) keep[at + kept + __popc(b1 & ((1u << lane) - 1))] = me;
                        if (b1) {
                            const int src = 31 - __clz(b1);
                            lastkept.x = __shfl_sync(0xffffffffu, me.x, src);
                            lastkept.y = __shfl_sync(0xffffffffu, me.y, src);
                        }
                        kept += __popc(b1);
                    }
                    if ((kept & 1) && lane == 0) keep[at + kept] = lastkept;
                    at += (kept + 1) & ~1;
                }
                if (lane == 0) s_csp[slot * (kClassMax + 1) + Kr] = at;
                if (lane < 8) keep[at + lane] = make_int2(0, kInf);
            }
        }
        for (int s = lane; s < S; s += 32) least = min(least, rm[s]);
        least = __reduce_min_sync(0xffffffffu, least);
        const int f = min(base + least, M + 1);
        if (lane == 0) { s_front[l & 3] = f; s_slot[l & 3] = slot; }
        __syncwarp();
        return f;
    };
    int front = 0;
    if (run) {
        if (warp == NW) {
            cp_async_wait<1>();
            __syncwarp();
            front = prepare(0, 0);
            if (Li > 1) front = prepare(1, front);
        } else {
            for (int k = 0; k < Kc; ++k)
                for (int x = tid; x < P; x += NW * 32) {
                    g0[k * P + x] = rank * W + x >= H ? 0 : kInf;           // column rank*W + x - H
                    if (x < H) g0[gints + k * P + x] = kInf;
                    if (ARG) {
                        a0[k * P + x] = 255;
                        if (x < H) a0[gints + k * P + x] = 255;
                    }
                }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");            // bulk copies write over the halo's initial values
    whole_barrier(CL);                                          // also: nobody leaves while its partial sums are being read
    if (!run) {
        if (warp == NW) cp_async_wait<0>();                     // nothing may land in shared memory that is no longer ours
        return;
    }

    Ctx c;
    c.S = S; c.M = M; c.W = W; c.H = H; c.P = P; c.G = W / 32; c.CL = CL; c.rank = rank; c.Li = Li; c.m_pitch = a.m_pitch; c.Kr = Kr; c.Kc = Kc;
    c.tmax = s_all.tmax; c.SP = a.SP; c.NW = NW; c.gints = gints;
    c.g0 = g0; c.a0 = a0; c.stage = stage_rows; c.rec = smem_addr(rec); c.S2 = S2; c.n_all = n_all; c.front = s_front; c.reach = s_reach; c.tsm = tsm; c.tmat = a.trans_layer ? tfull : 0;
    c.cs = s_first; c.csp = s_csp; c.slot = s_slot; c.cdelta = s_cdelta;
    c.slice = (size_t)S * a.m_pitch;
    c.C = STORE ? a.C + (size_t)i * Lmax * c.slice : nullptr;
    c.states = a.states ? a.states + (size_t)i * Lmax * c.slice : nullptr;
    if (a.states && rank == 0)
        for (int s = tid; s < S; s += NT) a.map[(size_t)i * S + s] = s_ccls[s];
    c.A = ARG ? a.A + (size_t)i * Lmax * c.slice : nullptr;
    c.C_last = a.C_last + (size_t)i * c.slice;
    c.bars = smem_addr(&s_bar[0]);
    c.halo_bytes = (uint32_t)(Kc * min(H, rank * W)) * (ARG ? 5u : 4u);
    c.strict = strict;
    c.late = s_late;
    if (CL > 1 && !c.strict) cluster_arrive();                  // nobody has read anything yet: the first copies may come
    if (warp == NW) {
        // ---------------------------------------------------------------- service warp
        for (int l = 0; l + 1 < Li; ++l) {
            if (l + 3 < Li) fetch(l + 3);
            cp_async_commit();
            if (a.trans_layer && l + 2 < Li) {                  // matrix l + 1 is in use in this layer
                const int32_t* const T = T0 + (size_t)(l + 2) * a.trans_layer;
                int32_t* const dst = tsm + ((l & 1) ? tfull : 0);
                for (int x = lane; x < S * S; x += 32) {
                    const int r = x / S, s = x - r * S;
                    cp_async_4(dst + r * a.SP + s, T + x);
                }
            }
            cp_async_commit();
            if (l + 2 < Li) {
                cp_async_wait<2>();                             // the rows of layer l + 2, asked for a layer ago
                __syncwarp();
                front = prepare(l + 2, front);
            }
            if (a.trans_layer) cp_async_wait<0>();
            if (STAGE) {
                if (lane == 0) bulk_wait_read();                // layer l - 1 has left its buffer, which layer l + 1 fills
                __syncwarp();
            }
            const bool on = *(volatile int*)(c.late + 1) > l - 2;            // see send_halo
            send_halo<ARG>(c, l, warp, lane, on && !(a.withhold && l == 0 && rank == 0));
            if (STAGE && lane == 0) {
                if (CL == 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                tensor_store_3d(&map_c, c.stage + (l & 1) * S * W, rank * (W / 32), (i * Lmax + l) * S);
                bulk_commit();
            }
            await_halo_service<STAGE>(c, l, lane, on);
        }
        if (STAGE) {
            if (lane == 0) bulk_wait_read();
            cta_barrier();                                      // the last layer's rows are collected
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                const int l = Li - 1;
                tensor_store_3d(&map_c, c.stage + (l & 1) * S * W, rank * (W / 32), (i * Lmax + l) * S);
                tensor_store_3d(&map_last, c.stage + (l & 1) * S * W, rank * (W / 32), i * S);
                bulk_commit();
                bulk_wait_all();
            }
            __syncwarp();
        }
    } else {
        if (classes) {
            if (K <= 4) run_layers<4, ARG ? 2 : STAGE ? 2 : STORE ? 6 : 5, false, STORE, ARG, STAGE>(c, warp, lane);
            else if (K <= 8) run_layers<8, ARG ? 2 : STAGE ? 2 : STORE ? 6 : 5, false, STORE, ARG, STAGE>(c, warp, lane);
            else run_layers<16, ARG ? 1 : 2, false, STORE, ARG, STAGE>(c, warp, lane);
        } else {
            run_layers<32, ARG ? 1 : 2, true, STORE, ARG, STAGE>(c, warp, lane);
        }
        if (STAGE) cta_barrier();                               // the last layer's rows are collected
    }
    if (CL > 1) {
        if (!c.strict) cluster_wait();
        if (s_late[1] != kNever && c.halo_bytes && warp == 0)    // copies of these two layers may still land here
            for (int l = s_late[1]; l <= s_late[1] + 1 && l + 1 < Li; ++l)
                for (int polls = 0; polls < kWaitPolls && !mbar_try(c.bars + 8u * (l & 1), (uint32_t)(l >> 1) & 1u); ++polls) { }
        whole_barrier(CL);                                      // nobody's shared memory goes away while it is being read or written
        if (s_late[0] && tid == 0) atomicOr(reinterpret_cast<int*>(a.status + i), GALV_STATUS_TIMEOUT);
    }
}

// Which matrices are worth the resident kernel's look: of kClassMax + 1 rows two are equal if there are at most kClassMax
// classes.  done[i] = 2: no two of the first rows are.  Not for matrices of fewer rows: those always have few enough classes
// (and the rows it reads are not there).  A kernel of a few hundred instructions, as it is latency alone: the
// same look inside the resident kernel cost a batch it turns away 15 us, most of them spent on fetching its code.
__global__ void __launch_bounds__(256) probe_kernel(int B, int S, int after_solo, const int32_t* __restrict__ trans_q, long long trans_inst, int32_t* __restrict__ done)
{
    constexpr int R = kClassMax + 1;
    __shared__ int32_t rows[R * kMaxS];
    __shared__ int s_pair;
    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    if (after_solo && done[i] == 3) return;
    if (S < R) {                                                // a matrix has S rows
        if (tid == 0) done[i] = 0;
        return;
    }
    const int32_t* const T = trans_q + (size_t)i * trans_inst;
    if (tid == 0) s_pair = 0;
    for (int k = tid; k < R * S; k += 256) rows[k] = T[k];
    __syncthreads();
    bool equal = false;                                         // the vote's answer: the same in all lanes, as the next vote needs it
    for (int x = tid >> 5; x < R * R && !equal; x += 8) {
        const int p = x / R, q = x - p * R;
        if (p >= q) continue;
        bool diff = false;
        for (int s = lane; s < S; s += 32) diff |= rows[p * S + s] != rows[q * S + s];
        equal = !__any_sync(0xffffffffu, diff);
    }
    if (equal && lane == 0) s_pair = 1;
    __syncthreads();
    if (tid == 0) done[i] = s_pair ? 0 : 2;
}

// ---------------------------------------------------------------- host side

typedef void (*RsKernel)(const RsArgs, const CUtensorMap, const CUtensorMap);
RsKernel kernel_of(bool store, bool arg, bool stage)
{
    if (stage) return resident_kernel<true, false, true>;
    return store ? (arg ? resident_kernel<true, true, false> : resident_kernel<true, false, false>)
                 : (arg ? resident_kernel<false, true, false> : resident_kernel<false, false, false>);
}

cudaError_t launch_resident(RsKernel k, const RsArgs& a, const RsPlan& p, const CUtensorMap& mc, const CUtensorMap& ml, cudaStream_t st, int* max_clusters)
{
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(a.B * p.cl));
    cfg.blockDim = dim3((unsigned)((p.nw + 1) * 32));
    cfg.dynamicSmemBytes = (size_t)p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (max_clusters) return cudaOccupancyMaxActiveClusters(max_clusters, k, &cfg);
    return cudaLaunchKernelEx(&cfg, k, a, mc, ml);
}

// Clusters of this plan's size and resources the device can hold at once (asked once per kind of launch).
int max_active_clusters(const galv_ctx* ctx, const RsPlan& p, bool store, bool arg)
{
    static std::map<unsigned long long, int> cache;          // shared by all contexts of the process
    static std::mutex cache_mutex;
    std::lock_guard<std::mutex> lock(cache_mutex);
    const unsigned long long key = ((unsigned long long)ctx->device << 48) | ((unsigned long long)p.cl << 40) | ((unsigned long long)p.stage << 38) | ((unsigned long long)store << 37) |
                                   ((unsigned long long)arg << 36) | ((unsigned long long)p.nw << 28) | (unsigned long long)((p.smem + 1023) / 1024);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    RsArgs a{};
    a.B = 1;
    int n = 0;
    CUtensorMap m{};
    if (launch_resident(kernel_of(store, arg, p.stage), a, p, m, m, nullptr, &n) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
    cache[key] = n;
    return n;
}

// Shared memory of a launch beside its state.
long long fixed_smem(const galv_shape* sh, bool dense)
{
    const int S = sh->S, SP = (S + 3) & ~3;
    const long long t = dense ? (long long)S * SP * ((sh->flags & GALV_TRANS_PER_LAYER) ? 2 : 1) : 0;
    return (t > kClassMax * kClassMax ? t : kClassMax * kClassMax) * 4 + (long long)4 * 24 * ((S + kClassMax + 11) & ~3) + (long long)8 * SP * 4 + 256;
}

// The best cluster size for a state of `rows` rows at least; false when none fits.
// (halo_fits: with room for the shifts to be expected; rounds: of clusters that the batch takes)
bool best_plan(const galv_ctx* ctx, const galv_shape* sh, int rows, bool dense, RsPlan* out, double* est)
{
    const int S = sh->S, Gt = sh->m_pitch / 32;
    const bool store = (sh->flags & GALV_STORE_C_FULL) != 0, arg = (sh->flags & GALV_STORE_ARGMIN) != 0;
    const int want = (sh->flags >> 16) & 31;                  // GALV_CLUSTER_SIZE(n) beside GALV_KERNEL_RESIDENT: only clusters of n CTAs
    const int per_word = arg ? 10 : 8;                        // two buffers of words, with argmin bytes beside
    const long long words = ((long long)ctx->smem_optin - kStaticSmem - fixed_smem(sh, dense)) / per_word;
    // halo to plan for: a few times what an even share of the budget gives a layer, and what large layers of the analytic
    // models ask for (a fifth of 2880 columns, 600 of 8192); beyond it a layer takes the slow way
    long long halo = 4ll * sh->M / sh->Lmax;
    if (!dense && halo < (sh->M / 5 < 600 ? sh->M / 5 : 600)) halo = sh->M / 5 < 600 ? sh->M / 5 : 600;
    if (halo < 64) halo = 64;
    if (halo > sh->M) halo = sh->M;
    bool found = false;
    for (int cl = 1; cl <= ctx->max_resident; ++cl) {
        if (want && cl != want) continue;
        const int g = (Gt + cl - 1) / cl;
        if (cl > 1 && (g < 2 || g * (cl - 1) >= Gt)) continue;      // no CTA without columns
        const int w = g * 32;
        RsPlan p;
        std::memset(&p, 0, sizeof(p));
        p.cl = cl; p.w = w; p.dense = dense;
        p.nw = g < kMaxWarps ? g : kMaxWarps;
        // rows collected in shared memory where there is room for them beside the state (a tensor box has 256 entries a
        // side at most) and where a layer is a chain of latencies rather than a stream of stores; room for shifts of a third
        // of the budget comes first (one instance of 50 layers whose shifts pass the halo: 436 us)
        const long long collected = (long long)2 * S * w * 4;
        p.stage = store && !arg && g <= 2 * kMaxWarps && (long long)rows * (w + (cl > 1 ? (halo > sh->M / 3 ? halo : sh->M / 3) : 0)) * per_word + collected <= words * per_word &&
                  (long long)sh->B * sh->Lmax * S < (1ll << 31);
        const long long room = p.stage ? words - collected / per_word : words;
        long long gi = (long long)(dense && S > kClassMax ? S : kClassMax) * (w + ((sh->M + 32) & ~31));    // all that could be used
        if (gi > room) gi = room;
        p.gints = (int)(gi & ~31ll);
        if ((long long)rows * w > p.gints) continue;
        p.smem = (int)(p.gints * (long long)per_word + fixed_smem(sh, dense));
        p.stage_at = (p.smem + 127) / 128 * 32;
        if (p.stage) p.smem = p.stage_at * 4 + (int)collected;
        const int slots = max_active_clusters(ctx, p, store, arg);
        if (slots < 1) continue;
        // SM cycles a layer, fitted on B200: the columns' work, issued at about one instruction a clock and scheduler
        // (with the stores 4.7 clocks a 128-byte line), or one warp's walk over the strategies of its widest tile at four
        // to five clocks an instruction, whichever is longer, and what a layer costs at any size.
        const double width = (g + p.nw - 1) / p.nw;            // column groups of the busiest warp
        const double work = g * (store ? S * 4.7 + 60.0 : S * 1.15 + 20.0);
        const double chain = S * (40.0 + 22.0 * width) + 400.0;
        double t = work > chain ? work : chain;
        if (store && !p.stage) t += S * 10.0;                  // loads wait behind stores
        t += cl == 1 ? 200.0 : (cl > 8 ? 1250.0 : 1100.0);
        const double share = (double)(sh->B < slots ? sh->B : slots) * cl / ctx->num_sms;      // several CTAs on an SM share its issue slots
        if (share > 1.0) t *= share;
        // layers with shifts beyond the halo are gathered four strategies and one column group at a time, at about the
        // latency of another CTA's memory
        p.halo_fits = cl == 1 || (long long)rows * (w + halo) <= p.gints;
        if (!p.halo_fits) t += S * width * 300.0;
        p.rounds = (sh->B + slots - 1) / slots;
        t *= p.rounds > 3 ? (double)sh->B / slots + 0.5 : p.rounds;          // ragged batches fill the last round
        // Of two sizes that come out about the same the finer one: ragged batches, whose lengths the host does not know,
        // fill the SMs better with it (64 instances of 1 to 96 layers: 0.79 ms on clusters of 2, 0.51 on clusters of 4;
        // with 96 layers each 0.79 and 0.94).
        if (!found || t < *est * (out->rounds == 1 && p.rounds <= 2 && sh->B > 1 ? 1.12 : 1.0)) {
            found = true;
            *est = t < *est || *est == 0.0 ? t : *est;
            p.sorted = sh->B > slots && sh->B <= kMaxSortedB;
            *out = p;
        }
    }
    return found;
}

}  // namespace

int galv_resident_plan(galv_ctx* ctx, const galv_shape* sh, const ClPlan* pushing, RsPlan plans[2])
{
    if (sh->flags & (GALV_KERNEL_REFERENCE | GALV_KERNEL_PER_LAYER | GALV_KERNEL_NO_CLUSTER)) return 0;
    if ((sh->flags & GALV_DEBUG_WITHHOLD_LOAD) && !(sh->flags & GALV_KERNEL_RESIDENT)) return 0;
    if (sh->S > kMaxS || (long long)sh->S * sh->m_pitch >= (1ll << 29)) return 0;      // row offsets are 32-bit
    if (ctx->plan_valid && std::memcmp(&ctx->plan_shape, sh, sizeof(*sh)) == 0) {       // the shape of the last call
        plans[0] = ctx->plans[0]; plans[1] = ctx->plans[1];
        return ctx->plan_launches;
    }
    double td = 0.0, tc = 0.0;
    int n = 0;
    const bool forced = (sh->flags & GALV_KERNEL_RESIDENT) != 0;
    const bool arg = (sh->flags & GALV_STORE_ARGMIN) != 0;
    // Unstructured matrices, measured on 48 layers of 2048 columns: S = 32, 16 instances 238 us here against 304 in the
    // pushing cluster kernel; S = 64 on 4000 columns 1.3 ms against 0.69 (its rows leave no room for the halo); 74
    // instances, which take two rounds, 0.77 ms against 0.49 in the tiled kernels without the dominated rows.  With an
    // argmin table, where only the tiled kernels compete, one instance 0.27 against 0.78 ms.
    bool d = (sh->S <= 32 || arg || forced) && best_plan(ctx, sh, sh->S, true, &plans[1], &td);
    if (d && !forced) d = plans[1].halo_fits && plans[1].rounds == 1;
    const bool c = !(sh->flags & GALV_TRANS_PER_LAYER) && sh->S > 8 && best_plan(ctx, sh, sh->S < 9 ? sh->S : 9, false, &plans[0], &tc);
    // Where the pushing kernel's clusters find room beside this one's, a state of S rows has to be worth it: about 260 cycles a
    // layer, strategy and column group (40 layers, 2880 columns, one instance, pushing / dense: S = 20 142 / 162 us,
    // S = 32 172 / 201).  Up to 16 strategies are classes whatever the matrix: k_max sees to those.  Without that room it would
    // start behind this kernel and cost structured batches 5 us (12 of S = 24: 99 / 106).
    if (d && !forced && c && pushing && sh->B * (plans[0].cl + pushing->cl) <= ctx->num_sms) {
        const int g = plans[1].w / 32, width = (g + plans[1].nw - 1) / plans[1].nw;
        d = sh->S > kClassMax && 1600.0 + 260.0 * sh->S * width <= 0.9 * pushing->est;
    }
    plans[0].est = tc; plans[1].est = td;
    // a launch that takes every instance spares the ones after it, which find nothing to do (20 us, 40 thousand cycles)
    if (d && (!c || forced || td * sh->Lmax <= tc * sh->Lmax * 1.05 + 40000.0)) { plans[0] = plans[1]; n = 1; }
    else if (c) n = d ? 2 : 1;
    if (c && n == 1 && !plans[0].dense && pushing) {
        // The pushing kernel's time does not depend on classes; here one costs about 400 cycles a layer and column group.
        // 40 layers, 2880 columns, one instance, pushing / 8 / 12 / 16 classes: S = 16 115 / 101 / 140 / 169 us,
        // S = 24 152 / 133 / 146 / 179, S = 48 268 / 162 / 196 / 237; 30 instances, pushing / 16: S = 16 187 / 257.
        const double width = plans[0].w / 32.0 / plans[0].nw, k = (0.9 * pushing->est - 1600.0 - 30.0 * (sh->S - 16)) / (400.0 * width);
        plans[0].follow = 1;
        plans[0].k_max = k < 8.0 ? 8 : k > kClassMax ? kClassMax : (int)k;
    }
    ctx->plan_shape = *sh; ctx->plans[0] = plans[0]; ctx->plans[1] = plans[1]; ctx->plan_launches = n; ctx->plan_valid = 1;
    return n;
}

cudaError_t galv_resident_configure(galv_ctx* ctx)
{
    ctx->max_resident = 16;                                     // beyond the portable 8 where the device allows it
    for (int k = 0; k < 5; ++k) {
        const RsKernel f = kernel_of(k & 1, (k & 2) != 0, k == 4);
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - kStaticSmem);
        if (e != cudaSuccess) return e;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) { (void)cudaGetLastError(); ctx->max_resident = 8; }
    }
    return cudaSuccess;
}

bool galv_probe_applies(const DpArgs& d) { return d.S > kClassMax && d.S <= kMaxS; }

void galv_probe_matrices(const DpArgs& d, cudaStream_t st) { probe_kernel<<<d.B, 256, 0, st>>>(d.B, d.S, d.after_solo, d.trans_q, d.trans_inst, d.done); }

cudaError_t galv_resident_launch(const RsPlan& p, int second, const DpArgs& d, cudaStream_t st)
{
    RsArgs a;
    a.B = d.B; a.Lmax = d.Lmax; a.S = d.S; a.M = d.M; a.m_pitch = d.m_pitch;
    a.CL = p.cl; a.W = p.w; a.gints = p.gints; a.sorted = p.sorted; a.second = second; a.withhold = d.withhold;
    a.follow = p.follow; a.k_max = p.k_max;
    a.probed = !p.dense && galv_probe_applies(d) && second == d.after_solo && !p.follow;       // the first launch of this kernel
    if (a.probed) galv_probe_matrices(d, st);
    a.SP = p.dense ? (d.S + 3) & ~3 : 0;                       // rows are read as int4, 32 entries at a time: what lies beyond a row is never kept
    a.L = d.L; a.time_q = d.time_q; a.mem_q = d.mem_q; a.trans_q = d.trans_q;
    a.trans_inst = d.trans_inst; a.trans_layer = d.trans_layer;
    const bool lean = d.lean_map != nullptr;
    a.C = lean ? nullptr : d.C; a.states = lean ? d.C : nullptr; a.map = d.lean_map;
    a.A = d.A; a.C_last = d.C_last; a.status = d.status; a.path = d.err; a.done = d.done;
    a.stage_at = p.stage_at;
    CUtensorMap mc, ml;
    std::memset(&mc, 0, sizeof(mc));
    std::memset(&ml, 0, sizeof(ml));
    if (p.stage) {
        cudaError_t e = galv_encode_table_3d(&ml, d.C_last, (size_t)d.B * d.S, d.m_pitch, d.S, p.w / 32);
        if (e == cudaSuccess) e = galv_encode_table_3d(&mc, d.C, (size_t)d.B * d.Lmax * d.S, d.m_pitch, d.S, p.w / 32);
        if (e != cudaSuccess) return e;
    }
    return launch_resident(kernel_of(a.C != nullptr, d.A != nullptr, p.stage), a, p, mc, ml, st, nullptr);
}
