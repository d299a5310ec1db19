// The whole recurrence of one instance on ONE SM: the state between two layers sits in its shared memory.
//
//   C[l][m][s] = time(l,s) + G[l][m - mem(l,s)][s],   G[l][m][s] = min_{s'} ( C[l-1][m][s'] + trans(s',s) )
//
// (Section 3 of the paper: dynamic-programming search over a performance model; Sections 3-4: it runs again while
// the job runs.)
//
// What makes an SM enough, and most of the arithmetic unnecessary:
//  - G has one row per DISTINCT COLUMN of the transition matrix (7 among the 64 strategies of a heterogeneous stack); a
//    matrix without such structure keeps all S rows.
//  - A column's rows lie within the largest transition entry of its best C: a base per column and 16-bit differences (32-bit
//    ones where the entries are larger).  8192 columns of 7 rows are 148 KB, 2048 columns of 32 rows 139 KB.
//  - C[l][m] is read at m - mem <= m only.  Taken from the highest columns down, a layer's new state can lie where the old
//    one was: one copy, no second buffer.
//  - C does not rise with m.  So a strategy's value at a tile's last column bounds it from below all over the tile, its value
//    at the first column from above: two cells a strategy say that it can neither win nor tie anywhere in the tile, nor come
//    within a transition entry of what wins.  A lane looks at a strategy, a warp at 32 of them; one or two of 64 pass on the
//    analytic models (tiles of 160 columns), three of 32 on measured tables whose transitions are a tenth of the times (tiles of 32),
//    and only those are relaxed.
//    Where they are of one row class k, G is base + T[k][.]: rows that hold T[k][.] already are left as they are.
//
// Taken where no table is written: optima, and the states that the host entry point's walk wants.  128 instances of 160 layers, 64
// strategies, 8192 columns, optima: 2976 us in the resident kernel, 1171 here; host entry point 3525 / 2078.  A step of tiles takes 2300
// cycles, latencies of its test, its walk and its writes in turn; one with the edge of the feasible region in it 5000.
//
// How many strategies pass depends on the tables: with times that lie close together, or transitions as large as the times, most of
// them do, and the kernels that relax every row of a register tile are several times as fast (40 instances of 40 layers, S = 64 of 4
// classes, 4000 columns, transitions up to a tenth / half / twice the median time: 480 / 975 / 1387 us here, 400 in the resident
// kernel).  So a batch is searched here only where a guess of that number (guess_kernel) says that it costs less.

#include <cstring>
#include <type_traits>

#include "galv_internal.h"

namespace {

constexpr uint32_t kInf = GALV_INF;
constexpr int kMaxWarps = 15;             // compute warps; with the service warp four a scheduler, of 128 registers
constexpr int kMaxSorted = 512;           // instances whose lengths fit the scratch below
constexpr int kMaxS = 128;
constexpr int kDenseMax = 64;             // rows of an unstructured state
constexpr int kClassMax = kResidentClassMax;
constexpr int kMaxTiles = 512;
constexpr int kStaticSmem = 7168;         // the kernel's static shared memory, rounded up
constexpr int kBatch = 8;                 // rows a warp writes at a time

struct SoArgs {
    int B, Lmax, S, M, m_pitch;
    int NW;            // compute warps
    int room;          // bytes for the state
    int mats;          // words of the transition matrices in shared memory
    int sorted;        // CTA c takes the c-th longest instance
    int dense;         // unstructured matrices are searched here (else left to the kernels behind)
    int packed;        // packed relaxations are allowed
    int certain;       // nothing is left to the kernels behind
    int guessed;       // `guess` holds the verdict on the batch; 0: every instance that fits is searched
    const float2* guess;
    const int32_t* L;
    const int32_t* time_q;
    const int32_t* mem_q;
    const int32_t* trans_q;
    long long trans_inst, trans_layer;
    int32_t* C_last;
    uint32_t* states;  // in the table's place, when nobody sees it: the states between the layers, [Lmax][1 + words][m_pitch] per instance; or NULL
    int32_t* map;      // [B][S] with `states`: state row of each strategy, kStateHalf or kStateWord added
    int32_t* status;
    int32_t* path;     // [4] device flags of the search; [3]: kernel that ran
    int32_t* done;     // [B] 3: this instance needs nothing more, 0: it does
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// Shared memory through 32-bit addresses, in the order written: loads in batches, so that a warp waits once for several.
template <int OFF>
__device__ __forceinline__ uint32_t lds(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
// How differences are kept.  kPacked, kHalf: 16 bits, rows 2p and 2p + 1 in the halves of a word (up to 65535); kPacked: up to
// 32767, so that a difference and a transition entry add up in 16 bits, and two rows are relaxed by one instruction.  kWord: 32 bits.
enum Form { kPacked, kHalf, kWord };
template <int F, int OFF>
__device__ __forceinline__ uint32_t ldd(uint32_t a) {
    uint32_t v;
    if constexpr (F != kWord) asm volatile("ld.shared.u16 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    else asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
__device__ __forceinline__ int4 lds4(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void cta_barrier() {                // all warps; its parties stand at different places in the code
    __syncwarp();
    asm volatile("bar.sync 0;" ::: "memory");
}
__device__ __forceinline__ void cp_async_4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Column groups of a tile, by rows of the state: as many as the registers hold.
__host__ __device__ constexpr int max_tile(int KC) { return KC == 8 ? 5 : KC == 16 ? 2 : 1; }

// What the layer loop needs; uniform over the CTA.  What is needed seldom stays in shared memory: registers are short.
struct Rare {
    int S, M, m_pitch;
    uint32_t all;          // records of all strategies: slot 0's list (see prepare)
    int32_t* C_last;
    uint32_t* states;
};
struct Ctx {
    const volatile Rare* rare;
    bool states;           // the states are kept
    int Mp, G, NW, Li, Kc;
    int TM, steps, per_step;       // column groups of a tile; runs of columns a layer, groups in one
    uint32_t tmax;
    uint32_t base, d;      // shared addresses of column 0 (row 0) of the bases and of the differences
    uint32_t base0, d0;    // ... of the first guard column, which records count from
    uint32_t keep;         // records of the strategies that can matter: slot 0's list
    uint32_t slot_bytes;   // from one slot's list to the next one's
    uint32_t slot;         // [4] the slot of layer l is slot[l & 3] (layers with the same rows share one)
    uint32_t nkeep;        // [4] entries of a slot's second list
    uint32_t front;        // [4] no column below front[l & 3] holds a finite value in layer l
    uint32_t hard;         // three words and a pad: which tiles are shared out (see step_end), then [NW][TM] two words of bits: their groups' strategies
    int* hard_bits;        // the three words
    uint32_t tags;         // [steps][NW] what a tile's differences are: T[k][.] of row class k, or -1
    uint32_t tsm, tmat;    // transition entries, KC to a row; from one matrix to the next with one per layer, else 0
};

// The columns [32 g, 32 g + 32) of kBatch rows from s0 on of the last layer.
template <int F>
__device__ __forceinline__ void put_values(const Ctx& c, int l, int g, int s0, int lane)
{
    const int col = 32 * g + lane, m_pitch = c.rare->m_pitch, M = c.rare->M, n = min(kBatch, c.rare->S - s0);
    int32_t* const out = c.rare->C_last + (size_t)s0 * m_pitch + col;
    const uint32_t bb = c.base0 + 4u * col, dd = c.d0 + 4u * col, rec = c.rare->all + lds<0>(c.slot + 4u * (l & 3)) * c.slot_bytes + 16u * s0;
    // all loads of a batch before its first store; rows past the last are the last again
    int4 r[kBatch];
    uint32_t b[kBatch], d[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) r[u] = lds4(rec + 16u * min(u, n - 1));
#pragma unroll
    for (int u = 0; u < kBatch; ++u) { b[u] = lds<0>(bb + r[u].y); d[u] = ldd<F, 0>(dd + r[u].x); }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
        if (u < n) out[(size_t)(uint32_t)(u * m_pitch)] = (int32_t)(col > M ? kInf : min(b[u] + d[u] + (uint32_t)r[u].z, kInf));
}

// The state that layer l reads, columns [32 g, 32 g + 32), to its place in `states`: a row of bases, and behind it those of the
// differences' words as they are; where nothing is finite, the bases alone.
template <int F>
__device__ __forceinline__ void put_state(const Ctx& c, int l, int g, int lane)
{
    const int col = 32 * g + lane, words = F == kWord ? c.Kc : (c.Kc + 1) >> 1;
    const int m_pitch = c.rare->m_pitch;
    uint32_t* out = c.rare->states + (size_t)l * (words + 1) * m_pitch + col;
    *out = lds<0>(c.base + 4u * col);
    if (32 * g + 31 < (int)lds<0>(c.front + 4u * ((l - 1) & 3))) return;
    uint32_t d = c.d + 4u * col;
#pragma unroll 4
    for (int p = 0; p < words; ++p) {
        out += m_pitch;
        *out = lds<0>(d);
        d += 4u * c.Mp;
    }
}

// Candidates v + T[k][q] of every row q of the next state, N words of them.
template <int KC, int N, int F>
__device__ __forceinline__ void relax(const Ctx& c, uint32_t row, uint32_t v, uint32_t (&acc)[N])
{
#pragma unroll
    for (int q = 0; q < N; q += 4) {
        if (KC <= 8 || q * (KC / N) < c.Kc) {
            const int4 t = lds4(row + 4u * q);
            if (F == kPacked) {
                acc[q] = __viaddmin_u16x2(v, (uint32_t)t.x, acc[q]);
                acc[q + 1] = __viaddmin_u16x2(v, (uint32_t)t.y, acc[q + 1]);
                acc[q + 2] = __viaddmin_u16x2(v, (uint32_t)t.z, acc[q + 2]);
                acc[q + 3] = __viaddmin_u16x2(v, (uint32_t)t.w, acc[q + 3]);
            } else {
                acc[q] = __viaddmin_u32(v, (uint32_t)t.x, acc[q]);
                acc[q + 1] = __viaddmin_u32(v, (uint32_t)t.y, acc[q + 1]);
                acc[q + 2] = __viaddmin_u32(v, (uint32_t)t.z, acc[q + 2]);
                acc[q + 3] = __viaddmin_u32(v, (uint32_t)t.w, acc[q + 3]);
            }
        }
    }
}

// The strategies of a column group that can matter: the first 64 of the list by their bits, what is beyond always.
struct Alive {
    uint32_t m0, m1;
    int e, n;              // next entry beyond 64, entries
    __device__ __forceinline__ bool some() const { return m0 || m1 || e < n; }
    __device__ __forceinline__ int next()                      // n, an entry of +inf, when none is left
    {
        if (m0) { const int q = __ffs(m0) - 1; m0 &= m0 - 1; return q; }
        if (m1) { const int q = __ffs(m1) + 31; m1 &= m1 - 1; return q; }
        return e < n ? e++ : n;
    }
};

// Four of them at a time: a chain of latencies for four.
template <int F>
struct Four {
    int4 r[4];
    uint32_t v[4];
    __device__ __forceinline__ void get(Alive& al, uint32_t list, uint32_t gb, uint32_t gd)
    {
        uint32_t b[4], d[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = lds4(list + 16u * al.next());
#pragma unroll
        for (int u = 0; u < 4; ++u) { b[u] = lds<0>(gb + r[u].y); d[u] = ldd<F, 0>(gd + r[u].x); }
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = min(b[u] + d[u] + (uint32_t)r[u].z, kInf);
    }
    __device__ __forceinline__ uint32_t least() const { return min(min(v[0], v[1]), min(v[2], v[3])); }
};

// A column's base and the difference of one of its rows, in TM column groups.
template <int F, int TM, int J = 0>
__device__ __forceinline__ void gather(uint32_t bb, uint32_t dd, uint32_t (&b)[TM], uint32_t (&d)[TM]) {
    b[J] = lds<128 * J>(bb);
    d[J] = ldd<F, 128 * J>(dd);
    if constexpr (J + 1 < TM) gather<F, TM, J + 1>(bb, dd, b, d);
}
template <int F, int TM>
__device__ __forceinline__ void values(uint32_t gb, uint32_t gd, const int4& r, uint32_t (&v)[TM])
{
    uint32_t b[TM], d[TM];
    gather<F, TM>(gb + r.y, gd + r.x, b, d);
#pragma unroll
    for (int j = 0; j < TM; ++j) v[j] = min(b[j] + d[j] + (uint32_t)r.z, kInf);
}

// The words of a column's differences from its accumulators.
template <int F, int N, int W>
__device__ __forceinline__ void differences(const uint32_t (&acc)[N], uint32_t v0, uint32_t (&out)[W])
{
#pragma unroll
    for (int p = 0; p < W; ++p) {
        if (F == kPacked) out[p] = acc[p % N];
        else if (F == kHalf) out[p] = (acc[2 * p % N] - v0) + (acc[(2 * p + 1) % N] - v0) * 65536u;
        else out[p] = acc[p % N] - v0;
    }
}

// One column group where several strategies can matter: a relaxation each.
template <int KC, int F, int W>
__device__ __forceinline__ void several(const Ctx& c, Alive al, uint32_t list, uint32_t tm, uint32_t gb, uint32_t gd, uint32_t& best, uint32_t (&out)[W])
{
    constexpr int N = F == kPacked ? KC / 2 : KC;              // words of a matrix row
    uint32_t acc[N], v0;
#pragma unroll
    for (int q = 0; q < N; ++q) acc[q] = ~0u;
    Four<F> f;
    f.get(al, list, gb, gd);
    v0 = f.least();
    // Packed: on differences to the column's best.  What lies further than tmax above it can neither win nor tie: clamped to tmax + 1.
    auto relax_four = [&]() {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            relax<KC, N, F>(c, tm + 4u * (f.r[u].w * N), F == kPacked ? min(f.v[u] - v0, c.tmax + 1) * 65537u : f.v[u], acc);
    };
    if (F == kPacked) {
        Alive first = al;
        Four<F> more;
#pragma unroll 1
        while (al.some()) { more.get(al, list, gb, gd); v0 = min(v0, more.least()); }
        relax_four();
#pragma unroll 1
        while (first.some()) { f.get(first, list, gb, gd); relax_four(); }
    } else {
        relax_four();
#pragma unroll 1
        while (al.some()) { f.get(al, list, gb, gd); v0 = min(v0, f.least()); relax_four(); }
    }
    best = v0;
    differences<F, N, W>(acc, v0, out);
}

template <int F, int W>
__device__ __forceinline__ void write_group(const Ctx& c, int g, int lane, uint32_t v0, const uint32_t (&out)[W])
{
    const uint32_t at = 4u * (32 * g + lane), row_bytes = 4u * c.Mp;
    const int words = F == kWord ? c.Kc : (c.Kc + 1) >> 1;
    sts(c.base + at, v0);
#pragma unroll
    for (int p = 0; p < W; ++p)
        if (p < words) sts(c.d + at + p * row_bytes, out[p]);
}

// Ends what a step reads.  The tiles that many strategies can matter in lie side by side, where C falls steeply: one warp would have
// such a tile to itself and the others would wait (6000 cycles against 1700).  So after a barrier the warps share out these
// tiles' column groups, one each and from the highest down, in as many rounds as that takes: what a round writes no later one
// reads.  Which tiles: bits of a word, three words in turn (step: steps counted through the layers), the next but one cleared.
__device__ __forceinline__ int rounds_of(int bits, int TM, int NW) { return (__popc(bits) * TM + NW - 1) / NW; }
template <int KC, int TM, int F>
__device__ __forceinline__ void step_end(const Ctx& c, int step, int lo, int hi, int warp, int lane, uint32_t list, int n, uint32_t tm)
{
    constexpr int W = F == kWord ? KC : KC / 2;
    cta_barrier();
    if (TM == 1) return;                                       // tiles of one group: nothing to share out
    const int bits = (int)lds<0>(c.hard + 4u * (step % 3));
    if (warp == 0) sts(c.hard + 4u * ((step + 2) % 3), 0u);
    if (bits == 0) return;
    const int total = __popc(bits) * TM;
#pragma unroll 1
    for (int e = warp; e - warp < total; e += c.NW) {
        int g = -1;
        uint32_t v0, out[W];
        if (e < total) {
            int left = bits;                                   // the tile: the (e / TM)-th highest bit
            for (int k = e / TM; k > 0; --k) left &= ~(1 << (31 - __clz(left)));
            const int t = 31 - __clz(left), j = TM - 1 - e % TM;
            g = min(lo + t * TM, hi - TM) + j;
            if (g < lo + t * TM) g = -1;                       // the tile below has this group too
            if (g >= 0) {
                const uint32_t at = c.hard + 16u + 8u * (t * TM + j), col = 32u * g + lane;
                several<KC, F, W>(c, Alive{lds<0>(at), lds<4>(at), 64, n}, list, tm, c.base0 + 4u * col, c.d0 + 4u * col, v0, out);
            }
        }
        cta_barrier();
        if (g >= 0) write_group<F, W>(c, g, lane, v0, out);
    }
}

// One layer of TM column groups from g on: the state behind layer l.  KC: rows of that state at most.  mine: this lane's entry
// of the list.  g < 0: no tile for this warp.  What is read comes before step_end, what is written behind it.
template <int KC, int TM, int F>
__device__ __forceinline__ void tile(const Ctx& c, int l, int g, int step, int lo, int hi, int warp, int lane, uint32_t list, int n, const int4& mine, uint32_t tag)
{
    constexpr int N = F == kPacked ? KC / 2 : KC, W = F == kWord ? KC : KC / 2;      // words of a matrix row, of a column's differences
    const int col0 = 32 * g, col = col0 + lane;
    const uint32_t wb = c.base + 4u * col, wd = c.d + 4u * col, row_bytes = 4u * c.Mp;
    const uint32_t gb = c.base0 + 4u * col, gd = c.d0 + 4u * col;
    const uint32_t tm = c.tsm + (((l + 1) & 1) ? c.tmat : 0u);
    const int words = F == kWord ? c.Kc : (c.Kc + 1) >> 1;
    auto end = [&]() { step_end<KC, TM, F>(c, step, lo, hi, warp, lane, list, n, tm); };

    if (g < 0 || n == 0 || col0 + 32 * TM - 1 < (int)lds<0>(c.front + 4u * (l & 3))) {       // +inf all over, and in the next layers too
        end();
        if (g >= 0)
#pragma unroll
            for (int j = 0; j < TM; ++j) sts(wb + 128u * j, kInf);
        return;
    }
    // ---- who can matter: a strategy a lane, its values at the tile's first column and at its last.  (Lanes read at shifts of
    // their own: three to four wavefronts a load, which is what the test costs.)
    uint32_t any0, any1 = 0;
    {
        auto bounds = [&](const int4& r, uint32_t& high, uint32_t& low) {
            const uint32_t b0 = c.base0 + 4u * col0 + r.y, d0 = c.d0 + 4u * col0 + r.x;
            const uint32_t b = lds<0>(b0), d = ldd<F, 0>(d0), b1 = lds<128 * TM - 4>(b0), d1 = ldd<F, 128 * TM - 4>(d0);
            high = min(high, b + d + (uint32_t)r.z);
            low = b1 + d1 + (uint32_t)r.z;
        };
        uint32_t high = kInf, low0, low1 = ~0u;
        bounds(mine, high, low0);
        if (n > 32) bounds(lds4(list + 16u * min(32 + lane, n)), high, low1);
        const uint32_t limit = __reduce_min_sync(0xffffffffu, high) + c.tmax;
        any0 = __ballot_sync(0xffffffffu, low0 <= limit && low0 < kInf);
        if (n > 32) any1 = __ballot_sync(0xffffffffu, low1 <= limit && low1 < kInf);
    }
    int alive = n > 64 ? 99 : __popc(any0) + __popc(any1);
    if (TM > 1 && alive > 4) {
        // the same group by group.  The first column of the next group bounds a group from below as well as its own last one.
        auto bounds = [&](const int4& r, uint32_t (&u)[TM + 1]) {
            const uint32_t b0 = c.base0 + 4u * col0 + r.y, d0 = c.d0 + 4u * col0 + r.x;
            uint32_t b[TM + 1], d[TM + 1];
#pragma unroll
            for (int j = 0; j < TM; ++j) { b[j] = lds<0>(b0 + 128u * j); d[j] = ldd<F, 0>(d0 + 128u * j); }
            b[TM] = lds<128 * TM - 4>(b0); d[TM] = ldd<F, 128 * TM - 4>(d0);
#pragma unroll
            for (int j = 0; j <= TM; ++j) u[j] = b[j] + d[j] + (uint32_t)r.z;
        };
        uint32_t u[TM + 1], w[TM + 1];
        bounds(mine, u);
        if (n > 32) {
            bounds(lds4(list + 16u * min(32 + lane, n)), w);
        } else {
#pragma unroll
            for (int j = 0; j <= TM; ++j) w[j] = ~0u;
        }
        any0 = any1 = 0;
#pragma unroll
        for (int j = 0; j < TM; ++j) {
            const uint32_t limit = min(__reduce_min_sync(0xffffffffu, min(u[j], w[j])), kInf) + c.tmax;
            const uint32_t m0 = __ballot_sync(0xffffffffu, u[j + 1] <= limit && u[j + 1] < kInf);
            const uint32_t m1 = n > 32 ? __ballot_sync(0xffffffffu, w[j + 1] <= limit && w[j + 1] < kInf) : 0u;
            any0 |= m0; any1 |= m1;
            if (lane == 0) { sts(c.hard + 16u + 8u * (warp * TM + j), m0); sts(c.hard + 20u + 8u * (warp * TM + j), m1); }
        }
        if (n <= 64) alive = __popc(any0) + __popc(any1);
    }
    Alive al{any0, any1, 64, n};
    if (alive <= 1) {
        // ---- one strategy in all of the tile: base = its values, differences = its class's row of the matrix
        const int4 r = lds4(list + 16u * al.next());
        uint32_t v[TM];
        values<F, TM>(gb, gd, r, v);
        const bool fresh = lds<0>(tag) != (uint32_t)r.w || c.tmat;
        end();
#pragma unroll
        for (int j = 0; j < TM; ++j) sts(wb + 128u * j, v[j]);
        if (fresh) {
            const uint32_t row = tm + 4u * (r.w * N);
#pragma unroll 1
            for (int p = 0; p < words; ++p) {
                const uint32_t t = F == kHalf ? lds<0>(row + 8u * p) | lds<4>(row + 8u * p) << 16 : lds<0>(row + 4u * p);
#pragma unroll
                for (int j = 0; j < TM; ++j) sts(wd + p * row_bytes + 128u * j, t);
            }
            __syncwarp();
            sts(tag, c.tmat ? ~0u : (uint32_t)r.w);
        }
        return;
    }
    uint32_t v0[TM], out[TM][W];
    if (alive <= 4) {
        // ---- two, or up to four: their values above the columns' smallest, and what those and the transition entries come to
        const bool more = alive > 2;
        uint32_t row[4], v[4][TM];
        {
            const int4 ra = lds4(list + 16u * al.next()), rb = lds4(list + 16u * al.next());
            row[0] = tm + 4u * (ra.w * N); row[1] = tm + 4u * (rb.w * N);
            values<F, TM>(gb, gd, ra, v[0]);
            values<F, TM>(gb, gd, rb, v[1]);
        }
#pragma unroll
        for (int j = 0; j < TM; ++j) v0[j] = min(v[0][j], v[1][j]);
        if (more) {
            const int4 rc = lds4(list + 16u * al.next()), rd = lds4(list + 16u * al.next());
            row[2] = tm + 4u * (rc.w * N); row[3] = tm + 4u * (rd.w * N);
            values<F, TM>(gb, gd, rc, v[2]);
            values<F, TM>(gb, gd, rd, v[3]);
#pragma unroll
            for (int j = 0; j < TM; ++j) v0[j] = min(v0[j], min(v[2][j], v[3][j]));
        }
        constexpr int PER = F == kHalf ? 2 : 1;                // matrix words to a word of differences
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u >= 2 && !more) break;
#pragma unroll
            for (int j = 0; j < TM; ++j) {
                v[u][j] -= v0[j];
                if (F == kPacked) v[u][j] = min(v[u][j], c.tmax + 1) * 65537u;       // beyond tmax it can neither win nor tie
            }
#pragma unroll
            for (int q = 0; q < N; q += 4)
                if (KC <= 8 || q * (KC / N) < c.Kc) {
                    const int4 t4 = lds4(row[u] + 4u * q);
                    const uint32_t t[4] = {(uint32_t)t4.x, (uint32_t)t4.y, (uint32_t)t4.z, (uint32_t)t4.w};
#pragma unroll
                    for (int p = 0; p < 4 / PER; ++p)
#pragma unroll
                        for (int j = 0; j < TM; ++j) {
                            uint32_t& o = out[j][q / PER + p];
                            if (F == kPacked) o = u ? __viaddmin_u16x2(v[u][j], t[p], o) : v[u][j] + t[p];
                            else if (F == kWord) o = u ? __viaddmin_u32(v[u][j], t[p], o) : v[u][j] + t[p];
                            else {
                                const uint32_t both = min(v[u][j] + t[2 * p % 4], 65535u) + min(v[u][j] + t[(2 * p + 1) % 4], 65535u) * 65536u;
                                o = u ? __vminu2(o, both) : both;
                            }
                        }
                }
        }
        end();
        sts(tag, ~0u);
#pragma unroll
        for (int j = 0; j < TM; ++j) sts(wb + 128u * j, v0[j]);
#pragma unroll
        for (int p = 0; p < W; ++p)
            if (p < words)
#pragma unroll
                for (int j = 0; j < TM; ++j) sts(wd + p * row_bytes + 128u * j, out[j][p]);
        return;
    }
    // ---- more
    if (TM > 1) {
        if (lane == 0) atomicOr(c.hard_bits + step % 3, 1 << warp);
        sts(tag, ~0u);
        end();
        return;
    }
    several<KC, F, W>(c, Alive{any0, any1, 64, n}, list, tm, gb, gd, v0[0], out[0]);
    end();
    sts(tag, ~0u);
    write_group<F, W>(c, g, lane, v0[0], out[0]);
}

// The layers, by the compute warps.  A layer is `steps` runs of columns from the highest down; in each the warps first read, and
// after the barrier write the new state over the old one.  One more barrier ends the layer.
template <int KC, int TM, int F>
__device__ __forceinline__ void run_layers(const Ctx& c, int warp, int lane)
{
    int step = 0;
#pragma unroll 1
    for (int l = 0; l + 1 < c.Li; ++l) {
        const uint32_t slot = lds<0>(c.slot + 4u * (l & 3));
        const int n = (int)lds<0>(c.nkeep + 4u * slot);
        const uint32_t list = c.keep + slot * c.slot_bytes;
        const int4 mine = lds4(list + 16u * min(lane, n));
        int hi = c.G;
#pragma unroll 1
        for (int t = 0; t < c.steps; ++t) {
            const int lo = max(0, hi - c.per_step), g = lo + warp * TM;
            if (c.states && l > 0)
                for (int x = lo + warp; x < hi; x += c.NW) put_state<F>(c, l, x, lane);
            // the last tile of a step may reach into the one before it: the same values are written twice
            tile<KC, TM, F>(c, l, g < hi ? min(g, hi - TM) : -1, step, lo, hi, warp, lane, list, n, mine, c.tags + 4u * (t * c.NW + warp));
            hi = lo; ++step;
        }
        cta_barrier();
    }
    const int l = c.Li - 1, nb = (c.rare->S + kBatch - 1) / kBatch;
    if (c.states && l > 0)
        for (int x = warp; x < c.G; x += c.NW) put_state<F>(c, l, x, lane);
#pragma unroll 1
    for (int u = warp; u < c.G * nb; u += c.NW) put_values<F>(c, l, u / nb, u % nb * kBatch, lane);
}

template <int KC, int F>
__device__ __forceinline__ void run(const Ctx& c, int warp, int lane)
{
    if (c.TM > 1) run_layers<KC, max_tile(KC), F>(c, warp, lane);
    else run_layers<KC, 1, F>(c, warp, lane);
}

// What a step of tiles costs here, in SM cycles: by how many strategies are listed, how many of them pass the test at a column group,
// and the share of tiles that are shared out group by group (and how many pass there).  Fitted on B200 to 460 shapes of analytic and
// of measured tables: tiles of one group to 15 %, of several groups to 25 % for the most part, below 700 columns to a factor of two.
// fill: the share of a step's column groups that there are.  states: they are written too.
struct Passing { float listed, alive, shared, shared_alive; };
__host__ __device__ inline float step_cycles(int KC, bool word, bool states, const Passing& p, float fill)
{
    const float past = p.listed > 64.0f ? p.listed - 64.0f : 0.0f, alive = p.alive + past;      // beyond the 64th of a list all of them pass
    const float shared_alive = p.shared_alive + past * p.shared;
    const float t = KC == 8    ? 1950.0f + 24.0f * p.listed + 210.0f * alive + (5600.0f * p.shared + 1320.0f * shared_alive) * fill
                    : KC == 16 ? 2280.0f + 26.0f * p.listed + 3000.0f * p.shared + 550.0f * shared_alive + 100.0f * alive
                    : KC == 32 ? 430.0f + 51.0f * p.listed + 640.0f * alive
                               : 2480.0f + 32.0f * p.listed + 1055.0f * alive;
    return t * (word ? 1.9f : 1.0f) + (states ? 2500.0f : 0.0f);
}

// What a layer costs a column group and an SM in the tiled kernels, which take unstructured matrices of large batches (to 12 %): the
// packed loop, and the 32-bit one with dominated rows left out.
__host__ __device__ inline float tiled_cycles(int S, bool packed, float alive)
{
    return packed ? 82.0f + 16.05f * S + 0.13f * S * S : 34.0f + 10.76f * S + 0.197f * S * S + 0.33f * alive * S;
}
// The resident kernel against its plan's estimate: stacks of layers that repeat (0.8 to 2.0 of it), of layers that all differ (1.6 to
// 3.5: a warp prepares each one's records), and what a strategy and column group of a warp adds where shifts pass the halo (40 to 230).
constexpr float kResidentRepeats = 1.2f, kResidentDiffers = 1.7f, kResidentPastHalo = 60.0f;

// Whether a batch is worth the solo kernel: the SM cycles it would take there, and elsewhere, if all its instances were like one, for up
// to kGuessed of them; -1: an instance that is not searched at all.
//
// What it costs hangs on how many strategies pass the test at a column group, which is guessed from a few layers' rows.  Where C
// falls by `slope` a column a strategy weighs time + slope * mem, and passes if that is within the largest transition entry of the
// layer's best; and there a layer of the best plan takes the mem of that best one.  So slopes from 0 (the budget is no bound)
// upwards, each with the layers and columns that lie between its mem and the next one's: within a quarter of what passes, on all
// tables tried (independent times and memories, less memory for more time, analytic models).
//
// One answer for the batch, as a mixed one pays for both kernels in turn (100 instances of 40 layers, S = 24 of 3000 columns, some of
// them taken: 1044 us against 542 and 575).  A kernel of its own, as the solo kernel's start is 20 thousand cycles, most of them
// spent on fetching its code: a batch that is turned away pays 15 to 20 us.  Taken where the guess leaves a tenth.
// Other kernels / solo kernel / with this rule, us: 64 instances of 60 layers of an analytic model, S = 32 of 2880 columns 278 / 482 / 295;
// 200 of 40, S = 64 of 4 classes and 4000 columns, transitions twice the layer times 1143 / 2700 / 1165; 200 of 40 of an analytic model,
// S = 64 of 2880 columns 2195 / 421 / 436; 300 of 30 measured, S = 24 of 3000 1529 / 799 / 825; host entry point, 130 of 60, S = 32 of 8192
// 4563 / 2159 / 2176.
constexpr int kGuessed = 32, kGuessThreads = 512, kGuessLayers = 8, kSlopes = 6;
constexpr float kGuessTaken = 0.9f, kGuessNoRoom = 1e30f, kGuessAway = -4.0f;
struct GuessArgs {
    int B, Lmax, S, M, n;
    int nw, groups, dense, states, room;
    SoOther other;
    const int32_t* L;
    const int32_t* time_q;
    const int32_t* mem_q;
    const int32_t* trans_q;
    long long trans_inst, trans_layer;
    float2* guess;
    int32_t* ticket;               // 0 before and afterwards
};

// What the looks at the instances come to, by one warp.  Where a round holds all instances the longest one counts, else their sum;
// what there is no room for goes elsewhere afterwards.
__device__ __forceinline__ bool turned_away(const float2* guess, int n, bool one_round, bool other_one_round)
{
    const int lane = threadIdx.x & 31;
    float2 mine = make_float2(-1.0f, 0.0f);
    if (lane < n) mine = __ldcg(guess + lane);
    const bool any = mine.x >= 0.0f, fits = mine.x < kGuessNoRoom;
    const float here = any && fits ? mine.x : 0.0f, after = any && !fits ? mine.y : 0.0f, other = any ? mine.y : 0.0f;
    auto all = [](float v, bool most) {
        for (int o = 16; o > 0; o >>= 1) { const float w = __shfl_xor_sync(0xffffffffu, v, o); v = most ? fmaxf(v, w) : v + w; }
        return v;
    };
    const float count = (float)__popc(__ballot_sync(0xffffffffu, any));
    const float cost = one_round ? count * all(here, true) : all(here, false), elsewhere = other_one_round ? count * all(other, true) : all(other, false);
    return cost + (other_one_round ? count * all(after, true) : all(after, false)) > kGuessTaken * elsewhere;
}

__global__ void __launch_bounds__(kGuessThreads) guess_kernel(const GuessArgs a)
{
    constexpr int NW = kGuessThreads / 32, kRows = 4;          // rows of the matrix a warp looks at together
    __shared__ uint32_t s_row[kMaxS + kRows * NW], s_col[kMaxS];
    __shared__ int s_next[kMaxS];                              // the next strategy of the same row and column, round and round
    __shared__ int2 s_at[kGuessLayers][kMaxS];                 // mem, time
    __shared__ float2 s_point[kGuessLayers][kMaxS];            // time, mem; +inf where it does not fit or another one of its kind is as good
    __shared__ float s_time[NW], s_mem[NW];
    __shared__ int s_tmax, s_kinds[2], s_listed, s_mmax, s_pass[kSlopes], s_used[kSlopes], s_shared[kSlopes], s_shared_pass[kSlopes];
    __shared__ uint32_t s_rows[kGuessLayers];
    __shared__ bool s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, S = a.S, M = a.M;
    const int i = a.n > 1 ? (int)((long long)blockIdx.x * (a.B - 1) / (a.n - 1)) : 0;
    const int Li = a.L[i];
    auto finish = [&](float2 mine) {                           // thread 0's; the CTA that comes last says what they all come to
        if (tid == 0) {
            a.guess[blockIdx.x] = mine;
            __threadfence();
            s_last = atomicAdd(a.ticket, 1) == a.n - 1;
        }
        __syncthreads();
        if (!s_last || warp != 0) return;
        __threadfence();
        const bool away = turned_away(a.guess, a.n, a.other.one_round, a.other.other_one_round);
        if (lane == 0) { if (away) a.guess[0].x = kGuessAway; *a.ticket = 0; }
    };
    if (Li < 1 || Li > a.Lmax) { finish(make_float2(-1.0f, 0.0f)); return; }
    const int32_t* const T = a.trans_q + (size_t)i * a.trans_inst;
    const int layers = min(Li, kGuessLayers);
    auto layer_of = [&](int q) { return layers > 1 ? (int)((long long)q * (Li - 1) / (layers - 1)) : 0; };
    if (tid < S) s_col[tid] = 0;
    if (tid < kSlopes) { s_pass[tid] = 0; s_used[tid] = 0; s_shared[tid] = 0; s_shared_pass[tid] = 0; }
    if (tid < kGuessLayers) s_rows[tid] = 0;
    if (tid == 0) { s_tmax = 0; s_kinds[0] = 0; s_kinds[1] = 0; s_listed = 0; s_mmax = 0; }
    __syncthreads();
    {
        float time = 0.0f, mem = 0.0f;
        for (int x = tid; x < layers * S; x += kGuessThreads) {
            const int q = x / S, s = x - q * S;
            const size_t at = ((size_t)i * a.Lmax + layer_of(q)) * S + s;
            const int2 me = make_int2(a.mem_q[at], a.time_q[at]);
            s_at[q][s] = me;
            atomicAdd(&s_rows[q], ((uint32_t)me.x * 0x85EBCA6Bu + (uint32_t)me.y) * ((uint32_t)s * 0x9E3779B2u + 0x7F4A7C15u));
            time += (float)me.y; mem += (float)min(me.x, M);
        }
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) { time += __shfl_xor_sync(0xffffffffu, time, o); mem += __shfl_xor_sync(0xffffffffu, mem, o); }
        if (lane == 0) { s_time[warp] = time; s_mem[warp] = mem; }
    }
    // ---- the matrix: sums over the words of its rows and columns, which tell the classes, and its largest entry.  Of matrices per
    // layer, whose rows are all kinds of their own, a few rows each.
    {
        int tmax = 0;
        if (!a.trans_layer) {
#pragma unroll 1
            for (int r0 = warp; r0 < S; r0 += kRows * NW) {
                uint32_t row[kRows] = {};
#pragma unroll 1
                for (int s = lane; s < S; s += 32) {
                    int v[kRows];
                    uint32_t col = 0;
#pragma unroll
                    for (int u = 0; u < kRows; ++u) v[u] = r0 + u * NW < S ? T[(r0 + u * NW) * S + s] : 0;
#pragma unroll
                    for (int u = 0; u < kRows; ++u) {
                        tmax = max(tmax, v[u]);
                        row[u] += (uint32_t)v[u] * ((uint32_t)s * 0x9E3779B2u + 0x7F4A7C15u);
                        col += (uint32_t)v[u] * ((uint32_t)(r0 + u * NW) * 0x9E3779B2u + 0x7F4A7C15u);
                    }
                    atomicAdd(&s_col[s], col);
                }
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    row[u] = __reduce_add_sync(0xffffffffu, row[u]);
                    if (lane == 0) s_row[r0 + u * NW] = row[u];
                }
            }
        } else if (warp < layers && layer_of(warp) > 0) {
            const int32_t* const Tl = T + (size_t)layer_of(warp) * a.trans_layer;
#pragma unroll 4
            for (int k = lane; k < min(S, 8) * S; k += 32) tmax = max(tmax, Tl[k]);
        }
        tmax = __reduce_max_sync(0xffffffffu, tmax);
        if (lane == 0) atomicMax(&s_tmax, tmax);
    }
    __syncthreads();
    if (!a.trans_layer && tid < S) {                            // the first ones of their rows and of their columns, and who shares both
        const uint32_t hr = s_row[tid], hc = s_col[tid];
        int row = 0, col = 0, both = tid, next = -1;
#pragma unroll 4
        for (int o = S - 1; o >= 0; --o) {
            const bool r = s_row[o] == hr, c = s_col[o] == hc;
            row += r && o < tid;
            col += c && o < tid;
            if (r && c) { both = o; if (o > tid) next = o; }
        }
        s_next[tid] = next < 0 ? both : next;
        if (row == 0) atomicAdd(&s_kinds[0], 1);
        if (col == 0) atomicAdd(&s_kinds[1], 1);
    }
    __syncthreads();
    const bool classes = !a.trans_layer && max(s_kinds[0], s_kinds[1]) <= kClassMax;
    const int Kr = classes ? s_kinds[0] : S, Kc = classes ? s_kinds[1] : S;
    const int KC = Kc <= 8 && Kr <= 16 ? 8 : Kc <= 16 ? 16 : Kc <= 32 ? 32 : 64;
    for (int x = tid; x < layers * S; x += kGuessThreads) {
        const int q = x / S, s = x - q * S;
        const int2 me = s_at[q][s];
        bool in = me.x <= M;
        if (classes)
#pragma unroll 1
            for (int o = s_next[s]; in && o != s; o = s_next[o]) {
                const int2 ot = s_at[q][o];
                in = ot.x > me.x || ot.y > me.y || (o > s && ot.y == me.y);
            }
        s_point[q][s] = in ? make_float2((float)me.y, (float)me.x) : make_float2(__uint_as_float(0x7f800000u), 0.0f);
        if (in) { atomicAdd(&s_listed, 1); atomicMax(&s_mmax, me.x); }
    }
    __syncthreads();
    // ---- a layer and a slope a warp
    float scale = 0.0f, over = 0.0f;                           // the slope at which time and memory weigh the same
#pragma unroll 1
    for (int q = 0; q < NW; ++q) { scale += s_time[q]; over += s_mem[q]; }
    scale /= fmaxf(over, 1.0f);
#pragma unroll 1
    for (int x = warp; x < layers * kSlopes; x += NW) {
        const int q = x / kSlopes, k = x - q * kSlopes;
        const float slope = k == 0 ? 0.0f : scale * (float)(1 << 2 * k) * 0.0078125f;       // 0, 1/32, 1/8, .. 8 times
        const uint32_t none = 0x7f800000u;                     // +inf as bits: sorts behind every weight
        uint32_t best = none, used = 0x7fffffffu;
        int pass = 0, tile = 0;
#pragma unroll 1
        for (int s = lane; s < S; s += 32) best = min(best, __float_as_uint(__fmaf_rn(slope, s_point[q][s].y, s_point[q][s].x)));
        best = __reduce_min_sync(0xffffffffu, best);
        const float limit = __uint_as_float(best) + (float)s_tmax + 32.0f * slope, tile_limit = limit + 32.0f * (float)(max_tile(KC) - 1) * slope;
#pragma unroll 1
        for (int s = lane; s < S; s += 32) {
            const float2 p = s_point[q][s];
            const float v = __fmaf_rn(slope, p.y, p.x);
            pass += __float_as_uint(v) != none && v <= limit;
            tile += __float_as_uint(v) != none && v <= tile_limit;
            if (__float_as_uint(v) == best) used = min(used, (uint32_t)p.y);
        }
        pass = __reduce_add_sync(0xffffffffu, pass);
        tile = __reduce_add_sync(0xffffffffu, tile);
        used = __reduce_min_sync(0xffffffffu, used);
        if (lane == 0 && best != none) {
            atomicAdd(&s_pass[k], pass); atomicAdd(&s_used[k], (int)used);
            if (tile > 4) { atomicAdd(&s_shared[k], 1); atomicAdd(&s_shared_pass[k], pass); }      // see tile
        }
    }
    __syncthreads();
    // ---- layers and columns below the line column = layer * mem, slope by slope
    float2 mine = make_float2(-1.0f, 0.0f);
    if (tid == 0) {
        const float cols = (float)(M + 1), deep = (float)Li, all = cols * deep, per = 1.0f / (float)layers;
        Passing sum{(float)s_listed * per, 0.0f, 0.0f, 0.0f};
        float left = all;
#pragma unroll 1
        for (int k = 0; k < kSlopes; ++k) {
            const float mem = (float)s_used[k] * per;
            const float below = fminf(left, mem * deep <= cols ? 0.5f * mem * deep * deep : all - 0.5f * cols * cols / mem);
            const float weight = (left - below) / all * per * (k == 0 ? 1.0f : 0.5f);
            const int b = max(k - 1, 0), both = k > 0;             // between a slope and the one before it: half of each
            sum.alive += weight * (float)(s_pass[k] + both * s_pass[b]);
            sum.shared += weight * (float)(s_shared[k] + both * s_shared[b]);
            sum.shared_alive += weight * (float)(s_shared_pass[k] + both * s_shared_pass[b]);
            left = below;
        }
        const int step = a.nw * max_tile(KC), steps = (a.groups + step - 1) / step;
        const float cost = a.other.rounds * (float)steps * step_cycles(KC, s_tmax > 65535, a.states, sum, (float)a.groups / (float)(steps * step));
        float other;
        if (classes && a.other.w && Kc * a.other.w <= a.other.gints) {
            bool repeats = layers < kGuessLayers;
            for (int q = 1; q < layers; ++q)
                for (int o = 0; o < q; ++o) repeats |= s_rows[o] == s_rows[q];
            other = a.other.resident * (repeats ? kResidentRepeats : kResidentDiffers);
            if (s_mmax > ((a.other.gints / Kc - a.other.w) & ~31)) other += a.other.past_halo * sum.listed;
        } else {
            other = a.other.tiled * tiled_cycles(S, a.other.packed && s_tmax <= 32767, sum.alive);
        }
        other = fminf(other, a.other.most);
        // as the solo kernel sees it, but for the largest shift, which is the sampled layers'
        const long long H = (s_mmax + 31) & ~31, words = s_tmax > 65535 ? Kc : (Kc + 1) >> 1, Mp = 32 * a.groups;
        const bool fits = (classes || a.dense) && 4 * (H + Mp) + 4 * (H + words * Mp) <= a.room && (!a.states || 1 + words <= S);
        mine = make_float2(fits ? cost * deep + a.other.start : kGuessNoRoom, other * deep);
    }
    __syncwarp();
    finish(mine);
}

__global__ void __launch_bounds__((kMaxWarps + 1) * 32, 1) solo_kernel(const SoArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(16) int s_hard[4 + 2 * kMaxWarps * max_tile(8)];
    __shared__ int s_tag[kMaxTiles], s_root[2 * kMaxS];
    __shared__ Rare s_rare;
    __shared__ uint32_t s_hash[2 * kMaxS];
    __shared__ int s_rcls[kMaxS], s_ccls[kMaxS], s_order[kMaxS], s_first[kClassMax], s_cnt[kClassMax], s_rep[2 * kClassMax];
    __shared__ int s_front[4], s_slot[4], s_nkeep[4], s_inst, s_K[2], s_differ;
    __shared__ struct { long long sum; int tmax, bad, mmax; } s_all;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x, NW = a.NW;
    const int S = a.S, M = a.M, Lmax = a.Lmax, Mp = a.m_pitch;

    // ---- shared memory: records, raw rows, matrices, state
    const int S1 = S + 1, S4 = (S + 3) & ~3;
    int4* const rec = reinterpret_cast<int4*>(smem_raw);                                  // [2][4][S1]: all strategies, those that can matter
    int32_t* const raw = reinterpret_cast<int32_t*>(rec + 8 * S1);                        // [4][2][S4] mem, time rows as they come
    int32_t* const tsm = raw + 8 * S4;
    unsigned char* const state = reinterpret_cast<unsigned char*>(tsm + a.mats);

    if (a.guessed && a.guess[0].x < kGuessAway * 0.5f) {
        if (tid == 0) a.done[blockIdx.x] = 0;
        if (blockIdx.x == 0 && tid == 0) a.path[3] = kPathSolo | kPathRest;
        return;
    }
    if (blockIdx.x == 0 && tid == 0) {
        if (a.certain) a.path[3] = kPathSolo;
        else atomicOr(a.path + 3, kPathSolo);                    // cleared before
    }

    // ---- which instance: CTAs are dispatched in order, so the longest instances go first
    int i = blockIdx.x;
    if (a.sorted) {
        int* const s_len = reinterpret_cast<int*>(state);       // the state is not in use yet
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
            if (before == (int)blockIdx.x) s_inst = j;
        }
        __syncthreads();
        i = s_inst;
    }
    const int G = Mp / 32;
    const int Li = a.L[i];
    if (Li < 1 || Li > Lmax) {
        if (tid == 0) { a.status[i] = GALV_STATUS_BAD_INPUT; a.done[i] = 3; }
        return;
    }
    const int32_t* const tq = a.time_q + (size_t)i * Lmax * S;
    const int32_t* const mq = a.mem_q + (size_t)i * Lmax * S;
    const int32_t* const T0 = a.trans_q + (size_t)i * a.trans_inst;

    // ---- validation
    int32_t* const stage = reinterpret_cast<int32_t*>(state);   // the matrix, while the state is not in use yet
    const int TP = S | 1;                                       // odd pitch: columns are read without bank conflicts too
    const bool staged = !a.trans_layer && (long long)S * TP * 4 <= a.room;
    auto fetch = [&](int l) {
        int32_t* const rm = raw + (l & 3) * 2 * S4;
        for (int s = lane; s < S; s += 32) {
            cp_async_4(rm + s, mq + (size_t)l * S + s);
            cp_async_4(rm + S4 + s, tq + (size_t)l * S + s);
        }
    };
    if (warp == NW) {                                           // the first layers' rows are under way while the rest is looked at
        fetch(0);
        cp_async_commit();
        if (Li > 1) fetch(1);
        cp_async_commit();
    }
    if (tid == 0) { s_all.sum = 0; s_all.tmax = 0; s_all.bad = 0; s_all.mmax = 0; s_differ = 0; }
    if (tid < 4) s_hard[tid] = 0;
    for (int x = tid; x < kMaxTiles; x += NT) s_tag[x] = -1;
    __syncthreads();
    {
        long long sum = 0;
        int bad = 0, tmax = 0, mmax = 0;                        // mmax: the largest shift that stays inside the budget
        if (!a.trans_layer) {
#pragma unroll 4
            for (int k = tid; k < S * S; k += NT) {
                const int v = T0[k];
                bad |= v < 0;
                tmax = max(tmax, v);
                if (staged) { const int q = k / S; stage[q * TP + k - q * S] = v; }
            }
        }
        constexpr int U = 4;                                    // layers a warp looks at together: their loads are one round trip
        for (int l0 = warp * U; l0 < Li; l0 += (NW + 1) * U) {
            int mx[U];
#pragma unroll
            for (int u = 0; u < U; ++u) mx[u] = 0;
            for (int s = lane; s < S; s += 32) {
                int tv[U], mv[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int l = min(l0 + u, Li - 1);
                    tv[u] = tq[(size_t)l * S + s];
                    mv[u] = mq[(size_t)l * S + s];
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    bad |= (tv[u] < 0) | (mv[u] < 0);
                    mx[u] = max(mx[u], tv[u]);
                    mmax = max(mmax, mv[u] <= M ? mv[u] : 0);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int m = __reduce_max_sync(0xffffffffu, mx[u]);
                if (lane == 0 && l0 + u < Li) sum += m;
            }
        }
        if (a.trans_layer) {
            const long long nx = (long long)(Li - 1) * S * S;                     // matrix 0 is unused
            const int32_t* const x = T0 + (size_t)S * S;
#pragma unroll 8
            for (long long k = tid; k < nx; k += NT) {
                const int v = x[k];
                bad |= v < 0;
                tmax = max(tmax, v);
            }
        }
        tmax = __reduce_max_sync(0xffffffffu, tmax);
        mmax = __reduce_max_sync(0xffffffffu, mmax);
        bad = __any_sync(0xffffffffu, bad != 0);
        if (lane == 0) {
            if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(&s_all.sum), static_cast<unsigned long long>(sum));
            atomicMax(&s_all.tmax, tmax);
            atomicMax(&s_all.mmax, mmax);
            if (bad) atomicOr(&s_all.bad, 1);
        }
    }
    __syncthreads();

    // ---- classes of equal rows and equal columns: by a sum over their words, then word by word against the first of the sum
    if (staged) {
        for (int x = warp; x < 2 * S; x += NW + 1) {
            const int me = x < S ? x : x - S, step = x < S ? TP : 1, word = x < S ? 1 : TP;
            uint32_t h = 0;
            for (int j = lane; j < S; j += 32) h += (uint32_t)stage[me * step + j * word] * ((uint32_t)j * 0x9E3779B2u + 0x7F4A7C15u);
            h = __reduce_add_sync(0xffffffffu, h);
            if (lane == 0) s_hash[x] = h;
        }
        __syncthreads();
        for (int x = tid; x < 2 * S; x += NT) {
            const int off = x < S ? 0 : S;
            const uint32_t mine = s_hash[x];
            int first = x - off;
#pragma unroll 8
            for (int o = S - 1; o >= 0; --o)
                if (o < first && s_hash[off + o] == mine) first = o;
            s_root[x] = first;
        }
        __syncthreads();
        for (int x = warp; x < 2 * S; x += NW + 1) {
            const int me = x < S ? x : x - S, step = x < S ? TP : 1, word = x < S ? 1 : TP, first = s_root[x];
            bool differ = false;
            if (first != me)
                for (int j = lane; j < S; j += 32) differ |= stage[first * step + j * word] != stage[me * step + j * word];
            if (differ) s_differ = 1;
        }
        // classes numbered in the order of their firsts: a row or a column a thread
        for (int x = tid; x < 2 * S; x += NT) {
            const int off = x < S ? 0 : S, first = s_root[x];
            int before = 0, all = 0;
#pragma unroll 4
            for (int o = 0; o < S; ++o) {
                const int opens = s_root[off + o] == o;
                all += opens;
                before += opens & (o < first);
            }
            (x < S ? s_rcls : s_ccls)[x - off] = before;
            if (first == x - off && before < kClassMax) s_rep[(x < S ? 0 : kClassMax) + before] = first;
            if (x == off) s_K[x < S ? 0 : 1] = all;
        }
        __syncthreads();
        // strategies in the order of their rows' classes, ascending inside one
        if (s_K[0] <= kClassMax)
            for (int s = tid; s < S; s += NT) {
                const int k = s_rcls[s];
                int at = 0, from = 0, cnt = 0;
#pragma unroll 4
                for (int o = 0; o < S; ++o) {
                    const int ko = s_rcls[o];
                    from += ko < k;
                    at += ko == k && o < s;
                    cnt += ko == k;
                }
                s_order[from + at] = s;
                if (at == 0) { s_first[k] = from; s_cnt[k] = cnt; }
            }
        __syncthreads();
    }
    const int K = staged && !s_differ ? max(s_K[0], s_K[1]) : S;
    const bool classes = staged && !s_differ && K <= kClassMax;
    const int Kr = classes ? s_K[0] : S, Kc = classes ? s_K[1] : S;
    const int KC = Kc <= 8 && Kr <= 16 ? 8 : Kc <= 16 ? 16 : Kc <= 32 ? 32 : 64;          // words of a matrix row
    const int st = s_all.bad ? GALV_STATUS_BAD_INPUT
                             : s_all.sum + (long long)(Li - 1) * s_all.tmax >= (long long)kInf ? GALV_STATUS_OVERFLOW_RISK : 0;
    // ---- the state: guard columns of +inf below column 0, as many as the largest shift; rows lie one behind the other, so what
    // a shift finds below its own row's column 0 is a difference of another column, or a zero before the first row
    const int form = s_all.tmax > 65535 ? kWord : a.packed && s_all.tmax <= 32767 ? kPacked : kHalf;
    const int H = (s_all.mmax + 31) & ~31, words = form == kWord ? Kc : (Kc + 1) >> 1;      // words of a column's differences
    const long long base_bytes = 4ll * (H + Mp), d_bytes = 4ll * (H + (long long)words * Mp);
    const int per_warp = max_tile(KC), steps = (G + NW * per_warp - 1) / (NW * per_warp), per_step = (G + steps - 1) / steps;
    const bool run_it = st == 0 && (classes || (a.dense && S <= kDenseMax)) && base_bytes + d_bytes <= a.room && steps * NW <= kMaxTiles &&
                        (!a.states || 1 + words <= S);          // the place of a table row each
    if (tid == 0) {
        a.status[i] = st; a.done[i] = st != 0 || run_it ? 3 : 0;
        if (st == 0 && !run_it) atomicOr(a.path + 3, kPathRest);
    }
    if (!run_it) {
        if (warp == NW) cp_async_wait<0>();                     // nothing may land in shared memory that is no longer ours
        return;
    }
    if (classes) {
        for (int x = tid; x < kClassMax * KC; x += NT) {
            const int k = x / KC, q = x - k * KC;
            int v = 0;
            if (k < Kr && q < Kc) v = stage[s_rep[k] * TP + s_rep[kClassMax + q]];
            if (form == kPacked) reinterpret_cast<uint16_t*>(tsm)[x] = (uint16_t)v;
            else tsm[x] = v;
        }
    } else {
        for (int s = tid; s < S; s += NT) { s_order[s] = s; s_rcls[s] = s; s_ccls[s] = s; }
        // the matrix paid between layers 0 and 1; with one matrix per layer, matrix l sits in buffer l & 1
        const int32_t* const T = T0 + (a.trans_layer ? a.trans_layer : 0);
        int32_t* const dst = tsm + (a.trans_layer ? S * KC : 0);
        for (int x = tid; x < S * KC; x += NT) {
            const int r = x / KC, s = x - r * KC;
            int v = 0;
            if (s < S && Li > 1) v = T[r * S + s];
            if (form == kPacked) reinterpret_cast<uint16_t*>(dst)[x] = (uint16_t)v;
            else dst[x] = v;
        }
        if (a.trans_layer)
            for (int x = tid; x < S * KC; x += NT) tsm[x] = 0;  // pad columns of the other buffer
    }
    __syncthreads();                                            // the staged matrix is no longer read

    // ---- records of a layer, by one warp: int4 (where the strategy's differences and bases are read, in bytes from the first guard
    // column on; time; row class); time = +inf where mem exceeds the budget.  Two lists: all strategies in the
    // table's order, for the last layer's values, and those that can matter in the order of their row classes: one whose row and column class has a member that needs no more memory and no more time (and is the lower one
    // where both are equal) never does, as C does not rise with the budget.  ZeRO stages and checkpointing mostly differ in
    // memory alone: about half drop out.
    auto prepare = [&](int l, int from) -> int {                // returns the new frontier
        const int32_t* const rm = raw + (l & 3) * 2 * S4;
        const int32_t* const rt = rm + S4;
        int slot = -1, least = M + 1;
        for (int back = 1; back <= 2 && back <= l && slot < 0; ++back) {          // a layer with the rows of one of the two before it
            const int32_t* const ro = raw + ((l - back) & 3) * 2 * S4;
            int diff = 0;
            for (int s = lane; s < S; s += 32) diff |= (rm[s] != ro[s]) | (rt[s] != ro[S4 + s]);
            if (!__any_sync(0xffffffffu, diff)) slot = s_slot[(l - back) & 3];
        }
        if (slot < 0) {
            unsigned used = 0;
            for (int back = 1; back <= 3 && back <= l; ++back) used |= 1u << s_slot[(l - back) & 3];
            slot = __ffs(~used) - 1;
            int4* const all = rec + slot * S1;
            int4* const keep = rec + (4 + slot) * S1;
            int at = 0;
            for (int e0 = 0; e0 < S; e0 += 32) {
                const int e = e0 + lane;
                bool in = e < S;
                int4 r = make_int4(0, 0, (int)kInf, 0);
                if (in) {
                    const int s = s_order[e], mem = rm[s], t = rt[s], rc = s_rcls[s], cc = s_ccls[s];
                    const bool fits = mem <= M;                 // else +inf everywhere: no shift, time +inf
                    const int at0 = H - (fits ? mem : 0);
                    r = make_int4(form == kWord ? 4 * (cc * Mp + at0) : 4 * ((cc >> 1) * Mp + at0) + 2 * (cc & 1), 4 * at0, fits ? t : (int)kInf, rc);
                    all[s] = r;
                    in = fits;
                    if (classes) {
                        const int first = s_first[rc], n = s_cnt[rc];
                        for (int q = 0; q < n; ++q) {
                            const int o = s_order[first + q], om = rm[o], ot = rt[o];
                            if (s_ccls[o] == cc && om <= mem && ot <= t && (o < s || ot < t)) in = false;
                        }
                    }
                }
                const unsigned b = __ballot_sync(0xffffffffu, in);
                if (in) keep[at + __popc(b & ((1u << lane) - 1u))] = r;
                at += __popc(b);
            }
            if (lane == 0) { s_nkeep[slot] = at; keep[at] = make_int4(4 * H, 4 * H, (int)kInf, 0); }    // none: +inf
        }
        for (int s = lane; s < S; s += 32) least = min(least, rm[s]);
        least = __reduce_min_sync(0xffffffffu, least);
        const int f = min(from + least, M + 1);
        if (lane == 0) { s_front[l & 3] = f; s_slot[l & 3] = slot; }
        __syncwarp();
        return f;
    };
    if (tid == 0) {
        s_rare.S = S; s_rare.M = M; s_rare.m_pitch = Mp; s_rare.all = smem_addr(rec);
        s_rare.C_last = a.C_last + (size_t)i * S * Mp;
        s_rare.states = a.states + (size_t)i * Lmax * S * Mp;
    }
    int front = 0;
    if (warp == NW) {
        cp_async_wait<1>();
        __syncwarp();
        front = prepare(0, 0);
    } else {
        // layer 0 reads a state of zeros: C[0] = time where mem fits
        int32_t* const base = reinterpret_cast<int32_t*>(state);
        for (int x = tid; x < H + Mp; x += 32 * NW) base[x] = x < H ? (int)kInf : 0;
        int4* const d = reinterpret_cast<int4*>(state + base_bytes);
        for (int x = tid; x < (int)(d_bytes / 16); x += 32 * NW) d[x] = make_int4(0, 0, 0, 0);
    }
    __syncthreads();

    if (warp < NW) {
        Ctx c;
        c.rare = &s_rare; c.states = a.states != nullptr; c.Mp = Mp; c.G = G; c.NW = NW; c.Li = Li; c.Kc = Kc; c.tmax = (uint32_t)s_all.tmax;
        c.TM = per_step > NW ? per_warp : 1; c.steps = steps; c.per_step = per_step;
        c.base0 = smem_addr(state); c.d0 = c.base0 + (uint32_t)base_bytes;
        c.base = c.base0 + 4u * H; c.d = c.d0 + 4u * H;
        c.keep = smem_addr(rec + 4 * S1); c.slot_bytes = 16u * S1;
        c.slot = smem_addr(s_slot); c.nkeep = smem_addr(s_nkeep); c.front = smem_addr(s_front); c.hard = smem_addr(s_hard); c.hard_bits = s_hard; c.tags = smem_addr(s_tag);
        c.tsm = smem_addr(tsm); c.tmat = a.trans_layer ? 4u * S * KC : 0u;
        if (a.states)
            for (int s = tid; s < S; s += 32 * NW) a.map[(size_t)i * S + s] = s_ccls[s] + (form == kWord ? kStateWord : kStateHalf);
        if (form == kPacked) {
            if (KC == 8) run<8, kPacked>(c, warp, lane);
            else if (KC == 16) run<16, kPacked>(c, warp, lane);
            else if (KC == 32) run<32, kPacked>(c, warp, lane);
            else run<64, kPacked>(c, warp, lane);
        } else if (form == kHalf) {
            if (KC == 8) run<8, kHalf>(c, warp, lane);
            else if (KC == 16) run<16, kHalf>(c, warp, lane);
            else if (KC == 32) run<32, kHalf>(c, warp, lane);
            else run<64, kHalf>(c, warp, lane);
        } else {
            if (KC == 8) run<8, kWord>(c, warp, lane);
            else if (KC == 16) run<16, kWord>(c, warp, lane);
            else if (KC == 32) run<32, kWord>(c, warp, lane);
            else run<64, kWord>(c, warp, lane);
        }
        return;
    }
    // ---- service warp: the records of layer l + 1 while layer l is searched
    const int elems = S * S;
    for (int l = 0; l + 1 < Li; ++l) {
        if (l + 2 < Li) fetch(l + 2);
        cp_async_commit();
        int32_t* const dst = tsm + ((l & 1) ? S * KC : 0);      // matrix l + 2; matrix l + 1 is in use in this layer
        if (a.trans_layer && l + 2 < Li && form != kPacked) {
            const int32_t* const T = T0 + (size_t)(l + 2) * a.trans_layer;
            for (int x = lane; x < elems; x += 32) {
                const int r = x / S, s = x - r * S;
                cp_async_4(dst + r * KC + s, T + x);
            }
        }
        cp_async_commit();
        cp_async_wait<2>();                                     // the rows of layer l + 1, asked for a layer ago
        __syncwarp();
        front = prepare(l + 1, front);
        if (a.trans_layer && l + 2 < Li) {
            if (form == kPacked) {
                const int32_t* const T = T0 + (size_t)(l + 2) * a.trans_layer;
#pragma unroll 8
                for (int x = lane; x < elems; x += 32) {
                    const int r = x / S, s = x - r * S;
                    reinterpret_cast<uint16_t*>(dst)[r * KC + s] = (uint16_t)T[x];
                }
            }
            cp_async_wait<0>();
            __syncwarp();
        }
        for (int t = 0; t < steps; ++t) {
            cta_barrier();
            if (per_step > NW)                                  // see step_end
                for (int r = rounds_of(*(volatile int*)(s_hard + (l * steps + t) % 3), per_warp, NW); r > 0; --r) cta_barrier();
        }
        cta_barrier();
    }
    cp_async_wait<0>();
}


// host side

// Bytes of the state: `rows` rows of differences of `size` bytes, guard columns for shifts of up to `shift`.
long long state_bytes(const galv_shape* sh, int rows, int size, long long shift)
{
    const long long Mp = sh->m_pitch, H = (shift + 31) / 32 * 32, words = size == 4 ? rows : (rows + 1) / 2;
    return 4 * (H + Mp) + 4 * (H + words * Mp);
}

}  // namespace

bool galv_solo_plan(const galv_ctx* ctx, const galv_shape* sh, bool states, SoPlan* p)
{
    std::memset(p, 0, sizeof(*p));
    if (sh->flags & (GALV_STORE_C_FULL | GALV_STORE_ARGMIN | GALV_KERNEL_REFERENCE | GALV_KERNEL_PER_LAYER | GALV_KERNEL_NO_CLUSTER | GALV_KERNEL_RESIDENT | GALV_KERNEL_CLUSTER | GALV_DEBUG_WITHHOLD_LOAD))
        return false;
    if ((sh->flags >> 16) & 31) return false;                 // GALV_CLUSTER_SIZE
    const int S = sh->S, G = sh->m_pitch / 32, mats = (sh->flags & GALV_TRANS_PER_LAYER) ? 2 : 1;
    if (S > kMaxS || (long long)sh->B * sh->Lmax >= (1ll << 31) || sh->m_pitch > (1 << 16)) return false;
    const int KC = S <= 8 ? 8 : S <= 16 ? 16 : S <= 32 ? 32 : 64;
    const int room_max = ctx->smem_optin - kStaticSmem;
    // Warps: as few as take the column groups in the same number of rounds.
    const int turns = (G + kMaxWarps - 1) / kMaxWarps;
    int nw = (G + turns - 1) / turns;
    if (nw < 4) nw = 4;
    p->nw = nw;
    // What the state may need is not known here: every row in 32 bits if that fits, else 16-bit rows of an unstructured matrix,
    // with room for shifts of an eighth of the budget at least, else those of 9 classes.
    const int rows[4] = {S, S, S, S < 9 ? S : 9}, size[4] = {4, 2, 2, 2}, shift[4] = {sh->M, sh->M, sh->M / 8, sh->M / 13};
    for (int need = S <= kDenseMax ? 0 : 3; need < 4; ++need) {
        p->dense = need < 3;
        if (mats == 2 && !p->dense) return false;
        p->mats = p->dense ? mats * S * KC : 0;
        if (p->mats < kClassMax * 16) p->mats = kClassMax * 16;
        const long long fixed = 128ll * (S + 1) + 32ll * ((S + 3) & ~3) + 4ll * p->mats;
        long long room = state_bytes(sh, rows[need], size[need], shift[need]);
        // the start of a search keeps the lengths and the matrix where the state will be
        if (room < 4ll * kMaxSorted) room = 4 * kMaxSorted;
        if (mats == 1 && room < 4ll * S * (S | 1) && need == 0) room = 4ll * S * (S | 1);
        room = (room + 15) & ~15ll;
        if (fixed + room > room_max) continue;
        p->certain = need == 0 && !states;
        p->smem = need == 0 ? (int)(fixed + room) : room_max;
        p->room = (int)((p->smem - fixed) & ~15ll);
        p->packed = !(sh->flags & GALV_KERNEL_NO_PACKED);
        p->sorted = sh->B > ctx->num_sms && sh->B <= kMaxSorted;
        return true;
    }
    return false;
}

// Whether the look at the tables is worth its launch: not for shapes that every batch is better off elsewhere with, not for a few
// instances (whose layers take clusters a few thousand cycles; and the look's answers want two words an instance), of a few hundred
// columns (step_cycles), nor for batches that are short everywhere.
bool galv_solo_worth(const galv_ctx* ctx, const galv_shape* sh, bool states, int n, const RsPlan resident[2], const ClPlan* pushing, SoPlan* p)
{
    const int S = sh->S, G = sh->m_pitch / 32;
    if (sh->B < 2 * kGuessed || sh->M < 1000) return false;
    SoOther& o = p->other;
    // CTAs an SM holds: four warps of 128 registers a scheduler, and its shared memory
    int per_sm = 16 / (p->nw + 1);
    if (per_sm > (ctx->smem_optin + 1024) / (p->smem + kStaticSmem + 1024)) per_sm = (ctx->smem_optin + 1024) / (p->smem + kStaticSmem + 1024);
    const int slots = ctx->num_sms * (per_sm > 1 ? per_sm : 1), rounds = (sh->B + slots - 1) / slots;
    o.rounds = rounds == 1 ? 1.0f : (float)sh->B / (float)slots + 0.5f;
    o.one_round = rounds == 1;
    o.start = 30000.0f;                                        // the look's launch, and half of this kernel's start, the half that the others do not have
    o.packed = S <= 64 && S % 4 == 0 && !(sh->flags & GALV_KERNEL_NO_PACKED);
    // a tile costs about the same whatever part of it there are columns for
    const int nsg = S < 64 ? (S + 7) / 8 : 8, tile = 16 / nsg * 4, tiles = (sh->M / 32 + tile) / tile * tile;
    o.tiled = 0.9f * (float)(tiles > G ? tiles : G) * (float)sh->B / (float)ctx->num_sms;
    o.most = pushing ? 0.9f * (float)pushing->est : 1e30f;
    if (n && resident[n - 1].dense && 1.5f * (float)resident[n - 1].est < o.most) o.most = 1.5f * (float)resident[n - 1].est;
    if (n && !resident[0].dense) {
        const RsPlan& r = resident[0];
        const int g = r.w / 32;
        o.resident = (float)r.est; o.gints = r.gints; o.w = r.w;
        o.past_halo = kResidentPastHalo * (float)((g + r.nw - 1) / r.nw * r.rounds);
        o.other_one_round = r.rounds == 1;
    }
    auto layer = [&](int KC, bool word, const Passing& pass) {
        const int step = p->nw * max_tile(KC);
        return o.rounds * (float)((G + step - 1) / step) * step_cycles(KC, word, states, pass, 1.0f) + o.start / (float)sh->Lmax;
    };
    // No batch of this shape is worth it: few strategies pass, and elsewhere it goes as badly as it can.
    const int KC = S <= 8 ? 8 : S <= 16 ? 16 : S <= 32 ? 32 : 64;
    const float s1 = (float)S, few = 0.7f;
    auto at_most = [&](float a) { return a < o.most ? a : o.most; };
    const float tiled = at_most(o.tiled * (tiled_cycles(S, false, (float)S) > tiled_cycles(S, true, 0.0f) ? tiled_cycles(S, false, (float)S) : tiled_cycles(S, true, 0.0f)));
    const float classes = o.w ? at_most(o.resident * kResidentDiffers + o.past_halo * (float)S) : tiled;
    p->dense = p->dense && layer(KC, false, Passing{s1, few, 0.0f, 0.0f}) <= kGuessTaken * tiled;
    const bool some = layer(8, false, Passing{s1 / 3.0f, few, 0.0f, 0.0f}) <= kGuessTaken * classes;
    if (!p->dense && !some) return false;
    // The look at the batch, 15 to 20 us where it is turned away, has to be small beside it.
    const float lowest = o.packed && tiled_cycles(S, true, 0.0f) < tiled_cycles(S, false, 0.0f) ? tiled_cycles(S, true, 0.0f) : tiled_cycles(S, false, 0.0f);
    const float least_tiled = at_most(o.tiled * lowest), least_classes = o.w ? at_most(o.resident * kResidentRepeats) : least_tiled;
    if ((p->dense && (!some || tiled > classes) ? tiled : classes) * (float)sh->Lmax < 800e3f) return false;
    if ((some && (!p->dense || least_classes < least_tiled) ? least_classes : least_tiled) * (float)sh->Lmax < 300e3f) return false;
    p->guessed = kGuessed;
    // Every batch of this shape is, whatever it holds.
    const float least = least_classes < least_tiled ? least_classes : least_tiled;
    bool all = p->certain && p->dense;
    for (int k = 8; k <= KC; k <<= 1) all = all && layer(k, true, Passing{s1, s1, 1.0f, s1}) <= kGuessTaken * least;
    p->certain = all;
    if (all) p->guessed = 0;
    return true;
}

cudaError_t galv_solo_configure(galv_ctx* ctx)
{
    return cudaFuncSetAttribute(solo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->smem_optin - kStaticSmem);
}

cudaError_t galv_solo_launch(const SoPlan& p, const DpArgs& d, cudaStream_t st)
{
    if (p.guessed) {
        GuessArgs g;
        g.B = d.B; g.Lmax = d.Lmax; g.S = d.S; g.M = d.M; g.n = p.guessed;
        g.nw = p.nw; g.groups = d.m_pitch / 32; g.dense = p.dense; g.states = d.lean_map != nullptr; g.room = p.room;
        g.other = p.other;
        g.L = d.L; g.time_q = d.time_q; g.mem_q = d.mem_q; g.trans_q = d.trans_q; g.trans_inst = d.trans_inst; g.trans_layer = d.trans_layer;
        g.guess = reinterpret_cast<float2*>(d.order); g.ticket = reinterpret_cast<int32_t*>(d.work);
        guess_kernel<<<p.guessed, kGuessThreads, 0, st>>>(g);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    SoArgs a;
    a.B = d.B; a.Lmax = d.Lmax; a.S = d.S; a.M = d.M; a.m_pitch = d.m_pitch;
    a.NW = p.nw; a.room = p.room; a.mats = p.mats; a.sorted = p.sorted; a.dense = p.dense;
    a.guessed = p.guessed; a.guess = reinterpret_cast<const float2*>(d.order);
    a.packed = p.packed; a.certain = p.certain;
    a.L = d.L; a.time_q = d.time_q; a.mem_q = d.mem_q; a.trans_q = d.trans_q;
    a.trans_inst = d.trans_inst; a.trans_layer = d.trans_layer;
    a.C_last = d.C_last; a.states = d.lean_map ? reinterpret_cast<uint32_t*>(d.C) : nullptr; a.map = d.lean_map;
    a.status = d.status; a.path = d.err; a.done = d.done;
    solo_kernel<<<d.B, (p.nw + 1) * 32, p.smem, st>>>(a);
    return cudaGetLastError();
}
