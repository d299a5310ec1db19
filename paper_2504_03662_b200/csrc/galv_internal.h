// Internal declarations shared by the translation units of libgalv.so.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "galv.h"

constexpr int kStateHalf = 1 << 16, kStateWord = 1 << 17;      // DpArgs::lean_map: states of bases and 16-bit (two rows a word) or 32-bit differences
// Which kernel ran: 1 the tiled kernels' packed loop, 0 their 32-bit one, these two, and with kPathRest the solo kernel has left something to
// the cluster kernels behind it (the tiled ones write their own).
constexpr int kPathCluster = 2, kPathSolo = 3, kPathRest = 4;
constexpr int kResidentClassMax = 16;      // classes beyond which a matrix counts as unstructured in the resident kernel

// How the resident kernel (one thread-block cluster per instance, the state between layers in shared memory) cuts an instance.
struct RsPlan {
    int cl;        // CTAs per cluster
    int w;         // budget columns per CTA (multiple of 32)
    int nw;        // compute warps per CTA
    int gints;     // words of one state buffer
    int dense;     // the state of an unstructured matrix (S rows and the matrix itself) fits: every instance can run
    int smem;      // dynamic shared memory bytes
    int sorted;    // clusters take the instances longest first
    int halo_fits, rounds;
    int stage;     // a layer's rows are collected in shared memory and leave with one tensor store
    int stage_at;  // word offset of the collected rows
    int follow;    // the pushing cluster kernel stands behind this launch: what it does better is left to it
    int k_max;     // ... instances of more classes
    double est;    // estimated SM cycles per layer, all rounds of clusters
};

// What a layer of a batch costs in the other kernels, in SM cycles, and what the solo kernel's own multiplies with.
struct SoOther {
    float resident;       // matrices of few classes, by the resident kernel's plan
    int gints, w;         // ... its room and columns (w = 0: it does not take them)
    float past_halo;      // ... for each strategy, where shifts pass the halo
    float tiled;          // the tiled kernels, for a cycle of a column group
    int packed;           // ... their packed loop is possible
    float most;           // the pushing kernel, or the resident one for any matrix
    float rounds;         // of instances on the solo kernel
    float start;          // its own start, once
    int one_round, other_one_round;        // all instances run at once, here, in the resident kernel
};

// How the solo kernel (an instance's state on one SM) cuts a batch.
struct SoPlan {
    int nw;        // compute warps per CTA
    int mats;      // words of the transition matrices in shared memory
    int smem;      // dynamic shared memory bytes
    int room;      // ... of which for the state
    int sorted;    // CTA c takes the c-th longest instance
    int dense;     // unstructured matrices fit, with transition entries up to 65535 at least
    int certain;   // every instance can run, and is worth it
    int packed;    // packed relaxations are allowed
    int guessed;   // instances that are looked at to see whether the batch is worth it; 0: it is
    SoOther other;
};

struct galv_ctx {
    int device;
    int num_sms;
    int smem_optin;      // max dynamic shared memory per block (bytes)
    int max_resident;    // the same for the resident kernel
    int max_cluster;     // largest thread-block cluster the cluster kernel may be launched with (8 portable, 16 where allowed)
    int profiling;       // record an event pair around the layer launches of every search
    int prof_count;      // searches profiled since profiling was switched on
    cudaEvent_t pev[2 * 64];   // ring of event pairs: search k uses pev[2*(k%64)], pev[2*(k%64)+1]
    galv_shape plan_shape;     // the resident kernel's plan for the shape of the last search
    RsPlan plans[2];
    int plan_launches, plan_valid;
    char err[512];
};

// How one layer of the recurrence is cut into work items (host-chosen, passed to the kernels).
struct DpPlan {
    int tm;        // 32-column groups per warp (register tile height)
    int sb;        // strategies per item (s-block), multiple of 8
    int nsb;       // s-blocks
    int nsg;       // warps along s  (= sb / 8)
    int nms;       // warps along m
    int tmb;       // budget columns per item = nms * 32 * tm
    int ks;        // previous-layer strategies staged per pipeline stage
    int nkc;       // chunks per item = ceil(S / ks)
    int nst;       // pipeline stages in shared memory
    int tma_t;     // trans rows are 16-byte aligned: staged by a tiled TMA box, else by plain copies
    int ntiles_m;  // ceil((M+1) / tmb)
    int threads;   // (nsg * nms + 4) * 32: consumer warps, producer, helper, store and publisher warps
    int smem;      // dynamic shared memory bytes
    int grid;      // resident CTAs
    int p16;       // the packed 16-bit path is possible for this shape (whether the costs allow it is known on the device)
    int p16_smem;  // its dynamic shared memory bytes
};

struct DpArgs {
    int B, Lmax, S, M, m_pitch;
    const int32_t* L;
    const int32_t* time_q;
    const int32_t* mem_q;
    const int32_t* trans_q;
    long long trans_inst;   // entries per instance in trans_q: S*S, or Lmax*S*S with one matrix per layer
    long long trans_layer;  // entries between the matrices of consecutive layers: 0 or S*S
    int32_t* C;          // full table or NULL
    uint8_t* A;          // argmin table or NULL
    int32_t* C_last;
    int32_t* roll;       // [2][B][S][m_pitch] when C == NULL
    int32_t* order;      // [B]   valid instances, longest first; before that, what the solo kernel would cost some of them
    int32_t* nactive;    // [Lmax+1] instances with L > l
    int32_t* scratch;    // [2*(Lmax+2)] histogram / fill counters, then the work counters below (zeroed together)
    unsigned long long* work;  // [Lmax+2] next item to hand out: [0] when all layers are one launch, else [l]
    long long* istart;   // [Lmax+1] items of the layers before l (layer 1 starts at 0); [Lmax] = all items
    int32_t* err;        // device error flag
    int32_t* tile_done;  // [B][ntiles_m] finished items per (instance, tile); NULL when layers are separate launches
    int32_t* maxmem;     // largest mem over the valid instances (min(.., M+1)); [1] largest trans entry; [2] 1: packed 16-bit path;
                         // [3] 1: trans_k holds shifted entries (keyed argmin loop); [4] 1: a quarter of the rows or more look dominated;
                         // [5], [6]: 64-bit count behind that
    uint32_t* trans_p;   // packed pairs of trans rows for the 16-bit path: [B][(Lmax)][S/2][S], entry = T[2q][s] | T[2q+1][s] << 16
    int32_t* trans_k;    // argmin table with keys: copy of trans_q with every entry << 6 (same place in the workspace as trans_p;
                         // a plain copy when the entries are too large for keys: maxmem[3] says which)
    int keyed_multi;     // the keys-only argmin kernel has been launched over all layers: launches per layer return when it ran
    int keyed;           // the shape allows the keyed argmin loop (S <= 64, all rows of a tile in one stage)
    int32_t* minmem_l;   // [Lmax+1] smallest mem of each layer over the valid instances
    int32_t* front;      // [B][Lmax] feasibility frontier (sum of the layers' smallest mem), or NULL when tiles are never skipped
    int32_t* ntiles;     // [Lmax+1] tiles per instance that can store anything in layer l
    int32_t* tcount;     // [Lmax][ntiles_m] layers 1..l whose items include tile t
    int32_t* status;
    int32_t* lean_map;   // host entry point (nobody sees the table): [B][S] state row of each strategy where the resident kernel has left
                         // the states between the layers in C in place of its values (with kStateHalf or kStateWord added: the solo
                         // kernel); -1 where C holds the values.  Else NULL
    int32_t* done;       // [B] 1: searched or flagged already, 3: by a kernel that has ended, 2: an unstructured matrix, not searched; or NULL when
                         // neither the resident nor the solo kernel was launched.
                         // Lies over tile_done: read until the schedule is made
    int withhold;        // test hook: CTA 0 never loads its first chunk, so that the bounded waits run out
    int after_solo;      // the solo kernel has run: done[] = 3 are its own
    int beside;          // the pushing kernel may start beside the kernel in front, the resident one
    int skip_dom;        // leave out rows (packed path: row pairs) that cannot win in any column of a warp group's tile
    int dom_auto;        // ... where a quarter of the rows or more look it (maxmem[4])
};

// records `text` as the context's last error and returns `code`
int galv_set_error(galv_ctx* ctx, int code, const char* text);

// workspace carve-up (offsets in bytes, all 256-aligned)
struct WsLayout { size_t order, done, nactive, scratch, err, minmem_l, ntiles, istart, tcount, front, tile_done, trans_p, roll, total; };
WsLayout galv_ws_layout(const galv_shape* sh);

// Tensor map of an int32 table [rows][m_pitch] seen as [rows][m_pitch / 32][32], box [box_rows][box_groups][32].
cudaError_t galv_encode_table_3d(CUtensorMap* map, void* base, size_t rows, int m_pitch, int box_rows, int box_groups);

// whether it can take the shape, which has no table to write; states: they are kept in its place
bool galv_solo_plan(const galv_ctx* ctx, const galv_shape* sh, bool states, SoPlan* plan);
cudaError_t galv_solo_configure(galv_ctx* ctx);
// whether a batch of some matrices can be worth it, given what the others' plans cost; n: of the resident kernel's launches; pushing: NULL when it cannot run the shape
bool galv_solo_worth(const galv_ctx* ctx, const galv_shape* sh, bool states, int n, const RsPlan resident[2], const struct ClPlan* pushing, SoPlan* plan);
cudaError_t galv_solo_launch(const SoPlan& plan, const struct DpArgs& a, cudaStream_t st);
// done[i] = 2 where no two of the first rows of a matrix are equal, else 0, but for those the solo kernel has finished; for the strategies that galv_probe_applies to
bool galv_probe_applies(const struct DpArgs& a);
void galv_probe_matrices(const struct DpArgs& a, cudaStream_t st);

// launches to make (0: the shape is left to the other kernels); the last one takes every instance when it is dense
// pushing: the plan of the pushing cluster kernel, which takes what is left; NULL when it cannot run the shape
int galv_resident_plan(galv_ctx* ctx, const galv_shape* sh, const struct ClPlan* pushing, RsPlan plans[2]);
cudaError_t galv_resident_configure(galv_ctx* ctx);
cudaError_t galv_resident_launch(const RsPlan& plan, int second, const struct DpArgs& a, cudaStream_t st);

// How the pushing cluster kernel (small batches of unstructured matrices: one thread-block cluster per instance) cuts an instance.
struct ClPlan {
    int cl;        // CTAs per cluster
    int w;         // budget columns per CTA (multiple of 32)
    int g;         // w / 32
    int nsg;       // ceil(S / 8)
    int sp8;       // nsg * 8
    int tm;        // 32-column groups per warp register tile
    int nct;       // column tiles per CTA
    int units;     // nct * nsg work units per CTA and layer
    int nw;        // warps per CTA
    int smem;      // dynamic shared memory bytes
    int sorted;    // clusters take the instances longest first
    double est;    // estimated SM cycles per layer
};
bool galv_cluster_plan(const galv_ctx* ctx, const galv_shape* sh, ClPlan* plan);
cudaError_t galv_cluster_configure(galv_ctx* ctx);
cudaError_t galv_cluster_launch(galv_ctx* ctx, const galv_shape* sh, const ClPlan& plan, const struct DpArgs& a, cudaStream_t st);

bool galv_dp_make_plan(const galv_ctx* ctx, const galv_shape* sh, DpPlan* plan);
cudaError_t galv_dp_configure(const galv_ctx* ctx);
cudaError_t galv_dp_launch(galv_ctx* ctx, const galv_shape* sh, const DpArgs& a, cudaStream_t st);
inline long long galv_trans_layer(const galv_shape* sh) { return (sh->flags & GALV_TRANS_PER_LAYER) ? (long long)sh->S * sh->S : 0; }
inline long long galv_trans_inst(const galv_shape* sh) { return (long long)sh->S * sh->S * ((sh->flags & GALV_TRANS_PER_LAYER) ? sh->Lmax : 1); }
cudaError_t galv_backtrack_launch(const galv_shape* sh, const int32_t* L, const int32_t* time_q,
                                  const int32_t* mem_q, const int32_t* trans_q, const int32_t* C,
                                  const uint8_t* A, const int32_t* C_last, const int32_t* lean_map, const int32_t* budget,
                                  int32_t* opt_cost, int32_t* plan, int32_t* mem_used, int32_t* status,
                                  cudaStream_t st);
cudaError_t galv_costs_launch(const galv_shape* sh, const int32_t* L, const galv_layer_desc* layers,
                              int64_t layer_stride_B, const galv_strategy_desc* strat,
                              const galv_inst_params* inst, double* time_s, double* mem_bytes,
                              int32_t* time_q, int32_t* mem_q, int32_t* trans_q, int32_t* status,
                              cudaStream_t st);
cudaError_t galv_probe_launch(const galv_ctx* ctx, int kind, int iters, int32_t* sink, cudaStream_t st,
                              long long* ops);
