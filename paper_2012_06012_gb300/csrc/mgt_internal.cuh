// Internal declarations shared by the mgt kernels and the host library.
//
// Pipeline of one transpose (the paper's LocalTranspose o ViewSwap, Sec. 3,
// realised as a two-level stable counting sort by column):
//   K0 prep       zeroes, end points, source-block cell offsets, row table, sentinels
//   K1 hist       per scatter tile, cell counts per column bucket (shared-memory histogram)
//   K2 scan_tiles per bucket, exclusive prefix over tiles (stable tile order); its last
//                 block: bucket bases (exclusive prefix over buckets)
//   K3a scatter   stable scatter of 12/16-byte cell records into <= 256
//                 super-buckets (high bits of the bucket id); P x P counts (the
//                 view swap's count matrices, Sec. 3) of aligned row blocks
//   K3b scatter2  stable split of each super-bucket into its buckets
//   K4 build_work value bases per bucket and the sort work list
//   K5/K6         per-column counts and cursors of the chunks of oversized buckets
//   K7a/K7b place one block per bucket or chunk: stable in-shared-memory split by
//                 column, coalesced output of row_ptr', col_idx', cell_ptr' and each
//                 run's source offset (plans that ask for sort clusters: one
//                 thread-block cluster per bucket, K7c for skewed ones)
//   K9 parts      P x P counts from the output, for all other row blocks
//   K8 copy       every value run, in output order, internal order kept
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/mgt.h"

namespace mgt {

// ------------------------------------------------------------ status word
// First bytes of every workspace: error bits written by the kernels.
enum : unsigned {
    ST_BADINPUT = 1u,  // column out of range, decreasing pointers, wrong totals
    ST_OVERFLOW = 2u,  // an internal per-tile limit was exceeded
    ST_TIMEOUT = 4u,   // a bounded wait expired
    ST_DEBUG_BOUNDS = 8u,  // debug builds: an access outside its array was caught and skipped
};
struct DevHeader {
    unsigned status;
    unsigned pad0;
    unsigned long long scan_done;      // K2 blocks that have written their bucket totals
    unsigned long long n_items;        // written by K4
    unsigned long long n_multi_items;  // written by K4
    unsigned long long n_multi_buckets;// written by K4
    unsigned long long n_fallback;     // buckets K7a left to K7c
    unsigned long long dbg_line;       // debug builds: source line of the first bad access,
    unsigned long long dbg_index;      //   its index
    unsigned long long dbg_bound;      //   and the bound it broke
    unsigned long long max_items;      // written by K4: fallback list capacity (debug checks)
    unsigned long long max_rows;       // written by K4: cursor rows of the chunk path
    unsigned long long unused[5];
};
static_assert(sizeof(DevHeader) <= 256, "header");

// ------------------------------------------------------------ records
// A cell record carries what the sort and the copy need: source row i (the
// output column index), the start of the value run, the column inside its
// bucket and the run length (clamped at 0xFFFF; longer runs are recovered
// from cell_ptr by binary search).
constexpr uint32_t LEN_ESC = 0xFFFFu;
struct RecC { uint32_t i, start, meta; };            // 12 bytes, V < 2^32
struct RecW { uint32_t i, meta; unsigned long long start; };  // 16 bytes
__host__ __device__ inline uint32_t pack_meta(uint32_t cl, uint64_t len) {
    return (cl << 16) | (uint32_t)(len < LEN_ESC ? len : LEN_ESC);
}

// ------------------------------------------------------------ work items
struct WorkItem {
    unsigned long long r0, r1;  // record range (global record indices)
    unsigned long long mc;      // row of the chunk-cursor matrix, or ~0 for single-chunk buckets
    uint32_t bucket;
    uint32_t chunk;             // chunk index inside its bucket
};
struct MultiBucket {
    unsigned long long mc0;     // first cursor-matrix row
    uint32_t bucket, nch;
    uint32_t done, pad;         // column slices that K6 has finished
};
// hist: a chunk's (cells, values) per column; scan: those of the bucket's earlier
// chunks, and in the first chunk's row (which has none) the column's start.
struct Cursor {
    uint32_t a, blo, bhi;
    __host__ __device__ Cursor() {}
    __host__ __device__ Cursor(uint32_t x, unsigned long long y) : a(x), blo((uint32_t)y), bhi((uint32_t)(y >> 32)) {}
    __host__ __device__ unsigned long long b() const { return (unsigned long long)bhi << 32 | blo; }
};

// ------------------------------------------------------------ launch params
struct Params {
    // problem
    int64_t R, N, C, V;
    int o;           // offset bytes
    int s;           // payload stride (1 for variable-width values)
    int P;
    int var;         // 1: variable-width values (byte offsets per value)
    int pp_out;      // 1: P x P counts by the pass over the output (else by the scatter pass)
    int pp_aligned;  // 1: every super-bucket lies in one row block
    int64_t nbytes;  // variable-width values: total bytes (set per call)
    // tiles
    int bshift;      // log2 columns per bucket
    int64_t B;       // buckets
    int tile;        // cells per K1/K3 tile
    int64_t T;       // tiles
    int cs;          // cluster size
    int cap;         // records per K7 CTA
    int64_t ch;      // records a sort cluster takes = cs * cap
    int chm;         // records per chunk of an oversized bucket (one CTA)
    int p2;          // bits of the bucket id handled by the second scatter pass (0: one pass)
    int item2;       // records per second-pass item, about
    bool wide_mid;   // wide records between the scatter passes (bshift + p2 > 16)
    int wide;        // 1: 16-byte records
    int unroll;      // copy unroll
    int cshift;      // log2 output cells per value-copy tile
    const long long *off_host;  // host address of the row-block offsets (read at launch; null: already in place)
    // derived bounds
    int64_t max_items, max_multi_rows, max_multi_buckets;
};

struct WsLayout {
    size_t header, cnt, bucket_tot, bucket_base, bucket_vtot, bucket_vbase, items, multi_items,
        multi_buckets, mc, recs, recs1, src, fallback, pcoff, poff, dblock, vblk, total;
};

struct Inputs {
    const void *row_ptr;
    const int32_t *col;
    const void *cell_ptr;
    const uint8_t *values;
    const long long *val_off;  // variable-width values: byte offset of each value (V + 1)
};
struct Outputs {
    void *row_ptr;
    int32_t *col;
    void *cell_ptr;
    uint8_t *values;
    long long *part_cells, *part_values;
    long long *val_off;        // variable-width values: output byte offsets (V + 1)
};

// pointers into one workspace
struct Ws {
    DevHeader *hdr;
    uint32_t *cnt;          // [T][B]
    unsigned long long *bucket_tot, *bucket_base, *bucket_vtot, *bucket_vbase;
    WorkItem *items;
    uint32_t *multi_items;  // indices of multi-chunk items
    MultiBucket *multi_buckets;
    Cursor *mc;             // [rows][w]
    void *recs;
    void *recs1;            // records after the first scatter pass (super-bucket order)
    void *src;              // per output cell: start of its value run in the input
    uint32_t *fallback;     // items K7a could not place
    long long *pcoff;       // P+1 cell offsets of the source blocks
    long long *poff;        // P+1 row offsets
    uint16_t *dblock;       // [B] destination block of each bucket (0xFFFF: spans two)
    unsigned long long *vblk;  // variable-width values: per-tile words of the chained byte scan, then a tile counter
};

// Row of every 2^ROWAT_SHIFT-th cell (K0, for the scatter pass), the last
// cell's row past the end.  It lies in the region of src, which is written only
// after the scatter passes (4 bytes a cell and at least 256 bytes: larger).
constexpr int ROWAT_SHIFT = 7;
__host__ __device__ inline int64_t row_table_entries(int64_t C) {
    return ((C + (1 << ROWAT_SHIFT) - 1) >> ROWAT_SHIFT) + 1;
}
__host__ __device__ inline uint32_t *row_table(const Ws &ws) { return static_cast<uint32_t *>(ws.src); }

// One matrix's launch context: problem and tile choice, its buffers and its
// workspace.  A kernel takes it by value for one transpose, or finds it in a
// device table when one launch serves a batch of matrices (BatchArgs).
struct Mat {
    Params p;
    Inputs in;
    Outputs out;
    Ws ws;
};

// Batch launch.  Phases with per-matrix grids: blocks [bstart[i],
// bstart[i + 1]) work on tab[i] as if they were a grid of their own.
// Persistent phases: the work units (items, groups of cells) of all members
// back to back, member i owning units [uprefix[i], uprefix[i + 1]), dealt
// to the whole grid.  n = 0: one matrix, passed by value.
struct BatchArgs {
    const Mat *tab;
    const uint32_t *bstart;
    const unsigned long long *uprefix;
    int n;
    bool late;  // not to be launched early (launch_kernel)
};

// One pipeline phase: the blocks it needs for one matrix (0: nothing to do;
// `share` = the matrix's share of the GPU for persistent grids, 1 when
// alone), its dynamic shared memory per block, and its launch (template
// dispatch on m0's formats; grid and smem cover the whole batch).
// Persistent phases also give, per matrix, a host bound on their work units
// (units != nullptr) and the grid that fills the GPU for `total` units of a
// batch; their batch launches deal units instead of blocks.
struct PhaseOps {
    const char *name;
    long long (*grid)(const Params &p, double share);
    size_t (*smem)(const Params &p);
    cudaError_t (*launch)(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                          cudaStream_t st);
    long long (*units)(const Params &p);
    long long (*full_grid)(const Params &p, long long total);
};

WsLayout layout_for(const Params &p);
int default_params(const mgt_desc *d, Params *p, bool compact = false);
Ws ws_from(void *base, const WsLayout &L);

// the pipeline, in order (phase 0 = setup); defined with the kernels
constexpr int kPhases = 14;
const PhaseOps &phase_op(int i);
extern const char *const kPhaseNames[kPhases];
int kernel_launches(const Params &p);
// phases 0-3 and 6 (k_bucket.cu), 4-5 (k_scatter.cu), 7-11 (k_place.cu), 12
// (k_parts.cu), 13: the value copy (k_place.cu, last entry of kPlacePhases)
extern const PhaseOps kBucketPhases[5];
extern const PhaseOps kScatterPhases[2];
extern const PhaseOps kPlacePhases[6];
extern const PhaseOps kPartsPhase;
// P x P counts from the output (k_parts.cu): up to this many row blocks, and
// whether a plan with these row-block offsets uses that pass.
constexpr int PC_MAX_PARTS = 2048;
bool parts_from_output(const Params &p, const long long *off, int *pp_aligned);
// Row-block offsets (P + 1) that travel as a parameter of the set-up kernel.
constexpr int PREP_OFF = 256;
size_t sort_smem_bytes(const Params &p, int cap);
int sort_cap_max();
size_t cluster_smem_bytes(const Params &p);
// The value copy of a variable-width plan (k_var.cu): per tile of output
// cells, the runs' byte sizes, the tile's byte base by a chained scan over the
// tiles, then the byte copy and the output value offsets.
constexpr int VAR_MIN_SHIFT = 6;  // log2 of the fewest cells of such a tile
cudaError_t launch_var_copy(const Mat &m, cudaStream_t st);
// Output cells of a value-copy tile (log2), by the cells of the launch and the mean run.
constexpr int COPY_MIN_SHIFT = 5;  // the fewest
int copy_shift(long long C, double run, int least);
inline double run_bytes(const Params &p) { return p.C > 0 ? (double)p.V * (double)p.s / (double)p.C : 0.0; }
// The kernel sequence of one transpose (everything after the workspace
// header is cleared and the row-block offsets are in place).  ev: optional
// events, ev[i] recorded after phase i (phase 0 = prep).
// Phases [first, last) of one transpose on st (ev: optional per-phase events).
int enqueue_kernels(const Params &p, const Inputs &I, const Outputs &O, const Ws &ws,
                    cudaStream_t st, cudaEvent_t *ev, int first = 0, int last = kPhases);
size_t scatter_smem_bytes(const Params &p);
// Whether the scatter pass counts P x P for a plan (row blocks, and the
// output pass not chosen): batch members differing in it launch apart.
__host__ __device__ inline bool scatter_counts_pp(const Params &p) { return p.P > 1 && !p.pp_out; }

int sm_count();

}  // namespace mgt

struct mgt_plan_s {
    mgt_desc desc;
    mgt::Params p;
    mgt::WsLayout L;
    mgt_tile_cfg cfg;
    long long *part_off_pinned;  // P + 1 row offsets (pinned host memory when available)
    bool pinned;
};

namespace mgt {
// Remembers (per host thread) the last failed CUDA call for mgt_last_error;
// returns MGT_ECUDA.
int note_cuda(cudaError_t e, const char *where);
// Batched launches (mgt_batch.cu): the launch-group key of a plan, the size
// of a batch's table region, and an enqueue that stages the tables through
// caller-provided pinned host memory (never blocks the host).
unsigned long long batch_group_key(const Params &p);
size_t batched_table_bytes(int n, mgt_plan_t *const *plans);
size_t batched_table_bound(int n, int max_parts);  // any n members of <= max_parts blocks
int batched_enqueue(int n, mgt_plan_t *const *plans, const mgt_xcsr_in *in, mgt_xcsr_out *out,
                    void *workspace, size_t workspace_bytes, cudaStream_t st, void *staging,
                    size_t staging_bytes);
// Argument checks shared by the single and batched calls.
int check_call(const mgt_plan_t *plan, const mgt_xcsr_in *in, const mgt_xcsr_out *out,
               const void *workspace, size_t workspace_bytes);
}  // namespace mgt

// ------------------------------------------------------------ device helpers
#ifdef __CUDACC__
namespace mgt {

// Launches one kernel of the pipeline.  Unless it is a batch's or a values-only
// call's (late), or has more than OVERLAP_GRID blocks, it may start while the
// kernel before it in the stream finishes: every kernel begins with
// pipeline_wait(), which returns once that kernel is complete and its writes
// are visible, so only launch latency overlaps (what that kernel writes is read
// by plain loads: ldp).  A 1,000-row transpose (ten launches; the memsets, the
// offsets copy and the bucket scan folded into other kernels) took 49 us, 68
// without the overlap; 715K cells 88 us, 100 without.  The line lies at two
// blocks per SM of this GPU's 152: the wait costs each block some 2 us, which
// grids of many short blocks pay again with every wave (overlap for all grids:
// 715K cells 107 us, 852K x 852K of 512 cells a row 28.6 instead of 26.8 ms, 48
// long columns 5.02 instead of 4.16 ms, 2M x 2M 1.80 instead of 1.74 ms).
constexpr unsigned OVERLAP_GRID = 304;
template <typename... KArgs, typename... Args>
static cudaError_t launch_kernel(void (*kern)(KArgs...), bool late, long long grid, int threads, size_t smem,
                                 cudaStream_t st, const Args &...args) {
    if (smem > 32 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = !late && grid <= OVERLAP_GRID ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
// First statement of a kernel: wait for the one before it, then (small grids)
// let the next one's blocks take the places that this one leaves.
template <bool BATCH>
__device__ __forceinline__ void pipeline_wait() {
    if constexpr (!BATCH) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (gridDim.x <= OVERLAP_GRID) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
}

// Offsets by the read-only path, whose contract is data that nothing writes while
// the kernel lives: the inputs, after the first kernel.
template <typename OffT>
__device__ __forceinline__ long long ldo(const void *p, long long i) {
    return (long long)__ldg(reinterpret_cast<const OffT *>(p) + i);
}
// ... by plain loads: what the pipeline writes itself, and what a caller's kernel
// may still write when a first kernel, launched early, becomes resident.
template <typename OffT>
__device__ __forceinline__ long long ldp(const void *p, long long i) {
    return (long long)reinterpret_cast<const OffT *>(p)[i];
}
template <typename OffT>
__device__ __forceinline__ void sto(void *p, long long i, long long v) {
    reinterpret_cast<OffT *>(p)[i] = (OffT)v;
}

__device__ __forceinline__ void flag(DevHeader *h, unsigned bit) { atomicOr(&h->status, bit); }

// Debug builds (-DMGT_DEBUG) check every index against its array before the
// access, record the first violation in the header (dbg_line, dbg_index,
// dbg_bound) and skip the access; release builds compile the checks away.
#ifdef MGT_DEBUG
__device__ __forceinline__ bool dbg_in(DevHeader *h, unsigned long long i, unsigned long long n,
                                       int line) {
    if (i < n) return true;
    if (atomicCAS(&h->dbg_line, 0ull, (unsigned long long)line) == 0ull) {
        h->dbg_index = i;
        h->dbg_bound = n;
    }
    atomicOr(&h->status, ST_DEBUG_BOUNDS);
    return false;
}
#define MGT_IN(h, i, n) dbg_in((h), (unsigned long long)(i), (unsigned long long)(n), __LINE__)
#else
#define MGT_IN(h, i, n) true
#endif

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned r;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
    return r;
}
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
// This warp's index in the block, as a value that the compiler knows to be the
// same for all its lanes (branches on it need no reconvergence).
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// The matrix this block works on, and the block's index and the grid size
// within that matrix's share of the launch.
struct VBlock {
    const Mat *m;
    long long b, g;
};
// BATCH = false: the context is the kernel's own (grid-constant) parameter,
// read straight from the parameter bank.
template <bool BATCH>
__device__ __forceinline__ VBlock vblock(const Mat &m0, const BatchArgs &ba) {
    if constexpr (!BATCH) return VBlock{&m0, (long long)blockIdx.x, (long long)gridDim.x};
    int lo = 0, hi = ba.n;  // bstart[lo] <= blockIdx.x < bstart[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (ba.bstart[mid] <= blockIdx.x) lo = mid;
        else hi = mid;
    }
    return VBlock{ba.tab + lo, (long long)(blockIdx.x - ba.bstart[lo]),
                  (long long)(ba.bstart[lo + 1] - ba.bstart[lo])};
}

// Work units of a persistent phase: j = first, first + stride, ... while
// j < count(matrix) for one matrix (count read from the device each time);
// in a batch, the units of all members back to back, each member's units
// at or beyond its own count skipped.  A caller's units only grow, so the
// member of the last unit (its unit range and count) is kept and the next
// unit usually falls in it or the member after it: no search per unit.
template <bool BATCH>
struct Units {
    const Mat &m0;
    const BatchArgs &ba;
    unsigned long long g, stride;
    const Mat *M = nullptr;
    unsigned long long j = 0;
    int lo = -1;                              // member of the last lookup (batch)
    unsigned long long lo_base = 0, lo_end = 0, lo_count = 0;
    __device__ Units(const Mat &m0_, const BatchArgs &ba_, unsigned long long first,
                     unsigned long long stride_)
        : m0(m0_), ba(ba_), g(first), stride(stride_) {}
    template <typename CountFn>
    __device__ __forceinline__ bool next(CountFn count) {
        if constexpr (!BATCH) {
            if (g >= (unsigned long long)count(m0)) return false;
            M = &m0;
            j = g;
            g += stride;
            return true;
        } else {
            const unsigned long long total = ba.uprefix[ba.n];
            for (; g < total; g += stride) {
                if (lo < 0 || g >= lo_end) {
                    if (lo >= 0 && lo + 2 <= ba.n && ba.uprefix[lo + 2] > g) {
                        ++lo;  // the member after the last one
                    } else {
                        int a = lo < 0 ? 0 : lo, b = ba.n;  // uprefix[a] <= g < uprefix[b]
                        while (b - a > 1) {
                            const int mid = (a + b) >> 1;
                            if (ba.uprefix[mid] <= g) a = mid;
                            else b = mid;
                        }
                        lo = a;
                    }
                    lo_base = ba.uprefix[lo];
                    lo_end = ba.uprefix[lo + 1];
                    lo_count = (unsigned long long)count(ba.tab[lo]);
                }
                const unsigned long long jj = g - lo_base;
                if (jj < lo_count) {
                    M = ba.tab + lo;
                    j = jj;
                    g += stride;
                    return true;
                }
            }
            return false;
        }
    }
};

// Lanes holding the same key as mine, a key being a value below nbins
// (nbins <= 256) or 0xFFFFFFFF for a lane without one, from one vote per key
// bit.  Its cost is the same whatever the keys, where the hardware peer
// match (__match_any_sync) takes longer the more distinct keys a warp holds.
__device__ __forceinline__ unsigned vote_peers(uint32_t key, int nbins) {
    const bool none = key == 0xFFFFFFFFu;
    unsigned m = __ballot_sync(0xffffffffu, none);
    if (!none) m = ~m;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        if ((1 << b) < nbins) {
            const bool bit = (key >> b) & 1u;
            const unsigned bb = __ballot_sync(0xffffffffu, bit);
            m &= bit ? bb : ~bb;
        }
    }
    return m;
}

// lanes whose `bits`-bit digit (bits <= 31) equals mine, among lanes with
// `valid` set (an invalid lane's own mask is meaningless)
__device__ __forceinline__ unsigned digit_peers(unsigned d, int bits, bool valid) {
    const unsigned key = valid ? (d & ((1u << bits) - 1u)) : 0xFFFFFFFFu;
    return __match_any_sync(0xffffffffu, key);
}

// Rank of this lane's key d among the warp's earlier keys of the same digit
// (rounds in order, then lanes), counted in cnt (this warp's own counters).
// The lanes of equal digit find one another through a mask word per digit:
// each sets its bit, all read the word back, the lowest lane adds the group
// to the counter and clears the mask for the next round (group: the word,
// 0 for a lane without a key).  On random digits of 7 or 8 bits this takes
// 16-17 cycles per 32 keys and SM, a vote per digit bit 25-28, the hardware
// peer match 56-60 (27 / 25-28 / 26 when 60 % of the keys are equal).
template <bool ALL>
__device__ __forceinline__ uint32_t warp_rank(uint16_t *cnt, uint32_t *msk, uint32_t d, bool valid,
                                              uint32_t &group) {
    if (ALL || valid) atomicOr(&msk[d], 1u << lane_id());
    __syncwarp();
    uint32_t m = 0, before = 0;
    if (ALL || valid) {
        m = msk[d];
        before = cnt[d];
    }
    const uint32_t lower = m & lanemask_lt();
    group = m;
    __syncwarp();
    if ((ALL || valid) && lower == 0) {
        cnt[d] = (uint16_t)(before + __popc(m));
        msk[d] = 0;
    }
    __syncwarp();
    return before + __popc(lower);
}

// Starts loading records src[0..n) into shared memory by a block of NT threads
// (16-byte asynchronous copies from the 16-byte boundary at or below src to
// the one at or above src + n: inside the records' 256-byte aligned workspace
// region) and returns where record 0 will lie.  wait_tile: this thread's
// copies are done (a barrier makes everyone's visible).
template <int NT, typename Rec>
__device__ __forceinline__ const Rec *start_tile(unsigned char *dst, const Rec *src, int n) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src);
    const unsigned skip = (unsigned)(a & 15);
    const unsigned chunks = (skip + (unsigned)n * (unsigned)sizeof(Rec) + 15u) >> 4;
    const unsigned sd = (unsigned)__cvta_generic_to_shared(dst);
    const char *g = reinterpret_cast<const char *>(a - skip);
    for (unsigned c = threadIdx.x; c < chunks; c += NT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sd + 16u * c), "l"(g + 16u * c) : "memory");
    return reinterpret_cast<const Rec *>(dst + skip);
}
__device__ __forceinline__ void wait_tile() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// 32-bit inclusive sum over the warp: the shuffle's own range predicate
// guards the add (two instructions a step).
__device__ __forceinline__ uint32_t warp_sum_scan(uint32_t v) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile(
            "{\n.reg .u32 t;\n.reg .pred p;\n"
            "shfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n"
            "@p add.u32 %0, %0, t;\n}"
            : "+r"(v)
            : "r"(d));
    return v;
}

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T n = __shfl_up_sync(0xffffffffu, v, d);
        if (lane_id() >= d) v += n;
    }
    return v;
}

// In-place exclusive scan of a[0..n) in shared memory by the whole block;
// returns the total.  scratch: >= 33 elements of T in shared memory.
template <typename T>
__device__ T block_exclusive_scan(T *a, long long n, T *scratch) {
    const int nt = blockDim.x, tid = threadIdx.x;
    long long per = (n + nt - 1) / nt;
    long long lo = (long long)tid * per, hi = lo + per;
    if (lo > n) lo = n;
    if (hi > n) hi = n;
    T sum = 0;
    for (long long i = lo; i < hi; ++i) sum += a[i];
    T incl = warp_inclusive_scan(sum);
    if (lane_id() == 31) scratch[tid >> 5] = incl;
    __syncthreads();
    if (tid < 32) {
        int nw = (nt + 31) >> 5;
        T v = tid < nw ? scratch[tid] : T(0);
        T vi = warp_inclusive_scan(v);
        scratch[tid] = vi - v;
        if (tid == 31) scratch[32] = vi;
    }
    __syncthreads();
    T run = scratch[tid >> 5] + incl - sum;
    for (long long i = lo; i < hi; ++i) {
        T x = a[i];
        a[i] = run;
        run += x;
    }
    T total = scratch[32];
    __syncthreads();
    return total;
}

// Per-(digit, warp) counters of a stable multisplit live warp-major with one
// word of padding per warp: index warp * (nbins + 1) + digit.  The leaders
// of one warp (distinct digits) and the threads of the scan below (one
// digit each) then fall on distinct banks.
__device__ __forceinline__ int wc_at(int digit, int warp, int nbins) {
    return warp * (nbins + 1) + digit;
}

// Turns the counters into exclusive offsets in (digit, warp) order -- the
// order that keeps equal digits in key order -- and writes each digit's
// first position to dstart[0..nbins] (dstart[nbins] = total).  scratch: >= 33
// words of shared memory.  Ends with a barrier.
__device__ __forceinline__ void wc_scan(uint32_t *wc, int nbins, int nwarps, uint32_t *dstart,
                                        uint32_t *scratch) {
    const int nt = blockDim.x, tid = threadIdx.x;
    for (int d = tid; d < nbins; d += nt) {
        uint32_t s = 0;
        for (int w = 0; w < nwarps; ++w) s += wc[w * (nbins + 1) + d];
        dstart[d] = s;
    }
    __syncthreads();
    const uint32_t total = block_exclusive_scan<uint32_t>(dstart, nbins, scratch);
    for (int d = tid; d < nbins; d += nt) {
        uint32_t run = dstart[d];
        for (int w = 0; w < nwarps; ++w) {
            const uint32_t x = wc[w * (nbins + 1) + d];
            wc[w * (nbins + 1) + d] = run;
            run += x;
        }
    }
    if (tid == 0) dstart[nbins] = total;
    __syncthreads();
}

// first index in [lo, hi) whose element is > key (OffT array in global memory)
template <typename OffT>
__device__ __forceinline__ long long upper_bound_g(const void *a, long long lo, long long hi,
                                                   long long key) {
    while (lo < hi) {
        long long mid = (lo + hi) >> 1;
        if (ldo<OffT>(a, mid) <= key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ long long upper_bound_ll(const long long *a, long long lo, long long hi,
                                                    long long key) {
    while (lo < hi) {
        long long mid = (lo + hi) >> 1;
        if (a[mid] <= key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// same, for a table in shared memory (plain loads)
__device__ __forceinline__ long long upper_bound_sm(const long long *a, long long lo, long long hi,
                                                    long long key) {
    while (lo < hi) {
        long long mid = (lo + hi) >> 1;
        if (a[mid] <= key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// true run length of a record (escape: search cell_ptr for the run's cell)
template <typename OffT>
__device__ __forceinline__ unsigned long long rec_len(uint32_t meta, unsigned long long start,
                                                      const void *cell_ptr, long long C, long long V) {
    uint32_t l = meta & 0xFFFFu;
    if (l != LEN_ESC) return l;
    if (C <= 0 || (long long)start >= V) return 0;
    long long k = upper_bound_g<OffT>(cell_ptr, 0, C + 1, (long long)start) - 1;
    if (k < 0) k = 0;
    if (k >= C) k = C - 1;
    long long end = ldo<OffT>(cell_ptr, k + 1);
    if (end > V) end = V;
    return end > (long long)start ? (unsigned long long)(end - (long long)start) : 0ull;
}

}  // namespace mgt
#endif
