// Level 2 of the transpose: per-bucket stable sort by column, output, value copy.
//
// A bucket holds the records of w consecutive columns in input order (K3).
// One block takes one bucket, or one chunk of a bucket too large for a block:
// it loads the records into shared memory, splits them by column and writes
// col_idx', cell_ptr' and each run's source offset in output order; chunks
// start at cursors that K5 and K6 make from per-chunk column counts.  (A plan
// may ask for thread-block clusters instead, whose CTAs exchange records
// through distributed shared memory.)  This is the paper's final "row-column
// ordering" of the received cells (Sec. 3, view swap step 2), with source
// order kept inside each output row.
#pragma once
#include "mgt_internal.cuh"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace mgt {

constexpr int P_THREADS = 512;

// ------------------------------------------------------------ value copy
template <int VEC>
struct VecT;
template <>
struct VecT<16> {
    using T = int4;
};
template <>
struct VecT<8> {
    using T = int2;
};
template <>
struct VecT<4> {
    using T = int;
};
template <>
struct VecT<1> {
    using T = unsigned char;
};

// Adds 1 and the run length of every valid lane to cnt[c] and vs[c] (c < w):
// one atomic pair per lane when a narrow bucket's columns are spread over
// the warp, one per distinct column otherwise (the hot columns of skewed
// inputs would serialize their lanes on one address).  Lengths of
// 2^16 and more (rare) are added one by one there.
template <typename CT>
__device__ __forceinline__ void warp_count_add(CT *cnt, unsigned long long *vs, uint32_t c,
                                               unsigned long long len, bool valid, int w) {
    // every valid lane on one column (the rounds of a hot column): no match
    const unsigned vm = __ballot_sync(0xffffffffu, valid);
    if (vm == 0) return;
    const int first = __ffs(vm) - 1;
    const uint32_t c0 = __shfl_sync(0xffffffffu, c, first);
    if (__all_sync(0xffffffffu, !valid || c == c0)) {
        const unsigned sum = __reduce_add_sync(0xffffffffu, (valid && len < 65536ull) ? (unsigned)len : 0u);
        if (lane_id() == first) {
            atomicAdd(&cnt[c0], (CT)__popc(vm));
            if (sum) atomicAdd(&vs[c0], (unsigned long long)sum);
        }
        if (valid && len >= 65536ull) atomicAdd(&vs[c0], len);
        return;
    }
    // narrow buckets (w <= 128 columns) whose columns are spread over the
    // warp (at most 4 lanes share the first lane's column, or the first
    // other one): one atomic pair per lane, cheaper than grouping the lanes
    // (measured: 64-column buckets 2.5x faster, 512-column ones slower);
    // otherwise one pair per group of equal columns
    const unsigned same0 = __ballot_sync(0xffffffffu, valid && c == c0);
    if (w <= 128 && __popc(same0) <= 4) {
        const unsigned rest = vm & ~same0;
        const uint32_t c1 = __shfl_sync(0xffffffffu, c, rest ? __ffs(rest) - 1 : first);
        if (__popc(__ballot_sync(0xffffffffu, valid && c == c1)) <= 4) {
            if (valid) {
                atomicAdd(&cnt[c], (CT)1);
                if (len) atomicAdd(&vs[c], len);
            }
            return;
        }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? c : 0xFFFFFFFFu);
    const unsigned small = (valid && len < 65536ull) ? (unsigned)len : 0u;
    const unsigned sum = __reduce_add_sync(peers, small);  // each group reduces over itself
    if (valid && (peers & lanemask_lt()) == 0) {
        atomicAdd(&cnt[c], (CT)__popc(peers));
        if (sum) atomicAdd(&vs[c], (unsigned long long)sum);
    }
    if (valid && len >= 65536ull) atomicAdd(&vs[c], len);
}

// Ranks of a warp's records [a, e) among equal bins (bin = bin_of(idx)),
// in rounds of 32 records: per-(bin, warp) counters in wc (padded layout,
// see wc_at), each record's rank written to rank_out[idx].  The peer
// matches of four rounds are issued together so that their latencies
// overlap; the counter updates stay in round order (stability).
template <typename BinFn>
__device__ __forceinline__ void warp_rank_pass(int a, int e, int nbins, uint32_t *wc,
                                               uint32_t *rank_out, BinFn bin_of) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    for (int base = a; base < e; base += 4 * 32) {
        uint32_t bk[4];
        unsigned pk[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = base + u * 32 + lane;
            bk[u] = idx < e ? bin_of(idx) : 0xFFFFFFFFu;
            // up to 64 bins: a vote per bin bit beats the hardware match on
            // spread keys (measured; wider buckets keep the match)
            pk[u] = nbins <= 64 ? vote_peers(bk[u], nbins) : __match_any_sync(0xffffffffu, bk[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = base + u * 32 + lane;
            const bool v = idx < e;
            const unsigned lower = pk[u] & lanemask_lt();
            uint32_t before = 0;
            if (v) before = wc[wc_at(bk[u], warp, nbins)];
            __syncwarp();
            if (v && lower == 0) wc[wc_at(bk[u], warp, nbins)] = before + __popc(pk[u]);
            if (v) rank_out[idx] = before + __popc(lower);
            __syncwarp();
        }
    }
}

// In-place exclusive scan of a[0..n) in shared memory with each warp owning
// a contiguous segment read 32 consecutive words at a time (no bank
// conflicts); returns nothing, ends with a barrier.  scratch: >= 33 words.
__device__ __forceinline__ void block_scan_segmented(uint32_t *a, int n, uint32_t *scratch) {
    const int lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int seg = (((n + nw - 1) / nw) + 31) & ~31;
    const int lo = min(n, warp * seg), hi = min(n, lo + seg);
    uint32_t sum = 0;
    for (int x = lo + lane; x < hi; x += 32) sum += a[x];
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) scratch[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        const uint32_t v = lane < nw ? scratch[lane] : 0u;
        const uint32_t inc = warp_inclusive_scan(v);
        if (lane < nw) scratch[lane] = inc - v;
    }
    __syncthreads();
    uint32_t carry = scratch[warp];
    for (int x0 = lo; x0 < hi; x0 += 32) {
        const int x = x0 + lane;
        const uint32_t v = x < hi ? a[x] : 0u;
        const uint32_t inc = warp_inclusive_scan(v);
        if (x < hi) a[x] = carry + inc - v;
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncthreads();
}

// ------------------------------------------------------- K5 chunk hist
// For chunks of buckets too large for one sort block: per-column cell counts
// and value sums of each chunk, into its row of the cursor matrix.  One block
// per chunk.  A shared-memory add per record and sum; when eight or more lanes
// of a warp share the first lane's column (a hot column's chunk, whose lanes
// would take turns on one word) they add up first.  32-bit sums: a chunk holds
// at most 8,192 records of less than 2^16 values, longer runs are added to the
// 64-bit sums one by one.
constexpr int K5_THREADS = 256;
template <typename OffT, typename Rec, bool BATCH>
__global__ void __launch_bounds__(K5_THREADS)
    k_chunk_hist(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const DevHeader *hdr = M.ws.hdr;
    if ((unsigned long long)vb.b >= hdr->n_multi_items) return;
    const Rec *__restrict__ recs = reinterpret_cast<const Rec *>(M.ws.recs);
    const WorkItem it = M.ws.items[M.ws.multi_items[vb.b]];
    const void *cell_ptr = M.in.cell_ptr;
    const long long C = M.p.C, V = M.p.V;
    const int w = 1 << M.p.bshift, tid = threadIdx.x, lane = tid & 31;
    if (!MGT_IN(M.ws.hdr, it.mc, hdr->max_rows)) return;
    unsigned long long *vl = reinterpret_cast<unsigned long long *>(smem);  // long runs
    uint32_t *cnt = reinterpret_cast<uint32_t *>(vl + w);
    uint32_t *vs = cnt + w;
    for (int c = tid; c < w; c += K5_THREADS) { cnt[c] = 0; vs[c] = 0; vl[c] = 0; }
    __syncthreads();
    const Rec *r = recs + it.r0;
    const int n = (int)(it.r1 - it.r0);
    constexpr int HU = 4;  // loads in flight per thread
    for (int x0 = 0; x0 < n; x0 += HU * K5_THREADS) {
        uint32_t meta[HU];
#pragma unroll
        for (int u = 0; u < HU; ++u) {
            const int x = x0 + u * K5_THREADS + tid;
            meta[u] = x < n && MGT_IN(M.ws.hdr, it.r0 + x, C) ? r[x].meta : 0u;
        }
#pragma unroll
        for (int u = 0; u < HU; ++u) {
            const int x = x0 + u * K5_THREADS + tid;
            bool v = x < n;
            const uint32_t c = meta[u] >> 16;
            uint32_t len = meta[u] & 0xFFFFu;
            if (v && len == LEN_ESC) {
                atomicAdd(&vl[c], rec_len<OffT>(meta[u], r[x].start, cell_ptr, C, V));
                len = 0;
            }
            const uint32_t c0 = __shfl_sync(0xffffffffu, c, 0);
            const unsigned same = __ballot_sync(0xffffffffu, v && c == c0);
            if (__popc(same) >= 8) {
                const uint32_t sum = __reduce_add_sync(0xffffffffu, v && c == c0 ? len : 0u);
                if (lane == 0) {
                    atomicAdd(&cnt[c0], (uint32_t)__popc(same));
                    atomicAdd(&vs[c0], sum);
                }
                v = v && c != c0;
            }
            if (v) {
                atomicAdd(&cnt[c], 1u);
                atomicAdd(&vs[c], len);
            }
        }
    }
    __syncthreads();
    Cursor *row = M.ws.mc + it.mc * (unsigned long long)w;
    for (int c = tid; c < w; c += K5_THREADS) {
        row[c] = Cursor(cnt[c], vl[c] + vs[c]);
    }
}

// ------------------------------------------------------- K6 chunk scan
// Per large bucket and column: the cells and values of its earlier chunks, in
// place of each chunk's own, and in the first chunk's row (which has none
// before it) the column's first output cell and value; row_ptr' of the
// bucket's columns.  The kernel lasts as long as the chain of cursor loads of
// the hottest bucket (thousands of chunks), so each column's chunks are cut
// into segments, one thread each (sums, a scan over the segments, the
// prefixes), and the bucket's columns into slices of 1,024 threads' worth that
// blocks take independently; the block that finishes a bucket's last slice
// scans its column totals.  Heterogeneous 8M x 8M 0.25 -> 0.19 ms, 48 columns of
// 415K cells 24 -> 8 us, 30M Zipf cells 67 -> 44 us (one 1,024-thread block per
// bucket before).
constexpr int K6_THREADS = 256;
constexpr int K6_UNITS = 32;  // units per bucket, its slices dealt to them
constexpr int K6_BLOCKS = 4;  // per SM
template <typename OffT, bool BATCH>
__global__ void __launch_bounds__(K6_THREADS, K6_BLOCKS)
    k_chunk_scan(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ uint32_t sc[K6_THREADS];
    __shared__ unsigned long long sv[K6_THREADS];
    __shared__ unsigned long long wsum[2][33];
    __shared__ int last;
    pipeline_wait<BATCH>();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    Units<BATCH> U(m0, ba, blockIdx.x, gridDim.x);
    while (U.next([](const Mat &X) { return X.ws.hdr->n_multi_buckets * K6_UNITS; })) {
        const Mat &M = *U.M;
        // (bucket by bucket first, so that the many buckets of one slice spread over all blocks)
        const unsigned long long buckets = M.ws.hdr->n_multi_buckets;
        MultiBucket *mb = M.ws.multi_buckets + U.j % buckets;
        const uint32_t nch = mb->nch, bucket = mb->bucket;
        const unsigned long long mc0 = mb->mc0;
        if (!MGT_IN(M.ws.hdr, mc0 + nch, M.ws.hdr->max_rows + 1)) continue;
        const int w = 1 << M.p.bshift;
        Cursor *rows = M.ws.mc + mc0 * (unsigned long long)w;
        // threads of a column: more for more chunks
        const int least = nch < 64 ? 1 : nch < 512 ? 4 : 32;
        const int cols = min(w, K6_THREADS / least), segs = K6_THREADS / cols, slices = w / cols;
        const int seg = tid / cols, ci = tid % cols;
        const uint32_t per = (nch + segs - 1) / segs;
        const uint32_t h0 = min(nch, (uint32_t)seg * per), h1 = min(nch, h0 + per);
        for (int s = (int)(U.j / buckets); s < slices; s += K6_UNITS) {
            Cursor *mine = rows + s * cols + ci;
            constexpr uint32_t CU = 8;  // loads in flight
            uint32_t rc = 0;
            unsigned long long rv = 0;
            Cursor x[CU];
            for (uint32_t hb = h0; hb < h1; hb += CU) {
#pragma unroll
                for (uint32_t u = 0; u < CU; ++u)
                    if (hb + u < h1) x[u] = mine[(unsigned long long)(hb + u) * w];
#pragma unroll
                for (uint32_t u = 0; u < CU; ++u)
                    if (hb + u < h1) {
                        rc += x[u].a;
                        rv += x[u].b();
                    }
            }
            sc[tid] = rc;
            sv[tid] = rv;
            __syncthreads();
            for (int d = 1; d < segs; d <<= 1) {  // inclusive over the segments
                const uint32_t pc = seg >= d ? sc[tid - d * cols] : 0u;
                const unsigned long long pv = seg >= d ? sv[tid - d * cols] : 0ull;
                __syncthreads();
                sc[tid] += pc;
                sv[tid] += pv;
                __syncthreads();
            }
            uint32_t ac = sc[tid] - rc;
            unsigned long long av = sv[tid] - rv;
            for (uint32_t hb = h0; hb < h1; hb += CU) {
                if (per > CU) {  // (else the chunks are still in registers)
#pragma unroll
                    for (uint32_t u = 0; u < CU; ++u)
                        if (hb + u < h1) x[u] = mine[(unsigned long long)(hb + u) * w];
                }
#pragma unroll
                for (uint32_t u = 0; u < CU; ++u)
                    if (hb + u < h1) {
                        if (hb + u > 0) mine[(unsigned long long)(hb + u) * w] = Cursor(ac, av);
                        ac += x[u].a;
                        av += x[u].b();
                    }
            }
            if (slices > 1) {
                __syncthreads();
                if (seg == segs - 1) rows[s * cols + ci] = Cursor(sc[tid], sv[tid]);  // the column's totals
                __threadfence();
                __syncthreads();
                if (tid == 0) last = atomicAdd(&mb->done, 1u) == (uint32_t)slices - 1u;
                __syncthreads();
                if (!last) continue;
                __threadfence();
            }
            const unsigned long long bb = M.ws.bucket_base[bucket], vb = M.ws.bucket_vbase[bucket];
            const long long c0 = (long long)bucket << M.p.bshift;
            unsigned long long carry_c = bb, carry_v = vb;
            for (int b0 = 0; b0 < w; b0 += K6_THREADS) {
                const int c = b0 + tid;
                unsigned long long xc = 0, xv = 0;
                if (c < w && slices > 1) {
                    const uint32_t *r = reinterpret_cast<const uint32_t *>(rows + c);
                    xc = __ldcg(r);
                    xv = (unsigned long long)__ldcg(r + 2) << 32 | __ldcg(r + 1);
                } else if (c < w) {  // one slice: the totals are here
                    xc = sc[(segs - 1) * cols + c];
                    xv = sv[(segs - 1) * cols + c];
                }
                const unsigned long long ic = warp_inclusive_scan(xc), iv = warp_inclusive_scan(xv);
                if (lane == 31) {
                    wsum[0][warp] = ic;
                    wsum[1][warp] = iv;
                }
                __syncthreads();
                if (warp < 2) {
                    const unsigned long long v = lane < K6_THREADS / 32 ? wsum[warp][lane] : 0ull, vi = warp_inclusive_scan(v);
                    wsum[warp][lane] = vi - v;
                    if (lane == 31) wsum[warp][32] = vi;
                }
                __syncthreads();
                if (c < w) {
                    const unsigned long long at = carry_c + wsum[0][warp] + ic - xc;
                    rows[c] = Cursor((uint32_t)at, carry_v + wsum[1][warp] + iv - xv);
                    if (c0 + c < M.p.N) sto<OffT>(M.out.row_ptr, c0 + c, (long long)at);
                }
                carry_c += wsum[0][32];
                carry_v += wsum[1][32];
                __syncthreads();
            }
        }
    }
}

// ------------------------------------------------ shared-memory layouts
constexpr int P_WARPS = P_THREADS / 32;

struct ClLayout {
    size_t in, inv, lpre, wc, cst, ocnt, olen, pub_cnt, pub_len, allc, alll, scratch, misc, total;
};
// per-owner stride of the (owner, round, warp) counters, odd so that one
// warp's leaders for different owners fall on different banks
__host__ __device__ inline int ocnt_stride(int cap) {
    return ((cap + P_THREADS - 1) / P_THREADS) * (P_THREADS / 32) + 1;
}
template <typename Rec, int CS>
__host__ __device__ inline ClLayout cl_layout(int cap, int wsub) {
    ClLayout L;
    size_t o = 0;
    const int rmax = (cap + P_THREADS - 1) / P_THREADS;
#define MGT_TAKE(field, bytes) L.field = o; o = (o + (size_t)(bytes) + 15) & ~size_t(15);
    MGT_TAKE(in, (size_t)cap * sizeof(Rec))
    MGT_TAKE(inv, (size_t)cap * 2)
    MGT_TAKE(lpre, (size_t)(cap + 1) * 4)
    MGT_TAKE(wc, (size_t)(wsub + 1) * P_WARPS * 4)
    MGT_TAKE(cst, (size_t)(wsub + 1) * 4)
    MGT_TAKE(ocnt, (size_t)CS * ocnt_stride(cap) * 4)
    MGT_TAKE(olen, (size_t)CS * 8)
    MGT_TAKE(pub_cnt, (size_t)CS * 4)
    MGT_TAKE(pub_len, (size_t)CS * 8)
    MGT_TAKE(allc, (size_t)CS * CS * 4)
    MGT_TAKE(alll, (size_t)CS * CS * 8)
    MGT_TAKE(scratch, 48 * 8)
    MGT_TAKE(misc, 64)
#undef MGT_TAKE
    L.total = o;
    return L;
}

// -------------------------------------------------- K7a with clusters
// For plans that ask for clusters: one of CS = 2, 4 or 8 CTAs per bucket (at most CS x cap
// records).  CTA r owns the bucket's columns [r w/CS, (r+1) w/CS):
//   1. each CTA counts, per owner, the records of its slice of the bucket
//      (slices in input order) and their value totals; cluster barrier;
//   2. from the CS x CS counts every CTA knows where its records go in each
//      owner's buffer; it stores them there through distributed shared
//      memory (stable: slices in order, records in order); cluster barrier;
//   3. each owner sorts its records by column with a one-pass stable
//      multisplit (per-warp counters), writes row_ptr' for its columns and,
//      in output order, col_idx', cell_ptr' and each run's source offset.
// An owner receiving more than cap records is left to K7c (fallback list).
template <typename OffT, typename Rec, int CS, bool BATCH>
__global__ void __launch_bounds__(P_THREADS, 2)
    k_place_cluster(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    pipeline_wait<BATCH>();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned rank = cg::this_cluster().block_rank();
    // one work item per cluster at a time (same sequence on all its CTAs)
    Units<BATCH> U(m0, ba, blockIdx.x / CS, gridDim.x / CS);
    while (U.next([](const Mat &X) { return X.ws.hdr->n_items; })) {
    const Mat &M = *U.M;
    const unsigned long long j = U.j;
    const Rec *__restrict__ recs = reinterpret_cast<const Rec *>(M.ws.recs);
    const WorkItem *__restrict__ items = M.ws.items;
    const int bshift = M.p.bshift, cap = M.p.cap;
    const long long N = M.p.N, C = M.p.C, V = M.p.V;
    const unsigned long long *__restrict__ bucket_base = M.ws.bucket_base;
    const unsigned long long *__restrict__ bucket_vbase = M.ws.bucket_vbase;
    const void *cell_ptr = M.in.cell_ptr;
    void *out_row_ptr = M.out.row_ptr;
    int32_t *__restrict__ out_col = M.out.col;
    void *out_cell_ptr = M.out.cell_ptr;
    decltype(Rec::start) *__restrict__ src_start = reinterpret_cast<decltype(Rec::start) *>(M.ws.src);
    uint32_t *fallback = M.ws.fallback;
    DevHeader *hdr = M.ws.hdr;
    constexpr int LOGCS = CS == 2 ? 1 : CS == 4 ? 2 : 3;
    const int w = 1 << bshift;
    const int osh = bshift - LOGCS;
    const int wsub = 1 << osh;
    const ClLayout L = cl_layout<Rec, CS>(cap, wsub);
    const int rmax = (cap + P_THREADS - 1) / P_THREADS;
    Rec *IN = reinterpret_cast<Rec *>(smem + L.in);
    uint16_t *inv = reinterpret_cast<uint16_t *>(smem + L.inv);
    uint32_t *lpre = reinterpret_cast<uint32_t *>(smem + L.lpre);
    uint32_t *wc = reinterpret_cast<uint32_t *>(smem + L.wc);
    uint32_t *cst = reinterpret_cast<uint32_t *>(smem + L.cst);
    uint32_t *ocnt = reinterpret_cast<uint32_t *>(smem + L.ocnt);
    unsigned long long *olen = reinterpret_cast<unsigned long long *>(smem + L.olen);
    uint32_t *pub_cnt = reinterpret_cast<uint32_t *>(smem + L.pub_cnt);
    unsigned long long *pub_len = reinterpret_cast<unsigned long long *>(smem + L.pub_len);
    uint32_t *allc = reinterpret_cast<uint32_t *>(smem + L.allc);
    unsigned long long *alll = reinterpret_cast<unsigned long long *>(smem + L.alll);
    unsigned long long *scratch = reinterpret_cast<unsigned long long *>(smem + L.scratch);
    (void)w;
    const int ostr = ocnt_stride(cap);
    const int nocnt = CS * ostr;
    (void)rmax;
    {
        const WorkItem it = items[j];
        if (it.mc != ~0ull) continue;  // chunk of an oversized bucket: K7b
        const unsigned long long n = it.r1 - it.r0;
        uint32_t nin = 0;
        unsigned long long slot0 = bucket_base[it.bucket], vb0 = bucket_vbase[it.bucket];
        {
        const unsigned long long lo = it.r0 + n * rank / CS, hi = it.r0 + n * (rank + 1) / CS;
        const int m = n > (unsigned long long)CS * (unsigned long long)cap ? 0 : (int)(hi - lo);
        for (int x = tid; x < nocnt; x += P_THREADS) ocnt[x] = 0;
        if (tid < CS) olen[tid] = 0;
        __syncthreads();
        // ---- 1. per-owner counts and value totals of my slice (four
        // rounds of loads in flight at a time)
        unsigned long long lsum[CS];
#pragma unroll
        for (int q = 0; q < CS; ++q) lsum[q] = 0;
        for (int k0 = 0; k0 * P_THREADS < m; k0 += 4) {
            Rec r4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = (k0 + u) * P_THREADS + warp * 32 + lane;
                if (idx < m && MGT_IN(hdr, lo + idx, C)) r4[u] = recs[lo + idx];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u;
                const int idx = k * P_THREADS + warp * 32 + lane;
                const bool v = idx < m;
                uint32_t o = 0;
                if (v) {
                    o = (r4[u].meta >> 16) >> osh;
                    const unsigned long long len = rec_len<OffT>(r4[u].meta, r4[u].start, cell_ptr, C, V);
#pragma unroll
                    for (int q = 0; q < CS; ++q)
                        if ((int)o == q) lsum[q] += len;
                }
                const unsigned peers = digit_peers(o, LOGCS, v);
                if (v && (peers & lanemask_lt()) == 0) ocnt[(int)o * ostr + k * P_WARPS + warp] = __popc(peers);
            }
        }
#pragma unroll
        for (int q = 0; q < CS; ++q) {
            unsigned long long x = lsum[q];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
            if (lane == 0 && x) atomicAdd(&olen[q], x);
        }
        __syncthreads();
        // owner segment totals, then offsets in (owner, round, warp) order
        if (tid < CS) {
            uint32_t s = 0;
            for (int x = 0; x < ostr; ++x) s += ocnt[tid * ostr + x];
            pub_cnt[tid] = s;
            pub_len[tid] = olen[tid];
        }
        __syncthreads();
        block_exclusive_scan<uint32_t>(ocnt, nocnt, reinterpret_cast<uint32_t *>(scratch));
        cg::this_cluster().sync();  // #1: counts published
        // ---- 2. all CTAs' counts; shuffle to owners
        if (tid < CS * CS) {
            const int rr = tid / CS, q = tid % CS;
            auto cl = cg::this_cluster();
            allc[tid] = *cl.map_shared_rank(&pub_cnt[q], rr);
            alll[tid] = *cl.map_shared_rank(&pub_len[q], rr);
        }
        __syncthreads();
        bool overflow = n > (unsigned long long)CS * (unsigned long long)cap;  // defensive
#pragma unroll
        for (int q = 0; q < CS; ++q) {
            uint32_t s = 0;
            for (int rr = 0; rr < CS; ++rr) s += allc[rr * CS + q];
            overflow |= s > (uint32_t)cap;
        }
        if (!overflow) {
            for (int k0 = 0; k0 * P_THREADS < m; k0 += 4) {
                Rec r4[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int idx = (k0 + u) * P_THREADS + warp * 32 + lane;
                    if (idx < m) r4[u] = recs[lo + idx];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0 + u;
                    const int idx = k * P_THREADS + warp * 32 + lane;
                    const bool v = idx < m;
                    const uint32_t o = v ? (r4[u].meta >> 16) >> osh : 0u;
                    const unsigned peers = digit_peers(o, LOGCS, v);
                    if (v) {
                        uint32_t before = 0;
                        for (unsigned rr = 0; rr < rank; ++rr) before += allc[rr * CS + o];
                        const uint32_t segstart = ocnt[(int)o * ostr];
                        const uint32_t pos = before + ocnt[(int)o * ostr + k * P_WARPS + warp] - segstart +
                                             __popc(peers & lanemask_lt());
                        if (MGT_IN(hdr, pos, cap) && MGT_IN(hdr, o, CS)) {
                            Rec *dst = cg::this_cluster().map_shared_rank(IN, o);
                            dst[pos] = r4[u];
                        }
                    }
                }
            }
        }
        cg::this_cluster().sync();  // #2: shuffle complete
        if (overflow) {
            if (rank == 0 && tid == 0) {
                const unsigned long long fi = atomicAdd(&hdr->n_fallback, 1ull);
                if (MGT_IN(hdr, fi, hdr->max_items)) fallback[fi] = (uint32_t)j;
            }
            continue;
        }
        for (int q = 0; q < CS; ++q) {
            uint32_t s = 0;
            unsigned long long vs = 0;
            for (int rr = 0; rr < CS; ++rr) { s += allc[rr * CS + q]; vs += alll[rr * CS + q]; }
            if ((unsigned)q < rank) { slot0 += s; vb0 += vs; }
            if ((unsigned)q == rank) nin = s;
        }
        }
        // ---- 3. my columns: stable multisplit by column, then outputs
        const int seg = ((((int)nin + P_WARPS - 1) / P_WARPS) + 31) & ~31;
        const int a = warp * seg, e = min((int)nin, a + seg);
        for (int x = tid; x < (wsub + 1) * P_WARPS; x += P_THREADS) wc[x] = 0;
        __syncthreads();
        const uint32_t binbase = (uint32_t)rank << osh;
        // ranks among equal columns: one peer match per record, the rank
        // kept in lpre until the lengths need it
        warp_rank_pass(a, e, wsub, wc, lpre,
                       [&](int idx) { return (uint32_t)((IN[idx].meta >> 16) - binbase); });
        __syncthreads();
        wc_scan(wc, wsub, P_WARPS, cst, reinterpret_cast<uint32_t *>(scratch));
        {
            const long long c0 = ((long long)it.bucket << bshift) + binbase;
            for (int bin = tid; bin < wsub; bin += P_THREADS)
                if (c0 + bin < N && MGT_IN(hdr, c0 + bin, N + 1))
                    sto<OffT>(out_row_ptr, c0 + bin, (long long)(slot0 + cst[bin]));
        }
        for (int base = a; base < e; base += 32) {
            const int idx = base + lane;
            if (idx < e) {
                const uint32_t bin = (IN[idx].meta >> 16) - binbase;
                inv[wc[wc_at(bin, warp, wsub)] + lpre[idx]] = (uint16_t)idx;
            }
        }
        __syncthreads();
        // one gather per record in output order: its row and run start go out
        // now, its length to the scan for cell_ptr'
        for (int p = tid; p < (int)nin; p += P_THREADS) {
            const Rec r = IN[inv[p]];
            const unsigned long long q = slot0 + p;
            lpre[p] = (uint32_t)rec_len<OffT>(r.meta, r.start, cell_ptr, C, V);
            if (MGT_IN(hdr, q, C)) {
                out_col[q] = (int32_t)r.i;
                src_start[q] = r.start;
            }
        }
        __syncthreads();
        block_scan_segmented(lpre, (int)nin, reinterpret_cast<uint32_t *>(scratch));
        for (int p = tid; p < (int)nin; p += P_THREADS) {
            const unsigned long long q = slot0 + p;
            if (MGT_IN(hdr, q, C)) sto<OffT>(out_cell_ptr, (long long)q, (long long)(vb0 + lpre[p]));
        }
        __syncthreads();
    }
    }
}

// ------------------------------------------------------ K7a / K7b place
// One block per work item: a bucket of at most cap records (K7a), or a chunk
// of a larger one (K7b, whose columns start at the cursors of K6).  The
// records are loaded into shared memory once and split by column like the
// scatter passes split by digit (per-warp mask words and counters, an index
// permutation); each warp then takes a contiguous piece of the output order:
// row ids and run starts go out, a warp scan of the run lengths with a carry
// gives cell_ptr', with the pieces' totals exchanged once.  Bound by issue
// slots and the shared-memory pipe.  As many blocks as items: the hardware
// deals them, so buckets of uneven size leave no tail on a fixed share.
// Threads x rounds, blocks per SM, on the balanced 4M x 4M matrix: 256 x 20,
// three 1.09 ms, four 1.40 (spills); 384 x 14, three 1.26, two 1.21; 512 x 10,
// two 1.34; the sort it replaces (two 512-thread blocks, a hardware peer match
// per record, separate passes for lengths) 1.62.  With the outputs of buckets
// and chunks in loops of their own and the search for escaped lengths out of
// them 0.98 ms; heterogeneous 8M x 8M (buckets and chunks) 2.88 -> 1.72 ms.
constexpr int PL_THREADS = 256;
constexpr int PL_WARPS = PL_THREADS / 32;
constexpr int PL_ROUNDS = 20;
constexpr int PL_BLOCKS = 3;  // per SM, with the planner's shared memory
constexpr int PL_CAP = 5120;  // most records of a block (a multiple of 512 below PL_ROUNDS * PL_THREADS)
static_assert((PL_CAP + PL_WARPS - 1) / PL_WARPS <= PL_ROUNDS * 32, "a warp's piece fits its rounds");

struct PlLayout {
    size_t in, msk, cnt, adjv, adj, total;
};
template <typename Rec>
__host__ __device__ inline PlLayout pl_layout(int cap, int w) {
    PlLayout L;
    size_t o = 0;
    const size_t m = (size_t)(w + 1) * PL_WARPS * 4, inv = (size_t)cap * 2;
#define MGT_TAKE(field, bytes) L.field = o; o = (o + (size_t)(bytes) + 15) & ~size_t(15);
    MGT_TAKE(in, (size_t)cap * sizeof(Rec) + 16)
    MGT_TAKE(msk, m > inv ? m : inv)               // mask words; later the index permutation
    MGT_TAKE(cnt, (size_t)(w + 2) * PL_WARPS * 2)
    MGT_TAKE(adjv, (size_t)w * 8)                  // chunks: value cursor less the values before it here
    MGT_TAKE(adj, (size_t)w * 4)                   // chunks: cell cursor less the column's first position
#undef MGT_TAKE
    L.total = o;
    return L;
}

template <typename OffT, typename Rec, bool BATCH>
__global__ void __launch_bounds__(PL_THREADS, PL_BLOCKS)
    k_place(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long wtot[PL_WARPS];
    __shared__ uint32_t scratch[PL_WARPS];
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    DevHeader *hdr = M.ws.hdr;
    if ((unsigned long long)vb.b >= hdr->n_items) return;
    const WorkItem it = M.ws.items[vb.b];
    const bool chunk = it.mc != ~0ull;
    if (!chunk && M.p.cs > 1) return;  // a cluster's
    const int bshift = M.p.bshift, w = 1 << bshift, cap = M.p.cs > 1 ? M.p.chm : M.p.cap;
    const long long N = M.p.N, C = M.p.C, V = M.p.V;
    const void *cell_ptr = M.in.cell_ptr;
    int32_t *__restrict__ out_col = M.out.col;
    void *out_cell_ptr = M.out.cell_ptr;
    using SrcT = decltype(Rec::start);
    SrcT *__restrict__ src_start = reinterpret_cast<SrcT *>(M.ws.src);
    const int tid = threadIdx.x, lane = tid & 31, warp = warp_index();
    const int n = (int)(it.r1 - it.r0);
    const long long c0 = (long long)it.bucket << bshift;
    const uint32_t slot0 = (uint32_t)M.ws.bucket_base[it.bucket];
    if (n == 0) {  // an empty bucket: its columns' row pointers
        for (int c = tid; c < w; c += PL_THREADS)
            if (c0 + c < N) sto<OffT>(M.out.row_ptr, c0 + c, (long long)slot0);
        return;
    }
    if (!MGT_IN(hdr, n, cap + 1) || !MGT_IN(hdr, it.r1, C + 1)) return;
    const PlLayout L = pl_layout<Rec>(cap, w);
    uint32_t *wmsk = reinterpret_cast<uint32_t *>(smem + L.msk);
    uint16_t *wcnt = reinterpret_cast<uint16_t *>(smem + L.cnt);
    uint16_t *inv = reinterpret_cast<uint16_t *>(smem + L.msk);
    unsigned long long *adjv = reinterpret_cast<unsigned long long *>(smem + L.adjv);
    uint32_t *adj = reinterpret_cast<uint32_t *>(smem + L.adj);
    const Rec *IN = start_tile<PL_THREADS>(smem + L.in, reinterpret_cast<const Rec *>(M.ws.recs) + it.r0, n);
    const int cstr = w + 2, mstr = w + 1;
    {
        uint32_t *z = reinterpret_cast<uint32_t *>(smem + L.cnt);
        for (int i = tid; i < cstr * PL_WARPS / 2; i += PL_THREADS) z[i] = 0;
        for (int i = tid; i < mstr * PL_WARPS; i += PL_THREADS) wmsk[i] = 0;
    }
    wait_tile();
    __syncthreads();
    uint16_t *mycnt = wcnt + warp * cstr;
    uint32_t *mymsk = wmsk + warp * mstr;
    // this warp's piece of the records, and later of the positions: m of them
    // from a on, in `rounds` rounds (the same for the whole warp)
    const int seg = ((n + PL_WARPS - 1) / PL_WARPS + 31) & ~31;
    const int a = warp * seg, m = min(n - a, seg), rounds = m > 0 ? (m + 31) >> 5 : 0;
    const Rec *mine = IN + a + lane;
    uint32_t rk[PL_ROUNDS];
#pragma unroll
    for (int u = 0; u < PL_ROUNDS; ++u) {
        if (u < rounds) {
            const bool v = u * 32 + lane < m;
            const uint32_t d = v ? mine[u * 32].meta >> 16 : 0u;
            uint32_t group;
            rk[u] = (d << 16) | warp_rank<false>(mycnt, mymsk, d, v, group);
        }
    }
    __syncthreads();
    // positions in (column, warp) order; row_ptr' or the chunk's cursors
    {
        const Cursor *crow = chunk ? M.ws.mc + it.mc * (unsigned long long)w : nullptr;
        const Cursor *cfirst = chunk ? M.ws.mc + (it.mc - it.chunk) * (unsigned long long)w : nullptr;
        uint32_t carry = 0;
        for (int d0 = 0; d0 < w; d0 += PL_THREADS) {
            const int d = d0 + tid;
            uint32_t c[PL_WARPS], tot = 0;
#pragma unroll
            for (int q = 0; q < PL_WARPS; ++q) {
                c[q] = d < w ? wcnt[q * cstr + d] : 0u;
                tot += c[q];
            }
            const uint32_t inc = warp_sum_scan(tot);
            if (lane == 31) scratch[warp] = inc;
            __syncthreads();
            uint32_t run = carry + inc - tot;
#pragma unroll
            for (int q = 0; q < PL_WARPS; ++q) {
                const uint32_t s = scratch[q];
                run += q < warp ? s : 0u;
                carry += s;
            }
            if (d < w) {
                if (!chunk) {
                    if (c0 + d < N) sto<OffT>(M.out.row_ptr, c0 + d, (long long)(slot0 + run));
                } else {
                    const Cursor x = cfirst[d];
                    uint32_t xa = x.a;
                    unsigned long long xv = x.b();
                    if (it.chunk) {
                        const Cursor y = crow[d];
                        xa += y.a;
                        xv += y.b();
                    }
                    adj[d] = xa - run;
                    adjv[d] = xv;
                }
#pragma unroll
                for (int q = 0; q < PL_WARPS; ++q) {
                    wcnt[q * cstr + d] = (uint16_t)run;
                    run += c[q];
                }
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int u = 0; u < PL_ROUNDS; ++u)
        if (u < rounds && u * 32 + lane < m)
            inv[mycnt[rk[u] >> 16] + (rk[u] & 0xFFFFu)] = (uint16_t)(a + u * 32 + lane);
    __syncthreads();
    // this warp's positions: row ids and run starts; exclusive run-length sums
    const uint16_t *at = inv + a + lane;
    uint32_t pre[PL_ROUNDS];
    unsigned long long sum = 0;
    // 32 bits hold the sums of a piece (at most 640 records) without escaped
    // lengths; one with them leaves those out here and adds up in 64 bits below
    bool escaped = false;
    auto length = [&](const Rec &r) {
        const uint32_t len = r.meta & 0xFFFFu;
        escaped |= len == LEN_ESC;
        return len == LEN_ESC ? 0u : len;
    };
    auto prefix = [&](int u, uint32_t len) {
        const uint32_t inc = warp_sum_scan(len);
        pre[u] = (uint32_t)sum + inc - len;
        sum += __shfl_sync(0xffffffffu, inc, 31);
    };
    const size_t first = (size_t)slot0 + a + lane;  // K7a: consecutive places
    if (!chunk) {
        int32_t *pc = out_col + first;
        SrcT *ps = src_start + first;
#pragma unroll
        for (int u = 0; u < PL_ROUNDS; ++u) {
            if (u < rounds) {
                uint32_t len = 0;
                if (u * 32 + lane < m) {
                    const Rec r = IN[at[u * 32]];
                    len = length(r);
                    if (MGT_IN(hdr, first + u * 32, C)) {
                        pc[u * 32] = (int32_t)r.i;
                        ps[u * 32] = r.start;
                    }
                }
                prefix(u, len);
            }
        }
    } else {
#pragma unroll
        for (int u = 0; u < PL_ROUNDS; ++u) {
            if (u < rounds) {
                uint32_t len = 0;
                if (u * 32 + lane < m) {
                    const Rec r = IN[at[u * 32]];
                    len = length(r);
                    const uint32_t q = adj[r.meta >> 16] + (uint32_t)(a + u * 32 + lane);
                    if (MGT_IN(hdr, q, C)) {
                        out_col[q] = (int32_t)r.i;
                        src_start[q] = r.start;
                    }
                }
                prefix(u, len);
            }
        }
    }
    // fn(u, sum of the piece's lengths before it) for this lane's records, and the
    // piece's total, from the records again (runs of 2^16 values and more are few:
    // their copy takes far longer than the searches for their lengths)
    auto wide_prefixes = [&](auto fn) {
        unsigned long long run = 0;
#pragma unroll 1
        for (int u = 0; u < rounds; ++u) {
            const bool v = u * 32 + lane < m;
            unsigned long long len = 0;
            if (v) {
                const Rec r = IN[at[u * 32]];
                len = rec_len<OffT>(r.meta, r.start, cell_ptr, C, V);
            }
            const unsigned long long inc = warp_inclusive_scan(len);
            if (v) fn(u, run + inc - len);
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        return run;
    };
    const bool wide = __any_sync(0xffffffffu, escaped);
    if (wide) sum = wide_prefixes([](int, unsigned long long) {});
    if (lane == 0) wtot[warp] = sum;
    __syncthreads();
    unsigned long long base = chunk ? 0ull : M.ws.bucket_vbase[it.bucket];
#pragma unroll
    for (int q = 0; q < PL_WARPS; ++q) base += q < warp ? wtot[q] : 0ull;
    if (!chunk) {
        OffT *po = reinterpret_cast<OffT *>(out_cell_ptr) + first;
        if (wide) {
            wide_prefixes([&](int u, unsigned long long before) {
                if (MGT_IN(hdr, first + u * 32, C)) po[u * 32] = (OffT)(base + before);
            });
            return;
        }
#pragma unroll
        for (int u = 0; u < PL_ROUNDS; ++u)
            if (u < rounds && u * 32 + lane < m && MGT_IN(hdr, first + u * 32, C))
                po[u * 32] = (OffT)(base + pre[u]);
        return;
    }
    // a column's first position takes the values before it off its cursor
    auto take_first = [&](int u, unsigned long long before) {
        const uint32_t c = IN[at[u * 32]].meta >> 16;
        if (a + u * 32 + lane == 0 || IN[at[u * 32 - 1]].meta >> 16 != c) adjv[c] -= base + before;
    };
    auto put = [&](int u, unsigned long long before) {
        const uint32_t c = IN[at[u * 32]].meta >> 16, q = adj[c] + (uint32_t)(a + u * 32 + lane);
        if (MGT_IN(hdr, q, C)) sto<OffT>(out_cell_ptr, q, (long long)(adjv[c] + base + before));
    };
    if (wide) {
        wide_prefixes(take_first);
    } else {
#pragma unroll
        for (int u = 0; u < PL_ROUNDS; ++u)
            if (u < rounds && u * 32 + lane < m) take_first(u, pre[u]);
    }
    __syncthreads();
    if (wide) {
        wide_prefixes(put);
    } else {
#pragma unroll
        for (int u = 0; u < PL_ROUNDS; ++u)
            if (u < rounds && u * 32 + lane < m) put(u, pre[u]);
    }
}

// --------------------------------------------------- K7c fallback place
// One CTA per bucket that overflowed a K7a owner (a few very frequent
// columns): per-column counts and value sums, column starts, then one warp
// deals the records in input order to their columns' cursors.
template <typename OffT, typename Rec, bool BATCH>
__global__ void __launch_bounds__(P_THREADS, 1)
    k_place_fallback(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    pipeline_wait<BATCH>();
    Units<BATCH> U(m0, ba, blockIdx.x, gridDim.x);
    while (U.next([](const Mat &X) { return X.ws.hdr->n_fallback; })) {
    const Mat &M = *U.M;
    const unsigned long long jj = U.j;
    const Rec *__restrict__ recs = reinterpret_cast<const Rec *>(M.ws.recs);
    const WorkItem *__restrict__ items = M.ws.items;
    const uint32_t *__restrict__ fallback = M.ws.fallback;
    const int bshift = M.p.bshift;
    const long long N = M.p.N, C = M.p.C, V = M.p.V;
    const unsigned long long *__restrict__ bucket_base = M.ws.bucket_base;
    const unsigned long long *__restrict__ bucket_vbase = M.ws.bucket_vbase;
    const void *cell_ptr = M.in.cell_ptr;
    void *out_row_ptr = M.out.row_ptr;
    int32_t *__restrict__ out_col = M.out.col;
    void *out_cell_ptr = M.out.cell_ptr;
    decltype(Rec::start) *__restrict__ src_start = reinterpret_cast<decltype(Rec::start) *>(M.ws.src);
    const DevHeader *hdr = M.ws.hdr;
    const int w = 1 << bshift;
    unsigned long long *cur = reinterpret_cast<unsigned long long *>(smem);  // [w] slots
    unsigned long long *vcur = cur + w;                                       // [w] values
    unsigned long long *scratch = vcur + w;                                   // [48]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const WorkItem it = items[fallback[jj]];
        if (!MGT_IN(const_cast<DevHeader *>(hdr), it.r1, C + 1)) continue;
        for (int c = tid; c < w; c += P_THREADS) { cur[c] = 0; vcur[c] = 0; }
        __syncthreads();
        for (unsigned long long r0 = it.r0; r0 < it.r1; r0 += P_THREADS) {
            const unsigned long long r = r0 + tid;
            const bool v = r < it.r1;
            uint32_t c = 0;
            unsigned long long len = 0;
            if (v) {
                const Rec rc = recs[r];
                c = rc.meta >> 16;
                len = rec_len<OffT>(rc.meta, rc.start, cell_ptr, C, V);
            }
            warp_count_add(cur, vcur, c, len, v, 1 << bshift);
        }
        __syncthreads();
        block_exclusive_scan<unsigned long long>(cur, w, scratch);
        block_exclusive_scan<unsigned long long>(vcur, w, scratch);
        const unsigned long long bb = bucket_base[it.bucket], vb = bucket_vbase[it.bucket];
        const long long c0 = (long long)it.bucket << bshift;
        for (int c = tid; c < w; c += P_THREADS) {
            cur[c] += bb;
            vcur[c] += vb;
            if (c0 + c < N) sto<OffT>(out_row_ptr, c0 + c, (long long)cur[c]);
        }
        __syncthreads();
        if (warp == 0) {
            for (unsigned long long r0 = it.r0; r0 < it.r1; r0 += 32) {
                const unsigned long long r = r0 + lane;
                const bool v = r < it.r1;
                Rec rc{};
                uint32_t c = 0xFFFFFFFFu;
                unsigned long long len = 0;
                if (v) {
                    rc = recs[r];
                    c = rc.meta >> 16;
                    len = rec_len<OffT>(rc.meta, rc.start, cell_ptr, C, V);
                }
                const unsigned peers = digit_peers(v ? c : 0u, bshift, v);
                const unsigned lower = peers & lanemask_lt();
                unsigned long long pre = 0, tot = 0;
                for (int l = 0; l < 32; ++l) {
                    const unsigned long long x = __shfl_sync(0xffffffffu, len, l);
                    if ((peers >> l) & 1u) {
                        tot += x;
                        if ((lower >> l) & 1u) pre += x;
                    }
                }
                unsigned long long s = 0, vv = 0;
                if (v && lower == 0) {
                    s = cur[c];
                    vv = vcur[c];
                    cur[c] = s + __popc(peers);
                    vcur[c] = vv + tot;
                }
                const int leader = __ffs(peers) - 1;
                s = __shfl_sync(0xffffffffu, s, leader);
                vv = __shfl_sync(0xffffffffu, vv, leader);
                if (v) {
                    const unsigned long long q = s + __popc(lower);
                    if (MGT_IN(const_cast<DevHeader *>(hdr), q, C)) {
                    out_col[q] = (int32_t)rc.i;
                    sto<OffT>(out_cell_ptr, (long long)q, (long long)(vv + pre));
                    src_start[q] = rc.start;
                    }
                }
                __syncwarp();
            }
        }
        __syncthreads();
    }
    }
}

// ------------------------------------------------------------- K8 copy
constexpr int CP_THREADS = 256;
constexpr int CP_WARPS = CP_THREADS / 32;
constexpr int CP_CELLS = 512;    // most output cells of one tile
constexpr int CP_GROUPS = 2048;  // most groups of 32 units of one tile (longer tiles: run by run)

// One unit of VEC bytes, through registers.
template <int VEC>
struct Unit {
    typename VecT<VEC>::T v;
    __device__ __forceinline__ void load(const uint8_t *p) { v = __ldg(reinterpret_cast<const typename VecT<VEC>::T *>(p)); }
    __device__ __forceinline__ void store(uint8_t *p) const { *reinterpret_cast<typename VecT<VEC>::T *>(p) = v; }
};
template <>
struct Unit<32> {  // one whole sector per lane
    int4 a, b;
    __device__ __forceinline__ void load(const uint8_t *p) {
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                     : "l"(p));
    }
    __device__ __forceinline__ void store(uint8_t *p) const {
        asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(a.x), "r"(a.y), "r"(a.z),
                     "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w), "l"(p)
                     : "memory");
    }
};

// The tile's runs, back to back in the output, in units of VEC bytes:
// off[0..n] their unit offsets (no run is empty), sb[i] where the input's unit 0
// would lie for the run (its units follow the tile's numbering), gcell[g] the
// run of unit 32 g.
// A warp takes U groups of 32 units at a time, their loads all in flight.  The
// runs that start inside a group mark their first unit in a 32-bit word (one
// warp-wide OR); the number of marks at or below a lane is its run.  off[n + 1
// .. n + 32] hold ~0 (off has CP_OFF entries).  Narrow
// units take more of them in flight for the same bytes: 12-byte values in runs
// of 72 bytes 1.71 -> 1.18 ms with 16 words instead of 2, 4-byte values in runs
// of 44 bytes 1.19 -> 0.90 ms (32M runs).
__device__ __forceinline__ uint32_t bit_or_none(uint32_t s) {  // 1 << s, 0 for s >= 32
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(s));  // (PTX clamps the shift)
    return r;
}
constexpr int CP_OFF = CP_CELLS + 1 + 32;  // off[]: 32 entries past the end for copy_tile's look-ahead
template <int VEC, int U>
__device__ __forceinline__ void copy_tile(uint8_t *__restrict__ out, const uint32_t *off,
                                          const uint8_t *const *sb, const uint16_t *gcell, uint32_t units) {
    const int lane = threadIdx.x & 31, warp = warp_index();
    const unsigned le = lanemask_lt() | (1u << lane);
    const uint32_t groups = (units + 31) >> 5;
    const uint32_t *ahead = off + 1 + lane;
    for (uint32_t g0 = warp * U; g0 < groups; g0 += CP_WARPS * U) {
        Unit<VEC> x[U];
        const uint32_t u0 = (g0 << 5) + lane;
        uint8_t *to = out + (size_t)u0 * VEC;
        if (((g0 + U) << 5) <= units) {
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const uint32_t c0 = gcell[g0 + j];
                const unsigned marks = __reduce_or_sync(0xffffffffu, bit_or_none(ahead[c0] - ((g0 + j) << 5)));
                x[j].load(sb[c0 + __popc(marks & le)] + (size_t)(u0 * VEC) + j * 32 * VEC);
            }
#pragma unroll
            for (int j = 0; j < U; ++j) x[j].store(to + j * 32 * VEC);
        } else {  // the tile's last groups
#pragma unroll
            for (int j = 0; j < U; ++j) {
                if (g0 + j < groups) {
                    const uint32_t c0 = gcell[g0 + j];
                    const unsigned marks = __reduce_or_sync(0xffffffffu, bit_or_none(ahead[c0] - ((g0 + j) << 5)));
                    if (u0 + j * 32 < units)
                        x[j].load(sb[c0 + __popc(marks & le)] + (size_t)(u0 * VEC) + j * 32 * VEC);
                }
            }
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (u0 + j * 32 < units) x[j].store(to + j * 32 * VEC);
        }
    }
}

// One run of `units` units by `nt` threads of which this is thread t.
template <int VEC>
__device__ __forceinline__ void copy_long(const uint8_t *__restrict__ in, uint8_t *__restrict__ out,
                                          unsigned long long units, int t, int nt) {
    unsigned long long u = t;
    for (; u + 3ull * nt < units; u += 4ull * nt) {
        Unit<VEC> x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j].load(in + (u + (unsigned long long)j * nt) * VEC);
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j].store(out + (u + (unsigned long long)j * nt) * VEC);
    }
    for (; u < units; u += nt) {
        Unit<VEC> x;
        x.load(in + u * VEC);
        x.store(out + u * VEC);
    }
}

// Every value run, in output order: source offset from src_start, target and
// length from cell_ptr'.  One block per tile of 2^cshift output cells, in
// output order, as many tiles as there are: the hardware deals them in order,
// so that all blocks in flight write one narrow window of the output that
// moves through it.  (A grid that fills the GPU once and strides through the
// output has its warps drift apart: random 32-byte runs over 4.3 GB moved at
// 34.5 G runs/s that way against 48 in order, 160-byte runs at 13.4 against
// 20.1, i.e. 6.4 TB/s, 95 % of the measured copy.)  Whole kernel, before and
// after: heterogeneous 8M x 8M 13.3 -> 8.55 ms (6.3 TB/s; 8.95 on some boxes),
// balanced 4M x 4M 3.86 -> 2.79 ms (3.37), 640-byte runs 5.62 -> 3.80 ms (7.0 TB/s).  It is bound by
// DRAM: short runs by the rate of random sectors, long ones by bandwidth.
template <typename OffT, typename SrcT, int U, bool BATCH>
__global__ void __launch_bounds__(CP_THREADS, U >= 4 ? 4 : U == 2 ? 5 : 6)
    k_copy_values(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ uint32_t off[CP_OFF];
    __shared__ const uint8_t *sb[CP_CELLS];
    __shared__ uint16_t gcell[CP_GROUPS];
    __shared__ int wcount[CP_CELLS / 32];
    __shared__ unsigned walign[CP_WARPS];
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    DevHeader *hdr = M.ws.hdr;
    // nothing for a matrix whose sort kernels placed nothing (malformed input or an internal limit);
    // threads of a block may read different words (other blocks flag too): they decide together below
    const bool stopped = (hdr->status & (ST_BADINPUT | ST_OVERFLOW)) != 0;
    const SrcT *__restrict__ src_start = reinterpret_cast<const SrcT *>(M.ws.src);
    const void *__restrict__ cp = M.out.cell_ptr;
    const long long C = M.p.C, V = M.p.V;
    const int stride = M.p.s, cells = 1 << M.p.cshift;
    const long long q0 = vb.b << M.p.cshift;
    const int n0 = (int)min((long long)cells, C - q0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long d_first = ldp<OffT>(cp, q0), d_last = ldp<OffT>(cp, q0 + n0);
    // this thread's cells (at most two); empty runs are left out
    constexpr int PER = CP_CELLS / CP_THREADS;
    long long d0[PER], d1[PER], sv[PER];
    unsigned mask[PER], align = 0;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = tid + k * CP_THREADS;
        d0[k] = d1[k] = sv[k] = 0;
        if (i < n0) {
            d0[k] = ldp<OffT>(cp, q0 + i);
            d1[k] = ldp<OffT>(cp, q0 + i + 1);
            sv[k] = (long long)src_start[q0 + i];
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const long long len = d1[k] - d0[k];
        if (tid + k * CP_THREADS < n0)  // never for consistent outputs
            bad |= d0[k] < 0 || len < 0 || d1[k] > V || sv[k] < 0 || sv[k] > V - len || d0[k] < d_first || d1[k] > d_last;
        const bool full = len > 0;
        mask[k] = __ballot_sync(0xffffffffu, full);
        if (lane == 0) wcount[k * CP_WARPS + warp] = __popc(mask[k]);
        if (full) align |= (unsigned)(sv[k] * stride) | (unsigned)(d0[k] * stride) | (unsigned)(len * stride);
    }
    align = __reduce_or_sync(0xffffffffu, align);
    if (lane == 0) walign[warp] = align;
    if (__syncthreads_or(bad || stopped)) {
        if (bad && !stopped) flag(hdr, ST_OVERFLOW);
        return;
    }
    const uint8_t *in = M.in.values;
    uint8_t *out = M.out.values + d_first * stride;
#pragma unroll
    for (int w = 0; w < CP_WARPS; ++w) align |= walign[w];
    align |= (unsigned)(reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(M.out.values));
    const int vshift = (align & 31) == 0 ? 5 : (align & 15) == 0 ? 4 : (align & 7) == 0 ? 3 : 2;
    const long long units = ((d_last - d_first) * stride) >> vshift;
    if (units > 32LL * CP_GROUPS) {
        // long runs: one warp per run, the whole block for the very long ones
        constexpr long long WIDE = 1 << 16;  // bytes
        for (int pass = 0; pass < 2; ++pass) {
            for (int i = pass ? 0 : warp; i < n0; i += pass ? 1 : CP_WARPS) {
                const long long a = ldp<OffT>(cp, q0 + i), len = (ldp<OffT>(cp, q0 + i + 1) - a) * stride;
                if ((len >= WIDE) != (pass != 0)) continue;
                const uint8_t *pi = in + (long long)src_start[q0 + i] * stride;
                uint8_t *po = M.out.values + a * stride;
                const int t = pass ? tid : lane, nt = pass ? CP_THREADS : 32;
                if (vshift == 5) copy_long<32>(pi, po, len >> 5, t, nt);
                else if (vshift == 4) copy_long<16>(pi, po, len >> 4, t, nt);
                else if (vshift == 3) copy_long<8>(pi, po, len >> 3, t, nt);
                else copy_long<4>(pi, po, len >> 2, t, nt);
            }
        }
        return;
    }
    int n = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int at = n + __popc(mask[k] & lanemask_lt());
#pragma unroll
        for (int w = 0; w < CP_WARPS; ++w) {
            const int c = wcount[k * CP_WARPS + w];
            at += w < warp ? c : 0;
            n += c;
        }
        if (d1[k] > d0[k]) {
            const uint32_t o0 = (uint32_t)(((d0[k] - d_first) * stride) >> vshift);
            const uint32_t o1 = (uint32_t)(((d1[k] - d_first) * stride) >> vshift);
            off[at] = o0;
            sb[at] = in + (sv[k] - (d0[k] - d_first)) * stride;
            for (uint32_t g = (o0 + 31) >> 5; (g << 5) < o1; ++g) gcell[g] = (uint16_t)at;
        }
    }
    if (warp == 0) off[n + 1 + lane] = ~0u;
    if (tid == 0) off[n] = (uint32_t)units;
    __syncthreads();
    if (vshift == 5) copy_tile<32, U>(out, off, sb, gcell, (uint32_t)units);
    else if (vshift == 4) copy_tile<16, 2 * U>(out, off, sb, gcell, (uint32_t)units);
    else if (vshift == 3) copy_tile<8, 4 * U>(out, off, sb, gcell, (uint32_t)units);
    else copy_tile<4, (U < 2 ? 8 : 16)>(out, off, sb, gcell, (uint32_t)units);
}

// Launch of one level-2 phase for one (offset, record) format; `which`:
// 0 = chunk hist (K5), 1 = chunk scan (K6), 2 = place (K7a / K7b), 3 = place
// with clusters, 4 = fallback place (K7c), 5 = value copy (K8).
template <typename OffT, typename Rec>
cudaError_t launch_level2_t(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                            cudaStream_t st, int which);

template <typename OffT, typename Rec, int CS>
static cudaError_t launch_cluster_cs(const Mat &m0, const BatchArgs &ba, long long grid,
                                     size_t smem, cudaStream_t st) {
    auto kern = ba.n ? k_place_cluster<OffT, Rec, CS, true> : k_place_cluster<OffT, Rec, CS, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(P_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.gridDim = dim3((unsigned)grid);
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, kern, m0, ba);
}

// Sort clusters of the cluster-place kernel that fit on the GPU at once.
template <typename OffT, typename Rec, int CS>
static long long resident_clusters_cs(size_t smem) {
    auto kern = k_place_cluster<OffT, Rec, CS, false>;  // same limits as the batch variant
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(P_THREADS);
    cfg.gridDim = dim3(CS);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) return 0;
    return n;
}

template <typename OffT, typename Rec>
long long resident_clusters_t(int cs, size_t smem) {
    switch (cs) {
    case 2: return resident_clusters_cs<OffT, Rec, 2>(smem);
    case 4: return resident_clusters_cs<OffT, Rec, 4>(smem);
    default: return resident_clusters_cs<OffT, Rec, 8>(smem);
    }
}

template <typename OffT, typename Rec>
cudaError_t launch_level2_t(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                            cudaStream_t st, int which) {
    using SrcT = decltype(Rec::start);
    cudaError_t e = cudaSuccess;
    switch (which) {
    case 0: {
        auto kern = ba.n ? k_chunk_hist<OffT, Rec, true> : k_chunk_hist<OffT, Rec, false>;
        e = launch_kernel(kern, ba.n > 0, grid, K5_THREADS, smem, st, m0, ba);
        break;
    }
    case 1: {
        auto kern = ba.n ? k_chunk_scan<OffT, true> : k_chunk_scan<OffT, false>;
        e = launch_kernel(kern, ba.n > 0, grid, K6_THREADS, smem, st, m0, ba);
        break;
    }
    case 2: {
        auto kern = ba.n ? k_place<OffT, Rec, true> : k_place<OffT, Rec, false>;
        e = launch_kernel(kern, ba.n > 0, grid, PL_THREADS, smem, st, m0, ba);
        break;
    }
    case 3:
        switch (m0.p.cs) {
        case 2: e = launch_cluster_cs<OffT, Rec, 2>(m0, ba, grid, smem, st); break;
        case 4: e = launch_cluster_cs<OffT, Rec, 4>(m0, ba, grid, smem, st); break;
        default: e = launch_cluster_cs<OffT, Rec, 8>(m0, ba, grid, smem, st); break;
        }
        break;
    case 4: {
        auto kern = ba.n ? k_place_fallback<OffT, Rec, true> : k_place_fallback<OffT, Rec, false>;
        e = launch_kernel(kern, ba.n > 0, grid, P_THREADS, smem, st, m0, ba);
        break;
    }
    default:
        auto kern = m0.p.unroll >= 4 ? (ba.n ? k_copy_values<OffT, SrcT, 4, true> : k_copy_values<OffT, SrcT, 4, false>)
                    : m0.p.unroll == 2 ? (ba.n ? k_copy_values<OffT, SrcT, 2, true> : k_copy_values<OffT, SrcT, 2, false>)
                                       : (ba.n ? k_copy_values<OffT, SrcT, 1, true> : k_copy_values<OffT, SrcT, 1, false>);
        e = launch_kernel(kern, ba.n > 0 || ba.late, grid, CP_THREADS, 0, st, m0, ba);
        break;
    }
    return e;
}

}  // namespace mgt
