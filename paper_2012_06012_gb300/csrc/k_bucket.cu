// Level 1 of the transpose: stable scatter of cell records into column buckets.
//
// The paper exchanges cells between ranks by destination (Sec. 3, view swap:
// metadata, then values).  On one GPU the destination of a cell is a bucket of
// consecutive output rows (= input columns); K1-K3 deal every cell's record
// into its bucket, keeping row-major input order inside each bucket, so that
// the per-bucket sort of K7 only has to order by column.  Here: set-up, counts,
// scans and the sort's work list (the scatter passes are in k_scatter.cu).
#include "mgt_internal.cuh"

#include <algorithm>

namespace mgt {

constexpr int K_THREADS = 512;

// ------------------------------------------------------------------ K0 prep
// Zeroes what a transpose starts from (header, value totals, P x P counts, the
// variable-width copy's tile words), checks the pointer arrays' end points,
// puts the row-block offsets in place and derives the source blocks' cell
// offsets pcoff[s] = row_ptr[off[s]]; writes the output sentinels
// row_ptr'[N] = C and cell_ptr'[C] = V and the P = 1 counts, and the row table.
// (The header is written by one thread of the first block; no other block
// touches it here, so that nothing has to be cleared before.)
struct PrepOff {
    long long v[PREP_OFF];
    int n;  // P + 1, or 0: the offsets are in the workspace already
};
template <typename OffT, bool BATCH>
__global__ void __launch_bounds__(K_THREADS)
    k_prep(const __grid_constant__ Mat m0, const BatchArgs ba, const __grid_constant__ PrepOff given) {
    __shared__ uint32_t lrow[K_THREADS];  // long rows of the block's round and their row table entries
    __shared__ long long lbeg[K_THREADS], lend[K_THREADS];
    __shared__ int nlong;
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const void *row_ptr = M.in.row_ptr, *cell_ptr = M.in.cell_ptr;
    const long long R = M.p.R, N = M.p.N, C = M.p.C, V = M.p.V, B = M.p.B;
    const int P = M.p.P, bshift = M.p.bshift;
    long long *poff = M.ws.poff;
    long long *pcoff = M.ws.pcoff;
    uint16_t *dblock = M.ws.dblock;
    long long *part_cells = M.out.part_cells, *part_values = M.out.part_values;
    long long gid = vb.b * (long long)blockDim.x + threadIdx.x;
    long long stride = vb.g * (long long)blockDim.x;
    if (gid == 0) {
        const bool bad = ldp<OffT>(row_ptr, 0) != 0 || ldp<OffT>(row_ptr, R) != C || ldp<OffT>(cell_ptr, 0) != 0 ||
                         ldp<OffT>(cell_ptr, C) != V;
        unsigned long long *h = reinterpret_cast<unsigned long long *>(M.ws.hdr);
        for (int i = 1; i < 32; ++i) h[i] = 0;
        h[0] = bad ? ST_BADINPUT : 0u;  // status
        sto<OffT>(M.out.row_ptr, N, C);
        sto<OffT>(M.out.cell_ptr, C, V);
        if (P == 1 && part_cells) part_cells[0] = C;
        if (P == 1 && part_values) part_values[0] = V;
    }
    for (long long b = gid; b < B; b += stride) M.ws.bucket_vtot[b] = 0;
    if (P > 1 && part_cells)
        for (long long i = gid; i < (long long)P * P; i += stride) part_cells[i] = part_values[i] = 0;
    if (M.p.var)
        for (long long i = gid; i <= (C + (1LL << M.p.cshift) - 1) >> M.p.cshift; i += stride) M.ws.vblk[i] = 0;
    auto off = [&](long long s) { return given.n ? given.v[s] : poff[s]; };
    for (long long s = gid; s <= P; s += stride) {
        const long long r = off(s);
        if (given.n) poff[s] = r;
        pcoff[s] = (r >= 0 && r <= R) ? ldp<OffT>(row_ptr, r) : 0;
    }
    // destination block of each bucket's columns, or 0xFFFF when they span two
    // (for the scatter pass that searches the block of a cell)
    if (scatter_counts_pp(M.p) && !M.p.pp_aligned) {
        auto block_of = [&](long long c) {
            long long lo = 0, hi = P + 1;  // first offset above c
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                if (off(mid) <= c) lo = mid + 1;
                else hi = mid;
            }
            return lo < 1 ? 0 : (lo > P ? P - 1 : lo - 1);
        };
        for (long long b = gid; b < B; b += stride) {
            const long long c0 = b << bshift, c1 = min(N, c0 + (1LL << bshift)) - 1;
            const long long da = block_of(c0), db = block_of(c1);
            dblock[b] = (da == db) ? (uint16_t)da : (uint16_t)0xFFFFu;
        }
    }
    // row of every 2^ROWAT_SHIFT-th cell, for the scatter pass: each row writes
    // the entries of its cells, a warp together for its longer rows, the block for
    // its longest (one dependent load where a search per entry takes a dozen)
    if (R > 0 && C > 0) {
        uint32_t *rowat = row_table(M.ws);
        const int lane = threadIdx.x & 31;
        const long long nb = row_table_entries(C), up = (1 << ROWAT_SHIFT) - 1;
        constexpr long long LONG_ROW = 1024;  // entries
        // Entries that the longer rows of this warp and of this block may still write: a valid
        // matrix's rows share the table.  Malformed row pointers (K1 checks their order) may claim it
        // once per row: 2M rows that claim all of 16M cells took 85 ms (a valid matrix of the size 0.7).
        long long warp_left = nb, block_left = nb;
        for (long long b0 = vb.b * (long long)blockDim.x; b0 < R; b0 += stride) {
            const long long i = b0 + threadIdx.x;
            long long e0 = 0, e1 = 0;  // entries [e0, e1)
            if (i < R) {
                const long long k0 = ldp<OffT>(row_ptr, i), k1 = ldp<OffT>(row_ptr, i + 1);
                e0 = min(max((k0 + up) >> ROWAT_SHIFT, 0ll), nb);
                e1 = min(max((k1 + up) >> ROWAT_SHIFT, 0ll), nb);
                if (k0 < C && k1 >= C) rowat[nb - 1] = (uint32_t)i;  // the last cell's row
            }
            const long long len = e1 - e0;
            if (len <= 4)
                for (long long e = e0; e < e1; ++e) rowat[e] = (uint32_t)i;
            for (unsigned todo = __ballot_sync(0xffffffffu, len > 4 && len < LONG_ROW); todo; todo &= todo - 1) {
                const int l = __ffs(todo) - 1;
                const long long a = __shfl_sync(0xffffffffu, e0, l), z = __shfl_sync(0xffffffffu, e1, l);
                const uint32_t r = __shfl_sync(0xffffffffu, (uint32_t)i, l);
                warp_left -= z - a;
                if (warp_left < 0) break;
                for (long long e = a + lane; e < z; e += 32) rowat[e] = r;
            }
            if (__syncthreads_or(len >= LONG_ROW)) {
                if (threadIdx.x == 0) nlong = 0;
                __syncthreads();
                if (len >= LONG_ROW) {
                    const int k = atomicAdd(&nlong, 1);
                    lrow[k] = (uint32_t)i;
                    lbeg[k] = e0;
                    lend[k] = e1;
                }
                __syncthreads();
                for (int k = 0; k < nlong; ++k) {
                    block_left -= lend[k] - lbeg[k];
                    if (block_left < 0) break;
                    for (long long e = lbeg[k] + threadIdx.x; e < lend[k]; e += K_THREADS) rowat[e] = lrow[k];
                }
                __syncthreads();
            }
        }
    }
}

static long long grid_prep(const Params &p, double share) {
    const long long full = 4LL * sm_count();
    long long n = std::max<long long>(p.R, p.B);
    if (p.P > 1) n = std::max<long long>(n, (long long)p.P * p.P);
    if (p.var) n = std::max<long long>(n, p.C >> p.cshift);
    long long want = (n + K_THREADS - 1) / K_THREADS;
    long long cap = (long long)(full * share + 0.999);
    if (cap < 1) cap = 1;
    if (want > cap) want = cap;
    return want < 1 ? 1 : want;
}
static size_t smem_none(const Params &) { return 0; }
static cudaError_t launch_prep(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                               cudaStream_t st) {
    PrepOff given;
    given.n = 0;
    if (!ba.n && m0.p.off_host && m0.p.P + 1 <= PREP_OFF) {
        given.n = m0.p.P + 1;
        for (int i = 0; i < given.n; ++i) given.v[i] = m0.p.off_host[i];
    }
    auto kern = m0.p.o == 4 ? (ba.n ? k_prep<int32_t, true> : k_prep<int32_t, false>)
                            : (ba.n ? k_prep<int64_t, true> : k_prep<int64_t, false>);
    return launch_kernel(kern, ba.n > 0, grid, K_THREADS, 0, st, m0, ba, given);
}

// ------------------------------------------------------------------ K1 hist
// Cells per bucket for one tile of `tile` consecutive cells, in a shared
// memory histogram; written as row t of the T x B count matrix.  Also checks
// that row_ptr never decreases (its rows dealt to all blocks; blocks past the
// last tile have nothing else to do).
template <typename OffT, bool BATCH>
__global__ void __launch_bounds__(1024) k_hist(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ uint32_t hist[];
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const int32_t *__restrict__ col = M.in.col;
    const long long C = M.p.C, N = M.p.N;
    const int bshift = M.p.bshift, B = (int)M.p.B, tile = M.p.tile;
    uint32_t *__restrict__ cnt = M.ws.cnt;
    DevHeader *hdr = M.ws.hdr;
    const long long t = vb.b;
    for (int b = threadIdx.x; b < B; b += blockDim.x) hist[b] = 0;
    __syncthreads();
    const long long k0 = t * (long long)tile;
    const long long k1 = min(C, k0 + tile);
    bool bad = false;
    for (long long i = t * (long long)blockDim.x + threadIdx.x; i < M.p.R; i += vb.g * (long long)blockDim.x)
        bad |= ldo<OffT>(M.in.row_ptr, i + 1) < ldo<OffT>(M.in.row_ptr, i);
    if (t >= M.p.T) {  // the check alone
        if (bad) flag(hdr, ST_BADINPUT);
        return;
    }
    const bool vec = ((reinterpret_cast<uintptr_t>(col) & 15) == 0);
    if (vec) {
        long long q0 = k0 >> 2, q1 = k1 >> 2;  // tile is a multiple of 4
        const int4 *c4 = reinterpret_cast<const int4 *>(col);
        auto count = [&](const int4 &v) {
            const int cs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                long long c = cs[u];
                if (c < 0 || c >= N) { bad = true; c = c < 0 ? 0 : N - 1; }
                atomicAdd(&hist[c >> bshift], 1u);
            }
        };
        constexpr int HU = 2;  // loads in flight per thread
        const int nt = blockDim.x;
        long long q = q0 + threadIdx.x;
        for (; q + (HU - 1) * nt < q1; q += HU * nt) {
            int4 v[HU];
#pragma unroll
            for (int j = 0; j < HU; ++j) v[j] = __ldcs(c4 + q + j * nt);
#pragma unroll
            for (int j = 0; j < HU; ++j) count(v[j]);
        }
        for (; q < q1; q += nt) count(__ldcs(c4 + q));
        for (long long k = (q1 << 2) + threadIdx.x; k < k1; k += blockDim.x) {
            long long c = __ldcs(col + k);
            if (c < 0 || c >= N) { bad = true; c = c < 0 ? 0 : N - 1; }
            atomicAdd(&hist[c >> bshift], 1u);
        }
    } else {
        for (long long k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
            long long c = __ldcs(col + k);
            if (c < 0 || c >= N) { bad = true; c = c < 0 ? 0 : N - 1; }
            atomicAdd(&hist[c >> bshift], 1u);
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) flag(hdr, ST_BADINPUT);
    uint32_t *row = cnt + t * (long long)B;
    for (int b = threadIdx.x; b < B; b += blockDim.x) row[b] = hist[b];
}

// A block per tile, and where rows are many times the cells a block per four
// rounds of rows (30M rows, 3,000 cells in the last ones: 25.4 ms in all with
// one block, 0.23 with 608).
static long long grid_hist(const Params &p, double share) {
    const long long cap = std::max(1LL, (long long)(4.0 * sm_count() * share + 0.999));
    return std::max<long long>(std::max<long long>(1, p.T), std::min<long long>(cap, p.R / (4 * K_THREADS)));
}
static size_t smem_hist(const Params &p) { return (size_t)p.B * sizeof(uint32_t); }
static cudaError_t launch_hist(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                               cudaStream_t st) {
    auto kern = m0.p.o == 4 ? (ba.n ? k_hist<int32_t, true> : k_hist<int32_t, false>)
                            : (ba.n ? k_hist<int64_t, true> : k_hist<int64_t, false>);
    // a histogram that leaves room for one block per SM: a wide block (32,768 buckets 0.22 ->
    // 0.17 ms; 3,328 buckets 0.27 ms with 512 threads, 0.28 with 1,024)
    return launch_kernel(kern, ba.n > 0, grid, smem > 64 * 1024 ? 1024 : 512, smem, st, m0, ba);
}

// ------------------------------------------------------------ K2 scan tiles
// For 32 K buckets per block: replace cnt[t][b] by the exclusive prefix over
// tiles t' < t (keeps tiles, hence input order, inside each bucket) and
// write the bucket totals; warp w takes tiles [T w / 32, T (w + 1) / 32).
// K = 1: a lane per bucket.  K = 4, for count matrices of many tiles: a lane
// per 4 neighbouring buckets (16-byte loads when B is a multiple of 4), so
// that a warp reads 512 contiguous bytes of a tile's row instead of 128 (the
// rows lie tens of kilobytes apart); with few tiles the 4x larger blocks
// would leave SMs idle.
__host__ __device__ inline int scan_tiles_k(const Params &p) { return p.T >= 4096 ? 4 : 1; }

template <int K>
__device__ __forceinline__ void scan_tiles_body(const Mat &M, long long blk,
                                                unsigned long long (*part)[32][33]) {
    uint32_t *cnt = M.ws.cnt;
    const long long T = M.p.T, B = M.p.B;
    unsigned long long *bucket_tot = M.ws.bucket_tot;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long b = blk * (32LL * K) + (long long)K * lane;  // buckets b .. b + K - 1
    const bool vec = K == 4 && (B & 3) == 0;
    const long long t0 = T * warp / nw, t1 = T * (warp + 1) / nw;
    auto load = [&](long long t, uint32_t *x) {
        const uint32_t *r = cnt + t * B;
        if (vec) {
            const uint4 v = *reinterpret_cast<const uint4 *>(r + b);
            x[0] = v.x;
            if (K == 4) { x[1] = v.y; x[2] = v.z; x[3] = v.w; }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) x[k] = b + k < B ? r[b + k] : 0u;
        }
    };
    unsigned long long sum[K];
#pragma unroll
    for (int k = 0; k < K; ++k) sum[k] = 0;
    if (b < B) {
        long long t = t0;
        for (; t + 4 / K <= t1 && K == 1; t += 4) {  // K = 1: four loads in flight
            uint32_t x0[K], x1[K], x2[K], x3[K];
            load(t, x0); load(t + 1, x1); load(t + 2, x2); load(t + 3, x3);
            sum[0] += (unsigned long long)x0[0] + x1[0] + x2[0] + x3[0];
        }
        for (; t + 2 <= t1 && K == 4; t += 2) {
            uint32_t x[K], y[K];
            load(t, x);
            load(t + 1, y);
#pragma unroll
            for (int k = 0; k < K; ++k) sum[k] += (unsigned long long)x[k] + y[k];
        }
        for (; t < t1; ++t) {
            uint32_t x[K];
            load(t, x);
#pragma unroll
            for (int k = 0; k < K; ++k) sum[k] += x[k];
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) part[k][warp][lane] = sum[k];
    __syncthreads();
    if (warp < K) {  // warp q: the prefix over warps of each lane's bucket b + q
        unsigned long long run = 0;
        for (int w = 0; w < nw; ++w) {
            const unsigned long long v = part[warp][w][lane];
            part[warp][w][lane] = run;
            run += v;
        }
        if (b + warp < B) bucket_tot[b + warp] = run;
    }
    __syncthreads();
    if (b < B) {
        unsigned long long run[K];
#pragma unroll
        for (int k = 0; k < K; ++k) run[k] = part[k][warp][lane];
        long long t = t0;
        for (; t + 4 <= t1 && K == 1; t += 4) {  // K = 1: four loads in flight
            uint32_t x0[K], x1[K], x2[K], x3[K];
            load(t, x0); load(t + 1, x1); load(t + 2, x2); load(t + 3, x3);
            uint32_t *r = cnt + t * B + b;
            r[0] = (uint32_t)run[0];
            r[B] = (uint32_t)(run[0] + x0[0]);
            r[2 * B] = (uint32_t)(run[0] + x0[0] + x1[0]);
            r[3 * B] = (uint32_t)(run[0] + x0[0] + x1[0] + x2[0]);
            run[0] += (unsigned long long)x0[0] + x1[0] + x2[0] + x3[0];
        }
        for (; t < t1; ++t) {
            uint32_t x[K];
            load(t, x);
            uint32_t *r = cnt + t * B;  // within-bucket offsets (< 2^32 by plan)
            if (vec) {
                *reinterpret_cast<uint4 *>(r + b) =
                    make_uint4((uint32_t)run[0], (uint32_t)run[K > 1 ? 1 : 0], (uint32_t)run[K > 2 ? 2 : 0],
                               (uint32_t)run[K > 3 ? 3 : 0]);
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (b + k < B) r[b + k] = (uint32_t)run[k];
            }
#pragma unroll
            for (int k = 0; k < K; ++k) run[k] += x[k];
        }
    }
}

// The block that finishes last also turns the buckets' totals into their
// bases (exclusive prefix), 4,096 buckets a round: a launch less, and 12
// instead of 64 us for 32,768 buckets (one block, 32 strided loads a thread).
template <bool BATCH>
__global__ void __launch_bounds__(1024) k_scan_tiles(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ unsigned long long part[4][32][33];
    __shared__ unsigned long long wsum[33];
    __shared__ int last;
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    if (scan_tiles_k(M.p) == 4) scan_tiles_body<4>(M, vb.b, part);
    else scan_tiles_body<1>(M, vb.b, part);
    __threadfence();
    __syncthreads();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) last = atomicAdd(&M.ws.hdr->scan_done, 1ull) == (unsigned long long)vb.g - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const unsigned long long *tot = M.ws.bucket_tot;
    unsigned long long *base = M.ws.bucket_base;
    const long long B = M.p.B;
    unsigned long long carry = 0;
    for (long long b0 = 0; b0 < B; b0 += 4096) {
        const long long b = b0 + 4 * tid;
        unsigned long long x[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[k] = b + k < B ? __ldcg(tot + b + k) : 0ull;
            sum += x[k];
        }
        const unsigned long long inc = warp_inclusive_scan(sum);
        __syncthreads();
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long v = wsum[lane], vi = warp_inclusive_scan(v);
            wsum[lane] = vi - v;
            if (lane == 31) wsum[32] = vi;
        }
        __syncthreads();
        unsigned long long run = carry + wsum[warp] + inc - sum;
        carry += wsum[32];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (b + k < B) base[b + k] = run;
            run += x[k];
        }
    }
}

static long long grid_scan_tiles(const Params &p, double) {
    const long long per = 32LL * scan_tiles_k(p);
    return (p.B + per - 1) / per;
}
static cudaError_t launch_scan_tiles(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                                     cudaStream_t st) {
    return launch_kernel(ba.n ? k_scan_tiles<true> : k_scan_tiles<false>, ba.n > 0, grid, 1024, 0, st, m0, ba);
}

static long long grid_none(const Params &, double) { return 0; }

// ------------------------------------------------------------ K4 build work
// Value bases per bucket (exclusive prefix of bucket_vtot) and the sort work
// list.  A bucket with at most `ch` records (one sort block or cluster) is one
// item; a larger one is cut into ceil(n / chm) chunks that get cursor-matrix
// rows.  A block per 1,024 buckets: it adds up the buckets before its own
// (values, items, chunk rows, chunked buckets), scans its own and writes their
// items, the chunks of hot buckets by all its threads.  Reading all earlier
// buckets again costs less than a second launch or a chain of waits: 32,768
// buckets 0.13 -> 0.03 ms, with 36,000 chunks 0.22 -> 0.04 ms (one block before).
constexpr int BW_THREADS = 1024;
template <bool BATCH>
__global__ void __launch_bounds__(BW_THREADS) k_build_work(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ unsigned long long sc[4][32], sum[4];
    __shared__ uint32_t huge[BW_THREADS];
    __shared__ int nhuge;
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const long long B = M.p.B, ch = M.p.ch, chm = M.p.chm, V = M.p.V;
    const unsigned long long *bucket_tot = M.ws.bucket_tot, *bucket_base = M.ws.bucket_base,
                             *bucket_vtot = M.ws.bucket_vtot;
    WorkItem *items = M.ws.items;
    DevHeader *hdr = M.ws.hdr;
    const unsigned long long max_items = M.p.max_items, max_rows = M.p.max_multi_rows,
                             max_mb = M.p.max_multi_buckets;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // one bucket's share of the four running sums
    auto shares = [&](long long b, unsigned long long *x) {
        const unsigned long long n = bucket_tot[b];
        const bool big = n > (unsigned long long)ch;
        x[0] = bucket_vtot[b];
        x[2] = big ? (n + chm - 1) / chm : 0ull;
        x[1] = big ? x[2] : 1ull;
        x[3] = big ? 1ull : 0ull;
        return n;
    };
    const long long own = vb.b * BW_THREADS;
    unsigned long long before[4] = {0, 0, 0, 0};
    {
#pragma unroll 4
        for (long long b = tid; b < own; b += BW_THREADS) {
            unsigned long long x[4];
            shares(b, x);
#pragma unroll
            for (int q = 0; q < 4; ++q) before[q] += x[q];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) before[q] += __shfl_xor_sync(0xffffffffu, before[q], d);
            if (lane == 0) sc[q][warp] = before[q];
        }
        if (tid == 0) nhuge = 0;
        __syncthreads();
        if (warp < 4) {
            unsigned long long v = sc[warp][lane];
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
            if (lane == 0) sum[warp] = v;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) before[q] = sum[q];
        __syncthreads();
    }
    const long long b = own + tid;
    const bool valid = b < B;
    unsigned long long x[4] = {0, 0, 0, 0}, at[4], n = 0;
    if (valid) n = shares(b, x);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned long long inc = warp_inclusive_scan(x[q]);
        if (lane == 31) sc[q][warp] = inc;
        at[q] = before[q] + inc - x[q];
    }
    __syncthreads();
    if (warp < 4) {
        const unsigned long long v = sc[warp][lane], inc = warp_inclusive_scan(v);
        sc[warp][lane] = inc - v;
        if (lane == 31) sum[warp] = inc;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        at[q] += sc[q][warp];
        before[q] += sum[q];  // through this block's buckets
    }
    // writes past the plan's capacities are skipped and reported by the last block
    if (valid) {
        const unsigned long long bb = bucket_base[b];
        M.ws.bucket_vbase[b] = at[0];
        if (x[3] == 0) {
            if (at[1] < max_items) {
                WorkItem it;
                it.r0 = bb;
                it.r1 = bb + n;
                it.bucket = (uint32_t)b;
                it.chunk = 0;
                it.mc = ~0ull;
                items[at[1]] = it;
            }
        } else if (at[3] < max_mb && at[2] + x[2] <= max_rows && at[1] + x[2] <= max_items) {
            MultiBucket mb;
            mb.mc0 = at[2];
            mb.bucket = (uint32_t)b;
            mb.nch = (uint32_t)x[2];
            mb.done = 0;
            M.ws.multi_buckets[at[3]] = mb;
            M.ws.multi_items[at[2]] = (uint32_t)at[1];  // the first chunk's item
            huge[atomicAdd(&nhuge, 1)] = (uint32_t)at[3];
        }
    }
    __syncthreads();
    // chunks: a warp per chunked bucket, or the whole block for the longest ones
    auto chunk_items = [&](const MultiBucket &mb, unsigned long long h0, unsigned long long hs) {
        const unsigned long long cells = bucket_tot[mb.bucket], bb = bucket_base[mb.bucket], nch = mb.nch;
        const unsigned long long first = M.ws.multi_items[mb.mc0];
        for (unsigned long long h = h0; h < nch; h += hs) {
            WorkItem it;
            it.r0 = bb + (cells * h) / nch;
            it.r1 = bb + (cells * (h + 1)) / nch;
            it.bucket = mb.bucket;
            it.chunk = (uint32_t)h;
            it.mc = mb.mc0 + h;
            items[first + h] = it;
            if (h > 0) M.ws.multi_items[mb.mc0 + h] = (uint32_t)(first + h);
        }
    };
    constexpr uint32_t LONG = 512;
    for (int k = warp; k < nhuge; k += 32) {
        const MultiBucket mb = M.ws.multi_buckets[huge[k]];
        if (mb.nch <= LONG) chunk_items(mb, lane, 32);
    }
    for (int k = 0; k < nhuge; ++k) {
        const MultiBucket mb = M.ws.multi_buckets[huge[k]];
        if (mb.nch > LONG) chunk_items(mb, tid, BW_THREADS);
    }
    if (vb.b == vb.g - 1 && tid == 0) {  // the totals
        const bool consistent = (hdr->status & ST_BADINPUT) == 0 && before[0] == (unsigned long long)V;
        const bool fits = before[1] <= max_items && before[2] <= max_rows && before[3] <= max_mb;
        if (!consistent) flag(hdr, ST_BADINPUT);
        else if (!fits) flag(hdr, ST_OVERFLOW);
        const bool go = consistent && fits;
        hdr->n_items = go ? before[1] : 0;
        hdr->n_multi_items = go ? before[2] : 0;
        hdr->n_multi_buckets = go ? before[3] : 0;
        hdr->max_items = max_items;  // bounds for debug-build checks
        hdr->max_rows = max_rows;
    }
}

static long long grid_build_work(const Params &p, double) { return (p.B + BW_THREADS - 1) / BW_THREADS; }
static cudaError_t launch_build_work(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                                     cudaStream_t st) {
    return launch_kernel(ba.n ? k_build_work<true> : k_build_work<false>, ba.n > 0, grid, BW_THREADS, 0, st, m0, ba);
}
static cudaError_t launch_none(const Mat &, const BatchArgs &, long long, size_t, cudaStream_t) { return cudaSuccess; }

const PhaseOps kBucketPhases[5] = {
    {"setup", grid_prep, smem_none, launch_prep, nullptr, nullptr},
    {"hist", grid_hist, smem_hist, launch_hist, nullptr, nullptr},
    {"scan_tiles", grid_scan_tiles, smem_none, launch_scan_tiles, nullptr, nullptr},
    {"scan_buckets", grid_none, smem_none, launch_none, nullptr, nullptr},  // in scan_tiles
    {"build_work", grid_build_work, smem_none, launch_build_work, nullptr, nullptr},
};

}  // namespace mgt
