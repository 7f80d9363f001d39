// Level 1 of the transpose: stable scatter of cell records into column buckets.
//
// The paper exchanges cells between ranks by destination (Sec. 3, view swap:
// metadata, then values).  On one GPU the destination of a cell is a bucket of
// consecutive output rows (= input columns); K1-K3 deal every cell's record
// into its bucket, keeping row-major input order inside each bucket, so that
// the per-bucket sort of K7 only has to order by column.
#include "mgt_internal.cuh"

#include <algorithm>

#include <cooperative_groups.h>

namespace mgt {

constexpr int K_THREADS = 512;

// ------------------------------------------------------------------ K0 prep
// Checks the pointer arrays' end points and that row_ptr never decreases;
// writes the source blocks' cell offsets pcoff[s] = row_ptr[off[s]], the
// output sentinels row_ptr'[N] = C and cell_ptr'[C] = V, and the P = 1 counts.
template <typename OffT, bool BATCH>
__global__ void __launch_bounds__(K_THREADS) k_prep(const __grid_constant__ Mat m0, const BatchArgs ba) {
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const void *row_ptr = M.in.row_ptr, *cell_ptr = M.in.cell_ptr;
    const long long R = M.p.R, N = M.p.N, C = M.p.C, V = M.p.V, B = M.p.B;
    const int P = M.p.P, bshift = M.p.bshift;
    const long long *poff = M.ws.poff;
    long long *pcoff = M.ws.pcoff;
    uint16_t *dblock = M.ws.dblock;
    void *out_row_ptr = M.out.row_ptr, *out_cell_ptr = M.out.cell_ptr;
    long long *part_cells = M.out.part_cells, *part_values = M.out.part_values;
    DevHeader *hdr = M.ws.hdr;
    long long gid = vb.b * (long long)blockDim.x + threadIdx.x;
    long long stride = vb.g * (long long)blockDim.x;
    if (gid == 0) {
        if (ldo<OffT>(row_ptr, 0) != 0 || ldo<OffT>(row_ptr, R) != C) flag(hdr, ST_BADINPUT);
        if (ldo<OffT>(cell_ptr, 0) != 0 || ldo<OffT>(cell_ptr, C) != V) flag(hdr, ST_BADINPUT);
        sto<OffT>(out_row_ptr, N, C);
        sto<OffT>(out_cell_ptr, C, V);
        if (P == 1 && part_cells) part_cells[0] = C;
        if (P == 1 && part_values) part_values[0] = V;
    }
    for (long long s = gid; s <= P; s += stride) {
        long long r = poff[s];
        pcoff[s] = (r >= 0 && r <= R) ? ldo<OffT>(row_ptr, r) : 0;
    }
    // destination block of each bucket's columns, or 0xFFFF when they span two
    for (long long b = gid; b < B && P > 1; b += stride) {
        const long long c0 = b << bshift, c1 = min(N, c0 + (1LL << bshift)) - 1;
        long long da = upper_bound_ll(poff, 0, P + 1, c0) - 1, db = upper_bound_ll(poff, 0, P + 1, c1) - 1;
        da = da < 0 ? 0 : (da >= P ? P - 1 : da);
        dblock[b] = (da == db) ? (uint16_t)da : (uint16_t)0xFFFFu;
    }
    // row of every 2^ROWAT_SHIFT-th cell, for the scatter pass: a warp takes 32
    // consecutive boundaries, finds the first and the last by a 32-way search
    // (few dependent loads) and each lane its own between them
    if (R > 0 && C > 0) {
        uint32_t *rowat = row_table(M.ws);
        const int lane = threadIdx.x & 31;
        const long long nb = row_table_entries(C);
        for (long long b0 = (gid >> 5) * 32; b0 < nb; b0 += stride) {
            auto find = [&](long long key) {  // entries of row_ptr at or below key
                long long a = 0, n = R + 1;
                while (n > 0) {
                    const long long step = (n + 31) / 32, i = a + (lane + 1) * step - 1;
                    const bool below = i < a + n && ldo<OffT>(row_ptr, i) <= key;
                    const int c = __popc(__ballot_sync(0xffffffffu, below));
                    const long long e = a + n;
                    a += c * step;
                    n = step > 1 ? min(step - 1, e - a) : 0;
                }
                return a;
            };
            const long long k = (b0 + lane) << ROWAT_SHIFT;
            const long long f = find(b0 << ROWAT_SHIFT), l = find(min(b0 + 31, nb - 1) << ROWAT_SHIFT);
            if (b0 + lane < nb) {
                long long r = k >= C ? R - 1 : upper_bound_g<OffT>(row_ptr, f - 1 < 0 ? 0 : f - 1, l, k) - 1;
                r = r < 0 ? 0 : (r > R - 1 ? R - 1 : r);
                rowat[b0 + lane] = (uint32_t)r;
            }
        }
    }
    bool bad = false;
    for (long long i = gid; i < R; i += stride)
        bad |= ldo<OffT>(row_ptr, i + 1) < ldo<OffT>(row_ptr, i);
    if (__syncthreads_or(bad) && threadIdx.x == 0) flag(hdr, ST_BADINPUT);
}

static long long grid_prep(const Params &p, double share) {
    const long long full = 4LL * sm_count();
    long long want = (std::max<long long>(p.R, row_table_entries(p.C)) + K_THREADS - 1) / K_THREADS;
    long long cap = (long long)(full * share + 0.999);
    if (cap < 1) cap = 1;
    if (want > cap) want = cap;
    return want < 1 ? 1 : want;
}
static size_t smem_none(const Params &) { return 0; }
static cudaError_t launch_prep(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                               cudaStream_t st) {
    auto kern = m0.p.o == 4 ? (ba.n ? k_prep<int32_t, true> : k_prep<int32_t, false>)
                            : (ba.n ? k_prep<int64_t, true> : k_prep<int64_t, false>);
    kern<<<(unsigned)grid, K_THREADS, 0, st>>>(m0, ba);
    return cudaGetLastError();
}

// Zeroes the header, the per-bucket value totals and the P x P outputs of
// every matrix of a batch (one transpose alone uses memsets instead).
template <bool BATCH>
__global__ void __launch_bounds__(K_THREADS) k_zero(const __grid_constant__ Mat m0, const BatchArgs ba) {
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const long long gid = vb.b * (long long)blockDim.x + threadIdx.x;
    const long long stride = vb.g * (long long)blockDim.x;
    unsigned long long *h = reinterpret_cast<unsigned long long *>(M.ws.hdr);
    for (long long i = gid; i < 32; i += stride) h[i] = 0;
    for (long long i = gid; i < M.p.B; i += stride) M.ws.bucket_vtot[i] = 0;
    const long long pp = (long long)M.p.P * M.p.P;
    if (M.out.part_cells)
        for (long long i = gid; i < pp; i += stride) { M.out.part_cells[i] = 0; M.out.part_values[i] = 0; }
}

long long grid_zero(const Params &p, double) {
    const long long n = std::max<long long>(std::max<long long>(32, p.B), (long long)p.P * p.P);
    const long long g = (n + K_THREADS - 1) / K_THREADS;
    return g < 64 ? g : 64;
}
cudaError_t launch_zero(const Mat &m0, const BatchArgs &ba, long long grid, size_t, cudaStream_t st) {
    k_zero<true><<<(unsigned)grid, K_THREADS, 0, st>>>(m0, ba);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ K1 hist
// Cells per bucket for one tile of `tile` consecutive cells, in a shared
// memory histogram; written as row t of the T x B count matrix.
template <bool BATCH>
__global__ void __launch_bounds__(K_THREADS) k_hist(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ uint32_t hist[];
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
    const bool vec = ((reinterpret_cast<uintptr_t>(col) & 15) == 0);
    if (vec) {
        long long q0 = k0 >> 2, q1 = k1 >> 2;  // tile is a multiple of 4
        const int4 *c4 = reinterpret_cast<const int4 *>(col);
        for (long long q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
            int4 v = __ldcs(c4 + q);
            int cs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                long long c = cs[u];
                if (c < 0 || c >= N) { bad = true; c = c < 0 ? 0 : N - 1; }
                atomicAdd(&hist[c >> bshift], 1u);
            }
        }
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

static long long grid_hist(const Params &p, double) { return p.T; }
static size_t smem_hist(const Params &p) { return (size_t)p.B * sizeof(uint32_t); }
static cudaError_t launch_hist(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                               cudaStream_t st) {
    auto kern = ba.n ? k_hist<true> : k_hist<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, K_THREADS, smem, st>>>(m0, ba);
    return cudaGetLastError();
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

template <bool BATCH>
__global__ void __launch_bounds__(1024) k_scan_tiles(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ unsigned long long part[4][32][33];
    const VBlock vb = vblock<BATCH>(m0, ba);
    if (scan_tiles_k(vb.m->p) == 4) scan_tiles_body<4>(*vb.m, vb.b, part);
    else scan_tiles_body<1>(*vb.m, vb.b, part);
}

static long long grid_scan_tiles(const Params &p, double) {
    const long long per = 32LL * scan_tiles_k(p);
    return (p.B + per - 1) / per;
}
static cudaError_t launch_scan_tiles(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                                     cudaStream_t st) {
    (ba.n ? k_scan_tiles<true> : k_scan_tiles<false>)<<<(unsigned)grid, 1024, 0, st>>>(m0, ba);
    return cudaGetLastError();
}

// ---------------------------------------------------------- K2b scan buckets
// One block: exclusive prefix of the 64-bit per-bucket totals.
template <bool BATCH>
__global__ void __launch_bounds__(1024) k_scan_u64(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ unsigned long long scratch[33];
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const unsigned long long *in = M.ws.bucket_tot;
    unsigned long long *out = M.ws.bucket_base;
    const long long n = M.p.B;
    const int nt = blockDim.x, tid = threadIdx.x;
    long long per = (n + nt - 1) / nt, lo = min(n, tid * per), hi = min(n, lo + per);
    unsigned long long sum = 0;
    for (long long i = lo; i < hi; ++i) sum += in[i];
    unsigned long long incl = warp_inclusive_scan(sum);
    if ((tid & 31) == 31) scratch[tid >> 5] = incl;
    __syncthreads();
    if (tid < 32) {
        unsigned long long v = tid < (nt >> 5) ? scratch[tid] : 0ull;
        unsigned long long vi = warp_inclusive_scan(v);
        scratch[tid] = vi - v;
    }
    __syncthreads();
    unsigned long long run = scratch[tid >> 5] + incl - sum;
    for (long long i = lo; i < hi; ++i) {
        unsigned long long x = in[i];
        out[i] = run;
        run += x;
    }
}

static long long grid_one_if_buckets(const Params &p, double) { return p.B > 0 ? 1 : 0; }
static cudaError_t launch_scan_buckets(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                                       cudaStream_t st) {
    (ba.n ? k_scan_u64<true> : k_scan_u64<false>)<<<(unsigned)grid, 1024, 0, st>>>(m0, ba);
    return cudaGetLastError();
}

// ------------------------------------------------------------ K4 build work
// One block: value bases per bucket (exclusive prefix of bucket_vtot) and the
// sort work list.  A bucket with at most `ch` records (one sort cluster) is
// one item; a larger one is cut into ceil(n / chm) chunks that get
// cursor-matrix rows.
template <bool BATCH>
__global__ void __launch_bounds__(1024) k_build_work(const __grid_constant__ Mat m0, const BatchArgs ba) {
    __shared__ unsigned long long sc[4][33];
    __shared__ uint32_t huge[64];
    __shared__ int nhuge;
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    const long long B = M.p.B, ch = M.p.ch, chm = M.p.chm, V = M.p.V;
    const unsigned long long *bucket_tot = M.ws.bucket_tot, *bucket_base = M.ws.bucket_base,
                             *bucket_vtot = M.ws.bucket_vtot;
    unsigned long long *bucket_vbase = M.ws.bucket_vbase;
    WorkItem *items = M.ws.items;
    uint32_t *multi_items = M.ws.multi_items;
    MultiBucket *multi_buckets = M.ws.multi_buckets;
    DevHeader *hdr = M.ws.hdr;
    const unsigned long long max_items = M.p.max_items, max_rows = M.p.max_multi_rows,
                             max_mb = M.p.max_multi_buckets;
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    if (tid == 0) nhuge = 0;
    // Rounds of nt consecutive buckets (coalesced loads, one bucket per
    // thread): a block scan of four running sums -- values, items,
    // multi-chunk rows, multi-chunk buckets -- gives each bucket its value
    // base and the place of its items.  A bucket of one sort cluster is one
    // item, written here; a larger one gets its MultiBucket entry, and the
    // index of its first item is parked in multi_items[mc0] for the last
    // pass, which writes its chunks' items.  Writes past the plan's
    // capacities are skipped and reported at the end.
    unsigned long long cv = 0, ci = 0, cr = 0, cm = 0;  // carries (block-uniform)
    for (long long c0 = 0; c0 < B; c0 += nt) {
        const long long b = c0 + tid;
        const bool valid = b < B;
        unsigned long long n = 0, vt = 0, bb = 0, nch = 0;
        if (valid) {
            n = bucket_tot[b];
            vt = bucket_vtot[b];
            bb = bucket_base[b];
        }
        const bool big = valid && n > (unsigned long long)ch;
        if (big) nch = (n + chm - 1) / chm;
        unsigned long long x[4] = {vt, valid ? (big ? nch : 1ull) : 0ull, nch, big ? 1ull : 0ull};
        unsigned long long inc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            inc[q] = warp_inclusive_scan(x[q]);
            if (lane == 31) sc[q][warp] = inc[q];
        }
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned long long v = lane < nw ? sc[q][lane] : 0ull;
                const unsigned long long vi = warp_inclusive_scan(v);
                sc[q][lane] = vi - v;
                if (lane == 31) sc[q][32] = vi;
            }
        }
        __syncthreads();
        const unsigned long long ev = cv + sc[0][warp] + inc[0] - x[0];
        const unsigned long long ei = ci + sc[1][warp] + inc[1] - x[1];
        const unsigned long long er = cr + sc[2][warp] + inc[2] - x[2];
        const unsigned long long em = cm + sc[3][warp] + inc[3] - x[3];
        if (valid) {
            bucket_vbase[b] = ev;
            if (!big) {
                if (ei < max_items) {
                    WorkItem it;
                    it.r0 = bb;
                    it.r1 = bb + n;
                    it.bucket = (uint32_t)b;
                    it.chunk = 0;
                    it.mc = ~0ull;
                    items[ei] = it;
                }
            } else if (em < max_mb && er + nch <= max_rows) {
                MultiBucket mb;
                mb.mc0 = er;
                mb.bucket = (uint32_t)b;
                mb.nch = (uint32_t)nch;
                multi_buckets[em] = mb;
                multi_items[er] = (uint32_t)ei;  // first item; the last pass completes the row
            }
        }
        cv += sc[0][32];
        ci += sc[1][32];
        cr += sc[2][32];
        cm += sc[3][32];
        __syncthreads();
    }
    const bool consistent = (hdr->status & ST_BADINPUT) == 0 && cv == (unsigned long long)V;
    const bool fits = consistent && ci <= max_items && cr <= max_rows && cm <= max_mb;
    // the chunks of multi-chunk buckets: one thread per bucket, the whole
    // block for the buckets of many chunks (the hot columns' buckets)
    auto chunk_items = [&](const MultiBucket &mb, unsigned long long h0, unsigned long long hs) {
        const unsigned long long n = bucket_tot[mb.bucket], bb = bucket_base[mb.bucket];
        const unsigned long long ri0 = multi_items[mb.mc0], nch = mb.nch;
        for (unsigned long long h = h0; h < nch; h += hs) {
            WorkItem it;
            it.r0 = bb + (n * h) / nch;
            it.r1 = bb + (n * (h + 1)) / nch;
            it.bucket = mb.bucket;
            it.chunk = (uint32_t)h;
            it.mc = mb.mc0 + h;
            items[ri0 + h] = it;
            multi_items[mb.mc0 + h] = (uint32_t)(ri0 + h);  // h = 0 rewrites the parked value
        }
    };
    if (fits) {
        for (unsigned long long m = tid; m < cm; m += nt) {
            const MultiBucket mb = multi_buckets[m];
            if (mb.nch > 64) {
                const int k = atomicAdd(&nhuge, 1);
                if (k < 64) {
                    huge[k] = (uint32_t)m;
                    continue;
                }
            }
            chunk_items(mb, 0, 1);
        }
        __syncthreads();
        const int nh = min(nhuge, 64);
        for (int k = 0; k < nh; ++k) chunk_items(multi_buckets[huge[k]], tid, nt);
    }
    if (tid == 0) {
        if (!consistent) flag(hdr, ST_BADINPUT);
        else if (!fits) flag(hdr, ST_OVERFLOW);
        hdr->n_items = fits ? ci : 0;
        hdr->n_multi_items = fits ? cr : 0;
        hdr->n_multi_buckets = fits ? cm : 0;
        hdr->max_items = max_items;  // bounds for debug-build checks
        hdr->max_rows = max_rows;
    }
}

static cudaError_t launch_build_work(const Mat &m0, const BatchArgs &ba, long long grid, size_t,
                                     cudaStream_t st) {
    (ba.n ? k_build_work<true> : k_build_work<false>)<<<(unsigned)grid, 1024, 0, st>>>(m0, ba);
    return cudaGetLastError();
}

const PhaseOps kBucketPhases[5] = {
    {"setup", grid_prep, smem_none, launch_prep, nullptr, nullptr},
    {"hist", grid_hist, smem_hist, launch_hist, nullptr, nullptr},
    {"scan_tiles", grid_scan_tiles, smem_none, launch_scan_tiles, nullptr, nullptr},
    {"scan_buckets", grid_one_if_buckets, smem_none, launch_scan_buckets, nullptr, nullptr},
    {"build_work", grid_one_if_buckets, smem_none, launch_build_work, nullptr, nullptr},
};

}  // namespace mgt
