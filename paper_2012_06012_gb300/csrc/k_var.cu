// Value copy for values of individual byte widths: the paper's second
// variation of the exchange (Sec. 2, heterogeneous datatypes across edges,
// one MPI datatype per edge through MPI_Alltoallw).
//
// The cells are placed by the same kernels as for fixed-width values; their
// runs are then moved as byte ranges.  Every output cell q knows the first
// input value of its run (src) and its value count (from cell_ptr'); the
// run's bytes are [val_off[src], val_off[src + len]).  One kernel, a block per
// tile of 2^cshift output cells, tiles taken in order from a counter:
//   1. each cell's run start and byte size (its val_off end points), the
//      cells' byte offsets in the tile (block scan) and the tile's byte total;
//   2. the tile's byte base from the tiles before it: a chained scan (each
//      tile publishes its total, then its inclusive prefix, and adds up its
//      predecessors' words, 32 at a time, until one holds an inclusive prefix
//      -- Merrill and Garland's decoupled look-back); the wait is bounded;
//   3. the bytes, by the tile copy of the fixed-width values (units as wide as
//      every offset and length allows), and the output value offsets.
// A tile only ever waits for tiles taken before it, by blocks that are
// running and publish their totals without waiting, so the chain always
// completes; a wait that runs out of iterations flags MGT_ETIMEOUT and the
// tile publishes anyway so that no later tile waits on it.
//
// Bound by random sectors: a run costs its val_off entries and its bytes at
// two random places.  1.5M x 1.5M, 30M runs of 130 bytes: 5.26 -> 2.95 ms against
// a persistent grid of 2,048-cell tiles that found its runs by 64-bit shuffles.
#include "k_place_impl.cuh"

namespace mgt {

__device__ __forceinline__ bool structure_ok(const DevHeader *hdr) {
    return (*(volatile const unsigned *)&hdr->status & (ST_BADINPUT | ST_OVERFLOW)) == 0;
}

// Tile words of the chained scan: flag in the top two bits, bytes below.
constexpr unsigned long long TW_AGG = 1ull << 62;  // the tile's own byte total
constexpr unsigned long long TW_PRE = 2ull << 62;  // its inclusive prefix
constexpr unsigned long long TW_VAL = (1ull << 62) - 1;
constexpr int LOOKBACK_POLLS = 1 << 22;            // polls of one group of predecessors before giving up

// Bytes before tile t (one warp, 32 words a step; 256 a step was slower, 3.39
// instead of 3.34 ms, more so on smaller tiles); false if a wait ran out.
__device__ __forceinline__ bool look_back(const unsigned long long *words, long long t, unsigned long long *prefix) {
    const int lane = lane_id();
    unsigned long long sum = 0;
    for (long long p = t - 1; p >= 0; p -= 32) {
        unsigned pre = 0;
        int polls = 0;
        for (;;) {
            const unsigned long long w =
                p - lane >= 0 ? *reinterpret_cast<const volatile unsigned long long *>(words + p - lane) : TW_PRE;
            pre = __ballot_sync(0xffffffffu, (w & TW_PRE) != 0);
            const unsigned missing = __ballot_sync(0xffffffffu, (w & ~TW_VAL) == 0);
            // the words down to the nearest prefix are needed
            const unsigned need = pre ? (pre & (0u - pre)) | ((pre & (0u - pre)) - 1u) : 0xffffffffu;
            if ((missing & need) == 0) {
                unsigned long long x = (need >> lane) & 1u ? w & TW_VAL : 0ull;
#pragma unroll
                for (int d = 16; d >= 1; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
                sum += x;
                break;
            }
            if (++polls > LOOKBACK_POLLS) {
                *prefix = sum;
                return false;
            }
            __nanosleep(32);
        }
        if (pre) break;
    }
    *prefix = sum;
    return true;
}

template <typename OffT, typename SrcT>
__global__ void __launch_bounds__(CP_THREADS, 4) k_var_copy(const __grid_constant__ Mat m) {
    __shared__ uint32_t off[CP_OFF];          // runs in the byte copy (units), then values of the runs
    __shared__ const uint8_t *sb[CP_CELLS];   // ... and where their units come from
    __shared__ long long vs[CP_CELLS];        // ... and their value offsets
    __shared__ long long add[CP_CELLS];       // what turns an input value offset into the output's
    __shared__ long long last[CP_CELLS];      // the input offset after the run's last value
    __shared__ uint16_t gcell[CP_GROUPS];
    __shared__ int wcount[2][CP_CELLS / 32];  // non-empty runs (bytes, values) per 32 cells
    __shared__ unsigned long long wsum[CP_CELLS / 32 + 1];
    __shared__ unsigned walign[CP_WARPS];
    __shared__ unsigned long long base_sh;
    __shared__ long long tile_sh;
    __shared__ int stop_sh;
    pipeline_wait<false>();
    DevHeader *hdr = m.ws.hdr;
    const long long C = m.p.C, V = m.p.V, nb = m.p.nbytes;
    const SrcT *__restrict__ src = reinterpret_cast<const SrcT *>(m.ws.src);
    const void *cp = m.out.cell_ptr;
    const long long *__restrict__ vo = m.in.val_off;
    long long *__restrict__ ovo = m.out.val_off;
    const uint8_t *in = m.in.values;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cshift = m.p.cshift;
    const long long ntiles = (C + (1LL << cshift) - 1) >> cshift;
    unsigned long long *words = m.ws.vblk;        // [ntiles], zeroed by the set-up kernel
    unsigned long long *counter = words + ntiles;  // next tile to take, zeroed too
    if (blockIdx.x == 0 && tid == 0) {
        if (__ldg(vo) != 0 || __ldg(vo + V) != nb) flag(hdr, ST_BADINPUT);
        ovo[0] = 0;
        ovo[V] = nb;
    }
    if (!structure_ok(hdr)) {  // malformed input: the cells were not placed (one decision for the block)
        if (tid == 0) tile_sh = -1;
    } else if (tid == 0) {
        tile_sh = (long long)atomicAdd(counter, 1ull);
    }
    __syncthreads();
    const long long t = tile_sh;
    if (t < 0 || t >= ntiles) return;
    const long long q0 = t << cshift;
    const int n0 = (int)min(1LL << cshift, C - q0);
    const long long v_first = ldp<OffT>(cp, q0), v_last = ldp<OffT>(cp, q0 + n0);
    // 1. this thread's cells (at most two): values [s, s + len), bytes [a, b)
    constexpr int PER = CP_CELLS / CP_THREADS;
    long long s[PER], c0[PER], len[PER], a[PER], b[PER];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = tid + k * CP_THREADS;
        s[k] = c0[k] = len[k] = a[k] = b[k] = 0;
        if (i < n0) {
            s[k] = (long long)src[q0 + i];
            c0[k] = ldp<OffT>(cp, q0 + i);
            len[k] = ldp<OffT>(cp, q0 + i + 1) - c0[k];
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (tid + k * CP_THREADS < n0) {
            if (s[k] < 0 || len[k] < 0 || s[k] > V - len[k] || c0[k] < v_first || c0[k] + len[k] > v_last) {
                bad = true;
                len[k] = 0;
            } else {
                a[k] = __ldg(vo + s[k]);
                b[k] = __ldg(vo + s[k] + len[k]);
            }
        }
    }
    unsigned maskb[PER], maskv[PER];
    unsigned long long inc[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (a[k] < 0 || b[k] < a[k] || b[k] > nb) {
            bad = true;
            a[k] = b[k] = 0;
        }
        maskb[k] = __ballot_sync(0xffffffffu, b[k] > a[k]);
        maskv[k] = __ballot_sync(0xffffffffu, len[k] > 0);
        inc[k] = warp_inclusive_scan((unsigned long long)(b[k] - a[k]));
        if (lane == 0) {
            wcount[0][k * CP_WARPS + warp] = __popc(maskb[k]);
            wcount[1][k * CP_WARPS + warp] = __popc(maskv[k]);
        }
        if (lane == 31) wsum[k * CP_WARPS + warp] = inc[k];
    }
    const bool any_bad = __syncthreads_or(bad);
    if (warp == 0) {
        constexpr int NW = PER * CP_WARPS;
        static_assert(NW <= 32, "one warp scans the warps' sums");
        const unsigned long long x = lane < NW ? wsum[lane] : 0ull, xi = warp_inclusive_scan(x);
        __syncwarp();
        if (lane < NW) wsum[lane] = xi - x;
        const unsigned long long agg = __shfl_sync(0xffffffffu, xi, 31);
        if (lane == 0) {
            wsum[NW] = agg;
            atomicExch(words + t, (t == 0 ? TW_PRE : TW_AGG) | (agg & TW_VAL));
        }
        // 2. the tile's byte base
        unsigned long long prefix = 0;
        const bool ok = look_back(words, t, &prefix);
        if (lane == 0) {
            // published even after a timeout, so that no later tile waits on this one
            if (t > 0) atomicExch(words + t, TW_PRE | ((prefix + agg) & TW_VAL));
            if (!ok) flag(hdr, ST_TIMEOUT);
            base_sh = prefix;
            stop_sh = !ok || prefix + agg > (unsigned long long)nb;
            // the runs do not cover the value bytes exactly
            if (ok && (stop_sh || (t == ntiles - 1 && prefix + agg != (unsigned long long)nb))) flag(hdr, ST_BADINPUT);
        }
    }
    __syncthreads();
    if (any_bad && tid == 0) flag(hdr, ST_BADINPUT);
    if (stop_sh || any_bad) return;
    const long long tb = (long long)base_sh, tbytes = (long long)wsum[PER * CP_WARPS];
    // the cells' byte offsets in the tile, and the copy's unit
    long long rel[PER];
    unsigned align = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        rel[k] = (long long)(wsum[k * CP_WARPS + warp] + inc[k]) - (b[k] - a[k]);
        if (b[k] > a[k]) align |= (unsigned)a[k] | (unsigned)(tb + rel[k]) | (unsigned)(b[k] - a[k]);
    }
    align = __reduce_or_sync(0xffffffffu, align);
    if (lane == 0) walign[warp] = align;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < CP_WARPS; ++w) align |= walign[w];
    align |= (unsigned)(reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(m.out.values));
    const int vshift = (align & 31) == 0 ? 5 : (align & 15) == 0 ? 4 : (align & 7) == 0 ? 3 : (align & 3) == 0 ? 2 : 0;
    // this thread's cells among the tile's non-empty ones
    auto place_of = [&](const int *counts, const unsigned (&mask)[PER], int k, int *total) {
        int at = __popc(mask[k] & lanemask_lt()), all = 0;
#pragma unroll
        for (int w = 0; w < PER * CP_WARPS; ++w) {
            at += w < k * CP_WARPS + warp ? counts[w] : 0;
            all += counts[w];
        }
        *total = all;
        return at;
    };
    // 3a. the bytes
    const long long units = tbytes >> vshift;
    uint8_t *out = m.out.values + tb;
    if (units > 32LL * CP_GROUPS) {  // long runs: a warp per run, the whole block for the very long ones
        constexpr long long WIDE = 1 << 16;
        long long *ra = vs, *rr = add, *rl = last;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int i = tid + k * CP_THREADS;
            if (i < n0) { ra[i] = a[k]; rr[i] = rel[k]; rl[i] = b[k] - a[k]; }
        }
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {
            for (int i = pass ? 0 : warp; i < n0; i += pass ? 1 : CP_WARPS) {
                if ((rl[i] >= WIDE) != (pass != 0)) continue;
                const int x = pass ? tid : lane, nx = pass ? CP_THREADS : 32;
                if (vshift == 5) copy_long<32>(in + ra[i], out + rr[i], rl[i] >> 5, x, nx);
                else if (vshift == 4) copy_long<16>(in + ra[i], out + rr[i], rl[i] >> 4, x, nx);
                else if (vshift == 3) copy_long<8>(in + ra[i], out + rr[i], rl[i] >> 3, x, nx);
                else if (vshift == 2) copy_long<4>(in + ra[i], out + rr[i], rl[i] >> 2, x, nx);
                else copy_long<1>(in + ra[i], out + rr[i], rl[i], x, nx);
            }
        }
        __syncthreads();
    } else {
        int n = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int at = place_of(wcount[0], maskb, k, &n);
            if (b[k] > a[k]) {
                const uint32_t o0 = (uint32_t)(rel[k] >> vshift), o1 = (uint32_t)((rel[k] + b[k] - a[k]) >> vshift);
                off[at] = o0;
                sb[at] = in + (a[k] - rel[k]);
                for (uint32_t g = (o0 + 31) >> 5; (g << 5) < o1; ++g) gcell[g] = (uint16_t)at;
            }
        }
        if (warp == 0) off[n + 1 + lane] = ~0u;
        if (tid == 0) off[n] = (uint32_t)units;
        __syncthreads();
        if (vshift == 5) copy_tile<32, 2>(out, off, sb, gcell, (uint32_t)units);
        else if (vshift == 4) copy_tile<16, 4>(out, off, sb, gcell, (uint32_t)units);
        else if (vshift == 3) copy_tile<8, 8>(out, off, sb, gcell, (uint32_t)units);
        else if (vshift == 2) copy_tile<4, 16>(out, off, sb, gcell, (uint32_t)units);
        else copy_tile<1, 16>(out, off, sb, gcell, (uint32_t)units);
        __syncthreads();
    }
    // 3b. the output value offsets, value by value
    const long long nv = v_last - v_first;
    int n = 0;
    const bool mapped = nv <= 32LL * CP_GROUPS;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int at = place_of(wcount[1], maskv, k, &n);
        if (len[k] > 0) {
            if (mapped) {
                const uint32_t o0 = (uint32_t)(c0[k] - v_first), o1 = o0 + (uint32_t)len[k];
                off[at] = o0;
                for (uint32_t g = (o0 + 31) >> 5; (g << 5) < o1; ++g) gcell[g] = (uint16_t)at;
            }
            const int x = mapped ? at : tid + k * CP_THREADS;
            vs[x] = mapped ? s[k] - (c0[k] - v_first) : s[k];
            add[x] = tb + rel[k] - a[k];
            last[x] = b[k];
        }
    }
    if (mapped && warp == 0) off[n + 1 + lane] = ~0u;
    if (mapped && tid == 0) off[n] = (uint32_t)nv;
    __syncthreads();
    bool wrong = false;
    if (mapped) {
        const unsigned le = lanemask_lt() | (1u << lane);
        const uint32_t groups = ((uint32_t)nv + 31) >> 5;
        constexpr int VU = 4;
        for (uint32_t g0 = warp * VU; g0 < groups; g0 += CP_WARPS * VU) {
            long long x[VU], y[VU];
            int c[VU];
#pragma unroll
            for (int j = 0; j < VU; ++j) {
                const uint32_t g = g0 + j, u = (g << 5) + lane;
                x[j] = y[j] = 0;
                c[j] = 0;
                if (g < groups) {
                    const int cc = gcell[g];
                    const unsigned marks = __reduce_or_sync(0xffffffffu, bit_or_none(off[cc + 1 + lane] - (g << 5)));
                    if (u < (uint32_t)nv) {
                        c[j] = cc + __popc(marks & le);
                        x[j] = __ldg(vo + vs[c[j]] + u);
                        y[j] = __ldg(vo + vs[c[j]] + u + 1);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < VU; ++j) {
                const uint32_t u = ((g0 + j) << 5) + lane;
                if (u < (uint32_t)nv) {
                    wrong |= y[j] < x[j] || y[j] > last[c[j]];
                    ovo[v_first + u] = x[j] + add[c[j]];
                }
            }
        }
    } else {  // long runs: a warp per run, the whole block for the very long ones
        constexpr long long WIDE = 1 << 13;
        for (int pass = 0; pass < 2; ++pass) {
            for (int i = pass ? 0 : warp; i < n0; i += pass ? 1 : CP_WARPS) {
                const long long c = ldp<OffT>(cp, q0 + i), l = ldp<OffT>(cp, q0 + i + 1) - c;
                if ((l >= WIDE) != (pass != 0)) continue;
                for (long long u = pass ? tid : lane; u < l; u += pass ? CP_THREADS : 32) {
                    const long long x = __ldg(vo + vs[i] + u), y = __ldg(vo + vs[i] + u + 1);
                    wrong |= y < x || y > last[i];
                    ovo[c + u] = x + add[i];
                }
            }
        }
    }
    if (wrong) flag(hdr, ST_BADINPUT);
}

template <typename OffT, typename SrcT>
static cudaError_t launch_var_t(const Mat &m, cudaStream_t st) {
    const long long ntiles = (m.p.C + (1LL << m.p.cshift) - 1) >> m.p.cshift;
    return launch_kernel(k_var_copy<OffT, SrcT>, false, ntiles < 1 ? 1 : ntiles, CP_THREADS, 0, st, m);
}

cudaError_t launch_var_copy(const Mat &m, cudaStream_t st) {
    if (m.p.o == 4)
        return m.p.wide ? launch_var_t<int32_t, unsigned long long>(m, st)
                        : launch_var_t<int32_t, uint32_t>(m, st);
    return m.p.wide ? launch_var_t<int64_t, unsigned long long>(m, st)
                    : launch_var_t<int64_t, uint32_t>(m, st);
}

}  // namespace mgt
