// Level 1 of the transpose, the scatter passes: two stable passes, like the
// digit passes of a radix sort, so that every pass writes runs of records
// instead of isolated ones.
//   K3a (cells -> super-buckets): one block per tile of `tile` cells, a few
//       thousand at a time.  Each warp builds the records of its piece in
//       shared memory; the block splits them by super-bucket (bucket >> p2,
//       <= 256) and writes runs at the super-bucket cursors.
//   K3b (super-bucket -> buckets): one block per (super-bucket, group of
//       tiles) item, the same split by the low p2 bits of the bucket, written
//       at the final bucket cursors.
// Cursors come from the tile-by-bucket offsets of K2, so input order is kept
// inside every bucket.  K3a also produces the P x P counts (source block from
// the cell index, destination block per super-bucket, or per cell where a
// super-bucket spans two destination blocks) when the planner leaves them to
// it; K3b the per-bucket value totals (K3a when there is a single pass).
//
// Both are bound by issue slots and the shared-memory pipe, not by DRAM (a
// record is 12 bytes in, 12 out), so they save instructions: no vote per digit
// bit, no second copy of a record, no search per thread for the rows.  K3a on
// the heterogeneous 8M x 8M matrix 2.77 -> 1.43 ms, balanced 4M x 4M (with
// P x P counts) 2.49 -> 1.31, 852K x 852K of 512 cells a row 7.68 -> 4.1;
// K3b 2.49 -> 1.40, 1.87 -> 1.02 and 6.66 -> 3.4 ms.
#include "mgt_internal.cuh"

#include <algorithm>
#include <climits>
#include <type_traits>

namespace mgt {

constexpr int SA_PSMEM = 256;                 // P up to which block tables live in shared memory
constexpr uint16_t SC_STRADDLE = 0xFFFFu;     // spans a destination block boundary

// The second-pass digit (low p2 bits of the bucket) rides in a record
// between the passes: above the column bits of meta for compact records
// (the planner keeps bshift + p2 <= 16 there, else it uses wide records
// between the passes), in bits 48.. of start for wide ones (V < 2^48).
__device__ __forceinline__ void put_d2(RecC &r, uint32_t d2, int bshift) { r.meta |= d2 << (16 + bshift); }
__device__ __forceinline__ void put_d2(RecW &r, uint32_t d2, int) {
    r.start |= (unsigned long long)d2 << 48;
}
__device__ __forceinline__ uint32_t take_d2(RecC &r, int bshift, int p2) {
    const uint32_t m = ((1u << p2) - 1u) << (16 + bshift);
    const uint32_t d = (r.meta & m) >> (16 + bshift);
    r.meta &= ~m;
    return d;
}
__device__ __forceinline__ uint32_t take_d2(RecW &r, int, int) {
    const uint32_t d = (uint32_t)(r.start >> 48);
    r.start &= (1ull << 48) - 1ull;
    return d;
}
__device__ __forceinline__ void rec_convert(const RecC &a, RecC &b) { b = a; }
__device__ __forceinline__ void rec_convert(const RecW &a, RecW &b) { b = a; }
__device__ __forceinline__ void rec_convert(const RecW &a, RecC &b) {
    b.i = a.i;
    b.meta = a.meta;
    b.start = (uint32_t)a.start;
}

// ------------------------------------------------- split of a tile of records
// Stable split, by a digit below nbins <= 256, of a tile of records that lies
// in shared memory in input order: each warp owns a contiguous piece, lane l
// its record 32 u + l in round u.
//   1. warp_rank: each record's rank among its warp's earlier ones of the
//      same digit, and the warp's counts;
//   2. ms_scan: positions in (digit, warp) order;
//   3. the index permutation inv[position] = record;
//   4. records in position order to their cursors: consecutive lanes write
//      the consecutive records of a run.
constexpr int MS_THREADS = 256;
constexpr int MS_WARPS = MS_THREADS / 32;
constexpr int MS_BLOCKS = 4;  // per SM
// Rounds of a warp per tile: 3,072 compact or 2,048 wide records leave room
// for four blocks per SM.  Measured in K3b on the balanced 4M x 4M matrix: 512
// threads x 8 rounds, two blocks 1.31 ms (its 16 warps wait at every
// barrier); 256 x 16, three blocks 0.98; 256 x 12, four 1.01; 256 x 8, four
// 1.08 (shorter runs).  1M x 1M, 512 cells a row, wide: 256 x 16 4.96 ms,
// 256 x 8 3.87.  Smaller matrices gain by the smaller tile (2M x 2M: 0.26 ms
// with 16 rounds, 0.23 with 12).
template <typename Rec>
__host__ __device__ constexpr int ms_rounds() { return sizeof(Rec) == 12 ? 12 : 8; }
template <typename Rec>
__host__ __device__ constexpr int ms_tile() { return MS_THREADS * ms_rounds<Rec>(); }

// Per-warp counters (u16) and mask words; the permutation lies over the mask
// words, which are all zero again when step 3 begins and are zeroed again
// after step 4.  PermT: uint16_t, or uint32_t to carry the digit along (digit
// << 16 | record), where the record does not hold it.
__host__ __device__ constexpr int ms_cstride(int nbins) { return nbins + 2; }
__host__ __device__ constexpr int ms_mstride(int nbins) { return nbins + 1; }
template <typename Rec, typename PermT>
__host__ __device__ constexpr size_t ms_mask_bytes(int nbins) {
    const size_t a = (size_t)ms_mstride(nbins) * MS_WARPS * 4, b = (size_t)ms_tile<Rec>() * sizeof(PermT);
    return a > b ? a : b;
}
__host__ __device__ constexpr size_t ms_cnt_bytes(int nbins) { return (size_t)ms_cstride(nbins) * MS_WARPS * 2; }

// sums[d] += x for every lane's digit: one add per lane; the lanes of a large
// group (a hot column's bucket), which would take turns on one word, add up
// first.  group: the lane's word from warp_rank.
__device__ __forceinline__ void warp_add(uint32_t *sums, uint32_t d, uint32_t x, uint32_t group) {
    const unsigned hot = __ballot_sync(0xffffffffu, __popc(group) >= 8);
    if (hot) {
        const uint32_t dh = __shfl_sync(0xffffffffu, d, __ffs(hot) - 1);
        const uint32_t sum = __reduce_add_sync(0xffffffffu, group && d == dh ? x : 0u);
        if (lane_id() == 0) atomicAdd(&sums[dh], sum);
        if (d == dh) x = 0;
    }
    if (x) atomicAdd(&sums[d], x);
}

// Turns the per-(digit, warp) counts into positions in (digit, warp) order,
// which keeps equal digits in input order, and calls fn(digit, first
// position, count) once per digit.  scratch: >= 8 words.  Every warp's counts
// must be visible; ends with a barrier.
template <typename Fn>
__device__ __forceinline__ void ms_scan(uint16_t *wcnt, int nbins, uint32_t *scratch, Fn fn) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t c[MS_WARPS], tot = 0;
#pragma unroll
    for (int w = 0; w < MS_WARPS; ++w) {
        c[w] = tid < nbins ? wcnt[w * ms_cstride(nbins) + tid] : 0u;
        tot += c[w];
    }
    const uint32_t inc = warp_sum_scan(tot);
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    if (tid < nbins) {
        uint32_t run = inc - tot;
#pragma unroll
        for (int w = 0; w < MS_WARPS; ++w) run += w < warp ? scratch[w] : 0u;
        fn(tid, run, tot);
#pragma unroll
        for (int w = 0; w < MS_WARPS; ++w) {
            wcnt[w * ms_cstride(nbins) + tid] = (uint16_t)run;
            run += c[w];
        }
    }
    __syncthreads();
}

// Steps 2 to 4 for the tile's n records (FULL: n = the tile's size): rk[u] =
// digit << 16 | rank of the lane's record of round u.  put(p, e): the record of
// permutation entry e to its place, position p; PAD: record x lies at x + x /
// 32, and that is what the entry names.  Leaves the counters and mask words zero for this
// warp's next tile; starts and ends with a barrier.
template <bool FULL, bool PAD, typename PermT, int ROUNDS, typename ScanFn, typename PutFn>
__device__ __forceinline__ void ms_place(const uint32_t (&rk)[ROUNDS], int n, int nbins, uint16_t *wcnt,
                                         uint32_t *wmsk, uint32_t *scratch, ScanFn on_digit, PutFn put) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint16_t *mycnt = wcnt + warp * ms_cstride(nbins);
    PermT *inv = reinterpret_cast<PermT *>(wmsk);
    __syncthreads();
    ms_scan(wcnt, nbins, scratch, on_digit);
#pragma unroll
    for (int u = 0; u < ROUNDS; ++u) {
        const int x = (warp * ROUNDS + u) * 32 + lane;
        if (FULL || x < n) {
            const uint32_t p = mycnt[rk[u] >> 16] + (rk[u] & 0xFFFFu);
            const uint32_t e = (uint32_t)(PAD ? x + warp * ROUNDS + u : x);
            inv[p] = (PermT)(sizeof(PermT) == 4 ? (rk[u] & 0xFFFF0000u) | e : e);
        }
    }
    __syncwarp();
    for (int d = lane; d < nbins; d += 32) mycnt[d] = 0;
    __syncthreads();
    if (FULL) {
#pragma unroll 4
        for (int u = 0; u < ROUNDS; ++u) put(u * MS_THREADS + tid, (uint32_t)inv[u * MS_THREADS + tid]);
    } else {
        for (int p = tid; p < n; p += MS_THREADS) put(p, (uint32_t)inv[p]);
    }
    __syncthreads();
    uint32_t *mymsk = wmsk + warp * ms_mstride(nbins);
    for (int d = lane; d < nbins; d += 32) mymsk[d] = 0;
    __syncwarp();
}

// Blocks per SM that the shared memory allows (228 KB, 1 KB a block reserved,
// room for the static arrays).
static int ms_blocks(size_t smem) {
    const int fit = (int)((size_t)228 * 1024 / (smem + 2304));
    return fit < 1 ? 1 : (fit < MS_BLOCKS ? fit : MS_BLOCKS);
}

// ---------------------------------------------------------------- K3a scatter
struct SaLayout {
    size_t in, msk, cnt, cur, delta, tcnt, tvs, tvs32, sblk, slo, shi, sspl, pcs, pos, ppt, ppc, ppc32, scratch,
        misc, total;
};
// vals: value totals per super-bucket are counted; P: row blocks whose tables
// lie in shared memory (0 without P x P counting)
template <typename Rec>
__host__ __device__ inline SaLayout sa_layout(int nbins, bool vals, int P) {
    SaLayout L;
    size_t o = 0;
    const int Ps = P <= SA_PSMEM ? P : 0, nb = P > 0 ? nbins : 0, nv = vals ? nbins : 0;
#define MGT_TAKE(field, bytes) L.field = o; o = (o + (size_t)(bytes) + 15) & ~size_t(15);
    MGT_TAKE(in, (size_t)(ms_tile<Rec>() / 32 * 33) * sizeof(Rec))  // one record of padding per 32
    MGT_TAKE(msk, (ms_mask_bytes<Rec, uint32_t>(nbins)))
    MGT_TAKE(cnt, ms_cnt_bytes(nbins))
    MGT_TAKE(cur, (size_t)nbins * 4)
    MGT_TAKE(delta, (size_t)nbins * 4)
    MGT_TAKE(tcnt, (size_t)nb * 4)
    MGT_TAKE(tvs, (size_t)nv * 8)
    MGT_TAKE(tvs32, (size_t)nv * 4)
    MGT_TAKE(sblk, (size_t)nb * 2)
    MGT_TAKE(slo, (size_t)nb * 2)
    MGT_TAKE(shi, (size_t)nb * 2)
    MGT_TAKE(sspl, (size_t)nb * 4)
    MGT_TAKE(pcs, (size_t)(Ps + 1) * 8)
    MGT_TAKE(pos, (size_t)(Ps + 1) * 8)
    MGT_TAKE(ppt, (size_t)2 * Ps * 8)
    MGT_TAKE(ppc, (size_t)4 * Ps * 8)
    MGT_TAKE(ppc32, (size_t)4 * Ps * 4)
    MGT_TAKE(scratch, 48 * 4)
    MGT_TAKE(misc, 32)
#undef MGT_TAKE
    L.total = o;
    return L;
}

// MODE 0: no P x P counting (the counts come from the output pass, or none are
// asked for).  MODE 1: every super-bucket lies in one destination block: the
// cells are taken source block by source block, and a super-bucket's count and
// value total go to its block (nothing per cell but the value total).  MODE 2:
// row blocks cut super-buckets and are too many for the output pass: a
// destination search per cell where needed (more registers, three blocks).
template <typename OffT, typename Rec, bool BATCH, int MODE>
__global__ void __launch_bounds__(MS_THREADS, MODE == 2 ? 3 : MS_BLOCKS)
    k_scatter(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int ROUNDS = ms_rounds<Rec>(), TILE = ms_tile<Rec>(), SEG = ROUNDS * 32;
    constexpr bool PP = MODE != 0;
    pipeline_wait<BATCH>();
    const VBlock vb = vblock<BATCH>(m0, ba);
    const Mat &M = *vb.m;
    DevHeader *hdr = M.ws.hdr;
    // malformed row pointers or columns: nothing is placed (the row table could be anything).  One
    // decision for the block: other blocks of this launch set the bit too, when cell_ptr decreases
    if (__syncthreads_or((hdr->status & ST_BADINPUT) != 0)) return;
    const void *__restrict__ row_ptr = M.in.row_ptr;
    const int32_t *__restrict__ col = M.in.col;
    const void *__restrict__ cell_ptr = M.in.cell_ptr;
    const long long R = M.p.R, N = M.p.N, C = M.p.C;
    const int bshift = M.p.bshift, B = (int)M.p.B, p2 = M.p.p2, tile = M.p.tile;
    const int P = M.p.P;
    const uint32_t *__restrict__ cnt = M.ws.cnt;
    const unsigned long long *__restrict__ bucket_base = M.ws.bucket_base;
    unsigned long long *bucket_vtot = M.ws.bucket_vtot;
    Rec *__restrict__ out = reinterpret_cast<Rec *>(p2 > 0 ? M.ws.recs1 : M.ws.recs);
    const long long *__restrict__ pcoff = M.ws.pcoff;
    const long long *__restrict__ poff = M.ws.poff;
    const uint16_t *__restrict__ dblock = M.ws.dblock;
    const uint32_t *__restrict__ rowat = row_table(M.ws);
    long long *part_cells = M.out.part_cells, *part_values = M.out.part_values;
    const int nbins = (B + (1 << p2) - 1) >> p2;
    const bool want_pp = PP && (part_cells != nullptr) && P > 1 && !M.p.pp_out;
    const bool pp_smem = want_pp && P <= SA_PSMEM;
    const bool vals = PP || p2 == 0;
    const SaLayout L = sa_layout<Rec>(nbins, vals, PP ? P : 0);
    Rec *IN = reinterpret_cast<Rec *>(smem + L.in);
    uint32_t *wmsk = reinterpret_cast<uint32_t *>(smem + L.msk);
    uint16_t *wcnt = reinterpret_cast<uint16_t *>(smem + L.cnt);
    uint32_t *cur = reinterpret_cast<uint32_t *>(smem + L.cur);      // next record of each super-bucket
    uint32_t *delta = reinterpret_cast<uint32_t *>(smem + L.delta);  // record minus position in the tile
    uint32_t *tcnt = reinterpret_cast<uint32_t *>(smem + L.tcnt);
    unsigned long long *tvs = reinterpret_cast<unsigned long long *>(smem + L.tvs);
    uint32_t *tvs32 = reinterpret_cast<uint32_t *>(smem + L.tvs32);  // per sub-chunk
    uint16_t *sblk = reinterpret_cast<uint16_t *>(smem + L.sblk);  // destination block of a super-bucket (or STRADDLE)
    uint16_t *slo = reinterpret_cast<uint16_t *>(smem + L.slo);    // block of its first column
    uint16_t *shi = reinterpret_cast<uint16_t *>(smem + L.shi);    // block of its last column
    int32_t *sspl = reinterpret_cast<int32_t *>(smem + L.sspl);    // first column of block shi when it spans two
    long long *pcs = reinterpret_cast<long long *>(smem + L.pcs);
    long long *pos_ = reinterpret_cast<long long *>(smem + L.pos);
    unsigned long long *ppt = reinterpret_cast<unsigned long long *>(smem + L.ppt);  // [2][P]
    unsigned long long *ppc = reinterpret_cast<unsigned long long *>(smem + L.ppc);  // [2 blocks][2][P]
    uint32_t *ppc32 = reinterpret_cast<uint32_t *>(smem + L.ppc32);  // the same, per sub-chunk
    uint32_t *scratch = reinterpret_cast<uint32_t *>(smem + L.scratch);
    long long *sh = reinterpret_cast<long long *>(smem + L.misc);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned le = lanemask_lt() | (1u << lane);
    uint16_t *mycnt = wcnt + warp * ms_cstride(nbins);
    uint32_t *mymsk = wmsk + warp * ms_mstride(nbins);
    const long long t = vb.b;
    const long long kt0 = t * (long long)tile, kt1 = min(C, kt0 + tile);
    const long long *pc_tab = pp_smem ? pcs : pcoff;
    const long long *po_tab = pp_smem ? pos_ : poff;
    for (int i = tid; i < ms_cstride(nbins) * MS_WARPS; i += MS_THREADS) wcnt[i] = 0;
    for (int i = tid; i < ms_mstride(nbins) * MS_WARPS; i += MS_THREADS) wmsk[i] = 0;
    if (vals)
        for (int d = tid; d < nbins; d += MS_THREADS) { tvs[d] = 0; tvs32[d] = 0; }
    if (PP)
        for (int d = tid; d < nbins; d += MS_THREADS) tcnt[d] = 0;
    if (pp_smem) {
        for (int i = tid; i <= P; i += MS_THREADS) { pcs[i] = pcoff[i]; pos_[i] = poff[i]; }
        for (int i = tid; i < 2 * P; i += MS_THREADS) ppt[i] = 0;
        for (int i = tid; i < 4 * P; i += MS_THREADS) { ppc[i] = 0; ppc32[i] = 0; }
    }
    // cursors: super-bucket base + this tile's offsets inside its 2^p2
    // consecutive buckets; a warp per super-bucket, or a thread where they are few
    {
        const uint32_t *row = cnt + t * (long long)B;
        if (p2 >= 3) {
#pragma unroll 4
            for (int d = warp; d < nbins; d += MS_WARPS) {
                const int b0 = d << p2, b1 = min(B, b0 + (1 << p2));
                uint32_t v = 0;
                for (int b = b0 + lane; b < b1; b += 32) v += row[b];
                v = __reduce_add_sync(0xffffffffu, v);
                if (lane == 0) cur[d] = (uint32_t)bucket_base[b0] + v;
            }
        } else {
            for (int d = tid; d < nbins; d += MS_THREADS) {
                const int b0 = d << p2, b1 = min(B, b0 + (1 << p2));
                uint32_t v = (uint32_t)bucket_base[b0];
                for (int b = b0; b < b1; ++b) v += row[b];
                cur[d] = v;
            }
        }
    }
    if (PP && tid == 0) {
        const long long a = upper_bound_ll(pcoff, 0, P + 1, kt0) - 1, z = upper_bound_ll(pcoff, 0, P + 1, kt1 - 1) - 1;
        sh[0] = a < 0 ? 0 : a;
        sh[1] = z < 0 ? 0 : z;
    }
    __syncthreads();
    if (want_pp) {
        for (int d = tid; d < nbins; d += MS_THREADS) {
            // destination blocks of the super-bucket's first and last columns
            const long long c0 = (long long)d << (p2 + bshift);
            const long long c1 = min(N, ((long long)(d + 1)) << (p2 + bshift)) - 1;
            long long lo = (pp_smem ? upper_bound_sm(pos_, 0, P + 1, c0) : upper_bound_ll(poff, 0, P + 1, c0)) - 1;
            long long hi = (pp_smem ? upper_bound_sm(pos_, 0, P + 1, c1) : upper_bound_ll(poff, 0, P + 1, c1)) - 1;
            lo = lo < 0 ? 0 : (lo >= P ? P - 1 : lo);
            hi = hi < lo ? lo : (hi >= P ? P - 1 : hi);
            sblk[d] = lo == hi ? (uint16_t)lo : SC_STRADDLE;
            // spanning exactly two blocks: the split column decides per cell
            slo[d] = (uint16_t)lo;
            shi[d] = (uint16_t)hi;
            sspl[d] = hi == lo + 1 ? (int32_t)min(pp_smem ? pos_[hi] : poff[hi], (long long)INT_MAX) : -1;
        }
        __syncthreads();
    }
    long long s_first = PP ? sh[0] : 0;  // source block of the (first) cell
    const bool one_src = MODE != 2 || sh[1] == s_first;
    long long sp = s_first;  // MODE 2: source block of this lane's last cell (they ascend)
    const uint32_t mask2 = (1u << p2) - 1u;
    const uint32_t colmask = (1u << (bshift + (sizeof(Rec) == 12 ? p2 : 0))) - 1u;
    bool bad = false;
    for (long long s0 = kt0; s0 < kt1;) {
        long long s1 = min(kt1, s0 + TILE);
        if (MODE == 1 && want_pp) {  // up to the end of the source block
            while (s_first < P - 1 && pc_tab[s_first + 1] <= s0) ++s_first;
            if (s_first < P - 1) s1 = min(s1, pc_tab[s_first + 1]);
        }
        const int n = (int)(s1 - s0);
        // FULL: every lane of every round has a cell
        auto split = [&](auto full) {
            constexpr bool FULL = decltype(full)::value;
            constexpr int HALF = 4;  // rounds whose loads are in flight together
            // rows per cell of a warp's piece from which its cells' rows are searched for: a walk reads 32
            // rows in 0.14 us, the searches of a piece take some 0.1 ms (30M rows, 3,000 cells: 42 to
            // 156 ms a transpose by walks alone, 0.24 to 0.38 with searches)
            constexpr long long SPARSE = 64;
            const long long kw = s0 + warp * SEG;                // the warp's first cell
            const int nw = FULL ? SEG : min(SEG, n - warp * SEG);  // and its cells (none: <= 0)
            // padded: cells of one super-bucket often lie a multiple of 32 apart (rows of
            // 32 sorted cells), and would all be read back from the same banks
            Rec *W = IN + warp * ROUNDS * 33;
            uint32_t rk[ROUNDS];
            int cv[HALF];
            long long st[HALF], en[HALF];
            // columns and run bounds of HALF rounds
            auto load_half = [&](int h) {
#pragma unroll
                for (int j = 0; j < HALF; ++j) {
                    const int y = (h * HALF + j) * 32 + lane;
                    cv[j] = 0;
                    st[j] = en[j] = 0;
                    if (FULL || y < nw) {
                        cv[j] = __ldcs(col + kw + y);
                        st[j] = ldo<OffT>(cell_ptr, kw + y);
                        en[j] = ldo<OffT>(cell_ptr, kw + y + 1);
                    }
                }
            };
            load_half(0);
            // rows: r0 holds the first cell; each later row that starts inside
            // the piece and is not empty leaves its index + 1 in the record
            // of its first cell
            uint32_t row = 0;
            if (FULL || nw > 0) {
                const long long g = kw >> ROWAT_SHIFT, ge = (min(kw + nw, C) + (1 << ROWAT_SHIFT) - 1) >> ROWAT_SHIFT;
                const long long r0 = rowat[g], r1 = rowat[ge];
                row = (uint32_t)r0;
#pragma unroll
                for (int u = 0; u < ROUNDS; ++u) W[u * 33 + lane].i = 0;
                __syncwarp();
                long long r = r0 + 1 + lane;
                if (r1 - r0 > SPARSE * SEG) {  // a search per cell: its row + 1 is its own mark
#pragma unroll 1
                    for (int y = lane; y < nw; y += 32)
                        W[y + (y >> 5)].i = (uint32_t)upper_bound_g<OffT>(row_ptr, r0, r1 + 1, kw + y);
                    r = r1 + 1;
                }
                for (; r <= r1; r += 32) {
                    const long long a = ldo<OffT>(row_ptr, r) - kw, e = ldo<OffT>(row_ptr, r + 1) - kw;
                    if (a < e && a > 0 && a < SEG) W[a + (a >> 5)].i = (uint32_t)r + 1;
                    if (MODE == 1 && a < e && a <= 0) row = (uint32_t)r;  // (a piece need not start on the table's cells)
                }
                if (MODE == 1) row = __reduce_max_sync(0xffffffffu, row);
                __syncwarp();
            }
#pragma unroll
            for (int h = 0; h < ROUNDS / HALF; ++h) {
                if (h) load_half(h);
#pragma unroll
                for (int j = 0; j < HALF; ++j) {
                    const int u = h * HALF + j, y = u * 32 + lane;
                    const bool v = FULL || y < nw;
                    // the last mark at or below this lane, else the row so far
                    uint32_t mark = 0;
                    if (FULL || nw > 0) mark = W[u * 33 + lane].i;
                    const unsigned marks = __ballot_sync(0xffffffffu, mark != 0) & le;
                    const uint32_t got = __shfl_sync(0xffffffffu, mark, marks ? 31 - __clz(marks) : 0);
                    const uint32_t irow = marks ? got - 1 : row;
                    row = __shfl_sync(0xffffffffu, irow, 31);
                    uint32_t d = 0, len16 = 0;
                    if (v) {
                        int c = cv[j];
                        if ((unsigned)c >= (unsigned)N) { bad = true; c = c < 0 ? 0 : (int)(N - 1); }
                        // (start and end lie in [0, V]: the end points are checked, and so is every step)
                        long long len = en[j] - st[j];
                        if (len < 0) { bad = true; len = 0; }
                        const bool esc = len >= (long long)LEN_ESC;
                        len16 = esc ? LEN_ESC : (uint32_t)len;
                        const uint32_t b = (uint32_t)c >> bshift;
                        d = b >> p2;
                        Rec r;
                        r.i = irow;
                        r.start = (decltype(r.start))st[j];
                        r.meta = (((uint32_t)c & colmask) << 16) | len16;
                        if (sizeof(Rec) != 12 && p2 > 0) put_d2(r, b & mask2, bshift);
                        W[u * 33 + lane] = r;
                        if (p2 == 0 && esc) atomicAdd(&bucket_vtot[b], (unsigned long long)len);
                        if (MODE == 1 && want_pp && esc)
                            atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[s_first * P + sblk[d]]),
                                      (unsigned long long)len);
                        if (MODE == 2 && want_pp && (!one_src || esc || sblk[d] == SC_STRADDLE)) {
                            if (!one_src) while (sp < P - 1 && pc_tab[sp + 1] <= kw + y) ++sp;
                            // destination block of the column: the super-bucket's, the
                            // side of its split column, else the bucket's or a search
                            long long dd;
                            const uint16_t lo = slo[d], hi = shi[d];
                            if (lo == hi) {
                                dd = lo;
                            } else if (hi == lo + 1) {
                                dd = c < sspl[d] ? lo : hi;
                            } else {
                                const uint16_t db = dblock[b];
                                dd = db != SC_STRADDLE ? (long long)db
                                                       : (pp_smem ? upper_bound_sm(po_tab, 0, P + 1, c)
                                                                  : upper_bound_ll(po_tab, 0, P + 1, c)) - 1;
                            }
                            if (dd < 0) dd = 0;
                            if (dd >= P) dd = P - 1;
                            const bool by_tile = one_src && sblk[d] != SC_STRADDLE;
                            if (pp_smem && sp - s_first < 2 && !esc) {
                                // 32-bit counters per sub-chunk (< 2^16 cells x < 2^16 values),
                                // added to the tile's 64-bit ones after each sub-chunk
                                const int rowp = (int)(sp - s_first);
                                atomicAdd(&ppc32[(rowp * 2 + 0) * P + dd], 1u);
                                atomicAdd(&ppc32[(rowp * 2 + 1) * P + dd], len16);
                            } else {
                                if (!by_tile)
                                    atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[sp * P + dd]), 1ull);
                                if (!by_tile || esc)
                                    atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[sp * P + dd]),
                                              (unsigned long long)len);
                            }
                        }
                        if (esc) len16 = 0;
                    }
                    uint32_t group;
                    rk[u] = (d << 16) | warp_rank<FULL>(mycnt, mymsk, d, v, group);
                    // value totals per super-bucket: the tile's P x P values, or
                    // the bucket totals of a single pass
                    if (vals) warp_add(tvs32, d, len16, group);
                }
            }
            ms_place<FULL, true, uint32_t>(
                rk, n, nbins, wcnt, wmsk, scratch,
                [&](int d, uint32_t start, uint32_t tot) {
                    delta[d] = cur[d] - start;
                    cur[d] += tot;
                    if (PP) tcnt[d] += tot;
                    if (vals) {
                        tvs[d] += tvs32[d];
                        tvs32[d] = 0;
                    }
                },
                [&](int p, uint32_t e) {
                    const uint32_t q = delta[e >> 16] + (uint32_t)p;
                    if (MGT_IN(hdr, q, C)) out[q] = IN[e & 0xFFFFu];
                });
        };
        if (n == TILE) split(std::true_type());
        else split(std::false_type());
        if (MODE == 2 && pp_smem) {
            for (int i = tid; i < 4 * P; i += MS_THREADS) {
                if (ppc32[i]) {
                    ppc[i] += ppc32[i];
                    ppc32[i] = 0;
                }
            }
            __syncthreads();  // (the next sub-chunk's cells add to ppc32 before any other barrier)
        }
        if (MODE == 1 && want_pp && (s1 == kt1 || (s_first < P - 1 && pc_tab[s_first + 1] <= s1))) {
            // the source block's (or the tile's) last cells: its totals by destination block
            for (int d = tid; d < nbins; d += MS_THREADS) {
                if (tcnt[d]) {
                    if (pp_smem) {
                        atomicAdd(&ppt[sblk[d]], (unsigned long long)tcnt[d]);
                        atomicAdd(&ppt[P + sblk[d]], tvs[d]);
                    } else {
                        atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[s_first * P + sblk[d]]),
                                  (unsigned long long)tcnt[d]);
                        atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[s_first * P + sblk[d]]), tvs[d]);
                    }
                }
                if (p2 == 0 && tvs[d]) atomicAdd(&bucket_vtot[d], tvs[d]);
                tcnt[d] = 0;
                tvs[d] = 0;
            }
            if (pp_smem) {
                __syncthreads();
                for (int dd = tid; dd < P; dd += MS_THREADS) {
                    if (ppt[dd]) {
                        atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[s_first * P + dd]), ppt[dd]);
                        atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[s_first * P + dd]), ppt[P + dd]);
                    }
                    ppt[dd] = ppt[P + dd] = 0;
                }
                __syncthreads();
            }
        }
        s0 = s1;
    }
    __syncthreads();
    // tile totals: bucket value totals (single pass) and P x P by super-bucket
    for (int d = tid; d < nbins; d += MS_THREADS) {
        if (vals && p2 == 0 && tvs[d]) atomicAdd(&bucket_vtot[d], tvs[d]);
        if (MODE == 2 && want_pp && one_src && sblk[d] != SC_STRADDLE && tcnt[d]) {
            if (pp_smem) {
                atomicAdd(&ppt[sblk[d]], (unsigned long long)tcnt[d]);
                atomicAdd(&ppt[P + sblk[d]], tvs[d]);
            } else {
                atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[s_first * P + sblk[d]]),
                          (unsigned long long)tcnt[d]);
                atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[s_first * P + sblk[d]]), tvs[d]);
            }
        }
    }
    __syncthreads();
    if (MODE == 2 && pp_smem) {
        for (int dd = tid; dd < P; dd += MS_THREADS) {
            if (ppt[dd]) {
                atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[s_first * P + dd]), ppt[dd]);
                atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[s_first * P + dd]), ppt[P + dd]);
            }
            for (int rowp = 0; rowp < 2; ++rowp) {
                const long long sp = s_first + rowp;
                const unsigned long long cc = ppc[(rowp * 2 + 0) * P + dd], vv = ppc[(rowp * 2 + 1) * P + dd];
                if (sp < P && (cc || vv)) {
                    atomicAdd(reinterpret_cast<unsigned long long *>(&part_cells[sp * P + dd]), cc);
                    atomicAdd(reinterpret_cast<unsigned long long *>(&part_values[sp * P + dd]), vv);
                }
            }
        }
    }
    if (__syncthreads_or(bad) && tid == 0) flag(hdr, ST_BADINPUT);
}

// ---------------------------------------------------------------- K3b scatter2
// One item = (super-bucket S, tile group).  Its records are the contiguous
// K3a output for tiles [t0, t1) of S; they go to S's buckets at cursors
// bucket base + tile t0's offset inside the bucket.
struct Sb2Layout {
    size_t in, msk, cnt, cur, delta, vs, vs32, scratch, misc, total;
};
template <typename Rec1>
__host__ __device__ inline Sb2Layout sb2_layout(int nbins) {
    Sb2Layout L;
    size_t o = 0;
#define MGT_TAKE(field, bytes) L.field = o; o = (o + (size_t)(bytes) + 15) & ~size_t(15);
    MGT_TAKE(in, (size_t)ms_tile<Rec1>() * sizeof(Rec1) + 16)
    MGT_TAKE(msk, (ms_mask_bytes<Rec1, uint16_t>(nbins)))
    MGT_TAKE(cnt, ms_cnt_bytes(nbins))
    MGT_TAKE(cur, (size_t)nbins * 4)
    MGT_TAKE(delta, (size_t)nbins * 4)
    MGT_TAKE(vs, (size_t)nbins * 8)
    MGT_TAKE(vs32, (size_t)nbins * 4)
    MGT_TAKE(scratch, 48 * 4)
    MGT_TAKE(misc, 32)
#undef MGT_TAKE
    L.total = o;
    return L;
}

// Second-pass items of one matrix: each super-bucket's tiles in groups of
// about p.item2 records, by the super-bucket's own size (a Zipf column's
// super-bucket may hold a tenth of all cells: groups of equal tile counts left
// one block with 25 times the mean: 3.7 instead of 1.8 ms on the heterogeneous
// matrix).
__device__ __forceinline__ long long group_tiles(unsigned long long tot, long long T, long long want) {
    const unsigned long long g = tot > 0 ? (unsigned long long)(want * T) / tot : (unsigned long long)T;
    return g < 1 ? 1 : (g > (unsigned long long)T ? T : (long long)g);
}
// Host bound on their number: floor(x) >= x / 2 for x >= 1, one partial group each.
__host__ __device__ inline long long scatter2_items(const Params &p) {
    if (p.T == 0 || p.p2 == 0) return 0;
    return 2 * (p.C / p.item2) + 2 * ((p.B + (1LL << p.p2) - 1) >> p.p2);
}

template <typename OffT, typename Rec1, typename Rec, bool BATCH>
__global__ void __launch_bounds__(MS_THREADS, MS_BLOCKS)
    k_scatter2(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int ROUNDS = ms_rounds<Rec1>(), TILE = ms_tile<Rec1>();
    pipeline_wait<BATCH>();
    __shared__ uint32_t first[257];  // first item of each super-bucket
    __shared__ uint32_t wsum[MS_WARPS];
    const Mat *known = nullptr;      // the matrix of that table
    // items (super-bucket, tile group), dealt round-robin to the blocks
    Units<BATCH> U(m0, ba, blockIdx.x, gridDim.x);
    while (U.next([](const Mat &X) { return scatter2_items(X.p); })) {
    const Mat &M = *U.M;
    if (M.ws.hdr->status & ST_BADINPUT) {  // K3a may have left records unwritten
        if (!BATCH) return;
        continue;
    }
    const Rec1 *__restrict__ in = reinterpret_cast<const Rec1 *>(M.ws.recs1);
    Rec *__restrict__ out = reinterpret_cast<Rec *>(M.ws.recs);
    const long long C = M.p.C, V = M.p.V, T = M.p.T;
    const int bshift = M.p.bshift, B = (int)M.p.B, p2 = M.p.p2;
    const uint32_t *__restrict__ cnt = M.ws.cnt;
    const unsigned long long *__restrict__ bucket_base = M.ws.bucket_base;
    const unsigned long long *__restrict__ bucket_tot = M.ws.bucket_tot;
    unsigned long long *bucket_vtot = M.ws.bucket_vtot;
    const void *cell_ptr = M.in.cell_ptr;
    DevHeader *hdr = M.ws.hdr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nbins = 1 << p2;
    const Sb2Layout SL = sb2_layout<Rec1>(nbins);
    uint16_t *wcnt = reinterpret_cast<uint16_t *>(smem + SL.cnt);
    uint32_t *wmsk = reinterpret_cast<uint32_t *>(smem + SL.msk);
    uint16_t *mycnt = wcnt + warp * ms_cstride(nbins);
    uint32_t *mymsk = wmsk + warp * ms_mstride(nbins);
    uint32_t *cur = reinterpret_cast<uint32_t *>(smem + SL.cur);
    uint32_t *delta = reinterpret_cast<uint32_t *>(smem + SL.delta);
    unsigned long long *vs = reinterpret_cast<unsigned long long *>(smem + SL.vs);
    uint32_t *vs32 = reinterpret_cast<uint32_t *>(smem + SL.vs32);  // per sub-chunk
    uint32_t *scratch = reinterpret_cast<uint32_t *>(smem + SL.scratch);
    unsigned long long *lohi = reinterpret_cast<unsigned long long *>(smem + SL.misc);
    (void)hdr;
    const int nS = (B + nbins - 1) >> p2;
    auto group_of = [&](int S) {
        const unsigned long long end = S + 1 < nS ? bucket_base[(S + 1) << p2] : (unsigned long long)C;
        return group_tiles(end - bucket_base[S << p2], T, M.p.item2);
    };
    if (known != &M) {
        uint32_t groups = 0;
        if (tid < nS) {
            const long long G = group_of(tid);
            groups = (uint32_t)((T + G - 1) / G);
        }
        const uint32_t inc = warp_inclusive_scan(groups);
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        if (tid < nS) first[tid + 1] = before + inc;
        if (tid == 0) first[0] = 0;
        __syncthreads();
        known = &M;
    }
    if (U.j >= first[nS]) continue;
    {
        int S = 0, Se = nS;  // first[S] <= item < first[Se]
        while (Se - S > 1) {
            const int mid = (S + Se) >> 1;
            if (first[mid] <= U.j) S = mid;
            else Se = mid;
        }
        const long long G = group_of(S);
        const long long t0 = ((long long)U.j - first[S]) * G, t1 = min(T, t0 + G);
        // record range of this item inside K3a's output for S
        if (tid < 64) {
            // warp 0: offset of tile t0 inside S; warp 1: of tile t1 (S's total at T)
            const long long tt = tid < 32 ? t0 : t1;
            uint32_t off = 0;
            for (int d = tid & 31; d < nbins; d += 32) {
                const int b = (S << p2) + d;
                if (b < B) off += tt < T ? cnt[tt * B + b] : (uint32_t)bucket_tot[b];
            }
            off = __reduce_add_sync(0xffffffffu, off);
            if ((tid & 31) == 0) lohi[tid >> 5] = bucket_base[S << p2] + off;
        }
        for (int d = tid; d < nbins; d += MS_THREADS) {
            const int b = (S << p2) + d;
            cur[d] = b < B ? (uint32_t)(bucket_base[b] + cnt[t0 * B + b]) : 0u;
            vs[d] = 0;
            vs32[d] = 0;
        }
        // the ranks' counters and masks start at zero (the layout depends on
        // p2, which may change between the matrices of a batch)
        for (int i = tid; i < ms_cstride(nbins) * MS_WARPS; i += MS_THREADS) wcnt[i] = 0;
        for (int i = tid; i < ms_mstride(nbins) * MS_WARPS; i += MS_THREADS) wmsk[i] = 0;
        __syncthreads();
        const unsigned long long lo = lohi[0], hi = lohi[1];
        for (unsigned long long s0 = lo; s0 < hi; s0 += TILE) {
            const int n = (int)min((unsigned long long)TILE, hi - s0);
            const Rec1 *IN = start_tile<MS_THREADS>(smem + SL.in, in + s0, n);
            wait_tile();
            __syncthreads();
            // FULL: every lane of every round has a record
            auto split = [&](auto full) {
                constexpr bool FULL = decltype(full)::value;
                // ranks among equal digits; value totals
                uint32_t rk[ROUNDS];
#pragma unroll
                for (int u = 0; u < ROUNDS; ++u) {
                    const int x = (warp * ROUNDS + u) * 32 + lane;
                    const bool v = FULL || x < n;
                    uint32_t d = 0, len = 0;
                    if (v) {
                        Rec1 r1 = IN[x];
                        d = take_d2(r1, bshift, p2);
                        len = r1.meta & 0xFFFFu;
                        if (len == LEN_ESC) {
                            len = 0;
                            if ((S << p2) + (int)d < B)
                                atomicAdd(&bucket_vtot[(S << p2) + d],
                                          rec_len<OffT>(r1.meta, r1.start, cell_ptr, C, V));
                        }
                    }
                    uint32_t group;
                    rk[u] = (d << 16) | warp_rank<FULL>(mycnt, mymsk, d, v, group);
                    warp_add(vs32, d, len, group);
                }
                ms_place<FULL, false, uint16_t>(
                    rk, n, nbins, wcnt, wmsk, scratch,
                    [&](int d, uint32_t start, uint32_t tot) {
                        delta[d] = cur[d] - start;
                        cur[d] += tot;
                        vs[d] += vs32[d];
                        vs32[d] = 0;
                    },
                    [&](int p, uint32_t x) {
                        Rec1 r1 = IN[x];
                        const uint32_t d = take_d2(r1, bshift, p2);
                        Rec r;
                        rec_convert(r1, r);
                        const uint32_t q = delta[d] + (uint32_t)p;
                        if (MGT_IN(hdr, q, C)) out[q] = r;
                    });
            };
            if (n == TILE) split(std::true_type());
            else split(std::false_type());
        }
        for (int d = tid; d < nbins; d += MS_THREADS) {
            const int b = (S << p2) + d;
            if (b < B && vs[d]) atomicAdd(&bucket_vtot[b], vs[d]);
        }
        __syncthreads();
    }
    }
}

// Shared memory of the scatter pass; pp: with the P x P counter tables.
static size_t smem_scatter_pp(const Params &p, bool pp) {
    const int nbins = (int)((p.B + (1LL << p.p2) - 1) >> p.p2);
    const int P = pp ? p.P : 0;
    const bool vals = pp || p.p2 == 0;
    return p.wide || p.wide_mid ? sa_layout<RecW>(nbins, vals, P).total : sa_layout<RecC>(nbins, vals, P).total;
}
static size_t smem_scatter(const Params &p) { return smem_scatter_pp(p, true); }
static size_t smem_scatter2(const Params &p) {
    return p.wide || p.wide_mid ? sb2_layout<RecW>(1 << p.p2).total : sb2_layout<RecC>(1 << p.p2).total;
}
size_t scatter_smem_bytes(const Params &p) {
    const size_t a = smem_scatter(p), b = smem_scatter2(p);
    return a > b ? a : b;
}

static long long grid_scatter(const Params &p, double) { return p.T; }
// Items are dealt round-robin to resident blocks (one that started late would finish late).
static long long grid_scatter2(const Params &p, double share) {
    const long long items = scatter2_items(p);
    if (items == 0) return 0;
    long long grid = (long long)((double)ms_blocks(smem_scatter2(p)) * sm_count() * share + 0.999);
    if (grid < 1) grid = 1;
    return items < grid ? items : grid;
}
static long long units_scatter2(const Params &p) { return scatter2_items(p); }
static long long full_scatter2(const Params &, long long total) {
    // the members' sizes differ: as many as fit with the largest layout of compact records
    const long long g = (long long)ms_blocks(sb2_layout<RecC>(256).total) * sm_count();
    return total < g ? total : g;
}

template <typename OffT, typename Rec1>
static cudaError_t launch_scatter_t(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                                    cudaStream_t st) {
    // one transpose that counts P x P elsewhere (or not at all): the lean
    // instantiation with its own, smaller shared memory
    // (a batch: every member of the launch shares scatter_counts_pp, its group key)
    const bool pp = scatter_counts_pp(m0.p) && (ba.n || m0.out.part_cells != nullptr);
    auto kern = !pp ? (ba.n ? k_scatter<OffT, Rec1, true, 0> : k_scatter<OffT, Rec1, false, 0>)
                : m0.p.pp_aligned ? (ba.n ? k_scatter<OffT, Rec1, true, 1> : k_scatter<OffT, Rec1, false, 1>)
                                  : (ba.n ? k_scatter<OffT, Rec1, true, 2> : k_scatter<OffT, Rec1, false, 2>);
    // one transpose without P x P tables: its own, smaller shared memory (a
    // batch keeps the maximum over its members, which bounds the lean layout)
    if (!pp && !ba.n) smem = smem_scatter_pp(m0.p, false);
    return launch_kernel(kern, ba.n > 0, grid, MS_THREADS, smem, st, m0, ba);
}

template <typename OffT, typename Rec1, typename Rec>
static cudaError_t launch_scatter2_t(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                                     cudaStream_t st) {
    auto kern2 = ba.n ? k_scatter2<OffT, Rec1, Rec, true> : k_scatter2<OffT, Rec1, Rec, false>;
    return launch_kernel(kern2, ba.n > 0, grid, MS_THREADS, smem, st, m0, ba);
}

static cudaError_t launch_scatter(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                                  cudaStream_t st) {
    const Params &p = m0.p;
    const bool w1 = p.wide || p.wide_mid;
    if (p.o == 4)
        return w1 ? launch_scatter_t<int32_t, RecW>(m0, ba, grid, smem, st)
                  : launch_scatter_t<int32_t, RecC>(m0, ba, grid, smem, st);
    return w1 ? launch_scatter_t<int64_t, RecW>(m0, ba, grid, smem, st)
              : launch_scatter_t<int64_t, RecC>(m0, ba, grid, smem, st);
}

static cudaError_t launch_scatter2(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                                   cudaStream_t st) {
    const Params &p = m0.p;
    if (p.o == 4) {
        if (p.wide) return launch_scatter2_t<int32_t, RecW, RecW>(m0, ba, grid, smem, st);
        return p.wide_mid ? launch_scatter2_t<int32_t, RecW, RecC>(m0, ba, grid, smem, st)
                          : launch_scatter2_t<int32_t, RecC, RecC>(m0, ba, grid, smem, st);
    }
    if (p.wide) return launch_scatter2_t<int64_t, RecW, RecW>(m0, ba, grid, smem, st);
    return p.wide_mid ? launch_scatter2_t<int64_t, RecW, RecC>(m0, ba, grid, smem, st)
                      : launch_scatter2_t<int64_t, RecC, RecC>(m0, ba, grid, smem, st);
}

const PhaseOps kScatterPhases[2] = {
    {"scatter", grid_scatter, smem_scatter, launch_scatter, nullptr, nullptr},
    {"scatter2", grid_scatter2, smem_scatter2, launch_scatter2, units_scatter2, full_scatter2},
};

}  // namespace mgt
