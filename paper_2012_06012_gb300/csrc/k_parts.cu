// P x P cell and value counts from the transposed matrix (the metadata-count
// and value-count matrices of the paper's view swap, Sec. 3: how many cells
// and values source block s sends to destination block d).
//
// An output cell q belongs to destination block d when it lies in that
// block's output cell range [row_ptr'[off[d]], row_ptr'[off[d + 1]]); its
// source block is the block of its source row col_idx'[q].  So the counts
// need one sequential pass over col_idx' and cell_ptr' and P + 1 entries of
// row_ptr', with the counters of each tile of output cells in shared memory
// (a tile spans few destination blocks).  The planner picks this pass unless
// every row block starts on a super-bucket of the first scatter pass, which
// then counts per tile and super-bucket.
#include "mgt_internal.cuh"

namespace mgt {

constexpr int PC_THREADS = 512;
constexpr int PC_BLOCKS = 3;    // per SM
constexpr int PC_TAB = 4096;    // entries of the row -> block table
constexpr uint16_t PC_CUT = 0x8000u;  // table entry: a block boundary lies inside it

// Output cells per work unit: at most 65,536 (the 32-bit counters hold that
// many runs of less than 2^16 values), fewer where that would idle SMs.
__host__ __device__ inline long long parts_tile(const Params &p) {
    long long t = 65536;
    while (t > 2048 && p.C / t < 1024) t >>= 1;
    return t;
}
__host__ __device__ inline long long parts_units(const Params &p) {
    return (p.pp_out && p.P > 1 && p.C > 0) ? (p.C + parts_tile(p) - 1) / parts_tile(p) : 0;
}

// Shared memory: the blocks' first rows po[P+1] and first output cells
// co[P+1]; cell and value counters of one destination block, [P] each; a row
// -> block table: entry k is the block of row k << tsh, marked when rows of
// the entry belong to later blocks too.
__host__ __device__ inline size_t parts_smem(int P) {
    return (size_t)(P + 1) * 8 + (size_t)P * 8 + (size_t)PC_TAB * 2;
}

// One unit's cells in pieces of one destination block each, so that a counter
// is found by the source block alone.  A lane adds to shared counters on its
// own unless eight or more lanes share the first lane's block (the long rows
// of hot columns, whose neighbouring cells come from nearby rows): those add
// up first.  Bound by issue slots and the dependent table lookup, at a third
// of the copy rate in bytes: 168M cells, 256 blocks 0.79 -> 0.63 ms.
template <typename OffT, bool BATCH>
__global__ void __launch_bounds__(PC_THREADS, PC_BLOCKS)
    k_part_counts(const __grid_constant__ Mat m0, const BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char smem[];
    pipeline_wait<BATCH>();
    Units<BATCH> U(m0, ba, blockIdx.x, gridDim.x);
    const Mat *cur = nullptr;  // the matrix whose tables are in shared memory
    const int tid = threadIdx.x, lane = tid & 31;
    while (U.next([](const Mat &X) {
        return (X.out.part_cells == nullptr || (X.ws.hdr->status & (ST_BADINPUT | ST_OVERFLOW)))
                   ? 0ull
                   : (unsigned long long)parts_units(X.p);
    })) {
        const Mat &M = *U.M;
        const int P = M.p.P;
        const long long C = M.p.C, R = M.p.R, N = M.p.N;
        uint32_t *po = reinterpret_cast<uint32_t *>(smem);
        uint32_t *co = po + (P + 1);
        uint32_t *cnt = co + (P + 1);
        uint32_t *val = cnt + P;
        uint16_t *tab = reinterpret_cast<uint16_t *>(val + P);
        int tsh = 0;
        while ((R >> tsh) >= PC_TAB) ++tsh;
        if (cur != &M) {  // tables of this matrix (block-uniform: every thread has the same U.M)
            __syncthreads();
            for (int d = tid; d <= P; d += PC_THREADS) {
                const long long r0 = M.ws.poff[d];
                const long long r = r0 < 0 ? 0 : (r0 > N ? N : r0);
                po[d] = (uint32_t)r;
                co[d] = (uint32_t)ldp<OffT>(M.out.row_ptr, r);
            }
            for (int x = tid; x < P; x += PC_THREADS) cnt[x] = val[x] = 0;
            __syncthreads();
            auto block_of = [&](uint32_t row) {  // last block that starts at or before the row
                int lo = 0, hi = P;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (po[mid] <= row) lo = mid;
                    else hi = mid;
                }
                return lo;
            };
            for (long long k = tid; k <= (R - 1) >> tsh; k += PC_THREADS) {
                const int b = block_of((uint32_t)(k << tsh));
                const uint32_t last = (uint32_t)min(((k + 1) << tsh) - 1, R - 1);
                tab[k] = (uint16_t)(b | (b < P - 1 && po[b + 1] <= last ? PC_CUT : 0));
            }
            cur = &M;
        }
        const long long tile = parts_tile(M.p);
        const uint32_t q0 = (uint32_t)(U.j * tile), q1 = (uint32_t)min(C, (long long)(U.j + 1) * tile);
        __syncthreads();
        const int32_t *__restrict__ ocol = M.out.col;
        const void *ocp = M.out.cell_ptr;
        unsigned long long *part_cells = reinterpret_cast<unsigned long long *>(M.out.part_cells);
        unsigned long long *part_values = reinterpret_cast<unsigned long long *>(M.out.part_values);
        int d = 0;
        {
            int hi = P;  // last block that starts at or before q0
            while (hi - d > 1) {
                const int mid = (d + hi) >> 1;
                if (co[mid] <= q0) d = mid;
                else hi = mid;
            }
        }
        for (uint32_t qa = q0; qa < q1;) {
            while (d < P - 1 && co[d + 1] <= qa) ++d;  // (empty blocks hold no cells)
            const uint32_t qb = d < P - 1 ? min(q1, co[d + 1]) : q1;
            // rounds of PC_U x PC_THREADS consecutive cells, all their loads in
            // flight first (the same trip count for every thread: warp-wide votes)
            constexpr int PC_U = 4;
            for (uint32_t done = 0; done < qb - qa; done += PC_U * PC_THREADS) {
                const uint32_t base = qa + done;
                uint32_t iu[PC_U];
                long long lu[PC_U];
#pragma unroll
                for (int u = 0; u < PC_U; ++u) {
                    const uint32_t q = base + u * PC_THREADS + tid;
                    iu[u] = 0;
                    lu[u] = 0;
                    if (q < qb && q >= base) {
                        iu[u] = (uint32_t)ocol[q];
                        lu[u] = ldp<OffT>(ocp, (long long)q + 1) - ldp<OffT>(ocp, q);
                    }
                }
#pragma unroll
                for (int u = 0; u < PC_U; ++u) {
                    const uint32_t q = base + u * PC_THREADS + tid;
                    bool v = q < qb && q >= base;
                    const uint32_t i = min(iu[u], (uint32_t)(R - 1));
                    uint32_t s = tab[i >> tsh];
                    if (s & PC_CUT) {
                        s &= ~(uint32_t)PC_CUT;
                        while (s < (uint32_t)P - 1 && po[s + 1] <= i) ++s;
                    }
                    uint32_t len = lu[u] > 0 ? (uint32_t)min(lu[u], 0xFFFFFFFFll) : 0u;
                    if (len >= 65536u) {  // a very long run: straight to the global counter
                        atomicAdd(&part_values[(long long)s * P + d], (unsigned long long)lu[u]);
                        len = 0;
                    }
                    const uint32_t s0 = __shfl_sync(0xffffffffu, s, 0);
                    const unsigned same = __ballot_sync(0xffffffffu, v && s == s0);
                    if (__popc(same) >= 8) {
                        const uint32_t sum = __reduce_add_sync(0xffffffffu, v && s == s0 ? len : 0u);
                        if (lane == 0) {
                            atomicAdd(&cnt[s0], (uint32_t)__popc(same));
                            atomicAdd(&val[s0], sum);
                        }
                        v = v && s != s0;
                    }
                    if (v) {
                        atomicAdd(&cnt[s], 1u);
                        atomicAdd(&val[s], len);
                    }
                }
            }
            __syncthreads();
            for (int x = tid; x < P; x += PC_THREADS) {
                if (cnt[x] == 0) continue;
                atomicAdd(&part_cells[(long long)x * P + d], (unsigned long long)cnt[x]);
                atomicAdd(&part_values[(long long)x * P + d], (unsigned long long)val[x]);
                cnt[x] = val[x] = 0;
            }
            __syncthreads();
            qa = qb;
        }
    }
}

static long long grid_parts(const Params &p, double share) {
    const long long u = parts_units(p);
    if (u == 0) return 0;
    long long g = (long long)((double)PC_BLOCKS * sm_count() * share + 0.999);
    if (g < 1) g = 1;
    return u < g ? u : g;
}
static size_t smem_parts(const Params &p) { return p.pp_out ? parts_smem(p.P) : 0; }
static long long units_parts(const Params &p) { return parts_units(p); }
static long long full_parts(const Params &p, long long total) {
    const long long g = (long long)PC_BLOCKS * sm_count();
    return total < g ? (total < 1 ? 1 : total) : g;
}
static cudaError_t launch_parts(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                                cudaStream_t st) {
    if (ba.n == 0 && m0.out.part_cells == nullptr) return cudaSuccess;  // counts not asked for
    auto kern = m0.p.o == 4 ? (ba.n ? k_part_counts<int32_t, true> : k_part_counts<int32_t, false>)
                            : (ba.n ? k_part_counts<int64_t, true> : k_part_counts<int64_t, false>);
    return launch_kernel(kern, ba.n > 0, grid, PC_THREADS, smem, st, m0, ba);
}

const PhaseOps kPartsPhase = {"part_counts", grid_parts, smem_parts, launch_parts, units_parts, full_parts};

// Whether the planner hands the P x P counts to this pass: P within the
// shared-memory tables and some row block starts inside a super-bucket of the
// first scatter pass (whose totals per super-bucket would then not be those
// of a block).  pp_aligned: none does.
bool parts_from_output(const Params &p, const long long *off, int *pp_aligned) {
    *pp_aligned = 0;
    if (p.P <= 1 || p.B == 0 || !off) return false;
    const int sh = p.p2 + p.bshift;  // log2 of the columns of a super-bucket
    bool cut = false;
    for (int d = 1; d < p.P && !cut; ++d)
        cut = off[d] > 0 && off[d] < p.N && (off[d] & ((1LL << sh) - 1)) != 0;
    *pp_aligned = cut ? 0 : 1;
    return cut && p.P <= PC_MAX_PARTS;
}

}  // namespace mgt
