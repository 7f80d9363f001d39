// Dispatch of the level-2 phases (sort/place, the large-bucket chunk passes
// and the value copy) over offset width and record format, and their grid
// and shared-memory sizes.
#include "k_place_impl.cuh"

namespace mgt {

static cudaError_t level2(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                          cudaStream_t st, int which) {
    const Params &p = m0.p;
    if (p.o == 4)
        return p.wide ? launch_level2_t<int32_t, RecW>(m0, ba, grid, smem, st, which)
                      : launch_level2_t<int32_t, RecC>(m0, ba, grid, smem, st, which);
    return p.wide ? launch_level2_t<int64_t, RecW>(m0, ba, grid, smem, st, which)
                  : launch_level2_t<int64_t, RecC>(m0, ba, grid, smem, st, which);
}

// Shared memory of the one-block sort for `cap` records of w columns.
size_t sort_smem_bytes(const Params &p, int cap) {
    return p.wide ? pl_layout<RecW>(cap, 1 << p.bshift).total : pl_layout<RecC>(cap, 1 << p.bshift).total;
}
int sort_cap_max() { return PL_CAP; }
// Shared memory of a cluster's sort for p.cap records per CTA (p.cs = 1: the
// layout that bounds the capacities a shape may name).
size_t cluster_smem_bytes(const Params &p) {
    const int logcs = p.cs == 1 ? 0 : p.cs == 2 ? 1 : p.cs == 4 ? 2 : 3;
    const int wsub = 1 << (p.bshift - logcs);
    switch (p.cs) {
    case 1: return p.wide ? cl_layout<RecW, 1>(p.cap, wsub).total : cl_layout<RecC, 1>(p.cap, wsub).total;
    case 2: return p.wide ? cl_layout<RecW, 2>(p.cap, wsub).total : cl_layout<RecC, 2>(p.cap, wsub).total;
    case 4: return p.wide ? cl_layout<RecW, 4>(p.cap, wsub).total : cl_layout<RecC, 4>(p.cap, wsub).total;
    default: return p.wide ? cl_layout<RecW, 8>(p.cap, wsub).total : cl_layout<RecC, 8>(p.cap, wsub).total;
    }
}

// persistent grids: the matrix's share of `per_sm` blocks per SM, at most `work`
static long long share_grid(double per_sm, double share, long long work) {
    long long g = (long long)(per_sm * sm_count() * share + 0.999);
    if (g < 1) g = 1;
    return work < g ? work : g;
}

// Sort clusters the cluster-place kernel can keep resident, for this plan
// (0 without a device: the grid then takes one cluster per SM pair).
static long long resident_clusters(const Params &p) {
    const size_t smem = cluster_smem_bytes(p);
    long long n = p.o == 4 ? (p.wide ? resident_clusters_t<int32_t, RecW>(p.cs, smem)
                                     : resident_clusters_t<int32_t, RecC>(p.cs, smem))
                           : (p.wide ? resident_clusters_t<int64_t, RecW>(p.cs, smem)
                                     : resident_clusters_t<int64_t, RecC>(p.cs, smem));
    if (n < 1) n = sm_count() / (p.cs > 1 ? p.cs : 1);
    return n < 1 ? 1 : n;
}

static bool may_chunk(const Params &p) { return p.B > 0 && p.max_multi_rows > 0; }
static long long grid_chunk_hist(const Params &p, double) { return may_chunk(p) ? p.max_multi_rows : 0; }
static long long grid_chunk_scan(const Params &p, double share) {
    return may_chunk(p) ? share_grid(K6_BLOCKS, share, p.max_multi_buckets * K6_UNITS) : 0;
}
// one block per work item; with clusters only the chunks are these blocks' work
static long long grid_place(const Params &p, double) {
    return p.B == 0 || (p.cs > 1 && !may_chunk(p)) ? 0 : p.max_items;
}
static long long grid_clusters(const Params &p, double share) {
    if (p.B == 0 || p.cs == 1) return 0;
    long long ncl = (long long)(resident_clusters(p) * share + 0.999);
    if (ncl < 1) ncl = 1;
    if (ncl > p.max_items) ncl = p.max_items < 1 ? 1 : p.max_items;
    return ncl * p.cs;
}
static long long grid_fallback(const Params &p, double share) {
    if (p.B == 0 || p.cs == 1) return 0;  // (only a cluster's owner can overflow)
    return share_grid(1.0, share, p.max_items);
}
static long long grid_copy(const Params &p, double) {
    if (p.var) return 1;  // variable-width values: launch_var_copy sizes its own grids
    if (p.C == 0 || p.V == 0) return 0;
    return (p.C + (1LL << p.cshift) - 1) >> p.cshift;  // one block per tile of output cells
}

static size_t smem_chunk_hist(const Params &p) {
    const size_t w = (size_t)1 << p.bshift;
    return w * 16;
}
static size_t smem_wide_scan(const Params &p) { return ((size_t)1 << p.bshift) * 16 + 48 * 8; }
static size_t smem_place(const Params &p) { return sort_smem_bytes(p, p.cs > 1 ? p.chm : p.cap); }
static size_t smem_clusters(const Params &p) { return cluster_smem_bytes(p); }
static size_t smem_zero(const Params &) { return 0; }

#define MGT_L2(fn, which)                                                                    \
    static cudaError_t fn(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem, \
                          cudaStream_t st) {                                                  \
        return level2(m0, ba, grid, smem, st, which);                                         \
    }
MGT_L2(launch_chunk_hist, 0)
MGT_L2(launch_chunk_scan, 1)
MGT_L2(launch_place, 2)
MGT_L2(launch_clusters, 3)
MGT_L2(launch_place_fallback, 4)
#undef MGT_L2
static cudaError_t launch_copy(const Mat &m0, const BatchArgs &ba, long long grid, size_t smem,
                               cudaStream_t st) {
    if (m0.p.var) return launch_var_copy(m0, st);  // single transposes only
    return level2(m0, ba, grid, smem, st, 5);
}

// Host bounds on the work units of the persistent phases (a batch deals
// them to one GPU-filling grid), and that grid for `total` units.
static long long units_multi_buckets(const Params &p) { return p.B == 0 ? 0 : p.max_multi_buckets * K6_UNITS; }
static long long units_clusters(const Params &p) { return p.B == 0 || p.cs == 1 ? 0 : p.max_items; }
static long long cap_total(long long g, long long total) { return total < g ? (total < 1 ? 1 : total) : g; }
static long long full_chunk_scan(const Params &, long long total) { return cap_total((long long)K6_BLOCKS * sm_count(), total); }
static long long full_one_per_sm(const Params &, long long total) { return cap_total(sm_count(), total); }
static long long full_clusters(const Params &p, long long total) {
    return cap_total(resident_clusters(p), total) * p.cs;
}

const PhaseOps kPlacePhases[6] = {
    {"chunk_hist", grid_chunk_hist, smem_chunk_hist, launch_chunk_hist, nullptr, nullptr},
    {"chunk_scan", grid_chunk_scan, smem_zero, launch_chunk_scan, units_multi_buckets, full_chunk_scan},
    {"place", grid_place, smem_place, launch_place, nullptr, nullptr},
    {"place_clusters", grid_clusters, smem_clusters, launch_clusters, units_clusters, full_clusters},
    {"place_fallback", grid_fallback, smem_wide_scan, launch_place_fallback, units_clusters, full_one_per_sm},
    {"copy", grid_copy, smem_zero, launch_copy, nullptr, nullptr},
};

}  // namespace mgt
