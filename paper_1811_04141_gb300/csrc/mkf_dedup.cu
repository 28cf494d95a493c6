// Seed cleaning before finding and duplicate-track removal after it (Sec. 2.2:
// repeated seeds of one particle are removed using the identity of their hits
// and their fitted pT, eta and phi; Sec. 3: duplicate tracks from several seeds
// per particle are to be removed after finding).
//
// Both are decisions over the graph of items (seeds or tracks) that share hits.
// The graph is built as an inverse index, hit -> items using it (a count pass,
// the binning's exclusive scan, a fill pass), after which one thread per item
// walks its hits and the items listed on them.  An item is dropped when a
// duplicate that ranks above it exists, whether or not that one is dropped
// itself, so no decision waits on another and the result does not depend on
// the order of the threads.
#include <cuda_runtime.h>

#include "mkf_internal.h"

namespace {

constexpr int kThreads = 256;

// Entries of a list that are valid hits; a hit listed twice appears twice in the
// index (the decisions ask only whether an item is listed there, so that does
// not matter, and looking back along the list for every entry would make both
// passes quadratic in its rows: 8.0 and 9.4 us then, 5.6 and 7.6 us now, for
// 44 000 tracks of 23 rows).
__global__ void __launch_bounds__(kThreads) count_kernel(const int32_t *lists, int32_t rows, int32_t n,
                                                         int32_t n_hits, int32_t *cnt) {
    after_previous();
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= (int64_t)rows * n) return;
    const int32_t h = lists[t];
    if (h >= 0 && h < n_hits) atomicAdd(&cnt[h], 1);
}

// Slots are handed out per hit with the counters running back to zero, so the
// counters are ready for the next call.
__global__ void __launch_bounds__(kThreads) fill_kernel(const int32_t *lists, int32_t rows, int32_t n, int32_t n_hits,
                                                        const int32_t *off, int32_t *cnt, int32_t *items) {
    after_previous();
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= (int64_t)rows * n) return;
    const int32_t h = lists[t];
    if (h < 0 || h >= n_hits) return;
    items[off[h + 1] - atomicSub(&cnt[h], 1)] = static_cast<int32_t>(t % n);
}

// Whether item i lists hit h before row k.
__device__ __forceinline__ bool listed_before(const int32_t *lists, int32_t k, int32_t n, int32_t i, int32_t h) {
    for (int32_t r = 0; r < k; ++r)
        if (lists[(int64_t)r * n + i] == h) return true;
    return false;
}

// eta of a polar angle, in double (both sides of a threshold test see the same
// value up to the last bit of a double).
__device__ __forceinline__ double eta_of(float theta) { return -log(tan(0.5 * static_cast<double>(theta))); }

// |eta_of(ta) - eta_of(tb)| <= tol.  The double logarithms and tangents are slow
// (FP64 units), so the difference is taken in FP32 first, which decides unless it
// lies within 1e-4 of the tolerance (FP32 eta: a few 1e-7 of itself, and |eta| is
// below 104 for a finite one).
__device__ __forceinline__ bool eta_within(float ta, float tb, double tol) {
    const float ea = -logf(tanf(0.5f * ta)), eb = -logf(tanf(0.5f * tb));
    const float d = fabsf(ea - eb), t = static_cast<float>(tol);
    const float margin = 1e-4f * (1.f + t);
    if (d < t - margin) return true;
    if (d > t + margin && d < 1e30f) return false;
    return fabs(eta_of(ta) - eta_of(tb)) <= tol;
}

// |a| wrapped into [0, pi].
__device__ __forceinline__ double wrapped_abs(double a) {
    constexpr double kPiD = 3.14159265358979323846;
    a = a + kPiD;
    if (!(a >= 0.0 && a < 2.0 * kPiD)) {  // else fmod returns it as it is
        a = fmod(a, 2.0 * kPiD);
        if (a < 0.0) a += 2.0 * kPiD;
    }
    return fabs(a - kPiD);
}

// Seeds: drop i when a seed u < i shares a hit with it and their fitted q/pT,
// eta and phi agree within the tolerances (differences in double on the given
// float parameters).  Bound: latency of the chain hit -> range -> items, and of
// FP64 where it is needed: 30.5 us for 44 000 seeds with every eta in double and
// every range walked, 12.6 us now.
__global__ void __launch_bounds__(kThreads) seeds_decide_kernel(const int32_t *seed_hits, int32_t n, int32_t n_hits,
                                                                const float *par, double max_dqpt, double max_deta,
                                                                double max_dphi, const int32_t *off,
                                                                const int32_t *items, int32_t *keep) {
    after_previous();
    const int32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    // the three hits' ranges at once: most seeds share none and end there
    int32_t b[3], e[3];
#pragma unroll
    for (int32_t r = 0; r < 3; ++r) {
        const int32_t h = seed_hits[(int64_t)r * n + i];
        const bool valid = h >= 0 && h < n_hits;
        b[r] = valid ? off[h] : 0;
        e[r] = valid ? off[h + 1] : 0;
    }
    bool k_ = true;
#pragma unroll
    for (int32_t r = 0; r < 3; ++r) {
        if (e[r] - b[r] < 2) continue;  // listed by this seed only
        for (int32_t p = b[r]; p < e[r] && k_; ++p) {
            const int32_t u = items[p];
            if (u >= i) continue;
            const double dw = static_cast<double>(par[3 * (int64_t)n + i]) - par[3 * (int64_t)n + u];
            const double dph = static_cast<double>(par[4 * (int64_t)n + i]) - par[4 * (int64_t)n + u];
            if (fabs(dw) <= max_dqpt && wrapped_abs(dph) <= max_dphi &&
                eta_within(par[5 * (int64_t)n + i], par[5 * (int64_t)n + u], max_deta))
                k_ = false;
        }
    }
    keep[i] = k_ ? 1 : 0;
}

// Tracks: drop i when a better track u (more hits, then lower chi2, then lower
// index) shares at least max(1, min_frac x the shorter one's hit count) hits.
// Bound: latency of the chain hit -> range -> items -> the other track, taken for
// several rows together.  Whether the other track lists a hit is looked up among
// the hit's items where these are no more than a list has rows (a few, mostly:
// 92 -> 30 us for 44 000 tracks of 23 rows, a tenth of them duplicates), else
// along the other track's list, or the work would grow with the square of the
// tracks on a hit.  20 000 tracks of 23 rows in groups that share 40 % of their
// hits, 128 / 1000 tracks a group: 27.5 / 248 ms; 55.4 / 2960 ms by the items
// alone, 52.6 / 415 ms along the lists alone.  Groups of equal tracks are bound by
// the best one's walk over every item, one item ahead of its test: 3.8 ms for
// 1000 a group (4.2 without, 3.95 along the lists alone).
__global__ void __launch_bounds__(kThreads) tracks_decide_kernel(const int32_t *hit_idx, int32_t rows, int32_t n,
                                                                 int32_t n_hits, const int32_t *nh, const float *chi2,
                                                                 float min_frac, const int32_t *off,
                                                                 const int32_t *items, int32_t *keep) {
    after_previous();
    const int32_t i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const int32_t ni = nh[i];
    const float ci = chi2[i];
    bool k_ = true;
    // kBatch rows at a time: their index ranges load together
    constexpr int32_t kBatch = 8;
    for (int32_t r0 = 0; r0 < rows && k_; r0 += kBatch) {
        int32_t b[kBatch], e[kBatch];
#pragma unroll
        for (int32_t j = 0; j < kBatch; ++j) {
            const int32_t h = r0 + j < rows ? hit_idx[(int64_t)(r0 + j) * n + i] : -1;
            const bool valid = h >= 0 && h < n_hits;
            b[j] = valid ? off[h] : 0;
            e[j] = valid ? off[h + 1] : 0;
        }
#pragma unroll
        for (int32_t j = 0; j < kBatch; ++j) {
            if (e[j] - b[j] < 2) continue;  // listed by this track only
            int32_t next = items[b[j]];  // loaded while the one before it is tested
            for (int32_t p = b[j]; p < e[j] && k_; ++p) {
                const int32_t u = next;
                if (p + 1 < e[j]) next = items[p + 1];
                if (u == i) continue;
                const int32_t nu = nh[u];
                const float cu = chi2[u];
                const bool better = nu > ni || (nu == ni && (cu < ci || (cu == ci && u < i)));
                if (!better) continue;
                // hits of i (as a set) that u lists; enough of them end the
                // count.  Looked up among the hit's items or, where these are
                // more than a list has rows, along u's own list.
                const double need = fmax(1.0, static_cast<double>(min_frac) * min(ni, nu));
                int32_t shared = 0;
                for (int32_t a = 0; a < rows && shared < need; ++a) {
                    const int32_t ha = hit_idx[(int64_t)a * n + i];
                    if (ha < 0 || ha >= n_hits) continue;
                    const int32_t q0 = off[ha], q1 = off[ha + 1];
                    // one loop for both (a loop each: 7 % slower where few share a hit)
                    const bool crowded = q1 - q0 > rows;
                    const int32_t *L = crowded ? hit_idx + u : &items[q0];
                    const int64_t stride = crowded ? n : 1;
                    const int32_t len = crowded ? rows : q1 - q0, want = crowded ? ha : u;
                    bool has = false;
                    for (int32_t c = 0; c < len && !has; ++c, L += stride) has = *L == want;
                    if (has && !listed_before(hit_idx, a, n, i, ha)) ++shared;
                }
                if (shared >= need) k_ = false;
            }
        }
    }
    keep[i] = k_ ? 1 : 0;
}

// Inverse index hit -> items of `lists` [rows][n]; scratch carved from the
// context: counters, offsets, scan sums, item slots.
mkf_status build_index(mkf_ctx *ctx, const int32_t *lists, int32_t rows, int32_t n, int32_t n_hits,
                       const int32_t **off_out, const int32_t **items_out) {
    const int64_t pairs = (int64_t)rows * n;
    const int64_t nts = mkf_scan_tilesums(n_hits);
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    const int64_t b_cnt = up(4 * (int64_t)n_hits), b_off = up(4 * ((int64_t)n_hits + 1)), b_ts = up(4 * (nts + 1)),
                  b_items = up(4 * pairs);
    void *scr = nullptr;
    const mkf_status st = mkf_scratch(ctx, b_cnt + b_off + b_ts + b_items, &scr);
    if (st != MKF_OK) return st;
    char *c = static_cast<char *>(scr);
    int32_t *cnt = reinterpret_cast<int32_t *>(c);
    int32_t *off = reinterpret_cast<int32_t *>(c + b_cnt);
    int32_t *ts = reinterpret_cast<int32_t *>(c + b_cnt + b_off);
    int32_t *items = reinterpret_cast<int32_t *>(c + b_cnt + b_off + b_ts);
    cudaStream_t s = ctx->stream;
    MKF_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)n_hits, s));
    const unsigned blocks = static_cast<unsigned>((pairs + kThreads - 1) / kThreads);
    if (pairs > 0) {
        MKF_CUDA_TRY(mkf_launch(count_kernel, blocks, kThreads, 0, s, lists, rows, n, n_hits, cnt));
    }
    const mkf_status ss = mkf_run_scan(s, cnt, n_hits, ts, off);
    if (ss != MKF_OK) return ss;
    if (pairs > 0) {
        MKF_CUDA_TRY(mkf_launch(fill_kernel, blocks, kThreads, 0, s, lists, rows, n, n_hits, off, cnt, items));
    }
    *off_out = off;
    *items_out = items;
    return MKF_OK;
}

}  // namespace

extern "C" mkf_status mkf_seeds_clean(mkf_ctx *ctx, const int32_t *seed_hits, int32_t n_seeds, int32_t n_hits,
                                      const float *seed_par, float max_dqpt, float max_deta, float max_dphi,
                                      int32_t *keep) {
    if (!ctx) return MKF_ERR_ARG;
    if (n_seeds < 0 || n_hits < 0) return MKF_ERR_ARG;
    if (n_hits > MKF_MAX_HITS) return MKF_ERR_CAPACITY;
    if (!(max_dqpt >= 0.f) || !(max_deta >= 0.f) || !(max_dphi >= 0.f)) return MKF_ERR_ARG;
    if (n_seeds == 0) return MKF_OK;
    if (!seed_hits || !seed_par || !keep) return MKF_ERR_ARG;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    const int32_t *off = nullptr, *items = nullptr;
    const mkf_status st = build_index(ctx, seed_hits, 3, n_seeds, n_hits, &off, &items);
    if (st != MKF_OK) return st;
    MKF_CUDA_TRY(mkf_launch(seeds_decide_kernel, (n_seeds + kThreads - 1) / kThreads, kThreads, 0, ctx->stream, seed_hits,
                            n_seeds, n_hits, seed_par, max_dqpt, max_deta, max_dphi, off, items, keep));
    return MKF_OK;
}

extern "C" mkf_status mkf_tracks_dedup(mkf_ctx *ctx, const int32_t *hit_idx, int32_t max_hits, int32_t n,
                                       int32_t n_hits, const int32_t *track_nhits, const float *chi2, float min_frac,
                                       int32_t *keep) {
    if (!ctx) return MKF_ERR_ARG;
    if (n < 0 || n_hits < 0 || max_hits < 1) return MKF_ERR_ARG;
    if (max_hits > MKF_MAX_LAYERS + 8) return MKF_ERR_CAPACITY;
    if (n_hits > MKF_MAX_HITS) return MKF_ERR_CAPACITY;
    if (!(min_frac >= 0.f && min_frac <= 1.f)) return MKF_ERR_ARG;
    if (n == 0) return MKF_OK;
    if (!hit_idx || !track_nhits || !chi2 || !keep) return MKF_ERR_ARG;
    DeviceGuard g(ctx->device);
    if (!g.ok) return MKF_ERR_CUDA;
    const int32_t *off = nullptr, *items = nullptr;
    const mkf_status st = build_index(ctx, hit_idx, max_hits, n, n_hits, &off, &items);
    if (st != MKF_OK) return st;
    MKF_CUDA_TRY(mkf_launch(tracks_decide_kernel, (n + kThreads - 1) / kThreads, kThreads, 0, ctx->stream, hit_idx, max_hits,
                            n, n_hits, track_nhits, chi2, min_frac, off, items, keep));
    return MKF_OK;
}
