// Host driver of the finder's two kernels for seeds with wide windows (tests
// only): find_kernel, as one warp of 32 lane threads, lists the seeds it leaves;
// find_wide_kernel then runs as one block of one warp, which it is for beam
// widths 1 and 2.  The hit bins are built as in find_emu.cpp.
#include "warp_emu.h"

template <class T>
inline T __shfl_xor_sync(unsigned m, T v, int mask) {
    return __shfl_sync(m, v, static_cast<int>(threadIdx.x & 31) ^ mask);
}
inline unsigned __reduce_max_sync(unsigned m, unsigned v) {
    for (int off = 16; off > 0; off >>= 1) v = std::max(v, __shfl_xor_sync(m, v, off));
    return v;
}
inline bool __syncthreads_or(bool p) { return __any_sync(0xffffffffu, p); }
inline int atomicOr(unsigned *p, unsigned v) { return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }

#include "find_dev.inc"
#include "mkf_geom.h"

#include <thread>
#include <vector>

thread_local dim3 threadIdx, blockIdx;
dim3 blockDim;
WarpEmu *g_warp;
unsigned char *g_smem;

template <class F>
static void run_warp(size_t smem_bytes, F f) {
    std::vector<unsigned char> smem(smem_bytes);
    g_smem = smem.data();
    WarpEmu w;
    g_warp = &w;
    blockDim.x = 32;
    std::vector<std::thread> lanes;
    for (int l = 0; l < 32; ++l)
        lanes.emplace_back([&, l] {
            threadIdx.x = l;
            blockIdx.x = 0;
            f();
        });
    for (auto &t : lanes) t.join();
}

// line: the extent of a wide window in bins; 0: the library's rule; negative: no
// seed is left.  *left: the seeds find_kernel left.
extern "C" int emu_wide(const mkf_layer *layers, int nl, float bz, float material, float eloss, const float *X,
                        const float *Y, const float *Z, const int *layer, int n_hits, const int *event_offsets,
                        int n_events, const int *seed_hits, const int *seed_event, int n_seeds, int N, float cut,
                        int max_out, float line, float *out_par, float *out_cov, float *out_chi2, int *out_nh,
                        int *out_hits, unsigned *out_status, int *counters, int *fault_out, int *left) {
    static Geom G;
    if (mkf_build_geom(layers, nl, nullptr, 0, nullptr, bz, G) != MKF_OK) return -1;
    for (int l = 0; l < nl; ++l) {  // as mkf_geometry_material sets them
        G.L[l].x0 = material;
        G.L[l].eloss = eloss;
    }
    const int64_t n_bins = static_cast<int64_t>(n_events) * G.bins_per_event;
    std::vector<int> key(n_hits);
    for (int i = 0; i < n_hits; ++i) {
        int ev = 0;
        while (ev < n_events && event_offsets[ev + 1] <= i) ++ev;
        const LayerDesc &Ld = G.L[layer[i]];
        const float zr = Ld.kind == 0 ? Z[i] : sqrtf(fmaf(X[i], X[i], Y[i] * Y[i]));
        const int pb =
            std::min(std::max(static_cast<int>(floorf((atan2f(Y[i], X[i]) + kPi) * Ld.phi_scale)), 0), Ld.nphi - 1);
        const int zb = std::min(std::max(static_cast<int>(floorf((zr - Ld.lo) * Ld.zr_scale)), 0), Ld.nzr - 1);
        key[i] = ev * G.bins_per_event + Ld.bin_base + pb * Ld.nzr + zb;
    }
    std::vector<int> offsets(n_bins + 1, 0), fill(n_bins, 0);
    for (int i = 0; i < n_hits; ++i) offsets[key[i] + 1]++;
    for (int64_t b = 0; b < n_bins; ++b) offsets[b + 1] += offsets[b];
    std::vector<float4> rec(n_hits);
    std::vector<int> inv(n_hits);
    std::vector<uint8_t> layer8(n_hits);
    std::vector<float> zhit(Z, Z + n_hits);
    for (int i = 0; i < n_hits; ++i) {
        const int k = offsets[key[i]] + fill[key[i]]++;
        rec[k] = float4{X[i], Y[i], G.L[layer[i]].kind == 0 ? Z[i] : sqrtf(fmaf(X[i], X[i], Y[i] * Y[i])),
                        __int_as_float(i)};
        inv[i] = k;
        layer8[i] = static_cast<uint8_t>(layer[i]);
    }
    std::vector<float> seedbuf(static_cast<size_t>(kSeedFields) * n_seeds);
    std::vector<float> lists(static_cast<size_t>(kListFields) * n_seeds * N);
    std::vector<int> wide(n_seeds + 2, 0);
    mkf_fault fault{0, 0};
    int work = 0;
    FindArgs A;
    std::memset(&A, 0, sizeof(A));
    A.G = G;
    A.rec = rec.data();
    A.inv = inv.data();
    A.layer8 = layer8.data();
    A.zhit = zhit.data();
    A.offsets = offsets.data();
    A.n_hits = n_hits;
    A.n_events = n_events;
    A.seed_hits = seed_hits;
    A.seed_event = seed_event;
    A.n_seeds = n_seeds;
    A.n_best = N;
    A.cut = cut;
    A.max_consec = 3;
    A.max_steps = find_max_steps(nl);
    A.out_par = out_par;
    A.out_cov = out_cov;
    A.out_chi2 = out_chi2;
    A.out_nhits = out_nh;
    A.out_hits = out_hits;
    A.max_out = max_out;
    A.out_status = out_status;
    A.counters = counters;
    A.fault = &fault;
    A.seedbuf = seedbuf.data();
    A.beam = lists.data();
    A.step1 = 1;
    A.work_counter = &work;
    if (line >= 0.f) {
        A.wide_list = wide.data();
        A.wide_count = &wide[n_seeds];
        A.wide_next = &wide[n_seeds + 1];
        A.wide_bins = line > 0.f ? line : wide_bins(1, n_seeds, N, false, n_hits, n_bins, n_events, nl);
    }
    blockDim.x = 128;
    for (int t = 0; t < n_seeds; ++t) {
        blockIdx.x = t / 128;
        threadIdx.x = t % 128;
        seed_kernel<1>(A);
    }
    run_warp(find_smem_bytes(nl, N, 32), [&] {
        if (N == 1) find_kernel<false, 1, 1>(A);
        else find_kernel<false, 1, 0>(A);
    });
    *left = wide[n_seeds];
    if (line >= 0.f && N <= 2) run_warp(wide_smem_bytes(nl, N), [&] { find_wide_kernel<false, 1>(A); });
    fault_out[0] = fault.code;
    fault_out[1] = fault.where;
    return 0;
}
