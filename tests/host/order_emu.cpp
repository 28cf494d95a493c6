// Host run of the finder's seed kernel and order kernel (tests only), thread by
// thread: the processing order of a call on a list of seeds, in a buffer that
// holds what an earlier call left there.
#include "find_dev.inc"
#include "mkf_geom.h"

#include <vector>

thread_local dim3 threadIdx, blockIdx;
dim3 blockDim;
WarpEmu *g_warp;
unsigned char *g_smem;

// One event without hits (no seed is valid: all have the same key).  order
// [n_seeds]: as an earlier call left it; returns the number of seeds in the call.
extern "C" int emu_order(const mkf_layer *layers, int nl, const int *seed_hits, const int *seed_event, int n_seeds,
                         int n_events, const int *list, int count, int *order, int *fault_out) {
    static Geom G;
    if (mkf_build_geom(layers, nl, nullptr, 0, nullptr, 3.8f, G) != MKF_OK) return -1;
    std::vector<float> seedbuf(static_cast<size_t>(kSeedFields) * n_seeds);
    const int n_keys = n_events * kOrderBuckets;
    std::vector<int> key(n_seeds, -9), pos(n_seeds, -9), counts(n_keys + 1, 0);
    mkf_fault fault{0, 0};
    int work = 0;
    FindArgs A;
    std::memset(&A, 0, sizeof(A));
    A.G = G;
    A.n_events = n_events;
    A.seed_hits = seed_hits;
    A.seed_event = seed_event;
    A.n_seeds = n_seeds;
    A.n_best = 1;
    A.seedbuf = seedbuf.data();
    A.fault = &fault;
    A.work_counter = &work;
    A.seed_list = list;
    A.seed_count = list ? &count : nullptr;
    A.order_key = key.data();
    A.order_pos = pos.data();
    A.order_counts = counts.data();
    blockDim.x = 128;
    for (int t = 0; t < n_seeds; ++t) {
        blockIdx.x = t / 128;
        threadIdx.x = t % 128;
        seed_kernel<0>(A);
    }
    int total = 0;
    for (int k = 0; k < n_keys; ++k) {
        const int c = counts[k];
        counts[k] = total;
        total += c;
    }
    counts[n_keys] = total;
    blockDim.x = 256;
    for (int t = 0; t < n_seeds; ++t) {
        blockIdx.x = t / 256;
        threadIdx.x = t % 256;
        order_scatter_kernel(key.data(), pos.data(), counts.data(), n_seeds, list, A.seed_count, order);
    }
    fault_out[0] = fault.code;
    fault_out[1] = fault.where;
    return total;
}
