// fp_device.cu -- resident forests and the classification entry points.
//
// fp_upload copies a packed image to the device; fp_predict launches the
// persistent traversal kernel (fp_traverse.cuh) on the caller's stream, in the
// shape that plan_rows chooses for the batch.  The kernel needs scratch memory
// only where bins are split over CTAs and more than votes is asked for: one
// counter per observation tile, and an accumulator (of votes, unless they add
// up in the caller's buffer; of leaf values).  Bins of a forest of one pass are
// not split for it under capture or in fp_predict_noalloc.  The scratch comes
// from a library-owned stream-ordered memory pool, so calls on different
// streams never share it.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/forest_pack.h"
#include "fp_common.h"
#include "fp_internal.h"
#include "fp_traverse.cuh"

struct fp_device_forest {
    int device = -1;
    FpImageHeader hdr{};
    std::vector<FpBin> bins;
    std::vector<FpPass> passes;
    uint8_t *d_image = nullptr;
    uint8_t *d_compact = nullptr;  // one-word level heads, after their bins (NULL: none)
    int64_t compact_bins_bytes = 0;
    int32_t *d_status = nullptr;
    int64_t l2_bytes = 0;     // of the device's L2
    int32_t R = 0;            // observation tile actually launched (fits shared memory)
    int32_t threads = 0;
    int32_t refill = 8;
    int32_t levels = 0;       // head kind of a launch of this forest alone (TravParams::levels)
    int32_t head_smem = 0;    // bytes of one of its bin-block buffers ...
    int32_t head_plan = 0;    // ... of one with the packed blocks, which tiles are fitted beside ...
    int32_t head_shared = 0;  // ... and of one in a launch with other forests
    int32_t nbuf = 3;                          // bin-block buffers
    size_t smem_votes = 0, smem_leaves = 0, smem_values = 0;
    int32_t grid_votes = 0, grid_leaves = 0, grid_values = 0;  // resident CTAs for a persistent launch
    double cost_fixed = 0.0, cost_row = 0.0, cost_task = 0.0;  // of an item (fit_costs) ...
    double deep_levels = 0.0;                                  // of a tree's walk, below the heads (fit_costs)
    double cost_finish = 0.0;                                  // ... and, per row and thread, of a split tile's classes
    int32_t spin_limit = FP_SPIN_LIMIT;       // fault injection may lower it
    int32_t stall = 0;                        // fault injection: bin waits run out
};

namespace {

std::mutex g_pool_mu;
std::vector<int> g_pool_ready;
std::atomic<int64_t> g_fail_allocs{0};  // fault injection: device allocations still to fail ...
std::atomic<int64_t> g_pass_allocs{0};  // ... after this many that go through

// true when fault injection takes this allocation
bool injected_alloc_failure(const char *what) {
    int64_t pass = g_pass_allocs.load();
    while (pass > 0 && !g_pass_allocs.compare_exchange_weak(pass, pass - 1)) {
    }
    if (pass > 0) return false;
    int64_t k = g_fail_allocs.load();
    while (k > 0 && !g_fail_allocs.compare_exchange_weak(k, k - 1)) {
    }
    if (k <= 0) return false;
    fp_set_error("%s: injected allocation failure", what);
    return true;
}

int cuda_fail(cudaError_t e, const char *what) {
    fp_set_error("%s: %s", what, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? FP_ENOMEM : FP_ECUDA;
}

// Per-call scratch comes from the device's stream-ordered memory pool
// (cudaMallocAsync), which CUDA-graph capture turns into graph memory nodes.
// The first use on a device keeps freed blocks in the pool between calls.  A
// failed allocation is reported by the return code alone: the runtime's own
// record of it (the thread's last error) is cleared, since the caller may go
// on without scratch.  An injected failure asks the runtime for more than any
// device has, so that it leaves the state that a real one does.
int scratch_alloc(int device, void **out, size_t bytes, cudaStream_t s) {
    {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        if ((int)g_pool_ready.size() <= device) g_pool_ready.resize((size_t)device + 1, 0);
        if (!g_pool_ready[device]) {
            cudaMemPool_t pool;
            cudaError_t e = cudaDeviceGetDefaultMemPool(&pool, device);
            if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetDefaultMemPool");
            uint64_t keep = UINT64_MAX;
            e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) return cuda_fail(e, "cudaMemPoolSetAttribute");
            g_pool_ready[device] = 1;
        }
    }
    const bool injected = injected_alloc_failure("cudaMallocAsync(scratch)");
    cudaError_t e = cudaMallocAsync(out, injected ? (size_t)1 << 60 : bytes, s);
    if (injected && e == cudaSuccess) cudaFreeAsync(*out, s);  // not on any device there is
    if (injected || e != cudaSuccess) {
        cudaGetLastError();
        return injected ? FP_ENOMEM : cuda_fail(e, "cudaMallocAsync(scratch)");
    }
    return FP_OK;
}

// bytes of a slab: 32 rows of F features and C counters (none for leaf ids)
size_t slab_bytes(int F, int C, bool leaves) { return 128 * ((size_t)F + (leaves ? 0 : C)); }

// the tile's slabs + nbuf bin blocks + per-warp task rings (R is a multiple of 32)
size_t smem_bytes(int R, int F, int head_smem, int nbuf, int C, int warps, bool leaves) {
    return (size_t)(R / 32) * slab_bytes(F, C, leaves) + (size_t)nbuf * (size_t)head_smem +
           (size_t)warps * FP_RING * 8;
}

// The kernel variant for a forest and block size: its kind of super-node
// (two levels, three of format 1 or 2), and up to 768 threads run the build
// for several CTAs per SM (<= 42 registers), larger blocks the one-CTA build ...
template <int MODE, int DK, int HK>
void (*traverse_kernel_sized(const fp_device_forest *f))(TravParams) {
    return f->threads <= 768 ? fp_traverse_kernel<MODE, 2, DK, HK, false> : fp_traverse_kernel<MODE, 1, DK, HK, false>;
}

// ... and its head kind (compiled in: 0 ranked, 1 level slots, 2 paired, 3
// level slots of one word).
template <int MODE, int DK>
void (*traverse_kernel_deep(const fp_device_forest *f))(TravParams) {
    // Shallow forests: one build for every CTA size.  Its 39 to 64 registers
    // keep a second CTA of 24 warps, or a third of 16, off the SM, and the large
    // CTA is the fastest all the same (256 boosted trees, 1 M rows: 580 us with
    // 32 warps, 615 with 24, 616 to 656 with 16).
    if (f->hdr.n_super == 0) {
        switch (f->levels) {
            case 1: return fp_traverse_kernel<MODE, 1, DK, 1, true>;
            case 2: return fp_traverse_kernel<MODE, 1, DK, 2, true>;
            default: return fp_traverse_kernel<MODE, 1, DK, 0, true>;
        }
    }
    switch (f->levels) {  // level slots of one word have keys only
        case 1:
            // with keys, only where the one-word heads found no memory: one build for every CTA size
            return DK == 2 ? traverse_kernel_sized<MODE, 2, 1>(f) : fp_traverse_kernel<MODE, 1, DK == 2 ? 3 : DK, 1, false>;
        case 2: return traverse_kernel_sized<MODE, DK, 2>(f);
        case 3: return traverse_kernel_sized<MODE, DK, DK == 2 ? 0 : 3>(f);
        default: return traverse_kernel_sized<MODE, DK, 0>(f);
    }
}

// The kernel's super-node kind of a packed header: 2, 3 (format 1) or 4 (format 2).
int deep_kind(const FpImageHeader &h) { return h.deep_levels != 3 ? 2 : (h.deep_format == 2 ? 4 : 3); }

template <int MODE>
void (*traverse_kernel(const fp_device_forest *f))(TravParams) {
    switch (deep_kind(f->hdr)) {
        case 3: return traverse_kernel_deep<MODE, 3>(f);
        case 4: return traverse_kernel_deep<MODE, 4>(f);
        default: return traverse_kernel_deep<MODE, 2>(f);
    }
}

// Every instance of the batched kernel: super-node kind (0 mixed, 2, 3, 4) x
// head kind (-1 mixed, 0 ranked, 1, 2, 3; two-level forests have no one-word heads).
template <int KIND>
void add_batched(std::vector<void (*)(BatchParams)> &v) {
    v.push_back(fp_traverse_batched_kernel<KIND, -1>);
    v.push_back(fp_traverse_batched_kernel<KIND, 0>);
    v.push_back(fp_traverse_batched_kernel<KIND, 1>);
    v.push_back(fp_traverse_batched_kernel<KIND, 2>);
    v.push_back(fp_traverse_batched_kernel<KIND, KIND == 2 ? -1 : 3>);
}

const std::vector<void (*)(BatchParams)> &batched_kernels() {
    static const std::vector<void (*)(BatchParams)> v = [] {
        std::vector<void (*)(BatchParams)> k;
        add_batched<0>(k);
        add_batched<2>(k);
        add_batched<3>(k);
        add_batched<4>(k);
        return k;
    }();
    return v;
}

// The instance for a launch: index 5 * kind + (head kind + 1) into batched_kernels().
void (*batched_kernel(int kind, int hk))(BatchParams) {
    const int ki = kind >= 2 ? kind - 1 : 0;  // 0 mixed, 1 two levels, 2 format 1, 3 format 2
    return batched_kernels()[(size_t)(5 * ki + (hk + 1))];
}

// The dynamic shared-memory limit is an attribute of the kernel instance,
// which every resident forest of the same kind of super-node, head kind and
// CTA size shares: it is raised to the device's whole budget (a limit, not a
// reservation; each launch asks for its own forest's bytes), so configuring
// one forest never lowers it below another's need.  The grid comes from the
// occupancy at this forest's own bytes.
template <int MODE>
int configure(fp_device_forest *f, size_t smem, size_t budget, int32_t *grid) {
    auto kern = traverse_kernel<MODE>(f);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, f->threads, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (per_sm < 1) {
        fp_set_error("traversal kernel does not fit on an SM (%zu bytes of shared memory)", smem);
        return FP_EUNSUPPORTED;
    }
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, f->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    *grid = per_sm * sms;
    return FP_OK;
}

// Fit the observation tile to shared memory and size the persistent grid.
int launch_setup(fp_device_forest *f, int32_t tile, int32_t warps, int32_t refill, int32_t nbuf) {
    if (tile < 32 || tile > 2048 || tile % 32 || warps < 1 || warps > 32 || refill < 1 || refill > 32 ||
        (nbuf != 2 && nbuf != 3)) {
        fp_set_error("launch parameters out of range (obs_tile %d, warps %d, refill %d, bin_buffers %d)", tile, warps,
                     refill, nbuf);
        return FP_EINVAL;
    }
    int max_optin = 0;
    cudaError_t e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, f->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    const size_t budget = (size_t)max_optin - 256;  // leaves room for the static shared variables
    const int C = f->hdr.n_classes, F = f->hdr.n_features;
    int R = tile;
    while (R > 32 && smem_bytes(R, F, f->head_plan, nbuf, C, warps, false) > budget) R -= 32;
    if (smem_bytes(R, F, f->head_plan, nbuf, C, warps, false) > budget) {
        fp_set_error("a 32-row tile, the bin-block buffers and the task rings need %zu bytes of shared memory (limit %zu)",
                     smem_bytes(R, F, f->head_plan, nbuf, C, warps, false), budget);
        return FP_EUNSUPPORTED;
    }
    fp_device_forest g = *f;
    g.R = R;
    g.threads = 32 * warps;
    g.refill = refill;
    g.nbuf = nbuf;
    g.smem_votes = smem_bytes(R, F, f->head_smem, nbuf, C, warps, false);
    g.smem_leaves = smem_bytes(R, F, f->head_smem, nbuf, C, warps, true);
    int rc = configure<FP_MODE_VOTES>(&g, g.smem_votes, budget, &g.grid_votes);
    if (rc) return rc;
    rc = configure<FP_MODE_LEAVES>(&g, g.smem_leaves, budget, &g.grid_leaves);
    if (rc) return rc;
    if (f->hdr.n_values > 0) {  // one float per row instead of the class votes
        g.smem_values = smem_bytes(R, F, f->head_smem, nbuf, 1, warps, false);
        rc = configure<FP_MODE_VALUES>(&g, g.smem_values, budget, &g.grid_values);
        if (rc) return rc;
    }
    // the batched kernels may host any resident forest: allow them all of shared memory
    for (auto kern : batched_kernels()) {
        cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget);
        if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFuncSetAttribute(batched)");
    }
    f->R = g.R;
    f->threads = g.threads;
    f->refill = g.refill;
    f->nbuf = g.nbuf;
    f->smem_votes = g.smem_votes;
    f->smem_leaves = g.smem_leaves;
    f->grid_votes = g.grid_votes;
    f->grid_leaves = g.grid_leaves;
    f->smem_values = g.smem_values;
    f->grid_values = g.grid_values;
    return FP_OK;
}

// ------------------------------------------------------- shape of a launch
//
// A batch is cut into tiles of R rows, and a tile's bins into S splits.  Large
// batches fill the GPU with tiles (S = 1: a CTA sweeps the whole forest for
// its tile, the CTAs walking the same bins at about the same time, so that L2
// serves them; 256 trees of 208 MB of super-nodes, 4 M rows: 24.8 ms, 25.4 ms
// when swept pass by pass, for the rows staged and the votes added once per
// pass).  A batch too small for that leaves SMs idle, or its last wave nearly
// empty, unless the bins are split as well; the splits of a tile then add up
// in global memory (scratch, a memset, and the last CTA's second look at the
// tile: 3 to 4 us), where a 32-row request on 64 trees had one CTA walk 22
// bins one after another.
// A batch of a few waves is cut in two: the rows that fill whole waves of the
// largest tile, and the rest in the shape that is best for it.

struct Shape {
    int32_t R = 32, S = 1;
    double cost = 1e300;  // estimated nanoseconds
};

struct Part {
    int64_t row0 = 0, n = 0;
    Shape shape;
};

// Estimated time of one item, in nanoseconds, fitted to launches of one wave
// over forests of 16 to 256 trees, tiles of 32 to 864 rows and 1 to 86 bins
// (within 20 % for most; only the ratios matter):
//   - what it takes before and after its walks: the first rows and blocks from
//     memory, and the longest walks' last steps, one L2 latency each (19 us for
//     one bin of the 256-tree forest, 29 us for one of 784-feature trees, whose
//     heads are 4 levels);
//   - its rows through one SM's loads;
//   - its bins: 0.8 us in which the warps take their turn at a block, and its
//     tasks, 0.06 ns per level in the head and 0.21 ns per level below it;
//   - the classes of a tile whose bins are split: the last CTA reads the votes
//     of its rows anew, up to 32 lanes to a row, and every pass of its threads
//     over them waits for L2, 1.1 us.  Without this term 9000 rows of a forest
//     of 50 classes were split, 384 rows a tile: 68 us, 56 unsplit.
void fit_costs(fp_device_forest *f) {
    const FpImageHeader &h = f->hdr;
    double levels = 1.0;  // of a tree's walk
    for (int64_t m = h.n_internal / std::max<int32_t>(1, h.n_trees); m > 1; m >>= 1) levels += 1.4;
    const double head = std::min(levels, h.depth + 1.0), deep = h.n_super ? levels - head : 0.0;
    f->deep_levels = deep;
    f->cost_fixed = 4000.0 + 1000.0 * deep;
    f->cost_row = 0.08 * h.n_features;
    f->cost_task = h.n_super ? 0.3 + 0.06 * head + 0.21 * deep : 0.06 * head;
    int lanes = 1;
    while (lanes < h.n_classes && lanes < 32) lanes *= 2;
    f->cost_finish = h.n_values > 0 ? 0.0 : 1100.0 * lanes;
}

double item_cost(const fp_device_forest *f, int64_t R, int64_t bins) {
    return f->cost_fixed + f->cost_row * (double)R +
           (double)bins * (800.0 + f->cost_task * (double)R * f->hdr.bin_size);
}

// The best shape for n rows, fewer than a few waves' worth: in one split if
// `whole` allows it, in several (up to one per bin) if `split` does.  `extra`:
// what splitting costs the GPU besides, where the splits add up in scratch.
// The allocation, the memset and their place between kernels add 3 to 6 us to
// small calls that follow one another, so as much has to be saved as well, and
// 15 % of the estimate at least (256 shallow trees, 1000 rows: 21 us a call
// split, 17.5 unsplit).
Shape best_shape(const fp_device_forest *f, int64_t n, int32_t slots, bool whole, bool split, double extra) {
    const int32_t nb = f->hdr.n_bins;
    Shape best;
    auto try_splits = [&](int64_t S) {
        const int64_t room = slots / S;  // tiles at a time
        for (int64_t w = 1; w <= 4 && room > 0; ++w) {
            const int64_t fit = ((n + w * room - 1) / (w * room) + 31) / 32 * 32;
            const int64_t R = std::min<int64_t>(f->R, std::max<int64_t>(32, fit));
            const int64_t tiles = (n + R - 1) / R, turns = (tiles + room - 1) / room;
            // a slab of few rows is walked by as many warp steps in the heads, fewer below them
            const int64_t filled = n < R ? (n + R) / 2 : R;
            double c = (double)turns * item_cost(f, filled, (nb + S - 1) / S);
            if (S > 1 && extra > 0.0) c += extra + f->cost_finish * (double)R / f->threads;
            if (c < best.cost) {
                best.R = (int32_t)R;
                best.S = (int32_t)S;
                best.cost = c;
            }
            if (R == 32) break;
        }
    };
    if (whole) try_splits(1);
    const Shape unsplit = best;
    if (split) {
        for (int64_t S = 2; S < nb && S <= slots; S += 1 + S / 6) try_splits(S);
        if (nb > 1) try_splits(nb);
    }
    if (whole && extra > 0.0 && best.cost > std::min(0.85 * unsplit.cost, unsplit.cost - 6000.0)) return unsplit;
    return best;
}

// How n rows are launched: in one or two parts (returns how many).  split: a
// forest of one pass may have its bins split, which takes scratch (leaf ids
// take none).
int plan_rows(const fp_device_forest *f, int64_t n, int32_t grid, bool split, bool leaves, Part out[2]) {
    const FpImageHeader &h = f->hdr;
    const int64_t wave = (int64_t)grid * f->R;  // rows of a full wave of the largest tiles
    const bool passes = h.n_passes > 1;
    // A forest beyond L2 whose tiles are too small to use a bin's lines before
    // the next bin's evict them is swept pass by pass, all tiles of a pass
    // before the next pass.  256 trees of 208 MB, 400,000 rows: 11.1 ms by
    // passes, 12.3 in one sweep with 32-row tiles (167 bytes of the forest per
    // task of a wave), 6.22 and 6.45 with 64 rows (83 bytes), 4.10 and 3.87
    // with 128; in two to four waves (20,000 rows) one sweep is the faster.
    const int64_t deep = 32 * (int64_t)h.n_super;
    if (passes && deep > f->l2_bytes / 4 * 3 && deep > 64 * wave * h.n_trees && n >= 8 * wave) {
        const int64_t want = (n * h.n_passes + grid - 1) / grid;
        out[0].row0 = 0;
        out[0].n = n;
        out[0].shape = Shape();
        out[0].shape.R = (int32_t)std::min<int64_t>(f->R, std::max<int64_t>(32, (want + 31) / 32 * 32));
        out[0].shape.S = h.n_passes;
        return 1;
    }
    auto small = [&](int64_t m) {  // the best shape for less than a few waves
        if (leaves) return best_shape(f, m, grid, true, true, 0.0);
        // a forest of several passes has bins enough to split: it is kept
        // whole only for rows that fill the GPU with two slabs per CTA
        if (passes) return best_shape(f, m, grid, m >= 64 * (int64_t)grid, true, 4000.0);
        return best_shape(f, m, grid, true, split, 4000.0);
    };
    const int64_t full = n / wave;
    if (full == 0) {
        out[0].row0 = 0;
        out[0].n = n;
        out[0].shape = small(n);
        return 1;
    }
    // whole waves only, in tiles as even as 32-row steps allow ...
    const int64_t waves = (n + wave - 1) / wave;
    Shape even;
    even.R = (int32_t)std::min<int64_t>(f->R, ((n + waves * grid - 1) / (waves * grid) + 31) / 32 * 32);
    even.cost = (double)(((n + even.R - 1) / even.R + grid - 1) / grid) * item_cost(f, even.R, h.n_bins);
    out[0].row0 = 0;
    out[0].n = n;
    out[0].shape = even;
    const int64_t rest = n - full * wave;
    if (rest == 0) return 1;
    // ... or full waves and the rest apart
    const Shape tail = small(rest);
    if ((double)full * item_cost(f, f->R, h.n_bins) + tail.cost + 8000.0 >= even.cost) return 1;
    out[0].n = full * wave;
    out[0].shape.R = f->R;
    out[1].row0 = full * wave;
    out[1].n = rest;
    out[1].shape = tail;
    return 2;
}

// levels: the head kind that the launch walks this forest with.
TravParams base_params(const fp_device_forest *f, const float *X, int64_t n, int32_t levels) {
    TravParams p;
    memset(&p, 0, sizeof p);
    const FpImageHeader &h = f->hdr;
    p.deep = reinterpret_cast<const FpSuper *>(f->d_image + h.off_deep);
    p.heads = f->d_image + h.off_heads;
    p.bins = reinterpret_cast<const FpBin *>(f->d_image + h.off_bins);
    p.passes = reinterpret_cast<const FpPass *>(f->d_image + h.off_passes);
    p.pheads = reinterpret_cast<const int32_t *>(f->d_image + h.off_pheads);
    p.deep_leaf = reinterpret_cast<const int32_t *>(f->d_image + h.off_deep_leaf);
    p.X = X;
    p.n = n;
    p.F = h.n_features;
    p.C = h.n_classes;
    p.T = h.n_trees;
    p.R = f->R;
    p.slab = (uint32_t)slab_bytes(h.n_features, h.n_classes, false);  // other modes set their own
    p.n_tiles = (n + p.R - 1) / p.R;
    p.n_items = p.n_tiles;
    p.n_splits = 1;
    p.n_passes = h.n_passes;
    p.n_bins = h.n_bins;
    p.split_bins = h.n_bins;
    p.head_smem = levels == f->levels ? f->head_smem : f->head_shared;
    p.nbuf = f->nbuf;
    p.levels = levels;
    if (levels == 3) {
        p.packed_kind = h.head_select;
        p.packed_heads = p.heads;
        p.packed_bins = p.bins;
        p.bins = reinterpret_cast<const FpBin *>(f->d_compact);
        p.heads = f->d_compact + f->compact_bins_bytes;
    }
    p.leaf_val = reinterpret_cast<const float *>(f->d_image + h.off_values);
    p.n_vals = (uint32_t)h.n_values;
    p.depth = h.depth;
    p.refill = f->refill;
    p.step_bins = f->deep_levels >= 10.0;  // measured on both sides: 8 levels lose 12 %, 13 gain 15 %
    p.status = f->d_status;
    p.spin_limit = f->spin_limit;
    p.stall = f->stall;
    p.n_super = (uint32_t)h.n_super;
    p.deep_kind = deep_kind(h);
    if (p.deep_kind >= 3) {
        const uint32_t fb = (uint32_t)h.feature_bits, cb = (uint32_t)h.class_bits;
        p.cshl = (p.deep_kind == 4 ? 1 : 2) * fb;
        p.cshr = p.cshl + cb;
        p.tie = 1u << (p.cshr + cb);
        p.frot = (fb + 25u) & 31u;  // right by fb - 7
        p.fmask = (1u << fb) - 1u;
        p.cmask = (1u << cb) - 1u;
        p.klo = h.key_lo;
        p.khi = h.key_hi;
        p.kshl = h.key_shl;
        p.kflag = h.key_flag;
        p.kga = h.key_gap_a;
        p.kgb = h.key_gap_b;
        p.kgd = h.key_gap_d;
        p.vbase3 = (uint32_t)h.values3_base;
        p.deep_keys = reinterpret_cast<const uint32_t *>(f->d_image + h.off_deep_keys);
    }
    return p;
}

void set_shape(TravParams &p, const Shape &sh) {
    p.R = sh.R;
    p.n_tiles = (p.n + sh.R - 1) / sh.R;
    p.n_splits = sh.S;
    p.n_items = p.n_tiles * sh.S;
    p.split_bins = p.n_bins / sh.S;
    p.split_more = p.n_bins % sh.S;
}

// A kernel launch that returns its own result: the thread's last error, which
// is all that <<<>>> leaves, may be that of an earlier call.
template <class Params>
cudaError_t launch(void (*kern)(Params), int64_t ctas, int threads, size_t smem, cudaStream_t s, const Params &p) {
    void *args[] = {const_cast<Params *>(&p)};
    return cudaLaunchKernel(reinterpret_cast<const void *>(kern), dim3((unsigned)ctas), dim3((unsigned)threads), args,
                            smem, s);
}

// Launch one part of a call, shaped by set_shape.
template <int MODE>
cudaError_t launch_part(const fp_device_forest *f, const TravParams &p, int32_t grid, size_t smem, cudaStream_t s) {
    return launch(traverse_kernel<MODE>(f), std::min<int64_t>(p.n_items, grid), f->threads, smem, s, p);
}

// Whether a call on this stream may take scratch that it would not need
// otherwise: while the stream is captured it becomes a memory node, which
// limits what can be done with the graph.
bool may_split(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) == cudaSuccess) return st == cudaStreamCaptureStatusNone;
    cudaGetLastError();  // the call goes on: without scratch
    return false;
}

// plan_rows for a call that takes scratch where bins of a forest of one pass
// are split.  The stream is asked only then: most calls split nothing (a call
// of 32 rows of 16 trees takes the host 2.22 us, 2.34 when it asks, and 4.7
// where bins are split).
int plan_call(const fp_device_forest *f, int64_t n, int32_t grid, cudaStream_t s, Part out[2]) {
    int k = plan_rows(f, n, grid, true, false, out);
    if (f->hdr.n_passes == 1 && out[k - 1].shape.S > 1 && !may_split(s)) k = plan_rows(f, n, grid, false, false, out);
    return k;
}

// Scratch of a part whose splits add up in global memory: acc_per_row bytes of
// accumulator per row, then a counter per tile.
size_t scratch_bytes(const Part &pt, int64_t acc_per_row, size_t *acc_bytes) {
    *acc_bytes = 0;
    if (pt.shape.S == 1) return 0;
    *acc_bytes = ((size_t)pt.n * acc_per_row + 255) & ~(size_t)255;
    return *acc_bytes + (size_t)((pt.n + pt.shape.R - 1) / pt.shape.R) * 4;
}

int check_device(const fp_device_forest *f) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev != f->device) {
        fp_set_error("forest lives on device %d but device %d is current", f->device, dev);
        return FP_EINVAL;
    }
    return FP_OK;
}

}  // namespace

// The one-word level heads of an uploaded forest (fp_compact_heads_kernel) and
// their bins; the forest then walks those.  Waits for the stream.  FP_ENOMEM
// leaves the forest with its packed heads, which serve every launch.
static int compact_heads(fp_device_forest *f, cudaStream_t s) {
    const FpImageHeader &h = f->hdr;
    std::vector<FpBin> bins;
    try {
        bins = f->bins;
    } catch (const std::bad_alloc &) {
        return FP_ENOMEM;
    }
    const int32_t nodes = (1 << (h.depth + 1)) - 1;
    int64_t off = 0;
    int32_t largest = 0;
    for (FpBin &b : bins) {
        b.nranks = nodes;
        b.head_bytes = (uint32_t)(((int64_t)(nodes + b.nexits) * b.stride * 4 + 15) & ~(int64_t)15);
        b.head_off = (uint32_t)off;  // below the packed block's, which fits
        off += b.head_bytes;
        largest = std::max<int32_t>(largest, (int32_t)b.head_bytes);
    }
    f->compact_bins_bytes = ((int64_t)(bins.size() * sizeof(FpBin)) + 255) & ~(int64_t)255;
    cudaError_t e = cudaErrorMemoryAllocation;
    if (!injected_alloc_failure("cudaMalloc(heads)"))
        e = cudaMalloc(&f->d_compact, (size_t)(f->compact_bins_bytes + off));
    if (e != cudaSuccess) {
        f->d_compact = nullptr;
        cudaGetLastError();
        return cuda_fail(e, "cudaMalloc(heads)");
    }
    e = cudaMemcpyAsync(f->d_compact, bins.data(), bins.size() * sizeof(FpBin), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(heads)");
    fp_compact_heads_kernel<<<(unsigned)bins.size(), 256, 0, s>>>(
        f->d_compact + f->compact_bins_bytes, reinterpret_cast<const FpBin *>(f->d_compact),
        f->d_image + h.off_heads, reinterpret_cast<const FpBin *>(f->d_image + h.off_bins), h.head_select,
        (1u << h.feature_bits) - 1u);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // before the host's bins go
    if (e != cudaSuccess) return cuda_fail(e, "fp_compact_heads_kernel");
    f->head_shared = largest;
    // Alone, paired heads of at most four levels are walked as packed: their
    // records are few enough for a warp to read most of them without bank
    // conflicts (784-feature rows, heads 0..3, 250,000 rows: 1482 us, 1494 us
    // with one-word slots).
    if (f->levels == 1 || h.depth > 3) {
        f->levels = 3;
        f->head_smem = largest;
    }
    return FP_OK;
}

extern "C" int fp_upload(const fp_packed_forest *pf, void *stream, fp_device_forest **out) {
    if (!out || !pf) {
        fp_set_error("fp_upload: NULL argument");
        return FP_EINVAL;
    }
    *out = nullptr;
    fp_device_forest *f = new (std::nothrow) fp_device_forest;
    if (!f) {
        fp_set_error("fp_upload: out of host memory");
        return FP_ENOMEM;
    }
    const FpImageHeader *h = fp_packed_header(pf);
    f->hdr = *h;
    const uint8_t *img = fp_packed_bytes(pf);
    f->bins.assign(reinterpret_cast<const FpBin *>(img + h->off_bins),
                   reinterpret_cast<const FpBin *>(img + h->off_bins) + h->n_bins);
    f->passes.assign(reinterpret_cast<const FpPass *>(img + h->off_passes),
                     reinterpret_cast<const FpPass *>(img + h->off_passes) + h->n_passes);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int rc = FP_OK, l2 = 0;
    cudaError_t e = cudaGetDevice(&f->device);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaGetDevice"); goto fail; }
    e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, f->device);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaDeviceGetAttribute"); goto fail; }
    f->l2_bytes = l2;
    if (injected_alloc_failure("cudaMalloc(image)")) { rc = FP_ENOMEM; goto fail; }
    e = cudaMalloc(&f->d_image, (size_t)h->total_bytes);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMalloc(image)"); goto fail; }
    e = cudaMalloc(&f->d_status, 256);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMalloc(status)"); goto fail; }
    e = cudaMemsetAsync(f->d_status, 0, 256, s);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMemsetAsync"); goto fail; }
    e = cudaMemcpyAsync(f->d_image, img, (size_t)h->total_bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaMemcpyAsync(image)"); goto fail; }
    if (h->n_values > 0 && h->n_super == 0) {
        fp_inline_values_kernel<<<(unsigned)h->n_bins, 256, 0, s>>>(
            f->d_image + h->off_heads, reinterpret_cast<const FpBin *>(f->d_image + h->off_bins),
            reinterpret_cast<const float *>(f->d_image + h->off_values), (uint32_t)h->n_values,
            h->head_select == 2 ? 16u : 8u);
        e = cudaGetLastError();
        if (e != cudaSuccess) { rc = cuda_fail(e, "fp_inline_values_kernel launch"); goto fail; }
    }
    e = cudaStreamSynchronize(s);  // the caller may free the host image on return
    if (e != cudaSuccess) { rc = cuda_fail(e, "cudaStreamSynchronize"); goto fail; }
    f->head_smem = f->head_plan = f->head_shared = (h->max_head_bytes + 15) & ~15;
    f->levels = h->head_select == 3 ? 0 : h->head_select;
    fit_costs(f);
    if (h->n_super > 0 && deep_kind(*h) >= 3 && f->levels != 0) {
        rc = compact_heads(f, s);
        if (rc && rc != FP_ENOMEM) goto fail;
    }
    rc = launch_setup(f, h->obs_tile, h->warps_per_cta, h->refill_lanes, h->bin_buffers);
    if (rc) goto fail;
    *out = f;
    return FP_OK;
fail:
    if (f->d_compact) cudaFree(f->d_compact);
    if (f->d_image) cudaFree(f->d_image);
    if (f->d_status) cudaFree(f->d_status);
    delete f;
    return rc;
}

extern "C" int fp_configure(fp_device_forest *f, const fp_pack_params *params) {
    if (!f || !params) {
        fp_set_error("fp_configure: NULL argument");
        return FP_EINVAL;
    }
    const FpImageHeader &h = f->hdr;
    if ((params->bin_size && params->bin_size != h.bin_size) ||
        (params->interleave_depth > 0 && params->interleave_depth != h.depth) ||
        (params->pass_bytes && params->pass_bytes != h.pass_bytes)) {
        fp_set_error("fp_configure: layout parameters can only change by packing again");
        return FP_EINVAL;
    }
    int rc = check_device(f);
    if (rc) return rc;
    return launch_setup(f, params->obs_tile ? params->obs_tile : f->R,
                        params->warps_per_cta ? params->warps_per_cta : f->threads / 32,
                        params->refill_lanes ? params->refill_lanes : f->refill,
                        params->bin_buffers ? params->bin_buffers : f->nbuf);
}

namespace {

// fp_predict and fp_predict_noalloc: scratch_for(bytes, &ptr) supplies the
// scratch of a part, release(ptr) takes it back.  A part that gets none runs
// unsplit where the forest has one pass, or where `whole` says so (then a
// forest of one pass is not split at all).  Votes
// without classes take no scratch: the splits add up in the caller's votes and
// nothing is left to do after the last of them.  So such calls cannot fail for
// memory, put no memory node into a captured graph, and overlap freely when
// they are fp_predict_noalloc's.
template <class Scratch, class Release>
int predict_votes(const fp_device_forest *f, const float *X, int64_t n, uint32_t *out_votes, int32_t *out_class,
                  cudaStream_t s, bool whole, Scratch scratch_for, Release release) {
    const FpImageHeader &h = f->hdr;
    Part parts[2];
    const int k = whole || !out_class ? plan_rows(f, n, f->grid_votes, !whole, false, parts)
                                      : plan_call(f, n, f->grid_votes, s, parts);
    for (int i = 0; i < k; ++i) {
        Part &pt = parts[i];
        uint32_t *const votes = out_votes ? out_votes + pt.row0 * h.n_classes : nullptr;
        // the splits add up in scratch, or, where that would be large, in the
        // caller's votes (a second memset)
        const int64_t vote_bytes = 4 * (int64_t)h.n_classes;
        const bool votes_alone = !out_class;
        const bool in_votes = votes_alone || (votes && pt.n * vote_bytes > (4 << 20));
        size_t acc_bytes = 0;
        const size_t bytes = votes_alone ? 0 : scratch_bytes(pt, in_votes ? 0 : vote_bytes, &acc_bytes);
        void *scratch = nullptr;
        if (bytes) {
            const int rc = scratch_for(bytes, &scratch);
            if (rc && h.n_passes > 1 && !whole) return rc;
            if (rc) pt.shape.S = 1;  // the same rows without scratch
        }
        TravParams p = base_params(f, X + pt.row0 * h.n_features, pt.n, f->levels);
        set_shape(p, pt.shape);
        p.out_votes = votes;
        p.out_class = out_class ? out_class + pt.row0 : nullptr;
        cudaError_t e = cudaSuccess;
        if (p.n_splits > 1) {
            uint8_t *sc = static_cast<uint8_t *>(scratch);
            p.acc = in_votes ? votes : reinterpret_cast<uint32_t *>(sc);
            p.tile_done = votes_alone ? nullptr : reinterpret_cast<uint32_t *>(sc + acc_bytes);
            if (bytes) e = cudaMemsetAsync(scratch, 0, bytes, s);
            if (e == cudaSuccess && in_votes) e = cudaMemsetAsync(votes, 0, (size_t)(pt.n * vote_bytes), s);
        }
        if (e == cudaSuccess) e = launch_part<FP_MODE_VOTES>(f, p, f->grid_votes, f->smem_votes, s);
        if (scratch) release(scratch);
        if (e != cudaSuccess) return cuda_fail(e, "fp_traverse_kernel launch");
    }
    return FP_OK;
}

}  // namespace

extern "C" int fp_predict(const fp_device_forest *f, const float *X, int64_t n, uint32_t *out_votes,
                          int32_t *out_class, void *stream) {
    if (!f || n < 0 || (n > 0 && !X)) {
        fp_set_error("fp_predict: bad arguments");
        return FP_EINVAL;
    }
    if (f->hdr.n_values > 0) {
        fp_set_error("fp_predict: the forest has leaf values; use fp_predict_values");
        return FP_EINVAL;
    }
    if (n == 0 || (!out_votes && !out_class)) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return predict_votes(
        f, X, n, out_votes, out_class, s, false,
        [&](size_t bytes, void **out) { return scratch_alloc(f->device, out, bytes, s); },
        [&](void *ptr) { cudaFreeAsync(ptr, s); });
}

extern "C" int fp_predict_values(const fp_device_forest *f, const float *X, int64_t n, float scale, float bias,
                                 float *out, void *stream) {
    if (!f || n < 0 || (n > 0 && (!X || !out))) {
        fp_set_error("fp_predict_values: bad arguments");
        return FP_EINVAL;
    }
    if (f->hdr.n_values <= 0) {
        fp_set_error("fp_predict_values: the forest was packed without leaf values");
        return FP_EINVAL;
    }
    if (n == 0) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const FpImageHeader &h = f->hdr;
    Part parts[2];
    const int k = plan_call(f, n, f->grid_values, s, parts);
    for (int i = 0; i < k; ++i) {
        Part &pt = parts[i];
        size_t acc_bytes;  // a float accumulator per row, a counter per tile
        const size_t bytes = scratch_bytes(pt, 4, &acc_bytes);
        void *scratch = nullptr;
        if (bytes) {
            rc = scratch_alloc(f->device, &scratch, bytes, s);
            if (rc && h.n_passes > 1) return rc;
            if (rc) pt.shape.S = 1;  // the same rows without scratch
        }
        TravParams p = base_params(f, X + pt.row0 * h.n_features, pt.n, f->levels);
        set_shape(p, pt.shape);
        p.slab = (uint32_t)slab_bytes(h.n_features, 1, false);
        p.vscale = scale;
        p.vbias = bias;
        p.out_val = out + pt.row0;
        cudaError_t e = cudaSuccess;
        if (p.n_splits > 1) {
            e = cudaMemsetAsync(scratch, 0, bytes, s);
            p.acc_val = static_cast<float *>(scratch);
            p.tile_done = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(scratch) + acc_bytes);
        }
        if (e == cudaSuccess) e = launch_part<FP_MODE_VALUES>(f, p, f->grid_values, f->smem_values, s);
        if (scratch) cudaFreeAsync(scratch, s);
        if (e != cudaSuccess) return cuda_fail(e, "fp_traverse_kernel<values> launch");
    }
    return FP_OK;
}

// ---------------------------------------------------------------------------
// fp_predict_noalloc: fp_predict for callers that must not allocate device
// memory.  The scratch of a forest of several passes whose bins are split and
// whose classes are asked for (one counter per observation tile, and a vote
// accumulator unless the votes add up in a buffer of the caller's of more than
// 4 MiB) lives in this fixed array instead of the stream-ordered pool.  Every GPU that loads the library holds the array
// until the process exits.
#define FP_NOALLOC_SCRATCH_BYTES (16u << 20)
static __device__ __align__(256) unsigned char fp_noalloc_scratch[FP_NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_noalloc_mu;
std::vector<void *> g_noalloc_ptr;  // device address of the array, per device (set up once)

// Host code cannot use the array's name as a device address: look the
// address up once per device, with that device current.
int noalloc_scratch(int device, void **out) {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if ((int)g_noalloc_ptr.size() <= device) g_noalloc_ptr.resize((size_t)device + 1, nullptr);
    if (!g_noalloc_ptr[device]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, fp_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(fp_noalloc_scratch)");
        g_noalloc_ptr[device] = ptr;
    }
    *out = g_noalloc_ptr[device];
    return FP_OK;
}
}  // namespace

extern "C" int fp_predict_noalloc(const fp_device_forest *f, const float *X, int64_t n, uint32_t *out_votes,
                                  int32_t *out_class, void *stream) {
    if (!f || n < 0 || (n > 0 && !X)) {
        fp_set_error("fp_predict_noalloc: bad arguments");
        return FP_EINVAL;
    }
    if (f->hdr.n_values > 0) {
        fp_set_error("fp_predict_noalloc: the forest has leaf values; use fp_predict_values");
        return FP_EINVAL;
    }
    if (n == 0 || (!out_votes && !out_class)) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const FpImageHeader &h = f->hdr;
    if (h.n_passes > 1) {
        // the documented limit: a vote accumulator and tile counters for the
        // whole batch, with tiles small enough that every pass fills the GPU
        const int64_t grid = std::max<int64_t>(1, f->grid_votes), want = (n * h.n_passes + grid - 1) / grid;
        const int64_t R = std::min<int64_t>(f->R, std::max<int64_t>(32, (want + 31) / 32 * 32));
        const size_t vote_bytes = out_votes ? 0 : (size_t)n * h.n_classes * 4;
        const size_t cnt_bytes = out_class ? (size_t)((n + R - 1) / R) * 4 : 0;
        const size_t bytes = ((vote_bytes + 255) & ~(size_t)255) + cnt_bytes;
        if (bytes > FP_NOALLOC_SCRATCH_BYTES) {
            fp_set_error("fp_predict_noalloc: %lld rows need %zu bytes of scratch, more than the fixed %u; pass "
                         "out_votes, split the batch, or use fp_predict",
                         (long long)n, bytes, FP_NOALLOC_SCRATCH_BYTES);
            return FP_EINVAL;
        }
        void *scratch;  // the address is looked up whether this call needs the array or not
        rc = noalloc_scratch(f->device, &scratch);
        if (rc) return rc;
    }
    return predict_votes(
        f, X, n, out_votes, out_class, s, true,
        [&](size_t bytes, void **out) {
            if (bytes > FP_NOALLOC_SCRATCH_BYTES) {
                fp_set_error("fp_predict_noalloc: %zu bytes of scratch, more than the fixed %u", bytes,
                             FP_NOALLOC_SCRATCH_BYTES);
                return FP_EINVAL;
            }
            return noalloc_scratch(f->device, out);
        },
        [](void *) {});
}

extern "C" int fp_predict_leaves(const fp_device_forest *f, const float *X, int64_t n, int32_t *out_leaf,
                                 void *stream) {
    if (!f || n < 0 || (n > 0 && (!X || !out_leaf))) {
        fp_set_error("fp_predict_leaves: bad arguments");
        return FP_EINVAL;
    }
    if (n == 0) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    Part parts[2];
    const int k = plan_rows(f, n, f->grid_leaves, false, true, parts);
    for (int i = 0; i < k; ++i) {
        const Part &pt = parts[i];
        TravParams p = base_params(f, X + pt.row0 * f->hdr.n_features, pt.n, f->levels);
        set_shape(p, pt.shape);
        p.slab = (uint32_t)slab_bytes(f->hdr.n_features, 0, true);
        p.out_leaf = out_leaf + pt.row0 * f->hdr.n_trees;
        cudaError_t e = launch_part<FP_MODE_LEAVES>(f, p, f->grid_leaves, f->smem_leaves, s);
        if (e != cudaSuccess) return cuda_fail(e, "fp_traverse_kernel<leaves> launch");
    }
    return FP_OK;
}

extern "C" int fp_sync_status(const fp_device_forest *f, void *stream) {
    if (!f) {
        fp_set_error("fp_sync_status: NULL forest");
        return FP_EINVAL;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    int32_t word = 0;
    e = cudaMemcpy(&word, f->d_status, 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(status)");
    if (word != 0) {
        e = cudaMemset(f->d_status, 0, 4);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemset(status)");
        fp_set_error("a kernel reported status %d", word);
        return word < 0 ? word : FP_EDEVICE;
    }
    return FP_OK;
}

extern "C" int fp_inject_fault(fp_device_forest *f, int32_t kind, int64_t value) {
    switch (kind) {
    case FP_FAULT_ALLOC:
        if (value < 0) break;
        g_fail_allocs.store(value);
        if (value == 0) g_pass_allocs.store(0);
        return FP_OK;
    case FP_FAULT_ALLOC_AFTER:
        if (value < 0) break;
        g_pass_allocs.store(value);
        return FP_OK;
    case FP_FAULT_WAIT_LIMIT:
        if (!f || value < 1 || value > FP_SPIN_LIMIT) break;
        f->spin_limit = (int32_t)value;
        return FP_OK;
    case FP_FAULT_STALL_BIN_COPY:
        if (!f || (value != 0 && value != 1)) break;
        f->stall = (int32_t)value;
        return FP_OK;
    default:
        break;
    }
    fp_set_error("fp_inject_fault: bad kind %d, value %lld or forest", kind, (long long)value);
    return FP_EINVAL;
}

extern "C" int fp_device_info_get(const fp_device_forest *f, fp_packed_info *info) {
    if (!f || !info) {
        fp_set_error("fp_device_info_get: NULL argument");
        return FP_EINVAL;
    }
    fp_fill_info(&f->hdr, info);
    info->obs_tile = f->R;
    info->warps_per_cta = f->threads / 32;
    info->refill_lanes = f->refill;
    info->bin_buffers = f->nbuf;
    return FP_OK;
}

extern "C" void fp_release(fp_device_forest *f) {
    if (!f) return;
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != f->device) cudaSetDevice(f->device);
    cudaDeviceSynchronize();
    cudaFree(f->d_compact);
    cudaFree(f->d_image);
    cudaFree(f->d_status);
    if (prev >= 0 && prev != f->device) cudaSetDevice(prev);
    delete f;
}

// One batch of a launch of several: the numbers of splits that it may be cut
// into, with what the estimates need of each.  Formed once per call, since the
// search below asks for a shape for every length of item: with the estimates
// formed anew each time, 32 batches of a few rows kept the host planning for
// as long as the launch itself takes.
struct BatchCuts {
    struct Cut {
        int64_t S;
        double fixed, per_row, inv_row, more;  // an item's time without rows, per row, and for adding its votes up
        double top_item, top_cost;             // of one item of the largest tile, and of all of them with `more`
        int32_t best_top;                      // the least top_cost from this cut on
    };
    int64_t n = 0, top = 32;  // rows; the largest tile
    double least = 0.0;       // the shortest item there can be
    int32_t count = 0;
    Cut cut[40];

    void form(const fp_device_forest *f, int64_t rows, int32_t max_R) {
        const uint32_t nb = (uint32_t)f->hdr.n_bins;
        n = rows;
        top = std::min<int64_t>(max_R, (n + 31) / 32 * 32);
        const int64_t tiles = n <= top ? 1 : (n + top - 1) / top;
        for (uint32_t S = 1; count < 40; S = std::min(nb, S + 1 + S / 2)) {
            const uint32_t bins = (nb + S - 1) / S;
            Cut &c = cut[count++];
            c.S = S;
            c.fixed = item_cost(f, 0, bins);
            c.per_row = item_cost(f, 1, bins) - c.fixed;
            c.inv_row = 1.0 / c.per_row;
            c.more = S > 1 ? 1000.0 : 0.0;
            c.top_item = c.fixed + c.per_row * (double)top;
            c.top_cost = (double)(tiles * S) * (c.top_item + c.more);
            least = c.fixed + c.per_row * 32.0;
            if (S == nb) break;
        }
        for (int32_t i = count - 1; i >= 0; --i)
            cut[i].best_top = i + 1 < count && cut[cut[i + 1].best_top].top_cost < cut[i].top_cost ? cut[i + 1].best_top : i;
    }

    // The shape when no item is to take longer than `most` nanoseconds: the
    // splits whose items (as large as `most` lets them be) take the least time
    // together.  *item: the time of one, *items: how many there are.
    Shape within(double most, double *item, double *items) const {
        Shape best;
        auto take = [&](const Cut &c, int64_t R, double one, double cost) {
            if (cost >= best.cost) return;
            best.R = (int32_t)R;
            best.S = (int32_t)c.S;
            best.cost = cost;
            *item = one;
        };
        for (int32_t i = 0; i < count; ++i) {
            if (i > 0 && cut[i].top_item + cut[i].more <= most) {  // and so it is for more splits
                const Cut &c = cut[cut[i].best_top];
                take(c, top, c.top_item, c.top_cost);
                break;
            }
            const Cut &c = cut[i];
            int64_t R = top;
            double one = c.top_item, cost = c.top_cost;
            if (one > most) {
                R = (int64_t)std::max(32.0, std::min((most - c.fixed) * c.inv_row, (double)top)) & ~(int64_t)31;
                one = c.fixed + c.per_row * (double)R;
                cost = (n <= R ? 1.0 : std::ceil((double)n / (double)R)) * (double)c.S * (one + c.more);
            }
            if (one + c.more > most) cost *= (one + c.more) / most;  // too long all the same: it counts for more
            take(c, R, one, cost);
        }
        *items = std::ceil((double)n / best.R) * best.S;
        return best;
    }
};

// One persistent launch over up to FP_MAX_BATCH (forest, batch) pairs.  How
// long an item may take is chosen for the whole launch: of a few lengths, the
// one with the least estimated end: the longest item when all items run at
// once, else the items' sum over the GPU's CTAs and the longest item besides
// (it may begin last).  Tiles as large as each forest's
// own left the last of them running alone, and a batch of a few rows walked
// all bins of a pass in one CTA (four forests, 3 to 52,001 rows: 379 us; four
// of 33 to 178 rows: 76 us).
static int predict_batched_chunk(const fp_device_forest *const *forests, const fp_batch *batches, int32_t k,
                                 cudaStream_t s) {
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    int max_optin = 0;
    e = cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
    const size_t budget = (size_t)max_optin - 256;
    int warps = 1;
    for (int32_t j = 0; j < k; ++j) warps = std::max(warps, forests[j]->threads / 32);

    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");

    BatchParams bp;
    memset(&bp, 0, sizeof bp);
    size_t smem = 0;
    int32_t live[FP_MAX_BATCH], max_R[FP_MAX_BATCH];  // batches with work, and their largest tiles
    int32_t m = 0;
    for (int32_t j = 0; j < k; ++j) {
        const fp_device_forest *f = forests[j];
        const fp_batch &bt = batches[j];
        if (bt.n == 0 || (!bt.out_votes && !bt.out_class)) continue;
        const FpImageHeader &h = f->hdr;
        int R = f->R;
        while (R > 32 && smem_bytes(R, h.n_features, f->head_plan, f->nbuf, h.n_classes, warps, false) > budget) R -= 32;
        const size_t need = smem_bytes(R, h.n_features, f->head_shared, f->nbuf, h.n_classes, warps, false);
        if (smem_bytes(R, h.n_features, f->head_plan, f->nbuf, h.n_classes, warps, false) > budget) {
            fp_set_error("fp_predict_batched: batch %d does not fit shared memory with %d warps", j, warps);
            return FP_EUNSUPPORTED;
        }
        smem = std::max(smem, need);
        live[m] = j;
        max_R[m++] = R;
    }
    if (m == 0) return FP_OK;
    BatchCuts cuts[FP_MAX_BATCH];
    for (int32_t i = 0; i < m; ++i) cuts[i].form(forests[live[i]], batches[live[i]].n, max_R[i]);
    Shape shapes[FP_MAX_BATCH], tried[FP_MAX_BATCH];
    double best_end = 1e300, least = 0.0;  // the shortest item of some batch, which no shape undercuts
    for (int32_t i = 0; i < m; ++i) least = std::max(least, cuts[i].least);
    for (double len = 8000.0; len < 4e6; len *= 1.5) {
        if (len * 1.5 < least) continue;
        double sum = 0.0, longest = 0.0, items = 0.0;
        bool whole = true;
        for (int32_t i = 0; i < m; ++i) {
            double item = 0.0, count = 0.0;
            tried[i] = cuts[i].within(len, &item, &count);
            whole = whole && tried[i].S == 1 && tried[i].R == cuts[i].top;
            sum += item * count;
            items += count;
            longest = std::max(longest, item);
        }
        const double end = items <= sms ? longest : sum / sms + longest;
        if (end < best_end) {
            best_end = end;
            std::copy(tried, tried + m, shapes);
        }
        if (whole) break;  // longer items there are none
    }
    size_t scratch_bytes = 256;  // the work counter, then per-batch accumulators and tile counters
    size_t acc_off[FP_MAX_BATCH] = {0}, cnt_off[FP_MAX_BATCH] = {0};
    for (int32_t i = 0; i < m; ++i) {
        const fp_device_forest *f = forests[live[i]];
        const fp_batch &bt = batches[live[i]];
        // one-word heads for every forest that has them, so that most launches
        // need one kind of walk (mixed kinds: 4 % longer)
        TravParams p = base_params(f, bt.X, bt.n, f->d_compact ? 3 : f->levels);
        set_shape(p, shapes[i]);
        p.out_votes = bt.out_votes;
        p.out_class = bt.out_class;
        if (p.n_splits > 1) {
            const size_t votes = (size_t)bt.n * f->hdr.n_classes * 4;
            if (!bt.out_votes || votes <= (4u << 20)) {  // else they add up in the caller's votes
                acc_off[i] = scratch_bytes;
                scratch_bytes += (votes + 255) & ~(size_t)255;
            }
            cnt_off[i] = scratch_bytes;
            scratch_bytes += ((size_t)p.n_tiles * 4 + 255) & ~(size_t)255;
        }
        bp.p[i] = p;
        bp.item_begin[i + 1] = bp.item_begin[i] + p.n_items;
    }
    bp.k = m;
    void *scratch = nullptr;
    int rc = scratch_alloc(device, &scratch, scratch_bytes, s);
    if (rc) return rc;
    uint8_t *sc = static_cast<uint8_t *>(scratch);
    e = cudaMemsetAsync(scratch, 0, scratch_bytes, s);
    for (int32_t j = 0; j < m && e == cudaSuccess; ++j) {
        TravParams &p = bp.p[j];
        if (p.n_splits > 1) {
            p.acc = acc_off[j] ? reinterpret_cast<uint32_t *>(sc + acc_off[j]) : p.out_votes;
            p.tile_done = reinterpret_cast<uint32_t *>(sc + cnt_off[j]);
            if (!acc_off[j]) e = cudaMemsetAsync(p.out_votes, 0, (size_t)p.n * p.C * 4, s);
        }
    }
    bp.work = reinterpret_cast<unsigned long long *>(sc);
    // one walk compiled in when every forest has the same kind of super-node,
    // and the head kind when every forest has the same one
    int dk = bp.p[0].deep_kind, hk = bp.p[0].levels;
    for (int32_t j = 0; j < m; ++j) {
        if (bp.p[j].deep_kind != dk) dk = 0;
        if (bp.p[j].levels != hk) hk = -1;
    }
    void (*kern)(BatchParams) = batched_kernel(dk, hk);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * warps, smem);
    if (e == cudaSuccess) {
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(bp.item_begin[m], (int64_t)per_sm * sms));
        e = launch(kern, grid, 32 * warps, smem, s, bp);
    }
    cudaFreeAsync(scratch, s);
    if (e != cudaSuccess) return cuda_fail(e, "fp_predict_batched");
    return FP_OK;
}

extern "C" int fp_predict_batched(const fp_device_forest *const *forests, const fp_batch *batches, int32_t k,
                                  void *stream) {
    if (k < 0 || (k > 0 && (!forests || !batches))) {
        fp_set_error("fp_predict_batched: bad arguments");
        return FP_EINVAL;
    }
    for (int32_t i = 0; i < k; ++i) {
        if (!forests[i] || batches[i].n < 0 || (batches[i].n > 0 && !batches[i].X)) {
            fp_set_error("fp_predict_batched: bad batch %d", i);
            return FP_EINVAL;
        }
        if (forests[i]->hdr.n_values > 0) {
            fp_set_error("fp_predict_batched: forest %d has leaf values; use fp_predict_values", i);
            return FP_EINVAL;
        }
        int rc = check_device(forests[i]);
        if (rc) return rc;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int32_t i = 0; i < k; i += FP_MAX_BATCH) {
        int rc = predict_batched_chunk(forests + i, batches + i, std::min<int32_t>(FP_MAX_BATCH, k - i), s);
        if (rc) return rc;
    }
    return FP_OK;
}

// ------------------------------------------------- host buffers, pipelined

namespace {

std::mutex g_copy_mu;
// per device, created on first use, kept for the process: [0] the copy
// stream, [1] a second stream for every other chunk's kernel
std::vector<cudaStream_t> g_lib_stream[2];

int lib_stream(int device, int which, cudaStream_t *out) {
    std::lock_guard<std::mutex> lk(g_copy_mu);
    std::vector<cudaStream_t> &v = g_lib_stream[which];
    if ((int)v.size() <= device) v.resize((size_t)device + 1, nullptr);
    if (!v[device]) {
        cudaError_t e = cudaStreamCreateWithFlags(&v[device], cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            v[device] = nullptr;
            return cuda_fail(e, which ? "cudaStreamCreateWithFlags(compute)" : "cudaStreamCreateWithFlags(copy)");
        }
    }
    *out = v[device];
    return FP_OK;
}

// Rows from host memory through the device in chunks (eight by default):
// chunk c's rows are copied in on the library's copy stream into one of two
// device buffers while earlier chunks are classified; the chunks of buffer 0
// are classified on the caller's stream and those of buffer 1 on a second
// library stream, so that a chunk's kernel starts on the SMs that the
// previous chunk's kernel has left, instead of after its last CTA; each
// chunk's outputs are copied back on its kernel's stream.  The caller's
// stream waits for the second one before the buffers are released, so all
// the work is ordered before whatever the caller enqueues next.  out_bytes:
// bytes of output per row (one region per output); run(Xd, rows, outs,
// stream) launches the chunk's classification on `stream`.
template <class Run>
int pipeline_host(const fp_device_forest *f, const float *X_host, int64_t n, int64_t chunk_rows,
                  const int64_t out_bytes[2], void *const out_host[2], cudaStream_t s, const char *what, Run run) {
    const int64_t F = f->hdr.n_features;
    const int64_t chunk = std::min<int64_t>(n, chunk_rows > 0 ? chunk_rows : std::max<int64_t>(65536, (n + 7) / 8));
    const int nbuf = n > chunk ? 2 : 1;
    auto align = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
    const int64_t in_b = align(chunk * F * 4), o0 = align(chunk * out_bytes[0]), o1 = align(chunk * out_bytes[1]);
    const int64_t per_buf = in_b + o0 + o1;
    cudaStream_t cs = nullptr, s2 = nullptr;
    int rc = lib_stream(f->device, 0, &cs);
    if (rc == FP_OK && nbuf == 2) rc = lib_stream(f->device, 1, &s2);
    if (rc) return rc;
    void *block = nullptr;
    rc = scratch_alloc(f->device, &block, (size_t)(nbuf * per_buf), s);
    if (rc) return rc;
    cudaEvent_t ev[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};  // ready, in[2], free[2], s2 done
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 6 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev[0], s);  // the block is allocated; earlier work on s is ordered
    if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, ev[0], 0);
    if (e == cudaSuccess && s2) e = cudaStreamWaitEvent(s2, ev[0], 0);
    bool s2_used = false;
    uint8_t *base = static_cast<uint8_t *>(block);
    for (int64_t c = 0, r0 = 0; e == cudaSuccess && rc == FP_OK && r0 < n; ++c, r0 += chunk) {
        const int b = (int)(c % nbuf);
        cudaStream_t ks = b == 0 ? s : s2;  // the chunk's kernel and output copies
        s2_used |= b == 1;
        const int64_t rows = std::min<int64_t>(chunk, n - r0);
        uint8_t *buf = base + b * per_buf;
        if (c >= nbuf) e = cudaStreamWaitEvent(cs, ev[3 + b], 0);  // chunk c-2 is done with the buffer
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(buf, X_host + r0 * F, (size_t)(rows * F * 4), cudaMemcpyHostToDevice, cs);
        if (e == cudaSuccess) e = cudaEventRecord(ev[1 + b], cs);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ks, ev[1 + b], 0);
        if (e != cudaSuccess) break;
        void *outs[2] = {out_host[0] ? buf + in_b : nullptr, out_host[1] ? buf + in_b + o0 : nullptr};
        rc = run(reinterpret_cast<const float *>(buf), rows, outs, ks);
        for (int k = 0; k < 2 && rc == FP_OK && e == cudaSuccess; ++k)
            if (out_host[k])
                e = cudaMemcpyAsync(static_cast<uint8_t *>(out_host[k]) + r0 * out_bytes[k], outs[k],
                                    (size_t)(rows * out_bytes[k]), cudaMemcpyDeviceToHost, ks);
        if (e == cudaSuccess) e = cudaEventRecord(ev[3 + b], ks);
    }
    if (s2_used) {  // the caller's stream covers the second stream's work, errors or not
        cudaError_t e2 = cudaEventRecord(ev[5], s2);
        if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(s, ev[5], 0);
        if (e2 != cudaSuccess) cudaStreamSynchronize(s2);
        if (e == cudaSuccess) e = e2;
    }
    if (e != cudaSuccess || rc != FP_OK) cudaStreamSynchronize(cs);  // nothing of the copy stream outlives the block
    cudaFreeAsync(block, s);
    for (int i = 0; i < 6; ++i)
        if (ev[i]) cudaEventDestroy(ev[i]);
    if (e != cudaSuccess) return cuda_fail(e, what);
    return rc;
}

}  // namespace

extern "C" int fp_predict_host(const fp_device_forest *f, const float *X_host, int64_t n, uint32_t *out_votes_host,
                               int32_t *out_class_host, int64_t chunk_rows, void *stream) {
    if (!f || n < 0 || chunk_rows < 0 || (n > 0 && !X_host)) {
        fp_set_error("fp_predict_host: bad arguments");
        return FP_EINVAL;
    }
    if (f->hdr.n_values > 0) {
        fp_set_error("fp_predict_host: the forest has leaf values; use fp_predict_values_host");
        return FP_EINVAL;
    }
    if (n == 0 || (!out_votes_host && !out_class_host)) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t ob[2] = {4 * (int64_t)f->hdr.n_classes, 4};
    void *const oh[2] = {out_votes_host, out_class_host};
    return pipeline_host(f, X_host, n, chunk_rows, ob, oh, s, "fp_predict_host",
                         [&](const float *Xd, int64_t rows, void *const outs[2], cudaStream_t ks) {
                             return fp_predict(f, Xd, rows, static_cast<uint32_t *>(outs[0]),
                                               static_cast<int32_t *>(outs[1]), ks);
                         });
}

extern "C" int fp_predict_values_host(const fp_device_forest *f, const float *X_host, int64_t n, float scale,
                                      float bias, float *out_host, int64_t chunk_rows, void *stream) {
    if (!f || n < 0 || chunk_rows < 0 || (n > 0 && (!X_host || !out_host))) {
        fp_set_error("fp_predict_values_host: bad arguments");
        return FP_EINVAL;
    }
    if (f->hdr.n_values <= 0) {
        fp_set_error("fp_predict_values_host: the forest was packed without leaf values");
        return FP_EINVAL;
    }
    if (n == 0) return FP_OK;
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t ob[2] = {4, 0};
    void *const oh[2] = {out_host, nullptr};
    return pipeline_host(f, X_host, n, chunk_rows, ob, oh, s, "fp_predict_values_host",
                         [&](const float *Xd, int64_t rows, void *const outs[2], cudaStream_t ks) {
                             return fp_predict_values(f, Xd, rows, scale, bias, static_cast<float *>(outs[0]), ks);
                         });
}

// ------------------------------------------- statistics from observations

// Section III-A: the cardinalities that order a tree's nodes (Stat) may be
// measured on observations instead of taken from training.  The rows go
// through fp_predict_leaves in chunks (the leaf ids of one chunk sit in
// scratch), fp_count_leaves adds them up per node on the device, and the
// counts come back to the host, where each internal node becomes the sum of
// its children (fp_cardinality_from_leaf_counts).
extern "C" int fp_infer_cardinality(const fp_device_forest *f, const fp_forest_desc *desc, const float *X, int64_t n,
                                    int64_t chunk_rows, int64_t *out_card, void *stream) {
    if (!f || !desc || !out_card || n < 0 || chunk_rows < 0 || (n > 0 && !X) || !desc->tree_node_begin) {
        fp_set_error("fp_infer_cardinality: bad arguments");
        return FP_EINVAL;
    }
    const FpImageHeader &h = f->hdr;
    if (desc->n_trees != h.n_trees || desc->n_features != h.n_features || desc->n_classes != h.n_classes) {
        fp_set_error("fp_infer_cardinality: the descriptor (%d trees, %d features, %d classes) is not the forest's "
                     "(%d, %d, %d)", desc->n_trees, desc->n_features, desc->n_classes, h.n_trees, h.n_features,
                     h.n_classes);
        return FP_EINVAL;
    }
    int64_t n_internal = 0;
    const int64_t total = desc->tree_node_begin[desc->n_trees];
    if (desc->left)
        for (int64_t v = 0; v < total; ++v) n_internal += desc->left[v] >= 0;
    if (!desc->left || n_internal != h.n_internal) {
        fp_set_error("fp_infer_cardinality: the descriptor's internal nodes do not match the packed forest's");
        return FP_EINVAL;
    }
    int rc = check_device(f);
    if (rc) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t T = h.n_trees;
    const int64_t chunk = std::max<int64_t>(
        1, std::min<int64_t>(n, chunk_rows > 0 ? chunk_rows : std::max<int64_t>(1, (256 << 20) / (4 * T))));
    auto align = [](int64_t b) { return (b + 255) & ~(int64_t)255; };
    const int64_t cnt_b = align(total * 8), nb_b = align((T + 1) * 8), st_b = 256;
    const int64_t leaf_b = n > 0 ? align(chunk * T * 4) : 0;
    void *block = nullptr;
    rc = scratch_alloc(f->device, &block, (size_t)(cnt_b + nb_b + st_b + leaf_b), s);
    if (rc) return rc;
    uint8_t *base = static_cast<uint8_t *>(block);
    int64_t *d_cnt = reinterpret_cast<int64_t *>(base);
    int64_t *d_nb = reinterpret_cast<int64_t *>(base + cnt_b);
    int32_t *d_st = reinterpret_cast<int32_t *>(base + cnt_b + nb_b);
    int32_t *d_leaf = reinterpret_cast<int32_t *>(base + cnt_b + nb_b + st_b);
    int32_t st = 0;
    cudaError_t e = cudaMemsetAsync(block, 0, (size_t)(cnt_b + nb_b + st_b), s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_nb, desc->tree_node_begin, (size_t)(T + 1) * 8, cudaMemcpyHostToDevice, s);
    for (int64_t r0 = 0; e == cudaSuccess && rc == FP_OK && r0 < n; r0 += chunk) {
        const int64_t rows = std::min<int64_t>(chunk, n - r0);
        rc = fp_predict_leaves(f, X + r0 * h.n_features, rows, d_leaf, stream);
        if (rc == FP_OK) rc = fp_count_leaves(d_leaf, rows, (int32_t)T, d_nb, d_cnt, d_st, stream);
    }
    if (e == cudaSuccess && rc == FP_OK)
        e = cudaMemcpyAsync(out_card, d_cnt, (size_t)total * 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && rc == FP_OK) e = cudaMemcpyAsync(&st, d_st, 4, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(block, s);
    const cudaError_t es = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = es;
    if (rc != FP_OK) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "fp_infer_cardinality");
    if (st != 0) {
        fp_set_error("fp_infer_cardinality: a leaf id was not a node of its tree");
        return FP_EDEVICE;
    }
    rc = fp_sync_status(f, stream);  // an error the traversal kernel recorded
    if (rc) return rc;
    return fp_cardinality_from_leaf_counts(desc, out_card, out_card);
}
