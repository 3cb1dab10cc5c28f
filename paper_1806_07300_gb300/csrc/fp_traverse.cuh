// fp_traverse.cuh -- the packed-forest traversal kernel (sm_103a).
//
// One work item = an observation tile and one of the parts (splits) that the
// forest's bins are cut into: a single one for large batches, so that a CTA
// sweeps all bins for its tile; the CTAs sweep the same bins at about the same
// time, which keeps the bins' super-nodes in L2 while every tile walks them
// (the GPU counterpart of the paper's bins bound to cores, Section III).  How
// a call is cut up is chosen on the host (fp_device.cu).  For an item the CTA:
//   1. stages the tile's rows into shared memory in slabs of 32 rows: a slab
//      holds its F features and then its vote counters (one per class, or one
//      float sum), 32 words each, row l of the slab in column l.  32 lanes
//      holding the 32 rows of a slab read any features and count any votes in
//      32 different banks, and feature f of a row is 128 * f bytes past the
//      row's own address, so a task carries that one address and no step
//      multiplies by the tile size.  For a forest with three-level
//      super-nodes each value is turned into its order key (fp_internal.h)
//      and every compare is an unsigned integer compare, otherwise values and
//      compares stay float;
//   2. streams the bins' interleaved blocks (the heads of their trees,
//      Section III-A Bin) through nbuf (2 or 3) shared-memory buffers with TMA bulk
//      copies (cp.async.bulk) completing on mbarriers: a warp waits only for
//      the block of the bin it walks next, and the last warp done with a
//      bin's block refills that buffer with the bin nbuf places ahead;
//   3. walks (observation, tree) tasks in two kinds of warp steps:
//        burst -- the warp takes its next unit, the 32 rows of one slab and
//                 one tree, and all lanes walk their paths through the tree's
//                 head in shared memory together, with a branch-free step
//                 (level heads: exactly d+1 steps over implicit slots, or
//                 (d+1)/2 steps of two levels when the slots are paired;
//                 ranked heads: until the last lane leaves the head); paths
//                 that leave the head are pushed, compacted with
//                 __ballot_sync / __popc, into the warp's ring of pending
//                 tasks.  Units are claimed from a shared counter: dealt out
//                 to the warps in turn they cost no atomic, but the slowest
//                 warp then held up each bin's buffer, 8 % of the run;
//        deep  -- every lane holding a task resolves two or three more levels
//                 with one 32-byte super-node load (one L2 sector); a lane
//                 that reaches a leaf votes and takes the next pending task
//                 from the ring.
//      Bursts keep the ring topped up, so lanes stay busy while paths of very
//      different depth diverge -- the GPU form of the paper's round-robin over
//      independent tasks (Section III-B).  Pending and running tasks carry
//      over from one bin to the next, and nothing but the item's end makes a
//      warp wait for another;
//   4. counts votes per (row, class) with shared-memory atomics;
//   5. writes votes and the argmax class (lowest class on ties).  With one
//      split the tile's votes are complete in shared memory; with several, they
//      are added to a global accumulator and the CTA that finishes a tile's
//      last split takes the argmax (per-tile counter, no waiting; no counter
//      and no argmax when votes alone are asked for).
// Parity mode writes the leaf id reached in every (observation, tree)
// instead of voting.  Values mode (forests with real leaf values: regression
// and boosted trees) adds the leaf's value to a float per row instead, and
// writes bias + scale * sum (several splits: summed in global memory, the
// last split's CTA writes it).
//
// What bounds it (256 trees of 78.8k nodes, 28 features, 4 M rows, bins of 5
// trees with heads 0..9: 24.1 ms; 27.5 ms as one pass of L2 after another with
// steps of divergent branches): the load/store data pipe, 77 % busy with 5.7
// wavefronts per (row, tree), 4.5 sectors of super-nodes and rows and 2.5
// wavefronts of shared memory among them (6.3 before); 18.7 warp instructions
// per (row, tree) (23.4 before) take 63 % of the issue slots.
//
// Waits: __syncthreads is a hardware wait; a wait for
// a bin block polls its mbarrier at most spin_limit times (FP_SPIN_LIMIT
// unless a test lowers it), then records FP_ETIMEOUT in the status word and
// makes every warp skip the rest of its work; before exiting, the CTA waits
// (bounded by FP_SPIN_LIMIT polls) for its own bulk copies to land.  A test
// can set `stall` so that bin waits ignore completed copies and run out; the
// copies themselves still complete, so the exit path stays clean.  Every walk
// is bounded too.
#pragma once
#include <stdint.h>

#include "fp_internal.h"

struct TravParams {
    const FpSuper *deep;      // super-nodes
    const uint8_t *heads;     // interleaved blocks
    const FpBin *bins;
    const FpPass *passes;
    const int32_t *pheads;    // parity: leaf id per block exit
    const int32_t *deep_leaf; // parity: 4 leaf ids per super-node
    const float *X;
    int64_t n;
    int64_t n_tiles;
    int64_t n_items;          // n_tiles * n_splits
    int32_t n_splits;         // parts that a tile's bins are cut into, each an item of its own
    int32_t split_bins;       // bins of a split: n_bins / n_splits, one more in the first
    int32_t split_more;       // n_bins % n_splits
    int32_t n_bins;
    int32_t F, C, T, R;
    uint32_t slab;            // bytes of a slab: 32 rows of F features and the mode's counters
    int32_t n_passes;         // with as many splits, the splits are the packed passes
    int32_t head_smem;        // bytes reserved for one bin block
    int32_t nbuf;             // bin-block buffers (2 or 3)
    int32_t levels;           // head kind: 0 ranked, 1 level slots (depth+1 steps), 2 paired level slots,
                              // 3 level slots of one word (fp_compact_heads_kernel)
    int32_t packed_kind;      // head kind 3: the packed image's, 1 or 2 ...
    const uint8_t *packed_heads;  // ... its blocks and their bins, for key ties
    const FpBin *packed_bins;
    int32_t depth;            // d of the interleaved head
    int32_t refill;           // bursts start when the ring holds at most this many tasks
    int32_t step_bins;        // a deep step in every bin, also in bins of fewer units than warps
    uint32_t *out_votes;      // final votes (may be NULL, or acc)
    int32_t *out_class;       // may be NULL
    int32_t *out_leaf;        // parity mode
    uint32_t *acc;            // several splits: vote accumulator
    uint32_t *tile_done;      // several splits: per-tile counter of finished ones (NULL: votes alone are asked for)
    int32_t *status;          // device status word
    const float *leaf_val;    // forests with leaf values: value of each leaf slot
    uint32_t n_vals;          // slots in leaf_val
    float vscale, vbias;      // out = vbias + vscale * sum of leaf values
    float *out_val;           // values mode: output per row
    float *acc_val;           // values mode, several splits: per-row accumulator
    int32_t spin_limit;       // polls of a bin block's barrier before the wait gives up
    int32_t stall;            // fault injection: bin waits ignore completed copies (0 normally)
    int32_t deep_kind;        // super-nodes: 2 two levels, 3 three levels (format 1), 4 three levels (format 2)
    uint32_t tie;             // three levels: equal key prefixes of the last level differ only below this
                              // (2fb + 2cb bits in format 1, fb + 2cb in format 2)
    uint32_t frot;            // format 1: rotation that brings an upper slot's feature to bit 7
    uint32_t cshl, cshr;      // three levels: where a last-level word holds its left and right exits' classes
    uint32_t fmask, cmask;    // three levels: feature and class masks
    uint32_t vbase3;          // three levels, values mode: first per-exit value slot
    const uint32_t *deep_keys;  // three levels: full keys, 4 (format 1) or 8 (format 2) per super-node
    uint32_t klo, khi, kshl, kflag;  // format 2: the key remap V of the staged rows
    uint32_t kga, kgb, kgd;          // format 2: its collapsed run of keys
    uint32_t n_super;         // super-nodes (below 2^31)
};

// What a kernel computes per (row, tree) task it finishes.
#define FP_MODE_VOTES 0   // a vote for the leaf's class; then votes and the argmax class
#define FP_MODE_LEAVES 1  // the leaf id (parity mode)
#define FP_MODE_VALUES 2  // the leaf's value, summed per row; then bias + scale * sum

#define FP_ERR_FLAG_DEVICE (-6)
#define FP_ERR_FLAG_TIMEOUT (-5)
#define FP_NBUF 3             // bin-block buffers at most (a launch uses nbuf = 2 or 3)
#define FP_SPIN_LIMIT (1 << 24)
#define FP_RING 64            // pending tasks per warp
#define FP_NO_CLASS (FP_REF_LEAF | 0x7FFFFFFFu)
#define FP_NO_TASK 0xFFFFFFFFu  // a lane's ref when it holds no task (super-node indices are below 2^31)

// One super-node: a single 256-bit load (32-byte aligned, one L2 sector), for
// the lanes that hold a task (ref is no index otherwise).
// The lines are not allocated in L1: few super-nodes are read twice by one
// SM before eviction, and with most of the unified L1/shared array given to
// shared memory, allocating a line per lane for thousands of loads in
// flight throttles the load path (measured: twice the run time once shared
// memory takes more than about 196 KB).  The memory clobber keeps the load
// where it is written, ahead of the work meant to overlap its latency.
__device__ __forceinline__ void ld_super(const FpSuper *deep, uint32_t ref, uint32_t w[8]) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %9, %10;\n"
                 " @p ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n}\n"
                 : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7])
                 : "l"(deep + ref), "r"(ref), "n"(FP_NO_TASK)
                 : "memory");
}

__device__ __forceinline__ void report(int32_t *status, int32_t code) { atomicCAS(status, 0, code); }

// The order key of an observation value (fp_internal.h): compares like the
// float against threshold keys; NaN goes above every threshold (right).
__device__ __forceinline__ uint32_t obs_key(float v) {
    uint32_t u = __float_as_uint(v);
    if ((u & 0x7FFFFFFFu) > 0x7F800000u) return 0xFFFFFFFFu;
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The remapped key V of format 2 (fp_internal.h): the run of keys without a
// threshold collapsed, then clamped to the forest's threshold range and
// spread over the 31 bits below a set top bit.
__device__ __forceinline__ uint32_t remap_key(const TravParams &p, uint32_t k) {
    const uint32_t g = k >= p.kgb ? k - p.kgd : min(k, p.kga);
    return p.kflag | ((min(max(g, p.klo), p.khi) - p.klo) << p.kshl);
}

// A staged observation value for super-node kind DK: its float bits (2), or
// one less than its order key (3) or remapped key (4; no key is 0).  One less,
// so that a value equal to a threshold, as rows of whole numbers or of few
// distinct values have, shares no prefix with it where the bits below are
// zero: prefixes that are equal cost a look at the full keys (64 trees on 28
// binary features with thresholds on their values, 200,000 rows: 190 us, 327
// with the keys themselves).
template <int DK>
__device__ __forceinline__ uint32_t staged(const TravParams &p, float v) {
    return DK == 2 ? __float_as_uint(v) : (DK == 3 ? obs_key(v) : remap_key(p, obs_key(v))) - 1u;
}

// x <= t, the split's test (go left): keys compare as unsigned integers (the
// staged x being one less), otherwise as floats (a NaN x or t goes right either
// way).
template <bool KEYS>
__device__ __forceinline__ bool goes_left(uint32_t x, uint32_t t) {
    return KEYS ? x < t : __uint_as_float(x) <= __uint_as_float(t);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// true once the phase of the given parity has completed
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// CTA-wide state shared by the items a CTA runs.
struct __align__(16) CtaShared {
    FpBin desc[FP_NBUF];      // the record of each buffer's bin
    uint4 ahead[FP_NBUF];     // the first half of the record of the bin that refills the buffer
    uint64_t full[FP_NBUF];   // block staged (bulk copy done)
    int next[FP_NBUF];        // next untaken unit of the buffer's bin
    int done[FP_NBUF];        // warps done with the buffer's bin
    int issued[FP_NBUF];      // bulk copies issued into the buffer
    uint32_t phases;          // parities of issued[] when the current item started
    int bin0, bin1;           // the current item's bins
    int64_t tile;             // the current item's tile
    int last;
    int abort;
    long long next_item;
};

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Shared memory by 32-bit addresses.  The walks take theirs from one base that
// run_item keeps in a register: through pointers to the shared arrays, the
// compiler may form the array's address anew in every step (from a special
// register, since it depends on the CTA's place in its cluster), which cost
// the walks up to 9 % of their time.
__device__ __forceinline__ uint32_t lds(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}

__device__ __forceinline__ void sts64(uint32_t addr, uint32_t x, uint32_t y) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};\n" ::"r"(addr), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void add_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void add_shared(uint32_t addr, float v) {
    asm volatile("red.shared.add.f32 [%0], %1;\n" ::"r"(addr), "f"(v) : "memory");
}

// Per-lane state of a running task.  A corrupt record only sets `bad`,
// reported at the item's end, so that a step stays straight-line code.
struct LaneTask {
    uint32_t ref;     // current super-node (index into deep), or FP_NO_TASK
    uint32_t xb;      // shared-memory address of the row: feature f is 128 f bytes further on
    uint32_t rt;      // parity mode: row within the tile | tree << 11
    int bad;
};

// A lane before its first task.  The deep step's reads of the row are not
// predicated, so the row that such a lane reads (and makes nothing of) is
// one of the tile's own: the first, at `base`.
__host__ __device__ __forceinline__ LaneTask idle_task(uint32_t base) {
    LaneTask L;
    L.ref = FP_NO_TASK;
    L.xb = base;
    L.rt = 0;
    L.bad = 0;
    return L;
}

// A finished task's memory read whose result is not used at once: the leaf's
// value on its way to the row's sum (values mode), or its leaf id on its way
// to the output (parity mode).  Used right before the next deep step, which
// waits for its super-nodes there anyway; a use at once stalls the warp for a
// whole L2 latency in nearly every step, and one before the head walk between
// two steps waits where the walk could have hidden it (leaf ids of 64 trees,
// 100-feature rows, 100,000 rows: 160 -> 146 us, 155 before leaf ids were used
// late at all; 128 regression trees, 1 M rows: 2856 -> 2769 us).
struct Pending {
    bool on;
    uint32_t at;      // values: xb; parity: rt
    uint32_t word;
};

// A vote for class `cls` of the row at xb.  Class 0 is not counted: its votes
// are the item's trees less all the others'.  Returns false for a class that
// does not exist.
__device__ __forceinline__ bool vote(const TravParams &p, bool on, uint32_t xb, uint32_t cls) {
    const bool counted = cls - 1u < (uint32_t)p.C - 1u;
    if (on && counted) add_shared(xb + (((uint32_t)p.F + cls) << 7), 1u);
    return !on || counted || cls == 0u;
}

// The row's sum of leaf values (values mode).
__device__ __forceinline__ void add_value(const TravParams &p, uint32_t xb, float v) {
    add_shared(xb + ((uint32_t)p.F << 7), v);
}

// Parity mode; leaves: the output from the tile's first row on.
__device__ __forceinline__ void put_leaf(const TravParams &p, int32_t *leaves, uint32_t rt, int32_t leaf_id) {
    leaves[(uint64_t)(rt & 2047u) * (uint32_t)p.T + (rt >> 11)] = leaf_id;
}

template <int MODE>
__device__ __forceinline__ void settle(const TravParams &p, int32_t *leaves, Pending &pend) {
    if (MODE == FP_MODE_VOTES) return;
    if (pend.on) {
        if (MODE == FP_MODE_VALUES)
            add_value(p, pend.at, __uint_as_float(pend.word));
        else
            put_leaf(p, leaves, pend.at, (int32_t)pend.word);
    }
    pend.on = false;
}

// Lanes without a task take pending ones from the warp's ring.
template <int MODE>
__device__ __forceinline__ void pop_tasks(const TravParams &p, uint32_t base, uint32_t ring, int &head, int tail, LaneTask &L,
                                          unsigned lt_mask) {
    const bool free = L.ref == FP_NO_TASK;
    const unsigned idle = __ballot_sync(0xffffffffu, free);
    const int rk = __popc(idle & lt_mask);
    uint32_t &second = MODE == FP_MODE_LEAVES ? L.rt : L.xb;
    asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q ld.shared.v2.u32 {%0, %1}, [%2];\n}\n"
                 : "+r"(L.ref), "+r"(second)
                 : "r"(ring + (uint32_t)((head + rk) & (FP_RING - 1)) * 8u), "r"(free && rk < tail - head ? 1u : 0u)
                 : "memory");
    if (MODE == FP_MODE_LEAVES) L.xb = base + ((L.rt & 2047u) >> 5) * p.slab + (L.rt & 31u) * 4u;
    head = min(head + __popc(idle), tail);
}

// One deep step in two halves: the load is issued first and consumed after
// the warp has done other work (a head burst), so the L2 latency overlaps
// that work.  The second half is written without branches (but for key ties,
// which are rare): all lanes compute, and the lanes without a task keep
// nothing.  Its outcome:
struct DeepStep {
    bool leaf;
    uint32_t cls;         // the leaf's class (two levels, values mode: its value slot)
    uint32_t next;        // the next super-node
    uint32_t e;           // the exit taken
};

// Three levels: exit e is a leaf, or leads to one of the super-node's
// children, which sit side by side from the offset on, in exit order.
__device__ __forceinline__ void exit3(uint32_t ref, uint32_t w7, DeepStep &s) {
    // bit 24: exit e leads on; below it: the exits before e that lead on
    const uint32_t on = (~w7 & 0xFF000000u) >> s.e;
    s.leaf = (on & (1u << 24)) == 0u;
    s.next = ref + (w7 & FP_DEEP3_OFFSET_MASK) + __popc(on & 0xFFFFFFu);
}

// Three levels, format 1: full keys for the first two, and a key prefix for
// the last, whose tie (rare) is decided by the slot's full key from the side
// table.
__device__ __forceinline__ DeepStep deep_step3(const TravParams &p, uint32_t ref, uint32_t xb,
                                               const uint32_t w[8]) {
    const uint32_t fm7 = p.fmask << 7;
    const uint32_t k0 = lds(xb + (__funnelshift_r(w[3], w[3], p.frot) & fm7));
    const bool r0 = k0 >= w[0];
    const uint32_t n1 = r0 ? w[2] : w[1], m1 = r0 ? w[5] : w[4];
    const uint32_t k1 = lds(xb + (__funnelshift_r(m1, m1, p.frot) & fm7));
    const bool r1 = k1 >= n1;
    const uint32_t n2 = r0 ? (r1 ? w[6] : w[5]) : (r1 ? w[4] : w[3]);
    const uint32_t k2 = lds(xb + ((n2 & p.fmask) << 7));
    bool r2 = k2 >= n2;  // decided by the key bits, unless they are equal
    DeepStep s;
    s.e = (r0 ? 4u : 0u) + (r1 ? 2u : 0u);
    // behind a vote, so that the steps without a tie issue no load of the side
    // table; predicated off in every lane it still takes the load/store pipe
    // a wavefront a step (2 % of the run)
    const bool tie = (k2 ^ n2) < p.tie && ref != FP_NO_TASK;
    if (__any_sync(0xffffffffu, tie)) {
        if (tie) r2 = k2 >= __ldg(p.deep_keys + 4 * (int64_t)ref + (s.e >> 1));
        __syncwarp();
    }
    s.e += r2 ? 1u : 0u;
    s.cls = (n2 >> (r2 ? p.cshr : p.cshl)) & p.cmask;
    exit3(ref, w[7], s);
    return s;
}

// Three levels, format 2: every slot's word is the top bits of its remapped
// key over its feature (and classes), so comparing the staged V with the
// whole word decides the split wherever their top bits differ.  Where they
// are equal for any of the three slots of the walk (rare), the step is taken
// again with the slots' full keys from the side table.
__device__ __forceinline__ DeepStep deep_step3p(const TravParams &p, uint32_t ref, uint32_t xb,
                                                const uint32_t w[8]) {
    const uint32_t fm = p.fmask;
    const uint32_t k0 = lds(xb + ((w[0] & fm) << 7));
    bool r0 = k0 >= w[0];
    uint32_t n1 = r0 ? w[2] : w[1];
    const uint32_t k1 = lds(xb + ((n1 & fm) << 7));
    bool r1 = k1 >= n1;
    uint32_t n2 = r0 ? (r1 ? w[6] : w[5]) : (r1 ? w[4] : w[3]);
    uint32_t k2 = lds(xb + ((n2 & fm) << 7));
    bool r2 = k2 >= n2;
    // one test for the three slots, by the last level's shorter prefix: it
    // takes a few more steps again than need be
    const bool tie = min(min(k0 ^ w[0], k1 ^ n1), k2 ^ n2) < p.tie && ref != FP_NO_TASK;
    if (__any_sync(0xffffffffu, tie)) {
        if (tie) {
            const uint32_t *fk = p.deep_keys + 8 * (int64_t)ref;
            r0 = k0 >= __ldg(fk);
            n1 = r0 ? w[2] : w[1];
            r1 = lds(xb + ((n1 & fm) << 7)) >= __ldg(fk + 1 + (r0 ? 1 : 0));
            n2 = r0 ? (r1 ? w[6] : w[5]) : (r1 ? w[4] : w[3]);
            k2 = lds(xb + ((n2 & fm) << 7));
            r2 = k2 >= __ldg(fk + 3 + (r0 ? 2 : 0) + (r1 ? 1 : 0));
        }
        __syncwarp();
    }
    DeepStep s;
    s.e = (r0 ? 4u : 0u) + (r1 ? 2u : 0u) + (r2 ? 1u : 0u);
    s.cls = (n2 >> (r2 ? p.cshr : p.cshl)) & p.cmask;
    exit3(ref, w[7], s);
    return s;
}

// Two levels, float thresholds.
__device__ __forceinline__ DeepStep deep_step2(uint32_t xb, const uint32_t w[8]) {
    const bool r0 = !goes_left<false>(lds(xb + ((w[3] & 1023u) << 7)), w[0]);
    const uint32_t f1 = r0 ? (w[3] >> 20) & 1023u : (w[3] >> 10) & 1023u;
    const bool r1 = !goes_left<false>(lds(xb + (f1 << 7)), r0 ? w[2] : w[1]);
    const uint32_t x = r0 ? (r1 ? w[7] : w[6]) : (r1 ? w[5] : w[4]);
    DeepStep s;
    s.leaf = (x & FP_REF_LEAF) != 0u;
    s.cls = x & 0x7FFFFFFFu;
    s.next = x;
    s.e = (r0 ? 2u : 0u) + (r1 ? 1u : 0u);
    return s;
}

// DK: the forest's kind of super-node (p.deep_kind: 2, 3 or 4); a
// compile-time choice, so no kind's step carries another's code.
template <int MODE, int DK>
__device__ __forceinline__ void deep_finish(const TravParams &p, LaneTask &L, Pending &pend,
                                            const uint32_t w[8]) {
    const uint32_t ref = L.ref;
    const bool on = ref != FP_NO_TASK;
    const DeepStep s = DK == 3   ? deep_step3(p, ref, L.xb, w)
                       : DK == 4 ? deep_step3p(p, ref, L.xb, w)
                                 : deep_step2(L.xb, w);
    const bool leaf = on && s.leaf;
    if (MODE == FP_MODE_VOTES) {
        const uint32_t c1 = s.cls - 1u, nc = (uint32_t)p.C - 1u;
        asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %1, 0;\n @q red.shared.add.u32 [%0], 1;\n}\n" ::"r"(
                         L.xb + (((uint32_t)p.F + s.cls) << 7)),
                     "r"(leaf && c1 < nc ? 1u : 0u)
                     : "memory");
        if (leaf && s.cls > nc) L.bad = 1;
    } else if (MODE == FP_MODE_VALUES) {  // start the read of the leaf's value ...
        const uint32_t slot = DK == 2 ? s.cls : p.vbase3 + 8 * ref + s.e;
        const bool ok = slot < p.n_vals;
        L.bad |= leaf && !ok;
        if (leaf && ok) {
            pend.on = true;
            pend.at = L.xb;
            pend.word = __float_as_uint(__ldg(p.leaf_val + slot));
        }
    } else if (leaf) {  // ... or of its id
        pend.on = true;
        pend.at = L.rt;
        pend.word = (uint32_t)__ldg(p.deep_leaf + (DK == 2 ? 4 : 8) * (int64_t)ref + s.e);
    }
    // forward only, so every walk ends: 1 <= next - ref <= n_super - 1 - ref
    const bool ahead = s.next - ref - 1u < p.n_super - 1u - ref;
    const bool go = on && !s.leaf;
    if (go && !ahead) L.bad = 1;
    L.ref = go && ahead ? s.next : FP_NO_TASK;
}

// The walk of one row through a level head in the packed image itself, with
// full keys: the index of the exit it ends on.  Not inlined, to keep the walk
// that calls it (on key ties) as it is.
__device__ __noinline__ uint32_t packed_walk(const TravParams &p, int b, int k, uint32_t xb) {
    const FpBin bn = p.packed_bins[b];
    const uint8_t *blk = p.packed_heads + bn.head_off;
    uint32_t q = 0;
    if (p.packed_kind == 2) {
        for (int l = 0; l <= p.depth; l += 2) {
            const uint4 nd = __ldg(reinterpret_cast<const uint4 *>(blk) + q * bn.stride + k);
            const bool r0 = lds(xb + ((nd.w & 1023u) << 7)) >= nd.x;
            const bool r1 = lds(xb + (((nd.w >> (r0 ? 20 : 10)) & 1023u) << 7)) >= (r0 ? nd.z : nd.y);
            q = 4u * q + 1u + (r0 ? 2u : 0u) + (r1 ? 1u : 0u);
        }
    } else {
        for (int l = 0; l <= p.depth; ++l) {
            const uint2 nd = __ldg(reinterpret_cast<const uint2 *>(blk) + q * bn.stride + k);
            q = 2u * q + 1u + (lds(xb + ((nd.y >> 22) << 7)) >= nd.x ? 1u : 0u);
        }
    }
    return q - (uint32_t)bn.nranks;
}

// The walk of one row (at xb) through the head of tree column k of the bin
// block at blk, whose exits begin at `exits`: the address of the exit word it
// ends on, or FP_NO_EXIT (corrupt ranked heads only).  HK: the head
// kind when known at compile time (0 ranked, 1 level slots, 2 paired level
// slots), or -1 to read it from p.levels (the batched kernel, whose forests
// may differ); 3, only with keys: one-word level slots.  Record q of a level head lies at at0 + q * rec and exit e
// where record nranks + e would, scaled to 4-byte words, so the walks keep
// the record's offset itself and never its index.
#define FP_NO_EXIT 0xFFFFFFFFu

template <bool KEYS, int HK>
__device__ __forceinline__ uint32_t head_walk(const TravParams &p, int b, uint32_t blk, uint32_t exits, int k,
                                              int stride, int nranks, int nexits, uint32_t xb, bool my) {
    const int levels = HK >= 0 ? HK : p.levels;
    if (KEYS && levels == 3) {
        // one word per node: the top bits of its key over its feature, so that
        // comparing the whole word decides wherever the top bits differ;
        // children 2s+1, 2s+2, and exit e in slot nranks + e
        const uint32_t rec = (uint32_t)stride * 4u, at0 = blk + (uint32_t)k * 4u;
        const uint32_t left = rec - at0, right = left + rec;
        uint32_t at = at0, near = 0xFFFFFFFFu;
#pragma unroll 1  // two levels a turn: one saves loop control (1 % of the run), five or ten no more
        for (int l = p.depth; l > 0; l -= 2) {
            const uint32_t na = lds(at), xa = lds(xb + ((na & p.fmask) << 7));
            at = 2u * at + (xa >= na ? right : left);
            const uint32_t nb = lds(at), x2 = lds(xb + ((nb & p.fmask) << 7));
            near = min(near, min(xa ^ na, x2 ^ nb));
            at = 2u * at + (x2 >= nb ? right : left);
        }
        if (!(p.depth & 1)) {
            const uint32_t nd = lds(at), x = lds(xb + ((nd & p.fmask) << 7));
            near = min(near, x ^ nd);
            at = 2u * at + (x >= nd ? right : left);
        }
        const bool tie = my && near <= p.fmask;  // the top bits were equal somewhere (rare)
        if (__any_sync(0xffffffffu, tie)) {
            if (tie) at = exits + rec * packed_walk(p, b, k, xb) + (uint32_t)k * 4u;
            __syncwarp();
        }
        return at;
    }
    if (levels == 2) {
        // paired slots: a node and its two children per 16-byte record,
        // successors 4q+1 .. 4q+4; (depth+1)/2 records per walk
        const uint32_t rec = (uint32_t)stride * 16u, at0 = blk + (uint32_t)k * 16u;
        const uint32_t left = rec - 3u * at0, right = left + 2u * rec;
        uint32_t at = at0;
#pragma unroll 1  // measured: unrolling the head walk only adds instructions
        for (int l = 0; l <= p.depth; l += 2) {
            const uint4 nd = lds128(at);
            const bool r0 = !goes_left<KEYS>(lds(xb + ((nd.w & 1023u) << 7)), nd.x);
            const uint32_t f1 = nd.w >> (r0 ? 20 - 7 : 10 - 7);
            const bool r1 = !goes_left<KEYS>(lds(xb + (f1 & (1023u << 7))), r0 ? nd.z : nd.y);
            at = 4u * at + (r0 ? right : left) + (r1 ? rec : 0u);
        }
        return exits + ((at - exits) >> 2);
    }
    if (levels) {
        // implicit slots: every walk takes depth+1 steps, children 2s+1, 2s+2
        const uint32_t rec = (uint32_t)stride * 8u, at0 = blk + (uint32_t)k * 8u;
        const uint32_t left = rec - at0, right = left + rec;
        uint32_t at = at0;
#pragma unroll 1
        for (int l = 0; l <= p.depth; ++l) {
            const uint2 nd = lds64(at);
            at = 2u * at + (goes_left<KEYS>(lds(xb + ((nd.y >> 22) << 7)), nd.x) ? left : right);
        }
        return exits + ((at - exits) >> 1);
    }
    const uint32_t hn = blk + (uint32_t)k * 8u, rec = (uint32_t)stride * 8u;  // this tree's column of the block
    uint32_t hr = 0;  // head rank, then nranks + exit index
    bool busy = my;
    while (__any_sync(0xffffffffu, busy)) {  // ranked heads: until the last lane leaves
#pragma unroll
        for (int u = 0; u < 2; ++u) {  // two steps per vote
            if (busy) {
                const uint2 nd = lds64(hn + hr * rec);
                const uint32_t m = nd.y;
                uint32_t nh = goes_left<KEYS>(lds(xb + ((m >> 22) << 7)), nd.x)
                                  ? (m & FP_TARGET_MASK)
                                  : ((m >> FP_TARGET_BITS) & FP_TARGET_MASK);
                busy = nh < (uint32_t)nranks;
                if (busy && nh <= hr) {  // ranks grow along every path of a valid block
                    busy = false;
                    nh = (uint32_t)(nranks + nexits);
                }
                hr = nh;
            }
        }
    }
    const uint32_t e = hr - (uint32_t)nranks;
    return e < (uint32_t)nexits ? exits + 4u * (e * (uint32_t)stride + (uint32_t)k) : FP_NO_EXIT;
}

// The walks of one row through the paired heads of N neighbouring tree columns
// at once, each as in head_walk: the N trees' loads are in flight together.
template <bool KEYS, int N>
__device__ __forceinline__ void head_walks(const TravParams &p, uint32_t blk, uint32_t exits, int k, int stride,
                                           uint32_t xb, uint32_t exit_at[N]) {
    const uint32_t rec = (uint32_t)stride * 16u, at0 = blk + (uint32_t)k * 16u;
    const uint32_t left = rec - 3u * at0, right = left + 2u * rec;
    uint32_t at[N];
#pragma unroll
    for (int i = 0; i < N; ++i) at[i] = at0 + 16u * i;
#pragma unroll 1
    for (int l = 0; l <= p.depth; l += 2) {
        uint4 nd[N];
        uint32_t x[N];
        bool r0[N];
#pragma unroll
        for (int i = 0; i < N; ++i) nd[i] = lds128(at[i]);
#pragma unroll
        for (int i = 0; i < N; ++i) x[i] = lds(xb + ((nd[i].w & 1023u) << 7));
#pragma unroll
        for (int i = 0; i < N; ++i) {
            r0[i] = !goes_left<KEYS>(x[i], nd[i].x);
            x[i] = lds(xb + ((nd[i].w >> (r0[i] ? 20 - 7 : 10 - 7)) & (1023u << 7)));
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const bool r1 = !goes_left<KEYS>(x[i], r0[i] ? nd[i].z : nd[i].y);
            at[i] = 4u * at[i] + (r0[i] ? right : left) + (r1 ? rec : 0u) - 48u * i;  // column k + i begins 16 i later
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) exit_at[i] = exits + ((at[i] - exits) >> 2);
}

// Forests whose trees end in the interleaved heads (no super-nodes: shallow
// trees, such as boosted ones).  Every walk of a slab through a tree ends
// together, so nothing is pushed or popped: a warp takes a slab and a run of
// up to 32 of the bin's trees, keeps the row's sum of leaf values (or its votes
// for class 1 of 2) in a register over the run, and adds it to the slab's
// counter once.  A task costs the head walk, one exit word and one add; as a
// burst of its own it also paid for the claim, its division, the read of its
// value from global memory and an atomic.  FP_HEAD_TREES trees are walked at a
// time, since one tree's walk is a chain of shared-memory latencies.  256
// boosted trees of six levels, 2 M rows: 2.93 ms as bursts, 1.47 ms one tree at
// a time, 1.21, 1.19, 1.15 and 1.22 ms with 2, 3, 4 and 6 at a time (runs of
// 16; 1.145 ms with 4 in runs of 32); bound by instruction issue.
#define FP_HEAD_TREES 4

template <int MODE, bool KEYS, int HK>
__device__ __forceinline__ void walk_heads(const TravParams &p, uint32_t base, CtaShared &sh, const FpBin &bn,
                                           uint32_t blk, uint32_t exits, int buf, int rows, int G, uint32_t inv_g,
                                           int32_t *leaves, int &bad) {
    const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    // runs of 32 trees, shorter when the bin would leave warps without one
    const int run = max(1, min(32, bn.width * G / nwarps));
    const int units = (bn.width + run - 1) / run * G;
    for (;;) {
        int unit = 0;
        if (lane == 0) unit = atomicAdd(&sh.next[buf], 1);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= units) break;
        const int c = G > 1 ? (int)__umulhi((uint32_t)unit, inv_g) : unit, g = unit - c * G;
        const uint32_t xb = base + (uint32_t)g * p.slab + (uint32_t)lane * 4u;
        const int r = g * 32 + lane;
        const bool my = r < rows;
        const int k1 = min(bn.width, (c + 1) * run);
        float sum = 0.0f;
        uint32_t ones = 0;
        auto take = [&](int k, uint32_t at) {  // the row's walk through tree k ended on the exit word `at`
            if (MODE == FP_MODE_VALUES) {
                sum += __uint_as_float(lds(at));  // the exits hold the leaves' values themselves
            } else if (MODE == FP_MODE_LEAVES) {
                if (my)
                    put_leaf(p, leaves, (uint32_t)r | ((uint32_t)(bn.first_tree + k) << 11),
                             p.pheads[(bn.phead_off >> 2) + ((at - exits) >> 2)]);
            } else {
                const uint32_t cls = lds(at) & 0x7FFFFFFFu;
                if (p.C == 2) {
                    ones += cls & 1u;
                    bad |= my && cls > 1u;
                } else {
                    bad |= !vote(p, my, xb, cls);
                }
            }
        };
        int k = c * run;
        if (HK == 2) {
            for (; k + FP_HEAD_TREES <= k1; k += FP_HEAD_TREES) {
                uint32_t at[FP_HEAD_TREES];
                head_walks<KEYS, FP_HEAD_TREES>(p, blk, exits, k, bn.stride, xb, at);
#pragma unroll
                for (int i = 0; i < FP_HEAD_TREES; ++i) take(k + i, at[i]);
            }
        }
        for (; k < k1; ++k) {
            const uint32_t at = head_walk<KEYS, HK>(p, 0, blk, exits, k, bn.stride, bn.nranks, bn.nexits, xb, my);
            if (HK <= 0 && at == FP_NO_EXIT) {
                bad |= my;
                continue;
            }
            take(k, at);
        }
        if (MODE == FP_MODE_VALUES && my) add_value(p, xb, sum);
        if (MODE == FP_MODE_VOTES && my && p.C == 2 && ones)
            add_shared(xb + (((uint32_t)p.F + 1u) << 7), ones);
    }
}

// One thread: copy bin b's block into a buffer with the bulk-copy engine, its
// record beside it, and half the record of the bin that will follow it there,
// so that neither the warps that walk the bin nor the thread that refills the
// buffer wait for one from global memory.
__device__ __forceinline__ void stage_bin(const TravParams &p, CtaShared &sh, int b, uint32_t head_off,
                                          uint32_t head_bytes, int buf, uint8_t *dst) {
    const bool more = b + p.nbuf < p.n_bins;
    sh.next[buf] = 0;
    sh.done[buf] = 0;
    sh.issued[buf] += 1;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // earlier reads of dst come first
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;\n" ::"r"(
                     smem_u32(&sh.full[buf])),
                 "r"(head_bytes + (uint32_t)sizeof(FpBin) + (more ? 16u : 0u))
                 : "memory");
    bulk_copy(dst, p.heads + head_off, head_bytes, &sh.full[buf]);
    bulk_copy(&sh.desc[buf], p.bins + b, (uint32_t)sizeof(FpBin), &sh.full[buf]);
    if (more) bulk_copy(&sh.ahead[buf], p.bins + b + p.nbuf, 16u, &sh.full[buf]);
}

__device__ __forceinline__ void cta_init(CtaShared &sh) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < FP_NBUF; ++i) {
            mbar_init(&sh.full[i], 1);
            sh.issued[i] = 0;
        }
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    __syncthreads();
}

// After an abort, let this CTA's bulk copies land before it exits (bounded).
__device__ __forceinline__ void cta_finish(CtaShared &sh) {
    if (threadIdx.x == 0 && sh.abort) {
        for (int i = 0; i < FP_NBUF; ++i) {
            if (sh.issued[i] == 0) continue;
            const uint32_t parity = (uint32_t)(sh.issued[i] - 1) & 1u;
            for (int spin = 0; spin < FP_SPIN_LIMIT && !mbar_try_wait(&sh.full[i], parity); ++spin) {
            }
        }
    }
}

// Votes and classes of a tile whose splits were added up in p.acc (class 0:
// the trees that voted for no other): a row's classes are spread over a group
// of lanes, each reading its own (a thread per row reads them one after
// another, an L2 latency for every few classes), and the maximum is found by
// shuffles, lowest class on ties.  All threads of the CTA call this.
__device__ __forceinline__ void finish_rows(const TravParams &p, int64_t row0, int rows) {
    const int C = p.C;
    int width = 1;  // lanes per row
    while (width < C && width < 32) width *= 2;
    const int lane = threadIdx.x & 31, sub = lane & (width - 1);
    const int per_warp = 32 / width, per_cta = per_warp * (blockDim.x >> 5);
    for (int i0 = 0; i0 < rows; i0 += per_cta) {
        const int rr = i0 + (int)(threadIdx.x >> 5) * per_warp + lane / width;
        const int64_t at = (row0 + rr) * C;
        uint32_t bv = 0, others = 0;
        int best = 0;
        if (rr < rows) {
            for (int c = sub; c < C; c += width) {
                if (c == 0) continue;
                const uint32_t x = __ldcg(p.acc + at + c);
                others += x;
                if (x > bv) { bv = x; best = c; }
                if (p.out_votes && p.out_votes != p.acc) p.out_votes[at + c] = x;
            }
        }
        for (int m = width >> 1; m > 0; m >>= 1) {
            const uint32_t ov = __shfl_xor_sync(0xffffffffu, bv, m);
            const int oc = __shfl_xor_sync(0xffffffffu, best, m);
            others += __shfl_xor_sync(0xffffffffu, others, m);
            if (ov > bv || (ov == bv && oc < best)) { bv = ov; best = oc; }
        }
        if (rr < rows && sub == 0) {
            const uint32_t v0 = (uint32_t)p.T - others;
            if (p.out_votes) p.out_votes[at] = v0;
            if (p.out_class) p.out_class[row0 + rr] = v0 >= bv ? 0 : best;
        }
    }
}

// Votes and classes of an unsplit tile with many classes.  A thread per row
// keeps two of 32 warps busy in a 64-row tile, waits for shared memory once per
// class, and writes a row's votes 4 * C bytes apart.  So: the classes of a slab
// are spread over the warps, which meet in two words of the row that the walks
// have finished with, its first feature (the best class, as votes << 9 |
// 511 - class, so that the lowest wins ties; at most 2^20 trees and 512 classes)
// and its counter of class 0 (the others' sum, then its own votes); and the
// votes go out 8 classes of 4 rows at a time: whole sectors, at a quarter of
// the bank conflicts that 32 classes of one row would have.  300,000 rows, 64
// trees, votes and classes: 512 classes 5.90 -> 5.70 ms, 200 2.11 -> 1.99, 50
// 0.849 -> 0.826; classes alone: 512 5.68 -> 5.48 ms, 200 1.91 either way, 50
// 0.797 -> 0.801.  With 10 classes (128 trees, 100,000 rows) its two barriers
// cost more than it saves, 585 -> 598 us.  All threads of the CTA call this.
// Not inlined, to keep the walks as they are.
__device__ __forceinline__ bool many_classes(const TravParams &p) { return p.C >= (p.out_votes ? 32 : 128); }

__device__ __noinline__ void finish_many_classes(const TravParams &p, uint32_t at0, int64_t row0, int rows) {
    const int C = p.C, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int groups = (rows + 31) >> 5;
    const uint32_t zero_at = (uint32_t)p.F << 7;  // of a slab: its counters of class 0
    for (int g = warp; g < groups; g += nwarps)
        asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(at0 + (uint32_t)g * p.slab + (uint32_t)lane * 4u), "r"(0u) : "memory");
    __syncthreads();
    const int parts = max(1, min(nwarps / groups, (C + 6) / 8)), per = (C - 2 + parts) / parts;
    for (int u = warp; u < groups * parts; u += nwarps) {
        const int part = u / groups, g = u - part * groups;
        const uint32_t at = at0 + (uint32_t)g * p.slab + (uint32_t)lane * 4u;
        const int c1 = min(C, 1 + (part + 1) * per);
        uint32_t others = 0, best = 0;
#pragma unroll 4
        for (int c = 1 + part * per; c < c1; ++c) {
            const uint32_t v = lds(at + zero_at + ((uint32_t)c << 7));
            others += v;
            best = max(best, v << 9 | (uint32_t)(511 - c));
        }
        add_shared(at + zero_at, others);
        asm volatile("red.shared.max.u32 [%0], %1;\n" ::"r"(at), "r"(best) : "memory");
    }
    __syncthreads();
    for (int rr = tid; rr < rows; rr += blockDim.x) {
        const uint32_t at = at0 + (uint32_t)(rr >> 5) * p.slab + (uint32_t)(rr & 31) * 4u;
        const uint32_t v0 = (uint32_t)p.T - lds(at + zero_at), best = lds(at);
        asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(at + zero_at), "r"(v0) : "memory");
        if (p.out_class) p.out_class[row0 + rr] = v0 >= (best >> 9) ? 0 : 511 - (int)(best & 511u);
    }
    if (!p.out_votes) return;
    __syncthreads();
    const int chunks = (C + 7) >> 3;
    uint32_t *out = p.out_votes + row0 * C;
    for (int u = warp; u < ((rows + 3) >> 2) * chunks; u += nwarps) {
        const int quad = u / chunks, c = (u - quad * chunks) * 8 + (lane & 7), rr = quad * 4 + (lane >> 3);
        if (c < C && rr < rows)
            out[(int64_t)rr * C + c] =
                lds(at0 + (uint32_t)(rr >> 5) * p.slab + (uint32_t)(rr & 31) * 4u + zero_at + ((uint32_t)c << 7));
    }
}

// A split's votes for class 0, where votes alone are asked for: no CTA looks at
// the tile again, so each split adds its own (its trees less the votes for the
// others).  Not inlined, to keep the walks of the kernels that call it as they
// are.
__device__ __noinline__ void add_class0(const TravParams &p, const CtaShared &sh, uint32_t at0, int64_t row0,
                                        int rows) {
    const int end = sh.bin1 < p.n_bins ? p.bins[sh.bin1].first_tree : p.T;
    const uint32_t trees = (uint32_t)(end - p.bins[sh.bin0].first_tree);
    for (int rr = threadIdx.x; rr < rows; rr += blockDim.x) {
        const uint32_t at = at0 + (uint32_t)(rr >> 5) * p.slab + ((uint32_t)p.F << 7) + (uint32_t)(rr & 31) * 4u;
        uint32_t rest = trees;
        for (int c = 1; c < p.C; ++c) rest -= lds(at + ((uint32_t)c << 7));
        if (rest) atomicAdd(p.acc + (row0 + rr) * p.C, rest);
    }
}

// 8 features of a row from a 32-byte aligned address, past L1.
__device__ __forceinline__ void load_row8(const float4 *at, float4 &a, float4 &b) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(at));
}

// The start of an item: its bins and their first blocks in flight, its rows in
// shared memory as order keys, its counters cleared.
template <int MODE, int DK>
__device__ __forceinline__ void begin_item(const TravParams &p, uint8_t *smem, CtaShared &sh, int64_t tile, int split,
                                        uint32_t hbuf0) {
    const int F = p.F, VR = MODE == FP_MODE_LEAVES ? 0 : (MODE == FP_MODE_VALUES ? 1 : p.C);
    const uint32_t slab = p.slab;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5, nbuf = p.nbuf;
    const int64_t row0 = tile * p.R;
    const int rows = (int)(p.n - row0 < (int64_t)p.R ? p.n - row0 : (int64_t)p.R);
    const int G = (rows + 31) >> 5;
    if (tid < 32) {
        int b0 = 0, b1 = p.n_bins;
        if (p.n_splits > 1 && p.n_splits == p.n_passes) {
            const FpPass ps = p.passes[split];
            b0 = ps.bin_begin;
            b1 = ps.bin_end;
        } else if (p.n_splits > 1) {
            b0 = split * p.split_bins + min(split, p.split_more);
            b1 = b0 + p.split_bins + (split < p.split_more ? 1 : 0);
        }
        if (tid == 0) {
            sh.bin0 = b0;
            sh.bin1 = b1;
            sh.tile = tile;
            uint32_t ph = 0;
            for (int i = 0; i < FP_NBUF; ++i) ph |= ((uint32_t)sh.issued[i] & 1u) << i;
            sh.phases = ph;
        }
        __syncwarp();
        if (tid < nbuf && b0 + tid < b1) {  // a lane per buffer, so that the records' latencies overlap
            const FpBin bn = p.bins[b0 + tid];
            stage_bin(p, sh, b0 + tid, bn.head_off, bn.head_bytes, tid, smem + hbuf0 + tid * p.head_smem);
        }
    }
    {
        // lane = row of a slab, 8 features at a time: loads along the row, and
        // each store of a warp fills the 32 columns of one feature.  The
        // (slab, 8 features) units are dealt out to all warps, so that a tile
        // of few wide rows (784 features, 64 rows) is staged by every warp,
        // not by two.  A lane's 8 features are one 32-byte load where its
        // address allows it: each sector is asked for once and used whole, and
        // nothing is left for L1 to hold.  64-row tiles of 784 features (250 k
        // rows): 1407 us, 1467 with four 16-byte loads a lane (16 features),
        // 1435 with two (8 features); more loads in flight a lane, or runs of
        // neighbouring features to one warp, 1480 to 1810.
        const float *src = p.X + row0 * F;
        const bool vec_rows = (F & 3) == 0 && (reinterpret_cast<uintptr_t>(p.X) & 15) == 0;
        const int fblocks = (F + 7) >> 3;
        for (int u = warp; u < G * fblocks; u += nwarps) {
            const int fq = u / G, g = u - fq * G, f0 = fq * 8;
            const int r = g * 32 + lane;
            if (r >= rows) continue;
            const float *rp = src + (int64_t)r * F + f0;
            uint32_t *dst = reinterpret_cast<uint32_t *>(smem + (uint32_t)g * slab) + f0 * 32 + lane;
            auto put4 = [&](int k, float4 v) {
                uint32_t *d = dst + 128 * k;
                d[0] = staged<DK>(p, v.x);
                d[32] = staged<DK>(p, v.y);
                d[64] = staged<DK>(p, v.z);
                d[96] = staged<DK>(p, v.w);
            };
            const float4 *rq = reinterpret_cast<const float4 *>(rp);
            if (vec_rows && f0 + 8 <= F) {
                float4 v[2];
                if ((reinterpret_cast<uintptr_t>(rq) & 31) == 0) {
                    load_row8(rq, v[0], v[1]);
                } else {  // rows of 4, 12, ... features: every second one; or rows from the middle of a sector
                    v[0] = __ldg(rq);
                    v[1] = __ldg(rq + 1);
                }
                put4(0, v[0]);
                put4(1, v[1]);
            } else if (vec_rows) {
                put4(0, __ldg(rq));  // the last 4 of F
            } else {
                const int m = F - f0 < 8 ? F - f0 : 8;
#pragma unroll 4
                for (int k = 0; k < m; ++k) dst[32 * k] = staged<DK>(p, __ldg(rp + k));
            }
        }
    }
    for (int u = warp; u < G * VR; u += nwarps) {
        const int g = u / VR;
        reinterpret_cast<uint32_t *>(smem + (uint32_t)g * slab)[(F + u - g * VR) * 32 + lane] = 0;
    }
}

// The end of an item, once every warp has finished its walks.
template <int MODE>
__device__ __forceinline__ void end_item(const TravParams &p, uint8_t *smem, CtaShared &sh) {
    constexpr bool VALUES = MODE == FP_MODE_VALUES;
    const int F = p.F, C = p.C, tid = threadIdx.x;
    const uint32_t slab = p.slab;
    const int64_t base = sh.tile * p.R;
    const int nrows = (int)(p.n - base < (int64_t)p.R ? p.n - base : (int64_t)p.R);

    // 5. the tile's results: from this CTA's shared memory, or, for a tile that
    //    is cut into several splits, added up in global memory, where the CTA
    //    that finishes the tile last completes it
    const bool alone = p.n_splits == 1;
    const bool go = !*(volatile int *)&sh.abort;
    const uint32_t at0 = smem_u32(smem);
    auto counter = [&](int rr, int c) {  // where a row's counter c lies
        return at0 + (uint32_t)(rr >> 5) * slab + ((uint32_t)(F + c) << 7) + (uint32_t)(rr & 31) * 4u;
    };
    auto last_split = [&]() {  // true in the CTA that finishes the tile last
        __threadfence();
        __syncthreads();
        if (tid == 0) sh.last = atomicAdd(p.tile_done + sh.tile, 1u) == (unsigned)(p.n_splits - 1);
        __syncthreads();
        if (sh.last) __threadfence();
        return sh.last != 0;
    };
    if (VALUES && go) {
        if (alone) {
            for (int rr = tid; rr < nrows; rr += blockDim.x)
                p.out_val[base + rr] = p.vbias + p.vscale * __uint_as_float(lds(counter(rr, 0)));
        } else {
            float *dst = p.acc_val + base;
            for (int rr = tid; rr < nrows; rr += blockDim.x) {
                const float v = __uint_as_float(lds(counter(rr, 0)));
                if (v != 0.0f) atomicAdd(dst + rr, v);
            }
            if (last_split())
                for (int rr = tid; rr < nrows; rr += blockDim.x)
                    p.out_val[base + rr] = p.vbias + p.vscale * __ldcg(dst + rr);
        }
    }
    if (MODE == FP_MODE_VOTES && go) {
        if (alone && many_classes(p)) {
            finish_many_classes(p, at0, base, nrows);
        } else if (alone) {  // a thread per row; class 0 has the votes that no other class got
            for (int rr = tid; rr < nrows; rr += blockDim.x) {
                uint32_t *d = p.out_votes ? p.out_votes + (base + rr) * C : nullptr;
                uint32_t rest = (uint32_t)p.T, bv = 0;
                int best = 0;
                for (int c = 1; c < C; ++c) {
                    const uint32_t v = lds(counter(rr, c));
                    rest -= v;
                    if (v > bv) { bv = v; best = c; }
                    if (d) d[c] = v;
                }
                if (d) d[0] = rest;
                if (p.out_class) p.out_class[base + rr] = rest >= bv ? 0 : best;
            }
        } else {
            // a warp per 32 rows and class: all of the CTA's warps have some,
            // however few rows the tile has
            const int groups = (nrows + 31) >> 5, lane = tid & 31;
            for (int u = tid >> 5; u < groups * (C - 1); u += blockDim.x >> 5) {
                const int c = u / groups + 1, rr = (u - (c - 1) * groups) * 32 + lane;
                const uint32_t v = rr < nrows ? lds(counter(rr, c)) : 0u;
                if (v) atomicAdd(p.acc + (base + rr) * C + c, v);
            }
            if (p.tile_done) {
                if (last_split()) finish_rows(p, base, nrows);
            } else {
                add_class0(p, sh, at0, base, nrows);
            }
        }
    }
}

// One work item: one of the parts (splits) that the forest's bins are cut
// into, and one observation tile.  The item's bins go through the buffers in
// turn; the k-th copy ever issued into a buffer completes its barrier's phase
// k, and every warp keeps the parities it waits for next (phases, from the
// buffers' copy counts when the item starts).  Counting per buffer keeps the
// phases right when items of forests with different nbuf share a CTA.  Every
// warp waits for every bin's block, also for one it has no unit in: a warp
// that ran ahead of a buffer's phases could not tell them apart.
// HEADS: the forest has no super-nodes (walk_heads); its own build, since the
// two walks in one kernel cost the other 8 % more instructions.
template <int MODE, int DK, int HK, bool HEADS>
__device__ __forceinline__ void run_item(const TravParams &p, int64_t tile, int split, uint8_t *smem,
                                         CtaShared &sh) {
    constexpr bool D3 = DK >= 3;  // rows and thresholds are (remapped) order keys
    constexpr bool LEAVES = MODE == FP_MODE_LEAVES, VALUES = MODE == FP_MODE_VALUES;
    const int levels = HK >= 0 ? HK : p.levels;
    const int R = p.R;
    const uint32_t slab = p.slab;
    const uint32_t hbuf0 = (uint32_t)(R >> 5) * slab;  // nbuf bin-block buffers from here, head_smem bytes each
    const int nbuf = p.nbuf;
    const int tid = threadIdx.x, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int lane = __shfl_sync(0xffffffffu, tid & 31, tid & 31);
    // through a shuffle, which the compiler cannot redo in every step
    const uint32_t base = __shfl_sync(0xffffffffu, smem_u32(smem), lane);
    const uint32_t ring = base + hbuf0 + (uint32_t)(nbuf * p.head_smem + warp * FP_RING * 8);
    const unsigned lt_mask = __shfl_sync(0xffffffffu, (1u << lane) - 1u, lane);

    // A CTA that gave up a wait skips its remaining items; each one records
    // the timeout in its own forest's status, since its outputs stay unwritten
    // (sh.abort is uniform here: it changes only inside the bin loop, and the
    // previous item ended with a CTA barrier).
    if (*(volatile int *)&sh.abort) {
        if (tid == 0) report(p.status, FP_ERR_FLAG_TIMEOUT);
        return;
    }
    const int64_t row0 = tile * R;
    const int rows = (int)(p.n - row0 < (int64_t)R ? p.n - row0 : (int64_t)R);
    const int G = (rows + 31) >> 5;  // slabs in use
    int32_t *const leaves = LEAVES ? p.out_leaf + row0 * p.T : nullptr;

    begin_item<MODE, DK>(p, smem, sh, tile, split, hbuf0);
    __syncthreads();

    LaneTask L = idle_task(base);
    uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // feature 0 in every slot
    Pending pend, hpend;  // of the last deep step, of the last burst (values mode)
    pend.on = hpend.on = false;
    pend.at = hpend.at = 0;
    pend.word = hpend.word = 0;
    int head = 0, tail = 0;  // warp-uniform ring cursors
    bool carried = false;    // the lanes' loads were issued in the bin before

    // unit u of a bin is slab u % G of its tree u / G: ceil(2^32 / G) divides by G
    const uint32_t inv_g = G > 1 ? 0xFFFFFFFFu / (uint32_t)G + 1u : 0u;

    uint32_t phases = sh.phases;  // bit b: the phase parity that buffer b's next block completes
    int buf = 0;
    for (int b = sh.bin0; b < sh.bin1; ++b) {
        {  // wait until the bin's block has landed
            const uint32_t parity = (phases >> buf) & 1u;
            phases ^= 1u << buf;
            bool ok = false;
            for (int spin = 0; spin < p.spin_limit; ++spin) {
                if (*(volatile int *)&sh.abort) break;
                if (mbar_try_wait(&sh.full[buf], parity) && !p.stall) {
                    ok = true;
                    break;
                }
            }
            if (!__all_sync(0xffffffffu, ok)) {
                if (lane == 0 && !*(volatile int *)&sh.abort) {
                    report(p.status, FP_ERR_FLAG_TIMEOUT);
                    *(volatile int *)&sh.abort = 1;
                }
                break;
            }
        }
        const FpBin bn = sh.desc[buf];
        const int stride = bn.stride, nranks = bn.nranks, nexits = bn.nexits;
        const uint32_t blk = base + hbuf0 + (uint32_t)(buf * p.head_smem);
        const uint32_t exits = blk + (uint32_t)(nranks * stride * (levels == 2 ? 16 : (levels == 3 ? 4 : 8)));

        if (HEADS) walk_heads<MODE, D3, HK>(p, base, sh, bn, blk, exits, buf, rows, G, inv_g, leaves, L.bad);
        const int units = bn.width * G;
        if (!HEADS) {
            if (carried && p.step_bins) {  // the load of the bin before has had that bin's time to arrive
                settle<MODE>(p, leaves, pend);
                if (__any_sync(0xffffffffu, L.ref != FP_NO_TASK)) deep_finish<MODE, DK>(p, L, pend, w);
                pop_tasks<MODE>(p, base, ring, head, tail, L, lt_mask);
                carried = false;
            }
            for (;;) {
                // deep steps until the ring runs low
                if (!carried) ld_super(p.deep, L.ref, w);
                carried = false;
                settle<MODE>(p, leaves, hpend);
                while (__any_sync(0xffffffffu, tail - head > p.refill)) {
                    settle<MODE>(p, leaves, pend);
                    deep_finish<MODE, DK>(p, L, pend, w);
                    pop_tasks<MODE>(p, base, ring, head, tail, L, lt_mask);
                    ld_super(p.deep, L.ref, w);
                }
                int unit = 0;
                if (lane == 0) unit = atomicAdd(&sh.next[buf], 1);
                unit = __shfl_sync(0xffffffffu, unit, 0);
                if (__any_sync(0xffffffffu, unit >= units)) break;  // all taken
                const int uk = G > 1 ? (int)__umulhi((uint32_t)unit, inv_g) : unit, ug = unit - uk * G;
                const uint32_t xb = base + (uint32_t)ug * slab + (uint32_t)lane * 4u;
                const int r2 = ug * 32 + lane;
                const bool my = r2 < rows;
                const uint32_t at =
                    head_walk<D3, HK>(p, b, blk, exits, uk, stride, nranks, nexits, xb, my);
                const bool ok = HK > 0 || at != FP_NO_EXIT;
                const uint32_t er = ok ? lds(at) : FP_NO_CLASS;
                const bool push = my && !(er & FP_REF_LEAF);
                if (my && !push) {  // a leaf in the head, or right below it
                    const uint32_t cls = er & 0x7FFFFFFFu;
                    if (LEAVES) {
                        L.bad |= !ok;
                        if (ok)
                            put_leaf(p, leaves, (uint32_t)r2 | ((uint32_t)(bn.first_tree + uk) << 11),
                                     __ldg(p.pheads + (bn.phead_off >> 2) + ((at - exits) >> 2)));
                    } else if (VALUES) {
                        L.bad |= cls >= p.n_vals;
                        hpend.on = cls < p.n_vals;
                        hpend.at = xb;
                        if (hpend.on) hpend.word = __float_as_uint(__ldg(p.leaf_val + cls));
                    } else {
                        L.bad |= !vote(p, true, xb, cls);
                    }
                }
                const unsigned pm = __ballot_sync(0xffffffffu, push);
                if (push)
                    sts64(ring + (uint32_t)((tail + __popc(pm & lt_mask)) & (FP_RING - 1)) * 8u, er,
                          LEAVES ? (uint32_t)r2 | ((uint32_t)(bn.first_tree + uk) << 11) : xb);
                tail += __popc(pm);
                __syncwarp();
                settle<MODE>(p, leaves, pend);
                // where nearly all paths end in the heads, most bursts find no
                // lane with a task: 16 trees of 80 nodes, 400,000 rows: 87.0 us
                // with the step taken all the same, 80.0 without; the vote
                // costs forests of deep trees 0.3 %
                if (__any_sync(0xffffffffu, L.ref != FP_NO_TASK)) deep_finish<MODE, DK>(p, L, pend, w);
                pop_tasks<MODE>(p, base, ring, head, tail, L, lt_mask);
            }
        }
        // this warp reads the bin's block no more; the last warp refills the buffer
        __syncwarp();
        if (lane == 0) {
            const int done = atomicAdd(&sh.done[buf], 1);
            if (done == nwarps - 1 && b + nbuf < sh.bin1 && !*(volatile int *)&sh.abort) {
                const uint4 next = sh.ahead[buf];
                stage_bin(p, sh, b + nbuf, next.x, next.y, buf, smem + hbuf0 + buf * p.head_smem);
            }
        }
        __syncwarp();
        // the load in flight is used here, or, where a bin has fewer units than
        // there are warps, carried into the next bins: waiting for it in every
        // bin would cost most warps an L2 latency for nothing (64 trees, 13
        // nodes a walk, 100,000 rows of 100 features: 175 us, 196 with a step
        // in every bin).  Trees of many levels below the heads (step_bins)
        // need those steps, which else all come after the last bin: 41 trees,
        // 22 nodes a walk, 3777 rows: 22.7 us, 26.6 without.
        carried = units < nwarps;
        if (!HEADS && !carried && __any_sync(0xffffffffu, L.ref != FP_NO_TASK)) {
            settle<MODE>(p, leaves, pend);
            deep_finish<MODE, DK>(p, L, pend, w);
            pop_tasks<MODE>(p, base, ring, head, tail, L, lt_mask);
        }
        if (++buf == nbuf) buf = 0;
    }
    const bool aborted = *(volatile int *)&sh.abort != 0;
    if (!HEADS && carried && !aborted) {
        settle<MODE>(p, leaves, pend);
        deep_finish<MODE, DK>(p, L, pend, w);
    }
    // drain: the item's last pending and running tasks
    for (; !HEADS && !aborted;) {
        __syncwarp();
        pop_tasks<MODE>(p, base, ring, head, tail, L, lt_mask);
        if (!__any_sync(0xffffffffu, L.ref != FP_NO_TASK)) break;
        ld_super(p.deep, L.ref, w);
        settle<MODE>(p, leaves, pend);
        deep_finish<MODE, DK>(p, L, pend, w);
    }
    settle<MODE>(p, leaves, pend);
    settle<MODE>(p, leaves, hpend);
    if (L.bad) report(p.status, FP_ERR_FLAG_DEVICE);
    __syncthreads();

    end_item<MODE>(p, smem, sh);
    __syncthreads();  // the next item reuses shared memory
}

// Forests with leaf values and no super-nodes: every exit of the heads becomes
// the value of the leaf that it names (once, after the upload), so that a
// walk ends on the value instead of on its slot in a table in global memory.
// One block per bin.
__global__ void fp_inline_values_kernel(uint8_t *heads, const FpBin *bins, const float *leaf_val, uint32_t n_vals,
                                        uint32_t node_bytes) {
    const FpBin bn = bins[blockIdx.x];
    uint32_t *exits = reinterpret_cast<uint32_t *>(heads + bn.head_off + (size_t)bn.nranks * bn.stride * node_bytes);
    for (int i = threadIdx.x; i < bn.nexits * bn.stride; i += blockDim.x) {
        const uint32_t slot = exits[i] & 0x7FFFFFFFu;
        exits[i] = slot < n_vals ? __float_as_uint(leaf_val[slot]) : 0u;  // entries that no walk reaches: 0
    }
}

// Level heads of a forest with order keys (three-level super-nodes), rewritten
// once after the upload: one word per node, the top bits of its key over its
// feature, in breadth-first slots, tree by tree side by side as in the packed
// block.  A 16-byte record of two levels costs a warp at random slots about
// nine wavefronts of the load/store pipe, a word one to three (none of the
// upper levels' 32 words share a bank), and the block is a seventh smaller.
// Heads of ten levels: regression forest, 1 M rows, 3.01 -> 2.86 ms; 256 trees
// of 78.8k nodes, 4 M rows, 24.46 -> 24.00 ms.  One block per bin; bins and
// blocks to write, bins and blocks to read.
__global__ void fp_compact_heads_kernel(uint8_t *out, const FpBin *out_bins, const uint8_t *heads, const FpBin *bins,
                                        int32_t kind, uint32_t fmask) {
    const FpBin src = bins[blockIdx.x], dst = out_bins[blockIdx.x];
    const uint8_t *from = heads + src.head_off;
    uint32_t *to = reinterpret_cast<uint32_t *>(out + dst.head_off);
    const int nodes = dst.nranks * dst.stride;
    for (int i = threadIdx.x; i < nodes; i += blockDim.x) {
        const int s = i / dst.stride, k = i - s * dst.stride;
        uint32_t thr, feature;
        if (kind == 2) {
            // slot s of an even level opens a record, its children lie in it
            const int level = 31 - __clz(s + 1), top = level & 1 ? (s - 1) / 2 : s, lt = level & ~1;
            const int q = ((1 << lt) - 1) / 3 + top - ((1 << lt) - 1), c = level & 1 ? 2 - (s & 1) : 0;
            const uint32_t *rec = reinterpret_cast<const uint32_t *>(from + ((size_t)q * src.stride + k) * 16);
            thr = rec[c];
            feature = (rec[3] >> (10 * c)) & 1023u;
        } else {
            const uint32_t *rec = reinterpret_cast<const uint32_t *>(from + ((size_t)s * src.stride + k) * 8);
            thr = rec[0];
            feature = rec[1] >> 22;
        }
        to[i] = (thr & ~fmask) | feature;
    }
    const uint32_t *exits =
        reinterpret_cast<const uint32_t *>(from + (size_t)src.nranks * src.stride * (kind == 2 ? 16 : 8));
    const int words = (int)(dst.head_bytes / 4);
    for (int i = threadIdx.x; nodes + i < words; i += blockDim.x)
        to[nodes + i] = i < src.nexits * src.stride ? exits[i] : 0u;
}

// MINB = 1: one CTA of up to 1024 threads per SM (up to 64 registers a thread);
// MINB = 2: CTAs of up to 768 threads, at most 42 registers a thread, so that
// two 24-warp or three 16-warp CTAs share an SM when shared memory allows:
// more warps to hide the latency of the dependent loads of each walk.
template <int MODE, int MINB, int DK, int HK, bool HEADS>
__global__ void __launch_bounds__(MINB == 1 ? 1024 : 768, MINB) fp_traverse_kernel(const __grid_constant__ TravParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ CtaShared sh;
    cta_init(sh);
    // all tiles of a split, then the next one's, so that the CTAs walk the same
    // bins at a time
    int64_t tile = blockIdx.x;
    int split = 0;
    for (;;) {
        for (; tile >= p.n_tiles && split < p.n_splits; tile -= p.n_tiles) ++split;
        if (split >= p.n_splits) break;
        run_item<MODE, DK, HK, HEADS>(p, tile, split, smem, sh);
        tile += gridDim.x;
    }
    cta_finish(sh);
}

// Several forests and batches in one persistent launch: the work items of
// all batches form one list (batch by batch, split by split within a batch),
// handed out to CTAs through a global counter so uneven batches balance; how
// long items are is chosen for the launch (fp_device.cu).
#define FP_MAX_BATCH 32

struct BatchParams {
    int32_t k;
    int64_t item_begin[FP_MAX_BATCH + 1];
    TravParams p[FP_MAX_BATCH];
    unsigned long long *work;  // zeroed before the launch
};

// KIND: 2, 3 or 4 when every forest of the launch has that kind of
// super-node (one walk compiled in), 0 for a mix (all, chosen per item).  HK:
// the head kind when all forests share it (0 ranked, 1, 2, 3), else -1.
template <int KIND, int HK>
__global__ void __launch_bounds__(1024, 1) fp_traverse_batched_kernel(const __grid_constant__ BatchParams bp) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ CtaShared sh;
    cta_init(sh);
    const int64_t total = bp.item_begin[bp.k];
    for (;;) {
        if (threadIdx.x == 0) sh.next_item = (long long)atomicAdd(bp.work, 1ull);
        __syncthreads();
        const int64_t item = sh.next_item;
        __syncthreads();
        if (item >= total) break;
        int j = 0;
        while (j + 1 < bp.k && bp.item_begin[j + 1] <= item) ++j;
        const int64_t own = item - bp.item_begin[j];
        const int split = (int)(own / bp.p[j].n_tiles);
        const int64_t tile = own - split * bp.p[j].n_tiles;
        if (KIND == 3 || (KIND == 0 && bp.p[j].deep_kind == 3))
            run_item<FP_MODE_VOTES, 3, HK, false>(bp.p[j], tile, split, smem, sh);
        else if (KIND == 4 || (KIND == 0 && bp.p[j].deep_kind == 4))
            run_item<FP_MODE_VOTES, 4, HK, false>(bp.p[j], tile, split, smem, sh);
        else
            run_item<FP_MODE_VOTES, 2, HK, false>(bp.p[j], tile, split, smem, sh);
    }
    cta_finish(sh);
}
