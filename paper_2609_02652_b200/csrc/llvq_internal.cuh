// Internal declarations shared by the translation units of the library (not part of the ABI).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "../../include/llvq.h"
#include "llvq_tables.h"
#include "llvq_unrank.cuh"

namespace llvq {

// Geometry of the 14-byte layout (see include/llvq.h).
constexpr int kRowsPerGroup = 32;
constexpr int kCellBytes = 448;        // 32 rows x 14 bytes
constexpr int kTileCells = 4;
constexpr int kTileBytes = 1792;
constexpr int kOneHotCellBytes = 640;  // 32 rows x 20 bytes
constexpr int kCell13Bytes = 416;      // 13-byte layout: 32 rows x 13 bytes
constexpr int kTile13Bytes = 1664;
constexpr int kTile10Bytes = 1280;     // 10-byte layout: 9 words a lane and 128 header bytes a tile; its leftover blocks are 13-byte cells
constexpr int kMaxGridCtas = 256;      // the GEMV launches one CTA a multiprocessor; more multiprocessors than this share the work of 256

// The 10-byte layout's buffer: row groups, then (128-byte aligned) the index, then (128-byte aligned) the exception table.
__host__ __device__ inline size_t overlay_group_bytes(int64_t nb) { return (size_t)(nb / kTileCells) * kTile10Bytes + (size_t)(nb % kTileCells) * kCell13Bytes; }
__host__ __device__ inline size_t overlay_index_offset(int64_t rows, int64_t nb) {
    return ((size_t)((rows + kRowsPerGroup - 1) / kRowsPerGroup) * overlay_group_bytes(nb) + 127) / 128 * 128;
}
__host__ __device__ inline size_t overlay_table_offset(int64_t rows, int64_t nb) {
    // the index: one entry a tile, and one more
    return overlay_index_offset(rows, nb) + ((size_t)((rows + kRowsPerGroup - 1) / kRowsPerGroup * (nb / kTileCells) + 1) * 4 + 127) / 128 * 128;
}

struct DeviceTables {
    const ClassDesc *desc;           // num_classes
    const float *cls_scale;          // 512
    const uint32_t *cls_parity;      // 512
    const float *cls_value;          // 512 x 8
    const uint8_t *cls_dist;         // 512 x 8
    const float2 *cls_block;         // 512 x {1 / (4 sqrt m), parity - 16}
    const uint4 *lane_table;         // 32 x {b0, b1, b2, xs}: a lane's operand offsets in two consecutive x records
    uint64_t num_points;
};

// n / d by one multiply-high and one shift, for 0 <= n < 2^31 and a divisor fixed per launch
// (mul = floor(2^(31+l) / d) + 1, shift = l - 1, l = ceil(log2 d); mul = 0 stands for d = 1)
struct FastDiv {
    uint32_t mul, shift;
};
inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f = {0u, 0u};
    if (d <= 1) return f;
    uint32_t l = 0;
    while ((1ull << l) < d) l++;
    f.mul = (uint32_t)(((1ull << (31 + l)) / d) + 1);
    f.shift = l - 1;
    return f;
}

struct GemvProblemDev {
    const uint8_t *layout;
    const __half *row_scale;
    float *y;
    int rows;
    int group_begin;   // index of this matrix's first row group in the concatenation
    float gain0, gain1;
    int qexp_base;     // log2 of this matrix's fixed-point quantum, before the exponent of max |x| is added
    const uint32_t *exc_index;   // 10-byte layout: entry i = exception-table entries of this matrix's tiles before tile i (row group by row group)
    const uint4 *exc_table;      // 10-byte layout: the exact records the short records leave out
};

// A CTA's share of a launch, planned on the host: its first unit, and the blocks of x [blk_lo, blk_hi) its units touch
// (the whole panels its range of units meets).  Eight bytes, because they are parameters of every launch.
struct CtaShare {
    int first;
    uint16_t blk_lo, blk_hi;
};

// What gemv_plan works out from the shapes of a launch alone.
struct GemvPlan {
    int units_base, units_rem;   // total_units divided by the warps of the grid (the one-hot arm's order)
    int panel, npanels;          // unit columns a panel, panels (the 14-byte layout's order of work)
    FastDiv div_panel, div_last; // by panel, by the last panel's width
    int xblocks;                 // most blocks of x any CTA needs
    uint32_t group_bytes;        // bytes of a row group's records
    int rot_span;                // most coordinates of the rotation blocks any CTA's blocks of x lie in
    int rot_keep;                // most of them any CTA keeps after the first stages (rot_first)
    CtaShare cta[kMaxGridCtas + 1];    // the share of every CTA of the grid; [grid].first is the total
};

// One launch's own: the caller's arguments and the context's tables.  The matrices come first and the plan behind: with the plan's
// 2 KB ahead of them a decoder layer's launches take 1.5 % longer (4096 to 12288: 87.3 us a layer, 86.0 this way).
struct GemvCall {
    GemvProblemDev prob[LLVQ_MAX_GROUP];
    int nprob;
    const __half *x;             // batch vectors of 24 nb halves, one after the other
    int batch;                   // activation vectors of the launch (1; up to LLVQ_MAX_BATCH through llvq_gemv_batch)
    int y_stride;                // floats between the outputs of consecutive vectors
    int nb, tiles, tail_cells;
    int units;             // units a row group: tiles, plus one for the nb mod 4 last columns
    int total_groups;
    int total_units;       // total_groups * units
    unsigned long long *accum;   // total_groups x 32 fixed-point row accumulators (context scratch, zero between launches)
    const float *cls_value;
    const float2 *cls_block;     // 512 x {1 / (4 sqrt m), parity - 16 as an integer's bits}; zeros for an unused class slot
    const uint4 *lane_table;     // 32 x this lane's offsets of its operand words in the x records of a half-step
    int *error;               // set when a bounded wait ran out
    // rotation of x inside the GEMV (llvq_gemv_rotated); rot_log2 = 0 means none
    int rot_log2;             // log2 of the rotation's block length (3..)
    int rot_n;                // coordinates rotated: a multiple of the block length, at most 24 nb
    const uint32_t *rot_negate;   // sign-flip bits, or null
    double rot_scale;         // 2^1008 / sqrt(block length): the sums are those of x times 2^-1008 (rot_widen)
    float shell_inv_norm[16];         // [m] = 1 / (4 sqrt m)
};

struct GemvParams : GemvCall, GemvPlan {};

struct GemvLaunch {
    int grid;
    size_t smem;
};
// The rotation inside the GEMV starts in one of two ways.  Blocks of 512 and more: the scan of x stores FP16 values, and the
// first pass over them runs the widest `stages` strides, 2^stride and more, down to pieces of 2^stride coordinates, of which a CTA
// keeps the ones that meet its blocks of x.  Shorter blocks have little to leave out: the scan runs their three narrowest
// stages on the eight values a thread holds (`stages` 0) and keeps whole blocks (`stride` the block).  Us a rotating launch of
// 4096 x 4096 with blocks of 8, 64, 128, 256, 512: FP16 values first 6.21, 6.12, 6.46, 6.41, 6.03; stages first 5.29, 5.89, 6.22, 6.21, -.
struct RotFirst {
    int stages, stride;
};
__host__ __device__ inline RotFirst rot_first(int block_log2) {
    RotFirst f;
    f.stages = block_log2 >= 9 ? 3 : 0;
    f.stride = block_log2 - f.stages;
    return f;
}
// Everything gemv_plan looks at, and what it made of it.
struct PlanKey {
    int layout, nb, batch, rot_log2, rot_n, nprob;
    int rows[LLVQ_MAX_GROUP];
};
// The plans of the last kKept shapes launched (a decoder has four or five): 2 KB and half a microsecond each.  Host threads
// that launch on one stream may ask at the same time: a plan is handed out whole, under the lock (20 ns where nobody waits).
class PlanCache {
public:
    // Copies the plan of `key` to `plan` and returns its launch: the kept one, or what make(plan) works out.
    template <typename F>
    GemvLaunch get(const PlanKey &key, GemvPlan &plan, F make) {
        std::lock_guard<std::mutex> lock(mutex_);
        for (int i = 0; i < used_; i++)
            if (std::memcmp(&kept_[i].key, &key, sizeof key) == 0) {
                plan = kept_[i].plan;
                return kept_[i].launch;
            }
        Entry &e = kept_[next_];
        e.launch = make(plan);
        e.key = key;
        e.plan = plan;
        if (used_ < kKept) used_++;
        next_ = (next_ + 1) % kKept;
        return e.launch;
    }

private:
    static constexpr int kKept = 8;
    struct Entry {
        PlanKey key;
        GemvPlan plan;
        GemvLaunch launch;
    };
    std::mutex mutex_;
    Entry kept_[kKept];
    int used_ = 0, next_ = 0;
};

// Three, four, seven and eight vectors have a kernel of their own, which takes them in sets of four (llvq_batch.cu).
// Five and six would leave half of the second set idle (us in sets and in pairs: five on 500 x 8192 10.8 and 8.3, 4096 x 4096 13.4 and 11.0,
// 34816 x 5120 50.5 and 47.4; six on 1024 x 2560 7.2 and 6.1, 8192 x 8192 24.9 and 22.5).
__host__ __device__ constexpr bool batch_in_sets(int batch) { return batch == 3 || batch == 4 || batch >= 7; }

constexpr int kVectorsPerPass = 4;      // activation vectors a pass that llvq_gemv_plan describes carries at most
constexpr int kTwoByTwo = 1;            // a pass's answer where three or four vectors have to go in passes of two
// Whether a pass fits a multiprocessor that grants `most` bytes of shared memory: LLVQ_OK or the pass's answer.  Three and four vectors that
// do not fit as a set go two by two where four did in pairs, whose records of x are 32 bytes a block less.
inline int pass_refusal(int batch, size_t smem, int xblocks, size_t most) {
    if (smem + 1024 <= most) return LLVQ_OK;
    return batch_in_sets(batch) && batch <= kVectorsPerPass && smem - 32 * (size_t)xblocks + 1024 <= most ? kTwoByTwo : LLVQ_ESIZE;
}
// The passes over the records that `batch` activation vectors take; pass(first, n) launches vectors [first, first + n) or says why not.
// One pass serves all of them, if the scratch has room for their sums and a multiprocessor for their records of x, which
// only devices of few multiprocessors lack (eight vectors, us in one pass and in two: 1024 x 2560 8.8 and 10.5, 4096 x 4096
// 15.1 and 16.5, 34816 x 5120 53.9 and 64.8).
template <typename Pass>
int batch_passes(int batch, Pass pass) {
    int rc = pass(0, batch);
    if (rc != kTwoByTwo && (rc != LLVQ_ESIZE || batch <= kVectorsPerPass)) return rc;
    // Otherwise passes of up to four, or of two, one after the other on the stream (they share the context's scratch).
    for (int first = 0, n; first < batch; first += n) {
        n = batch - first < kVectorsPerPass ? batch - first : kVectorsPerPass;
        rc = pass(first, n);
        if (rc == kTwoByTwo) rc = pass(first, n = 2);
        if (rc != LLVQ_OK) return rc;
    }
    return LLVQ_OK;
}

// A GEMV launched right behind an expansion must not read records ahead of its wait; behind a GEMV that was launched as an
// ordinary kernel after the expansion, it may.  Host threads that share the stream may ask at any point of one another's
// launches: an expansion counts once it is enqueued, and an ordinary launch, once it is enqueued itself, for the expansions that
// were counted before it.
class RecordOrder {
public:
    void expanded() { expansions_.fetch_add(1); }
    uint64_t expansions() const { return expansions_.load(); }
    bool behind(uint64_t expansions) const { return ordered_.load() >= expansions; }      // an ordinary launch lies behind all of them
    void ordered(uint64_t expansions) {
        uint64_t seen = ordered_.load();
        while (seen < expansions && !ordered_.compare_exchange_weak(seen, expansions)) {}
    }

private:
    std::atomic<uint64_t> expansions_{0}, ordered_{0};
};

}  // namespace llvq

struct llvq_ctx {
    int device;
    llvq::HostTables host;
    llvq::DeviceTables dev;
    llvq::UnrankView unrank;     // the expander's tables (device)
    void *table_blob;        // one allocation holding every table
    unsigned long long *accum;   // reduction scratch: one 64-bit accumulator a row of the largest launch
    size_t accum_slots;
    int *error;              // device flag: a kernel's bounded wait ran out
    uint32_t *bad_codes;     // device count: codes that named no point, over the expansions since the last llvq_status
    uint32_t *overflow;      // device count: exception-table entries that found no room, since the last llvq_status
    unsigned long long *counter;   // device scratch of llvq_overlay_count: two words, zero between calls
    unsigned long long *host_counter;   // page-locked: its result
    std::mutex count_mutex;  // one llvq_overlay_count at a time: the two above are its own from launch to result
    int use_pdl;             // launch the GEMV with programmatic stream serialization
    llvq::RecordOrder order; // whether a GEMV may read records ahead of its wait
    int sm_count;
    int max_smem_optin;
    llvq::PlanCache plans;
};

namespace llvq {
// A launch's status.  The runtime keeps a refused launch's error for whoever asks next; it is this call's, which reports it.
inline int launched(cudaError_t status) {
    if (status == cudaSuccess) return LLVQ_OK;
    cudaGetLastError();
    return LLVQ_ECUDA;
}
cudaError_t launch_expand(const llvq_ctx *ctx, int layout, const uint64_t *codes, int64_t rows, int64_t nb,
                          void *out, size_t out_bytes, uint32_t *bad_count, cudaStream_t s);
// writes the number of blocks the 10-byte layout would keep in its exception table to *host (page-locked); `counter` is two
// device words that are zero before and after
cudaError_t launch_overlay_count(const llvq_ctx *ctx, const uint64_t *codes, int64_t rows, int64_t nb, unsigned long long *counter,
                                 unsigned long long *host, cudaStream_t s);
// Completes the launch geometry in `p` (order of work, shares of x) and returns grid and dynamic shared memory.
GemvLaunch gemv_plan(int layout, GemvParams &p, int sm_count);
void gemv_lane_table(uint32_t (*out)[4]);      // fills the 32 entries of DeviceTables::lane_table (host)
cudaError_t launch_gemv(int layout, const GemvParams &p, const GemvLaunch &g, bool no_weights, bool pdl, cudaStream_t s);
cudaError_t launch_wait_limit_selftest(const llvq_ctx *ctx, cudaStream_t s);
cudaError_t launch_gemv_fp16(const __half *W, const __half *x, float *y, int64_t rows, int64_t k, cudaStream_t s);
cudaError_t launch_dequant(const llvq_ctx *ctx, int layout, const uint8_t *buf, const __half *row_scale, float g0, float g1,
                           __half *W, int64_t rows, int64_t nb, cudaStream_t s);
cudaError_t launch_decode_i8(const llvq_ctx *ctx, int layout, const uint8_t *buf, int8_t *coords, uint16_t *class_ids,
                             int64_t rows, int64_t nb, cudaStream_t s);
int expand_configure();                    // sets the expander's shared-memory attributes once a device
int gemv_configure(const llvq_ctx *ctx);   // sets the kernels' shared-memory attributes once

// activation rotation: blocks of at most 2^14 coordinates (64-bit partial sums in 128 KiB of shared memory)
constexpr int kRotMaxBlockLog2 = 14;
int rotate_block_log2(int64_t n, int64_t block);   // log2 of the block length used, -1 if `block` is not acceptable
int rotate_configure();                            // sets the kernel's shared-memory attribute once a device
cudaError_t launch_rotate(const __half *x, __half *y, const uint32_t *negate, int64_t n, int block_log2, bool pdl,
                          cudaStream_t s);
}  // namespace llvq
