// Internal types shared by the host runtime (runtime.cpp, server.cpp) and the
// kernels (count.cu, prep.cu).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tpcf {

// Catalog padding: every device catalog holds a multiple of this many
// points; points past n are zero vectors (never counted, see count.cu).
constexpr uint32_t kPad = 4096;

// Segments of a segmented catalog start on multiples of this many points (one
// warp's i-points of the 512 x 8 counting shape), so that a warp's i-points
// always belong to one segment.
constexpr uint32_t kSegAlign = 256;
// Bounding spheres for spatial pruning: one per kCapPoints consecutive
// points of a catalog's device layout.
constexpr uint32_t kCapPoints = 128;
// A catalog's FP32 points and tensor-core operands, in blocks of kBlk points:
// plane X (16 bytes a point), then the FP32 coordinates as x | y | z arrays.
// X = (x1, y1, z1, x2, y2, z2, n1, n2) is the binary16 split x = x1 + x2
// (likewise y, z).  Angular catalogs: n1 = n2 = 0.  3-D catalogs: of the point
// scaled by 2^-k to norm <= 1 (k from the largest norm, tc_exponent), and n1 +
// n2 splits -|v|^2 / 2; padding has a large negative n1.
constexpr uint32_t kBlk = 128;
constexpr uint32_t kBlkX = kBlk * 16;
constexpr uint32_t kBlkBytes = kBlkX + kBlk * 12;
// Bound on the distance of the tensor-core screen value from the binary64 dot
// product (44u, derived in count_tc.cu) with a margin.
constexpr double kTcGuard = 64.0 * 5.9604644775390625e-08;
// The same for 3-D counts: bound on the distance of the products' value from
// (a.b - |b|^2 / 2) scaled, plus that of the lane's threshold, per unit of
// max(s, 1/s), s the ratio of the catalogs' scales (57u, derived in count_tc.cu).
constexpr double kTcGuard3d = 128.0 * 5.9604644775390625e-08;
constexpr int kTcMaxRatio = 10;  // |log2 s| at most: s is a binary16 operand

// A k with 2^k >= sqrt(norm2): the smallest, or one more where norm2 is an even power of
// two (at least -100: its scale is an FP32 number).
__host__ __device__ inline int tc_exponent(unsigned long long norm2_bits) {
    const int e = (int)((norm2_bits >> 52) & 0x7ffu) - 1023;  // norm2 < 2^(e + 1)
    if (norm2_bits == 0ull) return 0;
    const int k = (e + 2) >> 1;
    return k < -100 ? -100 : k;
}
// 3-D catalogs store their spheres scaled by 2^-64 (exact), so that FP32
// squares of separations up to 2e28 stay finite.
constexpr double kCapScale3d = 5.421010862427522e-20;

// Lookup table from the FP32 screen value to the candidate histogram index
// range: cell k = rne(sat(e * lut_scale) * 2^14), k = 0 .. 2^14.
constexpr int kLutBits = 14;
constexpr int kLutCells = (1 << kLutBits) + 1;

// The chord refinement of unsettled pairs (count.cu, classify_unsettled) is proven for
// catalogs whose points satisfy | |v|^2 - 1 | <= kChordEpsRef.
constexpr double kChordEpsRef = 0x1p-40;

// Binary64 point (x, y, z, 0), 32-byte aligned for two 16-byte loads.
struct __align__(32) Point64 {
    double x, y, z, w;
};

// Device-resident description of one bin set (Section 3: angle -> bin).
// All arrays live in one device allocation owned by tpcf_bins.
// The FP32 screen value of a pair is e = fma(az,bz, fma(ay,by, fma(ax,bx, -T)))
// with T = fast_t; the e-space bounds below are the cos-space thresholds
// shifted by T and widened by the guard band.
struct BinsDev {
    const double* cos_thr;  // [nedges] C_k, decreasing (C_0 may be +inf)
    const float* lo;        // [nedges] RD(C_k - T - g)   (e-space)
    const float* hi;        // [nedges] RU(C_k - T + g)   (e-space)
    const float* cos32;     // [nedges] RN(C_k - T): FP32-only classification (statistics)
    const uint32_t* lut;    // [kLutCells] (P | Q << 16) per cell of e: see runtime.cpp
    const float* zlo;       // [nedges] chord-space bounds of Z_k = 2 (1 - C_k): z < zlo_k => not crossed
    const float* zhi;       // [nedges]                                          z >= zhi_k => crossed
    int nedges;             // B + 1
    float lut_scale;        // 2^-q with 2^q >= every in-range e: cell width 2^(q - 14)
    // 3-D variant (euclid = 1): cos_thr holds S_k (r >= r_k <=> d^2 >= S_k),
    // cos32 RN(S_k), fast_t the limit H of the fast test H - |a' - b'|^2 >= 0,
    // cos_last S_B; the LUT cell of z = fl32(|a' - b'|^2) is
    // clamp((bits(z) - zbits0) >> zshift, 0, kLutCells - 1).
    int euclid;
    int32_t zbits0;
    int zshift;
    float fast_t;           // T = RD(C_B - 10u): a screen value e < 0 is certainly overflow
    double cos_last;        // C_B (binary64 range limit, plain kernel)
};

// One histogram to fill: auto count over catalog A (B == A, pairs j > i) or
// cross count A x B (all pairs).  Work is cut into items: (i-block of I points)
// x (j-chunk of Jc points); an item is processed in j-tiles of J points.
struct SubProblem {
    const unsigned char* a_blk;  // FP32 points and operands of A and B in blocks (see kBlk), the
    const unsigned char* b_blk;  // sub-range's first block (catalogs are padded to kPad points)
    const Point64* a64;   // binary64 copy of A (padded)
    const Point64* b64;
    uint32_t na, nb;      // real point counts
    uint32_t n_iblk;      // ceil(na / I)
    uint32_t n_jchunk;    // ceil(nb / Jc)
    uint32_t auto_mode;   // 1: A == B, count j > i only
    uint32_t kratio;      // I / Jc (auto mode: first chunk of i-block ib is ib * kratio)
    uint64_t item_begin;  // global walk position of this sub-problem's first item
    uint64_t n_items;
    uint64_t walk_mult;   // position item_begin + k visits local item (k * walk_mult) mod n_items
    uint64_t walk_inv;          // floor((2^64 - 1) / n_items)
    unsigned long long* hist;   // B + 2 accumulators (device)
    const BinsDev* bins;        // device pointer to this sub-problem's bins
    // Row attribution (leave-one-out jackknife): pairs go to histogram
    // hist + row_seg[b] * row_stride, b the kSegAlign-point block of A holding
    // the pair's i-point (A's segments are aligned, so a warp's i-points share
    // one block).  row_seg == NULL: the one histogram `hist`.
    const uint32_t* row_seg;
    uint32_t row_stride;        // accumulator words between consecutive segments' histograms
    uint32_t no_self;           // 1: A == B counted over the full square except i == j
    // Bounding spheres (x, y, z, radius) of A's and B's kCapPoints-point groups,
    // starting at the sub-range's first point (spatial pruning).
    const float4* a_caps;
    const float4* b_caps;
    const float4* b_caps2;  // spheres of B's kPad-point blocks; NULL: the sub-range does not start on one
    // Tensor-core screen of 3-D counts: a block is kept where a lane's value reaches
    // fma(|tc_scale a|^2, tc_qmul, tc_qadd); tc_pad: the scales' ratio twice, binary16.
    float tc_scale, tc_qmul, tc_qadd;
    uint32_t tc_pad;
};

constexpr int kMaxInlineSub = 3;

// Device statistics words (per call, in the scratch slot after the histograms).
enum StatWord { kStatPairs = 0, kStatBand = 1, kStatMismatch = 2, kStatError = 3, kStatPruned = 4,
                kStatNextItem = 5,  // counting kernel: items drawn from the launch's dynamic pool
                kStatYield = 6,     // counting kernel: nonzero stops further draws (preemptible steps)
                kStatWords = 8 };

// Device error word bits.
enum : uint32_t { kErrWaitTimeout = 1u, kErrBadHist = 2u, kErrBadPoint = 4u, kErrSortOverflow = 8u };

struct WorkDesc {
    SubProblem sub[kMaxInlineSub];   // used when sub_dev == nullptr
    const SubProblem* sub_dev;       // device array of nsub sub-problems (batched launches)
    int nsub;
    uint64_t item_lo, item_hi;       // walk positions of this launch (shards)
    unsigned long long* stats;       // kStatWords words
    // Draw order: the launch draws the positions of [item_lo, item_hi)'s draw
    // order from pos_lo on, the order laid out for draw_warps warps (set by the
    // launcher), and stops drawing once stats[kStatYield] is nonzero (the job
    // server's preemptible steps); the item counter then says how many
    // positions it took.
    uint64_t pos_lo;
    uint32_t draw_warps;
    uint32_t draw_batch;             // tensor-core kernel: items per draw (1..32)
    uint32_t I, J, Jc;               // i-block (one warp's 32 R points), j-tile, j-chunk sizes (points)
    uint32_t stages;                 // stages of each warp's shared-memory ring S (2..16)
    uint32_t flags;                  // TPCF_F_* subset used on the device
    uint32_t force_idx;              // 1: always check indices (sub-ranges of segmented catalogs)
    int nedges_max;                  // largest B + 1 over the sub-problems (shared-memory sizing)
    uint64_t wait_limit_ns;          // bounded waits
    // Block constants, read by the kernel straight from its parameter (no
    // registers).  Bin scalars of the one bin set all sub-problems share
    // (set by the runtime) ...
    int ne;                          // B + 1
    float neg_fast_t;                // -T (screen offset)
    unsigned long long neg_fast_t2;  // the packed pair (-T, -T) (3-D: (-H, -H)): an FP32x2 operand
    float lut_scale;                 // 2^-q (LUT span)
    uint32_t need_idx;               // 1: check i < na, j < nb for every slow pair
    uint32_t chord_ok;               // 1: every catalog of the launch has | |v|^2 - 1 | <= kChordEpsRef
    uint32_t euclid;                 // 1: 3-D variant (distances); neg_fast_t then holds +H
    int32_t zbits0;                  // 3-D variant: LUT cell origin (bits of a float) and shift
    int zshift;
    double cos_last;                 // C_B (all-binary64 kernel)
    uint32_t prune;                  // 1: skip (warp, 128-j chunk) blocks proven beyond the range
    float prune_thr;                 // sphere-gap threshold of the pruning test (see prune_block)
    float near_thr;                  // sphere gap below which two point groups may hold pairs in
                                     // range (the last edge's chord; scheduling only, see heavy_item)
    float tc_thr;                    // tensor-core screen: blocks whose values are all below it are overflow
    // ... and the shared-memory layout of the shape (set by the launcher).
    uint32_t off_ctl, off_bars, off_meta, off_stage, off_hist, off_cthr, off_lo, off_hi, off_c32, off_zlo, off_zhi,
        off_lut, off_queue, off_icap, off_atile;
    uint32_t stage_bytes;            // J * bytes per staged point
    uint32_t flush_limit;            // j-points between merges of the 16-bit counters
};

// Kernel shape selected on the host.
struct Shape {
    int threads;   // T
    int ipt;       // R (a warp's items hold 32 R i-points)
    int jtile;     // J
    int jchunk;    // Jc
    int stages;    // S (per warp)
    int blocks;    // grid size
    size_t smem;   // dynamic shared memory bytes
    bool tc;       // tensor-core kernel (T, R, J and the i-block are its own)
};

// Kernel variants (mode argument of the launchers): FP32 screen of angles,
// all-binary64 comparator, FP32 screen of distances (3-D variant).
enum { kModeScreenScalar = 0, kModePlainFP64 = 1, kModeEuclidScreen = 3 };

// Launchers (count.cu, prep.cu).  All are asynchronous in `stream` and return a
// cudaError_t from the launch.
cudaError_t launch_count(const WorkDesc& wd, const Shape& sh, int mode, int nedges,
                         cudaStream_t stream);
// A served job with histograms too large for the tensor-core kernel (FP32
// screen of angles, shape 512 x 8): the kernel with preemptible draws (wd.pos_lo, stats[kStatYield]).
cudaError_t launch_count_preemptible(const WorkDesc& wd, const Shape& sh, cudaStream_t stream);
// The tensor-core counting kernel (count_tc.cu; angles, and distances where
// its screen applies): items of 512 i-points x Jc j-points in tiles of kBlk; preempt: draws from
// wd.pos_lo on, stopping at the yield word.
cudaError_t launch_count_tc(const WorkDesc& wd, const Shape& sh, bool preempt, cudaStream_t stream);
// The screen's values of 128 x 128 pairs (one block of either catalog; pad: the scales' ratio of a
// 3-D pair of catalogs twice, binary16) and their maxima of 32; err: device error word.
cudaError_t launch_screen_values(const unsigned char* a_blk, const unsigned char* b_blk, bool euclid, uint32_t pad,
                                 uint64_t limit_ns, float* values, float* maxima, unsigned long long* err,
                                 cudaStream_t stream);
size_t count_tc_smem_bytes(int stages, int nedges);
cudaError_t count_tc_set_smem_limit();
// count_over = 1: the kernel counted the overflow row (TPCF_F_CHECK_OVERFLOW);
// the finalize then checks that the histogram sums to the pair total.
cudaError_t launch_finalize(unsigned long long* acc, int nedges, unsigned long long* out,
                            unsigned long long total, int count_over, unsigned long long* err_word,
                            cudaStream_t stream);
cudaError_t launch_finalize_batch(const unsigned long long* acc, int acc_stride, int nedges,
                                  unsigned long long* out, int out_stride, const unsigned long long* totals,
                                  int count, int count_over, unsigned long long* err_word, cudaStream_t stream);
cudaError_t launch_prepare(const double* xyz_in, uint32_t n, const uint32_t* seg_of_point,
                           const uint32_t* seg_delta, int sort, int euclid, unsigned long long* bbox,
                           Point64* out64, unsigned char* blk, float4* caps, float4* caps2, uint32_t n_pad,
                           unsigned long long* key_scratch, uint32_t* val_scratch,
                           uint32_t n_pow2, unsigned long long* err_word, unsigned long long* eps_word,
                           cudaStream_t stream, uint32_t* launches);
size_t count_smem_bytes(int mode, int threads, int ipt, int jtile, int stages, int nedges);
bool count_shape_supported(int threads, int ipt);
bool derive_cos_thresholds(const double* edges, int nedges, double* cos_thr);
cudaError_t count_set_smem_limit(int mode, int threads, int ipt, size_t bytes);
cudaError_t count_preemptible_set_smem_limit(size_t bytes);

}  // namespace tpcf
