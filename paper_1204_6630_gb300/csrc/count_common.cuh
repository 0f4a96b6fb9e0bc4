// Device helpers shared by the counting kernels (count.cu: FP32 and binary64
// kernels of independent warps; count_tc.cu: the tensor-core screen): PTX
// wrappers, the lookup table's 16-bit codes, thread-private counters, the
// classification of pairs that the lookup table leaves open, the sphere test
// of spatial pruning.
//
// Paper: Ponce et al., "Application of GPUs for the calculation of two point
// correlation functions in cosmology", Section 3 (dot product, angle to bin,
// partial histograms combined into one).
#pragma once

#include <stdint.h>

#include "plan.h"
#include "tpcf.h"
#include "tpcf_internal.h"

namespace tpcf {

// Dynamic shared memory of the counting kernel.  Helpers address it through
// 32-bit byte offsets (one register each instead of a 64-bit pointer).
extern __shared__ __align__(128) unsigned char dyn_smem[];

template <class Tp>
__device__ __forceinline__ Tp* sptr(uint32_t off) {
    return reinterpret_cast<Tp*>(dyn_smem + off);
}

// ============================================================== PTX helpers
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// 1-D TMA bulk copy global -> shared, completion signalled on `bar`.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// One bounded probe of the barrier phase.  The suspend-time hint lets the
// hardware park the waiting warp until the phase completes or about
// kSuspendNs elapse, instead of spinning on the probe.
constexpr uint32_t kSuspendNs = 20000;

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for phase `parity` of `bar` to complete, giving up after limit_ns.
static __device__ __noinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
}

// Packed FP32x2 (sm_100+): two FP32 lanes in one 64-bit register pair.
typedef unsigned long long u64;
__device__ __forceinline__ u64 pack2(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo_of(u64 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_of(u64 v) { return __uint_as_float((uint32_t)(v >> 32)); }
// d = a * b + c on both halves, each rounded to nearest as fmaf rounds.
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// d = a - b on both halves, rounded to nearest.
__device__ __forceinline__ u64 fsub2(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Three-input AND / OR in one logic instruction.
__device__ __forceinline__ uint32_t and3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0x80;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t or3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xfe;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// AND (OR) of the bit patterns of N words as a tree of three-input operations.
template <int N, bool OR>
__device__ __forceinline__ uint32_t lop_tree(const uint32_t* v) {
    if constexpr (N == 1) {
        return v[0];
    } else if constexpr (N == 2) {
        return OR ? (v[0] | v[1]) : (v[0] & v[1]);
    } else {
        constexpr int A = N / 3, B = (N - A) / 2;
        const uint32_t x = lop_tree<A, OR>(v), y = lop_tree<B, OR>(v + A), z = lop_tree<N - A - B, OR>(v + A + B);
        return OR ? or3(x, y, z) : and3(x, y, z);
    }
}

// Kernel variants: FP32 screen (angles), all-binary64 comparator, FP32 screen
// of distances (3-D variant).
enum KernelMode { kModeScreen = 0, kModePlain = 1, kModeEuclid = 3 };

__host__ __device__ inline uint32_t align_up(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

// ============================================================== LUT entries
// A cell of the shared LUT is a 16-bit code, read sign-extended:
//   - settled in row P < ne (P == Q): P (0 <= code < kLutRowLimit);
//   - settled in the overflow row (P == Q == ne): kLutSkip, a non-negative
//     code >= kLutRowLimit, so the pair adds nothing (without
//     TPCF_F_CHECK_OVERFLOW the overflow row is never merged: the finalize
//     derives it from the pair total); with TPCF_F_CHECK_OVERFLOW the code is
//     the row ne itself, so overflow pairs are counted like the others;
//   - unsettled (edges [P, Q) open): bit 15 set (negative), P in bits 0..8,
//     min(Q - P, 63) in bits 9..14; the span 63 stands for Q = ne, a wider
//     range that every resolver handles with the same result (the edges
//     past the true Q are decided "not crossed" by their bounds).
// Rows fit 9 bits: ne <= TPCF_MAX_EDGES = 321.
constexpr uint32_t kLutRowLimit = 512;
constexpr uint32_t kLutSkip = 0x4000;
constexpr uint32_t kLutSpanCap = 63;

__device__ __forceinline__ unsigned short lut_code(uint32_t P, uint32_t Q, uint32_t ne, bool count_over) {
    if (P == Q) return (unsigned short)(P == ne && !count_over ? kLutSkip : P);
    return (unsigned short)(0x8000u | P | (min(Q - P, kLutSpanCap) << 9));
}
__device__ __forceinline__ int lut_P(int x) { return x & 0x1ff; }
__device__ __forceinline__ int lut_Q(int x, int ne) {
    const int span = (x >> 9) & 0x3f;
    return span == (int)kLutSpanCap ? ne : (x & 0x1ff) + span;
}

// Byte offset of histogram row h from a thread's column: h * (T/2) * 4 = h << log2(2T).
template <int T>
__host__ __device__ constexpr int row_shift() {
    static_assert(T == 128 || T == 256 || T == 512 || T == 1024, "power-of-two block");
    return T == 128 ? 8 : T == 256 ? 9 : T == 512 ? 10 : 11;
}

__device__ __forceinline__ int ld_shared_s16(uint32_t addr) {
    int v;
    asm volatile("ld.shared.s16 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// ============================================================== work items
// An item in progress: its sub-problem, geometry and current tile.
struct Cursor {
    uint32_t q;       // walk position of the item
    int sub;
    ItemGeom g;
    uint32_t t;       // current tile within the item
    bool valid;
};

__device__ __forceinline__ const SubProblem& sub_of(const WorkDesc& wd, int s) {
    return wd.sub_dev ? wd.sub_dev[s] : wd.sub[s];
}

static __device__ int find_sub(const WorkDesc& wd, uint64_t q) {
    int lo = 0, hi = wd.nsub;  // sub[lo].item_begin <= q < sub[hi].item_begin
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (sub_of(wd, mid).item_begin <= q) lo = mid; else hi = mid;
    }
    return lo;
}

template <bool BY_ROOT = true>
static __device__ bool load_item(const WorkDesc& wd, uint32_t q, Cursor& c) {
    c.q = q;
    c.sub = find_sub(wd, q);
    const SubProblem& sp = sub_of(wd, c.sub);
    const uint64_t local = walk_item_inv(q - sp.item_begin, sp.n_items, sp.walk_mult, sp.walk_inv);
    c.g = item_geom(local, sp.na, sp.nb, sp.n_iblk, sp.n_jchunk, sp.auto_mode != 0, wd.I, wd.Jc, wd.J,
                    BY_ROOT);
    c.t = c.g.t_first;
    return c.t < c.g.t_end;
}

// ============================================================== block helpers
// Block constants live in the kernel parameter (constant bank): the host fills
// the shared-memory offsets and the bin scalars of WorkDesc, so the kernel
// spends no registers on them.
template <int T>
__device__ void load_bins(const BinsDev* bd, const WorkDesc& wd, bool plain) {
    const int ne = wd.ne;
    double* c = sptr<double>(wd.off_cthr);
    float* lo = sptr<float>(wd.off_lo);
    float* hi = sptr<float>(wd.off_hi);
    float* c32 = sptr<float>(wd.off_c32);
    float* zlo = sptr<float>(wd.off_zlo);
    float* zhi = sptr<float>(wd.off_zhi);
    for (int k = threadIdx.x; k < ne; k += T) {
        c[k] = bd->cos_thr[k];
        lo[k] = bd->lo[k];
        hi[k] = bd->hi[k];
        c32[k] = bd->cos32[k];
        zlo[k] = bd->zlo[k];
        zhi[k] = bd->zhi[k];
    }
    if (!plain) {
        // Shared copy of the LUT as 16-bit entries (see lut_code).
        const bool count_over = (wd.flags & TPCF_F_CHECK_OVERFLOW) != 0;
        unsigned short* lut = sptr<unsigned short>(wd.off_lut);
#pragma unroll 8
        for (int k = threadIdx.x; k < kLutCells; k += T) {
            const uint32_t e = bd->lut[k];
            lut[k] = lut_code(e & 0xffffu, e >> 16, (uint32_t)ne, count_over);
        }
    }
}

// Thread-private 16-bit histogram counters, two per 32-bit shared word:
// thread t < T/2 owns the low halves of column t, thread t + T/2 the high
// halves of the same column, so every thread adds one fixed increment (1 or
// 2^16) and a row is a plain byte offset.  A counter has a single writer; the
// word's atomic add keeps the partner's half intact.  Lanes of a warp hold 32
// consecutive columns, so a warp's adds to any mix of rows hit 32 banks.
struct HistCol {
    uint32_t addr;  // shared byte address of the thread's word in row 0
    uint32_t inc;   // 1 (low half) or 65536 (high half)
};

template <int T>
__device__ __forceinline__ HistCol hist_col(const WorkDesc& wd) {
    const uint32_t t = threadIdx.x;
    return HistCol{smem_addr(dyn_smem) + wd.off_hist + (t % (T / 2)) * 4u, t < T / 2 ? 1u : 65536u};
}

__device__ __forceinline__ void red_add_shared(uint32_t addr, uint32_t v) {
    asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Histogram row h of the thread's column, one increment.
template <int T>
__device__ __forceinline__ void hist_inc(const HistCol& hc, int h) {
    red_add_shared(hc.addr + ((uint32_t)h << row_shift<T>()), hc.inc);
}

// One warp merges its 32 counters of every row into the global uint64 bins
// and clears them.  Rows 0..nedges-1 (underflow and the B bins) are merged;
// row nedges (pairs beyond the last edge) is merged only when overflow is
// counted (TPCF_F_CHECK_OVERFLOW), otherwise only cleared: the finalize
// kernel derives overflow from the pair total.  Each thread takes its own
// half out of the shared word with an atomic subtract, since the partner warp
// may be adding to the other half at the same time.
// Eight rows at a time: their loads, sums and atomics overlap (row by row a
// merge of 66 rows took 25000 cycles).
template <int T>
__device__ void warp_flush_hist(const HistCol& hc, int nedges, bool count_over, unsigned long long* out) {
    const int lane = threadIdx.x & 31;
    const uint32_t sh = hc.inc == 1u ? 0u : 16u;
    for (int h0 = 0; h0 <= nedges; h0 += 8) {
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            v[k] = h0 + k <= nedges ? (ld_shared_u32(hc.addr + ((uint32_t)(h0 + k) << row_shift<T>())) >> sh) & 0xffffu : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (v[k]) red_add_shared(hc.addr + ((uint32_t)(h0 + k) << row_shift<T>()), 0u - (v[k] << sh));
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t t = __reduce_add_sync(0xffffffffu, v[k]);
            if (lane == k) sum = t;
        }
        const int h = h0 + lane;  // lane k merges row h0 + k
        if (lane < 8 && sum != 0u && (h < nedges || (h == nedges && count_over))) atomicAdd(out + h, (unsigned long long)sum);
    }
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// ============================================================== per-pair classification
__device__ __forceinline__ Point64 ldg_point(const Point64* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    const double2 u = __ldg(q), v = __ldg(q + 1);
    Point64 r;
    r.x = u.x; r.y = u.y; r.z = v.x; r.w = v.y;
    return r;
}

// Binary64 dot product in the definition's order, no contraction.
__device__ __forceinline__ double dot64(const Point64& a, const Point64& b) {
    return __dadd_rn(__dadd_rn(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)), __dmul_rn(a.z, b.z));
}

// Exact histogram index of a band pair: h = nbv + #{m in [nbv, nav) : d <= C_m}
// with d the binary64 dot product (the edges below nbv are certainly crossed,
// those from nav on certainly not).  h32 is the FP32-only index; *mismatch
// is set when it differs (statistics).
__device__ __forceinline__ int band_index(const WorkDesc& wd, const SubProblem& sp, uint32_t ig, uint32_t jg,
                                          int nbv, int nav, int h32, uint32_t* mismatch) {
    const double* cthr = sptr<const double>(wd.off_cthr);
    const double d = dot64(ldg_point(sp.a64 + ig), ldg_point(sp.b64 + jg));
    int h = nbv;
    for (int m = nbv; m < nav; ++m) h += (d <= cthr[m]);
    *mismatch = (h != h32) ? 1u : 0u;
    return h;
}

// FP32 classification of a pair whose LUT entry left edges [P, Q) open:
// nb(c) = #{m : c < lo_m} (edges certainly crossed), na(c) = #{m : c <= hi_m}
// (edges possibly crossed); nb == na settles the index.  Otherwise h = -1
// with the band range [nbv, nav) and the FP32-only index h32.
struct Resolved {
    int h, nbv, nav, h32;
};

__device__ __forceinline__ Resolved resolve_f32(const WorkDesc& wd, float c, int P, int Q) {
    const float* lo = sptr<const float>(wd.off_lo);
    const float* hi = sptr<const float>(wd.off_hi);
    const float* c32 = sptr<const float>(wd.off_c32);
    int nb_ = P, na_ = P;
    for (int m = P; m < Q; ++m) {
        nb_ += (c < lo[m]);
        na_ += (c <= hi[m]);
    }
    if (nb_ == na_) return Resolved{nb_, 0, 0, 0};
    int h = nb_;
    for (int m = nb_; m < na_; ++m) h += (c <= c32[m]);
    return Resolved{-1, nb_, na_, h};
}

// FP32 coordinates of point i of a blocked catalog (lanes with consecutive
// points read consecutive words).
__device__ __forceinline__ float3 ldg_point32(const unsigned char* blk, uint32_t i) {
    const float* p = reinterpret_cast<const float*>(blk + (size_t)(i / kBlk) * kBlkBytes + kBlkX) + i % kBlk;
    return make_float3(__ldg(p), __ldg(p + kBlk), __ldg(p + 2 * kBlk));
}

// LUT entry of screen value e: cell k = rne(sat(e * 2^-q) * 2^14), read as the
// low bits of fma(v, 2^14, 2^23).
__device__ __forceinline__ int lut_entry(const WorkDesc& wd, float e) {
    const float v = __saturatef(e * wd.lut_scale);
    const float f = fmaf(v, (float)(1 << kLutBits), 8388608.0f);
    return ld_shared_s16(smem_addr(dyn_smem) + wd.off_lut + (__float_as_uint(f) - 0x4B000000u) * 2u);
}

// ---- 3-D variant (Euclidean separations)
// z = fl32(|a' - b'|^2): differences, then a fused sum of squares.
__device__ __forceinline__ float euclid_z(float ax, float ay, float az, float bx, float by, float bz) {
    const float dx = ax - bx, dy = ay - by, dz = az - bz;
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// LUT cell of z: constant-ratio cells, clamp((bits(z) - zbits0) >> zshift) (z >= 0).
__device__ __forceinline__ uint32_t euclid_cell_addr(const WorkDesc& wd, float z, uint32_t lut_base) {
    int k = ((int)__float_as_uint(z) - wd.zbits0) >> wd.zshift;
    k = min(max(k, 0), kLutCells - 1);
    return lut_base + (uint32_t)k * 2u;
}

// binary64 d^2 in the definition's order: differences, squares, left-to-right sum.
__device__ __forceinline__ double dist2_64(const Point64& a, const Point64& b) {
    const double dx = __dsub_rn(a.x, b.x), dy = __dsub_rn(a.y, b.y), dz = __dsub_rn(a.z, b.z);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// A 3-D pair whose LUT entry left edges [P, Q) open: z against the z-space
// bounds (increasing with the edge index; z >= zhi_m proves d^2 >= S_m, z <
// zlo_m proves d^2 < S_m).  Returns h >= 0 when z settles it; otherwise -1 and
// the edges still open, [*lo, *hi).
__device__ __forceinline__ int euclid_resolve(const WorkDesc& wd, float z, int ent, int* lo_out, int* hi_out) {
    const float* zlo = sptr<const float>(wd.off_zlo);
    const float* zhi = sptr<const float>(wd.off_zhi);
    const int Q = lut_Q(ent, wd.ne);
    int lo = lut_P(ent), hi = Q;
    while (lo < hi) {  // first m in [P, Q) with z < zhi[m]: the edges below are crossed
        const int mid = (lo + hi) >> 1;
        if (z >= zhi[mid]) lo = mid + 1; else hi = mid;
    }
    if (lo == Q || z < zlo[lo]) return lo;
    int a = lo + 1, c = Q;  // first m > lo with z < zlo[m]: the edges from there on are not crossed
    while (a < c) {
        const int mid = (a + c) >> 1;
        if (z >= zlo[mid]) a = mid + 1; else c = mid;
    }
    *lo_out = lo;
    *hi_out = a;
    return -1;
}

// Index of a 3-D pair decided in binary64 over the open edges [lo, hi)
// (S increasing: count the edges with d^2 >= S_m); h32 from the FP32 value
// against RN(S_m) for the statistics.
__device__ __forceinline__ int euclid_band_index(const WorkDesc& wd, const SubProblem& sp, uint32_t ig, uint32_t jg,
                                                 float z, int lo, int hi, uint32_t* mismatch) {
    const double* sthr = sptr<const double>(wd.off_cthr);
    const float* s32 = sptr<const float>(wd.off_c32);
    const double d2 = dist2_64(ldg_point(sp.a64 + ig), ldg_point(sp.b64 + jg));
    // two padding points (+inf) are NaN apart: not a pair (overflow, never merged);
    // real points are finite, |x| <= 1e28, so their binary64 d^2 is finite
    if (d2 != d2) {
        *mismatch = 0u;
        return wd.ne;
    }
    int h = lo, h32 = lo;
    for (int m = lo; m < hi; ++m) {
        h += (d2 >= sthr[m]);
        h32 += (z >= s32[m]);
    }
    *mismatch = (h != h32) ? 1u : 0u;
    return h;
}

// Histogram index of an unsettled pair (FP32 a, b; indices ig, jg).  Angles:
// the screen value and LUT entry are recomputed (bit-identical to the slow
// path's), the chord refinement decides the edges the entry leaves open where
// the catalogs allow it: z = fl32(|a' - b'|^2) is within 4u|a - b| + O(u |a -
// b|^2) of 2 (1 - d) (bounds zlo, zhi: runtime.cpp), far tighter than the
// screen value at the small and moderate angles of a histogram range; z-space
// bounds increase with the edge index, so a binary search over [P, Q) finds
// nb = #{crossed} and the pair is settled when z is also below zlo[nb].  Then
// the FP32 comparison with the open edges' screen bounds, else the binary64
// recomputation in the definition's order.  3-D: the z-space bounds of the
// open edges, else binary64.  Band statistics are added to band, mism.
template <bool EUCLID>
__device__ __forceinline__ int classify_unsettled(const WorkDesc& wd, const SubProblem& sp, float ax, float ay,
                                                  float az, float bx, float by, float bz, uint32_t ig, uint32_t jg,
                                                  uint32_t& band, uint32_t& mism) {
    if constexpr (EUCLID) {
        const float z = euclid_z(ax, ay, az, bx, by, bz);
        const int ent = ld_shared_s16(euclid_cell_addr(wd, z, smem_addr(dyn_smem) + wd.off_lut));
        if (ent >= 0) return ent == (int)kLutSkip ? wd.ne : ent;  // settled (not expected)
        int lo = 0, hi = 0;
        const int h0 = euclid_resolve(wd, z, ent, &lo, &hi);
        if (h0 >= 0) return h0;
        uint32_t mm;
        const int h = euclid_band_index(wd, sp, ig, jg, z, lo, hi, &mm);
        band += 1;
        mism += mm;
        return h;
    } else {
        const float e = fmaf(az, bz, fmaf(ay, by, fmaf(ax, bx, wd.neg_fast_t)));
        const int ent = lut_entry(wd, e);
        if (ent >= 0) return ent == (int)kLutSkip ? wd.ne : ent;  // settled (not expected)
        const int P = lut_P(ent), Q = lut_Q(ent, wd.ne);
        if (wd.chord_ok) {
            const float z = euclid_z(ax, ay, az, bx, by, bz);
            const float* zlo = sptr<const float>(wd.off_zlo);
            const float* zhi = sptr<const float>(wd.off_zhi);
            int lo = P, hi = Q;
            while (lo < hi) {  // first m in [P, Q) with z < zhi[m]
                const int mid = (lo + hi) >> 1;
                if (z >= zhi[mid]) lo = mid + 1; else hi = mid;
            }
            if (lo == Q || z < zlo[lo]) return lo;
        }
        const Resolved rs = resolve_f32(wd, e, P, Q);
        if (rs.h >= 0) return rs.h;
        uint32_t mm;
        const int h = band_index(wd, sp, ig, jg, rs.nbv, rs.nav, rs.h32, &mm);
        band += 1;
        mism += mm;
        return h;
    }
}

// ============================================================== spatial pruning
// Every point p of a group lies within radius r of the group's centre c
// (bounding spheres from prep_caps_kernel, in the catalog's scaled space).  By
// the triangle inequality, any pair (a, b) of two groups is at least
// |cA - cB| - rA - rB apart; when that gap exceeds prune_thr (the host's
// bound: every pair that far apart is overflow), the block is skipped.  The
// FP32 evaluation here under-estimates the gap (relative margin 2^-20 on the
// centre distance and on the radii, far above the few-ulp rounding of these
// FP32 operations).
constexpr float kPruneMargin = 9.5367431640625e-07f;  // 2^-20

__device__ __forceinline__ bool prune_block(const WorkDesc& wd, const float4& ic, const float4& jc) {
    const float dx = ic.x - jc.x, dy = ic.y - jc.y, dz = ic.z - jc.z;
    const float D = sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
    const float L = D * (1.0f - kPruneMargin) - (ic.w + jc.w) * (1.0f + kPruneMargin);
    return L > wd.prune_thr;
}

}  // namespace tpcf
