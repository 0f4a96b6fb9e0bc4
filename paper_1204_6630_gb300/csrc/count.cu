// CUDA counting kernel (sm_103a) for brute-force angular pair counting.
//
// Paper: Ponce et al., "Application of GPUs for the calculation of two point
// correlation functions in cosmology".  Section 3 lists the three features of
// its CUDA design: points staged in shared memory for the dot product and the
// angle, shared-memory atomic partial histograms combined into one global
// histogram, and the three histograms DD, DR, RR computed in parallel.  This
// file keeps those roles and re-designs them for GB300:
//   * every warp is an independent worker: it draws its own work items (its
//     32 R i-points x a chunk of j-points) from a per-launch counter and
//     streams the j-tiles of its items into its own ring of shared-memory
//     stages with TMA bulk copies (cp.async.bulk + mbarrier), so no warp ever
//     waits for another;
//   * j-tiles are staged as x | y | z arrays and i-points held in registers
//     as (a, a) pairs, so one fma.rn.f32x2 gives the screen values of two
//     pairs;
//   * the angle is never formed: an FP32 dot product is compared with
//     cos-space thresholds derived on the host from the host acos, and only
//     pairs inside a proven guard band around a threshold are recomputed in
//     binary64 (the exact definition);
//   * every thread owns private 16-bit counters in shared memory, merged by
//     its warp into uint64 global bins before any can wrap;
//   * the work is a list of (i-block x j-chunk) items over the upper triangle
//     (auto counts) or the rectangle (cross counts) of one or more histograms.
#include <stdint.h>

#include "count_common.cuh"

namespace tpcf {

// ============================================================== shared-memory layout
// Block-wide control words (int32): the abort flag.
enum Ctl { kCtlAbort = 0, kCtlWords = 32 };

// Per-warp queue of unsettled pairs of the current tile (32-bit codes): at most
// 31 left from earlier groups plus one per lane and round.
constexpr int kUQueue = 64;
constexpr int kMaskGroups = 32;     // fast loop: groups per warp reduction of the slow-group mask
constexpr uint32_t kPruneSlotBytes = 32;  // float4 i-sphere, B's sphere pointer, pruned pair slots (u64)

// One stage of a warp's ring: which item (walk position) and tile it holds.
// Stage record: the item (walk position, sub-problem, first i and j) and tile
// a stage holds, written by the warp's producer lane with the copy, so the
// consumer needs no item arithmetic of its own.
struct TileMeta {
    uint32_t q;
    uint32_t t_sub;  // tile | sub-problem << 16
    uint32_t i0, j0;
};

struct SmemLayout {
    uint32_t ctl;       // control words
    uint32_t bars;      // W x S full mbarriers (warp w: S consecutive)
    uint32_t meta;      // W x S TileMeta
    uint32_t stage;     // W x S stages of stage_bytes
    uint32_t hist;      // (nedges + 1) * T / 2 uint32: row h, column c at word h * T/2 + c (see HistCol)
    uint32_t cos_thr;   // nedges doubles
    uint32_t lo, hi, cos32, zlo, zhi;  // nedges floats each
    uint32_t lut;       // kLutCells 16-bit entries (screen kernels)
    uint32_t queue;     // W * kUQueue unsettled-pair codes (uint32, screen kernels)
    uint32_t icap;      // W pruning slots: the warp's i-sphere, B's sphere array, pruned pair slots
    uint32_t total;
};

// Bytes a staged j-point takes: x | y | z floats (screen kernels) or a
// binary64 (x, y, z, 0) record (all-binary64 kernel).
__host__ __device__ inline uint32_t staged_point_bytes(int mode) { return mode == kModePlain ? 32u : 12u; }

__host__ __device__ inline SmemLayout smem_layout(int mode, int T, int J, int S, int nedges) {
    SmemLayout L;
    const bool plain = mode == kModePlain;
    const uint32_t W = (uint32_t)T / 32;
    uint32_t off = 0;
    L.ctl = off; off += kCtlWords * 4;
    off = align_up(off, 8);
    L.bars = off; off += W * (uint32_t)S * 8;
    L.meta = off; off += W * (uint32_t)S * (uint32_t)sizeof(TileMeta);
    off = align_up(off, 128);
    L.stage = off; off += W * (uint32_t)S * (uint32_t)J * staged_point_bytes(mode);
    L.hist = off; off += (uint32_t)(nedges + 1) * (uint32_t)(T / 2) * 4;
    off = align_up(off, 16);
    L.cos_thr = off; off += (uint32_t)nedges * 8;
    L.lo = off; off += (uint32_t)nedges * 4;
    L.hi = off; off += (uint32_t)nedges * 4;
    L.cos32 = off; off += (uint32_t)nedges * 4;
    L.zlo = off; off += (uint32_t)nedges * 4;
    L.zhi = off; off += (uint32_t)nedges * 4;
    off = align_up(off, 16);
    L.lut = off; off += plain ? 0u : (uint32_t)kLutCells * 2;
    off = align_up(off, 16);
    L.queue = off; off += plain ? 0u : W * kUQueue * 4;
    off = align_up(off, 16);
    L.icap = off; off += W * kPruneSlotBytes;
    L.total = off;
    return L;
}

// ============================================================== work items
// Items are drawn dynamically: every warp takes walk position item_lo + k for
// the next k of a per-launch counter (a statistics word, zeroed before each
// launch), so warps that draw cheap items take more of them.  Within a
// sub-problem, position item_begin + k visits local item (k * walk_mult) mod
// n_items (walk_item).  Positions fit 32 bits (the host checks the count).
// Whether the item with first points i0 (of A) and j0 (of B) is heavy: at
// least a quarter of its j-chunk's kCapPoints-point groups come within
// near_thr of one of its i-groups, so that a large part of its pairs may take
// the slow path (an i-block and a j-chunk inside one dense cluster cost an
// order of magnitude more than an average item).  Called by every lane of the
// warp; one compiled body with explicitly rounded arithmetic and an integer
// reduction, so an item gets the same answer at every call.
__device__ __noinline__ bool heavy_item(const WorkDesc& wd, const SubProblem& sp, uint32_t i0, uint32_t j0) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t ng = wd.Jc / kCapPoints, ni = wd.I / kCapPoints;
    uint32_t near = 0;
    for (uint32_t k = lane; k < ng; k += 32) {
        const uint32_t j = j0 + k * kCapPoints;
        if (j >= sp.nb) break;
        const float4 jc = __ldg(sp.b_caps + j / kCapPoints);
        if (!(jc.w > -1e29f)) continue;  // an empty group
        bool nr = false;
        for (uint32_t a = 0; a < ni; ++a) {
            const uint32_t i = i0 + a * kCapPoints;
            if (i >= sp.na) break;
            const float4 ic = __ldg(sp.a_caps + i / kCapPoints);
            if (!(ic.w > -1e29f)) continue;
            const float dx = __fsub_rn(ic.x, jc.x), dy = __fsub_rn(ic.y, jc.y), dz = __fsub_rn(ic.z, jc.z);
            const float D = __fsqrt_rn(__fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx))));
            nr |= __fsub_rn(__fsub_rn(D, ic.w), jc.w) < wd.near_thr;
        }
        near += nr ? 1u : 0u;
    }
    near = __reduce_add_sync(0xffffffffu, near);
    return 4u * near >= ng;
}

// Order of a launch's items.  A warp that starts a heavy item near the end of
// the range would hold its block, and the launch, for the time of many
// average items; running all heavy items together, on the other hand, would
// load the slow path's shared-memory pipes while the FMA pipes idle.  So only
// the heavy items among the last L of the range are moved to the front; the
// rest of the range follows in walk order, then the light items of the last
// L, of which the last `tail` are handed out as kTailParts consecutive tile
// ranges each.  Draw positions:
//   [0, L)                     heavy items of the last L (light ones skipped),
//   [L, n)                     items 0 .. n - L - 1, all,
//   [n, n + L - tail)          light items of the last L but the last `tail`,
//   then kTailParts parts of each light item of the last `tail`.
// L = kLateRounds and tail = kTailRounds items per warp of the launch (at most
// n; the constants and the order's length, draw_positions, are in plan.h).

// Out of line, as the merge below: with both inlined at every use the loop over the
// tiles outgrew the instruction cache, and pruned launches, which are mostly draws,
// waited for instructions (200,000 + 200,000 points on the sphere to 2 degrees, 512 x 8:
// 2.94 ms inline, 2.47 ms so; 600,000 + 600,000: 16.3 and 13.6 ms).
__device__ __noinline__ bool load_item_ool(const WorkDesc& wd, uint32_t q, Cursor& c) {
    return load_item<false>(wd, q, c);
}
template <int T>
__device__ __noinline__ void merge_hist(HistCol hc, int ne, bool check, unsigned long long* out) {
    warp_flush_hist<T>(hc, ne, check, out);
}

// The warp's next item (or part) with countable tiles, drawing again past
// empty and skipped ones; called by every lane of the warp (lane 0 draws a
// position from `counter`, the position is broadcast).  A preemptible launch
// (PREEMPT) draws from pos_lo on and stops drawing once its yield word is set
// (the positions it took are the counter's value).
template <bool PREEMPT>
__device__ void draw_next(const WorkDesc& wd, Cursor& c, unsigned long long* counter) {
    const uint64_t n = wd.item_hi - wd.item_lo;
    const uint64_t warps = wd.draw_warps;
    const uint64_t L = umin64(n, warps * kLateRounds), tail = umin64(L, warps * kTailRounds);
    const uint64_t parts_at = n + L - tail, end = parts_at + tail * kTailParts;
    while (true) {
        unsigned long long p = ~0ull;  // (a yield: no position taken)
        if ((threadIdx.x & 31) == 0) {
            if constexpr (PREEMPT) {
                if (*reinterpret_cast<volatile unsigned long long*>(wd.stats + kStatYield) == 0ull)
                    p = wd.pos_lo + atomicAdd(counter, 1ull);
            } else {
                p = atomicAdd(counter, 1ull);
            }
        }
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= end) {
            c.valid = false;
            return;
        }
        // k: the item within the range; test: 0 none, 1 heavy only, 2 light only
        uint64_t k;
        int test;
        if (p < L) { k = n - L + p; test = 1; }
        else if (p < n) { k = p - L; test = 0; }
        else if (p < parts_at) { k = n - L + (p - n); test = 2; }
        else { k = n - tail + (p - parts_at) / kTailParts; test = 2; }
        if (!load_item_ool(wd, (uint32_t)(wd.item_lo + k), c)) continue;
        if (test != 0 && heavy_item(wd, sub_of(wd, c.sub), c.g.i0, c.g.j0) != (test == 1)) continue;
        if (p >= parts_at) {
            const uint32_t part = (uint32_t)((p - parts_at) % kTailParts), nt = c.g.t_end - c.g.t_first;
            const uint32_t t0 = c.g.t_first + nt * part / kTailParts, t1 = c.g.t_first + nt * (part + 1) / kTailParts;
            if (t0 == t1) continue;
            c.t = t0;
            c.g.t_end = t1;
        }
        // the pairs of the tiles drawn (a whole item's or a part's), counted once
        if ((threadIdx.x & 31) == 0) {
            const SubProblem& sp = sub_of(wd, c.sub);
            const uint64_t j0 = c.g.j0;
            atomicAdd(wd.stats + kStatPairs,
                      (unsigned long long)span_pairs(c.g.i0, wd.I, j0 + (uint64_t)c.t * wd.J,
                                                     j0 + (uint64_t)c.g.t_end * wd.J, sp.na, sp.nb,
                                                     sp.auto_mode != 0));
        }
        c.valid = true;
        return;
    }
}

template <bool PREEMPT>
__device__ __forceinline__ void advance(const WorkDesc& wd, Cursor& c, unsigned long long* counter) {
    if (!c.valid) return;
    if (++c.t < c.g.t_end) return;
    draw_next<PREEMPT>(wd, c, counter);
}

// ---- unsettled pairs
// A pair whose LUT cell leaves edges open is queued by its warp as a 32-bit
// code lane | r << 5 | j << 10 (the lane holding the i-point, its register r,
// the j-point's offset in the staged tile) and classified later, 32 at a time
// with one pair per lane: the i-point comes from its lane by shuffles, the
// j-point from the tile (the warp empties its queue before leaving a tile).
//
// The lane's i-points as scalars (register halves of the (a, a) pairs) and the
// staged tile: what classifying a queued pair needs.
template <int R>
struct PairSource {
    float x[R], y[R], z[R];
    const float* tile;  // blocks of kBlk points, x | y | z each
    uint32_t i0, jbase;
};

// Classifies the n <= 32 codes at q, one per lane, into the lanes' own columns.
template <int T, int R, bool EUCLID>
__device__ __forceinline__ void drain_batch(const WorkDesc& wd, const SubProblem& sp, const uint32_t* q, uint32_t n,
                                            const PairSource<R>& ps, const HistCol& hc, uint32_t& band,
                                            uint32_t& mism) {
    const uint32_t lane = threadIdx.x & 31u;
    const bool has = lane < n;
    const uint32_t code = has ? q[lane] : 0u;
    const int l = (int)(code & 31u), r = (int)((code >> 5) & 31u);
    const uint32_t jo = code >> 10;
    float ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
        const float x = __shfl_sync(0xffffffffu, ps.x[rr], l);
        const float y = __shfl_sync(0xffffffffu, ps.y[rr], l);
        const float z = __shfl_sync(0xffffffffu, ps.z[rr], l);
        if (rr == r) {
            ax = x;
            ay = y;
            az = z;
        }
    }
    if (has) {
        const uint32_t ig = ps.i0 + (uint32_t)l + 32u * (uint32_t)r, jg = ps.jbase + jo;
        const float* b = ps.tile + (jo / kBlk) * (3 * kBlk) + jo % kBlk;
        hist_inc<T>(hc, classify_unsettled<EUCLID>(wd, sp, ax, ay, az, b[0], b[kBlk], b[2 * kBlk], ig, jg,
                                                   band, mism));
    }
}

// Queues the lane's unsettled pairs of a group (bit U R - 1 - k for pair k =
// r U + u of the group at tile offset jj), one per lane and round (a ballot
// gives each lane its slot), and classifies every full batch of 32 (taken from
// the top of the queue); on return the warp's queue length qn (warp-uniform)
// is below 32.  nbatch counts the batches (each adds at most one to every
// lane's counters).
template <int T, int R, int U, bool EUCLID>
__device__ __forceinline__ void enqueue_unsettled(const WorkDesc& wd, const SubProblem& sp, uint32_t um, int jj,
                                                  uint32_t* q, uint32_t& qn, uint32_t& nbatch,
                                                  const PairSource<R>& ps, const HistCol& hc, uint32_t& band,
                                                  uint32_t& mism) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t below = (1u << lane) - 1u;
    uint32_t act = __ballot_sync(0xffffffffu, um != 0u);
    while (act) {
        if (um) {
            const int b = 31 - __clz(um);
            um &= ~(1u << b);
            const int k = U * R - 1 - b;
            q[qn + (uint32_t)__popc(act & below)] = lane | ((uint32_t)(k / U) << 5) | ((uint32_t)(jj + k % U) << 10);
        }
        qn += (uint32_t)__popc(act);
        if (qn >= 32) {
            __syncwarp();
            qn -= 32;
            drain_batch<T, R, EUCLID>(wd, sp, q + qn, 32u, ps, hc, band, mism);
            ++nbatch;
            __syncwarp();  // the batch is read before later codes overwrite it
        }
        act = __ballot_sync(0xffffffffu, um != 0u);
    }
}

// Diagonal handling of a tile (warp-uniform): none, keep j > i, keep j != i.
enum { kDiagNone = 0, kDiagAbove = 1, kDiagOffSelf = 2 };

// Which pairs of a group may be counted: bit r * U + u for i-point r and
// j-point u (sub-problem bounds, then the diagonal rule of the tile).
template <int R, int U>
__device__ __forceinline__ uint32_t valid_pairs(uint32_t ibase, uint32_t jg0, uint32_t na, uint32_t nb, int diag) {
    uint32_t v = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t ig = ibase + 32u * (uint32_t)r, jg = jg0 + (uint32_t)u;
            bool ok = ig < na && jg < nb;
            if (diag == kDiagAbove) ok = ok && jg > ig;
            else if (diag == kDiagOffSelf) ok = ok && jg != ig;
            v |= (ok ? 1u : 0u) << (r * U + u);
        }
    }
    return v;
}

// ---- packed screen values of a group of U j-points (x | y | z arrays at j)
// for R i-points held as (a, a) pairs: e[r][u] = fma(az,bz, fma(ay,by, fma(ax,bx, -T))).
template <int R, int U>
__device__ __forceinline__ void screen_group2(float (&e)[R][U], const u64 (&ax)[R], const u64 (&ay)[R],
                                              const u64 (&az)[R], const float* sx, const float* sy,
                                              const float* sz, int j, u64 nt2) {
    static_assert(U == 2 || U == 4, "j-points per group");
    if constexpr (U == 4) {
        const ulonglong2 bx = *reinterpret_cast<const ulonglong2*>(sx + j);
        const ulonglong2 by = *reinterpret_cast<const ulonglong2*>(sy + j);
        const ulonglong2 bz = *reinterpret_cast<const ulonglong2*>(sz + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const u64 v0 = ffma2(az[r], bz.x, ffma2(ay[r], by.x, ffma2(ax[r], bx.x, nt2)));
            const u64 v1 = ffma2(az[r], bz.y, ffma2(ay[r], by.y, ffma2(ax[r], bx.y, nt2)));
            e[r][0] = lo_of(v0);
            e[r][1] = hi_of(v0);
            e[r][2] = lo_of(v1);
            e[r][3] = hi_of(v1);
        }
    } else {
        const u64 bx = *reinterpret_cast<const u64*>(sx + j);
        const u64 by = *reinterpret_cast<const u64*>(sy + j);
        const u64 bz = *reinterpret_cast<const u64*>(sz + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const u64 v0 = ffma2(az[r], bz, ffma2(ay[r], by, ffma2(ax[r], bx, nt2)));
            e[r][0] = lo_of(v0);
            e[r][1] = hi_of(v0);
        }
    }
}

// ---- packed 3-D screen values: e'[r][u] = fma(dz,dz, fma(dy,dy, fma(dx,dx, -H)))
// with d = a - b, the negation of the fast test H - |a' - b'|^2: a pair can be
// in range only where e' <= 0 (sign bit set or zero).
template <int R, int U>
__device__ __forceinline__ void euclid_group2(float (&e)[R][U], const u64 (&ax)[R], const u64 (&ay)[R],
                                              const u64 (&az)[R], const float* sx, const float* sy,
                                              const float* sz, int j, u64 nh2) {
    static_assert(U == 2 || U == 4, "j-points per group");
    constexpr int P = U / 2;
    u64 bx[P], by[P], bz[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        bx[p] = *reinterpret_cast<const u64*>(sx + j + 2 * p);
        by[p] = *reinterpret_cast<const u64*>(sy + j + 2 * p);
        bz[p] = *reinterpret_cast<const u64*>(sz + j + 2 * p);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const u64 dx = fsub2(ax[r], bx[p]), dy = fsub2(ay[r], by[p]), dz = fsub2(az[r], bz[p]);
            const u64 v = ffma2(dz, dz, ffma2(dy, dy, ffma2(dx, dx, nh2)));
            e[r][2 * p] = lo_of(v);
            e[r][2 * p + 1] = hi_of(v);
        }
    }
}

// Slow path of the angular screen for a group of U j (warp-uniform), all R
// pairs of every lane, branch-free: the LUT cell of e is k = rne(sat(e *
// 2^-q) * 2^14), read as the low bits of fma(v, 2^14, 2^23); a settled entry
// is the pair's row, so the pair costs one shared load and one shared
// reduction.  The loads of i-point r + 1 are issued before the reductions of
// i-point r (shared loads and reductions stay in program order).  Pairs
// beyond the range land in the skip code or (TPCF_F_CHECK_OVERFLOW) the
// overflow row; on masked tiles, pairs that must not be counted (padding,
// j <= i on the diagonal) are forced to the skip code.  Returns the lane's
// unsettled pairs (bit 31 of the entry), pair k = r U + u at bit U R - 1 - k.
template <int T, int R, int U, bool MASKED>
__device__ __forceinline__ uint32_t slow_group(const WorkDesc& wd, const u64 (&ax2)[R], const u64 (&ay2)[R],
                                               const u64 (&az2)[R], const float* sx, const float* sy,
                                               const float* sz, int jj, uint32_t ibase, uint32_t jbase, int diag,
                                               uint32_t na, uint32_t nb, const HistCol& hc) {
    static_assert(U * R <= 32, "one bit per pair of the group");
    float e[R][U];
    screen_group2<R, U>(e, ax2, ay2, az2, sx, sy, sz, jj, wd.neg_fast_t2);  // as the fast loop
    uint32_t valid = ~0u;
    if constexpr (MASKED) valid = valid_pairs<R, U>(ibase, jbase + (uint32_t)jj, na, nb, diag);
    const uint32_t lut_adj = smem_addr(dyn_smem) + wd.off_lut - 0x4B000000u * 2u;  // + 2 bits(f): entry
    uint32_t ent[2][U];
    uint32_t um = 0;  // unsettled pairs of this lane: pair k = r * U + u at bit U * R - 1 - k
#pragma unroll
    for (int r = 0; r < R + 1; ++r) {
        if (r < R) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float v = __saturatef(e[r][u] * wd.lut_scale);
                const float f = fmaf(v, (float)(1 << kLutBits), 8388608.0f);
                asm volatile("ld.shared.s16 %0, [%1];" : "=r"(ent[r & 1][u]) : "r"(__float_as_uint(f) * 2u + lut_adj));
            }
        }
        if (r >= 1) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                uint32_t x = ent[(r - 1) & 1][u];
                if constexpr (MASKED) x = ((valid >> ((r - 1) * U + u)) & 1u) ? x : kLutSkip;
                // settled rows add one; skip and unsettled codes add nothing here
                if (x < kLutRowLimit) red_add_shared(hc.addr + (x << row_shift<T>()), hc.inc);
                um = __funnelshift_l(x, um, 1);  // (um << 1) | (x >> 31)
            }
        }
    }
    return um;
}

// ---- all-binary64 mode: comparisons on the integer units.  Dot products (finite):
// order_key(a) > order_key_thr(b) exactly when a > b, <= exactly when a <= b: the
// bits as a signed integer, the magnitude bits flipped below zero; a threshold of -0
// counts as +0, a value of -0 lies below it.  Squared distances (+0 and up, or NaN
// between two padding points of a jackknife's rows): the bits unsigned, in which a NaN
// of either sign lies above every threshold.
// The binary64 unit is the bound, and a comparison there costs as much as a
// product (six operations a pair with it, five without): 30,011 + 30,011 points
// on an octant 28.7 -> 26.0 ms with four warps an SM, 17.5 ms with sixteen.
__device__ __forceinline__ long long order_key(double a) {
    const long long b = __double_as_longlong(a);
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ long long order_key_thr(double a) {
    const long long b = __double_as_longlong(a);
    return (b << 1) == 0 ? 0 : b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}

__device__ __forceinline__ u64 distance_key(double a) { return (u64)__double_as_longlong(a); }
__device__ __forceinline__ u64 distance_key_thr(double a) {
    const u64 b = (u64)__double_as_longlong(a);
    return (b << 1) == 0ull ? 0ull : b;
}

// Slow path of the 3-D variant for a group of U j: z = fl32(|a' - b'|^2) is
// recomputed for all R pairs of every lane, its constant-ratio LUT cell gives
// a settled row (one shared load, one reduction) or the edges left open,
// which the warp's queue of unsettled pairs settles.  Same
// load-before-reduction pipelining, masking and return value as the angular
// slow path.
template <int T, int R, int U, bool MASKED>
__device__ __forceinline__ uint32_t slow_group_euclid(const WorkDesc& wd, const u64 (&ax2)[R],
                                                      const u64 (&ay2)[R], const u64 (&az2)[R], const float* sx,
                                                      const float* sy, const float* sz, int jj, uint32_t ibase,
                                                      uint32_t jbase, int diag, uint32_t na, uint32_t nb,
                                                      const HistCol& hc) {
    static_assert(U * R <= 32, "one bit per pair of the group");
    const uint32_t lut_base = smem_addr(dyn_smem) + wd.off_lut;
    float fx[R], fy[R], fz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        fx[r] = lo_of(ax2[r]);
        fy[r] = lo_of(ay2[r]);
        fz[r] = lo_of(az2[r]);
    }
    float bx[U], by[U], bz[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        bx[u] = sx[jj + u];
        by[u] = sy[jj + u];
        bz[u] = sz[jj + u];
    }
    uint32_t valid = ~0u;
    if constexpr (MASKED) valid = valid_pairs<R, U>(ibase, jbase + (uint32_t)jj, na, nb, diag);
    uint32_t ent[2][U];
    uint32_t um = 0;  // unsettled pairs of this lane: pair k = r * U + u at bit U * R - 1 - k
#pragma unroll
    for (int r = 0; r < R + 1; ++r) {
        if (r < R) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float z = euclid_z(fx[r], fy[r], fz[r], bx[u], by[u], bz[u]);
                asm volatile("ld.shared.s16 %0, [%1];" : "=r"(ent[r & 1][u]) : "r"(euclid_cell_addr(wd, z, lut_base)));
            }
        }
        if (r >= 1) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                uint32_t x = ent[(r - 1) & 1][u];
                if constexpr (MASKED) x = ((valid >> ((r - 1) * U + u)) & 1u) ? x : kLutSkip;
                if (x < kLutRowLimit) red_add_shared(hc.addr + (x << row_shift<T>()), hc.inc);
                um = __funnelshift_l(x, um, 1);
            }
        }
    }
    return um;
}

// The sphere of a warp's 32 R i-points (R / 4 consecutive groups): centre the
// FP32 mean of the groups' centres, radius max_k |c - c_k| + r_k (enlarged by
// 2^-20 relative); empty groups (radius -1e30) are left out.
template <int R>
__device__ __forceinline__ float4 warp_sphere(const float4* caps) {
    static_assert((32 * R) % kCapPoints == 0, "whole groups per warp");
    constexpr int K = 32 * R / kCapPoints;
    float4 g[K];
    float sx = 0.f, sy = 0.f, sz = 0.f;
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        g[k] = __ldg(caps + k);
        if (g[k].w > -1e29f) {
            sx += g[k].x;
            sy += g[k].y;
            sz += g[k].z;
            ++cnt;
        }
    }
    if (cnt == 0) return make_float4(0.f, 0.f, 0.f, -1e30f);
    const float inv = 1.0f / (float)cnt;
    const float cx = sx * inv, cy = sy * inv, cz = sz * inv;
    float r = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (g[k].w > -1e29f) {
            const float dx = cx - g[k].x, dy = cy - g[k].y, dz = cz - g[k].z;
            r = fmaxf(r, sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx))) + g[k].w);
        }
    }
    return make_float4(cx, cy, cz, r * (1.0f + kPruneMargin));
}

struct PruneSlot {
    float4 sphere;          // the warp's i-points
    const float4* b_caps;   // spheres of the current sub-problem's B
    unsigned long long pruned;  // pair slots skipped by this warp
};
static_assert(sizeof(PruneSlot) == kPruneSlotBytes, "prune slot layout");

// One pruning test for the warp's i-points against the kCapPoints-point group
// holding j-point jg0 of B (warp-uniform); lane 0 counts the skipped slots.
__device__ __forceinline__ bool prune_chunk(const WorkDesc& wd, uint32_t jg0, uint32_t slots) {
    PruneSlot* ps = sptr<PruneSlot>(wd.off_icap + (threadIdx.x >> 5) * kPruneSlotBytes);
    const float4 ic = ps->sphere;
    const float4 jc = __ldg(ps->b_caps + jg0 / kCapPoints);
    if (!prune_block(wd, ic, jc)) return false;
    if ((threadIdx.x & 31) == 0) ps->pruned += slots;
    return true;
}

// ============================================================== the counting kernel
// T threads, R i-points per thread, MODE: KernelMode.
//
// Every warp is a worker of its own: it draws items (its 32 R i-points x a
// j-chunk) from the launch's counter and streams their j-tiles through its
// own ring of S shared-memory stages; tile seq of the warp lives in stage
// seq % S, whose full mbarrier completes when the tile's TMA bulk copies land
// (the stage record says which item and tile it holds).  Lane 0 refills a
// stage with tile seq + S as soon as the warp has finished tile seq.  Warps
// share only read-only block data (bins, LUT) and the words of their 16-bit
// counters (two threads' halves each, updated atomically), so none ever
// waits for another.  Every wait is bounded; a timeout sets the block's abort
// word and the call's error word, after which no copy is issued, warps leave
// their loops and each waits (bounded) for its own copies in flight.
template <int T, int R, int MODE, bool PREEMPT>
__global__ void __launch_bounds__(T, 1) count_kernel(const __grid_constant__ WorkDesc wd) {
    constexpr bool PLAIN = MODE == kModePlain;
    constexpr bool EUCLID = MODE == kModeEuclid;
    constexpr int W = T / 32;
    constexpr int U = 32 / R;          // j-points per group (screen kernels)
    constexpr uint32_t IB = 32u * R;   // i-points per warp item
    const uint32_t S = wd.stages;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    volatile int* ctl = sptr<volatile int>(wd.off_ctl);
    const bool check = (wd.flags & TPCF_F_CHECK_OVERFLOW) != 0;

    // ---- block set-up: control words, counters, bins, barriers (all sub-problems share the bins)
    for (int k = tid; k < kCtlWords; k += T) ctl[k] = 0;
    if (tid < W) sptr<PruneSlot>(wd.off_icap + (uint32_t)tid * kPruneSlotBytes)->pruned = 0ull;
    {
        uint32_t* hist = sptr<uint32_t>(wd.off_hist);
        for (int k = tid; k < (wd.nedges_max + 1) * (T / 2); k += T) hist[k] = 0;
    }
    load_bins<T>(sub_of(wd, 0).bins, wd, PLAIN);
    // the warp's S barriers, stage records and stages (recomputed where used: no registers held)
#define TPCF_BARS (sptr<uint64_t>(wd.off_bars) + (uint32_t)warp * S)
#define TPCF_META (sptr<TileMeta>(wd.off_meta) + (uint32_t)warp * S)
#define TPCF_STAGE_BASE (wd.off_stage + (uint32_t)warp * S * wd.stage_bytes)
    if (lane == 0) {
        for (uint32_t s = 0; s < S; ++s) mbar_init(&TPCF_BARS[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    const HistCol hc = hist_col<T>(wd);

    // Lane 0 copies the tile at cursor p into stage seq % S and records it there.
    auto issue = [&](uint32_t seq, const Cursor& p) {
        if (lane != 0) return;
        if ((wd.flags & TPCF_F_TEST_WAIT_TIMEOUT) && seq == 0) return;  // test hook: never issued
        const uint32_t s = seq % S;
        const SubProblem& sp = sub_of(wd, p.sub);
        const uint32_t jbase = p.g.j0 + p.t * wd.J;
        TPCF_META[s] = TileMeta{p.q, p.t | ((uint32_t)p.sub << 16), p.g.i0, p.g.j0};
        unsigned char* dst = sptr<unsigned char>(TPCF_STAGE_BASE + s * wd.stage_bytes);
        uint64_t* bar = &TPCF_BARS[s];
        fence_proxy_async_smem();  // the warp's reads of the stage's previous tile come first
        mbar_expect_tx(bar, wd.stage_bytes);
        if constexpr (PLAIN) {
            bulk_copy_g2s(dst, sp.b64 + jbase, wd.stage_bytes, bar);
        } else {
            // the x | y | z arrays of the tile's blocks (J is a multiple of kBlk)
            const unsigned char* src = sp.b_blk + (size_t)(jbase / kBlk) * kBlkBytes + kBlkX;
            for (uint32_t o = 0; o < wd.stage_bytes; o += kBlk * 12u, src += kBlkBytes)
                bulk_copy_g2s(dst + o, src, kBlk * 12u, bar);
        }
    };

    // ---- the warp's state
    uint32_t seq = 0, issued = 0;  // tiles consumed / issued so far (tile k: stage k % S)
    int cur_sub = -1;
    uint32_t cur_q = 0xffffffffu;
    uint32_t g_i0 = 0, g_j0 = 0;  // first i and j of the item the warp counts
    unsigned long long* cur_hist = nullptr;  // the histogram this warp's counters belong to
    uint32_t inc_bound = 0;  // bound on the increments of any of the lane's counters since its merge
    u64 ax2[PLAIN ? 1 : R], ay2[PLAIN ? 1 : R], az2[PLAIN ? 1 : R];
    double dx[PLAIN ? R : 1], dy[PLAIN ? R : 1], dz[PLAIN ? R : 1];
    uint32_t ibase = 0;
    uint32_t band_cnt = 0, mism_cnt = 0;  // pairs rechecked in binary64 / whose FP32-only bin differed
    bool aborted = false;

    // ---- the warp's loop over its items: the first S tiles, then each tile in
    // turn, its stage refilled with the tile S ahead
    Cursor prod;
    draw_next<PREEMPT>(wd, prod, wd.stats + kStatNextItem);
    for (; issued < seq + S && prod.valid; ++issued) {
        issue(issued, prod);
        advance<PREEMPT>(wd, prod, wd.stats + kStatNextItem);
    }
    for (; seq < issued; ++seq) {
        // ---- wait for tile seq
        const uint32_t s = seq % S;
        const bool ok = mbar_wait_bounded(&TPCF_BARS[s], (seq / S) & 1u, wd.wait_limit_ns);
        if (__any_sync(0xffffffffu, !ok)) {
            if (lane == 0) {
                ctl[kCtlAbort] = 1;
                atomicOr(wd.stats + kStatError, (unsigned long long)kErrWaitTimeout);
            }
            aborted = true;
            break;
        }
        if (ctl[kCtlAbort]) { aborted = true; break; }
        const volatile TileMeta* vm = TPCF_META + s;
        const uint32_t tm_q = vm->q, tm_ts = vm->t_sub;
        const uint32_t tm_t = tm_ts & 0xffffu;

        if (tm_q != cur_q) {
            // ---- a new item (warp-uniform)
            const int c_sub = (int)(tm_ts >> 16);
            g_i0 = vm->i0;
            g_j0 = vm->j0;
            const SubProblem& sp = sub_of(wd, c_sub);
            unsigned long long* tgt = sp.hist;
            if (sp.row_seg) tgt += (size_t)__ldg(sp.row_seg + g_i0 / kSegAlign) * sp.row_stride;
            if (c_sub != cur_sub || tgt != cur_hist) {
                if (cur_sub >= 0 && tgt != cur_hist) {
                    merge_hist<T>(hc, wd.ne, check, cur_hist);
                    inc_bound = 0;
                }
                cur_sub = c_sub;
                cur_hist = tgt;
            }
            cur_q = tm_q;
            ibase = g_i0 + (uint32_t)lane;
            if (wd.prune) {
                const float4 sph = warp_sphere<R>(sp.a_caps + g_i0 / kCapPoints);
                if (lane == 0) {
                    PruneSlot* ps = sptr<PruneSlot>(wd.off_icap + (uint32_t)warp * kPruneSlotBytes);
                    ps->sphere = sph;
                    ps->b_caps = sp.b_caps;
                }
                __syncwarp();
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint32_t i = ibase + 32u * r;
                if constexpr (PLAIN) {
                    const Point64 p = ldg_point(sp.a64 + i);
                    dx[r] = p.x;
                    dy[r] = p.y;
                    dz[r] = p.z;
                } else {
                    const float3 p = ldg_point32(sp.a_blk, i);
                    ax2[r] = pack2(p.x, p.x);
                    ay2[r] = pack2(p.y, p.y);
                    az2[r] = pack2(p.z, p.z);
                }
            }
        }

        // ---- merge the 16-bit counters before any can wrap: during a tile a lane
        // adds one for each of its R J pairs that it settles itself (or, with
        // TPCF_F_CHECK_OVERFLOW, that the fast loop rejects) plus one per queue
        // batch of the warp (each pair is queued at most once: at most R J + 1
        // batches), so at most 2 R J + 1; after the tile, the R J and the
        // batches that actually ran are added to the bound
        if (inc_bound + 2u * R * wd.J + 1u > 0xffffu) {
            merge_hist<T>(hc, wd.ne, check, cur_hist);
            inc_bound = 0;
        }
        uint32_t nbatch = 0;

        const SubProblem& sp = sub_of(wd, cur_sub);
        const uint32_t na = sp.na, nb = sp.nb;
        const uint32_t jbase = g_j0 + tm_t * wd.J;
        const int J = (int)wd.J;
        // tiles that meet the diagonal: j > i (auto counts) or j != i (full square without self pairs)
        int diag = kDiagNone;
        if (jbase < g_i0 + IB) {
            if (sp.auto_mode) diag = kDiagAbove;
            else if (sp.no_self && jbase + wd.J > g_i0) diag = kDiagOffSelf;
        }
        // tiles holding padding (points past na or nb) are masked where padding could
        // look in range (need_idx) and whenever overflow is counted
        const bool edge = jbase + wd.J > nb || g_i0 + IB > na;
        const bool masked = diag != kDiagNone || (edge && (wd.need_idx || check));
        const uint32_t stage_off = TPCF_STAGE_BASE + s * wd.stage_bytes;

        if constexpr (PLAIN) {
            const Point64* sj = sptr<const Point64>(stage_off);
            const double* cthr = sptr<const double>(wd.off_cthr);
            const int ne = wd.ne;
            const long long last = order_key_thr(wd.cos_last);
            const u64 last2 = distance_key_thr(wd.cos_last);  // (3-D)
            for (int jj = 0; jj < J; ++jj) {
                const Point64 b = sj[jj];
                const uint32_t jg = jbase + (uint32_t)jj;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t ig = ibase + 32u * r;
                    const bool valid = ig < na && jg < nb && (!masked || (diag == kDiagAbove ? jg > ig
                                                                          : (diag == kDiagOffSelf ? jg != ig : true)));
                    if (wd.euclid) {
                        // 3-D: h = number of edges m with d^2 >= S_m (S increasing); d^2 >= S_B is overflow
                        const double ex = __dsub_rn(dx[r], b.x), ey = __dsub_rn(dy[r], b.y), ez = __dsub_rn(dz[r], b.z);
                        const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
                        const u64 k2 = distance_key(d2);
                        if (k2 < last2 && valid) {
                            int lo = 0, hi = ne;
                            while (lo < hi) {
                                const int mid = (lo + hi) >> 1;
                                if (k2 >= distance_key_thr(cthr[mid])) lo = mid + 1; else hi = mid;
                            }
                            hist_inc<T>(hc, lo);
                        } else if (check && valid) {
                            hist_inc<T>(hc, ne);
                        }
                        continue;
                    }
                    const double d = __dadd_rn(__dadd_rn(__dmul_rn(dx[r], b.x), __dmul_rn(dy[r], b.y)),
                                               __dmul_rn(dz[r], b.z));
                    const long long kd = order_key(d);
                    if (kd > last && valid) {
                        // h = number of edges m with d <= C_m (C decreasing)
                        int lo = 0, hi = ne;
                        while (lo < hi) {
                            const int mid = (lo + hi) >> 1;
                            if (order_key_thr(cthr[mid]) >= kd) lo = mid + 1; else hi = mid;
                        }
                        hist_inc<T>(hc, lo);
                    } else if (check && valid) {
                        hist_inc<T>(hc, ne);
                    }
                }
            }
        } else {
            // Fast loop: the screen values of a group of U j-points and the lane's R
            // i-points (packed FMA); one bit per group says whether some pair of the
            // lane may be in range (angles: some e >= 0; 3-D: some e' <= 0).  The loop
            // does not branch per group: after kMaskGroups groups one warp reduction
            // names the groups that take the slow path, which recomputes their values.
            // (the tile: blocks of kBlk points, x | y | z each)
            const float* const tile = sptr<const float>(stage_off);
            // angles: (-T, -T); 3-D: (-H, -H), read from the kernel parameter
            const u64 nt2 = wd.neg_fast_t2;
            constexpr int CH = kMaskGroups * U;                     // j-points per mask chunk
            uint32_t* uq = sptr<uint32_t>(wd.off_queue) + (uint32_t)warp * kUQueue;
            uint32_t qn = 0;  // codes in the warp's queue of unsettled pairs
            PairSource<R> src;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                src.x[r] = lo_of(ax2[r]);
                src.y[r] = lo_of(ay2[r]);
                src.z[r] = lo_of(az2[r]);
            }
            src.tile = tile;
            src.i0 = g_i0;
            src.jbase = jbase;
            static_assert(kMaskGroups <= 32, "one mask bit per group");
#pragma unroll 1
            for (int jc = 0; jc < J; jc += CH) {
                if (wd.prune && prune_chunk(wd, jbase + (uint32_t)jc, IB * CH)) continue;
                // a chunk lies in one block: its points j at sx[j], sy[j], sz[j] (j from the tile's first)
                static_assert((int)kBlk % CH == 0, "a chunk lies in one block");
                const float* const sx = tile + 2 * (jc & ~((int)kBlk - 1));
                const float* const sy = sx + kBlk;
                const float* const sz = sy + kBlk;
                uint32_t lane_mask = 0;
#pragma unroll 4
                for (int gi = 0; gi < kMaskGroups; ++gi) {
                    float e[R][U];
                    if constexpr (EUCLID) {
                        euclid_group2<R, U>(e, ax2, ay2, az2, sx, sy, sz, jc + gi * U, nt2);
                        // OR of the sign bits: 1 when some e' <= 0 (e' = -0 cannot occur)
                        lane_mask = __funnelshift_l(lop_tree<U * R, true>(reinterpret_cast<const uint32_t*>(&e[0][0])),
                                                    lane_mask, 1);
                    } else {
                        screen_group2<R, U>(e, ax2, ay2, az2, sx, sy, sz, jc + gi * U, nt2);
                        // (~AND) >> 31: 1 when some screen value of the group is >= 0
                        lane_mask = __funnelshift_l(~lop_tree<U * R, false>(reinterpret_cast<const uint32_t*>(&e[0][0])),
                                                    lane_mask, 1);
                    }
                }
                uint32_t m = __reduce_or_sync(0xffffffffu, lane_mask);  // bit kMaskGroups - 1 - gi: group gi
                if (check) {
                    // overflow counted: the lane's pairs of every group the fast loop
                    // rejected are overflow; masked tiles take every group slowly
                    if (masked) m = 0xffffffffu;
                    const uint32_t nfast = (uint32_t)kMaskGroups - (uint32_t)__popc(m);
                    if (nfast) red_add_shared(hc.addr + ((uint32_t)wd.ne << row_shift<T>()), hc.inc * nfast * (uint32_t)(U * R));
                }
#pragma unroll 1
                while (m) {
                    const int gi = kMaskGroups - __ffs(m);  // lowest set bit first
                    m &= m - 1u;
                    const int jj = jc + gi * U;
                    uint32_t um;
                    if constexpr (EUCLID) {
                        um = masked ? slow_group_euclid<T, R, U, true>(wd, ax2, ay2, az2, sx, sy, sz, jj, ibase, jbase, diag, na, nb, hc)
                                    : slow_group_euclid<T, R, U, false>(wd, ax2, ay2, az2, sx, sy, sz, jj, ibase, jbase, diag, na, nb, hc);
                    } else {
                        um = masked ? slow_group<T, R, U, true>(wd, ax2, ay2, az2, sx, sy, sz, jj, ibase, jbase, diag, na, nb, hc)
                                    : slow_group<T, R, U, false>(wd, ax2, ay2, az2, sx, sy, sz, jj, ibase, jbase, diag, na, nb, hc);
                    }
                    enqueue_unsettled<T, R, U, EUCLID>(wd, sp, um, jj, uq, qn, nbatch, src, hc, band_cnt, mism_cnt);
                }
            }
            // the queue's last codes, before the warp leaves the tile
            if (qn) {
                __syncwarp();
                drain_batch<T, R, EUCLID>(wd, sp, uq, qn, src, hc, band_cnt, mism_cnt);
                ++nbatch;
                __syncwarp();
            }
        }

        inc_bound += (uint32_t)R * wd.J + nbatch;

        // ---- refill this stage with tile seq + S
        __syncwarp();
        if (prod.valid && !ctl[kCtlAbort]) {
            issue(seq + S, prod);
            ++issued;
            advance<PREEMPT>(wd, prod, wd.stats + kStatNextItem);
        }
    }
    // ---- merge this warp's columns (skipped after an abort: outputs are invalid)
    if (!aborted && cur_sub >= 0) {
        merge_hist<T>(hc, wd.ne, check, cur_hist);
    }
    if constexpr (!PLAIN) {
        const unsigned long long b = warp_sum(band_cnt), mm = warp_sum(mism_cnt);
        if (lane == 0) {
            if (b) atomicAdd(wd.stats + kStatBand, b);
            if (mm) atomicAdd(wd.stats + kStatMismatch, mm);
        }
    }
    if (wd.prune && lane == 0) {
        const unsigned long long np = sptr<PruneSlot>(wd.off_icap + (uint32_t)warp * kPruneSlotBytes)->pruned;
        if (np) atomicAdd(wd.stats + kStatPruned, np);
    }
    // ---- after an abort, wait (bounded) for this warp's copies still in flight
    if (aborted && lane == 0) {
        for (uint32_t s2 = seq; s2 < issued; ++s2) {
            if ((wd.flags & TPCF_F_TEST_WAIT_TIMEOUT) && s2 == 0) continue;
            (void)mbar_wait_bounded(&TPCF_BARS[s2 % S], (s2 / S) & 1u, wd.wait_limit_ns);
        }
    }
#undef TPCF_BARS
#undef TPCF_META
#undef TPCF_STAGE_BASE
}

// ============================================================== finalize
// out[h] = acc[h] for h < nedges (underflow and bins).  Overflow: without
// count_over, out[nedges] = total - sum, or UINT64_MAX (and kErrBadHist in the
// error word) when the sum exceeds the total; with count_over (the kernel
// counted it), out[nedges] = acc[nedges] and the whole sum must equal the
// total (else kErrBadHist and overflow UINT64_MAX).  acc and out may alias.
__device__ void finalize_one(const unsigned long long* acc, int nedges, unsigned long long* out,
                             unsigned long long total, int count_over, unsigned long long* err_word,
                             unsigned long long* part) {
    const int nsum = count_over ? nedges + 1 : nedges;
    unsigned long long s = 0;
    for (int h = threadIdx.x; h < nsum; h += blockDim.x) s += acc[h];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
        __syncthreads();
    }
    const unsigned long long sum = part[0];
    const unsigned long long over = count_over ? acc[nedges] : 0ull;
    __syncthreads();  // every thread has read acc before out (possibly the same memory) is written
    for (int h = threadIdx.x; h < nedges; h += blockDim.x) out[h] = acc[h];
    if (threadIdx.x == 0) {
        // (count_over 2: a test hook that checks against total + 1, so the check fails)
        const bool bad = count_over ? sum != (count_over == 2 ? total + 1 : total) : sum > total;
        if (bad) {
            atomicOr(err_word, (unsigned long long)kErrBadHist);
            out[nedges] = ~0ull;  // sentinel
        } else {
            out[nedges] = count_over ? over : total - sum;
        }
    }
}

__global__ void finalize_kernel(unsigned long long* acc, int nedges, unsigned long long* out,
                                unsigned long long total, int count_over, unsigned long long* err_word) {
    __shared__ unsigned long long part[256];
    finalize_one(acc, nedges, out, total, count_over, err_word, part);
}

// Batched finalize: block b turns accumulator row b (stride acc_stride words)
// into histogram b of `out` (stride out_stride words) with pair total totals[b].
__global__ void finalize_batch_kernel(const unsigned long long* acc, int acc_stride, int nedges,
                                      unsigned long long* out, int out_stride, const unsigned long long* totals,
                                      int count_over, unsigned long long* err_word) {
    __shared__ unsigned long long part[256];
    finalize_one(acc + (size_t)blockIdx.x * acc_stride, nedges, out + (size_t)blockIdx.x * out_stride,
                 totals[blockIdx.x], count_over, err_word, part);
}

cudaError_t launch_finalize_batch(const unsigned long long* acc, int acc_stride, int nedges,
                                  unsigned long long* out, int out_stride, const unsigned long long* totals,
                                  int count, int count_over, unsigned long long* err_word, cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    finalize_batch_kernel<<<count, 256, 0, stream>>>(acc, acc_stride, nedges, out, out_stride, totals, count_over,
                                                     err_word);
    return cudaGetLastError();
}

cudaError_t launch_finalize(unsigned long long* acc, int nedges, unsigned long long* out,
                            unsigned long long total, int count_over, unsigned long long* err_word,
                            cudaStream_t stream) {
    finalize_kernel<<<1, 256, 0, stream>>>(acc, nedges, out, total, count_over, err_word);
    return cudaGetLastError();
}

// ============================================================== launchers
// Fills the block constants of the work description (shared-memory offsets of
// the shape, merge interval) and launches.
template <int T, int R, int MODE, bool PREEMPT = false>
static cudaError_t launch_t(const WorkDesc& wd_in, const Shape& sh, cudaStream_t stream) {
    WorkDesc wd = wd_in;
    const SmemLayout L = smem_layout(MODE, T, (int)wd.J, (int)wd.stages, wd.nedges_max);
    wd.off_ctl = L.ctl;
    wd.off_bars = L.bars;
    wd.off_meta = L.meta;
    wd.off_stage = L.stage;
    wd.off_hist = L.hist;
    wd.off_cthr = L.cos_thr;
    wd.off_lo = L.lo;
    wd.off_hi = L.hi;
    wd.off_c32 = L.cos32;
    wd.off_zlo = L.zlo;
    wd.off_zhi = L.zhi;
    wd.off_lut = L.lut;
    wd.off_queue = L.queue;
    wd.off_icap = L.icap;
    wd.stage_bytes = wd.J * staged_point_bytes(MODE);
    // the 16-bit counters' merge interval is bounded in the kernel, per tile
    wd.flush_limit = 0xffffu;
    if (L.total > sh.smem || wd.I != 32u * (uint32_t)R) return cudaErrorInvalidValue;
    // the draw order is laid out for this launch's warps unless the caller fixed it
    // (continuations of a preempted launch keep the order of the first)
    if (wd.draw_warps == 0) wd.draw_warps = (uint32_t)sh.blocks * (uint32_t)(T / 32);
    count_kernel<T, R, MODE, PREEMPT><<<sh.blocks, T, sh.smem, stream>>>(wd);
    return cudaGetLastError();
}

// The limit is raised to the device's opt-in maximum rather than to `bytes`:
// the attribute belongs to the kernel, not to a launch, so a smaller value set
// by one host thread could otherwise undercut a concurrent launch of another.
template <int T, int R, int MODE, bool PREEMPT = false>
static cudaError_t set_smem_t(size_t bytes) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (bytes > (size_t)optin) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(count_kernel<T, R, MODE, PREEMPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                optin);
}

// The job server's steps of jobs whose histograms do not fit the tensor-core
// kernel (133 to 136 edges) and of binary64 contexts: the 512 x 8 screen kernel
// with preemptible draws (a start position and the yield word).
cudaError_t launch_count_preemptible(const WorkDesc& wd, const Shape& sh, cudaStream_t stream) {
    if (sh.threads != 512 || sh.ipt != 8) return cudaErrorInvalidConfiguration;
    return launch_t<512, 8, kModeScreen, true>(wd, sh, stream);
}

cudaError_t count_preemptible_set_smem_limit(size_t bytes) {
    return set_smem_t<512, 8, kModeScreen, true>(bytes);
}

#define TPCF_SHAPES(X) X(128, 8) X(256, 8) X(512, 8) X(256, 16)

cudaError_t launch_count(const WorkDesc& wd, const Shape& sh, int mode, int nedges, cudaStream_t stream) {
    (void)nedges;
#define X(T_, R_)                                                                      \
    if (sh.threads == T_ && sh.ipt == R_) {                                            \
        if (mode == kModePlain) return launch_t<T_, R_, kModePlain>(wd, sh, stream);   \
        if (mode == kModeEuclid) return launch_t<T_, R_, kModeEuclid>(wd, sh, stream); \
        return launch_t<T_, R_, kModeScreen>(wd, sh, stream);                          \
    }
    TPCF_SHAPES(X)
#undef X
    return cudaErrorInvalidConfiguration;
}

cudaError_t count_set_smem_limit(int mode, int threads, int ipt, size_t bytes) {
#define X(T_, R_)                                                              \
    if (threads == T_ && ipt == R_) {                                          \
        if (mode == kModePlain) return set_smem_t<T_, R_, kModePlain>(bytes);  \
        if (mode == kModeEuclid) return set_smem_t<T_, R_, kModeEuclid>(bytes); \
        return set_smem_t<T_, R_, kModeScreen>(bytes);                         \
    }
    TPCF_SHAPES(X)
#undef X
    return cudaErrorInvalidConfiguration;
}

bool count_shape_supported(int threads, int ipt) {
#define X(T_, R_) if (threads == T_ && ipt == R_) return true;
    TPCF_SHAPES(X)
#undef X
    return false;
}

size_t count_smem_bytes(int mode, int threads, int ipt, int jtile, int stages, int nedges) {
    (void)ipt;
    return smem_layout(mode, threads, jtile, stages, nedges).total;
}

}  // namespace tpcf
