// CUDA counting kernel (sm_103a) whose screen runs on the tensor cores.
//
// Paper: Ponce et al., "Application of GPUs for the calculation of two point
// correlation functions in cosmology", Section 3: the dot product of each
// pair, its bin, partial histograms combined into one.  Here the dot products
// of a block of pairs are one small matrix product, which serves only to
// reject: a 32 x 32 block of pairs none of which can lie within the last edge
// is overflow and needs nothing more.  Every other block is classified as in
// count.cu: FP32 screen value, lookup table, chord refinement, binary64.
//
// The screen as a contraction.  The FP32 coordinates are split into two
// binary16 values, a = a1 + a2 + r with |r| <= 2^-22 |a| + 2^-25, and a pair's
// screen value is the K = 16 product
//   D = sum_c a1 b1 + a2 b2 + a1 b2 + a2 b1,   c = x, y, z:
// the j-side record is [X | X] and the i-side record [X | Y] with X = (x1, y1,
// z1, x2, y2, z2, 0, 0) and Y = (x2, y2, z2, x1, y1, z1, 0, 0).  Products of
// binary16 values are exact in binary32; with accumulation in at least single
// precision D is within 44u of the binary64 dot d (u = 2^-24: 2u from the FP32
// copies, 9.8u from the split, at most one unit 2u in the last place for each
// of 16 additions of partial sums below 1.002; measured, through
// tpcf_debug_screen_values: at most 4.3u).  A block is rejected when
// every D < tc_thr = RD(C_B - 64u), which proves d < C_B for all its pairs.
//
// 3-D counts (EUCLID) reject on D = a.b - |b|^2 / 2: d^2 >= S_B is D <= (|a|^2 -
// S_B) / 2, a threshold of the lane that holds a.  The operands hold the points
// scaled by powers of two to norm <= 1 (2^-ka, 2^-kb, one per catalog); the two
// spare places of X hold n1 + n2 = -|b|^2 / 2, which the i-side meets with 0 in X
// and with s = 2^(kb - ka) in Y, so that D comes out in units of 2^(ka + kb).
// Error with t = max(s, 1/s): 2u and 9.8u as above, 5u s from |b|^2 / 2 (three
// roundings, the copies, the split), 16 additions of partial sums below 2t at 2u t,
// 8u t from the threshold (three roundings of |a|^2 / 2s, the copies, the last
// addition where the screen rejects anything): 57u t in all, kTcGuard3d = 128u
// (measured without the threshold's part: at most 2.5u t).
// 300,000 + 300,000 points, distances to 0.05 of the box: 11.2 ms (FP32
// differences on the CUDA cores: 33.2 ms, bound by their nine operations a pair).
//
// One CTA per SM, 21 warps:
//   * warps 0..15, four groups of four: group g reads the accumulators of
//     i-points 128 g .. 128 g + 127 of the CTA's 512 (tcgen05.ld with a maximum
//     over 32 columns: one comparison per 32 x 32 pairs), releases them, and
//     classifies the blocks it kept, one i-point per lane;
//   * warps 16..19: group g's tcgen05.mma issuer (M 128 x N 128 x K 16);
//   * warp 20: draws items (512 i-points x a j-chunk), finds the tiles and
//     groups that can hold countable pairs, and copies operands with TMA.
// The j-tiles (operand and FP32 coordinates, one bulk copy) are shared by the
// four groups; a group that is busy classifying holds back its own
// accumulators only, and the others run up to the ring's depth ahead.
//
// What bounds it (octant of 1,000,000 + 1,000,000 points to 10 degrees 206 ms, the
// FP32 screen of count.cu 284 ms; sphere of 700,001 x 1,400,003 to 2 degrees 50.4 ms,
// there 108 ms):
//   * a rejected tile of 512 x 128 pairs takes about 1050 cycles.  The tensor core
//     needs 128 of them and reading the accumulators 344; the rest is the chain
//     from one product of a group to the next (product, commit, wait, load, vote,
//     arrival, wait): tensor memory holds one product of each group, so a group
//     has nothing else to do meanwhile;
//   * a kept 32 x 32 block takes about 2800 cycles of its warp, its unsettled pairs
//     500 (patches of close points: 1600), and, with all warps at it, the
//     shared-memory pipe: a lookup of 32 random cells is 3.9 wavefronts, with the
//     counter and the j-points 5.6 for 32 pairs.
#include <stdint.h>

#include "count_common.cuh"

namespace tpcf {

namespace {

constexpr int kWorkWarps = 16;                    // classifying warps
constexpr int kWorkThreads = 32 * kWorkWarps;
constexpr int kGroups = 4;                        // groups of four warps: 128 i-points each
constexpr int kIssueWarp = kWorkWarps;            // .. + kGroups - 1: the groups' mma issuers
constexpr int kLoadWarp = kWorkWarps + kGroups;
constexpr int kThreads = 32 * (kLoadWarp + 1);
constexpr int kTmemCols = 512;                    // 128 columns per group
constexpr uint32_t kABlock = 2 * kBlkX;            // i-side operand of 128 points: planes X and Y
constexpr uint32_t kABytes = kGroups * kABlock;   // ... of an item
constexpr uint32_t kStageX2 = kBlkBytes;          // a stage: the tile's block (X, x | y | z), then X once more
constexpr uint32_t kStageBytes = kBlkBytes + kBlkX;
constexpr int kQueueCodes = 64;                   // per-warp queue of unsettled pairs

// Control words.  kTcBeat changes with every batch of items the loader draws and with
// whatever the warps classify (tc_beat): a wait is bounded by the time without progress.
enum TcCtl { kTcAbort = 0, kTcTmem = 1, kTcBeat = 2, kTcCtlWords = 32 };

// A staged tile: what to do with it, first j of the tile, first i of the item.
struct __align__(16) TcMeta {
    uint32_t info;   // kInfo* below, sub-problem in bits 16..31
    uint32_t jbase, i0;
    uint32_t pad;
};
enum : uint32_t {
    kInfoGroups = 0xfu,   // groups of warps that work on this tile
    kInfoABuf = 0x10u,    // operand buffer of the item
    kInfoNew = 0x20u,     // first tile of an item
    kInfoLast = 0x40u,    // last tile of an item
    kInfoStop = 0x80u,    // no tile: the launch's (or slice's) items are done
    // (PRUNE) bits 8 + 2 g, 9 + 2 g: which 128 i-points of the item group g takes
};

// Barriers (8 bytes each): full[S], empty[S], a_full[2], a_empty[2], d_full[4], d_free[4].
__host__ __device__ constexpr uint32_t tc_bar_words(uint32_t S) { return 2 * S + 4 + 2 * kGroups; }

struct TcLayout {
    uint32_t ctl, bars, meta, atile, stage, hist, cos_thr, lo, hi, cos32, zlo, zhi, lut, queue, total;
};

__host__ __device__ inline TcLayout tc_layout(int S, int nedges) {
    TcLayout L;
    uint32_t off = 0;
    L.ctl = off; off += kTcCtlWords * 4;
    L.bars = off; off += tc_bar_words((uint32_t)S) * 8;
    off = align_up(off, 16);
    L.meta = off; off += (uint32_t)S * (uint32_t)sizeof(TcMeta);
    off = align_up(off, 128);
    L.atile = off; off += 2 * kABytes;
    L.stage = off; off += (uint32_t)S * kStageBytes;
    L.hist = off; off += (uint32_t)(nedges + 1) * (uint32_t)(kWorkThreads / 2) * 4;
    off = align_up(off, 16);
    L.cos_thr = off; off += (uint32_t)nedges * 8;
    L.lo = off; off += (uint32_t)nedges * 4;
    L.hi = off; off += (uint32_t)nedges * 4;
    L.cos32 = off; off += (uint32_t)nedges * 4;
    L.zlo = off; off += (uint32_t)nedges * 4;
    L.zhi = off; off += (uint32_t)nedges * 4;
    off = align_up(off, 16);
    L.lut = off; off += (uint32_t)kLutCells * 2;
    off = align_up(off, 16);
    L.queue = off; off += (uint32_t)kWorkWarps * kQueueCodes * 4;
    off = align_up(off, 16);
    L.total = align_up(off, 16);
    return L;
}

// ============================================================== tcgen05 wrappers
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Allocation of the tensor memory (whole warp; the address goes to the shared word at `dst`).
__device__ __forceinline__ void tc_alloc(uint32_t dst) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"((uint32_t)kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tc_dealloc(uint32_t tmem) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kTmemCols));
}
// A tile record (16-byte aligned shared address).
__device__ __forceinline__ void rec_load(uint32_t a, uint32_t& info, uint32_t& jbase, uint32_t& i0) {
    [[maybe_unused]] uint32_t unused;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(info), "=r"(jbase), "=r"(i0), "=r"(unused)
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void rec_store(uint32_t a, uint32_t info, uint32_t jbase, uint32_t i0) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %3};" ::"r"(a), "r"(info), "r"(jbase), "r"(i0) : "memory");
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major operand without swizzle: rows
// in groups of 8, a group's two 8 x 16-byte core matrices at `addr` + 0 and
// + `second` (its rows of the two planes of 128 points), groups 128 bytes apart.
__device__ __forceinline__ uint64_t op_desc(uint32_t addr, uint32_t second) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)(second >> 4) << 16) | ((uint64_t)(128u >> 4) << 32) |
           (1ull << 46);
}

// D (FP32, 128 x 128) = A B^T, K = 16, binary16 operands; issued by one thread.
constexpr uint32_t kIdesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, 0, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(kIdesc)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

// 32 columns of the lane's accumulator row and their maximum, valid after tc_wait_ld.
__device__ __forceinline__ float tc_row_max32(uint32_t addr, uint32_t (&r)[32]) {
    float m;
    asm volatile(
        "tcgen05.ld.red.sync.aligned.32x32b.x32.max.f32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, %32, [%33];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=f"(m)
        : "r"(addr));
    return m;
}
// The maximum alone.
__device__ __forceinline__ float tc_row_max32(uint32_t addr) {
    [[maybe_unused]] uint32_t r[32];
    return tc_row_max32(addr, r);
}
// Waits for the warp's tensor-memory loads; the operands tie the loaded values to the wait.
__device__ __forceinline__ void tc_wait_ld(float& a, float& b) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+f"(a), "+f"(b)::"memory");
}

__device__ __forceinline__ void tc_wait_ld(float& m, uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(m), "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14])
                 :: "memory");
    asm volatile("" : "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                      "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                      "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}

// Says that the block makes progress (a clock: any other value than before will do).
__device__ __forceinline__ void tc_beat(const WorkDesc& wd) {
    sptr<volatile int>(wd.off_ctl)[kTcBeat] = (int)clock();
}

// Bounded wait of a whole warp for phase `parity` of `bar`: false (with the
// block's abort word and the call's error word set) after limit_ns in which
// nothing was drawn or classified, and false as soon as another warp has aborted.
__device__ __noinline__ bool tc_wait_slow(uint64_t* bar, uint32_t parity, uint64_t limit_ns, volatile int* ctl,
                                          unsigned long long* stats) {
    uint64_t t0 = global_ns();
    int beat = ctl[kTcBeat];
    bool ok = false;
    while (true) {
        ok = mbar_try_wait(bar, parity);
        if (ok || ctl[kTcAbort]) break;
        const int b = ctl[kTcBeat];
        if (b != beat) {
            beat = b;
            t0 = global_ns();
        } else if (global_ns() - t0 > limit_ns) {
            ctl[kTcAbort] = 1;
            atomicOr(stats + kStatError, (unsigned long long)kErrWaitTimeout);
            break;
        }
    }
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns, volatile int* ctl,
                                        unsigned long long* stats) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return tc_wait_slow(bar, parity, limit_ns, ctl, stats);
}

// The i-side operand's planes X and Y of a catalog's operand record x: X (3-D: without
// the norm), and the halves' two triples exchanged (3-D: then the scales' ratio).
template <bool EUCLID>
__device__ __forceinline__ uint4 plane_x(const uint4& x) {
    return EUCLID ? make_uint4(x.x, x.y, x.z, 0u) : x;
}
template <bool EUCLID>
__device__ __forceinline__ uint4 plane_y(const uint4& x, uint32_t pad) {
    return make_uint4((x.y >> 16) | (x.z << 16), (x.z >> 16) | (x.x << 16), (x.x >> 16) | (x.y << 16),
                      EUCLID ? pad : 0u);
}

// A sphere that holds the (non-empty) spheres of an item's groups: centre the
// FP32 mean of their centres, radius max |c - c_g| + r_g, enlarged by 2^-20.
__device__ __forceinline__ float4 union_sphere(const float4 (&g)[kGroups]) {
    float x = 0.f, y = 0.f, z = 0.f, n = 0.f;
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
        if (g[k].w > -1e29f) {
            x += g[k].x;
            y += g[k].y;
            z += g[k].z;
            n += 1.f;
        }
    }
    if (n == 0.f) return make_float4(0.f, 0.f, 0.f, -1e30f);
    const float cx = x / n, cy = y / n, cz = z / n;
    float r = 0.f;
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
        if (g[k].w > -1e29f) {
            const float dx = cx - g[k].x, dy = cy - g[k].y, dz = cz - g[k].z;
            r = fmaxf(r, sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx))) + g[k].w);
        }
    }
    return make_float4(cx, cy, cz, r * (1.0f + kPruneMargin));
}

// ============================================================== classification of a kept block
// One i-point per lane (as (a, a) pairs) against 32 staged j-points: FP32
// screen value, LUT code, one counter increment per settled pair, as the slow
// path of count.cu (the codes of a group of four j are read before the
// increments of the group before it).  `valid` (MASKED) names the lane's pairs
// that may be counted.  Returns the unsettled pairs: pair j at bit 31 - j.
template <bool EUCLID, bool MASKED>
__device__ __forceinline__ uint32_t tc_block(const WorkDesc& wd, u64 ax, u64 ay, u64 az, const float* sx,
                                             uint32_t valid, const HistCol& hc) {
    const uint32_t lut_base = smem_addr(dyn_smem) + wd.off_lut;
    const uint32_t lut_adj = lut_base - 0x4B000000u * 2u;
    const u64 nt2 = wd.neg_fast_t2;
    uint32_t ent[2][4];
    uint32_t um = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if (k < 8) {
            const ulonglong2 bx = *reinterpret_cast<const ulonglong2*>(sx + 4 * k);
            const ulonglong2 by = *reinterpret_cast<const ulonglong2*>(sx + kBlk + 4 * k);
            const ulonglong2 bz = *reinterpret_cast<const ulonglong2*>(sx + 2 * kBlk + 4 * k);
            u64 v0, v1;
            if constexpr (EUCLID) {  // z as euclid_z rounds it
                const u64 dx0 = fsub2(ax, bx.x), dy0 = fsub2(ay, by.x), dz0 = fsub2(az, bz.x);
                const u64 dx1 = fsub2(ax, bx.y), dy1 = fsub2(ay, by.y), dz1 = fsub2(az, bz.y);
                v0 = ffma2(dz0, dz0, ffma2(dy0, dy0, ffma2(dx0, dx0, 0ull)));
                v1 = ffma2(dz1, dz1, ffma2(dy1, dy1, ffma2(dx1, dx1, 0ull)));
            } else {
                v0 = ffma2(az, bz.x, ffma2(ay, by.x, ffma2(ax, bx.x, nt2)));
                v1 = ffma2(az, bz.y, ffma2(ay, by.y, ffma2(ax, bx.y, nt2)));
            }
            const float e[4] = {lo_of(v0), hi_of(v0), lo_of(v1), hi_of(v1)};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if constexpr (EUCLID) {
                    ent[k & 1][u] = (uint32_t)ld_shared_s16(euclid_cell_addr(wd, e[u], lut_base));
                } else {
                    const float v = __saturatef(e[u] * wd.lut_scale);
                    const float f = fmaf(v, (float)(1 << kLutBits), 8388608.0f);
                    ent[k & 1][u] = (uint32_t)ld_shared_s16(__float_as_uint(f) * 2u + lut_adj);
                }
            }
        }
        if (k >= 1) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t x = ent[(k - 1) & 1][u];
                if constexpr (MASKED) x = ((valid >> (4 * (k - 1) + u)) & 1u) ? x : kLutSkip;
                if (x < kLutRowLimit) red_add_shared(hc.addr + (x << row_shift<kWorkThreads>()), hc.inc);
                um = __funnelshift_l(x, um, 1);
            }
        }
    }
    return um;
}

// Classifies the n <= 32 queued pairs at q, one per lane: code = lane holding
// the i-point | j-offset from jq0 << 5.
template <bool EUCLID>
__device__ __forceinline__ void tc_drain(const WorkDesc& wd, const SubProblem& sp, const uint32_t* q, uint32_t n,
                                         u64 ax, u64 ay, u64 az, uint32_t iw, uint32_t jq0, const HistCol& hc,
                                         uint32_t& band, uint32_t& mism) {
    tc_beat(wd);
    const uint32_t lane = threadIdx.x & 31u;
    const bool has = lane < n;
    const uint32_t code = has ? q[lane] : 0u;
    const int l = (int)(code & 31u);
    const uint32_t jg = jq0 + (code >> 5);
    const float x = __shfl_sync(0xffffffffu, lo_of(ax), l);
    const float y = __shfl_sync(0xffffffffu, lo_of(ay), l);
    const float z = __shfl_sync(0xffffffffu, lo_of(az), l);
    if (has) {
        const float3 b = ldg_point32(sp.b_blk, jg);
        hist_inc<kWorkThreads>(hc, classify_unsettled<EUCLID>(wd, sp, x, y, z, b.x, b.y, b.z, iw + (uint32_t)l, jg,
                                                             band, mism));
    }
}

// Merges the warp's counters (out of line: inlined three times it made the
// loop below spill).
static __device__ __noinline__ void tc_merge(HistCol hc, int ne, bool check, unsigned long long* out) {
    warp_flush_hist<kWorkThreads>(hc, ne, check, out);
}

// ============================================================== the kernel
// PREEMPT: draws start at wd.pos_lo and stop once stats[kStatYield] is set
// (the job server's steps of one large job).  PRUNE: tiles and groups whose
// bounding spheres are too far apart are left out, and a tile's i-groups go to
// the groups of warps in turn (without pruning group g always takes i-points
// 128 g .. of the item, and its loop is the shorter for it).  CHECK: the overflow
// row is counted too (TPCF_F_CHECK_OVERFLOW; never with PRUNE), for a tile that holds
// nothing within the range in one step (600,000 + 600,000 points on the sphere to 5
// degrees: 96 ms block by block, 45 ms so, 83 ms on the FP32 kernel).
template <bool PREEMPT, bool PRUNE, bool EUCLID, bool CHECK>
__global__ void __launch_bounds__(kThreads, 1) count_tc_kernel(const __grid_constant__ WorkDesc wd) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t S = wd.stages;
    volatile int* ctl = sptr<volatile int>(wd.off_ctl);
    uint64_t* bars = sptr<uint64_t>(wd.off_bars);
    uint64_t* const full = bars;
    uint64_t* const empty = bars + S;
    uint64_t* const a_full = bars + 2 * S;
    uint64_t* const a_empty = a_full + 2;
    uint64_t* const d_full = a_full + 4;
    uint64_t* const d_free = d_full + kGroups;
    const uint32_t meta = smem_addr(dyn_smem) + wd.off_meta;
    static_assert(!(PRUNE && CHECK), "skipped blocks would have to be counted");
    constexpr bool check = CHECK;
    const uint64_t limit = wd.wait_limit_ns;

    // ---- set-up: control words, barriers, tensor memory, counters, bins
    if (tid < kTcCtlWords) ctl[tid] = 0;
    if (tid == 0) {
        for (uint32_t s = 0; s < S; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, kWorkWarps + kGroups);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(a_full + k, 1);
            mbar_init(a_empty + k, kWorkWarps + kGroups);
        }
        for (int g = 0; g < kGroups; ++g) {
            mbar_init(d_full + g, 1);
            mbar_init(d_free + g, 4);
        }
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == kIssueWarp) {
        tc_alloc(smem_addr(dyn_smem) + wd.off_ctl + 4u * kTcTmem);
    }
    {
        uint32_t* hist = sptr<uint32_t>(wd.off_hist);
        for (int k = tid; k < (wd.nedges_max + 1) * (kWorkThreads / 2); k += kThreads) hist[k] = 0;
    }
    load_bins<kThreads>(sub_of(wd, 0).bins, wd, false);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = (uint32_t)ctl[kTcTmem];

    if (warp < kWorkWarps) {
        // ================================================== classifying warps
        const int g = warp >> 2;
        const uint32_t d_addr = tmem + (uint32_t)(g * 128) + ((uint32_t)(warp & 3) << 21);  // lane (w % 4) * 32
        const HistCol hc = hist_col<kWorkThreads>(wd);
        uint32_t* const uq = sptr<uint32_t>(wd.off_queue) + (uint32_t)warp * kQueueCodes;
        float thr = wd.tc_thr;  // (3-D: the i-point's own threshold)
        uint32_t stage = 0, phase = 0, dphase = 0;
        uint32_t iw = 0, qn = 0, jq0 = 0;  // first i of the warp, queue length, j origin of the queue's codes
        uint32_t na = 0, nb = 0, rule = 0;
        [[maybe_unused]] uint32_t cur_gi = 4u;  // which 128 of the item's i-points (4: none of this item yet)
        int cur_sub = -1;
        unsigned long long* cur_hist = nullptr;
        uint32_t inc_bound = 0, over = 0, band = 0, mism = 0;
        u64 ax = 0, ay = 0, az = 0;
        bool aborted = false;

        auto flush = [&]() {
            tc_merge(hc, wd.ne, check, cur_hist);
            if (check) {
                const unsigned long long o = warp_sum(over);
                if (lane == 0 && o) atomicAdd(cur_hist + wd.ne, o);
                over = 0;
            }
            inc_bound = 0;
        };

        uint32_t ninfo = 0, njbase = 0, ni0 = 0;
        bool have = false;  // the stage's record has been read ahead
        while (true) {
            uint32_t info = ninfo, jbase = njbase, i0 = ni0;
            if (!have) {
                if (!tc_wait(full + stage, phase, limit, ctl, wd.stats)) {
                    aborted = true;
                    break;
                }
                rec_load(meta + stage * (uint32_t)sizeof(TcMeta), info, jbase, i0);
            }
            have = false;
            if (info & kInfoStop) {
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + stage);
                break;
            }
            // other i-points: a new item's, or (PRUNE) another 128 of the item's
            bool turn = (info & kInfoNew) != 0u;
            uint32_t gi = (uint32_t)g;
            if constexpr (PRUNE) {
                if (turn) cur_gi = 4u;
                gi = (info >> (8 + 2 * g)) & 3u;
                turn = ((info >> g) & 1u) && gi != cur_gi;
            }
            if (turn) {
                if constexpr (PRUNE) {
                    if (qn) {
                        __syncwarp();
                        tc_drain<EUCLID>(wd, sub_of(wd, cur_sub), uq, qn, ax, ay, az, iw, jq0, hc, band, mism);
                        ++inc_bound;
                        qn = 0;
                        __syncwarp();
                    }
                    cur_gi = gi;
                }
                const int sub = (int)(info >> 16);
                const SubProblem& sp = sub_of(wd, sub);
                iw = i0 + kBlk * gi + 32u * (uint32_t)(warp & 3);
                jq0 = jbase;
                unsigned long long* tgt = sp.hist;
                if (sp.row_seg) tgt += (size_t)__ldg(sp.row_seg + iw / kSegAlign) * sp.row_stride;
                if (cur_sub >= 0 && tgt != cur_hist) flush();
                cur_sub = sub;
                cur_hist = tgt;
                na = sp.na;
                nb = sp.nb;
                rule = sp.auto_mode ? 1u : (sp.no_self ? 2u : 0u);
                const float3 p = ldg_point32(sp.a_blk, iw + (uint32_t)lane);
                if constexpr (EUCLID) {
                    const float ux = p.x * sp.tc_scale, uy = p.y * sp.tc_scale, uz = p.z * sp.tc_scale;
                    thr = fmaf(fmaf(uz, uz, fmaf(uy, uy, ux * ux)), sp.tc_qmul, sp.tc_qadd);
                }
                ax = pack2(p.x, p.x);
                ay = pack2(p.y, p.y);
                az = pack2(p.z, p.z);
            }
            if ((info >> g) & 1u) {
                // ---- the group's accumulators: one maximum per 32 x 32 pairs
                if (!tc_wait(d_full + g, dphase, limit, ctl, wd.stats)) {
                    aborted = true;
                    break;
                }
                dphase ^= 1u;
                tc_fence_after();
                // (votes after each pair of loads: without them four loads are in flight and their
                // registers spill)
                float m0 = tc_row_max32(d_addr), m1 = tc_row_max32(d_addr + 32u);
                tc_wait_ld(m0, m1);
                uint32_t kept = __any_sync(0xffffffffu, m0 >= thr) ? 1u : 0u;
                kept |= __any_sync(0xffffffffu, m1 >= thr) ? 2u : 0u;
                float m2 = tc_row_max32(d_addr + 64u), m3 = tc_row_max32(d_addr + 96u);
                // The next stage's record meanwhile, if it is there.  (A rejected tile is bound by
                // this loop's chain of waits, not by a unit: with this and the step below 700,001 x
                // 1,400,003 points on the sphere to 2 degrees 55.6 -> 50.4 ms, an octant of 1,000,000 +
                // 1,000,000 to 10 degrees 216.7 -> 213.3 ms; patches where every tile is classified
                // 49.3 -> 50.4 ms.  Most pruned tiles are classified: 26.2 -> 26.6 ms with both.)
                if constexpr (!PRUNE) {
                    const uint32_t ns = stage + 1u == S ? 0u : stage + 1u;
                    if (__all_sync(0xffffffffu, mbar_test_wait(full + ns, ns ? phase : phase ^ 1u))) {
                        rec_load(meta + ns * (uint32_t)sizeof(TcMeta), ninfo, njbase, ni0);
                        have = true;
                    }
                }
                tc_wait_ld(m2, m3);
                tc_fence_before();
                if (PRUNE && lane == 0) mbar_arrive(d_free + g);
                kept |= __any_sync(0xffffffffu, m2 >= thr) ? 4u : 0u;
                kept |= __any_sync(0xffffffffu, m3 >= thr) ? 8u : 0u;
                if constexpr (!PRUNE) {
                    // a tile with nothing to classify is done: its accumulators and its stage
                    // are given back in one step
                    bool done = kept == 0u && !(info & kInfoLast);
                    if constexpr (check) {
                        // off the diagonal and the catalogs' ends every pair of it is overflow
                        done = done && jbase + kBlk <= nb && iw + 32u <= na &&
                               (rule == 0u || jbase > iw || (rule == 2u && jbase + kBlk <= iw));
                        if (done) over += kBlk;
                    }
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(d_free + g);
                        if (done) mbar_arrive(empty + stage);
                    }
                    if (done) {
                        if (++stage == S) {
                            stage = 0;
                            phase ^= 1u;
                        }
                        continue;
                    }
                }
                // most tiles hold nothing within the range: on to the next
                if (kept != 0u || check) {
                    tc_beat(wd);
                    // a lane's counter gains at most one per pair of the tile and one per queue batch
                    // (one batch more when the queue is emptied at the item's end)
                    if (inc_bound + 2u * kBlk + 2u > 0xffffu || over > 0x40000000u) flush();
                    inc_bound += 32u * (uint32_t)__popc(kept);
                    const SubProblem& sp = sub_of(wd, cur_sub);
                    // blocks at or below the diagonal (j-block and i-block of 32 coincide or do not overlap)
                    uint32_t todo = check ? 0xfu : kept;
                    if (rule == 1u && jbase < iw) todo &= ~0u << ((iw - jbase) >> 5 < 4u ? (iw - jbase) >> 5 : 4u);
                    // (a counted block's overflow needs its pair mask; otherwise a mask is needed on the
                    // diagonal and, where padding could look in range, at the catalogs' ends)
                    const bool ends = (wd.need_idx || check) && (jbase + kBlk > nb || iw + 32u > na);
                    const float* sx = sptr<const float>(wd.off_stage + stage * kStageBytes + kBlkX);
                    while (todo) {
                        const uint32_t b = (uint32_t)__ffs((int)todo) - 1u;
                        todo &= todo - 1u;
                        const uint32_t jb = jbase + 32u * b;
                        const bool diag = rule != 0u && jb == iw;
                        uint32_t valid = ~0u;
                        if (diag || ends) {
                            const uint32_t left = nb > jb ? nb - jb : 0u;
                            if (left < 32u) valid = (1u << left) - 1u;
                            if (iw + (uint32_t)lane >= na) valid = 0u;
                            if (diag) valid &= rule == 1u ? (0xfffffffeu << lane) : ~(1u << lane);
                        }
                        if constexpr (check) {
                            if (!((kept >> b) & 1u)) {
                                over += (uint32_t)__popc(valid);
                                continue;
                            }
                        }
                        uint32_t um = (diag || ends) ? tc_block<EUCLID, true>(wd, ax, ay, az, sx + 32 * b, valid, hc)
                                                     : tc_block<EUCLID, false>(wd, ax, ay, az, sx + 32 * b, valid, hc);
                        // ---- queue the unsettled pairs; a full batch of 32 is classified at once
                        uint32_t act = __ballot_sync(0xffffffffu, um != 0u);
                        while (act) {
                            if (um) {
                                const int k = __clz((int)um);
                                um &= ~(0x80000000u >> k);
                                uq[qn + (uint32_t)__popc(act & ((1u << lane) - 1u))] =
                                    (uint32_t)lane | ((jb + (uint32_t)k - jq0) << 5);
                            }
                            qn += (uint32_t)__popc(act);
                            if (qn >= 32u) {
                                __syncwarp();
                                qn -= 32u;
                                tc_drain<EUCLID>(wd, sp, uq + qn, 32u, ax, ay, az, iw, jq0, hc, band, mism);
                                ++inc_bound;
                                __syncwarp();  // the batch is read before later codes overwrite it
                            }
                            act = __ballot_sync(0xffffffffu, um != 0u);
                        }
                    }
                }
            }
            if (info & kInfoLast) {
                if (lane == 0) mbar_arrive(a_empty + ((info & kInfoABuf) ? 1 : 0));
                if (qn) {
                    __syncwarp();
                    tc_drain<EUCLID>(wd, sub_of(wd, cur_sub), uq, qn, ax, ay, az, iw, jq0, hc, band, mism);
                    ++inc_bound;
                    qn = 0;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + stage);
            if (++stage == S) {
                stage = 0;
                phase ^= 1u;
            }
        }
        if (!aborted && cur_sub >= 0) flush();
        const unsigned long long b = warp_sum(band), mm = warp_sum(mism);
        if (lane == 0) {
            if (b) atomicAdd(wd.stats + kStatBand, b);
            if (mm) atomicAdd(wd.stats + kStatMismatch, mm);
        }
    } else if (warp < kLoadWarp) {
        // ================================================== mma issuers
        const int g = warp - kIssueWarp;
        uint32_t stage = 0, phase = 0, dphase = 0, acnt = 0;
        bool any = false;
        while (true) {
            if (!tc_wait(full + stage, phase, limit, ctl, wd.stats)) break;
            uint32_t info, jbase, i0;
            rec_load(meta + stage * (uint32_t)sizeof(TcMeta), info, jbase, i0);
            if (info & kInfoStop) {
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + stage);
                break;
            }
            const uint32_t buf = (info & kInfoABuf) ? 1u : 0u;
            if (info & kInfoNew) {
                if (!tc_wait(a_full + buf, (acnt >> 1) & 1u, limit, ctl, wd.stats)) break;
                ++acnt;
            }
            if ((info >> g) & 1u) {
                if (!tc_wait(d_free + g, dphase ^ 1u, limit, ctl, wd.stats)) break;
                dphase ^= 1u;
                tc_fence_after();
                if (lane == 0) {
                    tc_mma(tmem + (uint32_t)(g * 128),
                           op_desc(smem_addr(dyn_smem) + wd.off_atile + buf * kABytes +
                                   (PRUNE ? (info >> (8 + 2 * g)) & 3u : (uint32_t)g) * kABlock, kBlkX),
                           op_desc(smem_addr(dyn_smem) + wd.off_stage + stage * kStageBytes, kStageX2));
                    tc_commit(d_full + g);
                }
                any = true;
            }
            __syncwarp();
            if (lane == 0) {
                // (an issuer whose group has no tile in the item gives the operand back too: it has
                // waited for it, by parity, and must not see the buffer filled twice meanwhile)
                if (info & kInfoLast) mbar_arrive(a_empty + buf);
                mbar_arrive(empty + stage);
            }
            if (++stage == S) {
                stage = 0;
                phase ^= 1u;
            }
        }
        // after an abort: the last product finishes before the tensor memory is given back
        if (ctl[kTcAbort] && any) (void)mbar_wait_bounded(d_full + g, dphase ^ 1u, limit);
    } else {
        // ================================================== loader: items, tiles, copies
        const bool hook = (wd.flags & TPCF_F_TEST_WAIT_TIMEOUT) != 0;
        uint32_t stage = 0, phase = 0, acnt = 0, issued = 0, turn = 0;
        unsigned long long pruned = 0;
        bool ok = true;
        const uint64_t n = wd.item_hi - wd.item_lo;
        unsigned long long* const counter = wd.stats + kStatNextItem;
        // Items are drawn wd.draw_batch at a time, one per lane: a lane finds its
        // item's tiles and groups with countable pairs (bit t of gm[g]: tile t of the
        // chunk for group g), so that a launch that prunes nearly everything spends a
        // few instructions, not a draw, on an empty item.  A draw with its geometry
        // takes about 6500 cycles for one item or for 32 (full sphere, 1.5M + 3M,
        // 2 degrees: 145 ms with one item per draw, 40 ms with 32, 37 ms with the
        // chunk spheres, 26 ms with tiles given to the groups of warps in turn).
        const uint32_t batch = wd.draw_batch;
        // (lane 0's result counts; it is asked for a batch ahead, while the current one is issued)
        auto draw = [&]() {
            unsigned long long p = ~0ull;
            if (lane == 0) {
                if constexpr (PREEMPT) {
                    if (*reinterpret_cast<volatile unsigned long long*>(wd.stats + kStatYield) == 0ull)
                        p = wd.pos_lo + atomicAdd(counter, (unsigned long long)batch);
                } else {
                    p = atomicAdd(counter, (unsigned long long)batch);
                }
            }
            return p;
        };
        unsigned long long next = draw();
        while (ok) {
            const unsigned long long p = __shfl_sync(0xffffffffu, next, 0);
            if (p >= n || ctl[kTcAbort]) break;
            next = draw();
            if (lane == 0) ctl[kTcBeat] = ctl[kTcBeat] + 1;
            Cursor c;
            c.sub = 0;
            c.g = ItemGeom{0u, 0u, 0u, 0u};
            uint32_t gm[kGroups] = {0u, 0u, 0u, 0u};
            unsigned long long pairs = 0;
            if ((uint32_t)lane < batch && p + (uint32_t)lane < n &&
                load_item<!PRUNE>(wd, (uint32_t)(wd.item_lo + p + (uint32_t)lane), c)) {
                const SubProblem& sp = sub_of(wd, c.sub);
                pairs = span_pairs(c.g.i0, wd.I, (uint64_t)c.g.j0 + (uint64_t)c.t * wd.J,
                                   (uint64_t)c.g.j0 + (uint64_t)c.g.t_end * wd.J, sp.na, sp.nb, sp.auto_mode != 0);
#pragma unroll
                for (int gg = 0; gg < kGroups; ++gg) {
                    const uint32_t ib = c.g.i0 + kBlk * (uint32_t)gg;
                    uint32_t t0 = c.g.t_first;  // (auto counts: tiles from the group's own on)
                    if (sp.auto_mode && ib > c.g.j0) t0 = max(t0, (ib - c.g.j0) / kBlk);
                    if (ib < sp.na && t0 < c.g.t_end) gm[gg] = (0xffffffffu >> (32u - (c.g.t_end - t0))) << t0;
                }
                if (PRUNE && sp.b_caps2) {
                    // the item's i-points against the whole chunk
                    float4 ic[kGroups];
#pragma unroll
                    for (int gg = 0; gg < kGroups; ++gg)
                        ic[gg] = gm[gg] ? __ldg(sp.a_caps + c.g.i0 / kCapPoints + gg) : make_float4(0.f, 0.f, 0.f, -1e30f);
                    if (prune_block(wd, union_sphere(ic), __ldg(sp.b_caps2 + c.g.j0 / kPad))) {
#pragma unroll
                        for (int gg = 0; gg < kGroups; ++gg) {
                            pruned += (unsigned long long)__popc(gm[gg]) * (kBlk * kBlk);
                            gm[gg] = 0u;
                        }
                    }
                }
            }
            pairs = warp_sum(pairs);
            if (lane == 0) atomicAdd(wd.stats + kStatPairs, pairs);
            uint32_t items = __ballot_sync(0xffffffffu, (gm[0] | gm[1] | gm[2] | gm[3]) != 0u);
            while (ok && items) {
                const int l = __ffs((int)items) - 1;
                items &= items - 1u;
                const int sub = __shfl_sync(0xffffffffu, c.sub, l);
                const uint32_t i0 = __shfl_sync(0xffffffffu, c.g.i0, l), j0 = __shfl_sync(0xffffffffu, c.g.j0, l);
                uint32_t g0 = __shfl_sync(0xffffffffu, gm[0], l), g1 = __shfl_sync(0xffffffffu, gm[1], l),
                         g2 = __shfl_sync(0xffffffffu, gm[2], l), g3 = __shfl_sync(0xffffffffu, gm[3], l);
                const SubProblem& sp = sub_of(wd, sub);
                if constexpr (PRUNE) {
                    // every tile against every group, a tile per lane
                    const uint32_t has = ((g0 >> lane) & 1u) | (((g1 >> lane) & 1u) << 1) | (((g2 >> lane) & 1u) << 2) |
                                         (((g3 >> lane) & 1u) << 3);
                    uint32_t keep = 0;
                    if (has) {
                        const float4 jt = __ldg(sp.b_caps + j0 / kCapPoints + (uint32_t)lane);
#pragma unroll
                        for (int gg = 0; gg < kGroups; ++gg)
                            if (((has >> gg) & 1u) && !prune_block(wd, __ldg(sp.a_caps + i0 / kCapPoints + gg), jt))
                                keep |= 1u << gg;
                    }
                    pruned += (unsigned long long)__popc(has ^ keep) * (kBlk * kBlk);
                    g0 = __ballot_sync(0xffffffffu, keep & 1u);
                    g1 = __ballot_sync(0xffffffffu, keep & 2u);
                    g2 = __ballot_sync(0xffffffffu, keep & 4u);
                    g3 = __ballot_sync(0xffffffffu, keep & 8u);
                    if ((g0 | g1 | g2 | g3) == 0u) continue;
                }
                // ---- the item's i-side operand
                const uint32_t buf = acnt & 1u;
                if (!tc_wait(a_empty + buf, ((acnt >> 1) & 1u) ^ 1u, limit, ctl, wd.stats)) {
                    ok = false;
                    break;
                }
                {
                    const unsigned char* src = sp.a_blk + (size_t)(i0 / kBlk) * kBlkBytes;
                    uint4* const dst = sptr<uint4>(wd.off_atile + buf * kABytes);
#pragma unroll 1
                    for (int gg = 0; gg < kGroups; gg += 2) {  // (eight loads in flight)
                        uint4 x[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            x[k] = __ldg(reinterpret_cast<const uint4*>(src + (size_t)(gg + k / 4) * kBlkBytes) +
                                         32 * (k % 4) + lane);
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            uint4* const p = dst + (gg + k / 4) * (kABlock / 16) + 32 * (k % 4) + lane;
                            p[0] = plane_x<EUCLID>(x[k]);
                            p[kBlk] = plane_y<EUCLID>(x[k], sp.tc_pad);
                        }
                    }
                    fence_proxy_async_smem();  // the products read it through the asynchronous proxy
                    __syncwarp();
                    if (lane == 0) mbar_arrive(a_full + buf);
                }
                ++acnt;
                // ---- its tiles
                uint32_t first = kInfoNew, tiles = g0 | g1 | g2 | g3;
                while (tiles) {
                    const uint32_t t = (uint32_t)__ffs((int)tiles) - 1u;
                    tiles &= tiles - 1u;
                    if (!tc_wait(empty + stage, phase ^ 1u, limit, ctl, wd.stats)) {
                        ok = false;
                        break;
                    }
                    // the tile's i-groups; PRUNE: given to the groups of warps in turn, so that all work
                    const uint32_t gs = ((g0 >> t) & 1u) | (((g1 >> t) & 1u) << 1) | (((g2 >> t) & 1u) << 2) |
                                        (((g3 >> t) & 1u) << 3);
                    uint32_t who = gs;
                    if constexpr (PRUNE) {
                        who = 0u;
                        for (uint32_t m = gs; m; m &= m - 1u) {
                            who |= (1u << turn) | (((uint32_t)__ffs((int)m) - 1u) << (8u + 2u * turn));
                            turn = (turn + 1u) & 3u;
                        }
                    }
                    if (lane == 0) {
                        const uint32_t jt = j0 + t * kBlk;
                        rec_store(meta + stage * (uint32_t)sizeof(TcMeta),
                                  who | (buf ? kInfoABuf : 0u) | first | (tiles ? 0u : kInfoLast) | ((uint32_t)sub << 16),
                                  jt, i0);
                        fence_proxy_async_smem();  // the group's reads of the stage's previous tile come first
                        if (!(hook && issued == 0)) {  // (test hook: the first copy is never issued)
                            const unsigned char* src = sp.b_blk + (size_t)(jt / kBlk) * kBlkBytes;
                            unsigned char* const dst = sptr<unsigned char>(wd.off_stage + stage * kStageBytes);
                            mbar_expect_tx(full + stage, kStageBytes);
                            bulk_copy_g2s(dst, src, kBlkBytes, full + stage);
                            bulk_copy_g2s(dst + kStageX2, src, kBlkX, full + stage);
                        }
                    }
                    first = 0;
                    ++issued;
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
        if (ok && !ctl[kTcAbort] && tc_wait(empty + stage, phase ^ 1u, limit, ctl, wd.stats) && lane == 0) {
            rec_store(meta + stage * (uint32_t)sizeof(TcMeta), kInfoStop, 0u, 0u);
            mbar_arrive(full + stage);
        }
        __syncwarp();
        if constexpr (PRUNE) {
            pruned = warp_sum(pruned);
            if (lane == 0 && pruned) atomicAdd(wd.stats + kStatPruned, pruned);
        }
        // after an abort: copies still in flight land before the block leaves (bounded)
        if (ctl[kTcAbort]) {
            const uint32_t back = issued < S ? issued : S;
            for (uint32_t k = issued - back; k < issued; ++k)
                if (!(hook && k == 0)) (void)mbar_wait_bounded(full + k % S, (k / S) & 1u, limit);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kIssueWarp) tc_dealloc(tmem);
}

// ============================================================== the screen's values
// A self-check: the accumulators of one product of 128 i-points and 128 j-points (values: 128
// rows of 128) and the maxima of 32 that the kernel above compares (maxima: 128 rows of 4), by its
// instructions.  One block of four warps.
template <bool EUCLID>
__global__ void __launch_bounds__(128, 1) screen_values_kernel(const unsigned char* a, const unsigned char* b,
                                                               uint32_t pad, uint64_t limit_ns, float* values,
                                                               float* maxima, unsigned long long* err) {
    __shared__ __align__(128) unsigned char op[kABlock + 2 * kBlkX];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_word;
    const uint32_t t = threadIdx.x, warp = t >> 5;
    {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(a) + t), y = __ldg(reinterpret_cast<const uint4*>(b) + t);
        uint4* const p = reinterpret_cast<uint4*>(op) + t;
        p[0] = plane_x<EUCLID>(x);
        p[kBlk] = plane_y<EUCLID>(x, pad);
        p[2 * kBlk] = y;
        p[3 * kBlk] = y;
        fence_proxy_async_smem();
    }
    if (t == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == 0) tc_alloc(smem_addr(&tmem_word));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_word);
    if (t == 0) {
        tc_mma(tmem, op_desc(smem_addr(op), kBlkX), op_desc(smem_addr(op) + kABlock, kBlkX));
        tc_commit(&bar);
    }
    const bool ok = __all_sync(0xffffffffu, mbar_wait_bounded(&bar, 0u, limit_ns));
    if (ok) {
        tc_fence_after();
        for (uint32_t q = 0; q < 4; ++q) {
            uint32_t r[32];
            float m = tc_row_max32(tmem + (warp << 21) + 32u * q, r);
            tc_wait_ld(m, r);
            maxima[4u * t + q] = m;
#pragma unroll
            for (int k = 0; k < 32; ++k) values[128u * t + 32u * q + (uint32_t)k] = __uint_as_float(r[k]);
        }
        tc_fence_before();
    } else if ((t & 31u) == 0u) {
        atomicOr(err, (unsigned long long)kErrWaitTimeout);
    }
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tc_dealloc(tmem);
}

template <bool PREEMPT, bool PRUNE, bool EUCLID, bool CHECK = false>
cudaError_t launch_tc_t(const WorkDesc& wd_in, const Shape& sh, cudaStream_t stream) {
    WorkDesc wd = wd_in;
    const TcLayout L = tc_layout((int)wd.stages, wd.nedges_max);
    wd.off_ctl = L.ctl;
    wd.off_bars = L.bars;
    wd.off_meta = L.meta;
    wd.off_atile = L.atile;
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
    wd.stage_bytes = kStageBytes;
    if (L.total > sh.smem || wd.I != 128u * kGroups || wd.J != kBlk || wd.Jc > 32u * kBlk)
        return cudaErrorInvalidValue;
    count_tc_kernel<PREEMPT, PRUNE, EUCLID, CHECK><<<sh.blocks, kThreads, sh.smem, stream>>>(wd);
    return cudaGetLastError();
}

}  // namespace

size_t count_tc_smem_bytes(int stages, int nedges) { return tc_layout(stages, nedges).total; }

cudaError_t count_tc_set_smem_limit() {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // (the opt-in maximum: the attribute belongs to the kernel, not to a launch)
    const void* kernels[9] = {
        (const void*)count_tc_kernel<false, false, false, false>, (const void*)count_tc_kernel<true, false, false, false>,
        (const void*)count_tc_kernel<false, true, false, false>,  (const void*)count_tc_kernel<true, true, false, false>,
        (const void*)count_tc_kernel<false, false, true, false>,  (const void*)count_tc_kernel<false, true, true, false>,
        (const void*)count_tc_kernel<false, false, false, true>,  (const void*)count_tc_kernel<true, false, false, true>,
        (const void*)count_tc_kernel<false, false, true, true>};
    for (const void* k : kernels)
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    return e;
}

cudaError_t launch_screen_values(const unsigned char* a_blk, const unsigned char* b_blk, bool euclid, uint32_t pad,
                                 uint64_t limit_ns, float* values, float* maxima, unsigned long long* err,
                                 cudaStream_t stream) {
    if (euclid) screen_values_kernel<true><<<1, 128, 0, stream>>>(a_blk, b_blk, pad, limit_ns, values, maxima, err);
    else screen_values_kernel<false><<<1, 128, 0, stream>>>(a_blk, b_blk, pad, limit_ns, values, maxima, err);
    return cudaGetLastError();
}

cudaError_t launch_count_tc(const WorkDesc& wd, const Shape& sh, bool preempt, cudaStream_t stream) {
    const bool check = (wd.flags & TPCF_F_CHECK_OVERFLOW) != 0;
    if (check && wd.prune) return cudaErrorInvalidValue;
    if (wd.euclid) {  // (the job server, whose steps preempt, counts angles)
        if (preempt) return cudaErrorInvalidValue;
        if (check) return launch_tc_t<false, false, true, true>(wd, sh, stream);
        return wd.prune ? launch_tc_t<false, true, true>(wd, sh, stream) : launch_tc_t<false, false, true>(wd, sh, stream);
    }
    if (check)
        return preempt ? launch_tc_t<true, false, false, true>(wd, sh, stream)
                       : launch_tc_t<false, false, false, true>(wd, sh, stream);
    if (wd.prune)
        return preempt ? launch_tc_t<true, true, false>(wd, sh, stream) : launch_tc_t<false, true, false>(wd, sh, stream);
    return preempt ? launch_tc_t<true, false, false>(wd, sh, stream) : launch_tc_t<false, false, false>(wd, sh, stream);
}

}  // namespace tpcf
