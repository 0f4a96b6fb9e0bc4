// CUDA kernels (sm_103a) of catalog preparation: validation of the input
// points, a space-filling-curve sort, and the device copies the counting
// kernels read (binary64 points; blocks of 128 points that hold their
// tensor-core operand records and FP32 x | y | z arrays; bounding spheres per
// 128 and per 4096 points).
//
// Paper: Ponce et al., "Application of GPUs for the calculation of two point
// correlation functions in cosmology", Section 3 (the pair angle follows from
// the dot product of unit vectors; this file prepares those vectors once per
// catalog so that the O(N^2) counting kernel reads compact, sorted copies).
#include <cuda_fp16.h>
#include <stdint.h>

#include "tpcf.h"
#include "tpcf_internal.h"

namespace tpcf {
// ============================================================== catalog preparation
// Spatial key: cube face and a 14+14-bit Morton code of the face coordinates.
__device__ __forceinline__ uint32_t spread14(uint32_t v) {
    v &= 0x3fffu;
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

__device__ __forceinline__ uint32_t cell_key(double x, double y, double z) {
    const double ax = fabs(x), ay = fabs(y), az = fabs(z);
    uint32_t face;
    double u, v;
    if (ax >= ay && ax >= az) { face = x > 0 ? 0u : 1u; u = y / ax; v = z / ax; }
    else if (ay >= az)        { face = y > 0 ? 2u : 3u; u = x / ay; v = z / ay; }
    else                      { face = z > 0 ? 4u : 5u; u = x / az; v = y / az; }
    const double sc = 8192.0;  // (u + 1) * 2^13 in [0, 2^14]
    int qu = (int)((u + 1.0) * sc), qv = (int)((v + 1.0) * sc);
    qu = qu < 0 ? 0 : (qu > 16383 ? 16383 : qu);
    qv = qv < 0 ? 0 : (qv > 16383 ? 16383 : qv);
    return (face << 28) | (spread14((uint32_t)qu) << 1) | spread14((uint32_t)qv);
}

// Order-preserving map of a double to an unsigned 64-bit key (and back).
__device__ __forceinline__ unsigned long long dkey_of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dval_of(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

// Bounding box of a 3-D catalog: bbox[0..2] = min keys, bbox[3..5] = max keys
// (initialised to ~0 and 0 by the caller).
__global__ void prep_bbox_kernel(const double* __restrict__ xyz, uint32_t n, unsigned long long* bbox) {
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double v = xyz[3ull * i + c];
            if (!isfinite(v)) continue;
            const unsigned long long k = dkey_of(v);
            lo[c] = k < lo[c] ? k : lo[c];
            hi[c] = k > hi[c] ? k : hi[c];
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        atomicMin(bbox + c, lo[c]);
        atomicMax(bbox + 3 + c, hi[c]);
    }
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {  // 10 bits -> every third bit
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// 3-D Morton key (10 bits per axis) of a point inside the bounding box.
__device__ __forceinline__ uint32_t box_key(double x, double y, double z, const unsigned long long* bbox) {
    const double p[3] = {x, y, z};
    uint32_t q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double lo = dval_of(bbox[c]), hi = dval_of(bbox[3 + c]);
        const double t = hi > lo ? (p[c] - lo) / (hi - lo) * 1024.0 : 0.0;
        int v = (int)t;
        q[c] = (uint32_t)(v < 0 ? 0 : (v > 1023 ? 1023 : v));
    }
    return (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
}

// Sort keys and validation.  Unit-vector catalogs: every point finite with
// | |v| - 1 | <= 1e-6, eps_word receives the largest | |v|^2 - 1 |; 3-D
// catalogs (euclid): every point finite, eps_word receives the largest
// |v|^2 (both as the bits of a non-negative double, whose order is that of
// the integers).  Keys: cube-face curve of the direction (unit vectors) or a
// 3-D Morton curve over the bounding box (3-D).
__global__ void prep_keys_kernel(const double* __restrict__ xyz, uint32_t n,
                                 const uint32_t* __restrict__ seg_of_point, int sort, int euclid,
                                 const unsigned long long* __restrict__ bbox,
                                 unsigned long long* keys, uint32_t* vals, uint32_t n_pow2,
                                 unsigned long long* err_word, unsigned long long* eps_word) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pow2) return;  // n_pow2 is a multiple of the block size: whole warps leave
    double eps = 0.0;
    if (i >= n) {
        keys[i] = ~0ull;
        vals[i] = 0xffffffffu;
    } else {
        const double x = xyz[3ull * i], y = xyz[3ull * i + 1], z = xyz[3ull * i + 2];
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
        const bool finite = isfinite(x) && isfinite(y) && isfinite(z) && isfinite(r2);
        if (euclid) {
            // |coordinates| <= 1e28 keeps FP32 copies and differences finite
            if (!finite || !(fabs(x) <= 1e28 && fabs(y) <= 1e28 && fabs(z) <= 1e28))
                atomicOr(err_word, (unsigned long long)kErrBadPoint);
            else eps = r2;
        } else if (!finite || !(r2 >= 0.999998000001 && r2 <= 1.000002000001)) {
            // | |v| - 1 | <= 1e-6  <=>  r2 in [(1 - 1e-6)^2, (1 + 1e-6)^2]
            atomicOr(err_word, (unsigned long long)kErrBadPoint);
        } else {
            eps = fabs(r2 - 1.0);
        }
        const unsigned long long seg = seg_of_point ? seg_of_point[i] : 0u;
        const uint32_t ck = (sort && finite) ? (euclid ? box_key(x, y, z, bbox) : cell_key(x, y, z)) : 0u;
        keys[i] = (seg << 32) | ck;
        vals[i] = i;
    }
    unsigned long long eb = (unsigned long long)__double_as_longlong(eps);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, eb, o);
        eb = v > eb ? v : eb;
    }
    if ((threadIdx.x & 31) == 0 && eb != 0) atomicMax(eps_word, eb);
}

__device__ __forceinline__ bool kv_greater(unsigned long long ka, uint32_t va, unsigned long long kb,
                                           uint32_t vb) {
    return ka > kb || (ka == kb && va > vb);
}

// L global compare-exchange levels of the bitonic network in one pass over the
// data (block size k, strides j, j / 2, .. j >> (L - 1)): a thread holds the 2^L
// elements that these levels exchange with one another.  A pass costs a launch
// (about 3 us) more than it costs traffic at these sizes, so up to three levels
// share one (catalog of 100,003 points on the GPU: 323 us with a pass per level,
// 270 us; 200,006: 395 and 325 us; 3,000,000: 2.28 and 2.02 ms).
template <int L>
__global__ void bitonic_global_kernel(unsigned long long* keys, uint32_t* vals, uint32_t n_pow2, uint32_t k,
                                      uint32_t j) {
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_pow2 >> L) return;
    const uint32_t s = j >> (L - 1);  // smallest stride
    const uint32_t i0 = ((t & ~(s - 1u)) << L) | (t & (s - 1u));
    const bool up = (i0 & k) == 0;  // (2^L s = 2 j <= k: one block of k)
    unsigned long long kk[1 << L];
    uint32_t vv[1 << L];
#pragma unroll
    for (int m = 0; m < 1 << L; ++m) {
        kk[m] = keys[i0 + m * s];
        vv[m] = vals[i0 + m * s];
    }
#pragma unroll
    for (int d = 1 << (L - 1); d > 0; d >>= 1) {
#pragma unroll
        for (int m = 0; m < 1 << L; ++m) {
            if ((m & d) == 0 && kv_greater(kk[m], vv[m], kk[m + d], vv[m + d]) == up) {
                const unsigned long long tk = kk[m];
                kk[m] = kk[m + d];
                kk[m + d] = tk;
                const uint32_t tv = vv[m];
                vv[m] = vv[m + d];
                vv[m + d] = tv;
            }
        }
    }
#pragma unroll
    for (int m = 0; m < 1 << L; ++m) {
        keys[i0 + m * s] = kk[m];
        vals[i0 + m * s] = vv[m];
    }
}

// Shared-memory bitonic steps on 2048-element chunks: either the full sort of
// each chunk (k = 2 .. 2048) or, for a given k > 2048, the strides 1024 .. 1.
__global__ void __launch_bounds__(1024) bitonic_local_kernel(unsigned long long* keys, uint32_t* vals,
                                                             uint32_t n_pow2, uint32_t k_fixed) {
    __shared__ unsigned long long sk[2048];
    __shared__ uint32_t sv[2048];
    const uint32_t base = blockIdx.x * 2048u;
    const uint32_t t = threadIdx.x;
    sk[t] = keys[base + t];
    sk[t + 1024] = keys[base + t + 1024];
    sv[t] = vals[base + t];
    sv[t + 1024] = vals[base + t + 1024];
    __syncthreads();
    const uint32_t k_lo = k_fixed ? k_fixed : 2u;
    const uint32_t k_hi = k_fixed ? k_fixed : (n_pow2 < 2048u ? n_pow2 : 2048u);
    for (uint32_t k = k_lo; k <= k_hi; k <<= 1) {
        for (uint32_t j = (k_fixed ? 1024u : k / 2); j > 0; j >>= 1) {
            const uint32_t i = 2 * t - (t & (j - 1));
            const uint32_t l = i + j;
            const bool up = ((base + i) & k) == 0;
            const unsigned long long ki = sk[i], kl = sk[l];
            const uint32_t vi = sv[i], vl = sv[l];
            if (kv_greater(ki, vi, kl, vl) == up) {
                sk[i] = kl; sk[l] = ki;
                sv[i] = vl; sv[l] = vi;
            }
            // (strides up to 32 stay within a warp's 64 elements)
            if (j > 32u || (j == 1u && k > 32u)) __syncthreads(); else __syncwarp();
        }
    }
    __syncthreads();
    keys[base + t] = sk[t];
    keys[base + t + 1024] = sk[t + 1024];
    vals[base + t] = sv[t];
    vals[base + t + 1024] = sv[t + 1024];
}

// The binary16 split of an FP32 coordinate: v = hi + lo + r, |r| <= 2^-22 |v| + 2^-25.
__device__ __forceinline__ uint32_t split16(float v) {  // hi | lo << 16
    const __half h = __float2half_rn(v), l = __float2half_rn(v - __half2float(h));
    return (uint32_t)__half_as_ushort(h) | ((uint32_t)__half_as_ushort(l) << 16);
}

// Writes point q's FP32 coordinates and operand record into its block (3-D: the
// record of the point times `scale`).
__device__ __forceinline__ void put_block(unsigned char* blk, uint32_t q, float x, float y, float z, int euclid,
                                          float scale) {
    unsigned char* b = blk + (size_t)(q / kBlk) * kBlkBytes;
    const uint32_t o = q % kBlk;
    uint32_t norm = 0u;
    float ux = x, uy = y, uz = z;
    if (euclid) {
        if (isfinite(x)) {
            ux *= scale;
            uy *= scale;
            uz *= scale;
            norm = split16(-0.5f * fmaf(uz, uz, fmaf(uy, uy, ux * ux)));
        } else {  // padding: below every threshold (the screen need not reject it: its pairs are overflow)
            ux = uy = uz = 0.f;
            norm = 0xfbffu;  // -65504
        }
    }
    const uint32_t sx = split16(ux), sy = split16(uy), sz = split16(uz);
    reinterpret_cast<uint4*>(b)[o] =
        make_uint4(__byte_perm(sx, sy, 0x5410), __byte_perm(sz, sx, 0x7610), __byte_perm(sy, sz, 0x7632), norm);
    float* f = reinterpret_cast<float*>(b + kBlkX);
    f[o] = x;
    f[kBlk + o] = y;
    f[2 * kBlk + o] = z;
}

// Gather points in sorted order into the binary64 and FP32 device copies (the
// outputs are zeroed beforehand: padding and segment gaps hold zero vectors).
// Sorted point p of segment s goes to position p + seg_delta[s] (segments of a
// segmented catalog start on aligned positions; seg_delta = NULL: no shift).
__global__ void prep_gather_kernel(const double* __restrict__ xyz, uint32_t n,
                                   const uint32_t* __restrict__ order, const uint32_t* __restrict__ seg_of_point,
                                   const uint32_t* __restrict__ seg_delta, Point64* out64,
                                   unsigned char* blk, int euclid, const unsigned long long* __restrict__ norm2) {
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t s = order ? order[p] : p;
    const uint32_t q = seg_delta ? p + seg_delta[seg_of_point[s]] : p;
    const double x = xyz[3ull * s], y = xyz[3ull * s + 1], z = xyz[3ull * s + 2];
    const float fx = __double2float_rn(x), fy = __double2float_rn(y), fz = __double2float_rn(z);
    out64[q] = Point64{x, y, z, 0.0};
    put_block(blk, q, fx, fy, fz, euclid, euclid ? ldexpf(1.f, -tc_exponent(*norm2)) : 1.f);
}

// Padding of 3-D catalogs: (+inf, +inf, +inf).  A pair with a real point has
// screen value -inf (fails the fast test) and z = +inf; two padding points
// give NaN: both land in the overflow cell of the LUT, and where the screen
// cannot settle them (coordinates so large that the FP32 bounds overflow) the
// binary64 recheck maps the NaN distance to overflow, so padding is never
// counted (unit-vector catalogs are padded with zero vectors instead).
__global__ void prep_fill_kernel(Point64* out64, unsigned char* blk, uint32_t n_pad, double v) {
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pad) return;
    const float f = (float)v;
    out64[p] = Point64{v, v, v, 0.0};
    put_block(blk, p, f, f, f, 1, 1.f);
}

// Bounding sphere of each kCapPoints-point group of a prepared catalog (one
// warp per group), for spatial pruning: centre c = the FP32-rounded mean of
// the group's real points (padding left out: zero vectors of unit-vector
// catalogs, non-finite points of 3-D catalogs), radius = max |p - c| over
// them in binary64 from the binary64 points, enlarged by 2^-20 relative and
// rounded up to FP32; all multiplied by the exact power of two `scale`.  A
// group without real points gets radius -1e30: every block with it prunes
// (it holds nothing to count).
__global__ void prep_caps_kernel(const Point64* __restrict__ p64, uint32_t n_groups, int euclid, double scale,
                                 float4* caps) {
    const uint32_t grp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t lane = threadIdx.x & 31u;
    if (grp >= n_groups) return;  // warp-uniform
    constexpr int K = (int)kCapPoints / 32;
    Point64 q[K];
    bool real[K];
    double sx = 0.0, sy = 0.0, sz = 0.0;
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        q[k] = p64[(size_t)grp * kCapPoints + (uint32_t)k * 32u + lane];
        real[k] = euclid ? (isfinite(q[k].x) && isfinite(q[k].y) && isfinite(q[k].z))
                         : (q[k].x != 0.0 || q[k].y != 0.0 || q[k].z != 0.0);
        if (real[k]) {
            sx += q[k].x * scale;
            sy += q[k].y * scale;
            sz += q[k].z * scale;
            ++cnt;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, o);
        sy += __shfl_xor_sync(0xffffffffu, sy, o);
        sz += __shfl_xor_sync(0xffffffffu, sz, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (cnt == 0) {
        if (lane == 0) caps[grp] = make_float4(0.f, 0.f, 0.f, -1e30f);
        return;
    }
    const float cx = __double2float_rn(sx / cnt), cy = __double2float_rn(sy / cnt), cz = __double2float_rn(sz / cnt);
    double r = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (real[k]) {
            const double dx = q[k].x * scale - (double)cx, dy = q[k].y * scale - (double)cy,
                         dz = q[k].z * scale - (double)cz;
            r = fmax(r, sqrt(dx * dx + dy * dy + dz * dz));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = fmax(r, __shfl_xor_sync(0xffffffffu, r, o));
    if (lane == 0) caps[grp] = make_float4(cx, cy, cz, __double2float_ru(r * (1.0 + 0x1p-20)));
}

// Bounding sphere of each kPad-point block from its groups' spheres (one warp
// per block, a group per lane): centre the FP32 mean of the non-empty groups'
// centres, radius the largest |c - c_g| + r_g, enlarged by 2^-20; an empty
// block gets radius -1e30 like an empty group.
__global__ void prep_caps2_kernel(const float4* __restrict__ caps, uint32_t n_blocks, float4* caps2) {
    static_assert(kPad == 32 * kCapPoints, "one group per lane");
    const uint32_t blk = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (blk >= n_blocks) return;  // warp-uniform
    const float4 g = caps[(size_t)blk * 32u + (threadIdx.x & 31u)];
    const bool real = g.w > -1e29f;
    float x = real ? g.x : 0.f, y = real ? g.y : 0.f, z = real ? g.z : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    const int n = __popc(__ballot_sync(0xffffffffu, real));
    const float inv = 1.0f / (float)max(n, 1);
    const float cx = x * inv, cy = y * inv, cz = z * inv;
    const float dx = cx - g.x, dy = cy - g.y, dz = cz - g.z;
    float r = real ? sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx))) + g.w : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((threadIdx.x & 31u) == 0)
        caps2[blk] = n ? make_float4(cx, cy, cz, r * (1.0f + 9.5367431640625e-07f)) : make_float4(0.f, 0.f, 0.f, -1e30f);
}

cudaError_t launch_prepare(const double* xyz_in, uint32_t n, const uint32_t* seg_of_point,
                           const uint32_t* seg_delta, int sort, int euclid, unsigned long long* bbox,
                           Point64* out64, unsigned char* blk, float4* caps, float4* caps2, uint32_t n_pad,
                           unsigned long long* keys, uint32_t* vals, uint32_t n_pow2,
                           unsigned long long* err_word, unsigned long long* eps_word, cudaStream_t stream,
                           uint32_t* launches) {
    cudaError_t e;
    uint32_t nl = 0;
    if (n > 0) {
        if (euclid && sort) {
            prep_bbox_kernel<<<152, 256, 0, stream>>>(xyz_in, n, bbox);
            ++nl;
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        prep_keys_kernel<<<(n_pow2 + 255) / 256, 256, 0, stream>>>(xyz_in, n, seg_of_point, sort, euclid, bbox,
                                                                    keys, vals, n_pow2, err_word, eps_word);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const bool do_sort = sort && n > 1;
    if (do_sort) {
        // n_pow2 >= 2048 (the host rounds it up)
        const uint32_t chunks = n_pow2 / 2048u;
        bitonic_local_kernel<<<chunks, 1024, 0, stream>>>(keys, vals, n_pow2, 0u);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        for (uint32_t k = 4096; k <= n_pow2; k <<= 1) {
            for (uint32_t j = k / 2; j >= 2048;) {
                const uint32_t levels = j >= 8192 ? 3u : (j >= 4096 ? 2u : 1u), blocks = ((n_pow2 >> levels) + 255) / 256;
                if (levels == 3) bitonic_global_kernel<3><<<blocks, 256, 0, stream>>>(keys, vals, n_pow2, k, j);
                else if (levels == 2) bitonic_global_kernel<2><<<blocks, 256, 0, stream>>>(keys, vals, n_pow2, k, j);
                else bitonic_global_kernel<1><<<blocks, 256, 0, stream>>>(keys, vals, n_pow2, k, j);
                j >>= levels;
                ++nl;
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
            }
            bitonic_local_kernel<<<chunks, 1024, 0, stream>>>(keys, vals, n_pow2, k);
            ++nl;
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    if (n_pad > 0 && euclid) {
        prep_fill_kernel<<<(n_pad + 255) / 256, 256, 0, stream>>>(out64, blk, n_pad, (double)INFINITY);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else if (n_pad > 0) {
        if ((e = cudaMemsetAsync(out64, 0, (size_t)n_pad * sizeof(Point64), stream)) != cudaSuccess ||
            (e = cudaMemsetAsync(blk, 0, (size_t)(n_pad / kBlk) * kBlkBytes, stream)) != cudaSuccess)
            return e;
    }
    if (n > 0) {
        prep_gather_kernel<<<(n + 255) / 256, 256, 0, stream>>>(xyz_in, n, do_sort ? vals : nullptr, seg_of_point,
                                                               seg_delta, out64, blk, euclid, eps_word);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (n_pad > 0 && caps) {
        const uint32_t groups = n_pad / kCapPoints;  // n_pad is a multiple of kPad
        prep_caps_kernel<<<(groups + 7) / 8, 256, 0, stream>>>(out64, groups, euclid,
                                                               euclid ? kCapScale3d : 1.0, caps);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const uint32_t blocks = n_pad / kPad;
        prep_caps2_kernel<<<(blocks + 7) / 8, 256, 0, stream>>>(caps, blocks, caps2);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (launches) *launches = nl;
    return cudaSuccess;
}

}  // namespace tpcf

