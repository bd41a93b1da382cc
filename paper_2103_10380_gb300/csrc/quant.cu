// quant.cu -- cache storage conversion: binary32 source arrays -> FP32 / FP16 /
// FP8-E4M3 cache records, with per-channel FP8 scales from a device absmax.
//
// Densities are clamped to >= 0 (NaN -> 0) before storage. FP16 rounds to
// nearest even; FP8 stores E4M3(x / scale_c) rounded to nearest even and
// saturated to +-448, scale_c = absmax_c / 448 (binary32 division; 1 for an
// all-zero channel). For the (u, v, w) channels x is the residual from the
// cell's offset brick: the binary16 midrange of the channel over the brick. The (u, v, w) records are padded to rec_stride bytes with
// zeros so every record starts on a 16-byte (FP8: 8-byte) boundary.
// The brick occupancy bits are derived from the stored densities with the
// march's own dequantisation, so "brick empty" means exactly that every
// density the march could load there is 0.
//
// All of this is bound by memory bandwidth (4 (1 + 3D) bytes read per cell and
// pass), so the kernels over the channels share one mapping: a thread owns a
// fixed group of VEC consecutive floats of an x-row -- a fixed x, fixed channels
// and so one brick, one set of offsets and scales -- and walks the rows (y, z) of
// a square of rows, 64 for the offset bricks of k = 512. Index arithmetic, offset
// and scale loads are paid once per thread instead of once per element, a warp
// reads 512 consecutive bytes per row, and the loads of several rows are in
// flight together. E4M3 reads the source twice (min / max, then codes).
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "fnr_internal.h"
#include "march_device.cuh"

namespace fnr {

namespace {

__device__ __forceinline__ float clamp_density(float v) { return v > 0.0f ? v : 0.0f; }

__device__ __forceinline__ unsigned char to_e4m3(float v) {
    return static_cast<unsigned char>(__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3));
}

// W codes, four to a word, the conversions in pairs.
template <int W>
__device__ __forceinline__ unsigned to_e4m3_word(const float (&v)[W]) {
    if constexpr (W == 1) {
        return to_e4m3(v[0]);
    } else {
        unsigned q = 0u;
#pragma unroll
        for (int j = 0; j < W; j += 2)
            q |= static_cast<unsigned>(
                     __nv_cvt_float2_to_fp8x2(make_float2(v[j], v[j + 1]), __NV_SATFINITE, __NV_E4M3))
                 << (8 * j);
        return q;
    }
}

unsigned grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b > 152 * 64) b = 152 * 64;
    return static_cast<unsigned>(b < 1 ? 1 : b);
}

// Order-preserving uint key of a binary32 value (NaN excluded by the callers).
__device__ __forceinline__ unsigned order_key(float v) {
    const unsigned b = __float_as_uint(v);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_order_key(unsigned o) {
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// VEC consecutive floats of the source, one load.
template <int VEC>
__device__ __forceinline__ void load_floats(const float *__restrict__ p, float (&v)[VEC]) {
    if constexpr (VEC == 4) {
        const float4 q = __ldcs(reinterpret_cast<const float4 *>(p));
        v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else if constexpr (VEC == 2) {
        const float2 q = __ldcs(reinterpret_cast<const float2 *>(p));
        v[0] = q.x, v[1] = q.y;
    } else {
        v[0] = __ldcs(p);
    }
}

// The rows [ya, yb) of plane z that lie in the square of rows (by, .) of side
// 2^sh and in the slab's rows [r0, r1).
__device__ __forceinline__ void square_rows(int z, int by, int sh, int k, int64_t r0, int64_t r1, int &ya, int &yb) {
    const int64_t first = static_cast<int64_t>(z) * k;
    ya = static_cast<int>(max(static_cast<int64_t>(by << sh), r0 - first));
    yb = static_cast<int>(min(static_cast<int64_t>(min((by + 1) << sh, k)), r1 - first));
}

constexpr int kRowThreads = 256;

// Min and max per offset brick and channel (NaN ignored). Block (x, y, z):
// kRowThreads groups of VEC floats of the rows of offset-brick row (y, bz0 + z);
// each thread keeps its VEC minima and maxima in registers over the rows (min /
// max order -0 below +0, as the keys do), the block combines the cells of a brick
// in shared memory, and one atomic per (block, brick, channel) joins blocks and
// slabs. A group never crosses a brick: a brick's part of a row is 2^sh nch floats,
// a multiple of 4. k = 256, D = 8 (1.6 GB) took 2.41 ms with one thread per cell and
// its channels in a loop; k = 512 (12.9 GB) takes 1.73 ms here (7.4 TB/s read).
template <int VEC>
__global__ void __launch_bounds__(kRowThreads)
    brick_minmax_kernel(const float *__restrict__ uvw, int64_t r0, int64_t r1, int bz0, int k, int nch, int sh,
                        int dim, unsigned *__restrict__ kmin, unsigned *__restrict__ kmax) {
    // entries of a block: (bricks it touches) x nch <= VEC kRowThreads / 4 + 2 nch
    constexpr int kEntries = VEC * kRowThreads / 4 + 2 * 3 * FNR_MAX_D;
    __shared__ unsigned lo[kEntries], hi[kEntries];
    const int n_groups = k * nch / VEC;
    const int g0 = blockIdx.x * kRowThreads, g = g0 + threadIdx.x;
    const int g_last = min(g0 + kRowThreads, n_groups) - 1;
    const int b0 = (g0 * VEC / nch) >> sh, n_entries = (((g_last * VEC / nch) >> sh) - b0 + 1) * nch;
    for (int e = threadIdx.x; e < n_entries; e += kRowThreads) {
        lo[e] = 0xffffffffu;
        hi[e] = 0u;
    }
    __syncthreads();
    const int by = blockIdx.y, bz = bz0 + blockIdx.z;
    if (g < n_groups) {
        float mn[VEC], mx[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            mn[i] = __int_as_float(0x7f800000);
            mx[i] = -mn[i];
        }
        const int64_t row = static_cast<int64_t>(k) * nch;
        for (int z = bz << sh; z < min((bz + 1) << sh, k); ++z) {
            int ya, yb;
            square_rows(z, by, sh, k, r0, r1, ya, yb);
            const float *p = uvw + (static_cast<int64_t>(z) * k + ya - r0) * row + g * VEC;
#pragma unroll 8
            for (int y = ya; y < yb; ++y, p += row) {
                float v[VEC];
                load_floats<VEC>(p, v);
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    mn[i] = fminf(mn[i], v[i]);
                    mx[i] = fmaxf(mx[i], v[i]);
                }
            }
        }
        const int cell = g * VEC / nch, eb = ((cell >> sh) - b0) * nch;
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const int e = eb + (g * VEC + i) % nch;
            if (mn[i] <= mx[i]) {  // some value was not NaN
                atomicMin(&lo[e], order_key(mn[i]));
                atomicMax(&hi[e], order_key(mx[i]));
            }
        }
    }
    __syncthreads();
    const int64_t out = ((static_cast<int64_t>(bz) * dim + by) * dim + b0) * nch;
    for (int e = threadIdx.x; e < n_entries; e += kRowThreads)
        if (lo[e] != 0xffffffffu) {
            atomicMin(kmin + out + e, lo[e]);
            atomicMax(kmax + out + e, hi[e]);
        }
}

// Offsets: the binary16 (nearest even) value of (min + max) * 0.5 in binary32, 0 for a brick
// whose values were all NaN; the padding of each offset record is 0. Each channel's absmax of the
// residuals |binary32(u - offset)| (NaN skipped) goes to amax_bits[1 + c]: u - offset rounded is
// monotone in u, so over a brick it is reached at the brick's min or max (an infinite offset makes
// every residual infinite or NaN, the finite one of the two extremes among them), and no pass
// over the source is needed. A thread keeps one channel.
__global__ void brick_offsets_kernel(const unsigned *__restrict__ kmin, const unsigned *__restrict__ kmax,
                                     int64_t n_bricks, int nch, uint16_t *__restrict__ offs, int ostride,
                                     unsigned *__restrict__ amax_bits) {
    __shared__ unsigned smax[3 * FNR_MAX_D];
    for (int c = threadIdx.x; c < nch; c += blockDim.x) smax[c] = 0u;
    __syncthreads();
    const int per = blockDim.x / ostride;  // bricks per block and step
    const int c = threadIdx.x % ostride, lb = threadIdx.x / ostride;
    if (lb < per) {
        unsigned big = 0u;
        for (int64_t b = static_cast<int64_t>(blockIdx.x) * per + lb; b < n_bricks;
             b += static_cast<int64_t>(gridDim.x) * per) {
            float m = 0.0f;
            const unsigned ko = c < nch ? kmin[b * nch + c] : 0xffffffffu;
            const bool any = ko != 0xffffffffu;
            float lo = 0.0f, hi = 0.0f;
            if (any) {
                lo = from_order_key(ko);
                hi = from_order_key(kmax[b * nch + c]);
                m = (lo + hi) * 0.5f;
            }
            const __half mh = __float2half_rn(m);
            offs[b * ostride + c] = __half_as_ushort(mh);
            if (any) {
                const float mf = __half2float(mh), rl = fabsf(lo - mf), rh = fabsf(hi - mf);
                if (rl == rl) big = max(big, __float_as_uint(rl));
                if (rh == rh) big = max(big, __float_as_uint(rh));
            }
        }
        if (big) atomicMax(&smax[c], big);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nch; i += blockDim.x)
        if (smax[i]) atomicMax(&amax_bits[1 + i], smax[i]);
}

// four densities per thread and step when both sides are aligned for it, else one
template <int PREC, int VEC>
__global__ void convert_sigma_kernel(const float *__restrict__ in, void *__restrict__ out, int64_t n,
                                     const float *__restrict__ scale) {
    const float sc = PREC == FNR_PREC_FP8_E4M3 ? scale[0] : 1.0f;
    const int64_t groups = n / VEC, stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t first = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    auto store = [&](int64_t i, const auto &v) {
        constexpr int W = sizeof(v) / 4;
        if constexpr (PREC == FNR_PREC_FP32) {
            if constexpr (W == 4) reinterpret_cast<float4 *>(out)[i] = make_float4(v[0], v[1], v[2], v[3]);
            else static_cast<float *>(out)[i] = v[0];
        } else if constexpr (PREC == FNR_PREC_FP16) {
            if constexpr (W == 4) {
                const __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
                reinterpret_cast<uint2 *>(out)[i] =
                    make_uint2(*reinterpret_cast<const unsigned *>(&a), *reinterpret_cast<const unsigned *>(&b));
            } else static_cast<__half *>(out)[i] = __float2half_rn(v[0]);
        } else {
            float x[W];
#pragma unroll
            for (int j = 0; j < W; ++j) x[j] = __fdiv_rn(v[j], sc);
            const unsigned q = to_e4m3_word(x);
            if constexpr (W == 4) static_cast<unsigned *>(out)[i] = q;
            else static_cast<unsigned char *>(out)[i] = static_cast<unsigned char>(q);
        }
    };
#pragma unroll 4
    for (int64_t i = first; i < groups; i += stride) {
        float v[VEC];
        load_floats<VEC>(in + i * VEC, v);
#pragma unroll
        for (int j = 0; j < VEC; ++j) v[j] = clamp_density(v[j]);
        store(i, v);
    }
    if (VEC > 1 && first < n - groups * VEC) {
        float v[1] = {clamp_density(in[groups * VEC + first])};
        store(groups * VEC + first, v);
    }
}

// VEC channels of a record as stored (E4M3: residuals from the offsets m over the scales s) and their store.
template <int PREC, int VEC>
__device__ __forceinline__ void pack_channels(const float (&v)[VEC], const float (&m)[VEC], const float (&s)[VEC],
                                              unsigned (&w)[4]) {
    w[0] = w[1] = w[2] = w[3] = 0u;
    if constexpr (PREC == FNR_PREC_FP32) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) w[i] = __float_as_uint(v[i]);
    } else if constexpr (PREC == FNR_PREC_FP16) {
#pragma unroll
        for (int i = 0; i < VEC; ++i)
            w[i >> 1] |= static_cast<unsigned>(__half_as_ushort(__float2half_rn(v[i]))) << (16 * (i & 1));
    } else {
        float x[VEC];
#pragma unroll
        for (int i = 0; i < VEC; ++i) x[i] = __fdiv_rn(__fsub_rn(v[i], m[i]), s[i]);
        w[0] = to_e4m3_word(x);
    }
}
template <int BYTES>
__device__ __forceinline__ void put_channels(char *at, const unsigned (&w)[4]) {
    if constexpr (BYTES == 16) *reinterpret_cast<uint4 *>(at) = make_uint4(w[0], w[1], w[2], w[3]);
    else if constexpr (BYTES == 8) *reinterpret_cast<uint2 *>(at) = make_uint2(w[0], w[1]);
    else if constexpr (BYTES == 4) *reinterpret_cast<unsigned *>(at) = w[0];
    else if constexpr (BYTES == 2) *reinterpret_cast<uint16_t *>(at) = static_cast<uint16_t>(w[0]);
    else *reinterpret_cast<unsigned char *>(at) = static_cast<unsigned char>(w[0]);
}

// The records of the rows [r0, r1). VEC divides nch, so a thread's floats are
// channels c0 .. c0 + VEC - 1 of the cells at one x; the thread of a record's last
// channels also writes its padding (a multiple of the store's width: both divide
// the record's alignment). k = 256, D = 8 to E4M3 took 2.44 ms with one thread per
// element that found its cell, brick, offset and scale anew; k = 512 (16.1 GB read
// and written) takes 2.94 ms here, to FP16 2.92 ms (19.3 GB), to FP32 3.77 ms (25.8 GB).
template <int PREC, int VEC>
__global__ void __launch_bounds__(kRowThreads)
    convert_uvw_kernel(const float *__restrict__ in, char *__restrict__ out, int64_t r0, int64_t r1, int bz0, int k,
                       int nch, int rec_stride, const float *__restrict__ scales, const uint16_t *__restrict__ offs,
                       int sh, int dim, int ostride) {
    constexpr int kElem = PREC == FNR_PREC_FP32 ? 4 : PREC == FNR_PREC_FP16 ? 2 : 1;
    constexpr int kBytes = VEC * kElem;
    const int g = blockIdx.x * kRowThreads + threadIdx.x;
    if (g >= k * nch / VEC) return;
    const int by = blockIdx.y, bz = bz0 + blockIdx.z;
    const int x = g * VEC / nch, c0 = g * VEC - x * nch;
    const int pad = c0 + VEC == nch ? rec_stride - nch * kElem : 0;
    float m[VEC], s[VEC];
    if constexpr (PREC == FNR_PREC_FP8_E4M3) {
        const int64_t brick = (static_cast<int64_t>(bz) * dim + by) * dim + (x >> sh);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            m[i] = __half2float(__ushort_as_half(offs[brick * ostride + c0 + i]));
            s[i] = scales[1 + c0 + i];
        }
    }
    const int64_t row = static_cast<int64_t>(k) * nch, row_out = static_cast<int64_t>(k) * rec_stride;
    for (int z = bz << sh; z < min((bz + 1) << sh, k); ++z) {
        int ya, yb;
        square_rows(z, by, sh, k, r0, r1, ya, yb);
        const int64_t r = static_cast<int64_t>(z) * k + ya - r0;
        const float *p = in + r * row + g * VEC;
        char *q = out + r * row_out + static_cast<int64_t>(x) * rec_stride + c0 * kElem;
#pragma unroll 4
        for (int y = ya; y < yb; ++y, p += row, q += row_out) {
            float v[VEC];
            load_floats<VEC>(p, v);
            unsigned w[4];
            pack_channels<PREC, VEC>(v, m, s, w);
            put_channels<kBytes>(q, w);
            const unsigned zero[4] = {0u, 0u, 0u, 0u};
            for (int b = 0; b < pad; b += kBytes) put_channels<kBytes>(q + kBytes + b, zero);
        }
    }
}

__global__ void convert_beta_kernel(const float *__restrict__ in, void *__restrict__ out, int64_t n, int prec) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (prec == FNR_PREC_FP16) static_cast<__half *>(out)[i] = __float2half_rn(in[i]);
        else static_cast<float *>(out)[i] = in[i];
    }
}

// Absmax of the clamped densities into amax_bits[0]. Non-negative binary32
// values order like their bit patterns, so an unsigned max of the bits is exact
// (NaN is clamped to 0).
template <int VEC>
__global__ void sigma_absmax_kernel(const float *__restrict__ sigma, int64_t n, unsigned *__restrict__ amax_bits) {
    __shared__ unsigned smax;
    if (threadIdx.x == 0) smax = 0u;
    __syncthreads();
    unsigned big = 0u;
    const int64_t groups = n / VEC, stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t first = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
#pragma unroll 4
    for (int64_t i = first; i < groups; i += stride) {
        float v[VEC];
        load_floats<VEC>(sigma + i * VEC, v);
#pragma unroll
        for (int j = 0; j < VEC; ++j) big = max(big, __float_as_uint(clamp_density(v[j])));
    }
    if (first < n - groups * VEC) big = max(big, __float_as_uint(clamp_density(sigma[groups * VEC + first])));
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0 && big) atomicMax(&smax, big);
    __syncthreads();
    if (threadIdx.x == 0 && smax) atomicMax(&amax_bits[0], smax);
}

__global__ void scales_kernel(const unsigned *__restrict__ amax_bits, float *__restrict__ scales, int n) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) {
        const float a = __uint_as_float(amax_bits[c]);
        scales[c] = a > 0.0f ? __fdiv_rn(a, 448.0f) : 1.0f;
    }
}

// Brick occupancy bits. Bound by reading the density plane once: a thread reads V
// consecutive cells of an x-row (V divides k and the brick side, so the load is
// aligned and stays in one brick) over a square of rows of at most 8 x 8 inside a
// brick, and the lanes of a warp whose bricks share a word make one atomicOr.
// k = 512 (E4M3 / FP16 / FP32): one thread per cell, its coordinates by 64-bit
// divisions, took 317 / 341 / 364 us; this takes 68 / 53 / 84 us.
template <int PREC, int V>
__global__ void occupancy_kernel(const CacheView v, uint32_t *__restrict__ words) {
    constexpr int kElem = PREC == FNR_PREC_FP32 ? 4 : PREC == FNR_PREC_FP16 ? 2 : 1;
    constexpr int kBytes = V * kElem;
    const int k = v.k, cs = min(v.occ_shift, 3);
    const int n_slots = k / V, n_sq = (k + (1 << cs) - 1) >> cs;
    const int64_t id = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t line = id / n_slots;
    const int x = static_cast<int>(id - line * n_slots) * V;
    const int sz = static_cast<int>(line / n_sq), sy = static_cast<int>(line - static_cast<int64_t>(sz) * n_sq);
    unsigned lowest = 1u;  // E4M3: the lowest code whose dequantised value is > 0 (the scale may underflow it)
    if constexpr (PREC == FNR_PREC_FP8_E4M3)
        while (lowest < 0x7fu && !(__fmul_rn(dev::e4m3_to_float(lowest), v.scales[0]) > 0.0f)) ++lowest;
    bool any = false;
    if (sz < n_sq) {
        const int z1 = min((sz + 1) << cs, k), y0 = sy << cs, y1 = min((sy + 1) << cs, k);
        for (int z = sz << cs; z < z1; ++z) {
            const char *p = static_cast<const char *>(v.sigma) + ((static_cast<int64_t>(z) * k + y0) * k + x) * kElem;
#pragma unroll 8
            for (int y = y0; y < y1; ++y, p += static_cast<int64_t>(k) * kElem) {
                unsigned w[4] = {0u, 0u, 0u, 0u};
                if constexpr (kBytes == 16) {
                    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p));
                    w[0] = q.x, w[1] = q.y, w[2] = q.z, w[3] = q.w;
                } else if constexpr (kBytes == 8) {
                    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
                    w[0] = q.x, w[1] = q.y;
                } else if constexpr (kBytes == 4) {
                    w[0] = __ldg(reinterpret_cast<const unsigned *>(p));
                } else if constexpr (kBytes == 2) {
                    w[0] = __ldg(reinterpret_cast<const uint16_t *>(p));
                } else {
                    w[0] = __ldg(reinterpret_cast<const unsigned char *>(p));
                }
#pragma unroll
                for (int j = 0; j < (kBytes + 3) / 4; ++j) {
                    if constexpr (PREC == FNR_PREC_FP32) {
                        any = any || __uint_as_float(w[j]) > 0.0f;
                    } else if (w[j] != 0u) {
#pragma unroll
                        for (int e = 0; e < 4 / kElem; ++e) {
                            const unsigned q = (w[j] >> (8 * kElem * e)) & (kElem == 2 ? 0xffffu : 0xffu);
                            // binary16 in (0, +inf]; E4M3 codes from the lowest positive one to 448
                            any = any || (kElem == 2 ? q - 1u < 0x7c00u : q - lowest < 0x7fu - lowest);
                        }
                    }
                }
            }
        }
    }
    const int brick = ((((sz << cs) >> v.occ_shift) * v.occ_dim) + ((sy << cs) >> v.occ_shift)) * v.occ_dim +
                      (x >> v.occ_shift);
    const int word = any ? brick >> 5 : -1;
    const unsigned same = __match_any_sync(0xffffffffu, word);
    const unsigned bits = __reduce_or_sync(same, any ? 1u << (brick & 31) : 0u);
    if (any && (threadIdx.x & 31) == __ffs(same) - 1) atomicOr(words + word, bits);
}

// Distance field for passing over empty space: the Chebyshev (L-infinity)
// distance, in jump bricks (2^m occupancy bricks a side), from each jump brick
// to the nearest occupied one. dist_init_kernel writes 0 for jump bricks holding
// an occupied brick and 255 for the others; dist_fill_kernel, one block, turns
// that into distances.
__global__ void dist_init_kernel(const uint32_t *__restrict__ words, int nb, int m, uint8_t *__restrict__ dist,
                                 int nj) {
    const int64_t nj3 = static_cast<int64_t>(nj) * nj * nj;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; j < nj3; j += stride) {
        const int jx = static_cast<int>(j % nj), jy = static_cast<int>((j / nj) % nj), jz = static_cast<int>(j / nj / nj);
        bool occ = false;
        for (int z = jz << m; z < min((jz + 1) << m, nb) && !occ; ++z)
            for (int y = jy << m; y < min((jy + 1) << m, nb) && !occ; ++y)
                for (int x = jx << m; x < min((jx + 1) << m, nb) && !occ; ++x) {
                    const int64_t b = (static_cast<int64_t>(z) * nb + y) * nb + x;
                    occ = (words[b >> 5] >> (b & 31)) & 1u;
                }
        dist[j] = occ ? uint8_t(0) : uint8_t(255);
    }
}

// S_r, the jump bricks within distance r of an occupied one, is S_{r-1} dilated
// by the 3 x 3 x 3 cube, which splits into one dilation per axis. The grid has at
// most 32 jump bricks per axis, so a row along x is one word, a thread owns the
// row (y, z) and the x dilation is two shifts; the others go through shared
// memory. The distance (kDistCap + 1 where no S_r, r <= kDistCap, holds the brick)
// is the number of r in 0 .. kDistCap with the brick outside S_r, counted in bit
// planes. 32 jump bricks a side: 16 us, mostly the round trips of its loads (one
// launch per distance: 16 of 2.8 us).
__global__ void __launch_bounds__(1024) dist_fill_kernel(uint8_t *__restrict__ dist, int nj) {
    static_assert(kDistMaxDim == 32 && kDistCap < 31, "a row of jump bricks is one word, a distance five bits");
    __shared__ uint32_t sx[32 * 32], sy[32 * 32], plane[5][32 * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;  // this thread's row: y = lane, z = warp
    const uint32_t full = nj == 32 ? 0xffffffffu : (1u << nj) - 1u;
    const bool inside = lane < nj && warp < nj;
    sx[threadIdx.x] = 0u;
    __syncthreads();
    if (warp < nj) {
#pragma unroll 8
        for (int y = 0; y < nj; ++y) {  // the warp reads plane z row by row, one jump brick per lane
            const bool occ = lane < nj && dist[(static_cast<int64_t>(warp) * nj + y) * nj + lane] == 0;
            const uint32_t row = __ballot_sync(0xffffffffu, occ);
            if (lane == 0) sx[warp * 32 + y] = row;
        }
    }
    __syncthreads();
    uint32_t s = sx[threadIdx.x], count[5] = {0u, 0u, 0u, 0u, 0u};
    const int at = threadIdx.x;
    for (int r = 0; r <= kDistCap; ++r) {
        uint32_t carry = inside ? ~s & full : 0u;
#pragma unroll
        for (int p = 0; p < 5; ++p) {
            const uint32_t t = count[p] & carry;
            count[p] ^= carry;
            carry = t;
        }
        __syncthreads();  // the last round's reads of sy are done
        sx[at] = inside ? (s | (s << 1) | (s >> 1)) & full : 0u;
        __syncthreads();
        sy[at] = sx[at] | (lane > 0 ? sx[at - 1] : 0u) | (lane < 31 ? sx[at + 1] : 0u);
        __syncthreads();
        s = sy[at] | (warp > 0 ? sy[at - 32] : 0u) | (warp < 31 ? sy[at + 32] : 0u);
    }
#pragma unroll
    for (int p = 0; p < 5; ++p) plane[p][at] = count[p];
    __syncthreads();
    if (warp < nj && lane < nj)
        for (int y = 0; y < nj; ++y) {
            unsigned d = 0u;
#pragma unroll
            for (int p = 0; p < 5; ++p) d |= ((plane[p][warp * 32 + y] >> lane) & 1u) << p;
            dist[(static_cast<int64_t>(warp) * nj + y) * nj + lane] = static_cast<uint8_t>(d);
        }
}

// Brick slots in brick-index order, from the occupancy words. rank[w] = set bits
// of the words before w (one block: a scan of its share per thread, then of the
// shares), total = all set bits.
__global__ void __launch_bounds__(1024) brick_rank_kernel(const uint32_t *__restrict__ words, int64_t n_words,
                                                          uint32_t *__restrict__ rank, uint32_t *__restrict__ total) {
    __shared__ uint32_t part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0u;  // set bits of the words before this tile of 1024
    for (int64_t w0 = 0; w0 < n_words; w0 += 1024) {
        const int64_t w = w0 + threadIdx.x;
        const uint32_t own = w < n_words ? __popc(words[w]) : 0u;
        uint32_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        uint32_t sums = part[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, sums, d);
            if (lane >= d) sums += v;
        }
        const uint32_t before = warp ? __shfl_sync(0xffffffffu, sums, warp - 1) : 0u;
        if (w < n_words) rank[w] = carry + before + incl - own;
        carry += __shfl_sync(0xffffffffu, sums, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// page[b] = slot of brick b or -1, slot_brick[slot] = b.
__global__ void brick_pages_kernel(const uint32_t *__restrict__ words, const uint32_t *__restrict__ rank,
                                   int64_t n_bricks, int32_t *__restrict__ page, int32_t *__restrict__ slot_brick) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; b < n_bricks; b += stride) {
        const uint32_t w = words[b >> 5], bit = 1u << (b & 31);
        const int32_t slot = (w & bit) ? static_cast<int32_t>(rank[b >> 5] + __popc(w & (bit - 1u))) : -1;
        page[b] = slot;
        if (slot >= 0) slot_brick[slot] = static_cast<int32_t>(b);
    }
}

// The grid cell of pool element e (element slot B^3 + (lz B + ly) B + lx of brick
// slot_brick[slot]), or -1 past the grid's edge.
__device__ __forceinline__ int64_t pool_cell(int64_t e, const int32_t *__restrict__ slot_brick, int k, int shift,
                                             int dim) {
    const int mask = (1 << shift) - 1, local = static_cast<int>(e & ((int64_t(1) << (3 * shift)) - 1));
    const int brick = slot_brick[e >> (3 * shift)];
    const int by = (brick / dim) % dim, bz = brick / (dim * dim), bx = brick - (bz * dim + by) * dim;
    const int x = (bx << shift) + (local & mask), y = (by << shift) + ((local >> shift) & mask),
              z = (bz << shift) + (local >> (2 * shift));
    return x < k && y < k && z < k ? (static_cast<int64_t>(z) * k + y) * k + x : -1;
}

// One element T of `units` per cell and thread: densities (units = 1) or records in 16- or 8-byte
// pieces, so that a warp copies consecutive bytes. Cells past the grid edge are 0.
template <class T>
__global__ void gather_bricks_kernel(const T *__restrict__ plane, T *__restrict__ pool,
                                     const int32_t *__restrict__ slot_brick, int64_t n_elems, int units, int k,
                                     int shift, int dim) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x, n = n_elems * units;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t e = units == 1 ? i : i / units;
        const int64_t cell = pool_cell(e, slot_brick, k, shift, dim);
        pool[i] = cell >= 0 ? plane[cell * units + (i - e * units)] : T{};
    }
}

// The records of the pool's cells from the binary32 source: VEC channels per thread as
// convert_uvw_kernel packs them, read where the brick's cells lie (runs of B cells of an x-row), so
// empty bricks' channels are neither read nor stored. k = 250, D = 8, FP16, a quarter of the bricks kept:
// 104 us, against 369 us for all records and 79 us to gather them.
template <int PREC, int VEC>
__global__ void convert_bricks_kernel(const float *__restrict__ uvw, char *__restrict__ pool,
                                      const int32_t *__restrict__ slot_brick, int64_t n_elems, int k, int nch,
                                      int rec_stride, int shift, int dim, const float *__restrict__ scales,
                                      const uint16_t *__restrict__ offs, int oshift, int odim, int ostride) {
    constexpr int kElem = PREC == FNR_PREC_FP32 ? 4 : PREC == FNR_PREC_FP16 ? 2 : 1;
    constexpr int kBytes = VEC * kElem;
    const int groups = nch / VEC;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x, n = n_elems * groups;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t e = i / groups;
        const int c0 = static_cast<int>(i - e * groups) * VEC;
        const int64_t cell = pool_cell(e, slot_brick, k, shift, dim);
        unsigned w[4] = {0u, 0u, 0u, 0u};
        const unsigned zero[4] = {0u, 0u, 0u, 0u};
        if (cell >= 0) {
            float v[VEC], m[VEC], s[VEC];
            load_floats<VEC>(uvw + cell * nch + c0, v);
            if constexpr (PREC == FNR_PREC_FP8_E4M3) {
                const int row = static_cast<int>(cell / k), x = static_cast<int>(cell - static_cast<int64_t>(row) * k);
                const int z = row / k, y = row - z * k;
                const int64_t ob = (static_cast<int64_t>(z >> oshift) * odim + (y >> oshift)) * odim + (x >> oshift);
#pragma unroll
                for (int j = 0; j < VEC; ++j) {
                    m[j] = __half2float(__ushort_as_half(offs[ob * ostride + c0 + j]));
                    s[j] = scales[1 + c0 + j];
                }
            }
            pack_channels<PREC, VEC>(v, m, s, w);
        }
        char *q = pool + e * rec_stride + c0 * kElem;
        put_channels<kBytes>(q, w);
        if (c0 + VEC == nch)
            for (int b = nch * kElem; b < rec_stride; b += kBytes) put_channels<kBytes>(pool + e * rec_stride + b, zero);
    }
}

}  // namespace

cudaError_t launch_brick_rank(const uint32_t *words, int64_t n_words, uint32_t *rank, uint32_t *total,
                              cudaStream_t s) {
    brick_rank_kernel<<<1, 1024, 0, s>>>(words, n_words, rank, total);
    return cudaGetLastError();
}

cudaError_t launch_brick_pages(const uint32_t *words, const uint32_t *rank, int64_t n_bricks, int32_t *page,
                               int32_t *slot_brick, cudaStream_t s) {
    brick_pages_kernel<<<grid_for(n_bricks, 256), 256, 0, s>>>(words, rank, n_bricks, page, slot_brick);
    return cudaGetLastError();
}

namespace {

template <class T>
cudaError_t gather_as(const void *plane, void *pool, const int32_t *slot_brick, int64_t n, int units, int k, int shift,
                      int dim, cudaStream_t s) {
    gather_bricks_kernel<T><<<grid_for(n * units, 256), 256, 0, s>>>(
        static_cast<const T *>(plane), static_cast<T *>(pool), slot_brick, n, units, k, shift, dim);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gather_bricks(const void *plane, void *pool, const int32_t *slot_brick, int64_t n_bricks, int k,
                                 int shift, int dim, int stride, cudaStream_t s) {
    const int64_t n = n_bricks << (3 * shift);
    if (stride % 16 == 0) return gather_as<uint4>(plane, pool, slot_brick, n, stride / 16, k, shift, dim, s);
    if (stride % 8 == 0) return gather_as<uint2>(plane, pool, slot_brick, n, stride / 8, k, shift, dim, s);
    if (stride == 4) return gather_as<uint32_t>(plane, pool, slot_brick, n, 1, k, shift, dim, s);
    if (stride == 2) return gather_as<uint16_t>(plane, pool, slot_brick, n, 1, k, shift, dim, s);
    return gather_as<uint8_t>(plane, pool, slot_brick, n, stride, k, shift, dim, s);
}

namespace {

template <int PREC, int V>
void occupancy_v(const CacheView &v, uint32_t *words, int width, cudaStream_t s) {
    constexpr int kElem = PREC == FNR_PREC_FP32 ? 4 : PREC == FNR_PREC_FP16 ? 2 : 1;
    if constexpr (V * kElem < 16)
        if (width > V) return occupancy_v<PREC, 2 * V>(v, words, width, s);
    const int cs = std::min(v.occ_shift, 3);
    const int64_t sq = (v.k + (1 << cs) - 1) >> cs, n = sq * sq * (v.k / V);
    occupancy_kernel<PREC, V><<<static_cast<unsigned>((n + 127) / 128), 128, 0, s>>>(v, words);
}

}  // namespace

cudaError_t launch_occupancy(const CacheView &v, uint32_t *words, cudaStream_t s) {
    // cells per load: a power of two that divides the row and the brick side (at most 16 bytes)
    int width = 1;
    while (width < 16 && v.k % (2 * width) == 0 && width < (1 << v.occ_shift)) width *= 2;
    if (v.pos_prec == FNR_PREC_FP16) occupancy_v<FNR_PREC_FP16, 1>(v, words, width, s);
    else if (v.pos_prec == FNR_PREC_FP8_E4M3) occupancy_v<FNR_PREC_FP8_E4M3, 1>(v, words, width, s);
    else occupancy_v<FNR_PREC_FP32, 1>(v, words, width, s);
    return cudaGetLastError();
}

cudaError_t launch_brick_distance(const uint32_t *words, int nb, int occ_shift, uint8_t *dist, int nj,
                                  int dist_shift, cudaStream_t s) {
    const int64_t nj3 = static_cast<int64_t>(nj) * nj * nj;
    if (nj3 <= 0) return cudaSuccess;
    dist_init_kernel<<<grid_for(nj3, 256), 256, 0, s>>>(words, nb, dist_shift - occ_shift, dist, nj);
    dist_fill_kernel<<<1, 1024, 0, s>>>(dist, nj);
    return cudaGetLastError();
}

namespace {

bool aligned(const void *p, size_t bytes) { return reinterpret_cast<uintptr_t>(p) % bytes == 0; }

// Floats per load for a source at p whose groups must divide `unit` floats.
int group_width(const float *p, int64_t unit) {
    if (unit % 4 == 0 && aligned(p, 16)) return 4;
    return unit % 2 == 0 && aligned(p, 8) ? 2 : 1;
}

// Blocks over the rows [r0, r1): groups of an x-row, squares of rows along y, the squares along z that the
// rows reach (the first of them in *bz0).
dim3 row_grid(int64_t r0, int64_t r1, int k, int nch, int vec, int sh, int *bz0) {
    *bz0 = static_cast<int>(r0 / k) >> sh;
    const int bz1 = static_cast<int>((r1 - 1) / k) >> sh;
    const int groups = k * nch / vec;
    return dim3(static_cast<unsigned>((groups + kRowThreads - 1) / kRowThreads),
                static_cast<unsigned>((k + (1 << sh) - 1) >> sh), static_cast<unsigned>(bz1 - *bz0 + 1));
}

template <int PREC>
void convert_sigma_p(const float *in, void *out, int64_t n, const float *scale, cudaStream_t s) {
    constexpr size_t es = PREC == FNR_PREC_FP32 ? 4 : PREC == FNR_PREC_FP16 ? 2 : 1;
    if (aligned(in, 16) && aligned(out, 4 * es))
        convert_sigma_kernel<PREC, 4><<<grid_for((n + 3) / 4, 256), 256, 0, s>>>(in, out, n, scale);
    else
        convert_sigma_kernel<PREC, 1><<<grid_for(n, 256), 256, 0, s>>>(in, out, n, scale);
}

template <int PREC>
void convert_uvw_p(const float *in, char *out, int64_t r0, int64_t r1, int k, int nch, int rec_stride,
                   const float *scales, const uint16_t *offs, int sh, int dim, int ostride, cudaStream_t s) {
    const int vec = group_width(in, nch);
    int bz0;
    const dim3 grid = row_grid(r0, r1, k, nch, vec, sh, &bz0);
    if (vec == 4)
        convert_uvw_kernel<PREC, 4><<<grid, kRowThreads, 0, s>>>(in, out, r0, r1, bz0, k, nch, rec_stride, scales, offs,
                                                                 sh, dim, ostride);
    else if (vec == 2)
        convert_uvw_kernel<PREC, 2><<<grid, kRowThreads, 0, s>>>(in, out, r0, r1, bz0, k, nch, rec_stride, scales, offs,
                                                                 sh, dim, ostride);
    else
        convert_uvw_kernel<PREC, 1><<<grid, kRowThreads, 0, s>>>(in, out, r0, r1, bz0, k, nch, rec_stride, scales, offs,
                                                                 sh, dim, ostride);
}

}  // namespace

cudaError_t launch_convert_sigma(const float *in, void *out, int64_t n, int prec, const float *scale, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (prec == FNR_PREC_FP32) convert_sigma_p<FNR_PREC_FP32>(in, out, n, scale, s);
    else if (prec == FNR_PREC_FP16) convert_sigma_p<FNR_PREC_FP16>(in, out, n, scale, s);
    else convert_sigma_p<FNR_PREC_FP8_E4M3>(in, out, n, scale, s);
    return cudaGetLastError();
}

cudaError_t launch_convert_uvw(const float *in, char *out, int64_t r0, int64_t r1, int k, int D, int prec,
                               int rec_stride, const float *scales, const uint16_t *offs, int oshift, int odim,
                               int ostride, cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    constexpr int kSquare = 3;  // 8 x 8 rows per thread where no offset brick sets the square
    if (prec == FNR_PREC_FP32)
        convert_uvw_p<FNR_PREC_FP32>(in, out, r0, r1, k, 3 * D, rec_stride, scales, offs, kSquare, 0, 0, s);
    else if (prec == FNR_PREC_FP16)
        convert_uvw_p<FNR_PREC_FP16>(in, out, r0, r1, k, 3 * D, rec_stride, scales, offs, kSquare, 0, 0, s);
    else if (!offs)
        return cudaErrorInvalidValue;
    else
        convert_uvw_p<FNR_PREC_FP8_E4M3>(in, out, r0, r1, k, 3 * D, rec_stride, scales, offs, oshift, odim, ostride, s);
    return cudaGetLastError();
}

namespace {

template <int PREC, int VEC>
void convert_bricks_v(const float *uvw, char *pool, const int32_t *slot_brick, int64_t n, int k, int nch,
                      int rec_stride, int shift, int dim, const float *scales, const uint16_t *offs, int oshift,
                      int odim, int ostride, cudaStream_t s) {
    convert_bricks_kernel<PREC, VEC><<<grid_for(n * (nch / VEC), 256), 256, 0, s>>>(
        uvw, pool, slot_brick, n, k, nch, rec_stride, shift, dim, scales, offs, oshift, odim, ostride);
}

template <int PREC, class... A>
void convert_bricks_p(int vec, A... args) {
    if (vec == 4) convert_bricks_v<PREC, 4>(args...);
    else if (vec == 2) convert_bricks_v<PREC, 2>(args...);
    else convert_bricks_v<PREC, 1>(args...);
}

}  // namespace

cudaError_t launch_convert_bricks(const float *uvw, char *pool, const int32_t *slot_brick, int64_t n_bricks, int k,
                                  int D, int prec, int rec_stride, int shift, int dim, const float *scales,
                                  const uint16_t *offs, int oshift, int odim, int ostride, cudaStream_t s) {
    const int64_t n = n_bricks << (3 * shift);
    const int nch = 3 * D, vec = group_width(uvw, nch);
    if (n <= 0) return cudaSuccess;
    if (prec == FNR_PREC_FP32)
        convert_bricks_p<FNR_PREC_FP32>(vec, uvw, pool, slot_brick, n, k, nch, rec_stride, shift, dim, scales, offs,
                                        oshift, odim, ostride, s);
    else if (prec == FNR_PREC_FP16)
        convert_bricks_p<FNR_PREC_FP16>(vec, uvw, pool, slot_brick, n, k, nch, rec_stride, shift, dim, scales, offs,
                                        oshift, odim, ostride, s);
    else
        convert_bricks_p<FNR_PREC_FP8_E4M3>(vec, uvw, pool, slot_brick, n, k, nch, rec_stride, shift, dim, scales,
                                            offs, oshift, odim, ostride, s);
    return cudaGetLastError();
}

cudaError_t launch_brick_minmax(const float *uvw, int64_t r0, int64_t r1, int k, int nch, int oshift, int odim,
                                unsigned *kmin, unsigned *kmax, cudaStream_t s) {
    if (r1 <= r0) return cudaSuccess;
    const int vec = group_width(uvw, static_cast<int64_t>(k) * nch);
    int bz0;
    const dim3 grid = row_grid(r0, r1, k, nch, vec, oshift, &bz0);
    if (vec == 4)
        brick_minmax_kernel<4><<<grid, kRowThreads, 0, s>>>(uvw, r0, r1, bz0, k, nch, oshift, odim, kmin, kmax);
    else if (vec == 2)
        brick_minmax_kernel<2><<<grid, kRowThreads, 0, s>>>(uvw, r0, r1, bz0, k, nch, oshift, odim, kmin, kmax);
    else
        brick_minmax_kernel<1><<<grid, kRowThreads, 0, s>>>(uvw, r0, r1, bz0, k, nch, oshift, odim, kmin, kmax);
    return cudaGetLastError();
}

cudaError_t launch_brick_offsets(const unsigned *kmin, const unsigned *kmax, int64_t n_bricks, int nch,
                                 uint16_t *offs, int ostride, unsigned *amax_bits, cudaStream_t s) {
    if (n_bricks <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n_bricks * ostride + 255) / 256, 152 * 8);
    brick_offsets_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(kmin, kmax, n_bricks, nch, offs, ostride,
                                                                        amax_bits);
    return cudaGetLastError();
}

cudaError_t launch_convert_beta(const float *in, void *out, int64_t n, int prec, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    convert_beta_kernel<<<grid_for(n, 256), 256, 0, s>>>(in, out, n, prec);
    return cudaGetLastError();
}

cudaError_t launch_sigma_absmax(const float *sigma, int64_t n, unsigned *amax_bits, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (aligned(sigma, 16)) sigma_absmax_kernel<4><<<grid_for((n + 3) / 4, 256), 256, 0, s>>>(sigma, n, amax_bits);
    else sigma_absmax_kernel<1><<<grid_for(n, 256), 256, 0, s>>>(sigma, n, amax_bits);
    return cudaGetLastError();
}

cudaError_t launch_scales_from_absmax(const unsigned *amax_bits, float *scales, int n, cudaStream_t s) {
    scales_kernel<<<1, 64, 0, s>>>(amax_bits, scales, n);
    return cudaGetLastError();
}

}  // namespace fnr
