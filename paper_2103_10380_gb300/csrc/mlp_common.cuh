// mlp_common.cuh -- what the two forms of the tensor-core MLP kernel share
// (mlp.cu: one CTA per SM; mlp_pair.cu: a CTA pair per MMA): the launch
// arguments, the PTX wrappers, bounded waits and the positional encoding.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fnr_internal.h"

namespace fnr {
namespace mlp {

constexpr int kTileM = 128;
constexpr int kMaxK = 256;
constexpr int kMaxN = 256;
constexpr int kChunkK = 64;         // K columns per weight chunk: one 128-byte swizzle row
constexpr int kMaxK0 = kChunkK;     // the encoded input (layer 0's K) fits one staging chunk
constexpr int kMaxHeadOut = 64;     // outputs per point staged after the head
constexpr int kMaxLayers = 16;
constexpr int kPair = 2;            // tiles in flight per CTA
constexpr size_t kStageBytes = size_t(kTileM) * kMaxK0 * 2;  // 16 KB layer-0 input per tile
constexpr uint32_t kSuspendNs = 2000;                        // a poll may sleep this long: it leaves the issue slots
constexpr long long kWaitLimit = 1LL << 22;                  // try_wait polls before giving up
constexpr long long kDrainLimit = 1LL << 22;                 // polls for in-flight work at exit

struct MlpLayerDev {
    const __nv_bfloat16 *w;  // chunk-major: chunk c = [Np][64] in the 128-byte swizzled K-major layout
    int K, N;                // padded to multiples of 16
    int bias_off;            // offset of this layer's Np biases in the bias table
};

struct MlpArgs {
    MlpLayerDev L[kMaxLayers];
    const float *bias;       // all layers' padded biases
    int n_bias;
    int n_layers;
    int mode;        // 0: F_pos over the k^3 cell centres, 1: F_dir over the l x l bin centres
    int pe_freqs;
    int k, l;
    float bmin[3], h[3];
    long long n_points;                // or, with n_dev, their upper bound
    const unsigned long long *n_dev;   // the number of points, if the host does not know it
    // outputs
    void *sigma_out;   // mode 0
    char *uvw_out;     // mode 0
    int rec_stride, prec, D;
    void *beta_out;    // mode 1
    int dprec;
    // mode 2: F evaluated at listed points (positions, or unit directions for F_dir); the head's
    // first out_stride outputs go to out[p * out_stride + c] in FP32 (channel 0 through ReLU if relu0)
    const float *points;  // [n_points][3]
    float *out;
    int out_stride, relu0;
    int n_out;        // outputs stored per point: 1 + 3D (mode 0), D (mode 1), out_stride (mode 2)
    int head_stride;  // floats per staged head row: round16(n_out) + 4
    int *err;
    long long wait_limit;  // polls before a wait gives up (kWaitLimit unless a test armed a fault)
    long long withhold;    // test fault: the producer withholds its chunk of this index (-1: none)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// A poll sleeps up to kSuspendNs until the phase completes, so the waiting warps leave the issue slots to the others
// (192^3 in the single-CTA form: 1290 -> 1470 TFLOP/s with the sums of the epilogue in pairs).
// kCluster: acquire at cluster scope, for a barrier that the other CTA of the
// pair arrives on with data of its own to order (epilogue and encoder
// hand-offs); else the default CTA scope (weight chunks, slot releases,
// accumulators: completions of the pair's own copies and tensor-core work).
template <bool kCluster>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if (kCluster)
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendNs)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendNs)
            : "memory");
    return ok != 0;
}

// Bounded wait: false when `limit` polls run out (the error word and the
// CTA's abort flag -- and the peer CTA's, at cluster address peer_abort if
// non-zero -- are then set) or when another role has aborted.
template <bool kCluster>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int *err, volatile int *abort_flag,
                                          long long limit, uint32_t peer_abort) {
    for (long long it = 0; it < limit; ++it) {
        if (mbar_try_wait<kCluster>(bar, parity)) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
    }
    atomicExch(err, 1);
    *abort_flag = 1;
    if (peer_abort) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_abort), "r"(1) : "memory");
    return false;
}

// Bounded wait at exit for work this CTA has in flight, abort or not; false
// (and the error word set) if it does not complete within kDrainLimit polls.
template <bool kCluster>
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity, int *err) {
    for (long long it = 0; it < kDrainLimit; ++it)
        if (mbar_try_wait<kCluster>(bar, parity)) return true;
    atomicExch(err, 2);
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major with the 128-byte swizzle: rows of
// 64 bf16 (128 bytes), 8-row atoms of 1024 bytes stacked along M / N
// (stride 1024), the 16-byte pieces of row r stored at piece index ^ (r & 7).
// Atoms start on 1024-byte boundaries; a K step of 16 inside the atom row
// advances the start address by 32 bytes. The leading-dimension offset is
// unused by this layout (encoded as 1).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= uint64_t((addr >> 4) & 0x3FFFu);
    d |= uint64_t(1) << 16;                 // leading byte offset (unused), 16 bytes
    d |= uint64_t(1024 >> 4) << 32;         // stride byte offset: 8 rows x 128 bytes
    d |= uint64_t(1) << 46;                 // descriptor version for this architecture
    d |= uint64_t(2) << 61;                 // swizzle mode: 128 bytes
    return d;                               // base offset 0
}

// Instruction descriptor, kind::f16: bf16 A and B (both K-major), fp32 D.
__device__ __forceinline__ uint32_t instr_desc(int M, int N) {
    uint32_t d = 0;
    d |= 1u << 4;                            // D format fp32
    d |= 1u << 7;                            // A format bf16
    d |= 1u << 10;                           // B format bf16
    d |= uint32_t(N >> 3) << 17;
    d |= uint32_t(M >> 4) << 24;
    return d;
}

// 16 columns of this warp's TMEM lane quarter, without waiting (see tmem_wait).
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Byte offset of element (row, k) of the A tile (kTileM rows) in the 128-byte
// swizzled K-major layout: 64-column K blocks of kTileM / 8 atoms each.
__device__ __forceinline__ uint32_t a_offset(int row, int k) {
    return uint32_t((k >> 6) * (kTileM / 8) * 1024 + (row >> 3) * 1024 + (row & 7) * 128 +
                    ((((k >> 3) & 7) ^ (row & 7)) << 4) + (k & 7) * 2);
}

// ReLU(a), ReLU(b) rounded to bf16 (nearest even) and packed, a in the low
// half, in one conversion; a negative value rounds to a negative bf16, so
// clamping after rounding equals rounding after clamping.
__device__ __forceinline__ uint32_t pack_relu_bf16(float a, float b) {
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat16 x = __float2bfloat16_rn(a), y = __float2bfloat16_rn(b);
    return uint32_t(__bfloat16_as_ushort(x)) | (uint32_t(__bfloat16_as_ushort(y)) << 16);
}

__device__ __forceinline__ long long point_count(const MlpArgs &A) {
    return A.n_dev ? static_cast<long long>(*A.n_dev) : A.n_points;
}

// Positional encoding of point p into row `row` of a layer-0 A tile (K0 <= 64
// columns, one 128-byte swizzled row): column 2 P + 0 / 1 holds sin / cos(2^j
// pi x_a) with P = a L + j, rounded to bf16; columns from 6 L on, and every
// column of a point past the end, are 0.
__device__ __forceinline__ void encode_point(const MlpArgs &A, long long n_points, long long p, int row, char *sa) {
    const int K0 = A.L[0].K;
    float x0 = 0.0f, x1 = 0.0f, x2 = 0.0f;
    const bool valid = p < n_points;
    if (valid) {
        if (A.mode == 2) {
            x0 = A.points[3 * p];
            x1 = A.points[3 * p + 1];
            x2 = A.points[3 * p + 2];
        } else if (A.mode == 0) {
            int ix, iy, iz;
            if (A.n_points <= 0x7fffffffLL) {  // 32-bit index arithmetic
                const unsigned k = unsigned(A.k), q = unsigned(p);
                const unsigned yz = q / k;
                ix = int(q - yz * k);
                iz = int(yz / k);
                iy = int(yz - unsigned(iz) * k);
            } else {
                const long long kk = A.k;
                ix = int(p % kk);
                iy = int((p / kk) % kk);
                iz = int(p / (kk * kk));
            }
            x0 = fmaf(float(ix) + 0.5f, A.h[0], A.bmin[0]);
            x1 = fmaf(float(iy) + 0.5f, A.h[1], A.bmin[1]);
            x2 = fmaf(float(iz) + 0.5f, A.h[2], A.bmin[2]);
        } else {
            const unsigned q = unsigned(p), l = unsigned(A.l);
            const int it = int(q / l), ip = int(q - unsigned(it) * l);
            float st, ct, sp, cp;
            sincospif((float(it) + 0.5f) / float(A.l), &st, &ct);         // theta / pi
            sincospif(2.0f * (float(ip) + 0.5f) / float(A.l), &sp, &cp);  // phi / pi
            x0 = st * cp;
            x1 = st * sp;
            x2 = ct;
        }
    }
    const int nP = valid ? 3 * A.pe_freqs : 0;
    int a = 0, j = 0;  // (a, j) of P, advanced with P
    for (int g = 0; g < K0; g += 8) {  // 8 encoded values per 16-byte store
        float v[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int P = (g >> 1) + q;
            float sv = 0.0f, cv = 0.0f;
            if (P < nP) {
                const float xa = a == 0 ? x0 : (a == 1 ? x1 : x2);
                sincospif(xa * __int_as_float((127 + j) << 23), &sv, &cv);  // 2^j x_a, exact
                if (++j == A.pe_freqs) {
                    j = 0;
                    ++a;
                }
            }
            v[2 * q] = sv;
            v[2 * q + 1] = cv;
        }
        uint4 pk;
        pk.x = pack_bf16(v[0], v[1]);
        pk.y = pack_bf16(v[2], v[3]);
        pk.z = pack_bf16(v[4], v[5]);
        pk.w = pack_bf16(v[6], v[7]);
        *reinterpret_cast<uint4 *>(sa + a_offset(row, g)) = pk;
    }
}

__device__ __forceinline__ int n_chunks(int K) { return K / kChunkK; }  // K is padded to a multiple of 64

}  // namespace mlp

// One launch of either form on prepared arguments: one CTA (pair) per SM (pair)
// that can be resident at once, at most one per MMA tile.
fnr_status launch_mlp_single(const mlp::MlpArgs &A, int num_sms, cudaStream_t s);
fnr_status launch_mlp_pair(const mlp::MlpArgs &A, int num_sms, cudaStream_t s);

}  // namespace fnr
