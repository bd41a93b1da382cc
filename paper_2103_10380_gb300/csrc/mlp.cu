// mlp.cu -- cache build from the F_pos / F_dir MLPs on the 5th-generation
// tensor cores (Section 3.3: the caches hold F evaluated at every grid sample;
// Section 3.2 Eqs. 3-4 and Section 4: F_pos and F_dir are ReLU MLPs on
// positionally encoded inputs), and the same networks at listed points.
//
// One CTA per SM walks tiles of 128 points, two at a time. Per layer it computes
// D[128 points][N] = A[128][K] W^T in halves of up to 128 outputs, and the two
// tiles alternate, so the tensor core works on one while the other's outputs
// become its next inputs. What bounds such a kernel on one SM is shared memory:
// with both operands there, an MMA step of 128 x 256 x 16 (128 cycles) reads 12 KB
// of it, and the weights' arrival and the activations' way back come on top --
// together about 1.5 times the 128 bytes a cycle that it has. So
//   the activations never leave tensor memory: the epilogue reads a half's fp32
//     accumulator, adds the bias, applies ReLU, rounds to bf16 and stores it as
//     the next layer's A operand in tensor memory (tcgen05.mma with A in tmem);
//     only the encoded input of layer 0 lies in shared memory;
//   the weights are streamed once per layer for both tiles: 32 KB blocks (128
//     outputs x 128 inputs, two K-major 128-byte-swizzled parts) in a ring of 5
//     slots, a whole layer of 4 and one ahead.
// Tensor memory, 512 columns: A of tile 0 and of tile 1 (128 columns each, two
// bf16 a column) and two accumulator blocks (128 columns), one per half, which
// both tiles use in turn. A half takes 16 MMAs of 64 cycles, so the epilogue has
// 1024 cycles to read a block before the other tile's same half is due, and a
// whole step of the other tile (2048) to write A.
//
// Warp roles:
//   epilogue (warps 0-15, four per 32-lane quarter of tensor memory, 32 columns
//     of a half each): hidden layers, as above;
//   auxiliary (warps 16-19, one per quarter): encode the points of the next two
//     tiles (gamma(x) = sin / cos(2^j pi x), rounded to bf16) as soon as layer 0's
//     MMAs have read the buffer, and take the head's outputs from its accumulator
//     through a staging row per point to the cache -- sigma = ReLU(out_0), (u, v, w)
//     = out_1..3D (F_pos), beta = out_0..D-1 (F_dir) -- while the epilogue warps go
//     on with the other tile and the next pair;
//   producer (warp 20): the weight ring, by bulk async copies;
//   MMA issuer (warp 21, one lane).
//
// Order: every wait below is a bounded mbarrier wait. An accumulator block is
// written again after its readers have arrived (acc_free), A is read after its
// writers have (a_ready) and overwritten after the commit of the last MMA that
// read it (acc_full of the step's last half), a ring slot is refilled after the
// commit of its last MMA (empty). A wait that runs out sets the error word and
// the CTA's abort flag; every role leaves its loop, the producer waits (bounded)
// for the copies it has in flight, the MMA issuer for its tensor-core
// operations, and the tensor memory is freed.
//
// Measured on 512^3 + 512^2 (D = 8, FP32, the whole call with its 13.4 GB allocation): 84 ms, 1530 TFLOP/s,
// against 132 ms with the activations in shared memory, N = 256 MMAs and a two-slot ring loaded once per tile.
// On 192^3 alone: 1580 TFLOP/s; without the epilogue's work 1820, without the weights' 1680, without the encoding
// 1650, without any of them 1960. Tried in this layout: both halves in one N = 256 MMA but for the first and last
// quarter of the inputs 1190 (an accumulator block is read too late), halves of 64 inputs in turn 1360; the biases
// through L1 1470; polling by one lane of a warp and a shuffle 1070.
#include "mlp_common.cuh"

namespace fnr {

fnr_status fail(fnr_status st, const char *fmt, ...);
fnr_status cuda_fail(cudaError_t e, const char *what);

namespace {

using namespace mlp;

constexpr int kEpiWarps = 16, kAuxWarp0 = 16, kAuxWarps = 4, kProducerWarp = 20, kMmaWarp = 21;
constexpr int kThreads = 22 * 32;
constexpr int kHalfN = 128;                             // outputs of an accumulator block
constexpr int kSlots = 5;                               // ring slots of one weight block
constexpr uint32_t kPartBytes = kHalfN * kChunkK * 2;   // 128 outputs x 64 inputs: 16 KB
constexpr uint32_t kSlotBytes = 2 * kPartBytes;         // 128 outputs x 128 inputs
constexpr size_t kSmemRing = size_t(kSlots) * kSlotBytes;
constexpr size_t kSmemStage = size_t(kPair) * kStageBytes;
constexpr int kMaxOut = 1 + 3 * FNR_MAX_D;              // outputs stored per point
// full, empty per slot; acc_full, acc_free per half; a_ready, enc_ready, enc_free, head_full per tile; drain
constexpr int kBars = 2 * kSlots + 2 * 2 + 4 * kPair + 1;
constexpr int kHeadCols = 32, kHeadFloats = 32 * (kHeadCols + 1);  // per auxiliary warp: 32 rows, odd stride
constexpr size_t kSmemHead = size_t(kAuxWarps) * kHeadFloats * 4;
constexpr size_t kSmemBias = size_t(kMaxLayers) * kMaxN * 4;
constexpr size_t kSmemCtl = size_t(kBars) * 8 + 16;  // barriers, tensor memory address, abort flag
constexpr size_t kSmemBytes = kSmemRing + kSmemStage + kSmemBias + kSmemHead + kSmemCtl + 1024;  // + alignment slack
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
static_assert(kMaxK / kChunkK < kSlots, "a layer's weight blocks fit the ring, and one ahead");
constexpr uint32_t kTmemCols = 512, kAccCol = 256;      // A of tile t at column 128 t, block h at 256 + 128 h

// D (tmem) = or += A B^T for one K step of 16: A from shared memory, or from tensor memory. The whole warp
// executes these with uniform operands, the lane with `one` set issues: a branch around them instead would move
// the operands out of the uniform registers that the instruction reads (19 against 44 cycles of issue for each).
__device__ __forceinline__ void umma_ss(uint32_t one, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(one)
        : "memory");
}
__device__ __forceinline__ void umma_ts(uint32_t one, uint32_t d, uint32_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(one)
        : "memory");
}

// Arrive on the mbarrier at `bar` when every tcgen05 operation this thread has issued so far has completed.
__device__ __forceinline__ void umma_commit(uint32_t one, uint32_t bar) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
        "r"(one)
        : "memory");
}

// One lane of the (converged) warp, the same one every time.
__device__ __forceinline__ uint32_t elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p;
}

// The two halves of smem_desc_sw128: the low word of a tile's address (a K step of 16 adds 2), and the descriptor
// of a low word.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint64_t desc_sw128(uint32_t lo) {
    return (uint64_t((1024u >> 4) | (1u << 14) | (2u << 29)) << 32) | lo;
}

// One poll that does not sleep.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}

// 32 columns of this warp's lane quarter, read and waited for.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

// 16 columns of this warp's lane quarter, without waiting (tcgen05.wait::st).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

// ReLU(a + x), ReLU(b + y) as bf16, a's in the low half; the two binary32 sums in one instruction.
__device__ __forceinline__ uint32_t bias_relu_bf16(uint32_t a, uint32_t b, float x, float y) {
    uint32_t lo, hi;
    asm("{\n .reg .b64 u, v;\n mov.b64 u, {%2, %3};\n mov.b64 v, {%4, %5};\n add.rn.f32x2 u, u, v;\n"
        " mov.b64 {%0, %1}, u;\n}\n"
        : "=r"(lo), "=r"(hi)
        : "r"(a), "r"(b), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)));
    return pack_relu_bf16(__uint_as_float(lo), __uint_as_float(hi));
}

// 32 accumulator columns from output n0 on -> 16 columns of A: ReLU(acc + bias) as bf16, outputs past N as 0.
// bias: shared-memory address of output 0's. (The loads are volatile so that they stay beside their use: hoisted,
// they push the warp's 80 registers over into local memory by far more than the 20 bytes that ptxas spills now.)
__device__ __forceinline__ void relu_columns(const uint32_t (&r)[32], uint32_t bias, int n0, int N, uint32_t (&pk)[16]) {
#pragma unroll
    for (int u = 0; u < 32; u += 16) {
        if (n0 + u < N) {  // N is a multiple of 16
#pragma unroll
            for (int i = u; i < u + 16; i += 4) {
                float x, y, z, w;
                asm volatile("ld.volatile.shared::cta.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(x), "=f"(y), "=f"(z), "=f"(w)
                             : "r"(bias + uint32_t(n0 + i) * 4u));
                pk[i / 2] = bias_relu_bf16(r[i], r[i + 1], x, y);
                pk[i / 2 + 1] = bias_relu_bf16(r[i + 2], r[i + 3], z, w);
            }
        } else {
#pragma unroll
            for (int i = u / 2; i < u / 2 + 8; ++i) pk[i] = 0u;
        }
    }
}

// Bounded wait; false when `limit` polls run out (the error word and the abort flag are then set) or
// when another role has aborted.
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, uint32_t abort_flag, const MlpArgs &A) {
    for (uint32_t n = uint32_t(min(A.wait_limit, (long long)kWaitLimit)); n; --n) {
        if (mbar_try_wait<false>(bar, parity)) return true;
        uint32_t gone;
        asm volatile("ld.volatile.shared::cta.u32 %0, [%1];" : "=r"(gone) : "r"(abort_flag) : "memory");
        if (gone) return false;
    }
    atomicExch(A.err, 1);
    asm volatile("st.volatile.shared::cta.u32 [%0], %1;" ::"r"(abort_flag), "r"(1) : "memory");
    return false;
}

__global__ void __launch_bounds__(kThreads, 1) mlp_kernel(const __grid_constant__ MlpArgs A) {
    extern __shared__ __align__(1024) char smem_raw[];
    // the swizzled operand tiles start on 1024-byte boundaries
    char *ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    char *stage = ring + kSmemRing;  // layer-0 input of tile t at stage + t * kStageBytes
    float *sbias = reinterpret_cast<float *>(stage + kSmemStage);
    float *head = reinterpret_cast<float *>(stage + kSmemStage + kSmemBias);
    uint64_t *bars = reinterpret_cast<uint64_t *>(stage + kSmemStage + kSmemBias + kSmemHead);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kBars);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < A.n_bias; i += kThreads) sbias[i] = A.bias[i];
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * uint32_t(i); };
    auto full_bar = [&](int s) { return bar(s); };             // the slot's block has landed
    auto empty_bar = [&](int s) { return bar(kSlots + s); };   // its last MMA has completed
    constexpr int kB = 2 * kSlots;
    auto acc_full = [&](int h) { return bar(kB + h); };        // block h holds a finished half of a hidden layer
    auto acc_free = [&](int h) { return bar(kB + 2 + h); };    // block h has been read
    auto a_ready = [&](int t) { return bar(kB + 4 + t); };     // A of tile t holds the next layer's input
    auto enc_ready = [&](int t) { return bar(kB + 6 + t); };   // the staging buffer holds the next pair's points
    auto enc_free = [&](int t) { return bar(kB + 8 + t); };    // layer 0's MMAs have read it
    // block t holds the head's outputs of tile t (a barrier per tile: with narrow layers block 1 is used by heads
    // alone, and the other tile's next head may finish before this one's outputs have been taken)
    auto head_full = [&](int t) { return bar(kB + 10 + t); };
    const uint32_t drain_bar = bar(kB + 12);
    const uint32_t abort_flag = bar(kBars) + 4u;

    if (tid == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(acc_full(i), 1);
            mbar_init(acc_free(i), kEpiWarps);
            mbar_init(a_ready(i), kEpiWarps);
            mbar_init(enc_ready(i), kAuxWarps);
            mbar_init(enc_free(i), 1);
            mbar_init(head_full(i), 1);
        }
        mbar_init(drain_bar, 1);
        tmem_slot[1] = 0u;  // the abort flag
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // Tiles go to CTAs in pairs: pair r of CTA b holds tiles (2 r + t) * grid + b. The last pair may
    // hold one.
    const long long n_points = point_count(A);
    const int n_tiles = int((n_points + kTileM - 1) / kTileM), G = int(gridDim.x), bid = int(blockIdx.x);
    auto tile_of = [&](int r, int t) { return (kPair * r + t) * G + bid; };
    auto tiles_in = [&](int r) { return tile_of(r, 1) < n_tiles ? 2 : 1; };
    const int n_pairs = n_tiles > bid ? (n_tiles - bid + kPair * G - 1) / (kPair * G) : 0;
    const int last_layer = A.n_layers - 1;
    auto wait = [&](uint32_t b, uint32_t parity) { return bounded_wait(b, parity, abort_flag, A); };
    auto aborted = [&]() { return *static_cast<volatile uint32_t *>(tmem_slot + 1) != 0u; };
    // the same for a whole warp, with a uniform result
    auto warp_wait = [&](uint32_t b, uint32_t parity) {
        if (__all_sync(0xffffffffu, mbar_try_wait<false>(b, parity))) return true;
        return __all_sync(0xffffffffu, wait(b, parity)) != 0;
    };
    auto halves = [&](const MlpLayerDev &Ly) { return (Ly.N + kHalfN - 1) / kHalfN; };

    if (warp < kEpiWarps) {
        const int q = warp & 3, g = warp >> 2;  // lane quarter, 32-column group
        const uint32_t lanes = tmem + (uint32_t(q * 32) << 16);
        uint32_t full_par = 0u;  // bit h: parity of acc_full(h) to wait for
        bool stop = false;
        for (int r = 0; r < n_pairs && !stop; ++r) {
            const int nt = tiles_in(r);
            for (int li = 0; li < last_layer && !stop; ++li) {
                const MlpLayerDev &Ly = A.L[li];
                const int N = Ly.N, n_pad = (N + kChunkK - 1) / kChunkK * kChunkK, nh = halves(Ly);
                const uint32_t bias = smem_u32(sbias + Ly.bias_off);
                for (int t = 0; t < nt; ++t) {
                    uint32_t pk[2][16];
                    bool ok = true;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h >= nh) break;
                        if (!(ok = warp_wait(acc_full(h), (full_par >> h) & 1u))) break;
                        full_par ^= 1u << h;
                        tc_fence_after();
                        const int n0 = h * kHalfN + g * 32;
                        uint32_t acc[32];
                        if (n0 < N) tmem_ld32(lanes + kAccCol + uint32_t(n0), acc);
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acc_free(h));
                        if (n0 < n_pad) relu_columns(acc, bias, n0, N, pk[h]);
                    }
                    if (!ok) {
                        stop = true;
                        break;
                    }
                    // the step's MMAs have completed (its last half has): A may be overwritten
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int n0 = h * kHalfN + g * 32;
                        if (h < nh && n0 < n_pad) tmem_st16(lanes + uint32_t(t * 128 + n0 / 2), pk[h]);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(a_ready(t));
                }
            }
        }
    } else if (warp < kAuxWarp0 + kAuxWarps) {
        const int q = warp & 3;
        float *row = head + q * kHeadFloats;  // this warp's 32 staged head rows
        constexpr int hs = kHeadCols + 1;
        const int n = A.n_out;
        const float *bias = sbias + A.L[last_layer].bias_off;
        // encode tile t of pair r (its points past the end as zeros); false when aborted
        auto encode = [&](int r, int t) {
            // pair r - 1's layer-0 MMAs have read the buffer
            if (r > 0 && !warp_wait(enc_free(t), uint32_t((r - 1) & 1))) return false;
            encode_point(A, n_points, (long long)tile_of(r, t) * kTileM + q * 32 + lane, q * 32 + lane,
                         stage + size_t(t) * kStageBytes);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(enc_ready(t));
            return true;
        };
        // the head's outputs of tile t of pair r
        auto store_head = [&](int r, int t) {
            if (!warp_wait(head_full(t), uint32_t(r & 1))) return false;
            tc_fence_after();
            const long long p0 = (long long)tile_of(r, t) * kTileM + q * 32;
            const int nv = int(n_points - p0 < 32 ? (n_points > p0 ? n_points - p0 : 0) : 32);
#pragma unroll 1
            for (int c0 = 0; c0 < n; c0 += kHeadCols) {  // 32 outputs at a time
                const int nc = min(n - c0, kHeadCols);
#pragma unroll 1
                for (int u0 = 0; u0 < nc; u0 += 16) {
                    uint32_t acc[16];
                    tmem_ld16_nowait(tmem + (uint32_t(q * 32) << 16) + kAccCol + uint32_t(t * kHalfN + c0 + u0), acc);
                    tmem_wait();
#pragma unroll
                    for (int u = 0; u < 16; ++u)
                        if (u0 + u < nc) row[lane * hs + u0 + u] = __uint_as_float(acc[u]) + bias[c0 + u0 + u];
                }
                tc_fence_before();
                __syncwarp();  // also: the warp's rows are staged
                if (c0 + nc == n && lane == 0) mbar_arrive_n(acc_free(t), kEpiWarps / kAuxWarps);
                // rows of 32 consecutive points are contiguous in the cache (or in out): a warp writes row after row,
                // lane = output c0 + lane
                auto rows = [&](auto put) {
                    if (lane < nc)
#pragma unroll 4
                        for (int i = 0; i < nv; ++i) put(i, row[i * hs + lane]);
                };
                const int c = c0 + lane;
                if (A.mode == 0) {
                    if (c0 == 0 && lane < nv) {
                        const float sg = fmaxf(row[lane * hs], 0.0f);
                        if (A.prec == FNR_PREC_FP16) static_cast<__half *>(A.sigma_out)[p0 + lane] = __float2half_rn(sg);
                        else static_cast<float *>(A.sigma_out)[p0 + lane] = sg;
                    }
                    char *rec = A.uvw_out + p0 * A.rec_stride;
                    if (A.prec == FNR_PREC_FP16)
                        rows([&](int i, float v) {
                            if (c > 0) reinterpret_cast<__half *>(rec + size_t(i) * A.rec_stride)[c - 1] = __float2half_rn(v);
                        });
                    else
                        rows([&](int i, float v) {
                            if (c > 0) reinterpret_cast<float *>(rec + size_t(i) * A.rec_stride)[c - 1] = v;
                        });
                } else if (A.mode == 1 && A.dprec == FNR_PREC_FP16) {
                    rows([&](int i, float v) { static_cast<__half *>(A.beta_out)[(p0 + i) * n + c] = __float2half_rn(v); });
                } else {
                    float *out = A.mode == 1 ? static_cast<float *>(A.beta_out) : A.out;
                    const bool relu = A.mode == 2 && A.relu0 != 0 && c == 0;
                    rows([&](int i, float v) { out[(p0 + i) * n + c] = relu ? fmaxf(v, 0.0f) : v; });
                }
                __syncwarp();  // the staged rows have been read
            }
            return true;
        };
        bool ok = true;
        for (int t = 0; ok && n_pairs > 0 && t < tiles_in(0); ++t) ok = encode(0, t);
        for (int r = 0; ok && r < n_pairs; ++r) {
            const int nt = tiles_in(r), nt_next = r + 1 < n_pairs ? tiles_in(r + 1) : 0;
            // With one layer the head is layer 0, and the second tile's waits for the first's outputs to be
            // taken; else the next pair is encoded first, long before the heads are due.
            if (last_layer == 0)
                for (int t = 0; ok && t < nt; ++t) ok = store_head(r, t);
            for (int t = 0; ok && t < nt_next; ++t) ok = encode(r + 1, t);
            if (last_layer != 0)
                for (int t = 0; ok && t < nt; ++t) ok = store_head(r, t);
        }
    } else if (warp == kProducerWarp) {
        if (lane == 0) {
            long long it = 0, last = -1;  // index of the next block, of the last one copied
            int slot = 0;
            uint32_t round = 0u;          // of the ring, for the next block
            for (int r = 0; r < n_pairs && !aborted(); ++r)
                for (int li = 0; li < A.n_layers && !aborted(); ++li) {  // once for both tiles
                    const MlpLayerDev &Ly = A.L[li];
                    const int nc = n_chunks(Ly.K), nh = halves(Ly);
                    bool ok = true;
                    for (int h = 0; h < nh && ok; ++h) {
                        const uint32_t bytes = uint32_t(min(Ly.N - h * kHalfN, kHalfN)) * uint32_t(kChunkK) * 2u;
                        for (int c = 0; c < nc; c += 2, ++it) {
                            if (round > 0u && !(ok = wait(empty_bar(slot), (round - 1u) & 1u))) break;
                            if (it != A.withhold) {  // test fault: that block never arrives
                                const int parts = min(nc - c, 2);
                                mbar_expect_tx(full_bar(slot), bytes * uint32_t(parts));
                                for (int p = 0; p < parts; ++p)
                                    bulk_g2s(smem_u32(ring) + uint32_t(slot) * kSlotBytes + uint32_t(p) * kPartBytes,
                                             reinterpret_cast<const char *>(Ly.w) +
                                                 (size_t(c + p) * Ly.N + size_t(h) * kHalfN) * kChunkK * 2,
                                             bytes, full_bar(slot));
                                last = it;
                            }
                            if (++slot == kSlots) {
                                slot = 0;
                                ++round;
                            }
                        }
                    }
                }
            // Every copy issued has landed before the CTA's shared memory goes away (after an abort
            // some may not have been waited for): the last kSlots copies, one per slot; earlier ones were
            // consumed before their slot was reused.
            for (long long j = last >= kSlots ? last - kSlots + 1 : 0; j <= last; ++j)
                if (j != A.withhold) mbar_drain<false>(full_bar(int(j % kSlots)), uint32_t((j / kSlots) & 1), A.err);
        }
    } else {
        // The MMA issuer: the whole warp runs the loop, one elected lane issues. An N = 128 MMA takes 64 cycles,
        // so the issue of a block's eight, its wait and its commits have to fit into 512 (a single divergent lane
        // needed 100 to 190 cycles for each MMA: 512^3 in 247 ms).
        const uint32_t one = elect_one();
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t ring_lo = desc_lo(smem_u32(ring)), stage_lo = desc_lo(smem_u32(stage));
        int slot0 = 0;            // slot and ring round of the layer's first block
        uint32_t round0 = 0u;
        // bit h / t: parity of acc_free(h) to wait for (the first wait, on its phase before the first, passes at
        // once), and of a_ready(t)
        uint32_t free_par = 3u, a_par = 0u;
        int N = A.L[0].N, nc = n_chunks(A.L[0].K);
        bool ok = true;
        for (int r = 0; r < n_pairs && ok; ++r) {
            const int nt = tiles_in(r);
            for (int li = 0; li < A.n_layers && ok; ++li) {
                const int nh = (N + kHalfN - 1) / kHalfN;
                const bool is_head = li == last_layer;
                const int next = is_head ? 0 : li + 1, next_N = A.L[next].N, next_nc = n_chunks(A.L[next].K);
                int slot = slot0;
                uint32_t round = round0;
                for (int t = 0; t < nt && ok; ++t) {
                    slot = slot0;
                    round = round0;
                    for (int h = 0; h < nh && ok; ++h) {
                        // what this half waits for, polled together: its accumulator block, with the first half the
                        // layer's input, and with the layer's first tile the weight block
                        const int blk = is_head ? t : h;  // the two heads do not wait for one another
                        const uint32_t b_free = acc_free(blk), p_free = (free_par >> blk) & 1u;
                        const uint32_t b_in = li == 0 ? enc_ready(t) : a_ready(t);
                        const uint32_t p_in = li == 0 ? uint32_t(r & 1) : (a_par >> t) & 1u;
                        bool there = mbar_test(b_free, p_free);
                        if (h == 0) there = mbar_test(b_in, p_in) && there;
                        if (t == 0) there = mbar_test(full_bar(slot), round & 1u) && there;
                        if (!__all_sync(0xffffffffu, there))
                            ok = warp_wait(b_free, p_free) && (h > 0 || warp_wait(b_in, p_in)) &&
                                 (t > 0 || warp_wait(full_bar(slot), round & 1u));
                        if (!ok) break;
                        free_par ^= 1u << blk;
                        if (h == 0 && li > 0) a_par ^= 1u << t;
                        tc_fence_after();
                        const uint32_t idesc = instr_desc(kTileM, min(N - h * kHalfN, kHalfN));
                        const uint32_t d = tm + kAccCol + uint32_t(blk * kHalfN);
                        auto next_slot = [&]() {
                            if (t == nt - 1) umma_commit(one, empty_bar(slot));  // its last use: it may be refilled
                            if (++slot == kSlots) {
                                slot = 0;
                                ++round;
                            }
                        };
                        // one weight block: parts [0, n_parts) of 64 inputs from chunk c on
                        auto block = [&](int c, int n_parts) {
                            const uint32_t b_lo = ring_lo + uint32_t(slot) * (kSlotBytes >> 4);
                            const uint32_t a = tm + uint32_t(t * 128 + c * (kChunkK / 2));
#pragma unroll
                            for (int s = 0; s < 4; ++s)
                                umma_ts(one, d, a + 8 * s, desc_sw128(b_lo + 2 * s), idesc, (c > 0 || s > 0) ? 1u : 0u);
                            if (n_parts > 1) {
#pragma unroll
                                for (int s = 0; s < 4; ++s)
                                    umma_ts(one, d, a + 32 + 8 * s, desc_sw128(b_lo + (kPartBytes >> 4) + 2 * s), idesc, 1u);
                            }
                            next_slot();
                        };
                        auto next_block = [&]() {  // the block after the first has landed
                            if (t > 0) return true;
                            if (!warp_wait(full_bar(slot), round & 1u)) return false;
                            tc_fence_after();
                            return true;
                        };
                        if (li == 0) {
                            const uint32_t b_lo = ring_lo + uint32_t(slot) * (kSlotBytes >> 4);
                            const uint32_t a_lo = stage_lo + uint32_t(t) * uint32_t(kStageBytes >> 4);
#pragma unroll
                            for (int s = 0; s < 4; ++s)
                                umma_ss(one, d, desc_sw128(a_lo + 2 * s), desc_sw128(b_lo + 2 * s), idesc, s > 0 ? 1u : 0u);
                            next_slot();
                            if (h == nh - 1) umma_commit(one, enc_free(t));  // the staging buffer may be refilled
                        } else if (nc == 4) {
                            block(0, 2);
                            if (!(ok = next_block())) break;
                            block(2, 2);
                        } else {
                            for (int c = 0; c < nc && ok; c += 2)
                                if (c == 0 || (ok = next_block())) block(c, nc - c);
                            if (!ok) break;
                        }
                        umma_commit(one, is_head ? head_full(t) : acc_full(h));
                    }
                }
                slot0 = slot;
                round0 = round;
                N = next_N;
                nc = next_nc;
            }
        }
        // every tensor-core operation issued (and every commit before this one) has completed before the
        // tensor memory is freed and the CTA leaves
        umma_commit(one, drain_bar);
        if (one) mbar_drain<false>(drain_bar, 0u, A.err);
        __syncwarp();
    }
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// All layers' weights and biases, blockIdx.y = layer. W [N][K] row-major bf16
// bits -> padded, chunk-major 128-byte swizzled layout: chunk c holds columns
// [64 c, 64 c + 64) as [Np][64] K-major rows of 128 bytes, 8-row atoms of 1024
// bytes, piece (k / 8) of row n at (k / 8) ^ (n & 7); so rows [128 h, 128 h + 128)
// of a chunk are contiguous. Rows past the layer's N and columns past its K are 0.
struct PrepArgs {
    const uint16_t *w[kMaxLayers];
    const float *b[kMaxLayers];
    uint16_t *w_out[kMaxLayers];
    float *b_out[kMaxLayers];
    int N[kMaxLayers], K[kMaxLayers], Np[kMaxLayers], Kp[kMaxLayers];
};

__global__ void prepare_kernel(const __grid_constant__ PrepArgs P) {
    const int li = blockIdx.y, N = P.N[li], K = P.K[li], Np = P.Np[li], Kp = P.Kp[li];
    const int total = Np * Kp;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int n = e / Kp, k = e - n * Kp;
        const uint16_t v = (n < N && k < K) ? P.w[li][size_t(n) * K + k] : uint16_t(0);
        const int c = k / kChunkK, kk = k - c * kChunkK;
        const size_t off = size_t(c) * Np * kChunkK + size_t(n >> 3) * 512 + size_t(n & 7) * 64 +
                           size_t(((kk >> 3) ^ (n & 7)) & 7) * 8 + (kk & 7);
        P.w_out[li][off] = v;
        if (e < Np) P.b_out[li][e] = e < N ? P.b[li][e] : 0.0f;
    }
}

int round16(int v) { return (v + 15) / 16 * 16; }
int round64(int v) { return (v + 63) / 64 * 64; }

}  // namespace

fnr_status launch_mlp_single(const MlpArgs &A, int num_sms, cudaStream_t s) {
    cudaError_t e;
    // tile indices, one pair per CTA past the end included, are int
    if (A.n_points > (1LL << 37)) return fail(FNR_ERR_UNSUPPORTED, "MLP kernel: %lld points", A.n_points);
    const int tiles = int((A.n_points + kTileM - 1) / kTileM);
    if ((e = cudaFuncSetAttribute(mlp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes))) !=
        cudaSuccess)
        return cuda_fail(e, "MLP smem attribute");
    mlp_kernel<<<unsigned(tiles < num_sms ? tiles : num_sms), kThreads, kSmemBytes, s>>>(A);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "MLP launch");
    return FNR_OK;
}

// Validate one MLP description; n_out_min is the number of outputs needed.
fnr_status check_mlp(const fnr_mlp *m, int n_out_min, const char *name) {
    if (!m) return fail(FNR_ERR_INVALID_ARG, "%s is NULL", name);
    if (m->n_layers < 1 || m->n_layers > kMaxLayers)
        return fail(FNR_ERR_INVALID_ARG, "%s: n_layers %d outside [1, %d]", name, m->n_layers, kMaxLayers);
    if (m->pe_in != 3) return fail(FNR_ERR_UNSUPPORTED, "%s: pe_in must be 3", name);
    if (m->pe_freqs < 1 || 6 * m->pe_freqs > m->dims[0])
        return fail(FNR_ERR_INVALID_ARG, "%s: dims[0]=%d cannot hold 2*3*%d encoded inputs", name, m->dims[0],
                    m->pe_freqs);
    if (m->dims[0] > kMaxK0)
        return fail(FNR_ERR_UNSUPPORTED, "%s: encoded width dims[0]=%d above %d", name, m->dims[0], kMaxK0);
    for (int i = 0; i <= m->n_layers; ++i)
        if (m->dims[i] < 1 || round64(m->dims[i]) > kMaxK)
            return fail(FNR_ERR_UNSUPPORTED, "%s: layer width %d outside [1, %d]", name, m->dims[i], kMaxK);
    if (m->dims[m->n_layers] < n_out_min)
        return fail(FNR_ERR_INVALID_ARG, "%s: %d outputs, need %d", name, m->dims[m->n_layers], n_out_min);
    for (int i = 0; i < m->n_layers; ++i)
        if (!m->weights[i] || !m->biases[i]) return fail(FNR_ERR_INVALID_ARG, "%s: NULL layer %d", name, i);
    return FNR_OK;
}

namespace {

// Device copies of one network's weights and biases, and the error word of its launches.
struct MlpBuffers {
    TempBuf weights, biases, err;
    int num_sms = 0;
};

// Lay out the weights and biases of m and fill the layer table of A (A.mode and its outputs per point are set).
fnr_status mlp_prepare(const fnr_context *ctx, const fnr_mlp *m, MlpArgs &A, MlpBuffers &B, cudaStream_t s) {
    B.num_sms = ctx->num_sms;
    size_t welems = 0, belems = 0;
    for (int i = 0; i < m->n_layers; ++i) {
        welems += size_t(round16(m->dims[i + 1])) * round64(m->dims[i]);
        belems += size_t(round16(m->dims[i + 1]));
    }
    cudaError_t e;
    if ((e = B.weights.alloc(ctx, welems * 2, s)) != cudaSuccess) return cuda_fail(e, "MLP weights");
    if ((e = B.biases.alloc(ctx, belems * 4, s)) != cudaSuccess) return cuda_fail(e, "MLP biases");
    if ((e = B.err.alloc(ctx, 4, s)) != cudaSuccess) return cuda_fail(e, "MLP error word");
    if ((e = cudaMemsetAsync(B.err.p, 0, 4, s)) != cudaSuccess) return cuda_fail(e, "memset");
    A.n_out = A.mode == 0 ? 1 + 3 * A.D : (A.mode == 1 ? A.D : A.out_stride);
    if (A.n_out < 1 || A.n_out > kMaxOut || A.n_out > m->dims[m->n_layers])
        return fail(FNR_ERR_UNSUPPORTED, "MLP kernel: %d outputs per point (at most %d)", A.n_out, kMaxOut);
    A.head_stride = round16(A.n_out) + 4;
    size_t wo = 0, bo = 0;
    PrepArgs P;
    int max_elems = 0;
    for (int i = 0; i < m->n_layers; ++i) {
        // the head is evaluated up to the outputs that are stored
        const int K = m->dims[i], N = i + 1 == m->n_layers ? A.n_out : m->dims[i + 1], Kp = round64(K), Np = round16(N);
        uint16_t *wd = static_cast<uint16_t *>(B.weights.p) + wo;
        P.w[i] = m->weights[i];
        P.b[i] = m->biases[i];
        P.w_out[i] = wd;
        P.b_out[i] = static_cast<float *>(B.biases.p) + bo;
        P.N[i] = N;
        P.K[i] = K;
        P.Np[i] = Np;
        P.Kp[i] = Kp;
        if (Np * Kp > max_elems) max_elems = Np * Kp;
        A.L[i].w = reinterpret_cast<const __nv_bfloat16 *>(wd);
        A.L[i].bias_off = int(bo);
        A.L[i].K = Kp;
        A.L[i].N = Np;
        wo += size_t(Np) * Kp;
        bo += size_t(Np);
    }
    prepare_kernel<<<dim3(unsigned((max_elems + 255) / 256), unsigned(m->n_layers)), 256, 0, s>>>(P);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "MLP weight layout");
    A.bias = static_cast<const float *>(B.biases.p);
    A.n_bias = int(bo);
    A.n_layers = m->n_layers;
    A.pe_freqs = m->pe_freqs;
    A.err = static_cast<int *>(B.err.p);
    A.wait_limit = kWaitLimit;
    A.withhold = -1;
    take_mlp_fault(&A.wait_limit, &A.withhold);
    return FNR_OK;
}

// One launch over the points already in A.
fnr_status mlp_launch(const MlpArgs &A, int num_sms, cudaStream_t s) {
    if (A.n_points <= 0) return FNR_OK;
    return mlp_cta_pair() ? launch_mlp_pair(A, num_sms, s) : launch_mlp_single(A, num_sms, s);
}

// Wait for the launches on A and report their error word.
fnr_status mlp_finish(const MlpArgs &A, cudaStream_t s) {
    int herr = 0;
    cudaError_t e;
    if ((e = cudaMemcpyAsync(&herr, A.err, 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return cuda_fail(e, "MLP sync");
    if (herr == 1) return fail(FNR_ERR_DEVICE, "MLP kernel: an mbarrier wait ran out");
    if (herr) return fail(FNR_ERR_DEVICE, "MLP kernel: work in flight did not drain at exit");
    return FNR_OK;
}

}  // namespace

struct GridMlp::Impl {
    MlpArgs A;
    MlpBuffers B;
};

GridMlp::~GridMlp() { delete impl; }

fnr_status GridMlp::launch(const fnr_context *ctx, const fnr_mlp *m, int mode, const fnr_cache_desc &d,
                           const CacheView &v, cudaStream_t s) {
    impl = new Impl();
    MlpArgs &A = impl->A;
    memset(&A, 0, sizeof(A));
    A.mode = mode;
    A.k = d.k;
    A.l = d.l;
    for (int a = 0; a < 3; ++a) {
        A.bmin[a] = d.bmin[a];
        A.h[a] = static_cast<float>((static_cast<double>(d.bmax[a]) - d.bmin[a]) / d.k);
    }
    A.n_points = mode == 0 ? (long long)d.k * d.k * d.k : (long long)d.l * d.l;
    A.sigma_out = const_cast<void *>(v.sigma);
    A.uvw_out = const_cast<char *>(v.uvw);
    A.rec_stride = v.rec_stride;
    A.prec = d.pos_precision;
    A.D = d.D;
    A.beta_out = const_cast<void *>(v.beta);
    A.dprec = d.dir_precision;
    const fnr_status st = mlp_prepare(ctx, m, A, impl->B, s);
    return st == FNR_OK ? mlp_launch(A, impl->B.num_sms, s) : st;
}

fnr_status GridMlp::finish(cudaStream_t s) { return mlp_finish(impl->A, s); }

struct PointsMlp::Impl {
    MlpArgs A;
    MlpBuffers B;
};

PointsMlp::~PointsMlp() { delete impl; }

fnr_status PointsMlp::prepare(const fnr_context *ctx, const fnr_mlp *m, int out_stride, bool relu0, cudaStream_t s) {
    impl = new Impl();
    memset(&impl->A, 0, sizeof(impl->A));
    impl->A.mode = 2;
    impl->A.out_stride = out_stride;
    impl->A.relu0 = relu0 ? 1 : 0;
    return mlp_prepare(ctx, m, impl->A, impl->B, s);
}

fnr_status PointsMlp::launch(const float *points, long long max_n, const unsigned long long *n_dev, float *out,
                             cudaStream_t s) {
    MlpArgs A = impl->A;
    A.n_points = max_n;
    A.n_dev = n_dev;
    A.points = points;
    A.out = out;
    return mlp_launch(A, impl->B.num_sms, s);
}

const int *PointsMlp::error_word() const { return impl->A.err; }

fnr_status PointsMlp::finish(cudaStream_t s) { return mlp_finish(impl->A, s); }

}  // namespace fnr
