// mlp_pair.cu -- the CTA-pair form of the tensor-core MLP kernel (the default
// form and what the kernel computes: mlp.cu): a cluster of two CTAs on an SM pair
// walks tiles of 256 points, 128 per CTA; rank 0 issues M = 256 MMAs for both
// (tcgen05.mma.cta_group::2), which read each CTA's A rows and each CTA's half of
// the weight chunk from that CTA's own shared memory and accumulate into each
// CTA's own tensor memory, so each SM streams half of every chunk. Both forms
// compute every product in the same order, so their outputs are equal bit for
// bit. This form keeps the activations in shared memory and pays hand-offs
// between the two SMs; it measured slower and is chosen only through the test
// hook fnr_testing_mlp_cta_pair. Warp roles, in every CTA:
//   producer (warp 0): streams this CTA's half of each 64-column weight chunk
//     through a ring of 4 slots of 16 KB -- a whole layer -- by bulk async copy,
//     loaded once per layer for both tiles in flight;
//   two tiles are in flight: each has its own A tile (same swizzled layout)
//     and its own tensor-memory accumulator, so one tile's epilogue runs while
//     the other's MMAs do;
//   encoders (warps 2-3): encode each tile's points (gamma(x) = sin / cos(2^j
//     pi x), rounded to bf16) into the tile's layer-0 staging buffer one tile
//     pair ahead, as soon as the MMAs that read the buffer's previous contents
//     have completed, so encoding never waits between tiles;
//   MMA issuer (warp 1, one lane; in rank 0): waits for the layer
//     input and each chunk, issues tcgen05.mma (K=16 steps, bf16 x bf16 -> fp32
//     in tensor memory; layer 0 reads the staging buffer), releases each slot
//     with tcgen05.commit on its "empty" mbarrier and signals the finished
//     accumulator with one more commit; in rank 1 the same lane tells
//     rank 0 when each chunk half has landed;
//   epilogue (warps 4-19, four per 32-lane quarter of tensor memory): per
//     hidden layer read the accumulator (tcgen05.ld), add the bias, apply
//     ReLU, round to bf16 and write the next layer's A tile; after the head,
//     stage the outputs in the (now free) A tile as fp32 rows and write the
//     tile's sigma = ReLU(out_0), (u, v, w) = out_1..3D (F_pos) or beta =
//     out_0..D-1 (F_dir) -- contiguous ranges of the cache -- with coalesced
//     stores by all sixteen warps.
// Rank 0 issues each tcgen05.commit twice, on its own copy of the barrier and,
// through the barrier's cluster address, on rank 1's; rank 1's threads arrive on
// rank 0's barriers with remote mbarrier arrives. The next layer's weights load
// while the epilogue runs. Every mbarrier wait is bounded; a wait that runs out
// sets the error word and the abort flags of both CTAs, every role leaves its
// loop, each producer waits (bounded) for the copies it has in flight, rank 0's
// MMA issuer for its tensor-core operations and rank 1 for the same commit, and
// the tensor memory is freed.
#include "mlp_common.cuh"

namespace fnr {

fnr_status fail(fnr_status st, const char *fmt, ...);
fnr_status cuda_fail(cudaError_t e, const char *what);

namespace {

using namespace mlp;

// epilogue warp w reads tensor-memory lanes 32 (w % 4) .. 32 (w % 4) + 31
constexpr int kProducerWarp = 0, kMmaWarp = 1, kEncWarp0 = 2, kEncWarps = 2;
constexpr int kFirstEpiWarp = 4, kEpiWarps = 16;
constexpr int kThreads = (kFirstEpiWarp + kEpiWarps) * 32;
constexpr uint32_t kTmemCols = 256 * kPair;                   // one accumulator per tile
constexpr size_t kSmemA = size_t(kPair) * kTileM * kMaxK * 2;  // 64 KB activations per tile
constexpr size_t kSmemStage = size_t(kPair) * kStageBytes;
constexpr int kCtas = 2;
constexpr int kSuperM = kTileM * kCtas;                        // points per MMA tile
constexpr int kSlots = 2 * kCtas;                              // ring slots: a layer's chunk halves
constexpr int kSlotBytes = kMaxN / kCtas * kChunkK * 2;        // this CTA's rows of one weight chunk
constexpr size_t kSmemRing = size_t(kSlots) * kSlotBytes;
// full, empty, pair_full; per tile slot acc_full, a_ready, enc_ready, enc_free, head_ready; drain
constexpr int kBars = 3 * kSlots + 5 * kPair + 1;
constexpr size_t kSmemBars = (size_t(kBars) * 8 + 16 + 127) / 128 * 128;
constexpr size_t kSmemBytes = kSmemA + kSmemStage + kSmemRing + kSmemBars + 1024;  // + alignment slack
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
static_assert(kMaxK / kChunkK <= kSlots, "a layer's chunks fit the ring");
static_assert(size_t(kTileM) * (kMaxHeadOut + 4) * 4 <= size_t(kTileM) * kMaxK * 2, "head staging fits an A tile");

// The same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}

// Arrive on an mbarrier of the other CTA of the pair (address from cluster_addr).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::
            "r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive on the mbarrier at shared::cluster address `bar` when every tcgen05
// operation this thread has issued so far has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Tensor-memory allocation of `cols` columns by one whole warp (in both CTAs of a pair,
// together), its address written to shared memory at `slot`; and its release.
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1) mlp_pair_kernel(const __grid_constant__ MlpArgs A) {
    extern __shared__ __align__(1024) char smem_raw[];
    // the swizzled operand tiles start on 1024-byte boundaries
    char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    char *sa = smem;                 // A tile of slot t at sa + t * kTileM * kMaxK * 2
    char *stage = smem + kSmemA;     // layer-0 input of slot t at stage + t * kStageBytes
    char *ring = stage + kSmemStage;
    uint64_t *bars = reinterpret_cast<uint64_t *>(ring + kSmemRing);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kBars);
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Rank in the CTA pair: rank 0 issues the MMAs for both; every shared-memory
    // layout below is the same in both CTAs, so an address names the same
    // object in either.
    uint32_t rank = 0;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const bool leader = rank == 0;
    // bars: [0, kSlots) full, [kSlots, 2 kSlots) empty, [2 kSlots, 3 kSlots) pair_full, then per tile slot:
    // acc_full, a_ready, enc_ready, enc_free, head_ready
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * uint32_t(s); };
    auto empty_bar = [&](int s) { return bar0 + 8u * uint32_t(kSlots + s); };
    // pair_full(s) (rank 0): the other CTA's part of the chunk in slot s has landed
    auto pair_full = [&](int s) { return bar0 + 8u * uint32_t(2 * kSlots + s); };
    auto tile_bar = [&](int which, int t) { return bar0 + 8u * uint32_t(3 * kSlots + which * kPair + t); };
    // acc_full(t): the tile's accumulator holds a finished layer (one tcgen05.commit; rank 1: one relayed arrive)
    auto acc_full = [&](int t) { return tile_bar(0, t); };
    // a_ready(t) (rank 0): the accumulators have been read and the next layer's A tiles written (every epilogue
    // warp of both CTAs)
    auto a_ready = [&](int t) { return tile_bar(1, t); };
    // enc_ready(t) (rank 0): the staging buffers hold the encoded points of the tile's next pair (the encoder
    // warps of both CTAs)
    auto enc_ready = [&](int t) { return tile_bar(2, t); };
    // enc_free(t): the layer-0 MMAs that read the staging buffers have completed (commit; rank 1: relayed)
    auto enc_free = [&](int t) { return tile_bar(3, t); };
    // head_ready(t): every epilogue warp of this CTA has staged its head outputs
    auto head_ready = [&](int t) { return tile_bar(4, t); };
    // drain: every tensor-core operation of the pair has completed (commit; rank 1: relayed)
    const uint32_t drain_bar = bar0 + 8u * uint32_t(3 * kSlots + 5 * kPair);
    constexpr uint32_t kATileBytes = uint32_t(kTileM) * kMaxK * 2;
    // the same barrier in the other CTA of the pair, and arrivals that go to rank 0's copy
    auto other = [&](uint32_t bar) { return cluster_addr(bar, rank ^ 1u); };
    auto arrive_at_leader = [&](uint32_t bar) {
        if (leader) mbar_arrive(bar);
        else mbar_arrive_remote(other(bar));
    };
    const uint32_t peer_abort =
        cluster_addr(smem_u32(const_cast<int *>(&abort_flag)), rank ^ 1u);

    if (tid == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
            mbar_init(pair_full(s), 1);
        }
        for (int t = 0; t < kPair; ++t) {
            mbar_init(acc_full(t), 1);
            mbar_init(a_ready(t), kEpiWarps * kCtas);
            mbar_init(enc_ready(t), kEncWarps * kCtas);
            mbar_init(enc_free(t), 1);
            mbar_init(head_ready(t), kEpiWarps);
        }
        mbar_init(drain_bar, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), kTmemCols);  // both CTAs of a pair together
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // both CTAs' barriers are initialised before any remote arrive
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // MMA tiles of kSuperM points go to CTAs (pairs) in groups of kPair: group r holds tiles
    // (kPair r + t) * grid + bid, t < kPair; a tile past the end is carried as an empty one (no outputs).
    // CTA `rank` of a pair holds rows [rank kTileM, rank kTileM + kTileM) of each tile.
    const long long n_points = point_count(A), n_tiles = (n_points + kSuperM - 1) / kSuperM;
    const long long G = gridDim.x / kCtas;
    const long long bid = blockIdx.x / kCtas;
    auto pair_tile = [&](long long r, int t) { return (kPair * r + t) * G + bid; };
    const long long n_pairs = n_tiles > bid ? (n_tiles - bid + kPair * G - 1) / (kPair * G) : 0;
    // bounded waits: hand-offs between the CTAs of a pair (cluster scope), and completions
    // of copies and tensor-core work (CTA scope)
    auto wait = [&](uint32_t bar, uint32_t parity) {
        return mbar_wait<true>(bar, parity, A.err, &abort_flag, A.wait_limit, peer_abort);
    };
    auto wait_done = [&](uint32_t bar, uint32_t parity) {
        return mbar_wait<false>(bar, parity, A.err, &abort_flag, A.wait_limit, peer_abort);
    };
    // a warp-wide bounded wait on a completion or a hand-off within the CTA (lane 0 polls); false
    // when it ran out or another role aborted
    auto warp_wait = [&](uint32_t bar, uint32_t parity) {
        int ok = 1;
        if (lane == 0) ok = wait_done(bar, parity) ? 1 : 0;
        return __shfl_sync(0xffffffffu, ok, 0) != 0;
    };

    if (warp == kProducerWarp) {
        if (lane == 0) {
            long long it = 0, last = -1;  // last: index of the last chunk copied
            for (long long r = 0; r < n_pairs && !abort_flag; ++r)
                for (int li = 0; li < A.n_layers && !abort_flag; ++li)
                    {  // once for both tiles
                        const MlpLayerDev &Ly = A.L[li];
                        const int nc = n_chunks(Ly.K);
                        // this CTA's rows of each chunk: [rank N / kCtas, (rank + 1) N / kCtas), whole 8-row atoms
                        const uint32_t bytes = uint32_t(Ly.N / kCtas) * uint32_t(kChunkK) * 2u;
                        for (int c = 0; c < nc; ++c, ++it) {
                            const int slot = int(it % kSlots);
                            const long long round = it / kSlots;
                            if (round > 0 && !wait_done(empty_bar(slot), uint32_t((round - 1) & 1))) break;
                            if (it == A.withhold) continue;  // test fault: this chunk never arrives
                            mbar_expect_tx(full_bar(slot), bytes);
                            const char *src = reinterpret_cast<const char *>(Ly.w) + size_t(c) * Ly.N * kChunkK * 2 +
                                              size_t(rank) * bytes;
                            bulk_g2s(smem_u32(ring) + uint32_t(slot) * kSlotBytes, src, bytes, full_bar(slot));
                            last = it;
                        }
                    }
            // Every copy issued has landed before the CTA's shared memory goes away
            // (after an abort some may not have been waited for): the last kSlots
            // copies, one per slot; earlier ones were consumed before their slot was reused.
            for (long long j = last >= kSlots ? last - kSlots + 1 : 0; j <= last; ++j)
                if (j != A.withhold) mbar_drain<true>(full_bar(int(j % kSlots)), uint32_t((j / kSlots) & 1), A.err);
        }
    } else if (warp == kMmaWarp) {
        if (lane == 0 && leader) {
            long long it = 0, uses = 0;  // uses: (layer, tile) steps per slot t, same count for both
            for (long long r = 0; r < n_pairs && !abort_flag; ++r)
                for (int li = 0; li < A.n_layers && !abort_flag; ++li, ++uses)
                    for (int t = 0; t < kPair && !abort_flag; ++t) {
                        const MlpLayerDev &Ly = A.L[li];
                        if (t > 0) it -= n_chunks(Ly.K);  // the layer's chunks again, still in the ring
                        if (li == 0 && !wait(enc_ready(t), uint32_t(r & 1))) break;
                        if (!wait(a_ready(t), uint32_t(uses & 1))) break;
                        tc_fence_after();
                        const uint32_t idesc = instr_desc(kSuperM, Ly.N);
                        const uint32_t a_base =
                            li == 0 ? smem_u32(stage) + uint32_t(t) * uint32_t(kStageBytes)
                                    : smem_u32(sa) + uint32_t(t) * kATileBytes;
                        const uint32_t d_tmem = tmem + uint32_t(t * 256);
                        const int nc = n_chunks(Ly.K);
                        for (int c = 0; c < nc; ++c, ++it) {
                            const int slot = int(it % kSlots);
                            const uint32_t par = uint32_t((it / kSlots) & 1);
                            const bool first = t == 0;  // the chunk's first use: wait for it to land
                            if (first && !wait_done(full_bar(slot), par)) break;
                            if (first && !wait_done(pair_full(slot), par)) break;
                            tc_fence_after();
#pragma unroll
                            for (int s = 0; s < kChunkK / 16; ++s) {
                                const uint64_t ad = smem_desc_sw128(a_base + uint32_t(c) * (kTileM / 8) * 1024u +
                                                                    uint32_t(s) * 32u);
                                const uint64_t bd =
                                    smem_desc_sw128(smem_u32(ring) + uint32_t(slot) * kSlotBytes + uint32_t(s) * 32u);
                                umma_bf16(d_tmem, ad, bd, idesc, (c > 0 || s > 0) ? 1u : 0u);
                            }
                            if (t == kPair - 1) {  // its last use: the slot may be refilled
                                umma_commit(empty_bar(slot));
                                umma_commit(other(empty_bar(slot)));
                            }
                        }
                        if (abort_flag) break;
                        if (li == 0) {  // the staging buffers may be refilled
                            umma_commit(enc_free(t));
                            umma_commit(other(enc_free(t)));
                        }
                        umma_commit(acc_full(t));
                        umma_commit(other(acc_full(t)));
                    }
            // every tensor-core operation issued (and every commit before this one) has
            // completed before the tensor memory is freed and the CTAs leave
            umma_commit(drain_bar);
            umma_commit(other(drain_bar));
            mbar_drain<true>(drain_bar, 0u, A.err);
        } else if (lane == 0) {
            // rank 1: tell rank 0 when each of this CTA's chunk parts has landed, in chunk order
            long long it = 0;
            for (long long r = 0; r < n_pairs && !abort_flag; ++r)
                for (int li = 0; li < A.n_layers && !abort_flag; ++li)
                    {
                        const int nc = n_chunks(A.L[li].K);
                        for (int c = 0; c < nc; ++c, ++it) {
                            const int slot = int(it % kSlots);
                            if (!wait_done(full_bar(slot), uint32_t((it / kSlots) & 1))) break;
                            mbar_arrive_remote(other(pair_full(slot)));
                        }
                    }
            // rank 0's MMAs read this CTA's shared memory and write its tensor memory:
            // they have completed before either is released
            mbar_drain<true>(drain_bar, 0u, A.err);
        }
    } else if (warp >= kEncWarp0 && warp < kEncWarp0 + kEncWarps) {
        // encoders: rows (warp - kEncWarp0) * 32 + lane + 32 kEncWarps i of this CTA's part of each tile
        const int e = warp - kEncWarp0;
        for (long long r = 0; r < n_pairs && !abort_flag; ++r) {
            bool ok = true;
            for (int t = 0; t < kPair && ok; ++t) {
                // pair r - 1's layer-0 MMAs of this slot have read the buffers
                if (r > 0 && !(ok = warp_wait(enc_free(t), uint32_t((r - 1) & 1)))) break;
                const long long tile = pair_tile(r, t);
                char *st = stage + size_t(t) * kStageBytes;
                for (int row = e * 32 + lane; row < kTileM; row += 32 * kEncWarps) {
                    const long long p =
                        tile < n_tiles ? tile * kSuperM + rank * kTileM + row : n_points;  // past the end: zeros
                    encode_point(A, n_points, p, row, st);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) arrive_at_leader(enc_ready(t));
            }
            if (!ok) break;
        }
    } else if (warp >= kFirstEpiWarp) {
        const int q = warp & 3, g = (warp - kFirstEpiWarp) >> 2;  // lane quarter, column group
        const int row = q * 32 + lane;
        const int te = (warp - kFirstEpiWarp) * 32 + lane;       // 0 .. 32 kEpiWarps - 1
        long long uses = 0;
        bool stop = false;
        // the accumulators are free for the first pair's layer 0
        if (n_pairs > 0)
            for (int t = 0; t < kPair; ++t) {
                __syncwarp();
                if (lane == 0) arrive_at_leader(a_ready(t));
            }
        for (long long r = 0; r < n_pairs && !stop; ++r) {
            for (int li = 0; li < A.n_layers && !stop; ++li, ++uses) {
                const MlpLayerDev &Ly = A.L[li];
                const int N = Ly.N;
                const bool last = li + 1 == A.n_layers;
                const float *bias = A.bias + Ly.bias_off;
                for (int t = 0; t < kPair; ++t) {
                    if (!warp_wait(acc_full(t), uint32_t(uses & 1))) {
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    char *sa_t = sa + size_t(t) * kATileBytes;
                    const uint32_t trow = tmem + uint32_t(t * 256) + (uint32_t(q * 32) << 16);
                    if (!last) {
                        // this warp's 16-column chunks j = g, g+4, g+8, g+12, two loads in flight per wait
                        const int nj = N / 16;
                        auto process = [&](const uint32_t (&rr)[16], int j) {
                            const int c0 = j * 16;
#pragma unroll
                            for (int u = 0; u < 16; u += 8) {
                                const float4 b0 = __ldg(reinterpret_cast<const float4 *>(bias + c0 + u));
                                const float4 b1 = __ldg(reinterpret_cast<const float4 *>(bias + c0 + u + 4));
                                uint4 pk;
                                pk.x = pack_relu_bf16(__uint_as_float(rr[u + 0]) + b0.x, __uint_as_float(rr[u + 1]) + b0.y);
                                pk.y = pack_relu_bf16(__uint_as_float(rr[u + 2]) + b0.z, __uint_as_float(rr[u + 3]) + b0.w);
                                pk.z = pack_relu_bf16(__uint_as_float(rr[u + 4]) + b1.x, __uint_as_float(rr[u + 5]) + b1.y);
                                pk.w = pack_relu_bf16(__uint_as_float(rr[u + 6]) + b1.z, __uint_as_float(rr[u + 7]) + b1.w);
                                *reinterpret_cast<uint4 *>(sa_t + a_offset(row, c0 + u)) = pk;
                            }
                        };
                        for (int j0 = g; j0 < nj; j0 += 8) {  // warp-uniform
                            uint32_t r0[16], r1[16];
                            const bool two = j0 + 4 < nj;
                            tmem_ld16_nowait(trow + uint32_t(j0 * 16), r0);
                            if (two) tmem_ld16_nowait(trow + uint32_t((j0 + 4) * 16), r1);
                            tmem_wait();
                            process(r0, j0);
                            if (two) process(r1, j0 + 4);
                        }
                        // K padding of the next layer: columns [N, roundup(N, 64)) are 0
                        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
                        for (int c8 = N + 8 * g; c8 < ((N + 63) & ~63); c8 += 32)
                            *reinterpret_cast<uint4 *>(sa_t + a_offset(row, c8)) = z;
                        tc_fence_before();
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) arrive_at_leader(a_ready(t));
                        continue;
                    }
                    // head: stage out_c + bias (c < n_out) as fp32 rows of head_stride floats in the A tile,
                    // which the head's MMAs no longer read
                    float *hst = reinterpret_cast<float *>(sa_t);
                    const int hs = A.head_stride;
                    for (int j = g; j * 16 < A.n_out; j += 4) {  // warp-uniform
                        uint32_t rr[16];
                        tmem_ld16_nowait(trow + uint32_t(j * 16), rr);
                        tmem_wait();
#pragma unroll
                        for (int u = 0; u < 16; u += 4) {
                            const float4 b4 = __ldg(reinterpret_cast<const float4 *>(bias + j * 16 + u));
                            *reinterpret_cast<float4 *>(hst + row * hs + j * 16 + u) =
                                make_float4(__uint_as_float(rr[u + 0]) + b4.x, __uint_as_float(rr[u + 1]) + b4.y,
                                            __uint_as_float(rr[u + 2]) + b4.z, __uint_as_float(rr[u + 3]) + b4.w);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(head_ready(t));
                    if (!warp_wait(head_ready(t), uint32_t(r & 1))) {
                        stop = true;
                        break;
                    }
                    // this CTA's outputs of the tile are contiguous ranges of the cache (or of out):
                    // element e of the range belongs to row e / n and output e % n
                    const long long tile = pair_tile(r, t);
                    const long long p0 = tile * kSuperM + rank * kTileM;
                    const int nv = tile < n_tiles && p0 < n_points
                                       ? int(n_points - p0 < kTileM ? n_points - p0 : kTileM)
                                       : 0;
                    constexpr int kEpiThreads = 32 * kEpiWarps;
                    if (A.mode == 0) {
                        for (int i = te; i < nv; i += kEpiThreads) {
                            const float sg = fmaxf(hst[i * hs], 0.0f);
                            if (A.prec == FNR_PREC_FP16) static_cast<__half *>(A.sigma_out)[p0 + i] = __float2half_rn(sg);
                            else static_cast<float *>(A.sigma_out)[p0 + i] = sg;
                        }
                        const int n = 3 * A.D;
                        char *rec0 = A.uvw_out + p0 * A.rec_stride;
                        for (int e = te; e < nv * n; e += kEpiThreads) {
                            const int i = e / n, c = e - i * n;
                            const float o = hst[i * hs + 1 + c];
                            char *rec = rec0 + size_t(i) * A.rec_stride;
                            if (A.prec == FNR_PREC_FP16) reinterpret_cast<__half *>(rec)[c] = __float2half_rn(o);
                            else reinterpret_cast<float *>(rec)[c] = o;
                        }
                    } else if (A.mode == 1) {
                        const int n = A.D;
                        for (int e = te; e < nv * n; e += kEpiThreads) {
                            const int i = e / n, c = e - i * n;
                            const float o = hst[i * hs + c];
                            if (A.dprec == FNR_PREC_FP16)
                                static_cast<__half *>(A.beta_out)[p0 * n + e] = __float2half_rn(o);
                            else static_cast<float *>(A.beta_out)[p0 * n + e] = o;
                        }
                    } else {
                        const int n = A.out_stride;
                        for (int e = te; e < nv * n; e += kEpiThreads) {
                            const int i = e / n, c = e - i * n;
                            const float o = hst[i * hs + c];
                            A.out[p0 * n + e] = (c == 0 && A.relu0) ? fmaxf(o, 0.0f) : o;
                        }
                    }
                    // the staged rows have been read: the next pair's layer 0 may use the accumulator
                    // and its epilogue may overwrite the A tile
                    __syncwarp();
                    if (r + 1 < n_pairs && lane == 0) arrive_at_leader(a_ready(t));
                }
            }
        }
    }
    __syncthreads();
    // no arrive or MMA of one CTA of the pair targets the other after this point
    cluster_sync();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_free(tmem, kTmemCols);
    }
}

}  // namespace

fnr_status launch_mlp_pair(const MlpArgs &A, int num_sms, cudaStream_t s) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(mlp_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemBytes))) !=
        cudaSuccess)
        return cuda_fail(e, "MLP smem attribute");
    const long long tiles = (A.n_points + kSuperM - 1) / kSuperM;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(kCtas);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(unsigned(num_sms / kCtas * kCtas));
    int clusters = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&clusters, mlp_pair_kernel, &cfg)) != cudaSuccess)
        return cuda_fail(e, "MLP cluster occupancy");
    if (clusters < 1) return fail(FNR_ERR_UNSUPPORTED, "MLP kernel: no SM pair can hold a CTA pair");
    cfg.gridDim = dim3(unsigned((tiles < clusters ? tiles : clusters) * kCtas));
    if ((e = cudaLaunchKernelEx(&cfg, mlp_pair_kernel, A)) != cudaSuccess) return cuda_fail(e, "MLP launch");
    return FNR_OK;
}

}  // namespace fnr
