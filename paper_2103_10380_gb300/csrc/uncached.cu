// uncached.cu -- the uncached FastNeRF render: F_pos at every sample inside the
// box and F_dir per ray, evaluated by the tensor-core MLP kernel (mlp.cu), then
// composited with Eq. 5 and Eq. 1 exactly as the cached march does.
//
//   directions_kernel: every ray's unit direction, and F_dir over them;
//   then, batch by batch of rays (about 8 Mi samples, or 16 Ki rays if that
//     is more):
//   samples_kernel: the inside samples' positions in one compact list (a
//     warp-aggregated atomic hands each ray its range);
//   F_pos over the list (PointsMlp; its length stays on the device);
//   composite_kernel: per ray, beta from F_dir, then the samples in order:
//     sigma and (u, v, w) from F_pos, Eq. 5 + activation, Eq. 1 and the exact
//     integer termination; RGBA and counters;
//   publish_kernel: the finished image to the caller, unless a network's launch
//     failed.
// The networks' FLOPs are what the call cannot do without. The batches keep
// the temporaries at one GB and nothing waits between them: an 800 x 800 view of
// 128 samples has 9 GB of them in one piece, whose allocation and release and
// whose wait for the number of samples took 5 of 45 ms. Batches of 2 / 4 / 8 Mi
// samples: 44.0 / 40.6 / 39.0 ms (each launch has its ramp and its last wave).
// Compositing is a thread per ray, so a batch also holds at least 16 Ki rays:
// 256 x 256 x 4096 at 2 / 4 / 8 / 16 / 32 / 64 Ki rays 215 / 166 / 143 / 135 /
// 134 / 139 ms. All batches are of one size but for the last.
#include <algorithm>

#include "march_device.cuh"
#include "nvtx_range.h"

namespace fnr {

fnr_status fail(fnr_status st, const char *fmt, ...);
fnr_status cuda_fail(cudaError_t e, const char *what);
void clear_error();
fnr_status make_render_const(const fnr_render_params *p, RenderConst *rc);
fnr_status check_camera(const fnr_camera *c);
void fill_frame(FrameDesc *f, const fnr_camera *cam, float *rgba, fnr_ray_stats *stats, int32_t *cells,
                int tile_begin);
bool budget_charge(fnr_context *ctx, uint64_t bytes);
void budget_uncharge(fnr_context *ctx, uint64_t bytes);

namespace {

struct Ray {
    float d[3], o[3];
};

// a1 with the same binary32 sequence as the cached march
__device__ __forceinline__ Ray make_ray(const FrameDesc &F, int px, int py) {
    Ray r;
    const float dcx = __fdiv_rn(__fsub_rn(__fadd_rn(static_cast<float>(px), 0.5f), F.cx), F.fx);
    const float dcy = -__fdiv_rn(__fsub_rn(__fadd_rn(static_cast<float>(py), 0.5f), F.cy), F.fy);
    const float wx = __fmaf_rn(F.c2w[0], dcx, __fmaf_rn(F.c2w[1], dcy, -F.c2w[2]));
    const float wy = __fmaf_rn(F.c2w[4], dcx, __fmaf_rn(F.c2w[5], dcy, -F.c2w[6]));
    const float wz = __fmaf_rn(F.c2w[8], dcx, __fmaf_rn(F.c2w[9], dcy, -F.c2w[10]));
    const float n2 = __fmaf_rn(wx, wx, __fmaf_rn(wy, wy, __fmul_rn(wz, wz)));
    const float len = __fsqrt_rn(n2);
    r.d[0] = __fdiv_rn(wx, len);
    r.d[1] = __fdiv_rn(wy, len);
    r.d[2] = __fdiv_rn(wz, len);
    r.o[0] = F.c2w[3];
    r.o[1] = F.c2w[7];
    r.o[2] = F.c2w[11];
    return r;
}

struct Box {
    float lo[3], hi[3];
};

// sample i of the ray: position and whether it is inside the box
__device__ __forceinline__ bool sample_at(const Ray &r, const RenderConst &rc, const Box &b, int i, float p[3]) {
    const float t = __fmaf_rn(__fadd_rn(static_cast<float>(i), 0.5f), rc.dt, rc.t_near);
    bool in = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        p[a] = __fmaf_rn(t, r.d[a], r.o[a]);
        in = in && p[a] >= b.lo[a] && p[a] < b.hi[a];
    }
    return in;
}

__global__ void directions_kernel(const FrameDesc F, float *dirs) {
    const int ray = blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= F.W * F.H) return;
    const Ray r = make_ray(F, ray % F.W, ray / F.W);
    dirs[3 * ray] = r.d[0];
    dirs[3 * ray + 1] = r.d[1];
    dirs[3 * ray + 2] = r.d[2];
}

// Rays [ray0, ray0 + n_rays). A ray's inside samples are consecutive (t_i, and so each coordinate, is monotone in
// i), so a lane finds its ray's first and their number, and the warp writes the rays' positions one ray after the
// other, 32 samples at a time (a lane writing its own ray's scattered them: 328 us for 400 x 400 rays of 128).
__global__ void samples_kernel(const FrameDesc F, const RenderConst rc, const Box b, int ray0, int n_rays,
                               float *points, unsigned long long *total, long long *offset) {
    constexpr unsigned FULL = 0xffffffffu;
    const int i_ray = blockIdx.x * blockDim.x + threadIdx.x, ray = ray0 + i_ray, lane = threadIdx.x & 31;
    const bool active = i_ray < n_rays;
    Ray r = {};
    int first = 0, n = 0;
    if (active) {
        r = make_ray(F, ray % F.W, ray / F.W);
        float p[3];
        for (int i = rc.N - 1; i >= 0; --i)
            if (sample_at(r, rc, b, i, p)) {
                first = i;
                ++n;
            }
    }
    // one atomic per warp for the warp's rays
    int incl = n;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
        const int v = __shfl_up_sync(FULL, incl, dd);
        if (lane >= dd) incl += v;
    }
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(total, static_cast<unsigned long long>(incl));
    base = __shfl_sync(FULL, base, 31);
    if (active) offset[i_ray] = static_cast<long long>(base) + incl - n;
    float *out = points + 3 * base;
    for (int j = 0; j < 32; ++j) {
        const int nj = __shfl_sync(FULL, n, j), fj = __shfl_sync(FULL, first, j);
        Ray q;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            q.d[a] = __shfl_sync(FULL, r.d[a], j);
            q.o[a] = F.c2w[4 * a + 3];
        }
        for (int i = lane; i < nj; i += 32) {
            float p[3];
            sample_at(q, rc, b, fj + i, p);
            out[3 * i] = p[0];
            out[3 * i + 1] = p[1];
            out[3 * i + 2] = p[2];
        }
        out += 3 * nj;
    }
}

// Where the composited rays go, and the networks' error words: a ray is written only while both are 0. A view of
// one batch is written straight to the caller's arrays (its networks' launches are over by then); of several, to
// `rgba` and `counters` of the call (steps, lookups, occupied per ray), since a later batch may still fail, and
// from there by publish_kernel when the last has not. Either way a render that fails leaves the caller's arrays
// as they were.
struct Composited {
    float4 *rgba;
    int *counters;
    const int *err_pos, *err_dir;
    __device__ bool failed() const { return (*err_pos | *err_dir) != 0; }
};

template <int D>
__global__ void composite_kernel(const FrameDesc F, const RenderConst rc, const Box b, int ray0, int n_rays,
                                 const float *pos_out, const float *dir_out, const long long *offset,
                                 const Composited to) {
    const int i_ray = blockIdx.x * blockDim.x + threadIdx.x, ray = ray0 + i_ray;
    if (i_ray >= n_rays || to.failed()) return;
    const Ray r = make_ray(F, ray % F.W, ray / F.W);
    float beta[D];
#pragma unroll
    for (int i = 0; i < D; ++i) beta[i] = dir_out[static_cast<long long>(ray) * D + i];
    float T = 1.0f, C[3] = {0.0f, 0.0f, 0.0f};
    unsigned long long S = 0;
    int n_look = 0, n_occ = 0, n_steps = rc.N;
    long long j = offset[i_ray];
    float p[3];
    for (int i = 0; i < rc.N; ++i) {
        if (!sample_at(r, rc, b, i, p)) continue;
        const float *o = pos_out + j * (1 + 3 * D);
        ++j;
        ++n_look;
        const float sg = o[0];
        if (!(sg > 0.0f)) continue;
        ++n_occ;
        float col[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {  // Eq. 5, each channel's sum in order j = 0 .. D-1
            float x = 0.0f;
#pragma unroll
            for (int k = 0; k < D; ++k) x = __fmaf_rn(beta[k], o[1 + ch * D + k], x);
            col[ch] = rc.act == FNR_ACT_IDENTITY ? x : __fdividef(1.0f, 1.0f + __expf(-x));
        }
        float ext, alpha;
        dev::extinction(__fmul_rn(sg, rc.dt), ext, alpha);
        const float w = T * alpha;
        C[0] = __fmaf_rn(w, col[0], C[0]);
        C[1] = __fmaf_rn(w, col[1], C[1]);
        C[2] = __fmaf_rn(w, col[2], C[2]);
        T = T * ext;
        S += dev::fixed_depth(sg);
        if (S >= static_cast<unsigned long long>(rc.s_thr)) {
            n_steps = i + 1;
            break;
        }
    }
    float4 out;
    out.x = __fmaf_rn(T, rc.bg[0], C[0]);
    out.y = __fmaf_rn(T, rc.bg[1], C[1]);
    out.z = __fmaf_rn(T, rc.bg[2], C[2]);
    out.w = 1.0f - T;
    to.rgba[ray] = out;
    if (to.counters) {
        to.counters[3 * ray] = n_steps;
        to.counters[3 * ray + 1] = n_look;
        to.counters[3 * ray + 2] = n_occ;
    } else if (F.stats) {
        reinterpret_cast<int4 *>(F.stats)[ray] = make_int4(n_steps, n_look, n_occ, -1);
    }
}

// Bound by memory: 44 bytes a ray, 60 with counters. With it an 800 x 800 view of 128 samples takes 39.3 ms, without
// 39.2 (runs of one side differ by 0.3).
__global__ void publish_kernel(const FrameDesc F, const Composited from) {
    const int ray = blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= F.W * F.H || from.failed()) return;
    reinterpret_cast<float4 *>(F.rgba)[ray] = from.rgba[ray];
    const int *c = from.counters + 3 * ray;
    if (F.stats) reinterpret_cast<int4 *>(F.stats)[ray] = make_int4(c[0], c[1], c[2], -1);
}

template <int D>
cudaError_t launch_composite(const FrameDesc &F, const RenderConst &rc, const Box &b, int ray0, int n,
                             const float *pos_out, const float *dir_out, const long long *offset, const Composited &to,
                             cudaStream_t s) {
    composite_kernel<D><<<(n + 127) / 128, 128, 0, s>>>(F, rc, b, ray0, n, pos_out, dir_out, offset, to);
    return cudaGetLastError();
}

cudaError_t composite(int D, const FrameDesc &F, const RenderConst &rc, const Box &b, int ray0, int n,
                      const float *pos_out, const float *dir_out, const long long *offset, const Composited &to,
                      cudaStream_t s) {
    switch (D) {
        case 1: return launch_composite<1>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        case 2: return launch_composite<2>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        case 4: return launch_composite<4>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        case 6: return launch_composite<6>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        case 8: return launch_composite<8>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        case 16: return launch_composite<16>(F, rc, b, ray0, n, pos_out, dir_out, offset, to, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

}  // namespace fnr

using namespace fnr;

extern "C" fnr_status fnr_render_mlp(fnr_context *ctx, const fnr_mlp *pos_mlp, const fnr_mlp *dir_mlp, int32_t D,
                                     const float *bmin, const float *bmax, const fnr_camera *cam,
                                     const fnr_render_params *params, float *rgba_dev, fnr_ray_stats *stats_dev,
                                     fnr_stream_t stream) {
    clear_error();
    NvtxRange range("fnr_render_mlp");
    if (!ctx || !pos_mlp || !dir_mlp || !bmin || !bmax || !cam || !rgba_dev)
        return fail(FNR_ERR_INVALID_ARG, "NULL argument");
    if (D != 1 && D != 2 && D != 4 && D != 6 && D != 8 && D != 16)
        return fail(FNR_ERR_UNSUPPORTED, "the uncached render supports D in {1,2,4,6,8,16}, got %d", D);
    fnr_status st;
    if ((st = check_mlp(pos_mlp, 1 + 3 * D, "pos_mlp")) != FNR_OK) return st;
    if ((st = check_mlp(dir_mlp, D, "dir_mlp")) != FNR_OK) return st;
    Box b;
    for (int a = 0; a < 3; ++a) {
        if (!(isfinite(bmin[a]) && isfinite(bmax[a]) && bmax[a] > bmin[a]))
            return fail(FNR_ERR_INVALID_ARG, "invalid box");
        b.lo[a] = bmin[a];
        b.hi[a] = bmax[a];
    }
    RenderConst rc;
    if ((st = make_render_const(params, &rc)) != FNR_OK) return st;
    if (rc.flags != 0u) return fail(FNR_ERR_UNSUPPORTED, "the uncached render takes no render flags");
    if ((st = check_camera(cam)) != FNR_OK) return st;
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    FrameDesc F;
    fill_frame(&F, cam, rgba_dev, stats_dev, nullptr, 0);
    const long long n_rays = static_cast<long long>(cam->width) * cam->height;
    constexpr long long kBatchPoints = 1LL << 23, kBatchRays = 1LL << 14;
    const long long most = std::max<long long>(kBatchPoints / rc.N, kBatchRays);
    const long long n_batches = (n_rays + most - 1) / most, batch = (n_rays + n_batches - 1) / n_batches;
    const long long batch_pts = batch * rc.N;
    const bool staged = n_batches > 1;
    // the batch's sample list and F_pos over it, the directions and F_dir over them, the rays' places in the list, the
    // lists' lengths, the image
    const size_t sizes[] = {size_t(batch_pts) * 12, size_t(batch_pts) * (1 + 3 * D) * 4, size_t(n_rays) * 12,
                            size_t(n_rays) * D * 4, size_t(batch) * 8,                   size_t(n_batches) * 8,
                            staged ? size_t(n_rays) * 16 : 0};
    uint64_t bytes = 0;  // charged while the call runs
    for (size_t v : sizes) bytes += v;
    if (!budget_charge(ctx, bytes))
        return fail(FNR_ERR_BUDGET, "the uncached render needs %llu bytes of temporaries", (unsigned long long)bytes);
    TempBuf points, pos_out, dirs, dir_out, offset, totals, image;
    PointsMlp pos, dir;
    TempBuf *const bufs[] = {&points, &pos_out, &dirs, &dir_out, &offset, &totals, &image};
    for (int i = 0; i < 7 && st == FNR_OK; ++i)
        if (sizes[i] && (e = bufs[i]->alloc(ctx, sizes[i], s)) != cudaSuccess)
            st = cuda_fail(e, "uncached render temporaries");
    if (st == FNR_OK && (e = cudaMemsetAsync(totals.p, 0, size_t(n_batches) * 8, s)) != cudaSuccess)
        st = cuda_fail(e, "memset");
    if (st == FNR_OK) st = pos.prepare(ctx, pos_mlp, 1 + 3 * D, true, s);
    if (st == FNR_OK) st = dir.prepare(ctx, dir_mlp, D, false, s);
    if (st == FNR_OK) {
        directions_kernel<<<unsigned((n_rays + 127) / 128), 128, 0, s>>>(F, static_cast<float *>(dirs.p));
        if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "ray directions");
    }
    if (st == FNR_OK)
        st = dir.launch(static_cast<const float *>(dirs.p), n_rays, nullptr, static_cast<float *>(dir_out.p), s);
    Composited to = {};
    if (st == FNR_OK) {
        to.rgba = static_cast<float4 *>(staged ? image.p : static_cast<void *>(rgba_dev));
        to.counters = staged ? static_cast<int *>(dirs.p) : nullptr;  // F_dir has read the directions by then
        to.err_pos = pos.error_word();
        to.err_dir = dir.error_word();
    }
    for (long long i = 0; i < n_batches && st == FNR_OK; ++i) {
        const int ray0 = int(i * batch), n = int(std::min(batch, n_rays - i * batch));
        unsigned long long *total = static_cast<unsigned long long *>(totals.p) + i;
        samples_kernel<<<unsigned((n + 127) / 128), 128, 0, s>>>(F, rc, b, ray0, n, static_cast<float *>(points.p), total,
                                                                 static_cast<long long *>(offset.p));
        if ((e = cudaGetLastError()) != cudaSuccess) {
            st = cuda_fail(e, "sample positions");
            break;
        }
        st = pos.launch(static_cast<const float *>(points.p), (long long)n * rc.N, total,
                        static_cast<float *>(pos_out.p), s);
        if (st == FNR_OK &&
            (e = composite(D, F, rc, b, ray0, n, static_cast<const float *>(pos_out.p),
                           static_cast<const float *>(dir_out.p), static_cast<const long long *>(offset.p), to, s)) !=
                cudaSuccess)
            st = cuda_fail(e, "uncached composite");
    }
    if (st == FNR_OK && staged) {
        publish_kernel<<<unsigned((n_rays + 255) / 256), 256, 0, s>>>(F, to);
        if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "uncached image");
    }
    if (st == FNR_OK) st = pos.finish(s);
    if (st == FNR_OK) st = dir.finish(s);
    if (st != FNR_OK) cudaStreamSynchronize(s);  // whatever was launched has left the temporaries
    budget_uncharge(ctx, bytes);
    return st;
}
