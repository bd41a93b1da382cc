// march_voxels.cuh -- the voxel walk (FNR_RENDER_VOXELS): every cell a ray
// passes through is one sample whose delta is the ray's length inside the cell
// (Section 4 integrates every voxel a ray passes through once it has reached
// the density).
//
// One lane per ray, one warp per 8 x 4 pixel tile as in the uniform march. The
// walk itself (a 3-D digital differential analyser in binary32, the sequence
// fixed in fnr.h) is arithmetic only, so each lane generates three or four
// cells ahead (walk_group), issues their density loads together, composites
// them in walk order (weights, transmittance, exact fixed-point termination)
// and only then loads the records of the cells it composited; a group with no
// density in any lane of the warp ends at its density loads. What bounds it is
// the issue of the walk's instructions (k = 256, every cell / skipping: 0.76 /
// 0.78 issued per cycle and scheduler), so it is those that were cut: divisions
// through the ray's reciprocals (divide_by), short groups, empty groups left
// early, no code for outputs that are not asked for. 800 x 800, k = 512, FP32:
// 1064 -> 750 us, with skipping 876 -> 518; FP16, 512 x 512, k = 256: 230 -> 168,
// with skipping 265 -> 156; E4M3 with skipping 1486 -> 646. In this mode the
// launcher passes t_far in r.dt (the walk has no sample spacing) and r.s_thr is
// the threshold on sum floor(fp32(sigma delta) 2^32).
//
// The kernel is instantiated four times per (precision, D), one form per
// translation unit: the plain walk (march_voxels.cu), the walk that skips the
// density loads of empty bricks and passes over empty cubes in one step
// (march_voxels_jump.cu), and both without the passes when every walked cell is
// written (march_voxels_cells.cu, march_voxels_skip_cells.cu). Each form carries
// only its own code: the brick arithmetic alone cost the plain walk 10%.
#pragma once
#include <type_traits>

#include "march_device.cuh"

namespace fnr {

enum VoxelForm { kVoxPlain = 0, kVoxJump = 1, kVoxCells = 2, kVoxSkipCells = 3 };

namespace {

using namespace dev;

// Cells generated ahead of their density loads. Each is a copy of the step's code, and a skipping walk tries one pass
// over an empty cube per group: at 8 the skipping kernel stalled on instruction fetch (2.6 of 9.6 cycles an
// instruction) and walked up to 7 cells into empty space. 800 x 800, k = 512, 8 / 6 / 4 / 3 / 2 cells: FP32 with
// skipping 876 / 766 / 642 / 652 / 688 us, E4M3 1487 / 1233 / 885 / 776 / 795; FP32 plain 1064 / - / 1002.
// The forms that write every walked cell are bound by those stores, 4 bytes a cell at 3k cells a ray: eight at a time
// fill a lane's 32-byte sectors, and few blocks leave them in L2 until they are full. With skipping, 640 x 640, k = 128,
// FP32: 4 / 6 / 8 cells at 4 blocks 896 / 912 / 798 us, 8 cells at 4 / 5 / 6 / 7 blocks 798 / 814 / 855 / 850. Groups and
// blocks as the other forms' -> these, 640 x 640, k = 128 and 256 x 256, k = 192: FP32 956 -> 856 and 415 -> 299, with
// skipping 952 -> 798 and 423 -> 256; E4M3 971 -> 818 and 431 -> 254, with skipping 962 -> 793 and 451 -> 263; FP16 967 ->
// 852, with skipping 966 -> 814.
template <int PREC, int FORM>
constexpr int walk_group() {
    if (FORM == kVoxCells || FORM == kVoxSkipCells) return 8;
    return PREC == FNR_PREC_FP8_E4M3 && FORM == kVoxJump ? 3 : 4;
}

// Minimum resident blocks per SM (registers against latency), by precision and record length. us at 5 / 6 / 7 / 8 blocks,
// without and with skipping, 800 x 800, k = 350, and 512 x 512, k = 256:
//   FP32 D = 8    629 568 535 516, 491 437 408 392;  204 188 180 177, 174 164 158 164
//        D = 12   666 611 585 565, 568 547 533 545;  225 208 203 208, 227 226 232 246
//        D = 16   738 679 635 620, 586 541 509 490;  261 245 239 246, 235 239 241 251
//   FP16 D = 8    570 542 542 531, 498 446 414 391;  181 177 176 178, 179 170 163 167
//        D = 12   679 631 601 604, 611 565 537 546;  213 202 196 201, 228 221 226 237
//        D = 16   708 654 626 636, 563 506 473 454;  229 217 217 227, 212 207 209 218
//   E4M3 D = 4    821 785 773 817, 562 530 506 503;  256 249 247 263, 225 222 217 229
//        D = 8    677 655 674 691, 520 484 476 477;  218 215 227 237, 203 197 200 210
//        D = 12   753 764 771 783, 668 676 690 709;  245 252 257 268, 268 290 315 323
//        D = 16   850 889 888 894, 640 640 631 658;  278 304 319 340, 261 277 303 328
// E4M3 records are decoded with their offsets and scales in registers: at 8 blocks (64 registers) its kernels spill up
// to 550 bytes, so short ones run at 7 and long ones at 5. FP32 spills at most 44 bytes at 8 (D = 15: 220), FP16 24 at 7.
template <int PREC, int D, int FORM>
constexpr int walk_blocks() {
    if (FORM == kVoxCells || FORM == kVoxSkipCells) return 4;
    if (PREC == FNR_PREC_FP8_E4M3) return D <= 8 ? 7 : 5;
    return PREC == FNR_PREC_FP16 ? 7 : 8;
}

// a / b correctly rounded from y = 1 / b correctly rounded: Markstein's theorem (P. W. Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34(1), 1990) -- with q a faithful
// quotient and r = a - b q exact, q + r y rounds to the correctly rounded quotient. The first correction makes q
// faithful. Needs 2^-60 <= |b| <= 2^60 and a = +0 or 2^-60 <= |a| <= 2^61, so that no step leaves the normal range.
__device__ __forceinline__ float divide_by(float a, float b, float y) {
    float q = __fmul_rn(a, y);
    q = __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
    return __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
}

// The cells of one ray in walk order (fnr.h, FNR_RENDER_VOXELS). RECIP: the divisions by u_a through its
// reciprocal (every ray but the few whose coordinates are out of its range, see safe()): five multiplications and
// additions in line, without the division's branch to its general case.
template <bool RECIP>
struct VoxelWalk {
    float u0, u1, u2, w0, w1, w2;  // g_a(t) = t u_a + w_a in grid units
    float y0, y1, y2;              // 1 / u_a
    float tn0, tn1, tn2;           // next crossing per axis
    int c0, c1, c2;                // current cell
    float t, t1;
    int k;
    bool live;

    // Whether the ray's divisions can go through reciprocals. Every dividend is RN(m - w_a) for an integer
    // 0 <= m <= k: +0, or at least min(|w_a|, 2^-25).
    __device__ __forceinline__ static bool safe(const CacheView &cv, const float o[3], const float d[3]) {
        bool ok = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float u = fabsf(__fmul_rn(d[a], cv.scale[a]));
            const float w = fabsf(__fmul_rn(__fsub_rn(o[a], cv.bmin[a]), cv.scale[a]));
            ok = ok && (u == 0.0f || (u >= 0x1p-60f && u <= 0x1p60f)) && (w == 0.0f || w >= 0x1p-60f) && w <= 0x1p60f;
        }
        return ok;
    }

    __device__ __forceinline__ static float divide(float a, float u, float y) {
        return RECIP ? divide_by(a, u, y) : __fdiv_rn(a, u);
    }

    __device__ __forceinline__ static float crossing(int c, float u, float w, float y) {
        const float tc = divide(__fsub_rn(static_cast<float>(u > 0.0f ? c + 1 : c), w), u, y);
        return u == 0.0f ? __int_as_float(0x7f800000) : tc;  // +infinity
    }

    // Box clipping, start cell and first crossings; live = false if the ray
    // has no cells in [t_near, t_far].
    __device__ __forceinline__ void init(const CacheView &cv, const float o[3], const float d[3], float t_near,
                                         float t_far) {
        k = cv.k;
        const float kf = cv.kf;
        float uu[3], ww[3], yy[3];
        float t0 = t_near, te = t_far;
        live = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            uu[a] = __fmul_rn(d[a], cv.scale[a]);
            ww[a] = __fmul_rn(__fsub_rn(o[a], cv.bmin[a]), cv.scale[a]);
            yy[a] = RECIP ? __frcp_rn(uu[a]) : 0.0f;
            if (uu[a] != uu[a] || ww[a] != ww[a]) live = false;
            if (uu[a] == 0.0f) {
                if (!(ww[a] >= 0.0f && ww[a] < kf)) live = false;
            } else {
                const float ta = divide(-ww[a], uu[a], yy[a]);
                const float tb = divide(__fsub_rn(kf, ww[a]), uu[a], yy[a]);
                const float lo = ta < tb ? ta : tb, hi = ta < tb ? tb : ta;
                if (lo > t0) t0 = lo;
                if (hi < te) te = hi;
            }
        }
        if (!(t0 < te)) live = false;
        u0 = uu[0], u1 = uu[1], u2 = uu[2];
        w0 = ww[0], w1 = ww[1], w2 = ww[2];
        y0 = yy[0], y1 = yy[1], y2 = yy[2];
        t = t0;
        t1 = te;
        auto start = [&](float u, float w) {
            const int ci = __float2int_rd(__fmaf_rn(t0, u, w));
            return ci < 0 ? 0 : (ci > k - 1 ? k - 1 : ci);
        };
        c0 = live ? start(u0, w0) : 0;
        c1 = live ? start(u1, w1) : 0;
        c2 = live ? start(u2, w2) : 0;
        tn0 = crossing(c0, u0, w0, y0);
        tn1 = crossing(c1, u1, w1, y1);
        tn2 = crossing(c2, u2, w2, y2);
    }

    // The current cell, its occupancy brick (bricks of 2^sh cells, od per axis),
    // its E4M3 offset brick (2^osh cells, odim per axis) and its length;
    // advances to the next cell, or clears live after the last one. The step is
    // branch-free: lanes of a warp step different axes.
    __device__ __forceinline__ int next(float &delta, int &brick, int sh, int od, int &obrick, int osh, int odim) {
        const bool y = tn1 < tn0;
        const float txy = y ? tn1 : tn0;
        const bool z = tn2 < txy;
        const float tnext = z ? tn2 : txy;
        const float end = tnext < t1 ? tnext : t1;
        const int cell = (c2 * k + c1) * k + c0;  // k^3 < 2^31
        brick = ((c2 >> sh) * od + (c1 >> sh)) * od + (c0 >> sh);
        obrick = ((c2 >> osh) * odim + (c1 >> osh)) * odim + (c0 >> osh);
        delta = __fsub_rn(end, t);
        if (!(tnext < t1)) {
            live = false;
            return cell;
        }
        if (tnext > t) t = tnext;
        // the stepped axis has u != 0 (a +infinity crossing is never below t1)
        const float ua = z ? u2 : (y ? u1 : u0);
        const float wa = z ? w2 : (y ? w1 : w0);
        const float ya = z ? y2 : (y ? y1 : y0);
        const int ca = (z ? c2 : (y ? c1 : c0)) + (ua > 0.0f ? 1 : -1);
        const float tna = divide(__fsub_rn(static_cast<float>(ua > 0.0f ? ca + 1 : ca), wa), ua, ya);
        if (z) {
            c2 = ca;
            tn2 = tna;
        } else if (y) {
            c1 = ca;
            tn1 = tna;
        } else {
            c0 = ca;
            tn0 = tna;
        }
        if (ca < 0 || ca >= k) live = false;
        return cell;
    }

    // Crossings the walk makes along one axis from cell c on (n = 0: the one out
    // of c) at times before X, and at X too when `at`: counted with the crossing
    // formula itself, which is monotone in the cell index, from an estimate out
    // of the grid coordinate at X. -1 if the estimate is off by more than a few.
    // `next` receives the first crossing not counted: the one out of the cell
    // the axis has reached.
    __device__ __forceinline__ static int crossings_until(int c, float u, float w, float y, float X, bool at,
                                                              float &next) {
        next = __int_as_float(0x7f800000);
        if (u == 0.0f) return 0;
        const int s = u > 0.0f ? 1 : -1;
        auto before = [&](int n) {
            const float tc = crossing(c + s * n, u, w, y);
            const bool b = tc < X || (at && tc == X);
            if (!b) next = tc;
            return b;
        };
        const float g = floorf(__fmaf_rn(X, u, w));
        const float est = s > 0 ? g - static_cast<float>(c) : static_cast<float>(c) - g;
        int n = static_cast<int>(fminf(fmaxf(est, 0.0f), 16777216.0f));
        int fixes = 0;
        while (n > 0 && !before(n - 1))
            if (--n, ++fixes > 4) return -1;
        while (before(n))
            if (++n, ++fixes > 4) return -1;
        return n;
    }

    // One step over the cells of an empty cube [lo_a, hi_a] of cells that holds
    // the current cell: the number of cells the walk would return, one by one,
    // until it leaves the cube (or ends inside it), and its state after that,
    // both exactly as next() would leave them -- every crossing time comes from
    // a cell index alone, crossings at one time go in axis order, and each
    // crossing moves one axis by one cell. Returns the cells passed; at most
    // `cap`, which spends the walk; 0 if it took no step.
    __device__ __forceinline__ int pass_cube(const int lo[3], const int hi[3], int cap) {
        const float uu[3] = {u0, u1, u2}, ww[3] = {w0, w1, w2}, yy[3] = {y0, y1, y2};
        const int cc[3] = {c0, c1, c2};
        float X = __int_as_float(0x7f800000);
        int ax = 3;  // the axis whose crossing leaves the cube first (the lowest on a tie)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (uu[a] != 0.0f) {
                const float xa = crossing(uu[a] > 0.0f ? hi[a] : lo[a], uu[a], ww[a], yy[a]);
                if (xa < X) {
                    X = xa;
                    ax = a;
                }
            }
        const bool ends = !(X < t1);  // the walk ends inside the cube
        int n[3], total = ends ? 1 : 0;
        float nx[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            n[a] = crossings_until(cc[a], uu[a], ww[a], yy[a], ends ? t1 : X, !ends && a <= ax, nx[a]);
            if (n[a] < 0) return 0;
            total += n[a];
        }
        if (total <= 1) return 0;
        if (total >= cap) return cap;
        if (ends) {
            live = false;
            return total;
        }
        c0 = cc[0] + (uu[0] > 0.0f ? n[0] : -n[0]);
        c1 = cc[1] + (uu[1] > 0.0f ? n[1] : -n[1]);
        c2 = cc[2] + (uu[2] > 0.0f ? n[2] : -n[2]);
        if (X > t) t = X;
        tn0 = nx[0];  // = crossing(c0, u0, w0), computed by the count
        tn1 = nx[1];
        tn2 = nx[2];
        const int ca = ax == 0 ? c0 : (ax == 1 ? c1 : c2);
        if (ca < 0 || ca >= k) live = false;
        return total;
    }
};

template <int PREC, int D, int FORM>
__global__ void __launch_bounds__(FNR_BLOCK, (walk_blocks<PREC, D, FORM>()))
    march_voxels_kernel(const __grid_constant__ MarchArgs A) {
    allow_next_grid();
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int kVU = walk_group<PREC, FORM>();
    const int tile = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (tile >= A.total_tiles) return;  // whole warp
    int f = 0;
    while (f + 1 < A.n_frames && tile >= A.f[f + 1].tile_begin) ++f;
    const FrameDesc &F = A.f[f];
    const CacheView &c = A.c;
    const RenderConst &r = A.r;
    int x0, y0;
    tile_origin(F, tile - F.tile_begin, x0, y0);
    const int lane = threadIdx.x & 31;
    const int px = x0 + (lane & (kTileW - 1)), py = y0 + lane / kTileW;
    const bool active = px < F.W && py < F.H;
    constexpr bool kOffs = PREC == FNR_PREC_FP8_E4M3;
    __shared__ float sbeta[FNR_BLOCK / 32][D][32];
    __shared__ float wsc[FNR_BLOCK / 32][kOffs ? 3 * D : 1];  // E4M3: the (u, v, w) channel scales, per warp
    float (*qbeta)[32] = sbeta[threadIdx.x >> 5];
    float *ssc = wsc[threadIdx.x >> 5];
    if constexpr (kOffs) {
        for (int i = lane; i < 3 * D; i += 32) ssc[i] = __ldg(c.scales + 1 + i);
        __syncwarp();
    }

    RaySetup<PREC, D> R;  // a1/a2: direction cell and beta (the uniform-sample fields go unused)
    float dd[3] = {0.0f, 0.0f, 1.0f};
    const float oo[3] = {F.c2w[3], F.c2w[7], F.c2w[11]};
    R.dcell = 0;
    R.sigma_scale = 1.0f;
    if (active) {
        R.init(c, r, F, px, py, qbeta, lane);
        // the ray again (the fixed a1 sequence) for the walk
        const float dcx = __fdiv_rn(__fsub_rn(__fadd_rn(static_cast<float>(px), 0.5f), F.cx), F.fx);
        const float dcy = -__fdiv_rn(__fsub_rn(__fadd_rn(static_cast<float>(py), 0.5f), F.cy), F.fy);
        const float wx = __fmaf_rn(F.c2w[0], dcx, __fmaf_rn(F.c2w[1], dcy, -F.c2w[2]));
        const float wy = __fmaf_rn(F.c2w[4], dcx, __fmaf_rn(F.c2w[5], dcy, -F.c2w[6]));
        const float wz = __fmaf_rn(F.c2w[8], dcx, __fmaf_rn(F.c2w[9], dcy, -F.c2w[10]));
        const float n2 = __fmaf_rn(wx, wx, __fmaf_rn(wy, wy, __fmul_rn(wz, wz)));
        const float len = __fsqrt_rn(n2);
        dd[0] = __fdiv_rn(wx, len);
        dd[1] = __fdiv_rn(wy, len);
        dd[2] = __fdiv_rn(wz, len);
    }
    constexpr bool kCells = FORM == kVoxCells || FORM == kVoxSkipCells;
    constexpr bool kSkip = FORM == kVoxJump || FORM == kVoxSkipCells;
    // Skipping without per-cell output also passes over whole empty cubes of jump
    // bricks in one step (VoxelWalk::pass_cube), from the cache's distance field.
    constexpr bool kJump = FORM == kVoxJump;
    float T = 1.0f, Cr = 0.0f, Cg = 0.0f, Cb = 0.0f;
    unsigned long long S = 0;
    int n_gen = 0, n_steps = 0, n_look = 0, n_occ = 0;
    bool term = false;
    const long long pix = active ? static_cast<long long>(py) * F.W + px : 0;
    int32_t *cells_out = (kCells && active) ? F.cells + pix * r.N : nullptr;
    if (kCells) wait_prior_grid();  // cells are written while walking

    auto walk = [&](auto recip) {
        VoxelWalk<decltype(recip)::value> Wk;
        Wk.init(c, oo, dd, r.t_near, r.dt);  // r.dt holds t_far in this mode
        Wk.live = Wk.live && active;
        while (__any_sync(FULL, Wk.live && !term && n_gen < r.N)) {
            // kVU cells ahead, their densities loaded together
            int cell[kVU], brick[kVU], obr[kVU];
            float dl[kVU], sg[kVU];
            unsigned gen = 0u, looked = 0u;
#pragma unroll
            for (int u = 0; u < kVU; ++u) {
                cell[u] = 0;
                brick[u] = 0;
                obr[u] = 0;
                dl[u] = 0.0f;
                if (kJump && u == 0 && Wk.live && !term && n_gen < r.N) {
                    // One pass per group (more per group measured slower: each costs a dozen exact divisions
                    // and the lanes of a warp take different ones). d > 0: the jump bricks within Chebyshev
                    // distance d - 1 of the current one are empty.
                    const int sh = c.dist_shift;
                    const int d =
                        __ldg(c.dist + ((Wk.c2 >> sh) * c.dist_dim + (Wk.c1 >> sh)) * c.dist_dim + (Wk.c0 >> sh));
                    if (d > 0) {
                        const int cw[3] = {Wk.c0, Wk.c1, Wk.c2};
                        int lo[3], hi[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            lo[a] = max(((cw[a] >> sh) - (d - 1)) << sh, 0);
                            hi[a] = min((((cw[a] >> sh) + d) << sh) - 1, Wk.k - 1);
                        }
                        const int m = Wk.pass_cube(lo, hi, r.N - n_gen);
                        n_gen += m;
                        n_steps += m;
                    }
                }
                if (Wk.live && !term && n_gen < r.N) {
                    cell[u] = Wk.next(dl[u], brick[u], c.occ_shift, c.occ_dim, obr[u], c.offs_shift, c.offs_dim);
                    gen |= 1u << u;
                    ++n_gen;
                }
            }
            // The cell indices as they are: rebuilt from the walk's coordinates where they are used, they kept more
            // registers alive (FP32 plain 776 us, now 749; FP16 plain 174, now 168).
#pragma unroll
            for (int u = 0; u < kVU; ++u) asm volatile("" : "+r"(cell[u]));
#pragma unroll
            for (int u = 0; u < kVU; ++u) {
                sg[u] = 0.0f;
                if (((gen >> u) & 1u) && dl[u] > 0.0f) {
                    const bool load = !kSkip || brick_occupied(c, brick[u]) != 0u;
                    if (load) {
                        sg[u] = load_sigma<PREC>(c, cell[u], R.sigma_scale);
                        looked |= 1u << u;
                    }
                }
            }
            if (cells_out) {
                int j = n_steps;
#pragma unroll
                for (int u = 0; u < kVU; ++u)
                    if ((gen >> u) & 1u) cells_out[j++] = cell[u];  // past termination: overwritten by -2 below
            }
            unsigned dense = 0u;
#pragma unroll
            for (int u = 0; u < kVU; ++u) dense |= (sg[u] > 0.0f ? 1u : 0u) << u;
            if (!__any_sync(FULL, dense != 0u)) {  // empty space for the whole warp
                n_steps += __popc(gen);
                n_look += __popc(looked);
                continue;
            }
            // walk order: weights, transmittance and termination from the densities alone
            float wgt[kVU];
            unsigned occ = 0u, counted = gen;
#pragma unroll
            for (int u = 0; u < kVU; ++u) {
                wgt[u] = 0.0f;
                if (((dense >> u) & 1u) && !term) {
                    const float od = __fmul_rn(sg[u], dl[u]);
                    float ext, alpha;
                    extinction(od, ext, alpha);
                    wgt[u] = T * alpha;
                    T = T * ext;
                    occ |= 1u << u;
                    if (od > 0.0f) S += fixed_depth(od);
                    if (S >= static_cast<unsigned long long>(r.s_thr)) {
                        term = true;
                        counted = gen & ((2u << u) - 1u);
                    }
                }
            }
            n_steps += __popc(counted);
            n_look += __popc(looked & counted);
            n_occ += __popc(occ);
            // records of the composited cells, colour added in walk order
#pragma unroll
            for (int u = 0; u < kVU; ++u) {
                if (!((occ >> u) & 1u)) continue;
                Record<PREC, D> rec;
                rec.load(c.uvw + static_cast<long long>(cell[u]) * c.rec_stride);
                float col[3];
                if constexpr (kOffs) {
                    OffsetRecord<D> off;
                    off.load(c.offs + static_cast<long long>(obr[u]) * c.offs_stride);
                    shade_e4m3<D>(
                        rec, off, r.act, [&](int i) { return ssc[i]; }, [&](int j) { return qbeta[j][lane]; }, col);
                } else {
                    RaySetup<PREC, D>::shade_with(rec, r.act, [&](int ch, int j) { return qbeta[j][lane]; }, col);
                }
                Cr = __fmaf_rn(wgt[u], col[0], Cr);
                Cg = __fmaf_rn(wgt[u], col[1], Cg);
                Cb = __fmaf_rn(wgt[u], col[2], Cb);
            }
        }
    };
    if (__all_sync(FULL, VoxelWalk<true>::safe(c, oo, dd))) walk(std::true_type{});
    else walk(std::false_type{});
    wait_prior_grid();
    if (!active) return;
    if (cells_out)
        for (int j = n_steps; j < r.N; ++j) cells_out[j] = term ? -2 : -1;
    float4 o;
    o.x = __fmaf_rn(T, r.bg[0], Cr);
    o.y = __fmaf_rn(T, r.bg[1], Cg);
    o.z = __fmaf_rn(T, r.bg[2], Cb);
    o.w = 1.0f - T;
    reinterpret_cast<float4 *>(F.rgba)[pix] = o;
    if (F.stats) reinterpret_cast<int4 *>(F.stats)[pix] = make_int4(n_steps, n_look, n_occ, R.dcell);
}

template <int PREC, int D, int FORM>
cudaError_t launch_v(const MarchArgs &a, cudaStream_t s) {
    const int warps_per_block = FNR_BLOCK / 32;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((a.total_tiles + warps_per_block - 1) / warps_per_block));
    cfg.blockDim = dim3(FNR_BLOCK);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, march_voxels_kernel<PREC, D, FORM>, a);
}

template <int PREC, int FORM>
cudaError_t launch_vp(const MarchArgs &a, cudaStream_t s) {
    switch (a.c.D) {
        case 1: return launch_v<PREC, 1, FORM>(a, s);
        case 2: return launch_v<PREC, 2, FORM>(a, s);
        case 3: return launch_v<PREC, 3, FORM>(a, s);
        case 4: return launch_v<PREC, 4, FORM>(a, s);
        case 5: return launch_v<PREC, 5, FORM>(a, s);
        case 6: return launch_v<PREC, 6, FORM>(a, s);
        case 7: return launch_v<PREC, 7, FORM>(a, s);
        case 8: return launch_v<PREC, 8, FORM>(a, s);
        case 9: return launch_v<PREC, 9, FORM>(a, s);
        case 10: return launch_v<PREC, 10, FORM>(a, s);
        case 11: return launch_v<PREC, 11, FORM>(a, s);
        case 12: return launch_v<PREC, 12, FORM>(a, s);
        case 13: return launch_v<PREC, 13, FORM>(a, s);
        case 14: return launch_v<PREC, 14, FORM>(a, s);
        case 15: return launch_v<PREC, 15, FORM>(a, s);
        case 16: return launch_v<PREC, 16, FORM>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

// Every form dispatches on the position-cache precision the same way.
template <int FORM>
cudaError_t launch_voxels_prec(const MarchArgs &a, cudaStream_t s) {
    switch (a.c.pos_prec) {
        case FNR_PREC_FP32: return launch_vp<FNR_PREC_FP32, FORM>(a, s);
        case FNR_PREC_FP16: return launch_vp<FNR_PREC_FP16, FORM>(a, s);
        case FNR_PREC_FP8_E4M3: return launch_vp<FNR_PREC_FP8_E4M3, FORM>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// The other forms of the walk (march_voxels_jump.cu, march_voxels_cells.cu, march_voxels_skip_cells.cu).
cudaError_t launch_march_voxels_jump(const MarchArgs &a, cudaStream_t s);
cudaError_t launch_march_voxels_cells(const MarchArgs &a, cudaStream_t s);
cudaError_t launch_march_voxels_skip_cells(const MarchArgs &a, cudaStream_t s);

}  // namespace fnr
