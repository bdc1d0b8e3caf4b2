// exw_bwd.cu -- adjoint of stage (b) with respect to source colour and motion, and the fused training pass.
//
// A CTA owns a 32 x 32 SOURCE tile S and runs the fractions of its call one after another.  Per fraction, phase 1
// visits every source pixel p of S plus a one-pixel ring: if p won its target q = T(p) and q is not a hole, it
// stores the normalised weights w_t / sum w of its four taps and the upstream gradient g(q) in shared memory, and
// (for p inside S) adds dL/d mv(p) -- p wins at most one target per fraction, so each fraction adds one term and
// needs no atomics.  Phase 2 gives each source pixel s of S the contributions of the (at most 9) winners
// p = s - (dx, dy) that use s as a tap, in a fixed order, so dL/d colour(s) is summed by one thread
// deterministically.  The accumulators are read once, updated per fraction in fraction order and written once:
// a call over nfrac fractions equals nfrac one-fraction calls bit for bit.
//
// g(q) comes from grad_out (exw_warp_backward) or, in the fused training pass (exw_warp_l2_grad), from the
// forward value itself: q's colour is recomputed at its winner p with the arithmetic of stage (b) (same taps,
// weights and operation order, rounded to the storage type), g = 2 (out(q) - target(q)), and (out - target)^2 is
// added to the loss at q's winner, i.e. once per non-hole target.  The loss is summed in a fixed order: in FP32 by
// each thread over its few terms, then in FP64 across threads and CTAs (the FP64 pipe of this part issues about one
// operation per SM clock, so no FP64 arithmetic runs per pixel).
//
// Bound by issue.  The records are planes of words (each read without bank conflicts) with a mask of the directions a
// winner's taps lie in, so phase 2 tests nine bits and reads four records a pixel instead of nine; element addresses are
// 32-bit indices on per-plane pointers; the forward value is computed once for the loss and for the motion gradient.
// 1080p FP32, three fractions: 201 us a frame before (674 instructions per output pixel), 147 us now (events around the
// launch); splat 19 -> 15 us.
#include "exw_device.cuh"
#include "exw_internal.h"

namespace exw {

constexpr int kBwdThreads = 256;
constexpr int kStage = kFillTile + 4;  // S plus a two-pixel ring: the ring's winners and their taps
constexpr int kStageN = kStage * kStage;

// Shared memory of a CTA: the staged source depth (read once, used by every fraction for the taps' agreement; the
// motion and colour are read through L1), the per-fraction records of phase 1 and the motion accumulators of S.
template <typename CT>
struct BwdSmem {
    float w[4][kRegionN];   // w_t / S for taps (p), (p+sx), (p+sy), (p+sx+sy); a plane per word: no bank conflicts
    float g[3][kRegionN];   // g(q) rgb
    float2 gms[kFillTile * kFillTile];
    uint16_t dirs[kRegionN];  // bit 3 (dy + 1) + dx + 1: the source pixel p + (dx, dy) is a tap of p (0: p won nothing)
    float depth[kStageN];   // NaN outside the frame (never lands, never agrees)
    double red[kBwdThreads / 32];
};

// Every plane by its own pointer, so that an element's address is one wide multiply-add of a 32-bit index (a plane has
// at most 2^28 elements).
struct BwdArgs {
    const void *color[3];
    const float *depth;
    const float *mv[2];
    const unsigned long long *keys[kMaxFrac];
    const void *g[kMaxFrac][3];      // per fraction: the targets' channels (fused), or grad_out's (one fraction)
    int W, H, nfrac, k0, L;
    float *grad_color[3];
    float *grad_mv[2];
    bool store;                      // the gradients are written (as if they were zero before), not accumulated
    double *partial;                 // fused: one loss partial per CTA
};

template <typename CT, bool FUSED>
__global__ void __launch_bounds__(kBwdThreads, 4) bwd_tile_kernel(const __grid_constant__ BwdArgs a) {
    extern __shared__ __align__(16) unsigned char bwd_smem_raw[];
    BwdSmem<CT> &sm = *reinterpret_cast<BwdSmem<CT> *>(bwd_smem_raw);
    float2 *gms = sm.gms;
    double *red = sm.red;
    grid_dependency_wait();  // the splat before
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int W = a.W, H = a.H;
    const int X0 = blockIdx.x * kFillTile, Y0 = blockIdx.y * kFillTile;
    const uint32_t Wu = (uint32_t)W;
    // this thread's source pixels of phase 2 (rows wid + 8 j, column lane) and their colour accumulators
    const int sxg = X0 + lane;
    float gc[4][3];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int syg = Y0 + wid + 8 * j;
        const bool in = sxg < W && syg < H;
        const uint32_t s = (uint32_t)syg * Wu + (uint32_t)sxg;
#pragma unroll
        for (int c = 0; c < 3; ++c) gc[j][c] = in && !a.store ? a.grad_color[c][s] : 0.0f;
    }
    // the motion accumulators of S, in shared memory for the whole call
    for (int c = tid; c < kFillTile * kFillTile; c += kBwdThreads) {
        const int x = X0 + (c & (kFillTile - 1)), y = Y0 + c / kFillTile;
        const uint32_t i = (uint32_t)y * Wu + (uint32_t)x;
        gms[c] = (x < W && y < H && !a.store) ? make_float2(a.grad_mv[0][i], a.grad_mv[1][i]) : make_float2(0.f, 0.f);
    }
    // the source of S and its two-pixel ring, once for every fraction
    for (int c = tid; c < kStageN; c += kBwdThreads) {
        const int x = X0 - 2 + c % kStage, y = Y0 - 2 + c / kStage;
        const bool in = x >= 0 && x < W && y >= 0 && y < H;
        const uint32_t i = in ? (uint32_t)y * Wu + (uint32_t)x : 0u;
        sm.depth[c] = in ? __ldg(a.depth + i) : __int_as_float(0x7FC00000);
    }
    __syncthreads();  // phase 1 reads the stage and updates cells another thread loaded
    float lacc = 0.0f;  // this thread's loss terms (at most 5 cells x 3 fractions x 3 channels), then FP64
    for (int kk = 0; kk < a.nfrac; ++kk) {
        const int k = a.k0 + kk, L = a.L;
        const float kf = fraction_scale(k, L), limit = motion_limit(k, L), scale = -kf;
        const unsigned long long *keys = a.keys[kk];
        const void *const *gp = a.g[kk];
        int ry = tid / kRegion, rx = tid - ry * kRegion;  // cell r = tid, tid + 256, ...: 7 rows and 18 columns on
#pragma unroll 1
        for (int r = tid; r < kRegionN; r += kBwdThreads) {  // a cell belongs to the same thread in every fraction
            const int px = X0 - 1 + rx, py = Y0 - 1 + ry;
            const bool inside = rx >= 1 && rx <= kFillTile && ry >= 1 && ry <= kFillTile;
            uint32_t dirs = 0u;
            const int e = (ry + 1) * kStage + (rx + 1);  // p in the stage
            if (px >= 0 && px < W && py >= 0 && py < H) {
                const uint32_t i = (uint32_t)py * Wu + (uint32_t)px;
                const uint32_t db = __float_as_uint(sm.depth[e]);
                const float mx = __ldg(a.mv[0] + i), my = __ldg(a.mv[1] + i);
                if (depth_ok(db) && motion_lands(mx, my, limit)) {
                    const int ox = offset_of(mx, kf), oy = offset_of(my, kf);
                    const int qx = px + ox, qy = py + oy;
                    if ((unsigned)qx < (unsigned)W && (unsigned)qy < (unsigned)H) {
                        const uint32_t q = (uint32_t)qy * Wu + (uint32_t)qx;
                        // every global load of the cell at once: q's key, the depth words of its 4-neighbours', g's
                        // inputs
                        const unsigned long long kq = __ldg(keys + q);
                        const uint32_t *kd = reinterpret_cast<const uint32_t *>(keys + q) + 1;
                        const uint32_t k0 = qx > 0 ? __ldg(kd - 2) : 0xFFFFFFFFu;
                        const uint32_t k1 = qx < W - 1 ? __ldg(kd + 2) : 0xFFFFFFFFu;
                        const uint32_t *kw = reinterpret_cast<const uint32_t *>(keys) + 1;
                        const uint32_t k2 = qy > 0 ? __ldg(kw + 2u * (q - Wu)) : 0xFFFFFFFFu;
                        const uint32_t k3 = qy < H - 1 ? __ldg(kw + 2u * (q + Wu)) : 0xFFFFFFFFu;
                        float gin[3];
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            gin[c] = FUSED ? load_c<CT>((const CT *)gp[c] + q) : __ldg((const float *)gp[c] + q);
                        if (kq == pack_key_global(db, i)) {
                            if (!is_crack(db, k0, k1, k2, k3)) {
                                const float Dp = __uint_as_float(db);
                                int sx, sy;
                                const float rhox = residual(mx, k, L, ox, sx);
                                const float rhoy = residual(my, k, L, oy, sy);
                                const float wx1 = fabsf(rhox), wy1 = fabsf(rhoy);
                                const float wx0 = 1.f - wx1, wy0 = 1.f - wy1;
                                const int tx = px + sx, ty = py + sy;
                                const bool inx = sx != 0 && tx >= 0 && tx < W;
                                const bool iny = sy != 0 && ty >= 0 && ty < H;
                                const int e10 = e + sx, e01 = e + sy * kStage, e11 = e01 + sx;  // taps in the stage
                                const bool a10 = inx && tap_agrees(sm.depth[e10], Dp);
                                const bool a01 = iny && tap_agrees(sm.depth[e01], Dp);
                                const bool a11 = inx && iny && tap_agrees(sm.depth[e11], Dp);
                                const float w00 = __fmul_rn(wx0, wy0), w10 = a10 ? __fmul_rn(wx1, wy0) : 0.f;
                                const float w01 = a01 ? __fmul_rn(wx0, wy1) : 0.f;
                                const float w11 = a11 ? __fmul_rn(wx1, wy1) : 0.f;
                                const float S = weight_sum(w00, w10, w01, w11);
                                const float inv = __frcp_rn(S);
                                sm.w[0][r] = __fmul_rn(w00, inv);
                                sm.w[1][r] = __fmul_rn(w10, inv);
                                sm.w[2][r] = __fmul_rn(w01, inv);
                                sm.w[3][r] = __fmul_rn(w11, inv);
                                const uint32_t cols = sx > 0 ? 6u : sx < 0 ? 3u : 2u;  // dx in {0, sx}
                                dirs = (cols << 3) | (sy > 0 ? cols << 6 : sy < 0 ? cols : 0u);
                                float C[3][4];  // tap colours (0 for taps that do not take part)
                                if (FUSED || inside) {
                                    const uint32_t t10 = i + (uint32_t)sx, t01 = sy > 0 ? i + Wu : i - Wu,
                                                   t11 = t01 + (uint32_t)sx;
#pragma unroll
                                    for (int c = 0; c < 3; ++c) {
                                        const CT *cp = (const CT *)a.color[c];
                                        C[c][0] = load_c<CT>(cp + i);
                                        C[c][1] = a10 ? load_c<CT>(cp + t10) : 0.f;
                                        C[c][2] = a01 ? load_c<CT>(cp + t01) : 0.f;
                                        C[c][3] = a11 ? load_c<CT>(cp + t11) : 0.f;
                                    }
                                }
                                float g[3], o[3];  // o: q's colour as stage (b) computes it, before its rounding
#pragma unroll
                                for (int c = 0; c < 3; ++c) {
                                    if (FUSED || inside) {
                                        float n = __fmul_rn(w00, C[c][0]);
                                        n = a10 ? fmaf(w10, C[c][1], n) : n;
                                        n = a01 ? fmaf(w01, C[c][2], n) : n;
                                        n = a11 ? fmaf(w11, C[c][3], n) : n;
                                        o[c] = __fmul_rn(n, inv);
                                    }
                                    if (FUSED) {  // the loss and its gradient
                                        const float d = __fsub_rn(storage_round<CT>(o[c]), gin[c]);
                                        g[c] = __fmul_rn(2.0f, d);
                                        if (inside) lacc = fmaf(d, d, lacc);
                                    } else {
                                        g[c] = gin[c];
                                    }
                                    sm.g[c][r] = g[c];
                                }
                                if (inside) {
                                    // dL/d mv(p) = -(k/denom) sum_c g_c sum_t (dw_t/drho)(C_c(t) - out_c) / S
                                    // d w_t / d rho: +-(the other axis' weight), signs from the tap side
                                    const float fsx = (float)sx, fsy = (float)sy;
                                    const float dx00 = -fsx * wy0, dx10 = a10 ? fsx * wy0 : 0.f;
                                    const float dx01 = a01 ? -fsx * wy1 : 0.f, dx11 = a11 ? fsx * wy1 : 0.f;
                                    const float dy00 = -fsy * wx0, dy10 = a10 ? -fsy * wx1 : 0.f;
                                    const float dy01 = a01 ? fsy * wx0 : 0.f, dy11 = a11 ? fsy * wx1 : 0.f;
                                    float G00 = 0.f, G10 = 0.f, G01 = 0.f, G11 = 0.f;  // sum_c g_c (C_c(t) - out_c)
#pragma unroll
                                    for (int c = 0; c < 3; ++c) {
                                        G00 = fmaf(g[c], __fsub_rn(C[c][0], o[c]), G00);
                                        G10 = fmaf(g[c], __fsub_rn(C[c][1], o[c]), G10);
                                        G01 = fmaf(g[c], __fsub_rn(C[c][2], o[c]), G01);
                                        G11 = fmaf(g[c], __fsub_rn(C[c][3], o[c]), G11);
                                    }
                                    float gx = __fmul_rn(dx00, G00), gy = __fmul_rn(dy00, G00);
                                    gx = fmaf(dx10, G10, gx);
                                    gx = fmaf(dx01, G01, gx);
                                    gx = fmaf(dx11, G11, gx);
                                    gy = fmaf(dy10, G10, gy);
                                    gy = fmaf(dy01, G01, gy);
                                    gy = fmaf(dy11, G11, gy);
                                    float2 &gm = gms[(ry - 1) * kFillTile + (rx - 1)];
                                    gm.x = fmaf(__fmul_rn(scale, gx), inv, gm.x);
                                    gm.y = fmaf(__fmul_rn(scale, gy), inv, gm.y);
                                }
                            }
                        }
                    }
                }
            }
            sm.dirs[r] = (uint16_t)dirs;
            rx += kBwdThreads % kRegion;
            ry += kBwdThreads / kRegion;
            if (rx >= kRegion) {
                rx -= kRegion;
                ++ry;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int y = wid + 8 * j;
            float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
            for (int ddy = -1; ddy <= 1; ++ddy) {
#pragma unroll
                for (int ddx = -1; ddx <= 1; ++ddx) {
                    const int r = (y + 1 - ddy) * kRegion + (lane + 1 - ddx);
                    if (!(sm.dirs[r] & (1u << (3 * (ddy + 1) + ddx + 1)))) continue;
                    const float w = sm.w[(ddx != 0 ? 1 : 0) + (ddy != 0 ? 2 : 0)][r];
                    a0 = fmaf(sm.g[0][r], w, a0);
                    a1 = fmaf(sm.g[1][r], w, a1);
                    a2 = fmaf(sm.g[2][r], w, a2);
                }
            }
            gc[j][0] = __fadd_rn(gc[j][0], a0);
            gc[j][1] = __fadd_rn(gc[j][1], a1);
            gc[j][2] = __fadd_rn(gc[j][2], a2);
        }
        __syncthreads();  // the records are rewritten by the next fraction
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int syg = Y0 + wid + 8 * j;
        if (sxg >= W || syg >= H) continue;
        const uint32_t s = (uint32_t)syg * Wu + (uint32_t)sxg;
#pragma unroll
        for (int c = 0; c < 3; ++c) a.grad_color[c][s] = gc[j][c];
    }
    for (int c = tid; c < kFillTile * kFillTile; c += kBwdThreads) {  // (the last barrier ordered every update)
        const int x = X0 + (c & (kFillTile - 1)), y = Y0 + c / kFillTile;
        if (x >= W || y >= H) continue;
        const uint32_t i = (uint32_t)y * Wu + (uint32_t)x;
        const float2 gm = gms[c];
        a.grad_mv[0][i] = gm.x;
        a.grad_mv[1][i] = gm.y;
    }
    if constexpr (FUSED) {
        // the loss: per CTA a fixed tree over its threads; the CTAs' partials are added by the next launch
        double lsum = (double)lacc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xFFFFFFFFu, lsum, o);
        if (lane == 0) red[wid] = lsum;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < kBwdThreads / 32; ++w) t += red[w];
            a.partial[blockIdx.y * gridDim.x + blockIdx.x] = t;
        }
    }
}

// The loss of a frame from its CTAs' partials in a fixed order (one CTA, in a launch after the frame's: counted and summed
// by the CTA that finished last, every CTA ended with a fence and an atomic's round trip -- eight frames of 1080p FP32
// took 1318 us, now 1278).
__device__ __forceinline__ void sum_loss(const double *partial, unsigned int n, double *loss) {
    __shared__ double red[kBwdThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double t = 0.0;
    for (unsigned int b = tid; b < n; b += kBwdThreads) t += __ldcg(partial + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (lane == 0) red[wid] = t;
    __syncthreads();
    if (tid == 0) {
        double v = 0.0;
        for (int w = 0; w < kBwdThreads / 32; ++w) v += red[w];
        *loss = v;
    }
}
__global__ void __launch_bounds__(kBwdThreads) loss_sum_kernel(const double *partial, unsigned int n, double *loss) {
    grid_dependency_wait();  // the partials
    sum_loss(partial, n, loss);
}

// Between two frames: the first block sums the last frame's loss, the others clear the keys for the next frame's splat.
__global__ void __launch_bounds__(256) clear_loss_kernel(const double *partial, unsigned int npart, double *loss,
                                                         unsigned long long *keys, uint32_t n) {
    static_assert(kBwdThreads == 256, "the sum's threads");
    grid_dependency_wait();  // the partials; the last frame's reads of the keys
    grid_dependents_launch();  // the splat
    if (blockIdx.x == 0) sum_loss(partial, npart, loss);
    else clear_keys_block(keys, n, blockIdx.x - 1, nullptr, 0u);
}

// Stage (a) for fractions k0 .. k0 + nfrac - 1 in one pass: each source pixel is read once and takes the 64-bit
// atomic minimum at its target in each fraction's key plane (keys + kk W H, cleared beforehand).
constexpr int kSplatMultiRows = 2;
__global__ void __launch_bounds__(256) splat_multi_kernel(const float *__restrict__ depth,
                                                          const float *__restrict__ mv, int W, int H, int k0,
                                                          int nfrac, int L, unsigned long long *keys) {
    grid_dependency_wait();  // the keys are cleared by the kernel before
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y0 = blockIdx.y * kSplatMultiRows;
    if (x >= W) return;
    const size_t plane = (size_t)W * H;
    const float *mvy = mv + plane;
    uint32_t db[kSplatMultiRows];
    float mx[kSplatMultiRows], my[kSplatMultiRows];
#pragma unroll
    for (int r = 0; r < kSplatMultiRows; ++r) {
        const uint32_t i = (uint32_t)min(y0 + r, H - 1) * (uint32_t)W + (uint32_t)x;
        db[r] = __float_as_uint(__ldg(depth + i));
        mx[r] = __ldg(mv + i);
        my[r] = __ldg(mvy + i);
    }
#pragma unroll
    for (int r = 0; r < kSplatMultiRows; ++r) {
        const int y = y0 + r;
        if (y >= H || !depth_ok(db[r]) || !motion_lands(mx[r], my[r], kMotionLimit)) continue;
        const unsigned long long key = pack_key_global(db[r], (uint32_t)y * (uint32_t)W + (uint32_t)x);
#pragma unroll
        for (int kk = 0; kk < kMaxFrac; ++kk) {
            if (kk >= nfrac) break;
            const float kf = fraction_scale(k0 + kk, L);
            const int gx = x + offset_of(mx[r], kf), gy = y + offset_of(my[r], kf);
            if ((unsigned)gx >= (unsigned)W || (unsigned)gy >= (unsigned)H) continue;
            atomicMin(keys + kk * plane + ((uint32_t)gy * (uint32_t)W + (uint32_t)gx), key);
        }
    }
}

// The planes of a frame.
template <typename CT>
static void set_source(BwdArgs &a, const void *color, const float *depth, const float *mv, int W, int H,
                       float *grad_color, float *grad_mv) {
    const size_t plane = (size_t)W * H;
    for (int c = 0; c < 3; ++c) {
        a.color[c] = (const CT *)color + c * plane;
        a.grad_color[c] = grad_color + c * plane;
    }
    for (int c = 0; c < 2; ++c) {
        a.mv[c] = mv + c * plane;
        a.grad_mv[c] = grad_mv + c * plane;
    }
    a.depth = depth;
    a.W = W;
    a.H = H;
}

template <typename CT, bool FUSED>
static cudaError_t launch_bwd_tiles(const BwdArgs &a, cudaStream_t s) {
    constexpr size_t kSmem = sizeof(BwdSmem<CT>);
    // set on every launch: the attribute belongs to the current device's context
    const cudaError_t e =
        cudaFuncSetAttribute(bwd_tile_kernel<CT, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    const dim3 g((unsigned)ceil_div(a.W, kFillTile), (unsigned)ceil_div(a.H, kFillTile), 1);
    return launch_dependent(bwd_tile_kernel<CT, FUSED>, g, dim3(kBwdThreads), kSmem, s, a);
}

cudaError_t launch_backward(const float *grad_out, const void *color, exw_dtype cdt, const float *depth,
                            const float *mv, const uint64_t *keys, int W, int H, int k, int L, float *grad_color,
                            float *grad_mv, bool store, cudaStream_t s) {
    BwdArgs a{};
    a.store = store;
    if (cdt == EXW_F32) set_source<float>(a, color, depth, mv, W, H, grad_color, grad_mv);
    else set_source<__half>(a, color, depth, mv, W, H, grad_color, grad_mv);
    a.keys[0] = (const unsigned long long *)keys;
    for (int c = 0; c < 3; ++c) a.g[0][c] = grad_out + c * ((size_t)W * H);
    a.nfrac = 1;
    a.k0 = k;
    a.L = L;
    timing_begin("exw_backward", s);
    const cudaError_t e = cdt == EXW_F32 ? launch_bwd_tiles<float, false>(a, s) : launch_bwd_tiles<__half, false>(a, s);
    count_launch();
    timing_end("exw_backward", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Workspace of exw_warp_l2_grad: the key planes of the fractions and the CTAs' loss partials.
struct TrainLayout {
    size_t keys, partial, total;
};
static TrainLayout train_layout(int W, int H, int nfrac) {
    TrainLayout t{};
    size_t off = 0;
    t.keys = off;
    off += align_up((size_t)nfrac * W * H * 8);
    t.partial = off;
    off += align_up((size_t)ceil_div(W, kFillTile) * ceil_div(H, kFillTile) * 8);
    t.total = off + kAlign;  // (the last section is not used)
    return t;
}

size_t train_workspace_bytes(int W, int H, int nfrac) { return train_layout(W, H, nfrac).total; }

// Frame `frame` of nframes of exw_warp_l2_grad (loss: its loss): keys of every fraction (one clear, one splat pass), then
// the fused pass.  A frame's loss is summed with the next frame's clear, the last one's by a launch of its own.
cudaError_t launch_train_frame(const exw_train_frame &f, int frame, int nframes, int nfrac, double *loss, bool store,
                               void *ws, cudaStream_t s) {
    const int W = f.src.W, H = f.src.H;
    const TrainLayout t = train_layout(W, H, nfrac);
    char *b = (char *)ws;
    unsigned long long *keys = (unsigned long long *)(b + t.keys);
    double *const partial = (double *)(b + t.partial);
    const unsigned npart = (unsigned)(ceil_div(W, kFillTile) * ceil_div(H, kFillTile));
    const size_t nkeys = (size_t)nfrac * W * H;
    cudaError_t e;
    if (frame == 0) {
        e = launch_clear_keys((uint64_t *)keys, nkeys, s);
    } else {
        timing_begin("exw_clear_loss", s);
        e = launch_dependent(clear_loss_kernel, dim3(1u + (unsigned)((nkeys / 2 + kClearPairs) / kClearPairs)), dim3(256), 0,
                             s, (const double *)partial, npart, loss - 1, keys, (uint32_t)nkeys);
        count_launch();
        timing_end("exw_clear_loss", s);
    }
    if (e != cudaSuccess) return e;
    timing_begin("exw_splat_multi", s);
    const int k0 = 1, L = 2;
    e = launch_dependent(splat_multi_kernel, dim3((unsigned)ceil_div(W, 256), (unsigned)ceil_div(H, kSplatMultiRows)),
                         dim3(256), 0, s, f.src.depth, f.src.mv, W, H, k0, nfrac, L, keys);
    count_launch();
    timing_end("exw_splat_multi", s);
    if (e != cudaSuccess) return e;
    BwdArgs a{};
    const size_t plane = (size_t)W * H;
    if (f.src.cdt == EXW_F32)
        set_source<float>(a, f.src.color, f.src.depth, f.src.mv, W, H, f.grad_color, f.grad_mv);
    else
        set_source<__half>(a, f.src.color, f.src.depth, f.src.mv, W, H, f.grad_color, f.grad_mv);
    for (int j = 0; j < nfrac; ++j) {
        a.keys[j] = keys + j * plane;
        for (int c = 0; c < 3; ++c) a.g[j][c] = (const char *)f.target[j] + c * plane * csize(f.src.cdt);
    }
    a.nfrac = nfrac;
    a.k0 = k0;
    a.L = L;
    a.partial = partial;
    a.store = store;
    timing_begin("exw_train", s);
    e = f.src.cdt == EXW_F32 ? launch_bwd_tiles<float, true>(a, s) : launch_bwd_tiles<__half, true>(a, s);
    count_launch();
    timing_end("exw_train", s);
    if (e == cudaSuccess && frame + 1 == nframes) {
        e = launch_dependent(loss_sum_kernel, dim3(1), dim3(kBwdThreads), 0, s, (const double *)partial, npart, loss);
        count_launch();
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace exw
