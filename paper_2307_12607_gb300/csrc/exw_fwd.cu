// exw_fwd.cu -- the staged kernels (exw_warp's gather, exw_fill_holes' fill) and the coarse fix-up; the fused
// forward pass is the persistent engine (exw_engine.cuh).
#include "exw_items.cuh"

namespace exw {

// Plans: one warp per target tile (the first stream of an engine launch is planned ahead of the launch).
// Small CTAs: a small frame's plans (240 at 640 x 360) spread over the SMs instead of sharing 15 of them, and a large
// frame's last wave is short (4K: one frame's plans 26.5 us in CTAs of 16 warps, 24.4 in these; 640 x 360 13.1 and 11.7,
// events around the launch).
constexpr int kPlanThreads = 64;
template <typename CT, int WX, int WY>
__global__ void __launch_bounds__(kPlanThreads, 16) plan_kernel(const __grid_constant__ TileParams p) {
    grid_dependency_wait();  // the bounds kernel before
    grid_dependents_launch();
    const int tile = blockIdx.x * (kPlanThreads / 32) + (threadIdx.x >> 5);
    if (tile < p.n5x * p.n5y) plan_tile<CT, WX, WY>(p, tile);
}

// The same with four warps a tile, for frames whose CTAs are all resident with room to spare (four per SM): there the
// kernel is one plan's chain of dependent loads and reductions, and the visits of the bounds tiles are the part of it that
// warps can share.  One frame with fill, whole call, one warp / two / four: 320 x 180 26.6 / 25.8 / 25.2 us, 640 x 360 FP32
// 34.4 / 34.2 / 33.6, FP16 under a turning camera 34.4 / 33.3 / 32.9, 960 x 540 (510 tiles) 46.2 / 45.4 / 45.7; 1280 x 720
// (920 tiles) 55.2 / 55.7 / 56.8: the larger frames' plans are bound by their number.
constexpr int kPlanShare = 4;
constexpr int kPlanShareTiles = 4 * 152;
template <typename CT, int WX, int WY>
__global__ void __launch_bounds__(32 * kPlanShare) plan_shared_kernel(const __grid_constant__ TileParams p) {
    __shared__ PlanShare<kPlanShare> sh;
    grid_dependency_wait();  // the bounds kernel before
    grid_dependents_launch();
    plan_tile<CT, WX, WY, kPlanShare>(p, blockIdx.x, &sh, threadIdx.x >> 5);
}

// ------------------------------------------------------------------------------------------------------------
// Staged stage (b): keys from global memory (exw_splat_motion), one fraction.  FILL also fills the tile (stage (c)),
// CARRY also writes the depth and motion the warped frame carries (exw_carry_motion).
//
// Nothing passes through shared memory but the fill's pyramid: a warp reads the keys of its rows and the
// rows above and below as coalesced lines, the crack rule's left and right neighbours come from the lanes beside
// (the outer lanes load theirs), and the winners' motion, depth and colour go through L1.  The pixels' three dependent
// round trips -- key, motion, taps -- are taken for a thread's rows together.
//
// Bound by issue and latency (about 350 instructions a pixel; DRAM at a fifth of its rate).  One recursive step at 1080p
// FP32: gather, fill and carry 42 + 20 + 16 us as three kernels (keys through shared memory, a division per key), 34 us
// as this one; the gather alone at 720p FP16 21 -> 15 us (events around each launch).
// ------------------------------------------------------------------------------------------------------------

// Source index -> (x, y) without a division: inv = floor(2^32 / W) + 1 (saturated), so the quotient is at most one too
// large for indices below 2^28 (W = 1: one too small).
__device__ __forceinline__ void split_index(uint32_t idx, uint32_t inv, int W, int &x, int &y) {
    y = (int)__umulhi(idx, inv);
    x = (int)idx - y * W;
    if (x < 0) {
        x += W;
        --y;
    } else if (x >= W) {
        x -= W;
        ++y;
    }
}

struct WarpArgs {
    TileParams p;
    uint32_t inv;       // floor(2^32 / W) + 1, saturated
    float *depth_out;   // CARRY: [H][W]
    float *mv_out;      // CARRY: [2][H][W]
};

// Two rows per thread: 40 registers, three CTAs of 16 warps per SM (six of 8 without the fill, which needs whole tiles).
// Four rows took 64 registers for 32 warps per SM: a recursive chain 161-168 us against 156.
template <bool FILL> constexpr int kWarpThreads = FILL ? kTileThreads : kTileThreads / 2;

template <typename CT, bool FILL, bool CARRY>
__global__ void __launch_bounds__(kWarpThreads<FILL>, 1536 / kWarpThreads<FILL>)
    warp_kernel(const __grid_constant__ WarpArgs a) {
    __shared__ __align__(16) unsigned char pyramid[FILL ? sizeof(TilePyramid) : 1];
    grid_dependency_wait();  // the splat before
    constexpr int kRows = kTileRows;
    const TileParams &p = a.p;
    const int W = p.W, H = p.H, k = p.k0, L = p.L;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gx = blockIdx.x * kFillTile + lane, gy0 = (blockIdx.y * (kWarpThreads<FILL> / 32) + w) * kRows;
    const uint32_t npix = (uint32_t)W * (uint32_t)H;
    const size_t plane = (size_t)W * H;
    // keys: rows gy0 - 1 .. gy0 + kRows of this column, and beside the warp's columns for its outer lanes; outside the
    // frame, and for an index outside it (a malformed key), empty
    uint32_t idx[kRows], dw[kRows + 2], side[kRows];
    auto key = [&](int x, int y, uint32_t &i) -> uint32_t {
        uint64_t v = kKeyEmpty;
        if ((unsigned)x < (unsigned)W && (unsigned)y < (unsigned)H)
            v = __ldg((const unsigned long long *)p.keys + ((uint32_t)y * (uint32_t)W + (uint32_t)x));
        i = (uint32_t)v;
        return i < npix ? key_dbits(v) : 0xFFFFFFFFu;
    };
    uint32_t skip;
    dw[0] = key(gx, gy0 - 1, skip);
#pragma unroll
    for (int r = 0; r < kRows; ++r) dw[r + 1] = key(gx, gy0 + r, idx[r]);
    dw[kRows + 1] = key(gx, gy0 + kRows, skip);
#pragma unroll
    for (int r = 0; r < kRows; ++r)
        side[r] = lane == 0 || lane == 31 ? key(lane == 0 ? gx - 1 : gx + 1, gy0 + r, skip) : 0u;
    const GlobalAcc<CT> acc(p.color, p.depth, p.mv, W, H);
    float mx[kRows], my[kRows];
    bool ok[kRows];
    uint8_t m[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const uint32_t dq = dw[r + 1];
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, dq, 1), dn = __shfl_down_sync(0xFFFFFFFFu, dq, 1);
        const bool in = gx < W && gy0 + r < H, empty = dq == 0xFFFFFFFFu;
        const bool crack = !empty && is_crack(dq, lane == 0 ? side[r] : up, lane == 31 ? side[r] : dn, dw[r], dw[r + 2]);
        m[r] = !in ? (uint8_t)0 : empty ? (uint8_t)EXW_MASK_EMPTY : crack ? (uint8_t)EXW_MASK_CRACK : (uint8_t)0;
        ok[r] = in && !empty && !crack;
        idx[r] = ok[r] ? idx[r] : 0u;  // a pixel without a winner gathers at the first one, unused
        mx[r] = acc.mx(idx[r]);
        my[r] = acc.my(idx[r]);
    }
    float4 c[kRows];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        int px, py, sx, sy;
        split_index(idx[r], a.inv, W, px, py);
        const float rx = residual(mx[r], k, L, gx - px, sx);
        const float ry = residual(my[r], k, L, gy0 + r - py, sy);
        const float wx1 = fabsf(rx), wy1 = fabsf(ry);
        const float wx0 = 1.0f - wx1, wy0 = 1.0f - wy1;
        const bool ex = sx != 0 && (unsigned)(px + sx) < (unsigned)W;
        const bool ey = sy != 0 && (unsigned)(py + sy) < (unsigned)H;
        const uint32_t i00 = idx[r];
        const uint32_t i10 = ex ? i00 + (uint32_t)sx : i00;
        const uint32_t ir = sy > 0 ? i00 + acc.stride() : i00 - acc.stride();
        const uint32_t i01 = ey ? ir : i00;
        const uint32_t i11 = (ex && ey) ? ir + (uint32_t)sx : i00;
        const float Dp = __uint_as_float(dw[r + 1]);
        const bool a10 = ex && tap_agrees(acc.d(i10), Dp);
        const bool a01 = ey && tap_agrees(acc.d(i01), Dp);
        const bool a11 = ex && ey && tap_agrees(acc.d(i11), Dp);
        const float w00 = __fmul_rn(wx0, wy0);
        const float w10 = a10 ? __fmul_rn(wx1, wy0) : 0.0f;
        const float w01 = a01 ? __fmul_rn(wx0, wy1) : 0.0f;
        const float w11 = a11 ? __fmul_rn(wx1, wy1) : 0.0f;
        const float inv = __frcp_rn(weight_sum(w00, w10, w01, w11));
        float v[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            float n = __fmul_rn(w00, acc.c(ch, i00));
            const float c10 = acc.c(ch, i10), c01 = acc.c(ch, i01), c11 = acc.c(ch, i11);
            n = a10 ? fmaf(w10, c10, n) : n;
            n = a01 ? fmaf(w01, c01, n) : n;
            n = a11 ? fmaf(w11, c11, n) : n;
            v[ch] = ok[r] ? storage_round<CT>(__fmul_rn(n, inv)) : 0.0f;
        }
        c[r] = make_float4(v[0], v[1], v[2], ok[r] ? 1.0f : 0.0f);
        if (gx >= W || gy0 + r >= H) continue;
        const uint32_t q = (uint32_t)(gy0 + r) * (uint32_t)W + (uint32_t)gx;
        p.out_mask[0][q] = m[r];
        if constexpr (CARRY) {  // the winner's depth (its key's bits) and motion; NaN and 0 on a hole
            a.depth_out[q] = ok[r] ? Dp : __int_as_float(0x7FC00000);
            a.mv_out[q] = ok[r] ? mx[r] : 0.0f;
            (a.mv_out + plane)[q] = ok[r] ? my[r] : 0.0f;
        }
    }
    unsigned int have = (1u << kRows) - 1u;
    if constexpr (FILL) have = fill_columns(p, *reinterpret_cast<TilePyramid *>(pyramid), c, m, 0, blockIdx.y * p.n5x + blockIdx.x);
    CT *oc = (CT *)p.out_color[0], *oc1 = oc + plane, *oc2 = oc1 + plane;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        if (gx >= W || gy0 + r >= H) continue;
        const uint32_t q = (uint32_t)(gy0 + r) * (uint32_t)W + (uint32_t)gx;
        if (have & (1u << r)) {
            oc[q] = to_storage<CT>(c[r].x);
            oc1[q] = to_storage<CT>(c[r].y);
            oc2[q] = to_storage<CT>(c[r].z);
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// Staged stage (c): pull-push of an existing colour + mask, in place.
// ------------------------------------------------------------------------------------------------------------
template <typename CT>
__global__ void __launch_bounds__(kTileThreads, 3) fill_tiles_kernel(const __grid_constant__ TileParams p) {
    __shared__ TilePyramid pyramid;
    grid_dependency_wait();
    grid_dependents_launch();  // the coarse pass
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gx = blockIdx.x * kFillTile + lane, gy0 = blockIdx.y * kFillTile + kTileRows * w;
    const size_t plane = (size_t)p.W * p.H;
    CT *oc = (CT *)p.out_color[0];
    float4 c[kTileRows];
    uint8_t m[kTileRows];
#pragma unroll
    for (int r = 0; r < kTileRows; ++r) {
        c[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        m[r] = 1;
        if (gx < p.W && gy0 + r < p.H) {
            const size_t q = (size_t)((gy0 + r) * p.W + gx);
            m[r] = __ldg(p.mask_in + q);
            c[r] = make_float4(to_f<CT>(oc[q]), to_f<CT>(oc[plane + q]), to_f<CT>(oc[2 * plane + q]), 0.0f);
        }
    }
#pragma unroll
    for (int r = 0; r < kTileRows; ++r) {  // (a hole holds anything)
        if (m[r] != 0) c[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        else c[r].w = 1.0f;
    }
    const unsigned int have = fill_columns(p, pyramid, c, m, 0, blockIdx.y * p.n5x + blockIdx.x);
#pragma unroll
    for (int r = 0; r < kTileRows; ++r) {
        if (gx >= p.W || gy0 + r >= p.H || m[r] == 0 || !(have & (1u << r))) continue;
        const size_t q = (size_t)((gy0 + r) * p.W + gx);
        oc[q] = to_storage<CT>(c[r].x);
        oc[plane + q] = to_storage<CT>(c[r].y);
        oc[2 * plane + q] = to_storage<CT>(c[r].z);
    }
}

// The coarse values of a fill's tiles without a valid pixel (one CTA; nothing to do in most frames), then the fix-up: every
// such tile takes its own.  A launch of its own, after the tiles: with the tiles counted and the pass run by the CTA that
// finishes the last one, every CTA stayed on the SM for a fence and an atomic's round trip after its stores -- three
// recursive steps at 1080p FP32 took 138.7 us (120 without the count, and without the pass), now 121.0; splat, warp and
// fill at 720p FP16 27.3 and 25.5.
__global__ void __launch_bounds__(1024) coarse_kernel(const __grid_constant__ TileParams p) {
    grid_dependency_wait();  // the tiles' nodes
    grid_dependents_launch();  // the fix-up
    coarse_pass(p);
}
template <typename CT>
__global__ void __launch_bounds__(kThreads) fixup_kernel(const __grid_constant__ TileParams p) {
    grid_dependency_wait();  // the coarse values
    fixup_slice<CT>(p, blockIdx.x, gridDim.x, (int)threadIdx.x, (int)blockDim.x);
}

// ------------------------------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------------------------------
static dim3 tile_grid(const TileParams &p) { return dim3((unsigned)p.n5x, (unsigned)p.n5y, 1); }

cudaError_t launch_plan(const TileParams &p, exw_dtype cdt, int shape, cudaStream_t s) {
    const int ntiles = p.n5x * p.n5y;
    const unsigned g = (unsigned)ceil_div(ntiles, kPlanThreads / 32);
    timing_begin("exw_plan", s);
    using S0 = WinShape<0>;
    using S1 = WinShape<1>;
    const bool share = ntiles <= kPlanShareTiles;
    void (*k)(TileParams);
    if (share)
        k = shape == 0 ? (cdt == EXW_F32 ? plan_shared_kernel<float, S0::xf32, S0::yf32>
                                         : plan_shared_kernel<__half, S0::xf16, S0::yf16>)
                       : (cdt == EXW_F32 ? plan_shared_kernel<float, S1::xf32, S1::yf32>
                                         : plan_shared_kernel<__half, S1::xf16, S1::yf16>);
    else
        k = shape == 0 ? (cdt == EXW_F32 ? plan_kernel<float, S0::xf32, S0::yf32> : plan_kernel<__half, S0::xf16, S0::yf16>)
                       : (cdt == EXW_F32 ? plan_kernel<float, S1::xf32, S1::yf32> : plan_kernel<__half, S1::xf16, S1::yf16>);
    const cudaError_t e = launch_dependent(k, dim3(share ? (unsigned)ntiles : g), dim3(share ? 32 * kPlanShare : kPlanThreads),
                                           0, s, p);
    count_launch();
    timing_end("exw_plan", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename CT>
static cudaError_t launch_warp_as(const WarpArgs &a, bool fill, bool carry, cudaStream_t s) {
    void (*k)(WarpArgs) = fill ? (carry ? warp_kernel<CT, true, true> : warp_kernel<CT, true, false>)
                               : (carry ? warp_kernel<CT, false, true> : warp_kernel<CT, false, false>);
    const int threads = fill ? kWarpThreads<true> : kWarpThreads<false>;
    const dim3 g((unsigned)ceil_div(a.p.W, kFillTile), (unsigned)ceil_div(a.p.H, threads / 32 * kTileRows), 1);
    return launch_dependent(k, g, dim3(threads), 0, s, a);
}

cudaError_t launch_warp(const TileParams &p, exw_dtype cdt, bool fill, float *depth_out, float *mv_out,
                        cudaStream_t s) {
    WarpArgs a{};
    a.p = p;
    const uint64_t inv = (1ull << 32) / (uint32_t)p.W + 1u;
    a.inv = inv > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)inv;
    a.depth_out = depth_out;
    a.mv_out = mv_out;
    const bool carry = depth_out != nullptr;
    timing_begin("exw_warp_tiles", s);
    const cudaError_t e =
        cdt == EXW_F32 ? launch_warp_as<float>(a, fill, carry, s) : launch_warp_as<__half>(a, fill, carry, s);
    count_launch();
    timing_end("exw_warp_tiles", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_fill_tiles(const TileParams &p, exw_dtype cdt, cudaStream_t s) {
    timing_begin("exw_fill_tiles", s);
    void (*k)(TileParams) = cdt == EXW_F32 ? fill_tiles_kernel<float> : fill_tiles_kernel<__half>;
    const cudaError_t e = launch_dependent(k, tile_grid(p), dim3(kTileThreads), 0, s, p);
    count_launch();
    timing_end("exw_fill_tiles", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_fixup(const TileParams &p, exw_dtype cdt, cudaStream_t s) {
    const int n5 = p.n5x * p.n5y;
    const unsigned g = (unsigned)(n5 < 304 ? n5 : 304);
    timing_begin("exw_fixup", s);
    cudaError_t e = launch_dependent(coarse_kernel, dim3(1), dim3(1024), 0, s, p);
    count_launch();
    void (*k)(TileParams) = cdt == EXW_F32 ? fixup_kernel<float> : fixup_kernel<__half>;
    if (e == cudaSuccess) e = launch_dependent(k, dim3(g), dim3(kThreads), 0, s, p);
    count_launch();
    timing_end("exw_fixup", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace exw
