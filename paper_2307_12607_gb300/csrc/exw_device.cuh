// exw_device.cuh -- device-side building blocks of the warping fast path (sm_103a).
//
// What the staged kernels (exw_splat_motion, exw_warp, exw_fill_holes), the engine and the training pass compute per
// pixel, so that they agree bit for bit: offsets, residuals, keys, the crack and tap rules, the weights' sum, roundings
// and means.  The taps themselves are read and weighted in three places, each in its kernel's layout and all in the
// same order: warp_kernel (exw_fwd.cu), gather_pixel (exw_engine.cuh), phase 1 of bwd_tile_kernel (exw_bwd.cu).  Source
// data is read through an accessor (global memory or a staged shared-memory window).
#pragma once

#include <cstdint>
#include <cuda_fp16.h>

namespace exw {

constexpr uint64_t kKeyEmpty = ~0ull;
constexpr int kFillTile = 32;          // fill tile side: pyramid levels 1..5 live in shared memory
constexpr int kRegion = kFillTile + 2; // fill tile plus a one-pixel ring (the crack rule reads 4-neighbours)
constexpr int kRegionN = kRegion * kRegion;
constexpr int kBoundsBlock = 8;        // side of the motion-bounds tiles
constexpr int kMaxFrac = 3;

// Grids launched by launch_dependent: wait until the grids before this one on the stream have completed and their
// writes are visible (at once for a grid launched without programmatic serialisation), and let the next grid be
// scheduled (it waits in turn before touching memory).  Only a kernel that another one of the same entry point follows
// lets it be scheduled early, and after its own wait: what a kernel reads through the read-only path was then complete
// before its grid began, whoever launched the kernels before.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// ------------------------------------------------------------------------------------------------------------
// Validity of source pixels
// ------------------------------------------------------------------------------------------------------------

// Positive finite depth (subnormals included): bits in [1, 0x7F7FFFFF].
__device__ __forceinline__ bool depth_ok(uint32_t dbits) { return (dbits - 1u) < 0x7F7FFFFFu; }
__device__ __forceinline__ bool finite_bits(uint32_t b) { return (b & 0x7F800000u) != 0x7F800000u; }

__device__ __forceinline__ float pow2_neg(int n) {  // 2^-n for n in [-126, 126]
    return __int_as_float((127 - n) << 23);
}

// ------------------------------------------------------------------------------------------------------------
// Exact target offset off = floor(1/2 + k * mv / 2^L).
//
// kf = k / 2^L is exact in float, and so is the product inside a fused multiply-add.  Adding 2^22 * 3/2 + 1/2 rounded
// down leaves a float in [2^22, 2^23), whose last bit is worth 1/2: floor(2 (kf mv + 1/2)) / 2 above the base, and half
// of that, rounded down once more by the shift, is floor(kf mv + 1/2).  Three instructions per axis and fraction and
// nothing shared between them (the significand and exponent taken apart cost some ten per axis before the first).
// Holds while |kf mv + 1/2| < 2^21; a motion of 2^20 pixels or more lands in no frame for any k >= 1 (|off| >= 2^14).
// Engine time with the parts taken apart and with this: 4 frames of 1080p FP16 under a turning camera 423 and 392 us, the
// 60-frame 1080p sequence 3816 and 3708, 48 streams 5253 and 5072; 8 training frames 1371 and 1319 us.
// ------------------------------------------------------------------------------------------------------------
constexpr float kOffsetBias = 6291456.5f;           // 3/2 2^22 + 1/2
constexpr int kOffsetBase = 0x4AC00000 >> 1;        // half the bits of 3/2 2^22
constexpr float kMotionLimit = 1048576.0f;          // 2^20

__device__ __forceinline__ float fraction_scale(int k, int L) { return (float)k * pow2_neg(L); }
__device__ __forceinline__ int offset_raw(float mv, float kf) {  // the offset plus kOffsetBase
    return __float_as_int(__fmaf_rd(kf, mv, kOffsetBias)) >> 1;
}
__device__ __forceinline__ int offset_of(float mv, float kf) { return offset_raw(mv, kf) - kOffsetBase; }
// The motions that can land somewhere: below 2^20 for k >= 1; k = 0 (staged entry points) leaves a pixel where it is
// for any motion below 2^(23 + L), the range the offset is defined on.  A NaN is in neither.
__device__ __forceinline__ float motion_limit(int k, int L) { return k == 0 ? __int_as_float((150 + L) << 23) : kMotionLimit; }
__device__ __forceinline__ bool motion_lands(float mx, float my, float limit) {
    return fabsf(mx) < limit && fabsf(my) < limit;
}

// Residual rho = t - k*mv/2^L for a winner displaced by the whole-pixel offset t (|rho| <= 1/2).  One fused
// multiply-add computes the exact value rounded once, i.e. the correctly rounded residual.  Its sign is exact
// except when |rho| < 2^-150 rounds to zero, which needs t = 0 and a subnormal mv; with t = 0 the sign is that of
// -mv.  sgn is -1, 0 or +1.
__device__ __forceinline__ float residual(float mv, int k, int L, int t, int &sgn) {
    const float r = fmaf(-(float)k * pow2_neg(L), mv, (float)t);
    const float s = t == 0 && k != 0 ? -mv : r;
    sgn = (s > 0.0f) - (s < 0.0f);
    return r;
}

// Key packings.  In global memory: (depth bits << 32) | (y * W + x).  In shared memory the low word is
// (y << 14) | x, which orders exactly like y * W + x for x < 2^14 and needs no division to unpack.
__device__ __forceinline__ uint64_t pack_key_local(uint32_t dbits, int x, int y) {
    return ((uint64_t)dbits << 32) | (uint32_t)((y << 14) | x);
}
__device__ __forceinline__ uint64_t pack_key_global(uint32_t dbits, uint32_t idx) {
    return ((uint64_t)dbits << 32) | idx;
}
__device__ __forceinline__ uint32_t key_dbits(uint64_t key) { return (uint32_t)(key >> 32); }

// n keys (8-byte aligned) to empty, in 16-byte stores (the first and last key alone where they do not pair up), and
// zero_words words of a frame header to zero.  A block clears kClearPairs pairs, all of a thread's stores at immediate
// offsets: 6.2 M keys took 41 instructions a store in a grid-stride loop.
constexpr int kClearPerThread = 8, kClearPairs = 256 * kClearPerThread;
__device__ __forceinline__ void clear_keys_block(unsigned long long *keys, uint32_t n, uint32_t block, uint32_t *zero,
                                                 uint32_t zero_words) {
    const uint32_t head = ((uintptr_t)keys & 15u) ? 1u : 0u, npair = (n - head) / 2;
    const uint32_t first = block * (uint32_t)kClearPairs + threadIdx.x;
    ulonglong2 *pairs = reinterpret_cast<ulonglong2 *>(keys + head) + first;
    const ulonglong2 empty = make_ulonglong2(kKeyEmpty, kKeyEmpty);
    if (first + 256 * (kClearPerThread - 1) < npair) {
#pragma unroll
        for (int u = 0; u < kClearPerThread; ++u) pairs[256 * u] = empty;
    } else {
#pragma unroll
        for (int u = 0; u < kClearPerThread; ++u)
            if (first + 256 * u < npair) pairs[256 * u] = empty;
    }
    if (block != 0u) return;
    if (threadIdx.x == 0 && head) keys[0] = kKeyEmpty;
    if (threadIdx.x == 1 && head + 2 * npair < n) keys[n - 1] = kKeyEmpty;
    for (uint32_t i = threadIdx.x; i < zero_words; i += blockDim.x) zero[i] = 0u;
}

// ------------------------------------------------------------------------------------------------------------
// Colour types
// ------------------------------------------------------------------------------------------------------------
template <typename CT> __device__ __forceinline__ float to_f(CT v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }

template <typename CT> __device__ __forceinline__ float load_c(const CT *p) { return to_f<CT>(__ldg(p)); }

template <typename CT> __device__ __forceinline__ CT to_storage(float v);
template <> __device__ __forceinline__ float to_storage<float>(float v) { return v; }
template <> __device__ __forceinline__ __half to_storage<__half>(float v) { return __float2half_rn(v); }

template <typename CT> __device__ __forceinline__ float storage_round(float v) { return v; }
template <> __device__ __forceinline__ float storage_round<__half>(float v) {
    return __half2float(__float2half_rn(v));
}

// ------------------------------------------------------------------------------------------------------------
// Source accessors: global memory, or a shared-memory window [x0, x0 + WX) x [y0, y0 + WY) staged by TMA.
// ------------------------------------------------------------------------------------------------------------
template <typename CT>
struct GlobalAcc {  // 32-bit element indices (a plane has at most 2^28), so an address is one wide multiply-add
    const CT *col[3];
    const float *depth, *mvx, *mvy;
    uint32_t W;
    __device__ __forceinline__ GlobalAcc(const void *color, const float *depth_, const float *mv, int W_, int H)
        : depth(depth_), mvx(mv), W((uint32_t)W_) {
        const size_t plane = (size_t)W_ * H;
        mvy = mv + plane;
#pragma unroll
        for (int c = 0; c < 3; ++c) col[c] = (const CT *)color + c * plane;
    }
    __device__ __forceinline__ uint32_t at(int x, int y) const { return (uint32_t)y * W + (uint32_t)x; }
    __device__ __forceinline__ uint32_t stride() const { return W; }
    __device__ __forceinline__ int safe_x() const { return 0; }  // a pixel every access may use
    __device__ __forceinline__ int safe_y() const { return 0; }
    __device__ __forceinline__ float d(uint32_t i) const { return __ldg(depth + i); }
    __device__ __forceinline__ float mx(uint32_t i) const { return __ldg(mvx + i); }
    __device__ __forceinline__ float my(uint32_t i) const { return __ldg(mvy + i); }
    __device__ __forceinline__ float c(int ch, uint32_t i) const { return load_c<CT>(col[ch] + i); }
};

template <typename CT, int WX, int WY>
struct Window {  // TMA destinations: [y][x] per plane
    float depth[WY * WX];
    float mv[2][WY * WX];
    CT col[3][WY * WX];
};

template <typename CT, int WX, int WY>
struct WinAcc {
    const Window<CT, WX, WY> *w;
    int x0, y0;
    __device__ __forceinline__ int at(int x, int y) const { return (y - y0) * WX + (x - x0); }
    __device__ __forceinline__ int stride() const { return WX; }
    __device__ __forceinline__ int safe_x() const { return x0 + 1; }  // its taps stay inside the window
    __device__ __forceinline__ int safe_y() const { return y0 + 1; }
    __device__ __forceinline__ float d(int i) const { return w->depth[i]; }
    __device__ __forceinline__ float mx(int i) const { return w->mv[0][i]; }
    __device__ __forceinline__ float my(int i) const { return w->mv[1][i]; }
    __device__ __forceinline__ float c(int ch, int i) const { return to_f<CT>(w->col[ch][i]); }
};

// ------------------------------------------------------------------------------------------------------------
// Stage (b) for one target pixel
// ------------------------------------------------------------------------------------------------------------

// Crack rule: at least 3 non-empty 4-neighbours nearer than the target by more than D_q / 32.  Only the depth
// words of the keys matter: an empty key's word (all ones) is a NaN and never counts.  32 * (Dq - Dn) > Dq is
// exact in float: within a factor of 2 the difference is exact (Sterbenz), outside it both sides are far from
// the threshold.
__device__ __forceinline__ bool is_crack(uint32_t dq, uint32_t d0, uint32_t d1, uint32_t d2, uint32_t d3) {
    const float Dq = __uint_as_float(dq);
    int c = 0;
    c += (32.0f * (Dq - __uint_as_float(d0)) > Dq);
    c += (32.0f * (Dq - __uint_as_float(d1)) > Dq);
    c += (32.0f * (Dq - __uint_as_float(d2)) > Dq);
    c += (32.0f * (Dq - __uint_as_float(d3)) > Dq);
    return c >= 3;
}

// Tap agreement |D(t) - D(p)| <= D(p) / 32, exact in float by the same argument.  A NaN, infinite or
// non-positive tap depth fails it.
__device__ __forceinline__ bool tap_agrees(float Dt, float Dp) { return 32.0f * fabsf(Dt - Dp) <= Dp; }

// The products and sums of the gather are written with explicit round-to-nearest intrinsics (never fused into an
// FMA by the compiler), so every path that computes a gather -- the per-tile passes, the engine's window, uniform
// and smooth tiles, the recomputation in the fused training pass -- gets the same bits in any context.
// Sum of the bilinear weights of the participating taps (0 for the others), in the order 00, 10, 01, 11.
__device__ __forceinline__ float weight_sum(float w00, float w10, float w01, float w11) {
    return __fadd_rn(__fadd_rn(__fadd_rn(w00, w10), w01), w11);
}

// ------------------------------------------------------------------------------------------------------------
// Pull-push inside one 32 x 32 fill tile.  Tiles are aligned to 32, so every ancestor up to level 5 of a tile pixel
// is computed from that tile alone; out-of-frame pixels are invalid, which reproduces the ceil-halving level sizes.
// ------------------------------------------------------------------------------------------------------------

// Mean of the valid children, taken in the order (0,0),(0,1),(1,0),(1,1) (row, column); .w = validity.
__device__ __forceinline__ float4 mean4(float4 c0, float4 c1, float4 c2, float4 c3) {
    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
    int cnt = 0;
    if (c0.w != 0.0f) { a0 += c0.x; a1 += c0.y; a2 += c0.z; ++cnt; }
    if (c1.w != 0.0f) { a0 += c1.x; a1 += c1.y; a2 += c1.z; ++cnt; }
    if (c2.w != 0.0f) { a0 += c2.x; a1 += c2.y; a2 += c2.z; ++cnt; }
    if (c3.w != 0.0f) { a0 += c3.x; a1 += c3.y; a2 += c3.z; ++cnt; }
    if (cnt == 0) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float inv = cnt == 1 ? 1.0f : cnt == 2 ? 0.5f : cnt == 3 ? (1.0f / 3.0f) : 0.25f;
    return make_float4(__fmul_rn(a0, inv), __fmul_rn(a1, inv), __fmul_rn(a2, inv), 1.0f);
}

// The same where every .w is 0 or 1 and an invalid node's colour is 0 (all but the coarse levels): adding the zeros of
// the invalid children changes no bit, so nothing is selected.
// A third fewer instructions a node: a recursive chain at 1080p FP32 147.7 -> 139.6 us, splat + warp + fill at 720p FP16
// 29.2 -> 27.4.
__device__ __forceinline__ float4 mean4_01(float4 c0, float4 c1, float4 c2, float4 c3) {
    const float n = (c0.w + c1.w) + (c2.w + c3.w);
    const float inv = n == 1.0f ? 1.0f : n == 2.0f ? 0.5f : n == 3.0f ? (1.0f / 3.0f) : 0.25f;
    return make_float4(__fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(0.0f, c0.x), c1.x), c2.x), c3.x), inv),
                       __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(0.0f, c0.y), c1.y), c2.y), c3.y), inv),
                       __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(0.0f, c0.z), c1.z), c2.z), c3.z), inv), fminf(n, 1.0f));
}

__device__ __forceinline__ float4 shfl4_xor(float4 v, int m) {
    return make_float4(__shfl_xor_sync(0xFFFFFFFFu, v.x, m), __shfl_xor_sync(0xFFFFFFFFu, v.y, m),
                       __shfl_xor_sync(0xFFFFFFFFu, v.z, m), __shfl_xor_sync(0xFFFFFFFFu, v.w, m));
}

__device__ __forceinline__ float4 shfl4_idx(float4 v, int src) {
    return make_float4(__shfl_sync(0xFFFFFFFFu, v.x, src), __shfl_sync(0xFFFFFFFFu, v.y, src),
                       __shfl_sync(0xFFFFFFFFu, v.z, src), __shfl_sync(0xFFFFFFFFu, v.w, src));
}

// Ordered encoding of a non-NaN float for unsigned atomicMax: larger float <-> larger code, and 0 is below every
// code (the "nothing seen" value).
__device__ __forceinline__ uint32_t float_order(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float float_unorder(uint32_t c) {
    return __uint_as_float((c & 0x80000000u) ? (c & 0x7FFFFFFFu) : ~c);
}

}  // namespace exw
