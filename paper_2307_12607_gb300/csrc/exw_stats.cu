// exw_stats.cu -- frame statistics of the decision stage: the motion-variance features Var_x(F_mv), Var_y(F_mv) of
// the environment vector (Sec. IV-C, Eq. 1), and the colour MSE (PSNR) and SSIM of the reward (Sec. IV-C, Eq. 3).
//
// The sums keep FP64 accuracy without the FP64 pipe, which on this part takes one lane's operation per SM clock (a
// warp instruction 32 clocks; the FP32 pipe takes 128 lanes): a thread forms each difference and square as a pair of
// floats (two-difference, fused multiply-add residuals) and adds them error-free (two-sum) into words of falling size;
// every kFoldValues values these are folded into a second set.  Short inputs, and differences whose squares would
// leave float's range, go through FP64 value by value.  The error is at most that of
// sums on the FP64 pipe, whether the values differ or repeat (the same operations in the same order on a host, 40
// fields of each kind at 1080p and above, largest relative error: flat image pairs 2.4e-16 and 7.9e-15 in FP64, one
// motion per object 2.5e-16 and 4.7e-16, stripes of four motions 1.2e-15 and 6.4e-15).
//
// Every grid is a function of the sizes only and every sum has a fixed order: results are deterministic and do not
// depend on the GPU.  The blocks' partials are added by a one-block kernel launched behind them with programmatic
// serialisation, so no counter in the workspace has to be cleared first.
#include "exw_device.cuh"
#include "exw_internal.h"

namespace exw {
namespace {

// One block per SM of a 152-SM part: with 256 blocks (the earlier grid) 104 SMs had two and 48 one.
constexpr int kStatBlocks = 152, kStatThreads = 512;
constexpr int kFoldValues = 32;             // values a thread adds to its short sums between two folds
constexpr size_t kWideValues = 1u << 14;    // inputs shorter than this are summed in FP64 throughout
constexpr int kSumThreads = 256;            // the kernel that adds the partials
constexpr int kMaxPartials = 1280;          // doubles in the workspace

struct StatWs {
    double part[kMaxPartials];
    unsigned int reserved;  // keeps the workspace at its size
};

// ------------------------------------------------------------------------------------------------------------
// Error-free arithmetic on floats (Knuth's two-sum, Dekker's product by fused multiply-add).
// ------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void two_diff(float a, float b, float &h, float &l) {  // a - b = h + l exactly
    h = __fsub_rn(a, b);
    const float bv = __fsub_rn(a, h), av = __fadd_rn(h, bv);
    l = __fadd_rn(__fsub_rn(a, av), __fsub_rn(bv, b));
}

__device__ __forceinline__ float two_sum(float &s, float x) {  // s += x, returns the error of the addition
    const float t = __fadd_rn(s, x);
    const float xv = __fsub_rn(t, s), sv = __fsub_rn(t, xv);
    const float e = __fadd_rn(__fsub_rn(s, sv), __fsub_rn(x, xv));
    s = t;
    return e;
}

// A sum in words of falling size: s, the errors of its additions c, the errors of c's additions d.  What is left to
// plain additions is some 2^-72 of the sum.
struct Words {
    float s = 0.0f, c = 0.0f, d = 0.0f;
    __device__ __forceinline__ void small(float x) { d = __fadd_rn(d, two_sum(c, x)); }
    __device__ __forceinline__ void join(const Words &o) {
        small(two_sum(s, o.s));
        small(o.c);
        d = __fadd_rn(d, o.d);
    }
};

// The words of a short sum hold one kind of term each, and every addition to them is error-free down to k: a plain
// addition to any word but that rounds by up to 2^-48 of the sum, and where the values repeat -- one motion per object,
// a flat image -- every thread rounds the same way, so that nothing averages out.
struct LinearSum {  // of h + l: the short sum and the one it is folded into
    Words near, far;
    float k = 0.0f;
    __device__ __forceinline__ void add(float h, float l) {
        k = __fadd_rn(k, two_sum(near.c, two_sum(near.s, h)));
        k = __fadd_rn(k, two_sum(near.d, l));
    }
    __device__ __forceinline__ void fold() {
        far.small(near.d);
        near.d = k;
        far.join(near);
        near = Words{};
        k = 0.0f;
    }
};

struct FloatSum {  // of floats that are themselves rounded results: their sum to some 2^-48
    Words near, far;
    __device__ __forceinline__ void add(float x, float f) {  // x - f x, f x being smaller than x's last bit
        near.c = __fadd_rn(near.c, fmaf(-f, x, two_sum(near.s, x)));
    }
    __device__ __forceinline__ void fold() {
        far.join(near);
        near = Words{};
    }
};

// Of (h + l)^2 = p + e + q + r + l^2 with p = fl(h h), q = fl(2 h l) and their exact residuals e, r.
struct SquareSum {
    Words near, far;
    float g = 0.0f, k = 0.0f;
    __device__ __forceinline__ void add(float h, float l) {
        const float p = __fmul_rn(h, h), h2 = 2.0f * h, q = __fmul_rn(h2, l);
        const float r = fmaf(l, l, fmaf(h2, l, -q));
        k = __fadd_rn(k, two_sum(near.c, two_sum(near.s, p)));
        k = __fadd_rn(k, __fadd_rn(two_sum(near.d, fmaf(h, h, -p)), r));
        k = __fadd_rn(k, two_sum(g, q));
    }
    __device__ __forceinline__ void fold() {
        far.small(near.d);
        far.small(g);
        near.d = k;
        far.join(near);
        near = Words{};
        g = k = 0.0f;
    }
};

// Differences whose squares, their residuals and 2^28 squares added up stay inside float's range (zero included); NaN and infinities
// are not in it.  2^-39: the square's residual, down to 2^-48 of it, is still a multiple of 2^-149.
__device__ __forceinline__ bool float_range(float h) {
    const float m = fabsf(h);
    return m == 0.0f || (m >= 0x1p-39f && m < 0x1p40f);
}

// d += x - y and q += (x - y)^2 in FP64 (not inlined: the FP64 instructions of the rare values stay off the others'
// path).
__device__ __noinline__ void wide_square(float x, double y, double &d, double &q) {
    const double v = (double)x - y;
    d += v;
    q = fma(v, v, q);
}

constexpr int kStatWarps = kStatThreads / 32;
static_assert(kStatWarps <= 32, "one lane per warp in the last step");

// Block sum of the threads' words: a warp tree in FP32 (its roundings are independent over the thousands of warps of a
// grid), then one FP64 tree over the warps' words -- FP64 trees in every warp would take 160 times 32 clocks.  Every
// lane of warp 0 gets the sum.  sh: kStatWarps words, used by one sum only.  One block barrier.
__device__ __forceinline__ double block_words(Words v, Words *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Words x;
        x.s = __shfl_xor_sync(0xFFFFFFFFu, v.s, o);
        x.c = __shfl_xor_sync(0xFFFFFFFFu, v.c, o);
        x.d = __shfl_xor_sync(0xFFFFFFFFu, v.d, o);
        v.join(x);
    }
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        const Words x = lane < kStatWarps ? sh[lane] : Words{};
        t = (double)x.s + ((double)x.c + (double)x.d);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    }
    return t;
}

// Block sum of one double per thread (the values that went through FP64): thread 0 gets it.
__device__ __noinline__ double block_wide(double v, double *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kStatWarps; ++i) t += sh[i];
    return t;
}

// Sum of n partials, fixed order, by the calling warp (lane i takes i, i + 32, ...).
__device__ __forceinline__ double warp_sum(const double *p, int n) {
    double v = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) v += __ldcg(p + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// N consecutive values in one load where the addresses allow it (16 bytes), else one.
template <typename CT, int N> struct Pack { CT v[N]; };
template <typename CT, int N> __device__ __forceinline__ Pack<CT, N> load_pack(const CT *p) {
    Pack<CT, N> r;
    if constexpr (N == 1) {
        r.v[0] = __ldg(p);
    } else {
        static_assert(sizeof(r) == 16, "one 16-byte load");
        const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p));
        memcpy(&r, &u, 16);
    }
    return r;
}

// ------------------------------------------------------------------------------------------------------------
// Motion variance
// ------------------------------------------------------------------------------------------------------------

constexpr int kShiftScan = 1024;

// Shift of the variance's sums: the first finite vector among the first kShiftScan pixels (0 when there is none);
// every block finds the same one.  Any value of the field keeps the shifted sums' cancellation small.
// By warp 0 of a block, into its shared memory (a block barrier comes before the others read it).
__device__ __forceinline__ void find_shift(const float *__restrict__ mv, size_t n, float *shift) {
    if (threadIdx.x >= 32) return;
    int first = kShiftScan;
    for (int i0 = 0; i0 < kShiftScan && (size_t)i0 < n && first == kShiftScan; i0 += 32) {
        const int k = i0 + (int)threadIdx.x;
        const float x = (size_t)k < n ? __ldg(mv + k) : __int_as_float(0x7FC00000);
        const float y = (size_t)k < n ? __ldg(mv + n + k) : __int_as_float(0x7FC00000);
        const unsigned int b = __ballot_sync(0xFFFFFFFFu, isfinite(x) && isfinite(y));
        if (b) {
            const int src = __ffs(b) - 1;
            first = i0 + src;
            const float sx = __shfl_sync(0xFFFFFFFFu, x, src), sy = __shfl_sync(0xFFFFFFFFu, y, src);
            if (threadIdx.x == 0) {
                shift[0] = sx;
                shift[1] = sy;
            }
        }
    }
    if (threadIdx.x == 0 && first == kShiftScan) shift[0] = shift[1] = 0.0f;
}

// Inputs shorter than kWideValues: a vector per thread, FP64 throughout, over as many SMs as there are vectors for.  Both
// launches at 64 x 64: 7.2 us; 22.1 through the FP64 path of the kernel below, which puts 2048 vectors on an SM (and 16.5
// where all inputs were summed in FP64, 256 vectors a block).
constexpr int kShortThreads = 128;
static_assert((size_t)kStatBlocks * kShortThreads >= kWideValues, "a vector per thread");
__global__ void __launch_bounds__(kShortThreads) mv_variance_short_kernel(const float *__restrict__ mv, size_t n,
                                                                          double *__restrict__ part) {
    constexpr int kWarps = kShortThreads / 32;
    __shared__ float shift[2];
    __shared__ double red[kWarps][5];
    grid_dependency_wait();
    grid_dependents_launch();  // the kernel that adds the partials
    const size_t i = (size_t)blockIdx.x * kShortThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if ((size_t)blockIdx.x * kShortThreads >= n) {
        if (threadIdx.x < 5) part[threadIdx.x * kStatBlocks + blockIdx.x] = 0.0;
        return;
    }
    const float x = i < n ? __ldg(mv + i) : __int_as_float(0x7FC00000), y = i < n ? __ldg(mv + n + i) : x;
    find_shift(mv, n, shift);
    __syncthreads();
    const bool ok = isfinite(x) && isfinite(y);
    const double dx = ok ? (double)x - (double)shift[0] : 0.0, dy = ok ? (double)y - (double)shift[1] : 0.0;
    double v[4] = {dx, dy, dx * dx, dy * dy};
    const unsigned int count = __popc(__ballot_sync(0xFFFFFFFFu, ok));
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xFFFFFFFFu, v[c], o);
    if (lane == 0) {
        red[w][0] = (double)count;
#pragma unroll
        for (int c = 0; c < 4; ++c) red[w][c + 1] = v[c];
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double t = red[0][threadIdx.x];
        for (int q = 1; q < kWarps; ++q) t += red[q][threadIdx.x];
        part[threadIdx.x * kStatBlocks + blockIdx.x] = t;
    }
}

// Partials: count, sums of x - kx and y - ky, sums of their squares, [5][kStatBlocks].  8 bytes read
// and about 120 FP32 operations a pixel: 1080p 62 us with nine FP64 operations a pixel, 24 us now (events around
// both launches; 2.4 us of reads at the copy rate, the rest launches, tails and issue; 22 with the errors of the words
// added plainly, which biased repeated values).
template <int N>
__global__ void __launch_bounds__(kStatThreads) mv_variance_kernel(const float *__restrict__ mv, size_t n,
                                                                   double *__restrict__ part) {
    __shared__ float shift[2];
    __shared__ Words shp[4][kStatWarps];
    __shared__ double shw[32];
    grid_dependency_wait();
    grid_dependents_launch();  // the kernel that adds the partials
    constexpr int U = N == 1 ? 8 : 16 / N;  // packs in flight per plane
    const size_t npack = n / N, stride = (size_t)kStatBlocks * kStatThreads;
    const size_t first_pack = (size_t)blockIdx.x * kStatThreads + threadIdx.x;
    Pack<float, N> px[U], py[U];
    auto fetch = [&](size_t at) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t j = at + u * stride;
            if (j < npack) {
                px[u] = load_pack<float, N>(mv + j * N);
                py[u] = load_pack<float, N>(mv + n + j * N);
            }
        }
    };
    fetch(first_pack);  // the first values are on their way while the shift is found
    find_shift(mv, n, shift);
    __syncthreads();
    const float kx = shift[0], ky = shift[1];
    const double kxd = (double)kx, kyd = (double)ky;  // converted once: a conversion costs as much as an FP64 addition
    unsigned int cnt = 0u;
    bool any_rare = false;
    LinearSum sx, sy;                       // sums of (x - kx), (y - ky)
    SquareSum qx, qy;                       // and of their squares
    double r[4] = {0.0, 0.0, 0.0, 0.0};     // the same over the values that go through FP64
    // One vector: counted, added as pairs, or left for FP64 (true).
    auto take = [&](float x, float y) -> bool {
        const bool ok = isfinite(x) && isfinite(y);
        cnt += ok ? 1u : 0u;
        float hx, lx, hy, ly;
        two_diff(x, kx, hx, lx);
        two_diff(y, ky, hy, ly);
        const bool in = float_range(hx) && float_range(hy), use = ok && in;
        hx = use ? hx : 0.0f;
        lx = use ? lx : 0.0f;
        hy = use ? hy : 0.0f;
        ly = use ? ly : 0.0f;
        sx.add(hx, lx);
        sy.add(hy, ly);
        qx.add(hx, lx);
        qy.add(hy, ly);
        return ok && !in;
    };
    auto take_rare = [&](float x, float y) {
        wide_square(x, kxd, r[0], r[2]);
        wide_square(y, kyd, r[1], r[3]);
    };
    static_assert(kFoldValues % (U * N) == 0, "whole rounds between folds");
    int round = 1;
    for (size_t i = first_pack; i < npack; ++round) {
        unsigned int rare = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i + u * stride >= npack) break;
#pragma unroll
            for (int j = 0; j < N; ++j) rare |= take(px[u].v[j], py[u].v[j]) ? 1u << (u * N + j) : 0u;
        }
        if (rare != 0u) {
            any_rare = true;
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if (rare & (1u << (u * N + j))) take_rare(px[u].v[j], py[u].v[j]);
        }
        if (round % (kFoldValues / (U * N)) == 0) {
            sx.fold();
            sy.fold();
            qx.fold();
            qy.fold();
        }
        i += U * stride;
        fetch(i);
    }
    const size_t tail = npack * N + first_pack;  // fewer than N values are left
    if (tail < n) {
        const float x = __ldg(mv + tail), y = __ldg(mv + n + tail);
        if (take(x, y)) {
            any_rare = true;
            take_rare(x, y);
        }
    }
    sx.fold();
    sy.fold();
    qx.fold();
    qy.fold();
    double t[4] = {block_words(sx.far, shp[0]), block_words(sy.far, shp[1]), block_words(qx.far, shp[2]),
                   block_words(qy.far, shp[3])};
    if (__syncthreads_or(any_rare ? 1 : 0)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double w = block_wide(r[c], shw);
            if (threadIdx.x == 0) t[c] += w;
        }
    }
    cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
    __shared__ unsigned int counts[kStatWarps];
    if ((threadIdx.x & 31) == 0) counts[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int c = 0u;  // a block's pixels: at most 2^28 / 152
        for (int w = 0; w < kStatWarps; ++w) c += counts[w];
        part[blockIdx.x] = (double)c;
#pragma unroll
        for (int k = 0; k < 4; ++k) part[(k + 1) * kStatBlocks + blockIdx.x] = t[k];
    }
}

__global__ void __launch_bounds__(kSumThreads) mv_variance_sum_kernel(const double *part, double *out) {
    __shared__ double t[5];
    grid_dependency_wait();  // the partials
    const int w = threadIdx.x >> 5;
    if (w < 5) {
        const double v = warp_sum(part + w * kStatBlocks, kStatBlocks);
        if ((threadIdx.x & 31) == 0) t[w] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double cnt = t[0];
    out[0] = cnt;
    if (cnt == 0.0) {
        out[1] = out[2] = 0.0;
    } else {
        const double ax = t[1] / cnt, ay = t[2] / cnt;  // mean - shift
        out[1] = fmax(t[3] / cnt - ax * ax, 0.0);
        out[2] = fmax(t[4] / cnt - ay * ay, 0.0);
    }
}

// ------------------------------------------------------------------------------------------------------------
// Colour MSE
// ------------------------------------------------------------------------------------------------------------

// 2c bytes read a pixel and about 45 FP32 operations a value: 1080p FP32 79 us with four FP64 operations a value,
// 22.5 us now (events around both launches; 7.3 us of reads at the copy rate).
template <typename CT, int N>
__global__ void __launch_bounds__(kStatThreads) color_mse_kernel(const CT *__restrict__ a, const CT *__restrict__ b,
                                                                 size_t n, bool wide, double *__restrict__ part) {
    __shared__ Words shp[kStatWarps];
    __shared__ double shw[32];
    grid_dependency_wait();
    grid_dependents_launch();  // the kernel that adds the partials
    constexpr int U = N == 1 ? 8 : 16 / N;  // packs in flight per image
    const size_t npack = n / N, stride = (size_t)kStatBlocks * kStatThreads;
    const size_t first_pack = (size_t)blockIdx.x * kStatThreads + threadIdx.x;
    SquareSum q;
    double r = 0.0, unused = 0.0;
    bool any_rare = false;
    auto take = [&](CT va, CT vb) -> bool {
        float h, l;
        two_diff(to_f<CT>(va), to_f<CT>(vb), h, l);
        const bool in = wide && float_range(h);
        q.add(in ? h : 0.0f, in ? l : 0.0f);
        return !in;
    };
    static_assert(kFoldValues % (U * N) == 0, "whole rounds between folds");
    int round = 1;
    for (size_t i = first_pack; i < npack; i += U * stride, ++round) {
        Pack<CT, N> pa[U], pb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t j = i + u * stride;
            if (j < npack) {
                pa[u] = load_pack<CT, N>(a + j * N);
                pb[u] = load_pack<CT, N>(b + j * N);
            }
        }
        unsigned int rare = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i + u * stride >= npack) break;
#pragma unroll
            for (int j = 0; j < N; ++j) rare |= take(pa[u].v[j], pb[u].v[j]) ? 1u << (u * N + j) : 0u;
        }
        if (rare != 0u) {
            any_rare = true;
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if (rare & (1u << (u * N + j)))
                        wide_square(to_f<CT>(pa[u].v[j]), (double)to_f<CT>(pb[u].v[j]), unused, r);
        }
        if (round % (kFoldValues / (U * N)) == 0) q.fold();
    }
    const size_t tail = npack * N + first_pack;  // fewer than N values are left
    if (tail < n && take(a[tail], b[tail])) {
        any_rare = true;
        wide_square(to_f<CT>(a[tail]), (double)to_f<CT>(b[tail]), unused, r);
    }
    q.fold();
    double t = block_words(q.far, shp);
    if (__syncthreads_or(any_rare ? 1 : 0)) {
        const double w = block_wide(r, shw);
        if (threadIdx.x == 0) t += w;
    }
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void __launch_bounds__(32) color_mse_sum_kernel(const double *part, double n, double *out, bool psnr) {
    grid_dependency_wait();  // the partials
    const double t = warp_sum(part, kStatBlocks);
    if (threadIdx.x != 0) return;
    const double mse = t / n;
    out[0] = mse;
    // PSNR of colours in [0, 1] scaled by 255: 10 log10(255^2 / MSE) = -10 log10(MSE); +inf for equal images
    if (psnr) out[1] = mse == 0.0 ? __longlong_as_double(0x7FF0000000000000ll) : -10.0 * log10(mse);
}

// SSIM (Sec. IV-C, Eq. 3; the standard 11 x 11 Gaussian-window index, sigma 1.5, C1 = 1e-4, C2 = 9e-4 for colours in
// [0, 1]).  A warp takes 64 output columns (two per lane) of one channel and walks down its rows: the next rows' 74
// columns of both images are loaded two rows ahead into registers and staged in the warp's own shared memory; each
// lane filters its two columns horizontally from 12 neighbours and adds the result to the 11 outputs whose windows
// hold the row, which stay in registers (a ring unrolled by 11 rows).  Nothing but the raw rows passes through shared
// memory.  FP32, as the moments of s = (a - 1/2) + (b - 1/2) and d = a - b: with l the luminance term's and v the
// variance term's denominator the index is (1 - D^2 / l) (1 - var d / v), so its distance from 1 is formed directly and
// images that are alike lose nothing to cancellation.  The distances are added as float pairs, FP64 per warp and beyond.
// The window's weights are rounded to multiples of 2^-26 with a sum of exactly 1 (a sum off by an ulp gives a flat bright
// area a variance of its own).  Error against FP64 over 12 pairs of 1280 x 720 each, rms, and that of a kernel which filtered
// the moments of a and b through shared memory: smooth images half a pixel apart 5e-11 (2e-8), dark ones 3e-12 (3e-8),
// inverted 3e-8 (3e-6), dark noise 2e-8 (1e-5), unrelated noise 2e-10 (8e-10), flat against noise 2e-9 (2e-9; at
// 256 x 256 3e-9 and 2e-9).
//
// Bound by issue: per output 2 x 44 multiply-adds for the windows, 12 for the squares, about 34 for the index.  1080p
// FP32 136 us with the filtered maps in shared memory (a multiply-add per load, the sum on the FP64 pipe), 55 us from the
// moments of a and b, 53 us now (events around both launches).
constexpr int kSsimCols = 64, kSsimIn = kSsimCols + 10, kSsimPad = 80;
constexpr int kSsimWarps = 4, kSsimThreads = 32 * kSsimWarps;
constexpr int kSsimItems = 12 * 152;  // warps of one wave: 12 per SM of 152 at up to 168 registers

// Rows of outputs per warp, so that a frame gives about one wave of warps; 8 at least (each warp reads 10 rows more).
struct SsimGrid {
    int strips, rows, chunks;
    SsimGrid(int W, int H) {
        const int OH = H - 10;
        strips = ceil_div(W - 10, kSsimCols);
        int c = kSsimItems / (3 * strips);
        c = c < 1 ? 1 : c > ceil_div(OH, 8) ? ceil_div(OH, 8) : c;
        rows = ceil_div(OH, c);
        chunks = ceil_div(OH, rows);
    }
    int items() const { return 3 * strips * chunks; }
    int blocks() const { return ceil_div(items(), kSsimWarps); }
};

template <typename CT>
__global__ void __launch_bounds__(kSsimThreads, 3) ssim_kernel(const CT *__restrict__ a, const CT *__restrict__ b,
                                                               int W, int H, int strips, int rows, int chunks,
                                                               double *__restrict__ part) {
    __shared__ __align__(16) float stage[kSsimWarps][2][2][kSsimPad];  // [warp][row parity][image][column]
    __shared__ double red[kSsimWarps];
    grid_dependency_wait();
    grid_dependents_launch();  // the kernel that adds the partials
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int OW = W - 10, OH = H - 10;
    float g[6];  // the window's weights, symmetric (g[i] = weight i = weight 10 - i), their sum exactly 1
    {
        float e[11], sum = 0.0f;
        for (int i = 0; i < 11; ++i) {
            e[i] = expf(-(float)((i - 5) * (i - 5)) / 4.5f);
            sum += e[i];
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) g[i] = rintf(e[i] / sum * 67108864.0f) * (1.0f / 67108864.0f);
        g[5] = 1.0f - 2.0f * (((g[0] + g[1]) + (g[2] + g[3])) + g[4]);
    }
    const float C1 = 1e-4f, C2 = 9e-4f;
    double total = 0.0;
    const int item = blockIdx.x * kSsimWarps + wid;
    if (item < 3 * strips * chunks) {
        // a strip's chunks are neighbours, then its channels: warps of a block share rows
        const int strip = item % strips, rest = item / strips, chunk = rest % chunks, ch = rest / chunks;
        const int X0 = strip * kSsimCols, Y0 = chunk * rows;
        const int nrow = min(rows, OH - Y0) + 10;  // input rows
        const CT *pa = a + (size_t)ch * W * H + (size_t)Y0 * W + X0, *pb = b + (size_t)ch * W * H + (size_t)Y0 * W + X0;
        const int left = W - X0;  // columns of the frame from X0
        // this lane's columns of a row: lane, lane + 32, lane + 64 (the last for 10 lanes); outside the frame a value
        // that no output of the frame uses.  As loaded: converted and shifted when they are staged, two rows later
        struct Row {
            CT a[3], b[3];
        };
        auto fetch = [&](int r) {
            Row v;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int x = lane + 32 * i;
                const bool in = x < kSsimIn && x < left && r < nrow;
                const size_t o = (size_t)r * W + x;
                v.a[i] = in ? __ldg(pa + o) : CT(0.0f);
                v.b[i] = in ? __ldg(pb + o) : CT(0.0f);
            }
            return v;
        };
        const bool ok0 = X0 + 2 * lane < OW, ok1 = X0 + 2 * lane + 1 < OW;
        float acc[11][4][2];  // output row o in slot o mod 11: maps s, d, s^2, d^2 of the lane's two columns
        FloatSum sum;
        Row n0 = fetch(0), n1 = fetch(1);
        for (int base = 0; base < nrow; base += 11) {
#pragma unroll
            for (int u = 0; u < 11; ++u) {
                const int r = base + u;
                if (r >= nrow) break;
                float(*st)[kSsimPad] = stage[wid][r & 1];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    if (lane + 32 * i < kSsimPad) {
                        const float x = to_f<CT>(n0.a[i]), y = to_f<CT>(n0.b[i]);
                        st[0][lane + 32 * i] = (x - 0.5f) + (y - 0.5f);
                        st[1][lane + 32 * i] = x - y;
                    }
                }
                n0 = n1;
                n1 = fetch(r + 2);
                __syncwarp();  // the row is staged (the other parity's reads ended before this row's writes began)
                float vs[12], vd[12], h[4][2];
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    const float2 x = *reinterpret_cast<const float2 *>(&st[0][2 * lane + 2 * j]);
                    const float2 y = *reinterpret_cast<const float2 *>(&st[1][2 * lane + 2 * j]);
                    vs[2 * j] = x.x;
                    vs[2 * j + 1] = x.y;
                    vd[2 * j] = y.x;
                    vd[2 * j + 1] = y.y;
                }
#pragma unroll
                for (int j = 0; j < 12; ++j) {
                    const float x = vs[j], y = vd[j], q = x * x, p = y * y;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {  // column c takes neighbours c .. c + 10
                        const int i = j - c;
                        if (i < 0 || i > 10) continue;
                        const float w = g[i < 6 ? i : 10 - i];
                        h[0][c] = i == 0 ? w * x : fmaf(w, x, h[0][c]);
                        h[1][c] = i == 0 ? w * y : fmaf(w, y, h[1][c]);
                        h[2][c] = i == 0 ? w * q : fmaf(w, q, h[2][c]);
                        h[3][c] = i == 0 ? w * p : fmaf(w, p, h[3][c]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 11; ++i) {  // row r is window row i of output r - i, in slot (u - i) mod 11
                    const int slot = (u - i + 11) % 11;
                    const float w = g[i < 6 ? i : 10 - i];
#pragma unroll
                    for (int m = 0; m < 4; ++m)
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            acc[slot][m][c] = i == 0 ? w * h[m][c] : fmaf(w, h[m][c], acc[slot][m][c]);
                }
                if (r >= 10) {  // output row r - 10 is complete
                    const int slot = (u + 1) % 11;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float ms = acc[slot][0][c], md = acc[slot][1][c];
                        const float vs2 = fmaf(-ms, ms, acc[slot][2][c]), vd2 = fmaf(-md, md, acc[slot][3][c]);
                        const float S = ms + 1.0f, D2 = md * md;
                        const float l = fmaf(0.5f, fmaf(S, S, D2), C1);
                        const float t = 0.5f * (vs2 + vd2), v = __fadd_rn(t, C2);
                        const float e = fmaf(D2, v - vd2, vd2 * l) / (l * v);
                        // v loses C2's low bits, the same ones wherever the variances have one magnitude: where the
                        // images share nothing (e near 1) that alone moved the mean by 2e-9
                        const float lost = __fsub_rn(C2, __fsub_rn(v, t));
                        sum.add((c == 0 ? ok0 : ok1) ? e : 0.0f, __fdividef(lost, v));
                    }
                }
            }
            sum.fold();
        }
        total = (double)sum.far.s + ((double)sum.far.c + (double)sum.far.d);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, o);
    if (lane == 0) red[wid] = total;
    __syncthreads();
    if (threadIdx.x == 0) part[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
}

__global__ void __launch_bounds__(32) ssim_sum_kernel(const double *part, int nparts, double count, double *out) {
    grid_dependency_wait();  // the partials
    const double t = warp_sum(part, nparts);
    if (threadIdx.x == 0) out[0] = 1.0 - t / count;
}

}  // namespace

size_t stats_workspace_bytes() { return (sizeof(StatWs) + 255) & ~(size_t)255; }

cudaError_t launch_mv_variance(const float *mv, int W, int H, double *out, void *ws, cudaStream_t s) {
    static_assert(5 * kStatBlocks <= kMaxPartials, "the partials fit the workspace");
    double *const part = static_cast<StatWs *>(ws)->part;
    const size_t n = (size_t)W * H;
    const bool vec = ((uintptr_t)mv & 15u) == 0 && (n & 3u) == 0;  // both planes start on 16 bytes
    timing_begin("exw_mv_variance", s);
    cudaError_t e =
        n < kWideValues
            ? launch_dependent(mv_variance_short_kernel, dim3(kStatBlocks), dim3(kShortThreads), 0, s, mv, n, part)
            : launch_dependent(vec ? mv_variance_kernel<4> : mv_variance_kernel<1>, dim3(kStatBlocks),
                               dim3(kStatThreads), 0, s, mv, n, part);
    count_launch();
    if (e == cudaSuccess) {
        const double *cpart = part;
        e = launch_dependent(mv_variance_sum_kernel, dim3(1), dim3(kSumThreads), 0, s, cpart, out);
        count_launch();
    }
    timing_end("exw_mv_variance", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_color_mse(const void *a, const void *b, exw_dtype cdt, int W, int H, double *out, void *ws,
                             cudaStream_t s, bool psnr) {
    double *const part = static_cast<StatWs *>(ws)->part;
    const size_t n = 3 * (size_t)W * H;
    const bool vec = (((uintptr_t)a | (uintptr_t)b) & 15u) == 0, wide = n >= kWideValues;
    timing_begin("exw_color_mse", s);
    cudaError_t e;
    if (cdt == EXW_F16) {
        const __half *x = (const __half *)a, *y = (const __half *)b;
        e = launch_dependent(vec ? color_mse_kernel<__half, 8> : color_mse_kernel<__half, 1>, dim3(kStatBlocks),
                             dim3(kStatThreads), 0, s, x, y, n, wide, part);
    } else {
        const float *x = (const float *)a, *y = (const float *)b;
        e = launch_dependent(vec ? color_mse_kernel<float, 4> : color_mse_kernel<float, 1>, dim3(kStatBlocks),
                             dim3(kStatThreads), 0, s, x, y, n, wide, part);
    }
    count_launch();
    if (e == cudaSuccess) {
        const double *cpart = part;
        const double dn = (double)n;
        e = launch_dependent(color_mse_sum_kernel, dim3(1), dim3(32), 0, s, cpart, dn, out, psnr);
        count_launch();
    }
    timing_end("exw_color_mse", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_ssim(const void *a, const void *b, exw_dtype cdt, int W, int H, double *out, void *ws,
                        cudaStream_t s) {
    double *const part = static_cast<StatWs *>(ws)->part;
    const SsimGrid gr(W, H);
    timing_begin("exw_ssim", s);
    cudaError_t e;
    if (cdt == EXW_F16) {
        const __half *x = (const __half *)a, *y = (const __half *)b;
        e = launch_dependent(ssim_kernel<__half>, dim3(gr.blocks()), dim3(kSsimThreads), 0, s, x, y, W, H,
                             gr.strips, gr.rows, gr.chunks, part);
    } else {
        const float *x = (const float *)a, *y = (const float *)b;
        e = launch_dependent(ssim_kernel<float>, dim3(gr.blocks()), dim3(kSsimThreads), 0, s, x, y, W, H,
                             gr.strips, gr.rows, gr.chunks, part);
    }
    count_launch();
    if (e == cudaSuccess) {
        const double *cpart = part;
        const int nparts = gr.blocks();
        const double count = 3.0 * (double)(W - 10) * (double)(H - 10);
        e = launch_dependent(ssim_sum_kernel, dim3(1), dim3(32), 0, s, cpart, nparts, count, out);
        count_launch();
    }
    timing_end("exw_ssim", s);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace exw
