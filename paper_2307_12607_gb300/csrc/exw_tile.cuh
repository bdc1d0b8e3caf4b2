// exw_tile.cuh -- what the per-tile kernels and the engine share: the reach of a target tile under the motion bounds,
// and the fill's pull-push pyramid (levels 1 to 5 of a 32 x 32 tile, the coarse levels above them, the bookkeeping of
// tiles without a valid pixel).
#pragma once

#include "exw_device.cuh"
#include "exw_internal.h"

namespace exw {

constexpr int kThreads = 512;

// The fractions of the fused path are k / 4, k = 1 .. nfrac (Sec. IV-B): constants, so that no kernel keeps them in
// registers or converts them per pixel (4 frames of 1080p FP16 under a turning camera: engine 401 -> 394 us, 48 streams
// 5116 -> 5049).
constexpr int kEngineL = 2, kEngineK0 = 1;
__device__ __forceinline__ float engine_scale(int kk) { return 0.25f * (float)(kEngineK0 + kk); }

struct Rect {
    int x0, x1, y0, y1;
    __device__ __forceinline__ bool empty() const { return x1 < x0 || y1 < y0; }
};

// The block range that can reach region R (RX0, RY0 .. +33) under the frame-wide motion bounds, for fractions
// k0 .. k0+nfrac-1.  Returns false when nothing can land anywhere.
__device__ __forceinline__ bool frame_window(const TileParams &p, int RX0, int RY0, int &bx0, int &bx1, int &by0,
                                             int &by1) {
    const uint32_t a0 = __ldcg(&p.fh->acc[0]), a1 = __ldcg(&p.fh->acc[1]);
    const uint32_t a2 = __ldcg(&p.fh->acc[2]), a3 = __ldcg(&p.fh->acc[3]);
    if (a1 == 0u) return false;
    const float fx0 = -float_unorder(a0), fx1 = float_unorder(a1), fy0 = -float_unorder(a2), fy1 = float_unorder(a3);
    int xlo = 1 << 30, xhi = -(1 << 30), ylo = 1 << 30, yhi = -(1 << 30);
    for (int kk = 0; kk < p.nfrac; ++kk) {
        const float kf = engine_scale(kk);
        const int ox0 = offset_of(fx0, kf), ox1 = offset_of(fx1, kf);
        const int oy0 = offset_of(fy0, kf), oy1 = offset_of(fy1, kf);
        xlo = min(xlo, RX0 - ox1);
        xhi = max(xhi, RX0 + kRegion - 1 - ox0);
        ylo = min(ylo, RY0 - oy1);
        yhi = max(yhi, RY0 + kRegion - 1 - oy0);
    }
    bx0 = max(0, xlo >> 3);
    bx1 = min(p.nbx - 1, xhi >> 3);
    by0 = max(0, ylo >> 3);
    by1 = min(p.nby - 1, yhi >> 3);
    return bx0 <= bx1 && by0 <= by1;
}

// The offsets [ox0, ox1] x [oy0, oy1] of a fraction of a tile's motion bounds (the offset is monotone in the motion).
__device__ __forceinline__ void bounds_offsets(const float4 &b, float kf, int &ox0, int &ox1, int &oy0, int &oy1) {
    ox0 = offset_of(b.x, kf);
    ox1 = offset_of(b.y, kf);
    oy0 = offset_of(b.z, kf);
    oy1 = offset_of(b.w, kf);
}

// ------------------------------------------------------------------------------------------------------------
// Coarse levels and bookkeeping of the fill
// ------------------------------------------------------------------------------------------------------------

// Coarse levels of the pyramid (above level 5) for every fraction with invalid tiles, and the value each invalid
// tile receives (its first valid ancestor; 0 when the frame has no valid pixel).  Run by one CTA.
__device__ inline void coarse_pass(const TileParams &p) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int n5 = p.n5x * p.n5y;
    for (int kk = 0; kk < p.nfrac; ++kk) {
        const uint32_t cnt = __ldcg(&p.fh->ninvalid[kk]);
        if (cnt == 0u) continue;
        const float4 *child = p.nodes + (size_t)kk * n5;
        float4 *cz = p.coarse + (size_t)kk * p.ncoarse;
        int cw = p.n5x, ch = p.n5y, off = 0;
        while (cw > 1 || ch > 1) {
            const int pw = (cw + 1) / 2, ph = (ch + 1) / 2;
            float4 *par = cz + off;
            for (int node = tid; node < pw * ph; node += nt) {
                const int i = node / pw, j = node - i * pw;
                float4 c[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int ci = 2 * i + (q >> 1), cj = 2 * j + (q & 1);
                    c[q] = (ci < ch && cj < cw) ? __ldcg(child + ci * cw + cj) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                par[node] = mean4(c[0], c[1], c[2], c[3]);
            }
            __syncthreads();
            child = par;
            off += pw * ph;
            cw = pw;
            ch = ph;
        }
        for (uint32_t e = tid; e < cnt; e += nt) {
            const uint32_t tile = __ldcg(p.list + (size_t)kk * n5 + e);
            int ax = (int)(tile % (uint32_t)p.n5x), ay = (int)(tile / (uint32_t)p.n5x);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            int w = p.n5x, h = p.n5y, o = 0;
            while (w > 1 || h > 1) {
                const int pw = (w + 1) / 2, ph = (h + 1) / 2;
                ax >>= 1;
                ay >>= 1;
                const float4 c = __ldcg(cz + o + ay * pw + ax);
                if (c.w != 0.0f) {
                    v = c;
                    break;
                }
                o += pw * ph;
                w = pw;
                h = ph;
            }
            p.fillval[(size_t)kk * n5 + e] = make_float4(v.x, v.y, v.z, 1.0f);
        }
        __syncthreads();
    }
}

// Write the level-5 node of a tile for fraction kk; list the tile if it has no valid pixel.  Thread 0 only.
__device__ __forceinline__ void publish_node(const TileParams &p, float4 node, int kk, int tile) {
    const int n5 = p.n5x * p.n5y;
    p.nodes[(size_t)kk * n5 + tile] = node;
    if (node.w == 0.0f) {
        const uint32_t slot = atomicAdd(&p.fh->ninvalid[kk], 1u);
        p.list[(size_t)kk * n5 + slot] = (uint32_t)tile;
    }
}

// ------------------------------------------------------------------------------------------------------------
// Pull-push of one 32 x 32 tile by kTileThreads threads: lane = column, warp w the rows 2w and 2w + 1, so every row
// access is one line and a thread's pixels need no index arithmetic of their own.  Level 1 of two columns' pixels is
// formed with a shuffle, levels 2 to 5 by warp 0 from the tile's 256 level-1 nodes in shared memory; the others wait
// for them only where some hole has no valid level-1 ancestor.
// ------------------------------------------------------------------------------------------------------------
constexpr int kTileRows = 2;                              // rows per warp
constexpr int kTileThreads = kFillTile / kTileRows * 32;  // 512

struct TilePyramid {
    float4 l1[256], l2[64], l3[16], l4[4], l5;
};

// Levels 3, 4 and 5 of a tile from its level-2 nodes (one warp; every lane returns l5, lane L < 16 its level-3 node
// L = (L >> 2, L & 3), lane L < 4 its level-4 node).
__device__ __forceinline__ void upper_levels(const float4 *l2, float4 &l3, float4 &l4, float4 &l5) {
    const int lane = threadIdx.x & 31;
    const int L = lane & 15;
    const int I = L >> 2, J = L & 3;
    const float4 *c = l2 + (2 * I) * 8 + 2 * J;
    l3 = mean4_01(c[0], c[1], c[8], c[9]);
    const int b4 = 8 * ((lane & 3) >> 1) + 2 * (lane & 1);
    const float4 q0 = shfl4_idx(l3, b4), q1 = shfl4_idx(l3, b4 + 1), q2 = shfl4_idx(l3, b4 + 4),
                 q3 = shfl4_idx(l3, b4 + 5);
    l4 = mean4_01(q0, q1, q2, q3);
    l5 = mean4_01(shfl4_idx(l4, 0), shfl4_idx(l4, 1), shfl4_idx(l4, 2), shfl4_idx(l4, 3));
}

// Publishes the tile's level-5 node and replaces each hole of this thread's column (m[r] != 0) by its first valid
// ancestor inside the tile; returns a bit per row whose pixel has a value now (the others' tile has no valid pixel:
// the coarse fix-up writes them).  c[r].w = validity.  One block barrier, two where a hole lies that deep.
__device__ __forceinline__ unsigned int fill_columns(const TileParams &p, TilePyramid &t, float4 (&c)[kTileRows],
                                                     const uint8_t (&m)[kTileRows], int kk, int tile) {
    static_assert(kTileRows == 2, "one level-1 node per column pair");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float4 o0 = shfl4_xor(c[0], 1), o1 = shfl4_xor(c[1], 1);
    // children in the order (0,0), (0,1), (1,0), (1,1)
    const float4 n1 = (lane & 1) ? mean4_01(o0, c[0], o1, c[1]) : mean4_01(c[0], o0, c[1], o1);
    if ((lane & 1) == 0) t.l1[w * 16 + (lane >> 1)] = n1;
    const bool deep = __syncthreads_or((m[0] | m[1]) != 0 && n1.w == 0.0f) != 0;
    if (w == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int node = lane + 32 * h, i = node >> 3, j = node & 7;
            const float4 *q = t.l1 + (2 * i) * 16 + 2 * j;
            t.l2[node] = mean4_01(q[0], q[1], q[16], q[17]);
        }
        __syncwarp();
        float4 l3, l4, l5;
        upper_levels(t.l2, l3, l4, l5);
        if (lane < 16) t.l3[lane] = l3;
        if (lane < 4) t.l4[lane] = l4;
        if (lane == 0) {
            t.l5 = l5;
            publish_node(p, l5, kk, tile);
        }
    }
    float4 v = n1;
    if (deep) {
        __syncthreads();  // levels 2 to 5
        if (v.w == 0.0f) v = t.l2[(w >> 1) * 8 + (lane >> 2)];
        if (v.w == 0.0f) v = t.l3[(w >> 2) * 4 + (lane >> 3)];
        if (v.w == 0.0f) v = t.l4[(w >> 3) * 2 + (lane >> 4)];
        if (v.w == 0.0f) v = t.l5;
    }
    unsigned int have = 0u;
#pragma unroll
    for (int r = 0; r < kTileRows; ++r) {
        if (m[r] != 0) c[r] = v;
        have |= c[r].w != 0.0f ? 1u << r : 0u;
    }
    return have;
}

}  // namespace exw
