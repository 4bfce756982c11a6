// Learned first search radius: a 3-layer MLP (27 -> 64 -> 64 -> 1, ReLU)
// over log(1 + count) of a query chunk's 3x3x3 stencil cells, predicting
// log(largest Ndens-th-neighbour distance of the chunk / cell side).
// Weights are BF16 (an fp32 master copy is kept for training); products and
// sums are FP32.  Forward, backward and Adam are hand-written here.
#include "hop_internal.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <vector>

namespace {

constexpr int IN = HOP_MLP_IN, H = HOP_MLP_HID, NP = HOP_MLP_NPARAM;
constexpr int oW1 = 0, oB1 = H * IN, oW2 = oB1 + H, oB2 = oW2 + H * H, oW3 = oB2 + H, oB3 = oW3 + H;
static_assert(oB3 + 1 == NP, "parameter layout");
__device__ __forceinline__ float bf(const __nv_bfloat16 *w, int i) { return __bfloat162float(w[i]); }

// The first radius of every chunk in one pass, 32 chunks per warp.  Each
// lane finds its chunk's stencil level and centre cell (the same arithmetic
// as chunk_stencil) and spreads the three coordinates of each axis into
// Morton bits once.  The 32 x 27 stencil cells are then looked up as one flat
// list, kRadU independent cells per lane and step: this part is bound by the
// latency of the table reads and, in halos, of the searches below the dense
// level, so the searches of a lane's cells advance together.
// NET: the learned radius, R = side * exp(MLP + margin), the network as two
// small GEMMs of the warp's 32 chunks (an 8 x 8 register tile per lane, FP32-
// bound: 184 FMA instructions per chunk).  !NET: the closed form from the
// stencil total, R = side * cbrt(81 k / (4 pi total)) * exp(margin), the
// chunk's k-th-neighbour distance if the 27 cells held the mean density of
// their total.
// Measured (one chunk's cells at a time, the network one chunk per lane, in
// brackets): learned, 4.2M chunks of 16.8M particles 3.06 ms (3.98), issue
// 52 % busy; closed form, 750k chunks of 3M particles 0.31 ms (0.48).  Nine
// cells at once gave the same time.
constexpr int kRadThreads = 128;
constexpr int kRadWarps = kRadThreads / 32;
constexpr int kRadU = 3;              // cells a lane looks up at once
constexpr int kRadLog = 256;          // log(1 + count) from a table up to this count
constexpr int kLdX = 28, kLdH = 68;   // row strides: features (padded with a zero), hidden units
static_assert((27 * 32) % (32 * kRadU) == 0, "whole steps");

struct RadChunk {
    uint2 code[3][3];     // spread coordinates: axis, offset -1 / 0 / +1
    int64_t cell0;        // the subvolume's table
    int l, ld;            // stencil level, dense level
};
struct __align__(16) RadWarp {
    union {
        RadChunk ch[32];
        float h[32][kLdH];
    };
    float f[32][kLdX];    // log(1 + count); the counts' bits without the network
};
struct __align__(16) RadWeights {
    float w1[H][kLdX], w2[H][kLdH];
    float b1[H], b2[H], w3[H], b3;
    float lg[kRadLog];
};
// (rows are read 16 bytes at a time)
static_assert(sizeof(RadWeights) % 16 == 0 && sizeof(RadWarp) % 16 == 0 && offsetof(RadWarp, f) % 16 == 0 &&
                  offsetof(RadWeights, w2) % 16 == 0 && kLdX % 4 == 0 && kLdH % 4 == 0,
              "alignment of the rows");
template <bool NET> constexpr size_t rad_smem()
{
    return NET ? sizeof(RadWeights) + kRadWarps * sizeof(RadWarp) : kRadWarps * sizeof(RadWarp);
}

__device__ __forceinline__ void fma4(float &a, const float4 &u, const float4 &v)
{
    a = fmaf(u.x, v.x, a);
    a = fmaf(u.y, v.y, a);
    a = fmaf(u.z, v.z, a);
    a = fmaf(u.w, v.w, a);
}

template <bool NET>
__global__ void __launch_bounds__(kRadThreads, 3)
radius_kernel(const __nv_bfloat16 *__restrict__ w16, const float4 *__restrict__ spos,
              const uint64_t *__restrict__ keys, const uint32_t *__restrict__ cellT, int Ld,
              int64_t n, int64_t n_chunks, int Q, float box, float inv_box,
              const SegDesc *__restrict__ seg, int B, float margin, int k, float *__restrict__ chunk_r)
{
    extern __shared__ __align__(16) unsigned char rad_raw[];
    RadWeights &W = *(RadWeights *)rad_raw;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    RadWarp &S = *((RadWarp *)(rad_raw + (NET ? sizeof(RadWeights) : 0)) + w);
    if constexpr (NET) {
        for (int i = threadIdx.x; i < H * kLdX; i += kRadThreads) {
            const int j = i / kLdX, f = i % kLdX;
            W.w1[j][f] = f < IN ? bf(w16, oW1 + j * IN + f) : 0.f;
        }
        for (int i = threadIdx.x; i < H * H; i += kRadThreads) W.w2[i / H][i % H] = bf(w16, oW2 + i);
        for (int i = threadIdx.x; i < H; i += kRadThreads) {
            W.b1[i] = bf(w16, oB1 + i);
            W.b2[i] = bf(w16, oB2 + i);
            W.w3[i] = bf(w16, oW3 + i);
        }
        if (threadIdx.x == 0) W.b3 = bf(w16, oB3);
        for (int i = threadIdx.x; i < kRadLog; i += kRadThreads) W.lg[i] = log1pf((float)i);
        S.f[lane][IN] = 0.f;
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * kRadWarps * 32;
    for (int64_t base = ((int64_t)blockIdx.x * kRadWarps + w) * 32; base < n_chunks; base += stride) {
        const int nc = (int)min((int64_t)32, n_chunks - base);
        // ---- the lane's chunk: stencil level, centre cell, cell side
        const int64_t ch = base + (lane < nc ? lane : 0);
        int64_t s0 = ch * Q, nend = n, cell0 = 0;
        int ld = Ld;
        float bx = box, ibx = inv_box;
        if (seg) {
            const SegDesc &d = seg[seg_of_chunk(seg, B, ch)];
            s0 = d.base + (ch - d.chunk0) * Q;
            nend = d.base + d.n;
            cell0 = d.cell0;
            ld = d.level_dense;
            bx = (float)d.box;
            ibx = (float)(1.0 / d.box);
        }
        const int nq = (int)min((int64_t)Q, nend - s0);
        float lx = INFINITY, ly = INFINITY, lz = INFINITY, hx = -INFINITY, hy = -INFINITY, hz = -INFINITY;
        for (int q = 0; q < nq; ++q) {
            const float4 v = spos[s0 + q];
            lx = fminf(lx, v.x);
            ly = fminf(ly, v.y);
            lz = fminf(lz, v.z);
            hx = fmaxf(hx, v.x);
            hy = fmaxf(hy, v.y);
            hz = fmaxf(hz, v.z);
        }
        const float ext = fmaxf(hx - lx, fmaxf(hy - ly, hz - lz));
        int l = kMaxLevel;
        while (l > 2 && bx / (float)(1 << l) < ext) --l;
        const int G = 1 << l;
        const float sc = ibx * (float)G;
        const int c0[3] = {min((int)floorf((lx + hx) * 0.5f * sc), G - 1), min((int)floorf((ly + hy) * 0.5f * sc), G - 1),
                           min((int)floorf((lz + hz) * 0.5f * sc), G - 1)};
        const float side = (float)((double)bx / (double)G);
        {
            RadChunk &c = S.ch[lane];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const uint32_t x = (uint32_t)(c0[a] + d - 1) & (uint32_t)(G - 1);
                    c.code[a][d] = make_uint2(spread3_8(x) << a, spread3_8(x >> 8) << a);
                }
            c.cell0 = cell0;
            c.l = l;
            c.ld = ld;
        }
        __syncwarp();
        // ---- the stencil counts, kRadU cells per lane and step
#pragma unroll 1
        for (int i0 = 0; i0 < 27 * 32; i0 += 32 * kRadU) {
            uint32_t a[kRadU], b[kRadU], ha[kRadU], hb[kRadU];
            uint64_t k0[kRadU], k1[kRadU];
            int cj[kRadU], cc[kRadU];
#pragma unroll
            for (int u = 0; u < kRadU; ++u) {
                const int i = i0 + 32 * u + lane;
                cj[u] = i / 27;
                cc[u] = i - 27 * cj[u];
                const RadChunk &c = S.ch[cj[u]];
                const int dz = cc[u] / 9, r = cc[u] - 9 * dz, dy = r / 3, dx = r - 3 * dy;
                const uint2 x = c.code[0][dx], y = c.code[1][dy], z = c.code[2][dz];
                const uint64_t code = ((uint64_t)(x.y | y.y | z.y) << 24) | (x.x | y.x | z.x);
                const uint32_t *t = cellT + c.cell0;
                const int up = 3 * (c.l - c.ld);
                if (up <= 0) {
                    a[u] = t[code << -up];
                    b[u] = t[(code + 1) << -up];
                    ha[u] = a[u];
                    hb[u] = b[u];
                    k0[u] = k1[u] = 0;
                } else {
                    // below the dense level: first keys >= k0 and >= k1 in the
                    // dense cell's range
                    const uint64_t pc = code >> up;
                    const int ksh = 3 * (kMaxLevel - c.l);
                    a[u] = b[u] = t[pc];
                    ha[u] = hb[u] = t[pc + 1];
                    k0[u] = code << ksh;
                    k1[u] = (code + 1) << ksh;
                }
            }
            for (;;) {
                bool more = false;
                uint64_t x[kRadU], y[kRadU];
#pragma unroll
                for (int u = 0; u < kRadU; ++u) {
                    x[u] = y[u] = 0;
                    if (a[u] < ha[u]) x[u] = keys[(a[u] + ha[u]) >> 1];
                    if (b[u] < hb[u]) y[u] = keys[(b[u] + hb[u]) >> 1];
                }
#pragma unroll
                for (int u = 0; u < kRadU; ++u) {
                    if (a[u] < ha[u]) {
                        const uint32_t m = (a[u] + ha[u]) >> 1;
                        if (x[u] < k0[u]) a[u] = m + 1; else ha[u] = m;
                    }
                    if (b[u] < hb[u]) {
                        const uint32_t m = (b[u] + hb[u]) >> 1;
                        if (y[u] < k1[u]) b[u] = m + 1; else hb[u] = m;
                    }
                    more = more || a[u] < ha[u] || b[u] < hb[u];
                }
                if (!__any_sync(0xffffffffu, more)) break;
            }
#pragma unroll
            for (int u = 0; u < kRadU; ++u) {
                const uint32_t cnt = b[u] - a[u];
                if constexpr (NET)
                    S.f[cj[u]][cc[u]] = cnt < (uint32_t)kRadLog ? W.lg[cnt] : log1pf((float)cnt);
                else
                    S.f[cj[u]][cc[u]] = __uint_as_float(cnt);
            }
        }
        __syncwarp();
        if constexpr (!NET) {
            if (lane < nc) {
                uint32_t tot = 0;
                for (int c = 0; c < IN; ++c) tot += __float_as_uint(S.f[lane][c]);
                const double r = (double)side * cbrt(81.0 * k / (4.0 * 3.14159265358979323846 * (double)max(tot, 1u)));
                chunk_r[base + lane] = (float)(r * exp((double)margin));
            }
            __syncwarp();
            continue;
        }
        // ---- the network: outputs og + 8 a, chunks sg + 4 b
        const int og = lane & 7, sg = lane >> 3;
        float acc[8][8];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = W.b1[og + 8 * a];
#pragma unroll 1
        for (int kk = 0; kk < kLdX; kk += 4) {
            float4 wv[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) wv[a] = *(const float4 *)&W.w1[og + 8 * a][kk];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const float4 x = *(const float4 *)&S.f[sg + 4 * b][kk];
#pragma unroll
                for (int a = 0; a < 8; ++a) fma4(acc[a][b], wv[a], x);
            }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) S.h[sg + 4 * b][og + 8 * a] = fmaxf(acc[a][b], 0.f);
        __syncwarp();
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = W.b2[og + 8 * a];
#pragma unroll 1
        for (int kk = 0; kk < H; kk += 4) {
            float4 wv[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) wv[a] = *(const float4 *)&W.w2[og + 8 * a][kk];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const float4 x = *(const float4 *)&S.h[sg + 4 * b][kk];
#pragma unroll
                for (int a = 0; a < 8; ++a) fma4(acc[a][b], wv[a], x);
            }
        }
        // lane (og, sg) ends with the output of chunk sg + 4 og
        float out = 0.f;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            float y = 0.f;
#pragma unroll
            for (int a = 0; a < 8; ++a) y = fmaf(W.w3[og + 8 * a], fmaxf(acc[a][b], 0.f), y);
            y += __shfl_xor_sync(0xffffffffu, y, 1);
            y += __shfl_xor_sync(0xffffffffu, y, 2);
            y += __shfl_xor_sync(0xffffffffu, y, 4);
            if (og == b) out = y;
        }
        const int mine = sg + 4 * og;
        const float sd = __shfl_sync(0xffffffffu, side, mine);
        if (mine < nc) chunk_r[base + mine] = sd * expf(out + W.b3 + margin);
        __syncwarp();
    }
}

// The network over a set of samples (idx[] or 0..m-1): the outputs (GRAD
// false), or the mean-squared-error gradient scaled by `scale` (1 / batch
// size), of which every block writes its share to part[block][NP].
//
// A block of 128 threads takes tiles of 128 samples.  Each product is a small
// GEMM over the tile with an 8 x 8 register tile per thread (og, sg): 16
// reads of 16 bytes feed 256 FMAs, which is where shared-memory wavefronts
// (four per read) and the FMA pipe balance; one sample per thread needs a
// read per FMA.  Rows are padded so that the eight rows (or row parts) that a
// quarter of a warp reads lie in distinct banks.  The weight gradients stay
// in registers over all tiles of a block.  Weights are fp32 values of the
// bf16 copy; everything else is fp32, the blocks' shares are summed in fp64.
// FP32- and shared-memory-bound: 15.9k multiply-adds per sample forward and
// backward, 5.9k forward only.  Gradient and predictions of 262,147 samples:
// 3237 us with one sample per thread (rows 64 apart, every lane in one bank;
// shares added by atomics), 374 us now, of an FP32 floor of 140 us.
// The long register sums cost no accuracy at the sizes a box gives: against
// 64-bit sums the gradient is off by 3e-8 to 1.7e-7 (relative) at 262,147
// samples and by 8e-8 to 1.3e-7 at 33.5 million, where a fp32 share per 64
// samples added by atomics was off by 2.6e-7 to 3.5e-7 at either size.
constexpr int kNetThreads = 128, kNetTile = 128;
struct NetSmem {
    float w1[H][kLdX];
    float w2[H][kLdH];
    float b1[H], b2[H], w3[H];
    float x[kNetTile][kLdX];
    float h1[kNetTile][kLdH];                // h1, then d loss / d pre-activation 1
    float d2[kNetTile][kLdH];                // d loss / d pre-activation 2 (GRAD only, the last member)
};
static_assert(offsetof(NetSmem, w2) % 16 == 0 && offsetof(NetSmem, x) % 16 == 0 && offsetof(NetSmem, h1) % 16 == 0 &&
                  offsetof(NetSmem, d2) % 16 == 0,
              "alignment of the rows");
template <bool GRAD> constexpr size_t net_smem() { return GRAD ? sizeof(NetSmem) : offsetof(NetSmem, d2); }

template <bool GRAD>
__global__ void __launch_bounds__(kNetThreads, 2)
mlp_net_kernel(const __nv_bfloat16 *__restrict__ w16, const float *__restrict__ feat, const float *__restrict__ target,
               const uint32_t *__restrict__ idx, int64_t m, float scale, float *__restrict__ part,
               double *__restrict__ loss, float *__restrict__ out, const uint8_t *__restrict__ lvl, double box,
               float margin)
{
    extern __shared__ __align__(16) unsigned char net_raw[];
    NetSmem &S = *(NetSmem *)net_raw;
    const int t = threadIdx.x, og = t & 7, sg = t >> 3;   // outputs og + 8 j, samples sg + 16 j
    for (int i = t; i < H * kLdX; i += kNetThreads) {
        const int j = i / kLdX, f = i % kLdX;
        S.w1[j][f] = f < IN ? bf(w16, oW1 + j * IN + f) : 0.f;
    }
    for (int i = t; i < H * H; i += kNetThreads) S.w2[i / H][i % H] = bf(w16, oW2 + i);
    for (int i = t; i < H; i += kNetThreads) {
        S.b1[i] = bf(w16, oB1 + i);
        S.b2[i] = bf(w16, oB2 + i);
        S.w3[i] = bf(w16, oW3 + i);
    }
    const float b3 = bf(w16, oB3);
    for (int i = t; i < kNetTile; i += kNetThreads) S.x[i][IN] = 0.f;
    // gradient shares: W2 (8 x 8) and W1 (8 x 4) over half of the samples,
    // W3, b1 and b2 of the thread's eight units over its samples
    float g2[8][8], g1[8][4], gw3[8], gb2[8], gb1[8], gb3 = 0.f;
    double lsum = 0.0;
    if constexpr (GRAD) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
#pragma unroll
            for (int b = 0; b < 8; ++b) g2[a][b] = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) g1[a][b] = 0.f;
            gw3[a] = gb2[a] = gb1[a] = 0.f;
        }
    }
    const int half = t >> 6, u = t & 63, ua = u & 7, ub = u >> 3;   // weight-gradient tiles
    for (int64_t base = (int64_t)blockIdx.x * kNetTile; base < m; base += (int64_t)gridDim.x * kNetTile) {
        const int nt = (int)min((int64_t)kNetTile, m - base);
        __syncthreads();
        for (int i = t; i < kNetTile * IN; i += kNetThreads) {
            const int r = i / IN, f = i - r * IN;
            float v = 0.f;
            if (r < nt) v = idx ? feat[(int64_t)idx[base + r] * IN + f] : feat[base * IN + i];
            S.x[r][f] = v;
        }
        __syncthreads();
        float acc[8][8];   // [output][sample]
        // ---- layer 1
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = S.b1[og + 8 * a];
#pragma unroll 1
        for (int k = 0; k < kLdX; k += 4) {
            float4 w[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) w[a] = *(const float4 *)&S.w1[og + 8 * a][k];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const float4 x = *(const float4 *)&S.x[sg + 16 * b][k];
#pragma unroll
                for (int a = 0; a < 8; ++a) fma4(acc[a][b], w[a], x);
            }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) S.h1[sg + 16 * b][og + 8 * a] = fmaxf(acc[a][b], 0.f);
        __syncthreads();
        // ---- layer 2
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = S.b2[og + 8 * a];
#pragma unroll 1
        for (int k = 0; k < H; k += 4) {
            float4 w[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) w[a] = *(const float4 *)&S.w2[og + 8 * a][k];
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const float4 x = *(const float4 *)&S.h1[sg + 16 * b][k];
#pragma unroll
                for (int a = 0; a < 8; ++a) fma4(acc[a][b], w[a], x);
            }
        }
        // ---- output: the eight lanes of a sample sum their units
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            float y = 0.f;
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                acc[a][b] = fmaxf(acc[a][b], 0.f);
                y = fmaf(S.w3[og + 8 * a], acc[a][b], y);
            }
            y += __shfl_xor_sync(0xffffffffu, y, 1);
            y += __shfl_xor_sync(0xffffffffu, y, 2);
            y += __shfl_xor_sync(0xffffffffu, y, 4);
            y += b3;
            const int r = sg + 16 * b;
            if constexpr (!GRAD) {
                if (og == 0 && r < nt) {
                    // with lvl: the search radius side(lvl) * exp(y + margin)
                    if (lvl) y = (float)(box / (double)(1u << lvl[base + r])) * expf(y + margin);
                    out[base + r] = y;
                }
            } else {
                float e = 0.f;
                if (r < nt) e = y - target[idx ? (int64_t)idx[base + r] : base + r];
                const float dy = 2.f * e * scale;
                if (og == 0) {
                    lsum += (double)e * (double)e * (double)scale;
                    gb3 += dy;
                }
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const float d = acc[a][b] > 0.f ? dy * S.w3[og + 8 * a] : 0.f;
                    gw3[a] = fmaf(dy, acc[a][b], gw3[a]);
                    gb2[a] += d;
                    S.d2[r][og + 8 * a] = d;
                }
            }
        }
        if constexpr (GRAD) {
            __syncthreads();
            // ---- W2's gradient: units {4 ua, 32 + 4 ua} .. x {4 ub, 32 + 4 ub} ..
#pragma unroll 1
            for (int r = half * (kNetTile / 2); r < (half + 1) * (kNetTile / 2); ++r) {
                const float4 p = *(const float4 *)&S.d2[r][4 * ua], q = *(const float4 *)&S.d2[r][32 + 4 * ua];
                const float4 v = *(const float4 *)&S.h1[r][4 * ub], w = *(const float4 *)&S.h1[r][32 + 4 * ub];
                const float d[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                const float h[8] = {v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w};
#pragma unroll
                for (int a = 0; a < 8; ++a)
#pragma unroll
                    for (int b = 0; b < 8; ++b) g2[a][b] = fmaf(d[a], h[b], g2[a][b]);
            }
            // ---- back through W2: units {4 og, 32 + 4 og} .., samples sg + 16 b
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
#pragma unroll 1
            for (int o = 0; o < H; o += 4) {
                float4 x[8];
#pragma unroll
                for (int b = 0; b < 8; ++b) x[b] = *(const float4 *)&S.d2[sg + 16 * b][o];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float4 p = *(const float4 *)&S.w2[o + c][4 * og], q = *(const float4 *)&S.w2[o + c][32 + 4 * og];
                    const float w[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int b = 0; b < 8; ++b) {
                        const float d = c == 0 ? x[b].x : c == 1 ? x[b].y : c == 2 ? x[b].z : x[b].w;
#pragma unroll
                        for (int a = 0; a < 8; ++a) acc[a][b] = fmaf(w[a], d, acc[a][b]);
                    }
                }
            }
            __syncthreads();   // every read of h1 as activations is done
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                float4 *lo = (float4 *)&S.h1[sg + 16 * b][4 * og], *hi = (float4 *)&S.h1[sg + 16 * b][32 + 4 * og];
                const float4 p = *lo, q = *hi;
                const float h[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                float d[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    d[a] = h[a] > 0.f ? acc[a][b] : 0.f;
                    gb1[a] += d[a];
                }
                *lo = make_float4(d[0], d[1], d[2], d[3]);
                *hi = make_float4(d[4], d[5], d[6], d[7]);
            }
            __syncthreads();
            // ---- W1's gradient: units {4 ua, 32 + 4 ua} .. x features 4 ub ..
            if (ub < kLdX / 4) {
#pragma unroll 1
                for (int r = half * (kNetTile / 2); r < (half + 1) * (kNetTile / 2); ++r) {
                    const float4 p = *(const float4 *)&S.h1[r][4 * ua], q = *(const float4 *)&S.h1[r][32 + 4 * ua];
                    const float4 v = *(const float4 *)&S.x[r][4 * ub];
                    const float d[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                    const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int a = 0; a < 8; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) g1[a][b] = fmaf(d[a], x[b], g1[a][b]);
                }
            }
        }
    }
    if constexpr (GRAD) {
        // the block's share: the threads' parts meet in shared memory
        __syncthreads();
        float *G = &S.h1[0][0];
        static_assert(sizeof(S.h1) >= sizeof(float) * NP, "a gradient fits the activations' space");
        for (int i = t; i < NP; i += kNetThreads) G[i] = 0.f;
        __syncthreads();
        for (int h = 0; h < 2; ++h) {
            if (half == h) {
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const int ra = (a < 4 ? 4 * ua : 28 + 4 * ua) + a;
#pragma unroll
                    for (int b = 0; b < 8; ++b) G[oW2 + ra * H + (b < 4 ? 4 * ub : 28 + 4 * ub) + b] += g2[a][b];
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if (4 * ub + b < IN) G[oW1 + ra * IN + 4 * ub + b] += g1[a][b];
                }
            }
            __syncthreads();
        }
        // units' sums: the four lanes of a warp that share og, then the warps
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            float v[3] = {gw3[a], gb2[a], gb1[a]};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c] += __shfl_xor_sync(0xffffffffu, v[c], 8);
                v[c] += __shfl_xor_sync(0xffffffffu, v[c], 16);
            }
            if ((t & 31) < 8) {
                atomicAdd(&G[oW3 + og + 8 * a], v[0]);
                atomicAdd(&G[oB2 + og + 8 * a], v[1]);
                atomicAdd(&G[oB1 + (a < 4 ? 4 * og : 28 + 4 * og) + a], v[2]);
            }
        }
        if (og == 0) atomicAdd(&G[oB3], gb3);
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if ((t & 31) == 0) atomicAdd(loss, lsum);
        __syncthreads();
        for (int i = t; i < NP; i += kNetThreads) part[(int64_t)blockIdx.x * NP + i] = G[i];
    }
}

// grad = the sum of the blocks' shares, in fp64: eight warps per 32
// parameters, each over every eighth share.
__global__ void __launch_bounds__(256) grad_sum_kernel(const float *__restrict__ part, int blocks, float *__restrict__ grad)
{
    __shared__ double s[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    double v = 0.0;
    if (i < NP)
#pragma unroll 4
        for (int b = w; b < blocks; b += 8) v += (double)part[(int64_t)b * NP + i];
    s[w][lane] = v;
    __syncthreads();
    if (w == 0 && i < NP) {
        for (int k = 1; k < 8; ++k) v += s[k][lane];
        grad[i] = (float)v;
    }
}

__global__ void adam_kernel(float *__restrict__ w, __nv_bfloat16 *__restrict__ w16,
                            float *__restrict__ mo, float *__restrict__ ve,
                            const float *__restrict__ g, float lr, float bc1, float bc2)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < NP; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float m = b1 * mo[i] + (1.f - b1) * gi;
        const float v = b2 * ve[i] + (1.f - b2) * gi * gi;
        mo[i] = m;
        ve[i] = v;
        const float mh = m / bc1, vh = v / bc2;
        const float nw = w[i] - lr * mh / (sqrtf(vh) + eps);
        w[i] = nw;
        w16[i] = __float2bfloat16_rn(nw);
    }
}

__global__ void to_bf16_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ w16, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        w16[i] = __float2bfloat16_rn(w[i]);
}

// Blocks of the network kernels: a tile each, as many as are resident (two
// per SM with gradients, three without).
int64_t net_blocks(hop_ctx *c, int64_t m, int per_sm)
{
    return std::max<int64_t>(1, std::min<int64_t>((m + kNetTile - 1) / kNetTile, (int64_t)c->num_sms * per_sm));
}

// grad = the gradient (written whole), *loss += its loss.
int grad_launch(hop_ctx *c, const float *feat, const float *target, const uint32_t *idx, int64_t m,
                float scale, float *grad, double *loss)
{
    const int64_t blocks = net_blocks(c, m, 2);
    float *part = (float *)ctx_buf(c, S_MLP_PART, (size_t)blocks * NP * sizeof(float));
    if (!part) return HOP_ENOMEM;
    constexpr size_t smem = net_smem<true>();
    HOP_CUDA(c, cudaFuncSetAttribute(mlp_net_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    mlp_net_kernel<true><<<(unsigned)blocks, kNetThreads, smem, c->stream>>>(
        (const __nv_bfloat16 *)c->mlp->w16, feat, target, idx, m, scale, part, loss, nullptr, nullptr, 1.0, 0.f);
    HOP_LAUNCH(c);
    grad_sum_kernel<<<(NP + 31) / 32, 256, 0, c->stream>>>(part, (int)blocks, grad);
    HOP_LAUNCH(c);
    return HOP_OK;
}

// out[s] = MLP(feat[s]); with lvl != null the search radius side(lvl[s]) *
// exp(MLP + margin) instead.
int forward_launch(hop_ctx *c, const float *feat, int64_t m, float *out, const uint8_t *lvl, double box, float margin)
{
    constexpr size_t smem = net_smem<false>();
    HOP_CUDA(c, cudaFuncSetAttribute(mlp_net_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    mlp_net_kernel<false><<<(unsigned)net_blocks(c, m, 3), kNetThreads, smem, c->stream>>>(
        (const __nv_bfloat16 *)c->mlp->w16, feat, nullptr, nullptr, m, 0.f, nullptr, nullptr, out, lvl, box, margin);
    HOP_LAUNCH(c);
    return HOP_OK;
}

}  // namespace

int mlp_ensure(hop_ctx *c)
{
    if (c->mlp->w32) return HOP_OK;
    char *p = nullptr;
    const size_t bytes = sizeof(float) * NP * 4 + sizeof(uint16_t) * NP + 256;
    HOP_CUDA(c, cudaMalloc(&p, bytes));
    HOP_CUDA(c, cudaMemset(p, 0, bytes));
    c->mlp->w32 = (float *)p;
    c->mlp->m = c->mlp->w32 + NP;
    c->mlp->v = c->mlp->m + NP;
    c->mlp->g = c->mlp->v + NP;
    c->mlp->w16 = (uint16_t *)(c->mlp->g + NP);
    return HOP_OK;
}

void mlp_free(hop_ctx *c)
{
    for (MlpState &m : c->mlp_bank) {
        if (m.w32) cudaFree(m.w32);
        m = MlpState();
    }
}

int mlp_forward_dev(hop_ctx *c, const float *feat, int64_t m, float *out)
{
    return forward_launch(c, feat, m, out, nullptr, 1.0, 0.f);
}

namespace {

template <bool NET>
int radius_launch(hop_ctx *c, const void *spos, const uint64_t *keys, const uint32_t *cellT, int Ld, int64_t n,
                  int64_t n_chunks, int qpw, double box, const SegDesc *seg, int B, int k, float margin, float *chunk_r)
{
    constexpr size_t smem = rad_smem<NET>();
    HOP_CUDA(c, cudaFuncSetAttribute(radius_kernel<NET>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    HOP_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, radius_kernel<NET>, kRadThreads, smem));
    int64_t blocks = (n_chunks + kRadThreads - 1) / kRadThreads;
    blocks = std::min<int64_t>(blocks, (int64_t)c->num_sms * std::max(per_sm, 1));
    blocks = std::max<int64_t>(blocks, 1);
    radius_kernel<NET><<<(unsigned)blocks, kRadThreads, smem, c->stream>>>(
        NET ? (const __nv_bfloat16 *)c->mlp->w16 : nullptr, (const float4 *)spos, keys, cellT, Ld, n, n_chunks, qpw,
        (float)box, (float)(1.0 / box), seg, B, margin, k, chunk_r);
    HOP_LAUNCH(c);
    return HOP_OK;
}

}  // namespace

// The closed-form radius (float32 positions) with the same kernel.
int radius_closed(hop_ctx *c, const void *spos, const uint64_t *keys, const uint32_t *cellT, int Ld, int64_t n,
                  int64_t n_chunks, int qpw, double box, const SegDesc *seg, int B, int k, float log_margin,
                  float *chunk_r)
{
    return radius_launch<false>(c, spos, keys, cellT, Ld, n, n_chunks, qpw, box, seg, B, k, log_margin, chunk_r);
}

int mlp_radius(hop_ctx *c, const void *spos, const uint64_t *keys, const uint32_t *cellT, int Ld,
               int64_t n, const hop_params *p, int qpw, float *chunk_r)
{
    const int64_t nc = (n + qpw - 1) / qpw;
    if (!p->pos_is_f64) return radius_launch<true>(c, spos, keys, cellT, Ld, n, nc, qpw, p->box, nullptr, 0, 0, c->mlp->log_margin, chunk_r);
    float *feat = (float *)ctx_buf(c, S_MLP_TMP, nc * IN * sizeof(float));
    uint8_t *lvl = (uint8_t *)ctx_buf(c, S_CHUNK_LVL, nc);
    if (!feat || !lvl) return HOP_ENOMEM;
    int rc = chunk_features(c, spos, keys, cellT, Ld, n, p->pos_is_f64 != 0, p->box, qpw, feat, lvl,
                            nullptr, nullptr);
    if (rc) return rc;
    return forward_launch(c, feat, nc, chunk_r, lvl, p->box, c->mlp->log_margin);
}

// Batched pass: features of every chunk (with the cell side of its own
// subvolume in chunk_r), then radius = side * exp(MLP + margin) in place.
int mlp_radius_seg(hop_ctx *c, const void *spos, const uint64_t *keys, const uint32_t *cellT,
                   const SegDesc *seg, int B, int64_t n_chunks, int qpw, int k, float *chunk_r)
{
    if (!c->mlp->loaded) return ctx_fail(c, HOP_ENOMODEL, "no radius network loaded (hop_mlp_load)");
    (void)k;
    return radius_launch<true>(c, spos, keys, cellT, 0, 0, n_chunks, qpw, 1.0, seg, B, 0, c->mlp->log_margin, chunk_r);
}

extern "C" {

int hop_mlp_load(hop_ctx *c, const float *params_host, float log_margin)
{
    if (!c || !params_host) return HOP_EINVAL;
    HOP_CUDA(c, cudaSetDevice(c->device));
    int rc = mlp_ensure(c);
    if (rc) return rc;
    HOP_CUDA(c, cudaMemcpyAsync(c->mlp->w32, params_host, sizeof(float) * NP, cudaMemcpyHostToDevice, c->stream));
    HOP_CUDA(c, cudaMemsetAsync(c->mlp->m, 0, sizeof(float) * NP * 2, c->stream));
    to_bf16_kernel<<<8, 256, 0, c->stream>>>(c->mlp->w32, (__nv_bfloat16 *)c->mlp->w16, NP);
    HOP_LAUNCH(c);
    HOP_CUDA(c, cudaStreamSynchronize(c->stream));
    c->mlp->loaded = true;
    c->mlp->log_margin = log_margin;
    c->mlp->step = 0;
    return HOP_OK;
}

int hop_mlp_get(hop_ctx *c, float *params_host)
{
    if (!c || !params_host) return HOP_EINVAL;
    if (!c->mlp->loaded) return ctx_fail(c, HOP_ENOMODEL, "no network loaded");
    HOP_CUDA(c, cudaMemcpyAsync(params_host, c->mlp->w32, sizeof(float) * NP, cudaMemcpyDeviceToHost, c->stream));
    HOP_CUDA(c, cudaStreamSynchronize(c->stream));
    return HOP_OK;
}

int hop_mlp_samples(hop_ctx *c, float *feat, float *target, int64_t cap, int64_t *n_chunks)
{
    if (!c || !n_chunks) return HOP_EINVAL;
    if (!c->last_spos) return ctx_fail(c, HOP_EINVAL, "no density pass to take samples from");
    const int64_t nc = (c->last_n + c->last_qpw - 1) / c->last_qpw;
    *n_chunks = nc;
    if (!feat || !target) return HOP_OK;
    if (cap < nc) return ctx_fail(c, HOP_ETABLE, "sample capacity too small");
    HOP_CUDA(c, cudaSetDevice(c->device));
    uint8_t *lvl = (uint8_t *)ctx_buf(c, S_CHUNK_LVL, nc);
    if (!lvl) return HOP_ENOMEM;
    int rc = chunk_features(c, c->last_spos, c->last_keys, c->last_cellT, c->last_level_dense, c->last_n,
                            c->last_f64, c->last_box, c->last_qpw, feat, lvl, c->last_rk, target);
    if (rc) return rc;
    HOP_CUDA(c, cudaStreamSynchronize(c->stream));
    return HOP_OK;
}

int hop_mlp_forward(hop_ctx *c, const float *feat, int64_t m, float *out)
{
    if (!c || !feat || !out || m < 0) return HOP_EINVAL;
    if (!c->mlp->loaded) return ctx_fail(c, HOP_ENOMODEL, "no network loaded");
    HOP_CUDA(c, cudaSetDevice(c->device));
    if (m == 0) return HOP_OK;
    return mlp_forward_dev(c, feat, m, out);
}

int hop_mlp_grad(hop_ctx *c, const float *feat, const float *target, int64_t m, double *loss,
                 float *grad)
{
    if (!c || !feat || !target || !grad || !loss || m <= 0) return HOP_EINVAL;
    if (!c->mlp->loaded) return ctx_fail(c, HOP_ENOMODEL, "no network loaded");
    HOP_CUDA(c, cudaSetDevice(c->device));
    double *dl = (double *)ctx_buf(c, S_MISC, 256);
    if (!dl) return HOP_ENOMEM;
    HOP_CUDA(c, cudaMemsetAsync(dl, 0, sizeof(double), c->stream));
    int rc = grad_launch(c, feat, target, nullptr, m, 1.f / (float)m, grad, dl);
    if (rc) return rc;
    HOP_CUDA(c, cudaMemcpyAsync(c->h_pinned, dl, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    HOP_CUDA(c, cudaStreamSynchronize(c->stream));
    *loss = *(double *)c->h_pinned;
    return HOP_OK;
}

int hop_mlp_train(hop_ctx *c, const float *feat, const float *target, int64_t m, int32_t epochs,
                  int32_t batch, float lr, uint64_t seed, double *final_loss)
{
    if (!c || !feat || !target || m <= 0 || epochs <= 0 || batch <= 0) return HOP_EINVAL;
    if (!c->mlp->loaded) return ctx_fail(c, HOP_ENOMODEL, "load initial parameters first (hop_mlp_load)");
    HOP_CUDA(c, cudaSetDevice(c->device));
    uint32_t *perm = (uint32_t *)ctx_buf(c, S_MLP_TMP, m * sizeof(uint32_t));
    double *dl = (double *)ctx_buf(c, S_MISC, 256);
    if (!perm || !dl) return HOP_ENOMEM;
    std::vector<uint32_t> hp((size_t)m);
    uint64_t st = seed;
    auto next = [&]() {
        // SplitMix64 step (Steele, Lea & Flood 2014)
        uint64_t z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    double last = 0.0;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int64_t i = 0; i < m; ++i) hp[i] = (uint32_t)i;
        for (int64_t i = m - 1; i > 0; --i) std::swap(hp[i], hp[next() % (uint64_t)(i + 1)]);
        HOP_CUDA(c, cudaMemcpyAsync(perm, hp.data(), m * sizeof(uint32_t), cudaMemcpyHostToDevice, c->stream));
        HOP_CUDA(c, cudaMemsetAsync(dl, 0, sizeof(double), c->stream));
        for (int64_t b = 0; b < m; b += batch) {
            const int64_t bs = std::min<int64_t>(batch, m - b);
            // loss of each batch is its mean; weight it by bs/m for the epoch mean
            int rc = grad_launch(c, feat, target, perm + b, bs, 1.f / (float)bs, c->mlp->g, dl);
            if (rc) return rc;
            c->mlp->step += 1;
            const float bc1 = 1.f - powf(0.9f, (float)c->mlp->step);
            const float bc2 = 1.f - powf(0.999f, (float)c->mlp->step);
            adam_kernel<<<(NP + 255) / 256, 256, 0, c->stream>>>(c->mlp->w32, (__nv_bfloat16 *)c->mlp->w16,
                                                                c->mlp->m, c->mlp->v, c->mlp->g, lr, bc1, bc2);
            HOP_LAUNCH(c);
        }
        HOP_CUDA(c, cudaMemcpyAsync(c->h_pinned, dl, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        HOP_CUDA(c, cudaStreamSynchronize(c->stream));
        // sum over batches of (batch mean loss); convert to a per-sample mean
        const double nb = (double)((m + batch - 1) / batch);
        last = *(double *)c->h_pinned / nb;
    }
    if (final_loss) *final_loss = last;
    return HOP_OK;
}

}  // extern "C"
