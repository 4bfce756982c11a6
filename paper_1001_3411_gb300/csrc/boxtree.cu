// Bounding boxes over the Morton-sorted particles: level 0 holds the box of
// every eight consecutive particles, each further level the box of eight
// consecutive nodes below.  A node's children and particles follow from its
// number (child c of node i is 8 i + c, one level down), so the tree is two
// arrays of corners and nothing else.  A range search needs no cell lookups
// and no search in the sorted keys, and its leaves are 128-byte lines of
// positions whatever the local density.
#include "hop_internal.cuh"

#include <algorithm>

namespace {

constexpr int kBoxThreads = 512;   // inputs of a block: 64, 8 and 1 nodes of the next three levels

struct Aabb {
    float lx, ly, lz, hx, hy, hz;
    __device__ __forceinline__ void join(const Aabb &o)
    {
        lx = fminf(lx, o.lx);
        ly = fminf(ly, o.ly);
        lz = fminf(lz, o.lz);
        hx = fmaxf(hx, o.hx);
        hy = fmaxf(hy, o.hy);
        hz = fmaxf(hz, o.hz);
    }
    __device__ __forceinline__ void join_lanes(int o)
    {
        Aabb b;
        b.lx = __shfl_xor_sync(0xffffffffu, lx, o);
        b.ly = __shfl_xor_sync(0xffffffffu, ly, o);
        b.lz = __shfl_xor_sync(0xffffffffu, lz, o);
        b.hx = __shfl_xor_sync(0xffffffffu, hx, o);
        b.hy = __shfl_xor_sync(0xffffffffu, hy, o);
        b.hz = __shfl_xor_sync(0xffffffffu, hz, o);
        join(b);
    }
    __device__ __forceinline__ void store(float4 *lo, float4 *hi, int64_t i) const
    {
        lo[i] = make_float4(lx, ly, lz, 0.f);
        hi[i] = make_float4(hx, hy, hz, 0.f);
    }
};

// Three levels above the m inputs (particles, or the nodes at in_lo / in_hi):
// out[0], out[1], out[2] are their first nodes.  Nodes past the last input
// are empty (lo = +inf, hi = -inf).  HBM-bound: 16 bytes read and 4.6 written
// per particle.
template <bool LEAF>
__global__ void __launch_bounds__(kBoxThreads) box_levels_kernel(const float4 *__restrict__ in_lo,
                                                                 const float4 *__restrict__ in_hi, int64_t m,
                                                                 float4 *__restrict__ lo, float4 *__restrict__ hi,
                                                                 uint32_t out0, uint32_t out1, uint32_t out2)
{
    __shared__ Aabb sw[kBoxThreads / 32];
    const int64_t i = (int64_t)blockIdx.x * kBoxThreads + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Aabb b = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    if (i < m) {
        const float4 l = in_lo[i];
        float4 h = l;
        if constexpr (!LEAF) h = in_hi[i];
        b = {l.x, l.y, l.z, h.x, h.y, h.z};
    }
    b.join_lanes(1);
    b.join_lanes(2);
    b.join_lanes(4);
    if ((lane & 7) == 0) b.store(lo, hi, (int64_t)out0 + (i >> 3));
    b.join_lanes(8);
    b.join_lanes(16);
    if (lane == 0) sw[warp] = b;
    __syncthreads();
    if (threadIdx.x < 8) {
        b = sw[2 * threadIdx.x];
        b.join(sw[2 * threadIdx.x + 1]);
        b.store(lo, hi, (int64_t)out1 + (int64_t)blockIdx.x * 8 + threadIdx.x);
    }
    if (threadIdx.x == 0) {
        b = sw[0];
        for (int w = 1; w < kBoxThreads / 32; ++w) b.join(sw[w]);
        b.store(lo, hi, (int64_t)out2 + blockIdx.x);
    }
}

}  // namespace

// Builds the levels up to the first with at most kBoxTop nodes over all n
// particles.
int box_tree_build(hop_ctx *c, const float4 *spos, int64_t n, BoxTree *t)
{
    // blocks per triple of levels, a multiple of eight so that the children
    // of every node exist
    int64_t blocks[4], m = n, total = 0;
    int triples = 0;
    for (;;) {
        const int64_t b = ((m + kBoxThreads - 1) / kBoxThreads + 7) / 8 * 8;
        blocks[triples] = b;
        t->off[3 * triples] = (uint32_t)total;
        t->off[3 * triples + 1] = (uint32_t)(total + 64 * b);
        t->off[3 * triples + 2] = (uint32_t)(total + 72 * b);
        total += 73 * b;
        ++triples;
        m = (m + kBoxThreads - 1) / kBoxThreads;
        if (m <= kBoxTop) break;
        if (triples == 4) return ctx_fail(c, HOP_EINVAL, "too many particles for the box levels");
        m = b;
    }
    float4 *buf = (float4 *)ctx_buf(c, S_BOX, (size_t)total * 2 * sizeof(float4));
    if (!buf) return HOP_ENOMEM;
    float4 *lo = buf, *hi = buf + total;
    t->lo = lo;
    t->hi = hi;
    for (int i = 0; i < triples; ++i) {
        const uint32_t *o = t->off + 3 * i;
        if (i == 0)
            box_levels_kernel<true><<<(unsigned)blocks[0], kBoxThreads, 0, c->stream>>>(spos, nullptr, n, lo, hi, o[0],
                                                                                      o[1], o[2]);
        else
            box_levels_kernel<false><<<(unsigned)blocks[i], kBoxThreads, 0, c->stream>>>(lo + o[-1], hi + o[-1],
                                                                                       blocks[i - 1], lo, hi, o[0], o[1],
                                                                                       o[2]);
        HOP_LAUNCH(c);
    }
    return HOP_OK;
}
