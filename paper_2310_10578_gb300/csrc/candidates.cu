// candidates.cu -- the ray launch of the large-scene mode on the device.
//
// The paper's own path search is a ray tracer (Sec. III, BVH-accelerated);
// for order-3 reflections among ~100k faces this library takes candidate
// face sequences from a forward launch from the transmitter and validates
// each one exactly per receiver (the planar class kernel).  The launch rule
// (shared with the host launch in bvh.cu and with the oracle): n_rays
// directions of the spherical Fibonacci lattice; each ray is reflected
// specularly at the nearest triangle hit (Moller--Trumbore, parameter >
// 1e-9, the face it leaves excluded, equal parameters to the lower triangle
// index) up to max_order times; every prefix of its face sequence is a
// candidate; the distinct sequences sorted by (order, faces).
//
// Here: k_ray_launch, one warp per ray, walks the scene's triangle BVH (FP32
// box and triangle filters, both conservative; FP64 triangle tests of what
// passes); this file is compiled without FMA contraction, so every FP64
// operation rounds as in the host code (-ffp-contract=off) and both launches
// trace bit-identical rays from the same host-made directions and face
// normals.  Each sequence a warp finds goes into a hash set in device memory,
// and into the list when it is new.  k_cand_finish, one block, sorts the
// distinct (order, faces) keys in shared memory (bitonic) and writes the list
// with the source's FP64 images after each reflection, as rt_set_candidates
// would upload them.  Its length goes to device memory, where the class
// kernels read it: no host round trip.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace creep {

namespace {

constexpr int FINISH_THREADS = 1024;
constexpr unsigned long long KEY_NONE = ~0ull;

struct D3 { double x, y, z; };
__device__ __forceinline__ D3 d3(double x, double y, double z) { D3 r; r.x = x; r.y = y; r.z = z; return r; }
__device__ __forceinline__ D3 sub(D3 a, D3 b) { return d3(a.x - b.x, a.y - b.y, a.z - b.z); }
// the host's expression trees: ((a.x b.x + a.y b.y) + a.z b.z), a.y b.z - a.z b.y, ...
__device__ __forceinline__ double dotd(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 crossd(D3 a, D3 b) {
    return d3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

// nearest-hit parameter of the ray o + t d with the closed triangle, or -1
__device__ double ray_tri_d(D3 o, D3 d, D3 v0, D3 v1, D3 v2) {
    D3 e1 = sub(v1, v0), e2 = sub(v2, v0);
    D3 p = crossd(d, e2);
    double det = dotd(e1, p);
    if (fabs(det) < 1e-14) return -1.0;
    double inv = 1.0 / det;
    D3 sv = sub(o, v0);
    double u = dotd(sv, p) * inv;
    if (u < 0.0 || u > 1.0) return -1.0;
    D3 q = crossd(sv, e1);
    double v = dotd(d, q) * inv;
    if (v < 0.0 || u + v > 1.0) return -1.0;
    return dotd(e2, q) * inv;
}

// the ray's parameter interval [0, tmax] meets the box?  In FP32 on the
// rounded ray: conservative, since the node
// boxes are padded outwards by 1e-4 m + 1e-6 of the coordinate, far beyond
// the rounding of the ray and of this test over the scene's extent; tmax is
// rounded up.  It only prunes the walk: every box holding a triangle whose
// FP64 hit parameter is <= tmax is kept, so the nearest hit is the FP64 one.
__device__ __forceinline__ bool ray_box_f(const float o[3], const float d[3], float4 lo, float4 hi, float tmax) {
    float t0 = 0.0f, t1 = tmax;
    const float bl[3] = {lo.x, lo.y, lo.z}, bh[3] = {hi.x, hi.y, hi.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (d[k] == 0.0f) {
            if (o[k] < bl[k] || o[k] > bh[k]) return false;
            continue;
        }
        const float inv = 1.0f / d[k];
        float a = (bl[k] - o[k]) * inv, b = (bh[k] - o[k]) * inv;
        if (a > b) { const float w = a; a = b; b = w; }
        t0 = fmaxf(t0, a);
        t1 = fminf(t1, b);
        if (t0 > t1) return false;
    }
    return true;
}

__device__ __forceinline__ D3 vtx(const float4 *tri, int t, int k) {
    const float4 v = tri[3 * t + k];
    return d3(v.x, v.y, v.z);
}

// key of a prefix: order (2 bits), then face + 1 of each slot (20 bits, 0 = none)
__device__ __forceinline__ unsigned long long seq_key(int k, const int fs[3]) {
    return ((unsigned long long)k << 60) | ((unsigned long long)(fs[0] + 1) << 40) |
           ((unsigned long long)(fs[1] + 1) << 20) | (unsigned long long)(fs[2] + 1);
}

// May the FP64 test of this triangle find a hit with parameter in (0, best]?
// FP32, conservative: for each of u, v, 1 - u - v and t the numerator is
// compared with minus a bound of its rounding -- the coordinates' own (6e-8 of
// scale, the largest |coordinate| of the ray and the triangle) and that of
// some ten operations, 1e-5 (|s| + scale) |edge| in all, two orders above it.
// (The FP64 test divides by det; the signs of its u, v and 1 - u - v are those
// of the numerators here.)  FP64 decides, too, where a product overflows, with
// coordinates from 1e12 m on (vertices may be any finite floats).
__device__ __forceinline__ bool ray_tri_may(const float o[3], const float d[3], float4 a, float4 b, float4 c,
                                            float scale, float best) {
    const float e1x = b.x - a.x, e1y = b.y - a.y, e1z = b.z - a.z, e2x = c.x - a.x, e2y = c.y - a.y, e2z = c.z - a.z;
    const float sx = o[0] - a.x, sy = o[1] - a.y, sz = o[2] - a.z;
    const float px = d[1] * e2z - d[2] * e2y, py = d[2] * e2x - d[0] * e2z, pz = d[0] * e2y - d[1] * e2x;
    const float qx = sy * e1z - sz * e1y, qy = sz * e1x - sx * e1z, qz = sx * e1y - sy * e1x;
    float det = e1x * px + e1y * py + e1z * pz, u = sx * px + sy * py + sz * pz, v = d[0] * qx + d[1] * qy + d[2] * qz,
          t = e2x * qx + e2y * qy + e2z * qz;
    const float l1 = fabsf(e1x) + fabsf(e1y) + fabsf(e1z), l2 = fabsf(e2x) + fabsf(e2y) + fabsf(e2z);
    const float m = 1e-5f * (fabsf(sx) + fabsf(sy) + fabsf(sz) + scale), eu = m * l2, ev = m * l1;
    const float ed = 1e-5f * l1 * l2;
    if (fabsf(det) <= ed) return true;           // the plane nearly along the ray: let FP64 decide
    if (!(fabsf(det) + fabsf(u) + fabsf(v) + fabsf(t) < INFINITY)) return true;
    if (det < 0.0f) { det = -det; u = -u; v = -v; t = -t; }
    if (u < -eu || v < -ev || u + v > det + ed + eu + ev) return false;
    const float et = m * l1 * l2;
    return t > -et && t - et <= best * (det + ed);
}

// One warp per ray.  The walk takes up to 32 nodes at a time from the warp's
// stack in shared memory, a node a lane: an inner node's two children are
// tested together (they are adjacent) and the ones the ray meets pushed, far
// ones below near ones; a leaf's triangles are filtered in FP32 and the rest
// tested in FP64, and the nearest hit so far, shared by the warp, prunes the
// boxes.  The nearest hit is unique (equal parameters go to the lower
// triangle), so the order of the tests changes nothing.
//   What bounds it is the chain of a ray's bounces: per bounce some twenty
// stack rounds of two dependent loads, and about 1200 cycles per FP64 test
// (its division alone 430).  A thread per ray had run the nodes of a walk one
// after the other, with 3.7 lanes of a warp active and 1.6 % of the warps an
// SM can hold: 28.5 ms for 4096 rays of order 3 among 193 572 triangles, and
// 10.0 ms among 7 800; this one 0.24 ms and 0.10 ms.
constexpr int RAY_WARPS = 4;
constexpr int RAY_STACK = 1088;
__global__ void __launch_bounds__(32 * RAY_WARPS)
k_ray_launch(const float4 *__restrict__ tri, const float4 *__restrict__ bvh, const int *__restrict__ bvh_tri,
             const double *__restrict__ fn, const double *__restrict__ dir, double ox, double oy, double oz,
             int n_rays, int max_order, unsigned long long *__restrict__ table, unsigned long long *__restrict__ list,
             int *__restrict__ ctr) {
    __shared__ int s_stack[RAY_WARPS][RAY_STACK];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * RAY_WARPS + warp;
    if (i >= n_rays) return;
    int *stack = s_stack[warp];
    D3 o = d3(ox, oy, oz), d = d3(dir[3 * (size_t)i], dir[3 * (size_t)i + 1], dir[3 * (size_t)i + 2]);
    int fs[3] = {-1, -1, -1}, last = -1;
    for (int k = 0; k < max_order; ++k) {
        double best = INFINITY;
        int bt = -1, sp = 1;
        float bestf = INFINITY;
        const float of[3] = {(float)o.x, (float)o.y, (float)o.z}, df[3] = {(float)d.x, (float)d.y, (float)d.z};
        const float so = fmaxf(fmaxf(fabsf(of[0]), fabsf(of[1])), fabsf(of[2]));
        __syncwarp();
        if (lane == 0) stack[0] = 0;
        __syncwarp();
        while (sp > 0) {
            // near the stack's end nodes go one at a time: a plain depth-first
            // walk, which adds at most the tree's depth (<= 32) to it
            const int np = min(min(32, sp), max(1, RAY_STACK - 40 - sp));
            int first = 0, count = 0, push = 0;
            bool flip = false;
            sp -= np;
            if (lane < np) {
                const int nd = stack[sp + lane];
                const float4 lo = bvh[2 * nd], hi = bvh[2 * nd + 1];
                first = __float_as_int(lo.w);
                count = __float_as_int(hi.w);
                if (!ray_box_f(of, df, lo, hi, bestf)) {
                    count = 0;                    // (pushed before a nearer hit was found)
                } else if (count == 0) {
                    const float4 l0 = bvh[2 * first], h0 = bvh[2 * first + 1], l1 = bvh[2 * first + 2],
                                 h1 = bvh[2 * first + 3];
                    if (ray_box_f(of, df, l0, h0, bestf)) push |= 1;
                    if (ray_box_f(of, df, l1, h1, bestf)) push |= 2;
                    // the nearer child by its box's centre along the ray
                    flip = (l1.x + h1.x - l0.x - h0.x) * df[0] + (l1.y + h1.y - l0.y - h0.y) * df[1] +
                               (l1.z + h1.z - l0.z - h0.z) * df[2] > 0.0f;
                }
            }
            __syncwarp();
            // (an only child counts as near)
            const bool both = push == 3;
            const unsigned mb = __ballot_sync(0xffffffffu, both), m1 = __ballot_sync(0xffffffffu, push != 0);
            const unsigned lt = (1u << lane) - 1u;
            if (sp + __popc(mb) + __popc(m1) > RAY_STACK) {
                if (lane == 0) atomicExch(ctr + 1, 1);        // (a tree deeper than the build makes)
                break;
            }
            if (both) stack[sp + __popc(mb & lt)] = first + (flip ? 1 : 0);
            if (push) stack[sp + __popc(mb) + __popc(m1 & lt)] = first + (both ? (flip ? 0 : 1) : push - 1);
            sp += __popc(mb) + __popc(m1);
            __syncwarp();
            // leaves: which triangles pass the FP32 filter
            unsigned cand = 0;
            for (int j = 0; j < count; ++j) {
                const int t = bvh_tri[first + j];
                const float4 a = tri[3 * t], b = tri[3 * t + 1], c = tri[3 * t + 2];
                if (__float_as_int(a.w) == last) continue;
                const float sc = fmaxf(so, fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fabsf(a.z)));
                if (ray_tri_may(of, df, a, b, c, sc, bestf)) cand |= 1u << j;
            }
            bool hit = false;
            while (__any_sync(0xffffffffu, cand != 0)) {
                if (cand) {
                    const int t = bvh_tri[first + __ffs(cand) - 1];
                    cand &= cand - 1;
                    const double h = ray_tri_d(o, d, vtx(tri, t, 0), vtx(tri, t, 1), vtx(tri, t, 2));
                    if (h > 1e-9 && (h < best || (h == best && t < bt))) { best = h; bt = t; hit = true; }
                }
            }
            if (__any_sync(0xffffffffu, hit)) {
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) {
                    const double h = __shfl_xor_sync(0xffffffffu, best, w);
                    const int t = __shfl_xor_sync(0xffffffffu, bt, w);
                    if (t >= 0 && (bt < 0 || h < best || (h == best && t < bt))) { best = h; bt = t; }
                }
                bestf = __double2float_ru(best);
            }
        }
        if (bt < 0) break;
        const int f = __float_as_int(tri[3 * bt].w);
        fs[k] = f;
        if (lane == 0) {
            // into the set (open addressing, at most half full); new: into the list
            const unsigned long long key = seq_key(k + 1, fs);
            unsigned slot = (unsigned)((key * 0x9E3779B97F4A7C15ull) >> 40) & (RT_DEV_CAND_TABLE - 1);
            for (int n = 0; n < RT_DEV_CAND_TABLE; ++n) {
                const unsigned long long old = atomicCAS(table + slot, KEY_NONE, key);
                if (old == KEY_NONE) list[atomicAdd(ctr + 2, 1)] = key;
                if (old == KEY_NONE || old == key) break;
                slot = (slot + 1) & (RT_DEV_CAND_TABLE - 1);
            }
        }
        const D3 n = d3(fn[3 * (size_t)f], fn[3 * (size_t)f + 1], fn[3 * (size_t)f + 2]);
        o = d3(o.x + d.x * best, o.y + d.y * best, o.z + d.z * best);
        const double dn = 2.0 * dotd(d, n);
        d = d3(d.x - n.x * dn, d.y - n.y * dn, d.z - n.z * dn);
        last = f;
    }
}

// One block: sort the n_list[0] distinct keys of the list, write them and
// their images.  Bitonic over the next power of two (the launch reserves
// shared memory for every prefix being distinct): the steps of a warp's own 32
// slots run on registers by shuffles, so a stage of width k takes log2(k) - 4
// block barriers (2093 distinct keys of 12 288 prefixes: 0.08 ms, against 0.34
// ms for sorting every prefix and dropping the repeated ones after).
__global__ void __launch_bounds__(FINISH_THREADS) k_cand_finish(const unsigned long long *__restrict__ keys,
                                                                const int *__restrict__ n_list,
                                                                const dq4 *__restrict__ face64,
                                                                double tx, double ty, double tz,
                                                                int4 *__restrict__ cand, float4 *__restrict__ cimg,
                                                                int *__restrict__ n_out) {
    extern __shared__ unsigned long long sk[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int n_keys = *n_list;
    int n = 32;
    while (n < n_keys) n <<= 1;
    for (int i = tid; i < n; i += FINISH_THREADS) sk[i] = i < n_keys ? keys[i] : KEY_NONE;
    __syncthreads();
    for (int k = 32; k <= n; k <<= 1) {
        for (int j = k >> 1; j >= 32; j >>= 1) {
            for (int i = tid; i < n; i += FINISH_THREADS) {
                const int l = i ^ j;
                if (l > i) {
                    const unsigned long long a = sk[i], b = sk[l];
                    const bool up = (i & k) == 0;
                    if ((a > b) == up) { sk[i] = b; sk[l] = a; }
                }
            }
            __syncthreads();
        }
        for (int i = tid; i < n; i += FINISH_THREADS) {      // (n is a multiple of 32: whole warps)
            unsigned long long a = sk[i];
            for (int kk = (k == 32) ? 2 : k; kk <= k; kk <<= 1) {
                const bool up = (i & kk) == 0;
                for (int j = min(kk >> 1, 16); j > 0; j >>= 1) {
                    const unsigned long long b = __shfl_xor_sync(0xffffffffu, a, j);
                    const bool low = (lane & j) == 0;
                    if ((low == up) ? b < a : b > a) a = b;
                }
            }
            sk[i] = a;
        }
        __syncthreads();
    }
    if (tid == 0) *n_out = n_keys;
    for (int pos = tid; pos < n_keys; pos += FINISH_THREADS) {
        const unsigned long long key = sk[pos];
        const int k = (int)(key >> 60);
        const int f[3] = {(int)((key >> 40) & 0xFFFFFull) - 1, (int)((key >> 20) & 0xFFFFFull) - 1,
                          (int)(key & 0xFFFFFull) - 1};
        cand[pos] = make_int4(f[0], f[1], f[2], k);
        // the source's image after each reflection (FP64, as hi + lo floats)
        double X[3] = {tx, ty, tz};
        for (int m = 0; m < 3; ++m) {
            float4 h = make_float4(0.f, 0.f, 0.f, 0.f), l = h;
            if (m < k) {
                const dq4 F = face64[f[m]];
                const double dist = F.x * X[0] + F.y * X[1] + F.z * X[2] - F.w;
                X[0] = X[0] - F.x * (2.0 * dist);
                X[1] = X[1] - F.y * (2.0 * dist);
                X[2] = X[2] - F.z * (2.0 * dist);
                h = make_float4((float)X[0], (float)X[1], (float)X[2], 0.f);
                l = make_float4((float)(X[0] - (double)h.x), (float)(X[1] - (double)h.y), (float)(X[2] - (double)h.z), 0.f);
            }
            cimg[6 * (size_t)pos + 2 * m] = h;
            cimg[6 * (size_t)pos + 2 * m + 1] = l;
        }
    }
}

}  // namespace

int launch_ray_candidates(const float4 *tri, const float4 *bvh, const int *bvh_tri, const dq4 *face64,
                          const double tx[3], int n_rays, int max_order, const DevCandBufs &B, cudaStream_t st) {
    int n = 32;
    while (n < n_rays * max_order) n <<= 1;
    const size_t smem = sizeof(unsigned long long) * (size_t)n;
    cudaError_t e = cudaFuncSetAttribute(k_cand_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // B.n_cand: the list's length, [1] set if a traversal stack overflowed
    // (the build is far shallower than the stack; reported by
    // rt_get_candidates), [2] the distinct keys so far
    if (e == cudaSuccess) e = cudaMemsetAsync(B.n_cand + 1, 0, 2 * sizeof(int), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(B.table, 0xff, sizeof(unsigned long long) * RT_DEV_CAND_TABLE, st);
    if (e == cudaSuccess) {
        k_ray_launch<<<(n_rays + RAY_WARPS - 1) / RAY_WARPS, 32 * RAY_WARPS, 0, st>>>(
            tri, bvh, bvh_tri, B.fn, B.dir, tx[0], tx[1], tx[2], n_rays, max_order, B.table, B.keys, B.n_cand);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        k_cand_finish<<<1, FINISH_THREADS, smem, st>>>(B.keys, B.n_cand + 2, face64, tx[0], tx[1], tx[2], B.cand, B.cimg,
                                                       B.n_cand);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error(std::string("device ray launch: ") + cudaGetErrorString(e));
        return RT_ERR_CUDA;
    }
    return RT_OK;
}

}  // namespace creep
