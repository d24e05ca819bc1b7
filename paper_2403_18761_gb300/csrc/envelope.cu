// Geometric preservation (Sec. 4.3): distance from surface samples to the
// enveloping volume of the medial mesh.
//
// The medial mesh's primitives (Sec. 3.1, 3.2) are its vertices (spheres
// m_i = (c_i, r_i), one per RPC), its edges (medial cones, the spheres
// interpolated linearly between two vertices, one per RPF) and its triangles
// (medial slabs, interpolated between three, one per RPE).  The signed
// distance of a point s to a primitive is the minimum over its interpolated
// spheres of |s - c| - r; the sample's distance is the minimum over all
// primitives (negative inside the envelope).  Sec. 4.3 inserts a sphere at a
// sample whose distance exceeds delta times the bounding-box diagonal.
//
// |s - c(l)| - r(l) is convex in the interpolation weights l, so its minimum
// over a cone or slab is either at an interior stationary point or on the
// primitive's boundary, which is made of lower primitives (a cone's ends are
// spheres, a slab's edges are cones; every edge of an RPE is an RPF, every
// end of an RPF an RPC).  So each primitive contributes only its interior
// stationary point, found in closed form:
//  * cone (c1, r1) -> (c2, r2), axis u = (c2 - c1) / L, slope k = (r2 - r1) / L,
//    s at axial coordinate x and radial distance y from the axis: the
//    stationary point is at axial coordinate z = x + k y / sqrt(1 - k^2);
//    it counts when 0 < z < L (and |k| < 1);
//  * slab: the unit vector v from c(l) to s satisfies v.(c_j - c_1) = r_1 - r_j
//    (j = 2, 3), i.e. v is the normal of a plane tangent to the three
//    spheres; with v known, c(l) = s - rho v is solved in the plane of the
//    centres; it counts when l lies inside the triangle and rho > 0, and the
//    distance is then v.(s - c_1) - r_1.
//
// FP32 arithmetic on coordinates relative to mesh vertex 0 (the distances
// only decide a threshold); one lane per sample, the samples and the
// primitives in Morton order; a warp culls tiles of 32 primitives, then single
// primitives, by bounding balls (see k_env_dist).
#include <cuda_runtime.h>
#include <math.h>

#include "internal.cuh"
#include "prim.cuh"

namespace {

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int ENV_THREADS = 128;
constexpr int ENV_TILE = 64;    // primitives per tile of the tie order (k_env_dist)
constexpr int ENV_BLOCK = 256;  // samples that share a start of the tie order

// A primitive: up to three spheres (x, y, z, r) and its kind (1, 2, 3).
struct Prim {
    float4 s[3];
    int kind;
};

__device__ __forceinline__ float sphere_d(float3 p, float4 c) {
    const float dx = p.x - c.x, dy = p.y - c.y, dz = p.z - c.z;
    return sqrtf(dx * dx + dy * dy + dz * dz) - c.w;
}

// Interior stationary value of a cone, or +inf.
__device__ __forceinline__ float cone_d(float3 p, float4 a, float4 b) {
    const float ex = b.x - a.x, ey = b.y - a.y, ez = b.z - a.z;
    const float L2 = ex * ex + ey * ey + ez * ez;
    if (!(L2 > 0)) return INFINITY;
    const float L = sqrtf(L2), k = (b.w - a.w) / L;
    if (!(fabsf(k) < 1.0f)) return INFINITY;
    const float ax = p.x - a.x, ay = p.y - a.y, az = p.z - a.z;
    const float x = (ax * ex + ay * ey + az * ez) / L;
    const float y = sqrtf(fmaxf(ax * ax + ay * ay + az * az - x * x, 0.0f));
    const float z = x + k * y / sqrtf(1.0f - k * k);
    if (!(z > 0 && z < L)) return INFINITY;
    const float t = z / L;
    const float4 c = make_float4(a.x + t * ex, a.y + t * ey, a.z + t * ez, a.w + t * (b.w - a.w));
    return sphere_d(p, c);
}

// Interior stationary value of a slab, or +inf.
__device__ __forceinline__ float slab_d(float3 p, float4 c1, float4 c2, float4 c3) {
    const float3 e2 = make_float3(c2.x - c1.x, c2.y - c1.y, c2.z - c1.z);
    const float3 e3 = make_float3(c3.x - c1.x, c3.y - c1.y, c3.z - c1.z);
    const float g22 = e2.x * e2.x + e2.y * e2.y + e2.z * e2.z, g23 = e2.x * e3.x + e2.y * e3.y + e2.z * e3.z;
    const float g33 = e3.x * e3.x + e3.y * e3.y + e3.z * e3.z;
    const float det = g22 * g33 - g23 * g23;
    if (!(det > 1e-20f * g22 * g33)) return INFINITY;
    // in-plane part w = al e2 + be e3 of v: w.e2 = r1 - r2, w.e3 = r1 - r3
    const float b2 = c1.w - c2.w, b3 = c1.w - c3.w;
    const float al = (b2 * g33 - b3 * g23) / det, be = (b3 * g22 - b2 * g23) / det;
    const float3 w = make_float3(al * e2.x + be * e3.x, al * e2.y + be * e3.y, al * e2.z + be * e3.z);
    const float ww = w.x * w.x + w.y * w.y + w.z * w.z;
    if (!(ww < 1.0f)) return INFINITY;
    float3 n = make_float3(e2.y * e3.z - e2.z * e3.y, e2.z * e3.x - e2.x * e3.z, e2.x * e3.y - e2.y * e3.x);
    const float nn = sqrtf(n.x * n.x + n.y * n.y + n.z * n.z);
    n = make_float3(n.x / nn, n.y / nn, n.z / nn);
    const float3 a = make_float3(p.x - c1.x, p.y - c1.y, p.z - c1.z);
    const float h = a.x * n.x + a.y * n.y + a.z * n.z;
    const float gm = copysignf(sqrtf(1.0f - ww), h);
    const float3 v = make_float3(w.x + gm * n.x, w.y + gm * n.y, w.z + gm * n.z);
    // c1 + l2 e2 + l3 e3 + rho v = s: rho from the normal component, then the
    // in-plane weights from the 2x2 Gram system
    const float vn = v.x * n.x + v.y * n.y + v.z * n.z;
    if (!(fabsf(vn) > 0)) return INFINITY;
    const float rho = h / vn;
    if (!(rho > 0)) return INFINITY;
    const float3 q = make_float3(a.x - rho * v.x, a.y - rho * v.y, a.z - rho * v.z);
    const float q2 = q.x * e2.x + q.y * e2.y + q.z * e2.z, q3 = q.x * e3.x + q.y * e3.y + q.z * e3.z;
    const float l2 = (q2 * g33 - q3 * g23) / det, l3 = (q3 * g22 - q2 * g23) / det;
    if (!(l2 > 0 && l3 > 0 && l2 + l3 < 1)) return INFINITY;
    return a.x * v.x + a.y * v.y + a.z * v.z - c1.w;
}

__device__ __forceinline__ float prim_d(float3 p, const Prim& q) {
    if (q.kind == 1) return sphere_d(p, q.s[0]);
    if (q.kind == 2) return cone_d(p, q.s[0], q.s[1]);
    return slab_d(p, q.s[0], q.s[1], q.s[2]);
}

// Primitive table: kinds 1..3 from the element keys, sphere data relative to
// the centre `o` (grid units x unit, in FP32).
__global__ void k_env_prims(const int32_t* __restrict__ k1, long long n1, const int32_t* __restrict__ k2, long long n2,
                            const int32_t* __restrict__ k3, long long n3, const int32_t* __restrict__ Ci,
                            const long long* __restrict__ W, double unit, double3 o, Prim* __restrict__ out,
                            uint64_t* __restrict__ morton, uint32_t* __restrict__ idx, int3 gmin, int shift) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n1 + n2 + n3) return;
    Prim q;
    const int32_t* key;
    int kind;
    if (i < n1) {
        kind = 1;
        key = k1 + i;
    } else if (i < n1 + n2) {
        kind = 2;
        key = k2 + 2 * (i - n1);
    } else {
        kind = 3;
        key = k3 + 3 * (i - n1 - n2);
    }
    q.kind = kind;
    long long cx = 0, cy = 0, cz = 0;
    for (int z = 0; z < 3; z++) {
        const int s = key[z < kind ? z : 0];
        const int3 c = ld_int3(Ci, s);
        q.s[z] = make_float4((float)(c.x * unit - o.x), (float)(c.y * unit - o.y), (float)(c.z * unit - o.z),
                             (float)(sqrt((double)W[s]) * unit));
        if (z < kind) {
            cx += c.x;
            cy += c.y;
            cz += c.z;
        }
    }
    out[i] = q;
    // Morton code of the primitive's mean centre (21 bits per axis)
    auto spread = [](unsigned long long v) {
        v &= 0x1fffffull;
        v = (v | v << 32) & 0x1f00000000ffffull;
        v = (v | v << 16) & 0x1f0000ff0000ffull;
        v = (v | v << 8) & 0x100f00f00f00f00full;
        v = (v | v << 4) & 0x10c30c30c30c30c3ull;
        v = (v | v << 2) & 0x1249249249249249ull;
        return v;
    };
    const unsigned long long ux = (unsigned long long)((cx / kind - gmin.x) >> shift);
    const unsigned long long uy = (unsigned long long)((cy / kind - gmin.y) >> shift);
    const unsigned long long uz = (unsigned long long)((cz / kind - gmin.z) >> shift);
    morton[i] = spread(ux) | (spread(uy) << 1) | (spread(uz) << 2);
    idx[i] = (uint32_t)i;
}

// Morton code of a sample (world coordinates), in the primitives' code space.
__device__ __forceinline__ unsigned long long spread21(unsigned long long v) {
    v &= 0x1fffffull;
    v = (v | v << 32) & 0x1f00000000ffffull;
    v = (v | v << 16) & 0x1f0000ff0000ffull;
    v = (v | v << 8) & 0x100f00f00f00f00full;
    v = (v | v << 4) & 0x10c30c30c30c30c3ull;
    v = (v | v << 2) & 0x1249249249249249ull;
    return v;
}

__global__ void k_env_sample_keys(const double* __restrict__ samples, long long ns, double scale, int3 gmin, int shift,
                                  uint64_t* __restrict__ morton, uint32_t* __restrict__ idx) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns) return;
    unsigned long long u[3];
    const int gm[3] = {gmin.x, gmin.y, gmin.z};
    for (int a = 0; a < 3; a++) {
        double g = rint(samples[3 * i + a] * scale);
        g = fmin(fmax(g, (double)gm[a]), (double)(-gm[a] - 1));   // inside the code's range
        u[a] = (unsigned long long)(((long long)g - gm[a]) >> shift);
    }
    morton[i] = spread21(u[0]) | (spread21(u[1]) << 1) | (spread21(u[2]) << 2);
    idx[i] = (uint32_t)i;
}

// Primitives in Morton order, each with a bounding ball of its spheres (every
// point of its envelope is within the radius of the centre), and the bounding
// ball of each 32 of them (one warp).
__global__ void k_env_gather(const Prim* __restrict__ in, const uint32_t* __restrict__ order, long long n,
                             Prim* __restrict__ out, float4* __restrict__ balls, float4* __restrict__ tiles) {
    const unsigned FULL = 0xffffffffu;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if ((i & ~31ll) >= n) return;   // warp-uniform
    float4 b = make_float4(0, 0, 0, -INFINITY);
    if (i < n) {
        const Prim q = in[order[i]];
        out[i] = q;
        for (int z = 0; z < q.kind; z++) {
            b.x += q.s[z].x;
            b.y += q.s[z].y;
            b.z += q.s[z].z;
        }
        const float w = 1.0f / (float)q.kind;
        b.x *= w;
        b.y *= w;
        b.z *= w;
        for (int z = 0; z < q.kind; z++) {
            const float dx = q.s[z].x - b.x, dy = q.s[z].y - b.y, dz = q.s[z].z - b.z;
            b.w = fmaxf(b.w, sqrtf(dx * dx + dy * dy + dz * dz) + q.s[z].w);
        }
        b.w *= 1.0f + 0x1p-18f;
        balls[i] = b;
    }
    const int m = (int)(n - (i & ~31ll) < 32 ? n - (i & ~31ll) : 32);
    float sx = b.x, sy = b.y, sz = b.z;
    for (int off = 16; off; off >>= 1) {
        sx += __shfl_xor_sync(FULL, sx, off);
        sy += __shfl_xor_sync(FULL, sy, off);
        sz += __shfl_xor_sync(FULL, sz, off);
    }
    const float cx = sx / (float)m, cy = sy / (float)m, cz = sz / (float)m;
    const float dx = b.x - cx, dy = b.y - cy, dz = b.z - cz;
    float r = sqrtf(dx * dx + dy * dy + dz * dz) + b.w;   // -inf past the end
    for (int off = 16; off; off >>= 1) r = fmaxf(r, __shfl_xor_sync(FULL, r, off));
    if ((i & 31) == 0) tiles[i >> 5] = make_float4(cx, cy, cz, r * (1.0f + 0x1p-18f));
}

// First position whose key is >= key (n if there is none); the whole warp,
// 32 probes a step.
__device__ __forceinline__ long long warp_lower_bound(const uint64_t* __restrict__ keys, long long n, uint64_t key) {
    const int lane = threadIdx.x & 31;
    long long lo = 0, hi = n;   // the answer is in [lo, hi]
    while (lo < hi) {
        const long long pos = lo + (hi - lo) * lane / 32;   // < hi, ascending over the lanes
        const int below = __popc(__ballot_sync(0xffffffffu, keys[pos] < key));
        const long long at = __shfl_sync(0xffffffffu, pos, below > 0 ? below - 1 : 0);
        const long long up = __shfl_sync(0xffffffffu, pos, below < 32 ? below : 31);
        if (below < 32) hi = up;
        if (below > 0) lo = at + 1;
    }
    return lo;
}

// Order of floats as unsigned integers (no NaN).
__device__ __forceinline__ unsigned float_key(float f) {
    const unsigned u = __float_as_uint(f);
    return u ^ ((unsigned)((int)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? k ^ 0x80000000u : ~k);
}

// One block per 32 samples in Morton order: a lane is a sample in each of the
// block's warps, and the warps share out the tiles of 32 primitives.  Tiles
// are tested 32 at a time (one per lane) against the box of the samples and
// the largest of their best distances, R, then against each sample's own best
// distance; the primitives of an open tile likewise, and each that is left is
// evaluated by all lanes.  Groups of 32 tiles are taken outwards from the
// block's own place in the Morton order, so the distances fall early; the warps
// share them through shared memory.
//
// What bounds it: latency and issue on the primitives that a ball cannot
// reject (those whose envelope nearly touches a sample); the samples alone are
// too few warps to hide it, hence several per packet.  Culling by blocks of
// 256 samples and tiles of 64 primitives, with three block barriers per tile,
// evaluated every primitive of a tile for all 256: 5.8 ms for 58 k samples
// and 45 k primitives.
//
// Equal distances go to the primitive that comes first in an order fixed by
// the sample's place: tiles of 64 outwards (t0, t0 + 1, t0 - 1, ...) from t0, the
// tile where the codes reach that of the first of the sample's 256.
// Distance from a sample to a ball, from below (slack: the margin).
__device__ __forceinline__ float sample_gap(float3 p, float slack, float4 b) {
    const float dx = p.x - b.x, dy = p.y - b.y, dz = p.z - b.z;
    return sqrtf(dx * dx + dy * dy + dz * dz) * (1.0f - 0x1p-18f) - b.w - slack;
}

// Nearest of the (up to 32) primitives from e0 on to one sample, a primitive
// per lane: its distance and its place, the first of equals (INFINITY, 0 when
// none is nearer than the ball tests' limit).  A call, so that it takes none of
// the main loop's registers.
__device__ __noinline__ float2 one_sample(const Prim* __restrict__ prims, const float4* __restrict__ balls, long long np,
                                          long long e0, float3 p, float slack, float limit) {
    const unsigned FULL = 0xffffffffu;
    const long long k = e0 + (threadIdx.x & 31);
    float d = INFINITY;
    if (k < np && !(sample_gap(p, slack, balls[k]) > limit)) d = prim_d(p, prims[k]);
    if (!(d < INFINITY)) d = INFINITY;   // NaN: not taken
    const float least = key_float(__reduce_min_sync(FULL, float_key(d + 0.0f)));   // -0 as 0
    const int b = __ffs(__ballot_sync(FULL, d == least)) - 1;
    return make_float2(__shfl_sync(FULL, d, b), __int_as_float(b));
}

__global__ void __launch_bounds__(ENV_THREADS) k_env_dist(const double* __restrict__ samples, long long ns, double3 o,
                                                          const Prim* __restrict__ prims, long long np,
                                                          const float4* __restrict__ balls,
                                                          const float4* __restrict__ tiles,
                                                          const uint64_t* __restrict__ pkeys,
                                                          const uint32_t* __restrict__ porder,
                                                          const uint64_t* __restrict__ skeys,
                                                          const uint32_t* __restrict__ sorder, float* __restrict__ dist,
                                                          int32_t* __restrict__ arg) {
    const unsigned FULL = 0xffffffffu;
    constexpr int NW = ENV_THREADS / 32;
    __shared__ unsigned sbest[32];        // the samples' best distances so far (float_key)
    __shared__ float fd[NW][32];          // the warps' results
    __shared__ long long fr[NW][32];
    __shared__ int fi[NW][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long q0 = 32ll * blockIdx.x;
    const bool in = q0 + lane < ns;
    const long long i = (long long)sorder[in ? q0 + lane : q0];
    float3 p = make_float3((float)(samples[3 * i] - o.x), (float)(samples[3 * i + 1] - o.y),
                           (float)(samples[3 * i + 2] - o.z));
    // a sample whose squared distances are not finite has no nearest primitive
    // (INFINITY, -1), and must not open the tiles for the others of its packet
    const bool live = in && isfinite(p.x * p.x + p.y * p.y + p.z * p.z);
    if (!live) p = make_float3(0, 0, 0);
    if (warp == 0) sbest[lane] = float_key(INFINITY);
    float lo[3] = {p.x, p.y, p.z}, hi[3] = {p.x, p.y, p.z};
    const bool some = __any_sync(FULL, live);
    if (!live && some) {
        for (int a = 0; a < 3; a++) {
            lo[a] = INFINITY;
            hi[a] = -INFINITY;
        }
    }
    for (int a = 0; a < 3; a++)
        for (int off = 16; off; off >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(FULL, lo[a], off));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(FULL, hi[a], off));
        }
    // margin of the ball tests, far above their FP32 rounding
    float slack = 0.0f;
    for (int a = 0; a < 3; a++) slack = fmaxf(slack, fmaxf(fabsf(lo[a]), fabsf(hi[a])));
    slack *= 0x1p-18f;
    // distance from the samples' box, or from this sample, to a ball, from below
    auto gap = [&](float4 b) {
        const float dx = fmaxf(fmaxf(lo[0] - b.x, b.x - hi[0]), 0.0f), dy = fmaxf(fmaxf(lo[1] - b.y, b.y - hi[1]), 0.0f),
                    dz = fmaxf(fmaxf(lo[2] - b.z, b.z - hi[2]), 0.0f);
        return sqrtf(dx * dx + dy * dy + dz * dz) * (1.0f - 0x1p-18f) - b.w - slack;
    };
    // (a margin of the sample's own: a far one must not widen the others')
    const float own_slack = 0x1p-18f * fmaxf(fabsf(p.x), fmaxf(fabsf(p.y), fabsf(p.z)));
    const long long ntile64 = (np + ENV_TILE - 1) / ENV_TILE;
    const long long l0 = warp_lower_bound(pkeys, np, skeys[q0 / ENV_BLOCK * ENV_BLOCK]);
    const long long t0 = l0 < np ? l0 / ENV_TILE : ntile64 - 1;
    float best = INFINITY;   // this warp's
    long long brank = 0;
    int bi = -1;
    float bound = INFINITY, R = INFINITY;   // best of all the warps', and its largest over the samples
    auto refresh = [&]() {
        __syncwarp();
        bound = key_float(*(volatile unsigned*)&sbest[lane]);
        R = live ? bound : -INFINITY;
        for (int off = 16; off; off >>= 1) R = fmaxf(R, __shfl_xor_sync(FULL, R, off));
    };
    auto needs = [&](float4 b) { return __ballot_sync(FULL, live && !(sample_gap(p, own_slack, b) > fminf(bound, best))); };
    auto tile = [&](long long t, unsigned who) {   // the 32 primitives of tile t, for the samples `who`
        const long long k = 32 * t + lane;
        const long long t64 = t >> 1, j = t64 > t0 ? 2 * (t64 - t0) - 1 : 2 * (t0 - t64);
        const long long rank0 = j * ENV_TILE + 32 * (t & 1);
        auto take = [&](float d, int b) {
            const long long rank = rank0 + b;
            if (live && (d < best || (d == best && rank < brank))) {
                best = d;
                bi = (int)(32 * t + b);
                brank = rank;
            }
        };
        // few samples (one far from the shape needs every tile: its margin is wider
        // than the differences between the primitives' distances; the warp's
        // lanes, not its samples, then share them out: such a sample made
        // 24.7 k others take 6.8 ms instead of 1.35)
        if (__popc(who) <= 2) {
            for (; who; who &= who - 1) {
                const int z = __ffs(who) - 1;
                const float3 x = make_float3(__shfl_sync(FULL, p.x, z), __shfl_sync(FULL, p.y, z), __shfl_sync(FULL, p.z, z));
                const float2 r = one_sample(prims, balls, np, 32 * t, x, __shfl_sync(FULL, own_slack, z),
                                            __shfl_sync(FULL, fminf(bound, best), z));
                if (lane == z) take(r.x, __float_as_int(r.y));
            }
            who = 0;
        }
        unsigned open = who ? __ballot_sync(FULL, k < np && !(gap(balls[k < np ? k : np - 1]) > R)) : 0;
        for (; open; open &= open - 1) {
            const int b = __ffs(open) - 1;
            if (needs(balls[32 * t + b])) take(prim_d(p, prims[32 * t + b]), b);
        }
        if (best < bound) atomicMin(&sbest[lane], float_key(best));
        refresh();
    };
    const long long ntile = (np + 31) / 32, ngroup = (ntile + 31) / 32;
    long long start = warp_lower_bound(pkeys, np, skeys[q0]) / 32;
    if (start >= ntile) start = ntile - 1;
    __syncthreads();   // sbest
    // the tiles around the samples first, one per warp
    const long long s0 = start - NW / 2 + warp;
    if (s0 >= 0 && s0 < ntile) tile(s0, FULL);
    __syncthreads();
    refresh();
    const long long g0 = start / 32;
    for (long long jg = 0; jg < 2 * ngroup; jg++) {
        const long long g = (jg & 1) ? g0 + (jg + 1) / 2 : g0 - jg / 2;
        if (g < 0 || g >= ngroup) continue;
        const long long t = 32 * g + lane;
        const float gp = t < ntile ? gap(tiles[t]) : INFINITY;
        // this warp's tiles of the group: every NW-th
        for (unsigned open = __ballot_sync(FULL, t < ntile && !(gp > R) && (lane & (NW - 1)) == warp); open;
             open &= open - 1) {
            const int b = __ffs(open) - 1;
            if (__shfl_sync(FULL, gp, b) > R) continue;   // R has fallen since
            const unsigned who = needs(tiles[32 * g + b]);
            if (who) tile(32 * g + b, who);
        }
    }
    fd[warp][lane] = best;
    fr[warp][lane] = brank;
    fi[warp][lane] = bi;
    __syncthreads();
    if (warp == 0 && in) {
        for (int w = 1; w < NW; w++)
            if (fi[w][lane] >= 0 &&
                (bi < 0 || fd[w][lane] < best || (fd[w][lane] == best && fr[w][lane] < brank))) {
                best = fd[w][lane];
                brank = fr[w][lane];
                bi = fi[w][lane];
            }
        dist[i] = best;
        arg[i] = bi < 0 ? -1 : (int32_t)porder[bi];   // sorted position -> table row
    }
}

}  // namespace

size_t envelope_tmp_bytes(long long np, long long nsamp) {
    const size_t a = ((size_t)np * sizeof(Prim) + 255) & ~(size_t)255;
    const size_t t = (((size_t)(np + 31) / 32 + 1) * sizeof(float4) + 255) & ~(size_t)255;
    const size_t bl = ((size_t)np * sizeof(float4) + 255) & ~(size_t)255;
    const size_t k = ((size_t)(np + 1) * 8 + 255) & ~(size_t)255, v = ((size_t)(np + 1) * 4 + 255) & ~(size_t)255;
    const size_t ks = ((size_t)(nsamp + 1) * 8 + 255) & ~(size_t)255, vs = ((size_t)(nsamp + 1) * 4 + 255) & ~(size_t)255;
    return 2 * a + t + bl + 2 * k + 2 * v + 2 * ks + 2 * vs + radix_tmp_bytes(np > nsamp ? np : nsamp);
}

// Primitive table sorted by the Morton code of the primitive's mean centre,
// its tile bounds, then the distance of every sample (FP32, relative to o).
// prim_id: index into the unsorted table (spheres, then cones, then slabs).
void launch_envelope(const int32_t* k1, long long n1, const int32_t* k2, long long n2, const int32_t* k3, long long n3,
                     const int32_t* Ci, const long long* W, double unit, const double* o3, const double* samples,
                     long long nsamp, float* dist, int32_t* prim_id, void* tmp, int* d_err, cudaStream_t s) {
    const long long np = n1 + n2 + n3;
    if (np <= 0 || nsamp <= 0) return;
    const size_t a = ((size_t)np * sizeof(Prim) + 255) & ~(size_t)255;
    const size_t t = (((size_t)(np + 31) / 32 + 1) * sizeof(float4) + 255) & ~(size_t)255;
    const size_t bl = ((size_t)np * sizeof(float4) + 255) & ~(size_t)255;
    const size_t k = ((size_t)(np + 1) * 8 + 255) & ~(size_t)255, v = ((size_t)(np + 1) * 4 + 255) & ~(size_t)255;
    char* p = (char*)tmp;
    Prim* raw = (Prim*)p;
    p += a;
    Prim* sorted = (Prim*)p;
    p += a;
    float4* tiles = (float4*)p;
    p += t;
    float4* balls = (float4*)p;
    p += bl;
    uint64_t* m0 = (uint64_t*)p;
    p += k;
    uint64_t* m1 = (uint64_t*)p;
    p += k;
    uint32_t* i0 = (uint32_t*)p;
    p += v;
    uint32_t* i1 = (uint32_t*)p;
    p += v;
    const size_t ks = ((size_t)(nsamp + 1) * 8 + 255) & ~(size_t)255, vs = ((size_t)(nsamp + 1) * 4 + 255) & ~(size_t)255;
    uint64_t* sk0 = (uint64_t*)p;
    p += ks;
    uint64_t* sk1 = (uint64_t*)p;
    p += ks;
    uint32_t* so0 = (uint32_t*)p;
    p += vs;
    uint32_t* so1 = (uint32_t*)p;
    p += vs;
    const double3 o = make_double3(o3[0], o3[1], o3[2]);
    // grid coordinates are in (-2^21, 2^21): shifted by 2^21 and halved they fit 21 bits
    const int g0 = -(1 << 21);
    k_env_prims<<<nblk(np, 256), 256, 0, s>>>(k1, n1, k2, n2, k3, n3, Ci, W, unit, o, raw, m0, i0,
                                               make_int3(g0, g0, g0), 1);
    note_launch();
    radix_sort_pairs(m0, i0, m1, i1, np, 63, p, d_err, s);
    k_env_gather<<<nblk(np, 256), 256, 0, s>>>(raw, i1, np, sorted, balls, tiles);
    note_launch();
    k_env_sample_keys<<<nblk(nsamp, 256), 256, 0, s>>>(samples, nsamp, 1.0 / unit, make_int3(g0, g0, g0), 1, sk0, so0);
    note_launch();
    radix_sort_pairs(sk0, so0, sk1, so1, nsamp, 63, p, d_err, s);
    k_env_dist<<<nblk(nsamp, 32), ENV_THREADS, 0, s>>>(samples, nsamp, o, sorted, np, balls, tiles, m1, i1,
                                                                sk1, so1, dist, prim_id);
    note_launch();
}
