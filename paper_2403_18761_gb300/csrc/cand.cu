// A2 by packets: the candidate spheres of every tet.
//
// Sphere i is a candidate of tet t unless some sphere j is strictly closer (in
// power distance) at all four corners; pd(., i) - pd(., j) is affine, so i then
// owns no point of t.  The set does not depend on how it is found.  Here:
//
//  * Tets, vertices and spheres are put in the order of the cells of a bisected
//    box over the mesh (one counting pass for all three), so that consecutive
//    ones are close; 32 consecutive spheres make a leaf, 32 leaves a node, each
//    with the box of its centres and its largest weight.
//  * Over the box of a packet of 8 vertices or tets, a sphere j beats sphere i
//    everywhere when
//      pd(m, i) - pd(m, j) > 2 sum_a |c_i - c_j|_a e_a
//    (m the box's centre, e its half extents: the smallest value of the affine
//    difference over the box).  A leaf is beaten when the bound from its box
//    and largest weight is.  A warp tests 32 nodes, leaves or spheres at once.
//  * k_vertex_owners: a warp per 8 vertices walks the leaves that the sphere
//    near the box's centre does not beat; every vertex gets its owner, the
//    nearest sphere, and whether another one is as near.
//  * k_candidates_packet: a warp per 8 tets, a lane per corner.  A tet with one
//    owner at all corners (and no tie) has no other candidate.  For the others
//    the warp collects the spheres that none of their owners beats over their
//    box; every tet then gathers those that no owner of its corners beats at
//    all four, and applies the exact test among them.
//
// Everything is in exact integers (the box tests on doubled coordinates).
// What bounds it: integer issue and the latency of short dependent steps.
// Packets of 8 rather than 32 have smaller boxes (fewer spheres reach them), four
// times the warps to hide the latency with, and a tet's four corners side by
// side: with 32 tets a warp and a lane per tet the two kernels took 0.10 and
// 0.22 ms on the 205k-tet slab, most of it waiting for a few slow warps, now
// 0.045 and 0.18 (2 M-tet blob: 0.56 and 1.35).  Testing a leaf against the
// packet's corners one by one before its spheres did not pay.  The form before this one kept the k nearest spheres of every mesh vertex,
// one warp per vertex walking box shells of a grid (k_knn_warp), and merged
// four lists per tet with a warp (k_candidates_warp): on the 2 M-tet organic
// blob 2.4 and 1.5 ms, because a shell walk goes on until the largest weight
// of all spheres is out of reach, and k neighbours are far more than the 2 to 8
// candidates of a tet.  rpd_euler_static (which has no room for the orders) and
// the debug bit 4 still use that form.
#include <cuda_runtime.h>
#include <limits.h>

#include <algorithm>

#include "internal.cuh"
#include "prim.cuh"

namespace {

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int WARPS = 4;         // packets per block
constexpr int PACKET = 8;        // vertices or tets of a packet, four lanes each
constexpr int NEAR_CAP = 256;    // spheres collected by a packet (its tets go to the fallback above that)
constexpr int DOM_CAP = 16;      // owners that a packet tests the spheres against
// Up to this many spheres there are two leaves at most: the orders are not
// worth their launches.
constexpr long long ORDER_SPHERES = 64;

// ----------------------------------------------------------------- orders
// Bounds of a shape's vertices: the minima of x, y, z, -x, -y, -z in box[6 s].
__global__ void k_shape_box(CandArgs A, int* __restrict__ box) {
    __shared__ int red[6];
    const CandShape& S = A.shapes ? A.shapes[blockIdx.x] : A.one;
    if (threadIdx.x < 6) red[threadIdx.x] = INT_MAX;
    __syncthreads();
    int m[6] = {INT_MAX, INT_MAX, INT_MAX, INT_MAX, INT_MAX, INT_MAX};
    for (long long v = S.v0 + (long long)blockIdx.y * blockDim.x + threadIdx.x; v < S.v1;
         v += (long long)gridDim.y * blockDim.x) {
        const int3 x = ld_int3(A.Xi, v);
        m[0] = min(m[0], x.x);
        m[1] = min(m[1], x.y);
        m[2] = min(m[2], x.z);
        m[3] = min(m[3], -x.x);
        m[4] = min(m[4], -x.y);
        m[5] = min(m[5], -x.z);
    }
#pragma unroll
    for (int a = 0; a < 6; a++) {
        m[a] = __reduce_min_sync(0xffffffffu, m[a]);
        if ((threadIdx.x & 31) == 0) atomicMin(&red[a], m[a]);
    }
    __syncthreads();
    if (threadIdx.x < 6 && red[threadIdx.x] != INT_MAX) atomicMin(&box[6 * blockIdx.x + threadIdx.x], red[threadIdx.x]);
}

// Last shape whose member `field` is <= i.
template <typename F>
__device__ __forceinline__ int find_shape(const CandArgs& A, F field, long long i) {
    if (!A.shapes) return 0;
    int lo = 0, hi = A.nshapes - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (field(A.shapes[mid]) <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
__device__ __forceinline__ const CandShape& shape_at(const CandArgs& A, int s) { return A.shapes ? A.shapes[s] : A.one; }

// Cell of every tet (by the mean of its corners), vertex and sphere, and its
// place among the cell's items; items are numbered tets, vertices, spheres.
// The cells are the leaves of a number of halvings of the shape's box, each
// across the side that is the longest by then, and numbered by the halves
// taken: consecutive cells are near each other and nearly cubic.
__global__ void k_order_cells(CandArgs A, const int* __restrict__ box, int32_t* __restrict__ count,
                              uint32_t* __restrict__ cell, uint32_t* __restrict__ place) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.nt + A.nv + A.ns) return;
    long long base;
    int bits, sh;
    int3 x = make_int3(0, 0, 0);
    if (i < A.nt) {
        sh = find_shape(A, [](const CandShape& s) { return s.t0; }, i);
        base = shape_at(A, sh).ct;
        bits = shape_at(A, sh).bt;
        const int4 v = *reinterpret_cast<const int4*>(A.T + 4 * i);
        if (v.x >= 0 && v.x < A.nv && v.y >= 0 && v.y < A.nv && v.z >= 0 && v.z < A.nv && v.w >= 0 && v.w < A.nv) {
            const int3 p0 = ld_int3(A.Xi, v.x), p1 = ld_int3(A.Xi, v.y), p2 = ld_int3(A.Xi, v.z), p3 = ld_int3(A.Xi, v.w);
            x = make_int3((p0.x + p1.x + p2.x + p3.x) >> 2, (p0.y + p1.y + p2.y + p3.y) >> 2,
                          (p0.z + p1.z + p2.z + p3.z) >> 2);
        }
    } else if (i < A.nt + A.nv) {
        const long long v = i - A.nt;
        sh = find_shape(A, [](const CandShape& s) { return s.v0; }, v);
        base = shape_at(A, sh).cv;
        bits = shape_at(A, sh).bv;
        x = ld_int3(A.Xi, v);
    } else {
        const long long s = i - A.nt - A.nv;
        sh = find_shape(A, [](const CandShape& q) { return q.s0; }, s);
        base = shape_at(A, sh).cs;
        bits = shape_at(A, sh).bs;
        x = ld_int3(A.Ci, s);
    }
    const int* b = box + 6 * sh;
    // position relative to the current cell, and the cell's sides
    float px = (float)(x.x - b[0]), py = (float)(x.y - b[1]), pz = (float)(x.z - b[2]);
    float ex = (float)(-b[3] - b[0]), ey = (float)(-b[4] - b[1]), ez = (float)(-b[5] - b[2]);
    uint32_t q = 0;
    for (int k = 0; k < bits; k++) {
        q <<= 1;
        if (ex >= ey && ex >= ez) {
            ex *= 0.5f;
            if (px >= ex) {
                px -= ex;
                q |= 1;
            }
        } else if (ey >= ez) {
            ey *= 0.5f;
            if (py >= ey) {
                py -= ey;
                q |= 1;
            }
        } else {
            ez *= 0.5f;
            if (pz >= ez) {
                pz -= ez;
                q |= 1;
            }
        }
    }
    const uint32_t g = (uint32_t)(base + q);
    cell[i] = g;
    place[i] = (uint32_t)atomicAdd(&count[g], 1);
}

// order[] of the three kinds, one after the other (cells are numbered tets
// first, then vertices, then spheres, each kind shape by shape).
__global__ void k_order_fill(CandArgs A, const uint32_t* __restrict__ cell, const uint32_t* __restrict__ place,
                             const int64_t* __restrict__ start, int32_t* __restrict__ order) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.nt + A.nv + A.ns) return;
    const long long at = start[cell[i]] + place[i];
    order[at] = (int32_t)(i < A.nt ? i : (i < A.nt + A.nv ? i - A.nt : i - A.nt - A.nv));
}

// ----------------------------------------------------------------- leaves
// Spheres in order (centre and id, weight), one warp per leaf.
__global__ void k_leaves(CandArgs A, int4* __restrict__ sph, long long* __restrict__ sw, Leaf* __restrict__ leaf,
                         long long* __restrict__ lwmax) {
    const unsigned FULL = 0xffffffffu;
    const long long L = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (L >= A.nleaf) return;   // warp-uniform
    const CandShape& S = shape_at(A, find_shape(A, [](const CandShape& s) { return s.l0; }, L));
    const long long e = S.s0 + 32 * (L - S.l0) + lane;
    int3 lo = make_int3(INT_MAX, INT_MAX, INT_MAX), hi = make_int3(INT_MIN, INT_MIN, INT_MIN);
    long long wm = 0;
    if (e < S.s1) {
        const long long i = A.order_s ? A.order_s[e] : e;
        const int3 c = ld_int3(A.Ci, i);
        lo = hi = c;
        wm = A.W[i];
        sph[e] = make_int4(c.x, c.y, c.z, (int)i);
        sw[e] = wm;
    }
    lo = make_int3(__reduce_min_sync(FULL, lo.x), __reduce_min_sync(FULL, lo.y), __reduce_min_sync(FULL, lo.z));
    hi = make_int3(__reduce_max_sync(FULL, hi.x), __reduce_max_sync(FULL, hi.y), __reduce_max_sync(FULL, hi.z));
    for (int o = 16; o; o >>= 1) wm = max(wm, __shfl_xor_sync(FULL, wm, o));
    if (lane == 0) {
        leaf[L].lo = make_int4(lo.x, lo.y, lo.z, 0);
        leaf[L].hi = make_int4(hi.x, hi.y, hi.z, 0);
        lwmax[L] = wm;
    }
}

// One warp per node: 32 leaves of one shape.
__global__ void k_nodes(CandArgs A, const Leaf* __restrict__ leaf, const long long* __restrict__ lwmax,
                        Leaf* __restrict__ node, long long* __restrict__ nwmax) {
    const unsigned FULL = 0xffffffffu;
    const long long N = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (N >= A.nnode) return;   // warp-uniform
    const CandShape& S = shape_at(A, find_shape(A, [](const CandShape& s) { return s.n0; }, N));
    const long long L = S.l0 + 32 * (N - S.n0) + lane;
    int4 lo = make_int4(INT_MAX, INT_MAX, INT_MAX, 0), hi = make_int4(INT_MIN, INT_MIN, INT_MIN, 0);
    long long wm = 0;
    if (L < S.l0 + (S.s1 - S.s0 + 31) / 32) {
        lo = leaf[L].lo;
        hi = leaf[L].hi;
        wm = lwmax[L];
    }
    lo = make_int4(__reduce_min_sync(FULL, lo.x), __reduce_min_sync(FULL, lo.y), __reduce_min_sync(FULL, lo.z), 0);
    hi = make_int4(__reduce_max_sync(FULL, hi.x), __reduce_max_sync(FULL, hi.y), __reduce_max_sync(FULL, hi.z), 0);
    for (int o = 16; o; o >>= 1) wm = max(wm, __shfl_xor_sync(FULL, wm, o));
    if (lane == 0) {
        node[N].lo = lo;
        node[N].hi = hi;
        nwmax[N] = wm;
    }
}

// ---------------------------------------------------------------- box tests
struct Box {
    int lo[3], hi[3];
};

__device__ __forceinline__ void box_clear(Box& b) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        b.lo[a] = INT_MAX;
        b.hi[a] = INT_MIN;
    }
}
__device__ __forceinline__ void box_add(Box& b, int3 x) {
    b.lo[0] = min(b.lo[0], x.x);
    b.lo[1] = min(b.lo[1], x.y);
    b.lo[2] = min(b.lo[2], x.z);
    b.hi[0] = max(b.hi[0], x.x);
    b.hi[1] = max(b.hi[1], x.y);
    b.hi[2] = max(b.hi[2], x.z);
}
__device__ __forceinline__ void box_warp(Box& b) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        b.lo[a] = __reduce_min_sync(0xffffffffu, b.lo[a]);
        b.hi[a] = __reduce_max_sync(0xffffffffu, b.hi[a]);
    }
}

__device__ __forceinline__ int3 centre(int4 s) { return make_int3(s.x, s.y, s.z); }

// 4 pd(m, sphere) at the box's centre m = (lo + hi) / 2, in integers
// (|lo + hi - 2 c| < 2^23).
__device__ __forceinline__ long long pd4(const Box& b, int4 c, long long w) {
    const long long x = b.lo[0] + b.hi[0] - 2 * c.x, y = b.lo[1] + b.hi[1] - 2 * c.y, z = b.lo[2] + b.hi[2] - 2 * c.z;
    return x * x + y * y + z * z - 4 * w;
}

// Can sphere c (v = 4 pd) be as close as or closer than sphere cj (vj) at some
// point of the box?
__device__ __forceinline__ bool reaches(const Box& b, int4 c, long long v, int4 cj, long long vj) {
    const long long r = (long long)abs(c.x - cj.x) * (b.hi[0] - b.lo[0]) + (long long)abs(c.y - cj.y) * (b.hi[1] - b.lo[1]) +
                        (long long)abs(c.z - cj.z) * (b.hi[2] - b.lo[2]);
    return v - vj <= 4 * r;
}

// Lower bound of 4 pd(m, .) over a leaf or node.
__device__ __forceinline__ long long leaf_pd4(const Box& b, const Leaf& f, long long wmax) {
    const int lo[3] = {f.lo.x, f.lo.y, f.lo.z}, hi[3] = {f.hi.x, f.hi.y, f.hi.z};
    long long d2 = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int m2 = b.lo[a] + b.hi[a];
        const long long d = max(max(2 * lo[a] - m2, m2 - 2 * hi[a]), 0);
        d2 += d * d;
    }
    return d2 - 4 * wmax;
}

// Can a sphere of the leaf (v: its bound) be as close as sphere cj somewhere?
__device__ __forceinline__ bool leaf_reaches(const Box& b, const Leaf& f, long long v, int4 cj, long long vj) {
    const long long r = (long long)max(abs(f.lo.x - cj.x), abs(f.hi.x - cj.x)) * (b.hi[0] - b.lo[0]) +
                        (long long)max(abs(f.lo.y - cj.y), abs(f.hi.y - cj.y)) * (b.hi[1] - b.lo[1]) +
                        (long long)max(abs(f.lo.z - cj.z), abs(f.hi.z - cj.z)) * (b.hi[2] - b.lo[2]);
    return v - vj <= 4 * r;
}

__device__ __forceinline__ void warp_argmin(long long& v, int& i) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov < v || (ov == v && oi < i)) {
            v = ov;
            i = oi;
        }
    }
}

// Lower bound of pd(x, .) over the box's points x and the leaf's spheres.
__device__ __forceinline__ long long leaf_near(const Box& b, const Leaf& f, long long wmax) {
    const long long x = max(max(f.lo.x - b.hi[0], b.lo[0] - f.hi.x), 0), y = max(max(f.lo.y - b.hi[1], b.lo[1] - f.hi.y), 0),
                    z = max(max(f.lo.z - b.hi[2], b.lo[2] - f.hi.z), 0);
    return x * x + y * y + z * z - wmax;
}
// ... and one sphere.
__device__ __forceinline__ long long box_near(const Box& b, int4 c, long long w) {
    const long long x = max(max(c.x - b.hi[0], b.lo[0] - c.x), 0), y = max(max(c.y - b.hi[1], b.lo[1] - c.y), 0),
                    z = max(max(c.z - b.hi[2], b.lo[2] - c.z), 0);
    return x * x + y * y + z * z - w;
}
// ... over the leaf's spheres, at one point.
__device__ __forceinline__ long long leaf_near(int3 p, const Leaf& f, long long wmax) {
    const long long x = max(max(f.lo.x - p.x, p.x - f.hi.x), 0), y = max(max(f.lo.y - p.y, p.y - f.hi.y), 0),
                    z = max(max(f.lo.z - p.z, p.z - f.hi.z), 0);
    return x * x + y * y + z * z - wmax;
}

__device__ __forceinline__ long long warp_max(long long v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The shape's leaves that sphere (cj, vj) does not beat over the box and that
// may hold a sphere with pd <= R somewhere in it (fn may lower R): each with
// fn(leaf, first slot, number of spheres); the whole warp.
template <typename F>
__device__ __forceinline__ void walk(const CandArgs& A, const CandShape& S, const Box& b, int4 cj, long long vj,
                                     const long long& R, F fn) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long nl = (S.s1 - S.s0 + 31) / 32, nn = (nl + 31) / 32;
    auto open = [&](const Leaf& f, long long wmax) {
        return leaf_near(b, f, wmax) <= R && leaf_reaches(b, f, leaf_pd4(b, f, wmax), cj, vj);
    };
    for (long long n0 = 0; n0 < nn; n0 += 32) {
        const bool on = n0 + lane < nn && open(A.node[S.n0 + n0 + lane], A.nwmax[S.n0 + n0 + lane]);
        for (unsigned mn = __ballot_sync(FULL, on); mn; mn &= mn - 1) {
            const long long l0 = 32 * (n0 + __ffs(mn) - 1);
            const bool ol = l0 + lane < nl && open(A.leaf[S.l0 + l0 + lane], A.lwmax[S.l0 + l0 + lane]);
            for (unsigned ml = __ballot_sync(FULL, ol); ml; ml &= ml - 1) {
                const long long l = l0 + __ffs(ml) - 1;
                const long long e0 = S.s0 + 32 * l;
                fn(S.l0 + l, (int)e0, (int)min((long long)32, S.s1 - e0));
            }
        }
    }
}

// ------------------------------------------------------------------ owners
constexpr int TIE = 1 << 30;   // flag of an owner's slot: another sphere is as near

// Four lanes per vertex: each takes every fourth sphere.
__global__ void __launch_bounds__(32 * WARPS) k_vertex_owners(CandArgs A, int32_t* __restrict__ owner) {
    const unsigned FULL = 0xffffffffu;
    __shared__ int list_s[WARPS][32];   // slots of the leaf's spheres that are left
    const int lane = threadIdx.x & 31, sub = lane & 3;
    int* list = list_s[threadIdx.x >> 5];
    const long long pk = (long long)blockIdx.x * WARPS + (threadIdx.x >> 5);
    if (pk >= A.npv) return;   // warp-uniform
    const CandShape S = shape_at(A, find_shape(A, [](const CandShape& s) { return s.pv; }, pk));
    const long long at = S.v0 + PACKET * (pk - S.pv) + (lane >> 2);
    const bool in = at < S.v1;
    const long long v = in ? (A.order_v ? A.order_v[at] : at) : 0;
    int3 x = make_int3(0, 0, 0);
    Box b;
    box_clear(b);
    if (in) {
        x = ld_int3(A.Xi, v);
        box_add(b, x);
    }
    box_warp(b);
    // a sphere near the box's centre: the nearest of the most promising leaf
    // of the most promising node
    const long long nl = (S.s1 - S.s0 + 31) / 32, nn = (nl + 31) / 32;
    long long best = LLONG_MAX;
    int q = INT_MAX;
    for (long long k = lane; k < nn; k += 32) {
        const long long d = leaf_pd4(b, A.node[S.n0 + k], A.nwmax[S.n0 + k]);
        if (d < best) {
            best = d;
            q = (int)k;
        }
    }
    warp_argmin(best, q);
    const long long l0 = 32ll * q;
    best = LLONG_MAX;
    q = INT_MAX;
    if (l0 + lane < nl) {
        best = leaf_pd4(b, A.leaf[S.l0 + l0 + lane], A.lwmax[S.l0 + l0 + lane]);
        q = lane;
    }
    warp_argmin(best, q);
    const long long e0 = S.s0 + 32 * (l0 + q);
    best = LLONG_MAX;
    q = INT_MAX;
    if (e0 + lane < S.s1) {
        best = pd4(b, A.sph[e0 + lane], A.sw[e0 + lane]);
        q = (int)(e0 + lane);
    }
    warp_argmin(best, q);
    const int4 cj = A.sph[q];
    const long long vj = best;
    long long d0 = LLONG_MAX;   // this lane's; dv: the vertex's
    int own = 0;
    auto test = [&](int e) {
        const long long d = pd_exact(x, centre(A.sph[e]), A.sw[e]);
        if (d < d0) {
            d0 = d;
            own = e;
        } else if (d == d0) {
            own |= TIE;
        }
    };
    auto nearest = [&]() {
        const long long d = min(d0, __shfl_xor_sync(FULL, d0, 1));
        return min(d, __shfl_xor_sync(FULL, d, 2));
    };
    // that sphere's leaf whole, for every vertex a first distance
    const int n0 = (int)min(32ll, S.s1 - e0);
    for (int u = sub; u < n0; u += 4) test((int)e0 + u);
    const long long first = S.l0 + (e0 - S.s0) / 32;
    long long dv = nearest();
    long long R = warp_max(in ? dv : LLONG_MIN);
    walk(A, S, b, cj, vj, R, [&](long long l, int e, int n) {
        if (l == first || !__any_sync(FULL, in && leaf_near(x, A.leaf[l], A.lwmax[l]) <= dv)) return;
        bool take = false;
        if (lane < n) take = reaches(b, A.sph[e + lane], pd4(b, A.sph[e + lane], A.sw[e + lane]), cj, vj);
        const unsigned m = __ballot_sync(FULL, take);
        if (!m) return;
        if (take) list[__popc(m & ((1u << lane) - 1u))] = e + lane;
        __syncwarp();
        const int nt = __popc(m);
        for (int u = sub; u < nt; u += 4) test(list[u]);
        dv = nearest();
        R = warp_max(in ? dv : LLONG_MIN);
        __syncwarp();   // the list has been read before the next leaf's is written (shuffles order no memory)
    });
    // the nearest over the four lanes; two lanes as near: a tie
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        const long long d = __shfl_xor_sync(FULL, d0, o);
        const int w = __shfl_xor_sync(FULL, own, o);
        if (d < d0) {
            d0 = d;
            own = w;
        } else if (d == d0 && d != LLONG_MAX) {
            own = min(own & ~TIE, w & ~TIE) | TIE;
        }
    }
    if (in && sub == 0) owner[v] = own;
}

// -------------------------------------------------------------- candidates
// Four lanes per tet, one per corner.
__global__ void __launch_bounds__(32 * WARPS) k_candidates_packet(CandArgs A, const int32_t* __restrict__ owner) {
    const unsigned FULL = 0xffffffffu;
    struct alignas(16) Held {          // a tet's gathered sphere
        long long d[4];                // power distances of the corners
    };
    __shared__ Held held_s[WARPS][RPD_MAXC][PACKET];
    __shared__ int held_id[WARPS][RPD_MAXC][PACKET];
    __shared__ int near_s[WARPS][NEAR_CAP];     // the packet's spheres (slots)
    __shared__ int4 dom_c[WARPS][DOM_CAP];      // owners that the spheres are tested against: centre and slot,
    __shared__ long long dom_v[WARPS][DOM_CAP]; // 4 pd at the box's centre
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, a = lane & 3, g0 = lane & ~3;
    const long long pk = (long long)blockIdx.x * WARPS + warp;
    if (pk >= A.npt) return;   // warp-uniform
    const CandShape S = shape_at(A, find_shape(A, [](const CandShape& s) { return s.pt; }, pk));
    const long long at = S.t0 + PACKET * (pk - S.pt) + g;
    const bool in = at < S.t1;
    const long long t = in ? (A.order_t ? A.order_t[at] : at) : 0;
    // an earlier stage that raised an error, or a vertex id out of range (the
    // mesh check reports it): no candidates
    const int v = in ? A.T[4 * t + a] : -1;
    const bool good = v >= 0 && v < A.nv && *(volatile const int*)&A.st->err == 0;
    bool ok = ((__ballot_sync(FULL, good) >> g0) & 15u) == 15u;   // the same for a tet's four lanes
    if (in && !ok && a == 0) A.cand_cnt[t] = 0;
    int o = ok ? owner[v] : 0;
    {
        const bool same = o == __shfl_sync(FULL, o, g0) && !(o & TIE);
        const unsigned all = __ballot_sync(FULL, same);
        const bool single = ok && ((all >> g0) & 15u) == 15u;   // inside one cell
        if (single && a == 0) {
            A.cand[t * RPD_MAXC] = A.sph[o].w;
            A.cand_ord[t * RPD_MAXC] = 0;
            A.cand_cnt[t] = 1;
        }
        ok = ok && !single;
        o &= ~TIE;
    }
    if (!__any_sync(FULL, ok)) return;
    int3 x = make_int3(0, 0, 0);
    Box b;
    box_clear(b);
    if (ok) {
        x = ld_int3(A.Xi, v);
        box_add(b, x);
    }
    box_warp(b);
    // the distinct owners, up to DOM_CAP of them; the nearest to the centre
    int nd = 0;
    long long vj = LLONG_MAX;
    int4 cj = make_int4(0, 0, 0, 0);
    for (unsigned left = __ballot_sync(FULL, ok); left && nd < DOM_CAP; nd++) {
        const int e = __shfl_sync(FULL, o, __ffs(left) - 1);
        left &= ~__ballot_sync(FULL, o == e);
        const int4 s = A.sph[e];
        const long long ve = pd4(b, s, A.sw[e]);
        if (lane == 0) {
            dom_c[warp][nd] = make_int4(s.x, s.y, s.z, e);
            dom_v[warp][nd] = ve;
        }
        if (ve < vj) {
            vj = ve;
            cj = s;
        }
    }
    // M[z] = pd(X_a, owner of corner z); the owner with the tightest thresholds
    // bounds the walk (a candidate is within them at some corner) and serves
    // the fallback
    long long M[4], thr = 0, best = LLONG_MAX;
    int ref = 0;
#pragma unroll
    for (int z = 0; z < 4; z++) {
        const int e = __shfl_sync(FULL, o, g0 + z);
        M[z] = ok ? pd_exact(x, centre(A.sph[e]), A.sw[e]) : 0;
    }
    const long long mine = a == 0 ? M[0] : (a == 1 ? M[1] : (a == 2 ? M[2] : M[3]));
#pragma unroll
    for (int z = 0; z < 4; z++) {
        long long score = M[z] - mine;
        score = max(score, __shfl_xor_sync(FULL, score, 1));
        score = max(score, __shfl_xor_sync(FULL, score, 2));
        if (score < best) {
            best = score;
            ref = z;
            thr = M[z];
        }
    }
    const long long R = warp_max(ok ? thr : LLONG_MIN);
    __syncwarp();   // the owners' list
    // the spheres that none of the owners beats over the box
    int* near_l = near_s[warp];
    int nn = 0;
    walk(A, S, b, cj, vj, R, [&](long long, int e, int n) {
        int4 s = make_int4(0, 0, 0, 0);
        long long w = 0;
        bool take = lane < n;
        if (take) {   // within the thresholds at some point of the box?
            s = A.sph[e + lane];
            w = A.sw[e + lane];
            take = box_near(b, s, w) <= R;
        }
        if (!__any_sync(FULL, take)) return;
        if (take) {
            const long long vs = pd4(b, s, w);
            for (int k = 0; k < nd && take; k++) take = reaches(b, s, vs, dom_c[warp][k], dom_v[warp][k]);
        }
        const unsigned m = __ballot_sync(FULL, take);
        const int to = nn + __popc(m & ((1u << lane) - 1u));
        if (take && to < NEAR_CAP) near_l[to] = e + lane;
        nn += __popc(m);
    });
    __syncwarp();
    // gather: the spheres that no owner beats at all corners
    int nh = 0;
    if (nn <= NEAR_CAP)
        for (int u = 0; u < nn; u++) {
            const int e = near_l[u];
            const int4 s = A.sph[e];
            const long long d = pd_exact(x, centre(s), A.sw[e]);
            unsigned m4 = (d <= M[0] ? 1u : 0u) | (d <= M[1] ? 2u : 0u) | (d <= M[2] ? 4u : 0u) | (d <= M[3] ? 8u : 0u);
            m4 |= __shfl_xor_sync(FULL, m4, 1);
            m4 |= __shfl_xor_sync(FULL, m4, 2);
            if (ok && m4 == 15u) {
                if (nh < RPD_MAXC) {
                    held_s[warp][nh][g].d[a] = d;
                    if (a == 0) held_id[warp][nh][g] = s.w;
                }
                nh++;
            }
        }
    __syncwarp();
    const bool fallback = nn > NEAR_CAP || nh > A.gather;
    // exact corner filter among the gathered spheres, each lane every fourth
    unsigned keep = 0;
    if (ok && !fallback)
        for (int i = a; i < nh; i += 4) {
            const Held D = held_s[warp][i][g];
            bool stay = true;
            for (int z = 0; z < nh && stay; z++) {
                if (z == i) continue;
                const Held E = held_s[warp][z][g];
                stay = D.d[0] <= E.d[0] || D.d[1] <= E.d[1] || D.d[2] <= E.d[2] || D.d[3] <= E.d[3];
            }
            if (stay) keep |= 1u << i;
        }
    keep |= __shfl_xor_sync(FULL, keep, 1);
    keep |= __shfl_xor_sync(FULL, keep, 2);
    const int oref = __shfl_sync(FULL, o, g0 + ref);
    if (!ok) return;
    if (fallback) {
        if (a == 0) {
            A.fb_list[atomicAdd(A.fb_count, 1)] = (int32_t)t;
            A.cand_cnt[t] = 0;
            A.cand[t * RPD_MAXC] = A.sph[oref].w;
        }
        return;
    }
    // rank by id, and by (sum of corner distances, id)
    for (int i = a; i < nh; i += 4) {
        if (!((keep >> i) & 1u)) continue;
        const Held D = held_s[warp][i][g];
        const long long ki = D.d[0] + D.d[1] + D.d[2] + D.d[3];
        const int id = held_id[warp][i][g];
        int rank = 0, rank2 = 0;
        for (unsigned mz = keep; mz; mz &= mz - 1) {
            const int z = __ffs(mz) - 1;
            const Held E = held_s[warp][z][g];
            const long long kz = E.d[0] + E.d[1] + E.d[2] + E.d[3];
            const int id2 = held_id[warp][z][g];
            rank += id2 < id;
            rank2 += kz < ki || (kz == ki && id2 < id);
        }
        A.cand[t * RPD_MAXC + rank] = id;
        A.cand_ord[t * RPD_MAXC + rank2] = (uint8_t)rank;
    }
    if (a == 0) A.cand_cnt[t] = __popc(keep);
}

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// Halvings of a shape's box for n items: about two cells per item (a shape
// fills a part of its box, so a cell that is not empty holds a few), at most
// 2^20 cells.
int order_bits(long long n) {
    int b = 1;
    while (b < 20 && (1ll << b) < 2 * n) b++;
    return b;
}

}  // namespace

// Host-side plan: every shape's ranges, packets, leaves, nodes and cells.
void cand_plan(const long long* voff, const long long* toff, const long long* soff, int nshapes, long long nv,
               long long nt, long long ns, CandPlan& P) {
    P = CandPlan();
    P.ordered = ns > ORDER_SPHERES;
    P.shapes.resize(nshapes);
    long long cell = 0;
    for (int k = 0; k < nshapes; k++) {
        CandShape& s = P.shapes[k];
        const bool b = nshapes > 1;
        s.v0 = b ? voff[k] : 0;
        s.v1 = b ? voff[k + 1] : nv;
        s.t0 = b ? toff[k] : 0;
        s.t1 = b ? toff[k + 1] : nt;
        s.s0 = b ? soff[k] : 0;
        s.s1 = b ? soff[k + 1] : ns;
        s.pv = P.npv;
        s.pt = P.npt;
        s.l0 = P.nleaf;
        s.n0 = P.nnode;
        const long long nl = (s.s1 - s.s0 + 31) / 32;
        P.npv += (s.v1 - s.v0 + PACKET - 1) / PACKET;
        P.npt += (s.t1 - s.t0 + PACKET - 1) / PACKET;
        P.nleaf += nl;
        P.nnode += (nl + 31) / 32;
        s.bt = order_bits(s.t1 - s.t0);
        s.bv = order_bits(s.v1 - s.v0);
        s.bs = order_bits(s.s1 - s.s0);
    }
    // cells: all tets' first, then the vertices', then the spheres'
    for (CandShape& s : P.shapes) {
        s.ct = cell;
        cell += 1ll << s.bt;
    }
    for (CandShape& s : P.shapes) {
        s.cv = cell;
        cell += 1ll << s.bv;
    }
    for (CandShape& s : P.shapes) {
        s.cs = cell;
        cell += 1ll << s.bs;
    }
    P.ncell = cell;
}

size_t cand_tmp_bytes(const CandPlan& P, long long nt, long long nv, long long ns) {
    const size_t n = (size_t)(nt + nv + ns);
    size_t b = al(sizeof(CandShape) * P.shapes.size()) + al(sizeof(int4) * ns) + al(sizeof(long long) * ns) +
               al(sizeof(Leaf) * P.nleaf) + al(sizeof(long long) * P.nleaf) + al(sizeof(Leaf) * P.nnode) +
               al(sizeof(long long) * P.nnode) + al(sizeof(int32_t) * nv);
    if (!P.ordered) return b;
    return b + al(sizeof(int) * 6 * P.shapes.size()) + al(sizeof(int32_t) * P.ncell) +
           al(sizeof(int64_t) * (P.ncell + 1)) + 3 * al(sizeof(uint32_t) * n) + al(scan_tmp_bytes(P.ncell));
}

void launch_candidates_packet(CandArgs a, const CandPlan& P, const long long* voff, void* tmp, cudaStream_t s) {
    if (a.nt == 0) return;
    char* p = (char*)tmp;
    auto take = [&](size_t bytes) {
        char* q = p;
        p += al(bytes);
        return q;
    };
    const int S = (int)P.shapes.size();
    CandShape* shapes = (CandShape*)take(sizeof(CandShape) * S);
    int4* sph = (int4*)take(sizeof(int4) * a.ns);
    long long* sw = (long long*)take(sizeof(long long) * a.ns);
    Leaf* leaf = (Leaf*)take(sizeof(Leaf) * P.nleaf);
    long long* lwmax = (long long*)take(sizeof(long long) * P.nleaf);
    Leaf* node = (Leaf*)take(sizeof(Leaf) * P.nnode);
    long long* nwmax = (long long*)take(sizeof(long long) * P.nnode);
    int32_t* owner = (int32_t*)take(sizeof(int32_t) * a.nv);
    a.nshapes = S;
    a.one = P.shapes[0];
    a.shapes = nullptr;
    if (S > 1) {
        cudaMemcpyAsync(shapes, P.shapes.data(), sizeof(CandShape) * S, cudaMemcpyHostToDevice, s);
        a.shapes = shapes;
    }
    a.npv = P.npv;
    a.npt = P.npt;
    a.nleaf = P.nleaf;
    a.nnode = P.nnode;
    a.order_t = a.order_v = a.order_s = nullptr;
    cudaMemsetAsync(a.fb_count, 0, sizeof(int32_t), s);
    if (P.ordered) {
        const long long n = a.nt + a.nv + a.ns;
        int* box = (int*)take(sizeof(int) * 6 * S);
        int32_t* count = (int32_t*)take(sizeof(int32_t) * P.ncell);
        int64_t* start = (int64_t*)take(sizeof(int64_t) * (P.ncell + 1));
        uint32_t* cell = (uint32_t*)take(sizeof(uint32_t) * n);
        uint32_t* place = (uint32_t*)take(sizeof(uint32_t) * n);
        int32_t* order = (int32_t*)take(sizeof(uint32_t) * n);
        // box (minima, 0x7f..) and counters (0)
        cudaMemsetAsync(box, 0x7f, sizeof(int) * 6 * S, s);
        cudaMemsetAsync(count, 0, sizeof(int32_t) * P.ncell, s);
        const unsigned parts =
            S > 1 ? (S <= 1024 ? 8u : 1u) : (unsigned)std::min<long long>((a.nv + 1023) / 1024, 304);
        k_shape_box<<<dim3((unsigned)S, parts), 256, 0, s>>>(a, box);
        note_launch();
        k_order_cells<<<nblk(n, 256), 256, 0, s>>>(a, box, count, cell, place);
        note_launch();
        scan_excl(count, start, P.ncell, p, s);
        k_order_fill<<<nblk(n, 256), 256, 0, s>>>(a, cell, place, start, order);
        note_launch();
        a.order_t = order;
        a.order_v = order + a.nt;
        a.order_s = order + a.nt + a.nv;
    }
    k_leaves<<<nblk(32 * P.nleaf, 128), 128, 0, s>>>(a, sph, sw, leaf, lwmax);
    note_launch();
    k_nodes<<<nblk(32 * P.nnode, 128), 128, 0, s>>>(a, leaf, lwmax, node, nwmax);
    note_launch();
    a.sph = sph;
    a.sw = sw;
    a.leaf = leaf;
    a.lwmax = lwmax;
    a.node = node;
    a.nwmax = nwmax;
    k_vertex_owners<<<nblk(P.npv, WARPS), 32 * WARPS, 0, s>>>(a, owner);
    note_launch();
    k_candidates_packet<<<nblk(P.npt, WARPS), 32 * WARPS, 0, s>>>(a, owner);
    note_launch();
    FallbackTree tree;
    tree.shapes = a.shapes;
    tree.one = a.one;
    tree.leaf = leaf;
    tree.lwmax = lwmax;
    tree.sph = sph;
    launch_candidates_fallback(a.T, a.nv, a.Xi, a.Ci, a.W, tree, nullptr, 0, nullptr, nullptr, nullptr, nullptr,
                               a.fb_list, a.fb_count, a.cand_cnt, a.cand, a.cand_ord, a.st, voff, S, s);
}
