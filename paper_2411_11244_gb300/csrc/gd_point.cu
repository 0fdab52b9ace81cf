// Point-to-mesh distance (the 1-to-N direction the paper names as future
// work in Section 10, with points as the N queries): for each query point,
// the closest point of a mesh placed by a rigid transform, exact in float64.
//
// One warp per point walks the mesh's f12-BVH: a step takes up to four nodes
// off the warp's stack and tests their eight descendants three levels down,
// one per lane, so the nodes of one point are tested side by side and a point
// that many triangles surround at nearly one distance (the centre of a ring)
// takes 1/32 of the steps that a thread would need.  Float64 stays off the
// walk: boxes and triangles give rigorous float32 bounds (coordinates taken
// relative to the point, held in two floats), and only triangles whose lower
// bound does not exceed the least upper bound are listed for float64.  A warp
// collects the lists of the points it answers and evaluates them 32 at a time,
// one per lane; the least (d, original index) pair of each point wins.
// Pruning only ever drops triangles that are provably farther than a true
// distance, so the answer is the exact minimum over all triangles, the
// smallest original index among ties.
//
// What bounds it: issue slots and L1/L2 latency of the box tests (3,200 a point
// around a ring on average, most of them near-ties), not the bytes of the points.
// A thread per point, with float64 in the walk, left one lane of a warp
// working at a time: 262,144 device points against a 7.5 M-triangle ring took
// 258 ms, 1,000 host points against a 204,800-triangle gear 9.4 ms; one warp
// per point alone 13.6 ms (18.8 for another draw of the points, in which one
// walk of 500 K tests, with its neighbours, ran for half of that) and 0.29 ms;
// with long walks divided among idle warps 9.8 and 0.15 ms.  20, 24 and 28 warps
// an SM took 11.5, 10.9 and 10.4 ms at one stage of this, 32 (with 64 registers)
// 12.0.
#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "gd_geom.cuh"
#include "gd_internal.cuh"
#include "gd_launch.h"

namespace gd {

namespace {

constexpr int kPointWarps = 2;
constexpr int kPointThreads = 32 * kPointWarps;
constexpr int kPointCtas = 14;  // CTAs per SM the kernel is compiled for: 28 warps, 72 registers a thread
// The stack of a walk.  A step pushes at most 32 entries, each at least three
// levels below the shallowest entry it took; entries of a later step lie above
// those of an earlier one and are taken first, so the pushes alive at one time
// have depths three apart: with the start, at most 1 + 30 / 3 of them.
constexpr int kStack = 384;
constexpr int kTriWait = 96;   // < 32 waiting triangles before a step, at most 64 more after it
constexpr int kNearWait = 64;  // < 32 before a pass, at most 32 more after it
constexpr int kList = 96;      // <= 32 of finished points, <= 32 of this one, 32 more in a pass

// Walks differ by a factor of a thousand (a point that much of the mesh
// surrounds at nearly one distance), so a long walk gives half of its stack
// to a warp that has run out of points.
constexpr unsigned kShareMin = 16;  // least stack worth dividing
constexpr unsigned kChunk = 4;      // most points a warp takes at a time

struct PointWarp {
    unsigned node[kStack];      // the stack: node,
    unsigned short gap[kStack]; //   and its squared gap, rounded down to 16 bits
    unsigned tri[kTriWait];     // triangles whose leaf passed
    unsigned near[kNearWait];   // ... and that a plane through their centroid does not keep away
    unsigned cj[kList];         // candidates for float64: triangle,
    unsigned ci[kList];         //   point,
    float clow[kList];          //   lower bound (squared)
    float c[kChunk][6];         // the chunk's points: local coordinates, two floats each
    unsigned pi[kChunk];        //   and their indices (kNone: not finite)
};

constexpr unsigned kNone = 0xffffffffu;

__device__ __forceinline__ unsigned leaf_begin(long long T, int L, unsigned leaf) {
    return (unsigned)(((unsigned long long)leaf * (unsigned long long)T) >> L);
}

__device__ __forceinline__ void load_tri(const float4* tri, unsigned j, V3<float>* v, int* id) {
    const float4 p = __ldg(tri + 3ull * j), q = __ldg(tri + 3ull * j + 1), r = __ldg(tri + 3ull * j + 2);
    v[0] = mk3(p.x, p.y, p.z);
    v[1] = mk3(p.w, q.x, q.y);
    v[2] = mk3(q.z, q.w, r.x);
    *id = __float_as_int(r.y);
}

struct NodeBox {
    float lo[3], hi[3];
};

__device__ __forceinline__ NodeBox load_node(const float* box, unsigned node) {
    const float2* b = reinterpret_cast<const float2*>(box + 6ull * node);
    const float2 x = __ldg(b), y = __ldg(b + 1), z = __ldg(b + 2);
    return NodeBox{{x.x, x.y, y.x}, {y.y, z.x, z.y}};
}

// Squared distance from the box [cm, cp] (the point +- its float32 rounding)
// to the node's box; every float32 step rounds at most one unit, so the caller
// compares it against its bound grown by 2^-20 relative.
__device__ __forceinline__ float node_gap_sq(const NodeBox& b, V3<float> cm, V3<float> cp) {
    const float gx = fmaxf(0.f, fmaxf(b.lo[0] - cp.x, cm.x - b.hi[0]));
    const float gy = fmaxf(0.f, fmaxf(b.lo[1] - cp.y, cm.y - b.hi[1]));
    const float gz = fmaxf(0.f, fmaxf(b.lo[2] - cp.z, cm.z - b.hi[2]));
    return fmaf(gz, gz, fmaf(gy, gy, gx * gx));
}

// A rigorous upper bound of the squared distance from any point within E (per
// coordinate) of c to the mesh: the node's box is tight, so each of its faces
// holds a vertex, which is no farther than the face's farthest point.
__device__ __forceinline__ float node_upper_sq(const NodeBox& b, V3<float> c, float E) {
    const float cc[3] = {c.x, c.y, c.z};
    float n2[3], f2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float x = fabsf(b.lo[k] - cc[k]), y = fabsf(cc[k] - b.hi[k]);
        const float n = fminf(x, y) + E, f = fmaxf(x, y) + E;
        n2[k] = n * n;
        f2[k] = f * f;
    }
    const float u = fminf(n2[0] + f2[1] + f2[2], fminf(f2[0] + n2[1] + f2[2], f2[0] + f2[1] + n2[2]));
    return u * (1.f + 0x1p-20f);
}

__device__ __forceinline__ float abs_max(V3<float> a) { return fmaxf(fabsf(a.x), fmaxf(fabsf(a.y), fabsf(a.z))); }

// Rigorous float32 bounds of the squared distance from a point to a triangle
// whose vertices relative to the point are w, each coordinate off by at most
// 2.01 u X + e (u = 2^-24, X the largest coordinate, e for the point's own
// two-float form).  q, the float32 closest point, has weights clamped to the
// triangle, so it lies within 10 u X per coordinate (its products, sums and
// edge differences) of a point of the triangle with those weights: with the
// vertices' error less than 16 u X + e, and |q| grown by that bounds the
// distance from above.  The separation of the origin from the triangle along
// q bounds it from below (any axis does; this one is nearly the exact
// direction): each dot product is taken down by 4 u of its absolute terms,
// for its own rounding, and by 4 u X + e per unit of |q|_1, for the vertices'.
__device__ __forceinline__ void tri_bounds_sq(const V3<float>* w, float e, float* lower, float* upper) {
    bool inside;
    const V3<float> q = closest_on_triangle<float>(mk3(0.f, 0.f, 0.f), w[0], w[1], w[2], &inside);
    const float X = fmaxf(abs_max(w[0]), fmaxf(abs_max(w[1]), abs_max(w[2])));
    const float qq = dot(q, q);
    const float slack = __fmul_ru(1.7320509f, __fmaf_ru(X, 0x1p-20f, e));
    const float up = __fmaf_ru(__fsqrt_ru(qq), 1.f + 0x1p-20f, slack);
    *upper = __fmul_ru(up, up);
    float smin = INFINITY, mag = 0.f;
    const V3<float> aq = mk3(fabsf(q.x), fabsf(q.y), fabsf(q.z));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        smin = fminf(smin, dot(q, w[k]));
        mag = fmaxf(mag, aq.x * fabsf(w[k].x) + aq.y * fabsf(w[k].y) + aq.z * fabsf(w[k].z));
    }
    const float num = smin - mag * 0x1p-22f - (aq.x + aq.y + aq.z) * (X * 0x1p-22f + e);
    // (num * num leaves float32's range at a distance of 4e9, where num and qq are
    // still far inside it: an infinite bound would drop the nearest triangle.  Below
    // 1e-15 the terms' own roundings are no longer relative)
    *lower = num > 0.f && qq > 0x1p-100f ? num / qq * num * (1.f - 0x1p-20f) : 0.f;
}

// Whether the plane across the direction to the triangle's centroid keeps it
// farther than U (squared), with the margins of tri_bounds_sq, at a fifth of its
// cost.  A point far from the mesh sees a triangle nearly across that
// direction, so few get past it (of 428 M triangles whose leaf passed, in
// 262,144 points against a ring, 17 M).  v: the vertices, E: the point's
// float32 rounding (and more than 4 u |c|, for the differences taken here).
__device__ __forceinline__ bool centroid_apart(const V3<float>* v, V3<float> c, float E, float U) {
    const V3<float> w0 = v[0] - c, w1 = v[1] - c, w2 = v[2] - c;
    const V3<float> q = w0 + w1 + w2;
    const float X = fmaxf(abs_max(w0), fmaxf(abs_max(w1), abs_max(w2)));
    const float q1 = fabsf(q.x) + fabsf(q.y) + fabsf(q.z);
    // sum |q_i| |w_i| <= |q|_1 X: one margin for both of tri_bounds_sq's
    const float num = fminf(dot(q, w0), fminf(dot(q, w1), dot(q, w2))) - q1 * fmaf(X, 0x1p-21f, E);
    return num > 0.f && num * num * (1.f - 0x1p-20f) > U * dot(q, q);
}

__device__ __forceinline__ void load_local(const float4* tri, unsigned j, V3<float> c, V3<float> cl, V3<float>* w) {
    int id;
    load_tri(tri, j, w, &id);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        w[k] = mk3(__fsub_rn(__fsub_rn(w[k].x, c.x), cl.x), __fsub_rn(__fsub_rn(w[k].y, c.y), cl.y),
                   __fsub_rn(__fsub_rn(w[k].z, c.z), cl.z));
}

// The point in the mesh's frame: R^T (p - t) in float64.
__device__ __forceinline__ V3<double> to_local(const PointArgs& g, unsigned i) {
    const double* P = g.pts + 3ull * i;
    const double w0 = P[0] - g.x[3], w1 = P[1] - g.x[7], w2 = P[2] - g.x[11];
    return mk3(fma(g.x[0], w0, fma(g.x[4], w1, g.x[8] * w2)), fma(g.x[1], w0, fma(g.x[5], w1, g.x[9] * w2)),
               fma(g.x[2], w0, fma(g.x[6], w1, g.x[10] * w2)));
}

// The local point as two floats per coordinate.
__device__ __forceinline__ void split_local(V3<double> p, V3<float>* c, V3<float>* cl) {
    *c = mk3((float)p.x, (float)p.y, (float)p.z);
    *cl = mk3((float)(p.x - (double)c->x), (float)(p.y - (double)c->y), (float)(p.z - (double)c->z));
}

// float64 distance (squared) of candidate k of the warp's list on lane k -
// first, for the m <= 32 candidates from first: float64 costs a warp the same
// for one lane as for 32, so it only runs on lists.  Lanes beyond m (and a
// distance that is not a number) come back as (inf, 0x7fffffff).
__device__ __noinline__ void exact_candidates(const PointArgs& g, const PointWarp& W, unsigned first, unsigned m,
                                              double* d2, int* id, V3<double>* q) {
    const unsigned lane = threadIdx.x & 31;
    *d2 = INFINITY;
    *id = 0x7fffffff;
    *q = mk3(0.0, 0.0, 0.0);
    if (lane < m) {
        const V3<double> p = to_local(g, W.ci[first + lane]);
        V3<float> v[3];
        int t;
        load_tri(g.tri, W.cj[first + lane], v, &t);
        bool inside;
        *q = closest_on_triangle<double>(p, mk3((double)v[0].x, (double)v[0].y, (double)v[0].z),
                                         mk3((double)v[1].x, (double)v[1].y, (double)v[1].z),
                                         mk3((double)v[2].x, (double)v[2].y, (double)v[2].z), &inside);
        const V3<double> d = p - *q;
        const double n = dot(d, d);
        if (n <= INFINITY) {
            *d2 = n;
            *id = t;
        }
    }
    __syncwarp();
}

__device__ __forceinline__ bool nearer(double d2, int id, double od2, int oid) {
    return d2 < od2 || (d2 == od2 && id < oid);
}

// The lane with the least (d2, id) of the warp; *d2 becomes that least distance.
__device__ __forceinline__ unsigned nearest_lane(double& d2, int id) {
    unsigned win = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(kFull, d2, o);
        const int oi = __shfl_xor_sync(kFull, id, o);
        const unsigned ow = __shfl_xor_sync(kFull, win, o);
        if (nearer(od, oi, d2, id) || (od == d2 && oi == id && ow < win)) { d2 = od; id = oi; win = ow; }
    }
    return win;
}

// Replaces the last 32 candidates of the current point by the nearest of them
// and returns its squared distance (rounded up), a bound for the rest.
__device__ __noinline__ float thin_candidates(const PointArgs& g, PointWarp& W, unsigned end) {
    const unsigned lane = threadIdx.x & 31, first = end - 32;
    double d2;
    int id;
    V3<double> q;
    exact_candidates(g, W, first, 32, &d2, &id, &q);
    const unsigned win = nearest_lane(d2, id);
    const unsigned j = W.cj[first + win];
    const float low = W.clow[first + win];
    __syncwarp();
    if (lane == 0) {
        W.cj[first] = j;
        W.clow[first] = low;
    }
    __syncwarp();
    return __double2float_ru(d2);
}

__device__ __forceinline__ void point_failed(const PointArgs& g, unsigned i, unsigned status) {
    gd_point_result r{};
    r.d = status == GD_ERR_INVALID_ARG ? NAN : 0.0;
    r.tri = -1;
    r.status = status;
    g.out[i] = r;
    if (status == GD_ERR_TIMEOUT) atomicExch(g.ws + kPointTimeout, 1ull);
}

// The records of the finished points whose candidates fill the list's first m
// <= 32 entries, each point's in one run.
__device__ __noinline__ void finish_points(const PointArgs& g, const PointWarp& W, unsigned m) {
    const unsigned lane = threadIdx.x & 31;
    double d2;
    int id;
    V3<double> q;
    exact_candidates(g, W, 0, m, &d2, &id, &q);
    const unsigned i = lane < m ? W.ci[lane] : 0xffffffffu;
    // the least of each run, at its first lane
    unsigned win = lane;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double od = __shfl_down_sync(kFull, d2, o);
        const int oid = __shfl_down_sync(kFull, id, o);
        const unsigned ow = __shfl_down_sync(kFull, win, o), oi = __shfl_down_sync(kFull, i, o);
        if (lane + o < 32 && oi == i && nearer(od, oid, d2, id)) { d2 = od; id = oid; win = ow; }
    }
    const V3<double> c =
        mk3(__shfl_sync(kFull, q.x, win), __shfl_sync(kFull, q.y, win), __shfl_sync(kFull, q.z, win));
    const unsigned prev = __shfl_up_sync(kFull, i, 1);
    if (lane < m && (lane == 0 || prev != i)) {
        if (id == 0x7fffffff) {
            point_failed(g, i, GD_ERR_TIMEOUT);
        } else {
            gd_point_result r{};
            r.d = sqrt(d2);
            r.tri = id;
            // the closest point in the world frame: R q + t
            r.p[0] = fma(g.x[0], c.x, fma(g.x[1], c.y, fma(g.x[2], c.z, g.x[3])));
            r.p[1] = fma(g.x[4], c.x, fma(g.x[5], c.y, fma(g.x[6], c.z, g.x[7])));
            r.p[2] = fma(g.x[8], c.x, fma(g.x[9], c.y, fma(g.x[10], c.z, g.x[11])));
            r.status = GD_OK;
            g.out[i] = r;
        }
    }
    __syncwarp();
}

constexpr float kGrow = 1.f + 0x1p-20f;

// a stack entry's squared gap (never above the one it was pushed with)
__device__ __forceinline__ float stack_gap(unsigned short h) { return __uint_as_float((unsigned)h << 16); }
__device__ __forceinline__ unsigned short stack_gap(float g) { return (unsigned short)(__float_as_uint(g) >> 16); }

// A point whose walk is shared: its bound, the parts still running, and the
// chain of the parts' answers.
__device__ __forceinline__ float slot_bound(const PointSlot* s) { return __uint_as_float(ld_relaxed(&s->U)); }

// Gives every other of the lowest 64 entries of the stack (the shallowest:
// the largest subtrees) to an idle warp.  *slot: the point's slot, made on its
// first gift.  Returns the entries left.
__device__ __noinline__ unsigned give_half(const PointArgs& g, PointWarp& W, unsigned i, float U, unsigned sp,
                                           unsigned* slot) {
    const unsigned lane = threadIdx.x & 31;
    unsigned rec = kNone, sl = *slot;
    if (lane == 0) {
        if (sl == kNone) {
            const unsigned long long k = atomicAdd(g.ws + kPointSlots, 1ull);
            if (k < kPointMaxSlots) {
                sl = (unsigned)k;
                g.slots[sl] = PointSlot{__float_as_uint(U), 1u, kNone, i, 0u};
                // what stands if a part is lost to the deadline
                gd_point_result r{};
                r.tri = -1;
                r.status = GD_ERR_TIMEOUT;
                g.out[i] = r;
            }
        }
        if (sl != kNone) {
            const unsigned long long t = atomicAdd(g.ws + kPointTail, 1ull);
            if (t < kPointMaxShares) {
                rec = (unsigned)t;
                atomicAdd(&g.slots[sl].parts, 1u);
            }
        }
    }
    rec = __shfl_sync(kFull, rec, 0);
    *slot = sl = __shfl_sync(kFull, sl, 0);
    if (rec == kNone) return sp;
    const unsigned n = min(sp, 64u), ng = (n + 1u) / 2u, nk = n / 2u;  // entries 0, 2, ... go, 1, 3, ... stay
    PointShare& r = g.shares[rec];
    if (lane < ng) r.node[lane] = W.node[2u * lane];
    const unsigned mn = lane < nk ? W.node[2u * lane + 1u] : 0u;
    const unsigned short mg = lane < nk ? W.gap[2u * lane + 1u] : (unsigned short)0;
    __syncwarp();
    if (lane < nk) {
        W.node[lane] = mn;
        W.gap[lane] = mg;
    }
    for (unsigned k = 64u; k < sp; k += 32u) {
        const unsigned at = k + lane;
        const unsigned vn = at < sp ? W.node[at] : 0u;
        const unsigned short vg = at < sp ? W.gap[at] : (unsigned short)0;
        __syncwarp();
        if (at < sp) {
            W.node[at - 32u] = vn;
            W.gap[at - 32u] = vg;
        }
        __syncwarp();
    }
    if (lane == 0) {
        r.slot = sl;
        r.n = ng;
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) {
        __threadfence();
        atomicExch(&r.ready, g.epoch);
    }
    return sp - ng;
}

// One walk by a warp for point i (its local coordinates c + cl), from the sp
// entries of the warp's stack or the nt triangles waiting.  U, the same on every
// lane, is a true upper bound of the squared distance at every step; the
// candidates the point is left with, at most 32, follow the n0 entries of the
// warp's list.  *slot: the slot of a shared point, kNone before the first gift.
// Returns the number of candidates, kNone on a timeout.
__device__ __forceinline__ unsigned walk(const PointArgs& g, PointWarp& W, unsigned i, V3<float> c, V3<float> cl,
                                         float U, unsigned sp, unsigned nt, unsigned n0, unsigned* slot,
                                         unsigned* tests, unsigned* exact, unsigned long long deadline) {
    const unsigned lane = threadIdx.x & 31, lt = lanemask_lt();
    const unsigned first_leaf = 1u << g.L;
    // float32 rounding of the mapped point, plus margin; e: what its two-float form leaves
    const float ca = abs_max(c);
    const float E = ca * 0x1p-22f + FLT_MIN, e = ca * 0x1p-46f + FLT_MIN;
    const V3<float> cm = mk3(c.x - E, c.y - E, c.z - E), cp = mk3(c.x + E, c.y + E, c.z + E);
    unsigned nn = 0, nc = 0;
    bool seen = U < INFINITY;  // a triangle has lowered U (another part's, for a gift)
    unsigned hungry = 0;       // idle warps at the last look

    // keeps the current point's candidates within U (nc <= 64)
    auto compress = [&]() {
        unsigned j[2];
        float low[2];
        bool k[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned at = lane + 32u * h;
            k[h] = false;
            if (at < nc) {
                j[h] = W.cj[n0 + at];
                low[h] = W.clow[n0 + at];
                k[h] = low[h] <= U * kGrow;
            }
        }
        __syncwarp();
        unsigned n = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned m = __ballot_sync(kFull, k[h]);
            if (k[h]) {
                const unsigned at = n0 + n + (unsigned)__popc(m & lt);
                W.cj[at] = j[h];
                W.clow[at] = low[h];
            }
            n += (unsigned)__popc(m);
        }
        nc = n;
        __syncwarp();
    };

    for (unsigned iter = 1;; ++iter) {
        if ((iter & 63u) == 0u && __shfl_sync(kFull, (unsigned)(globaltimer() > deadline), 0)) return kNone;
        const bool last = sp == 0u || !seen;
        if (nt >= 32u || (nt > 0u && last)) {
            const unsigned m = min(nt, 32u);
            nt -= m;
            unsigned j = 0;
            bool in = false;
            if (lane < m) {
                j = W.tri[nt + lane];
                V3<float> v[3];
                int id;
                load_tri(g.tri, j, v, &id);
                in = !centroid_apart(v, c, E, U);
            }
            const unsigned mn = __ballot_sync(kFull, in);
            if (in) W.near[nn + (unsigned)__popc(mn & lt)] = j;
            nn += (unsigned)__popc(mn);
            __syncwarp();
        }
        if (nn >= 32u || (nn > 0u && last && nt == 0u)) {
            const unsigned m = min(nn, 32u);
            nn -= m;
            float low = INFINITY, up = INFINITY;
            unsigned j = 0;
            if (lane < m) {
                j = W.near[nn + lane];
                V3<float> w[3];
                load_local(g.tri, j, c, cl, w);
                tri_bounds_sq(w, e, &low, &up);
            }
            // non-negative floats order like their bits; a NaN (a point beyond float32's range) bounds nothing
            U = fminf(U, __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(fminf(up, INFINITY)))));
            if (!seen) {
                // most of what the descent left behind is beyond the first triangle's bound
                unsigned n = 0;
                for (unsigned k = 0; k < sp; k += 32u) {
                    const unsigned at = k + lane;
                    unsigned node = 0;
                    unsigned short gap = 0;
                    bool in2 = false;
                    if (at < sp) {
                        node = W.node[at];
                        gap = W.gap[at];
                        in2 = stack_gap(gap) <= U * kGrow;
                    }
                    const unsigned mk = __ballot_sync(kFull, in2);
                    if (in2) {
                        W.node[n + (unsigned)__popc(mk & lt)] = node;
                        W.gap[n + (unsigned)__popc(mk & lt)] = gap;
                    }
                    n += (unsigned)__popc(mk);
                    __syncwarp();
                }
                sp = n;
                seen = true;
            }
            const bool cand = lane < m && low <= U * kGrow;
            const unsigned mc = __ballot_sync(kFull, cand);
            if (cand) {
                const unsigned at = n0 + nc + (unsigned)__popc(mc & lt);
                W.cj[at] = j;
                W.ci[at] = i;
                W.clow[at] = low;
            }
            nc += (unsigned)__popc(mc);
            __syncwarp();
            if (nc > 32u) {
                compress();
                while (nc > 32u) {
                    // many triangles at one distance: float64 decides
                    U = fminf(U, thin_candidates(g, W, n0 + nc));
                    if (lane == 0) *exact += 32u;
                    nc -= 31u;
                    compress();
                }
            }
            continue;
        }
        if (nt >= 32u || (nt > 0u && last)) continue;
        if (sp == 0u) break;
        if (hungry && iter >= g.share_steps && sp >= kShareMin) sp = give_half(g, W, i, U, sp, slot);
        // four nodes, their eight descendants three levels down
        const unsigned grp = lane >> 3;
        bool on = grp < sp;
        unsigned node = 0;
        if (on) {
            node = 8u * W.node[sp - 1u - grp] + (lane & 7u);
            on = stack_gap(W.gap[sp - 1u - grp]) <= U * kGrow;
        }
        sp -= min(sp, 4u);
        // now and then a look at the idle warps and the shared bound, whose loads wait together with the boxes
        const bool look = (iter & g.share_mask) == 0u;
        unsigned long long head = 0, tail = 0;
        float Us = INFINITY;
        if (look) {
            head = ld_relaxed64(g.ws + kPointHead);
            tail = ld_relaxed64(g.ws + kPointTail);
            if (*slot != kNone) Us = slot_bound(g.slots + *slot);
        }
        float gap = INFINITY;
        NodeBox box;
        if (on) {
            box = load_node(g.box, node);
            gap = node_gap_sq(box, cm, cp);
            ++*tests;
        }
        if (!seen) {
            // (a triangle's bound is tighter than any box's)
            const float up = on ? fminf(node_upper_sq(box, c, E), INFINITY) : INFINITY;
            U = fminf(U, __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(up))));
        }
        hungry = 0;
        if (look) {
            hungry = __shfl_sync(kFull, (unsigned)(head > tail), 0);
            if (*slot != kNone) {
                Us = __shfl_sync(kFull, Us, 0);
                if (lane == 0 && U < Us) atomicMin(&g.slots[*slot].U, __float_as_uint(U));
                U = fminf(U, Us);
            }
        }
        const bool keep = on && gap <= U * kGrow;
        const bool leaf = node >= first_leaf;
        const unsigned mi = __ballot_sync(kFull, keep && !leaf), ml = __ballot_sync(kFull, keep && leaf);
        __syncwarp();
        if (mi) {
            const unsigned top = (unsigned)__popc(mi) - 1u;
            unsigned pos = (unsigned)__popc(mi & lt);
            if (!seen) {
                // the nearest node on top, so that the first descent is greedy
                const unsigned key = keep && !leaf ? __float_as_uint(gap) : 0xffffffffu;
                const unsigned best = __reduce_min_sync(kFull, key);
                const unsigned near = (unsigned)__ffs((int)__ballot_sync(kFull, key == best && keep && !leaf)) - 1u;
                const unsigned pn = __shfl_sync(kFull, pos, near);
                if (lane == near) pos = top;
                else if (pos == top) pos = pn;
            }
            if (keep && !leaf) {
                W.node[sp + pos] = node;
                W.gap[sp + pos] = stack_gap(gap);
            }
            sp += top + 1u;
        }
        if (ml) {
            unsigned j = 0, two = 0;
            if (keep && leaf) {
                const unsigned l = node - first_leaf;
                j = leaf_begin(g.T, g.L, l);
                two = leaf_begin(g.T, g.L, l + 1) - j > 1u;
            }
            // in leaf order, so that neighbouring lanes load neighbouring records
            const unsigned m2 = __ballot_sync(kFull, two);
            if (keep && leaf) {
                const unsigned at = nt + (unsigned)__popc(ml & lt) + (unsigned)__popc(m2 & lt);
                W.tri[at] = j;
                if (two) W.tri[at + 1u] = j + 1u;
            }
            nt += (unsigned)__popc(ml) + (unsigned)__popc(m2);
        }
        __syncwarp();
    }
    compress();
    return nc;
}

// A part of a shared walk is done: its nc candidates, which follow the n0
// entries of the warp's list, join the slot's chain (thinned to kPartCands by
// float64 if need be).  The last part of the point gathers the chain into the
// list and returns the number of candidates it is left with (kNone if a part
// ran into the deadline); any other returns 0.  Its float64 distances go to the
// call's count at once (a counter of the caller's, reached through a pointer, cost
// 8 % of a large call: the caller then holds it in memory).
__device__ __noinline__ unsigned join_part(const PointArgs& g, PointWarp& W, unsigned i, unsigned slot, unsigned n0,
                                           unsigned nc) {
    const unsigned lane = threadIdx.x & 31, lt = lanemask_lt();
    PointSlot& s = g.slots[slot];
    if (nc == kNone) {
        if (lane == 0) atomicExch(&s.failed, 1u);
    } else if (nc > 0u) {
        if (nc > kPartCands) {
            double d2;
            int id;
            V3<double> q;
            exact_candidates(g, W, n0, nc, &d2, &id, &q);
            if (lane == 0) atomicAdd(g.ws + kPointExact, (unsigned long long)nc);
            const unsigned win = nearest_lane(d2, id);
            const unsigned j = W.cj[n0 + win];
            const float low = W.clow[n0 + win];
            __syncwarp();
            if (lane == 0) {
                W.cj[n0] = j;
                W.clow[n0] = low;
            }
            __syncwarp();
            nc = 1u;
        }
        unsigned k = 0;
        if (lane == 0) k = (unsigned)atomicAdd(g.ws + kPointParts, 1ull);  // at most one a gift and one a slot
        k = __shfl_sync(kFull, k, 0);
        PointPart& p = g.parts[k];
        if (lane < nc) {
            p.tri[lane] = W.cj[n0 + lane];
            p.low[lane] = W.clow[n0 + lane];
        }
        if (lane == 0) {
            p.n = nc;
            p.next = atomicExch(&s.chain, k);
        }
    }
    __threadfence();
    __syncwarp();
    unsigned last = 0;
    if (lane == 0) {
        __threadfence();
        last = atomicSub(&s.parts, 1u) == 1u;
        __threadfence();
    }
    last = __shfl_sync(kFull, last, 0);
    __syncwarp();
    if (!last) return 0u;
    if (__shfl_sync(kFull, ld_relaxed(&s.failed), 0)) return kNone;
    float U = __shfl_sync(kFull, slot_bound(&s), 0);
    unsigned n = 0;
    for (unsigned k = __shfl_sync(kFull, ld_relaxed(&s.chain), 0); k != kNone;) {
        const PointPart& p = g.parts[k];
        const unsigned m = __ldcg(&p.n);
        unsigned j = 0;
        float low = INFINITY;
        if (lane < m) {
            j = __ldcg(&p.tri[lane]);
            low = __ldcg(&p.low[lane]);
        }
        const bool in = lane < m && low <= U * kGrow;
        const unsigned mk = __ballot_sync(kFull, in);
        if (in) {
            const unsigned at = n0 + n + (unsigned)__popc(mk & lt);
            W.cj[at] = j;
            W.ci[at] = i;
            W.clow[at] = low;
        }
        n += (unsigned)__popc(mk);
        __syncwarp();
        if (n > 32u) {
            U = fminf(U, thin_candidates(g, W, n0 + n));
            if (lane == 0) atomicAdd(g.ws + kPointExact, 32ull);
            n -= 31u;
        }
        k = __shfl_sync(kFull, __ldcg(&p.next), 0);
    }
    return n ? n : kNone;
}

// A warp takes chunks of points off a common counter, maps a chunk's points one
// per lane, walks them one after another and finishes them when their
// candidates fill a warp.  When the points have run out it takes gifts from
// the walks still running (it claims the next gift's place and waits for it,
// within the deadline) until every point is answered.  Only warps whose points
// are all answered wait, so the wait ends whatever part of the grid is resident.
__global__ void __launch_bounds__(kPointThreads, kPointCtas) k_point(const __grid_constant__ PointArgs g,
                                                                     unsigned long long chunks) {
    __shared__ PointWarp s_w[kPointWarps];
    __shared__ unsigned long long s_deadline;
    if (threadIdx.x == 0) {
        const unsigned long long now = globaltimer();
        const unsigned long long old = atomicCAS(g.ws + kPointT0, 0ull, now);
        s_deadline = (old ? old : now) + (unsigned long long)g.timeout_ns;
    }
    __syncthreads();
    const unsigned lane = threadIdx.x & 31;
    PointWarp& W = s_w[threadIdx.x >> 5];
    const unsigned* order = g.order && !*g.order_err ? g.order : nullptr;
    unsigned tests = 0, exact = 0;
    unsigned waiting = 0;  // candidates of finished points at the front of the list
    unsigned answered = 0; // points answered and not yet counted
    bool more = true;      // points left on the counter
    // (a lane's counts stay far below 2^32 between two calls: a call has a deadline, a chunk a few points)
    auto count = [&]() {
        unsigned long long nt = tests, ne = exact;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            nt += __shfl_down_sync(kFull, nt, o);
            ne += __shfl_down_sync(kFull, ne, o);
        }
        if (lane == 0) {
            if (nt) atomicAdd(g.ws + kPointTests, nt);
            if (ne) atomicAdd(g.ws + kPointExact, ne);
        }
        tests = exact = 0u;
    };
    for (;;) {
        if (__any_sync(kFull, (tests | exact) >= 1u << 30)) count();
        unsigned m = 0, gift = kNone;
        if (more) {
            unsigned long long t0 = 0;
            if (lane == 0) t0 = atomicAdd(g.ws + kPointTicket, 1ull);
            t0 = __shfl_sync(kFull, t0, 0);
            // the first tickets are whole chunks, the others single points
            m = t0 < chunks ? kChunk : 1u;
            t0 = t0 < chunks ? t0 * kChunk : t0 + chunks * (kChunk - 1u);
            if (t0 >= (unsigned long long)g.n) {
                m = 0u;
                more = false;
                continue;
            }
            bool fin = true;
            if (lane < m) {
                const unsigned i = order ? order[t0 + lane] : (unsigned)(t0 + lane);
                fin = isfinite(g.pts[3ull * i]) && isfinite(g.pts[3ull * i + 1]) && isfinite(g.pts[3ull * i + 2]);
                W.pi[lane] = fin ? i : kNone;
                if (fin) {
                    V3<float> c, cl;
                    split_local(to_local(g, i), &c, &cl);
                    float* o = W.c[lane];
                    o[0] = c.x; o[1] = c.y; o[2] = c.z; o[3] = cl.x; o[4] = cl.y; o[5] = cl.z;
                } else {
                    point_failed(g, i, GD_ERR_INVALID_ARG);
                }
            }
            answered += (unsigned)__popc(__ballot_sync(kFull, !fin));
            __syncwarp();
        } else {
            if (waiting) finish_points(g, W, waiting);
            waiting = 0u;
            if (lane == 0) {
                if (answered) {
                    __threadfence();
                    atomicAdd(g.ws + kPointAnswered, (unsigned long long)answered);
                }
                const unsigned long long k = atomicAdd(g.ws + kPointHead, 1ull);
                if (k < kPointMaxShares) {
                    for (unsigned spin = 0;; ++spin) {
                        if (ld_acquire(&g.shares[k].ready) == g.epoch) {
                            gift = (unsigned)k;
                            break;
                        }
                        if ((spin & 3u) == 3u &&
                            (ld_relaxed64(g.ws + kPointAnswered) >= (unsigned long long)g.n || globaltimer() > s_deadline))
                            break;
                        __nanosleep(spin < 16u ? 200u : 800u);
                    }
                }
            }
            answered = 0u;
            gift = __shfl_sync(kFull, gift, 0);
            __syncwarp();
            if (gift == kNone) break;
            m = 1u;
        }
        for (unsigned k = 0; k < m; ++k) {
            unsigned ik, sp, nt = 0, slot = kNone;
            V3<float> ck, clk;
            float U = INFINITY;
            if (gift != kNone) {
                const PointShare& r = g.shares[gift];
                slot = __ldcg(&r.slot);
                sp = __ldcg(&r.n);
                if (lane < sp) {
                    W.node[lane] = __ldcg(&r.node[lane]);
                    W.gap[lane] = 0;
                }
                ik = __ldcg(&g.slots[slot].i);
                U = __shfl_sync(kFull, slot_bound(g.slots + slot), 0);
                split_local(to_local(g, ik), &ck, &clk);
            } else {
                ik = W.pi[k];
                if (ik == kNone) continue;
                const float* o = W.c[k];
                ck = mk3(o[0], o[1], o[2]);
                clk = mk3(o[3], o[4], o[5]);
                // the root's descendants from which the leaves are a multiple of three levels down
                sp = 0;
                if (g.L < 3) {
                    nt = (unsigned)g.T;  // at most 7 triangles
                    if (lane < nt) W.tri[lane] = lane;
                } else {
                    sp = 1u << (g.L % 3);
                    if (lane < sp) {
                        W.node[lane] = sp | lane;
                        W.gap[lane] = 0;
                    }
                }
            }
            __syncwarp();
            unsigned nc = walk(g, W, ik, ck, clk, U, sp, nt, waiting, &slot, &tests, &exact, s_deadline);
            if (slot != kNone) {
                nc = join_part(g, W, ik, slot, waiting, nc);
                if (nc == 0u) continue;  // others still walk parts of the point
            } else if (nc == 0u) {
                nc = kNone;  // cannot happen: the nearest triangle is never dropped
            }
            if (lane == 0 && nc != kNone) exact += nc;
            ++answered;
            if (nc == kNone) {
                if (lane == 0) point_failed(g, ik, GD_ERR_TIMEOUT);
                continue;
            }
            if (waiting + nc > 32u) {
                finish_points(g, W, waiting);
                // this point's candidates move to the front
                unsigned j = 0;
                if (lane < nc) j = W.cj[waiting + lane];
                __syncwarp();
                if (lane < nc) {
                    W.cj[lane] = j;
                    W.ci[lane] = ik;
                }
                __syncwarp();
                waiting = 0u;
            }
            waiting += nc;
        }
    }
    count();
}

// 10 bits of v spread to every third bit
__device__ __forceinline__ unsigned long long spread10(unsigned v) {
    unsigned long long r = 0;
#pragma unroll
    for (int b = 0; b < 10; ++b) r |= (unsigned long long)((v >> b) & 1u) << (3 * b);
    return r;
}

// Morton key of each point in the mesh's frame, quantised in the root box
// (points outside clamp to its faces: the key only orders the work), and the
// counts of its digits for the sort's passes
constexpr int kKeyPasses = 4;  // 30 bits

__global__ void __launch_bounds__(256) k_point_keys(const __grid_constant__ PointArgs g, unsigned long long* keys,
                                                    unsigned* hist) {
    __shared__ unsigned h[kKeyPasses][256];
    for (int p = 0; p < kKeyPasses; ++p) h[p][threadIdx.x] = 0u;
    __syncthreads();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += (long long)gridDim.x * blockDim.x) {
        const double* P = g.pts + 3 * i;
        const double w0 = P[0] - g.x[3], w1 = P[1] - g.x[7], w2 = P[2] - g.x[11];
        const double l[3] = {g.x[0] * w0 + g.x[4] * w1 + g.x[8] * w2, g.x[1] * w0 + g.x[5] * w1 + g.x[9] * w2,
                             g.x[2] * w0 + g.x[6] * w1 + g.x[10] * w2};
        unsigned long long key = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float lo = g.box[6 + k], hi = g.box[9 + k];
            const float ext = hi - lo;
            float f = ext > 0.f ? (float)((l[k] - lo) / ext) : 0.f;
            f = f == f ? fminf(fmaxf(f, 0.f), 1.f) : 0.f;  // NaN (a non-finite point) to 0
            const unsigned c = min(1023u, (unsigned)(f * 1024.f));
            key |= spread10(c) << k;
        }
        keys[i] = key;
#pragma unroll
        for (int p = 0; p < kKeyPasses; ++p) atomicAdd(&h[p][(unsigned)(key >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = 0; p < kKeyPasses; ++p) {
        const unsigned n = h[p][threadIdx.x];
        if (n) atomicAdd(hist + 256 * p + threadIdx.x, n);
    }
}

__global__ void k_point_init(unsigned long long* ws) {
    static_assert(kPointWords <= 128, "one word a thread");
    if (threadIdx.x < kPointWords) ws[threadIdx.x] = 0ull;
}

}  // namespace

int sort_points(const PointArgs& g, const SortWork& w, unsigned long long* const keys[2], unsigned* const vals[2],
                cudaStream_t st) {
    sort_clear(w, g.n, st);
    k_point_keys<<<(unsigned)std::min(152ll * 8, (g.n + 255) / 256), 256, 0, st>>>(g, keys[0], w.hist);
    return radix_sort_pairs(w, keys, vals, g.n, 0, kKeyPasses, st);
}

cudaError_t launch_point(PointArgs g, int sms, cudaStream_t st) {
    k_point_init<<<1, 128, 0, st>>>(g.ws);
    if (g.n > 0) {
        const long long warps = (long long)sms * kPointCtas * kPointWarps;
        // the points in chunks, whose float64 mapping costs a warp as much as
        // one point's, but for the last 16 a warp, which go one by one to even
        // out the end
        const long long chunks = std::max(0ll, g.n - 16 * warps) / kChunk;
        // Four CTAs an SM beyond the points' own take parts of long walks.  A
        // call that leaves warps idle from the start divides walks early (1,000
        // points: 0.20 ms, 0.22 from 16 steps on, 0.25 from 32); one that keeps
        // them busy has only its tail to even out (0.6 ms; 0.8 from 64 steps on)
        const bool full = g.n >= 4 * warps;
        g.share_steps = full ? 32u : 8u;
        g.share_mask = full ? 7u : 3u;
        const long long ctas = std::min((long long)sms * kPointCtas, (g.n + kPointWarps - 1) / kPointWarps + 4 * sms);
        k_point<<<(unsigned)ctas, kPointThreads, 0, st>>>(g, (unsigned long long)chunks);
    }
    return cudaGetLastError();
}

}  // namespace gd
