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
// What bounds it: issue slots and L1/L2 latency of the box tests (about 4,000
// a point on a ring, most of them near-ties), not the bytes of the points.
// A thread per point, with float64 in the walk, left one lane of a warp
// working at a time: 262,144 device points against a 7.5 M-triangle ring took
// 258 ms, 1,000 host points against a 204,800-triangle gear 9.4 ms; this form
// 13.6 ms and 0.29 ms.
#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "gd_geom.cuh"
#include "gd_internal.cuh"
#include "gd_launch.h"

namespace gd {

namespace {

constexpr int kPointWarps = 4;
constexpr int kPointThreads = 32 * kPointWarps;
constexpr int kPointCtas = 8;  // CTAs per SM the kernel is compiled for: 32 warps, 64 registers a thread
// The stack of a walk.  A step pushes at most 32 entries, each at least three
// levels below the shallowest entry it took; entries of a later step lie above
// those of an earlier one and are taken first, so the pushes alive at one time
// have depths three apart and there are at most 1 + 30 / 3 of them.
constexpr int kStack = 384;
constexpr int kTriWait = 96;  // < 32 waiting triangles before a step, at most 64 more after it
constexpr int kList = 96;     // <= 32 of finished points, <= 32 of this one, 32 more in a pass

struct PointWarp {
    uint2 stack[kStack];     // node, bits of its squared gap
    unsigned tri[kTriWait];  // triangles whose leaf passed
    unsigned cj[kList];      // candidates for float64: triangle,
    unsigned ci[kList];      //   point,
    float clow[kList];       //   lower bound (squared)
};

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

// Squared distance from the box [c - E, c + E] to the node's box (every
// float32 step rounds at most one unit, so the caller compares it against its
// bound grown by 2^-20 relative), and *up, a rigorous upper bound of the
// squared distance from any point of [c - E, c + E] to the mesh: the node's
// box is tight, so each of its faces holds a vertex, which is no farther than
// the face's farthest point.
__device__ __forceinline__ float node_bounds_sq(const float* box, unsigned node, V3<float> c, float E, float* up) {
    const float2* b = reinterpret_cast<const float2*>(box + 6ull * node);
    const float2 x = __ldg(b), y = __ldg(b + 1), z = __ldg(b + 2);
    const float lo[3] = {x.x, x.y, y.x}, hi[3] = {y.y, z.x, z.y};
    const float cc[3] = {c.x, c.y, c.z};
    float s = 0.f, n2[3], f2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = lo[k] - cc[k], b2 = cc[k] - hi[k];
        const float g = fmaxf(0.f, fmaxf(a, b2) - E);
        s = fmaf(g, g, s);
        const float n = fminf(fabsf(a), fabsf(b2)) + E, f = fmaxf(fabsf(a), fabsf(b2)) + E;
        n2[k] = n * n;
        f2[k] = f * f;
    }
    const float u = fminf(n2[0] + f2[1] + f2[2], fminf(f2[0] + n2[1] + f2[2], f2[0] + f2[1] + n2[2]));
    *up = u * (1.f + 0x1p-20f);
    return s;
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
    *lower = num > 0.f && qq > 0.f ? num * num / qq * (1.f - 0x1p-20f) : 0.f;
}

// The point in the mesh's frame: R^T (p - t) in float64.
__device__ __forceinline__ V3<double> to_local(const PointArgs& g, unsigned i) {
    const double* P = g.pts + 3ull * i;
    const double w0 = P[0] - g.x[3], w1 = P[1] - g.x[7], w2 = P[2] - g.x[11];
    return mk3(fma(g.x[0], w0, fma(g.x[4], w1, g.x[8] * w2)), fma(g.x[1], w0, fma(g.x[5], w1, g.x[9] * w2)),
               fma(g.x[2], w0, fma(g.x[6], w1, g.x[10] * w2)));
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

// Replaces the last 32 candidates of the current point by the nearest of them
// and returns its squared distance (rounded up), a bound for the rest.
__device__ __noinline__ float thin_candidates(const PointArgs& g, PointWarp& W, unsigned end) {
    const unsigned lane = threadIdx.x & 31, first = end - 32;
    double d2;
    int id;
    V3<double> q;
    exact_candidates(g, W, first, 32, &d2, &id, &q);
    unsigned win = lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(kFull, d2, o);
        const int oi = __shfl_xor_sync(kFull, id, o);
        const unsigned ow = __shfl_xor_sync(kFull, win, o);
        if (nearer(od, oi, d2, id) || (od == d2 && oi == id && ow < win)) { d2 = od; id = oi; win = ow; }
    }
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

// One walk of the tree by a warp for point i (its local coordinates c + cl).
// U, the same on every lane, is a true upper bound of the squared distance at
// every step; the candidates the point is left with, at most 32, follow the
// n0 entries of the warp's list.  Returns their number, 0 on a timeout.
__device__ __forceinline__ unsigned walk(const PointArgs& g, PointWarp& W, unsigned i, V3<float> c, V3<float> cl,
                                         unsigned n0, unsigned* tests, unsigned* exact, unsigned long long deadline) {
    const unsigned lane = threadIdx.x & 31, lt = lanemask_lt();
    const unsigned first_leaf = 1u << g.L;
    // float32 rounding of the mapped point, plus margin; e: what its two-float form leaves
    const float cm = abs_max(c);
    const float E = cm * 0x1p-22f + FLT_MIN, e = cm * 0x1p-46f + FLT_MIN;
    float U = INFINITY;
    unsigned sp = 0, nt = 0, nc = 0;
    bool seen = false;  // a triangle has lowered U

    auto visit = [&](bool on, unsigned node) {
        float gap = INFINITY, up = INFINITY;
        if (on) {
            gap = node_bounds_sq(g.box, node, c, E, &up);
            ++*tests;
        }
        // non-negative floats order like their bits; a NaN (a point beyond float32's range) bounds nothing
        U = fminf(U, __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(fminf(up, INFINITY)))));
        const bool keep = on && gap <= U * kGrow;
        const bool leaf = node >= first_leaf;
        const unsigned mi = __ballot_sync(kFull, keep && !leaf);
        if (mi) {
            // the nearest node on top, so that the first descent is greedy
            const unsigned key = keep && !leaf ? __float_as_uint(gap) : 0xffffffffu;
            const unsigned best = __reduce_min_sync(kFull, key);
            const unsigned near = (unsigned)__ffs((int)__ballot_sync(kFull, key == best && keep && !leaf)) - 1u;
            const unsigned last = (unsigned)__popc(mi) - 1u;
            unsigned pos = (unsigned)__popc(mi & lt);
            const unsigned pn = __shfl_sync(kFull, pos, near);
            if (lane == near) pos = last;
            else if (pos == last) pos = pn;
            if (keep && !leaf) W.stack[sp + pos] = make_uint2(node, __float_as_uint(gap));
            sp += last + 1u;
        }
        const unsigned ml = __ballot_sync(kFull, keep && leaf);
        if (ml) {
            const unsigned l = node - first_leaf;
            unsigned j = 0, two = 0;
            if (keep && leaf) {
                j = leaf_begin(g.T, g.L, l);
                two = leaf_begin(g.T, g.L, l + 1) - j > 1u;
                W.tri[nt + (unsigned)__popc(ml & lt)] = j;
            }
            nt += (unsigned)__popc(ml);
            const unsigned m2 = __ballot_sync(kFull, two);
            if (two) W.tri[nt + (unsigned)__popc(m2 & lt)] = j + 1u;
            nt += (unsigned)__popc(m2);
        }
        __syncwarp();
    };

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

    // the root's descendants, so many levels down that the leaves are a multiple of three below
    const int e0 = g.L <= 5 ? g.L : 3 + (g.L % 3);
    visit(lane < (1u << e0), (1u << e0) | (lane & ((1u << e0) - 1u)));
    for (unsigned iter = 1;; ++iter) {
        if ((iter & 63u) == 0u && __shfl_sync(kFull, (unsigned)(globaltimer() > deadline), 0)) return 0u;
        if (nt >= 32u || (nt > 0u && (sp == 0u || !seen))) {
            const unsigned m = min(nt, 32u);
            nt -= m;
            float low = INFINITY, up = INFINITY;
            unsigned j = 0;
            if (lane < m) {
                j = W.tri[nt + lane];
                V3<float> v[3];
                int id;
                load_tri(g.tri, j, v, &id);
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    v[k] = mk3(__fsub_rn(__fsub_rn(v[k].x, c.x), cl.x), __fsub_rn(__fsub_rn(v[k].y, c.y), cl.y),
                               __fsub_rn(__fsub_rn(v[k].z, c.z), cl.z));
                tri_bounds_sq(v, e, &low, &up);
            }
            U = fminf(U, __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(fminf(up, INFINITY)))));
            seen = true;
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
        if (sp == 0u) break;
        const unsigned grp = lane >> 3;
        bool on = grp < sp;
        unsigned node = 0;
        if (on) {
            const uint2 s = W.stack[sp - 1u - grp];
            node = 8u * s.x + (lane & 7u);
            on = __uint_as_float(s.y) <= U * kGrow;
        }
        sp -= min(sp, 4u);
        __syncwarp();
        visit(on, node);
    }
    compress();
    return nc;
}

// A warp takes chunks of points off a common counter (the walks differ by
// orders of magnitude), maps a chunk's points one per lane, walks them one
// after another and finishes them when their candidates fill a warp.
__global__ void __launch_bounds__(kPointThreads, kPointCtas) k_point(const __grid_constant__ PointArgs g,
                                                                     unsigned chunk) {
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
    unsigned long long tests = 0, exact = 0;
    unsigned waiting = 0;  // candidates of finished points at the front of the list
    for (;;) {
        unsigned long long t0 = 0;
        if (lane == 0) t0 = atomicAdd(g.ws + kPointTicket, (unsigned long long)chunk);
        t0 = __shfl_sync(kFull, t0, 0);
        if (t0 >= (unsigned long long)g.n) break;
        const unsigned m = (unsigned)min((unsigned long long)chunk, (unsigned long long)g.n - t0);
        unsigned i = 0;
        bool fin = false;
        V3<float> c = mk3(0.f, 0.f, 0.f), cl = c;
        if (lane < m) {
            i = g.order ? g.order[t0 + lane] : (unsigned)(t0 + lane);
            fin = isfinite(g.pts[3ull * i]) && isfinite(g.pts[3ull * i + 1]) && isfinite(g.pts[3ull * i + 2]);
            if (fin) {
                const V3<double> p = to_local(g, i);
                c = mk3((float)p.x, (float)p.y, (float)p.z);
                cl = mk3((float)(p.x - (double)c.x), (float)(p.y - (double)c.y), (float)(p.z - (double)c.z));
            } else {
                point_failed(g, i, GD_ERR_INVALID_ARG);
            }
        }
        for (unsigned k = 0; k < m; ++k) {
            if (!__shfl_sync(kFull, (unsigned)fin, k)) continue;
            const unsigned ik = __shfl_sync(kFull, i, k);
            const V3<float> ck =
                mk3(__shfl_sync(kFull, c.x, k), __shfl_sync(kFull, c.y, k), __shfl_sync(kFull, c.z, k));
            const V3<float> clk =
                mk3(__shfl_sync(kFull, cl.x, k), __shfl_sync(kFull, cl.y, k), __shfl_sync(kFull, cl.z, k));
            unsigned nt = 0, ne = 0;
            const unsigned nc = walk(g, W, ik, ck, clk, waiting, &nt, &ne, s_deadline);
            tests += nt;
            exact += ne;
            if (nc == 0u) {
                if (lane == 0) point_failed(g, ik, GD_ERR_TIMEOUT);
                continue;
            }
            if (lane == 0) exact += nc;
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
    if (waiting) finish_points(g, W, waiting);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tests += __shfl_down_sync(kFull, tests, o);
        exact += __shfl_down_sync(kFull, exact, o);
    }
    if (lane == 0) {
        if (tests) atomicAdd(g.ws + kPointTests, tests);
        if (exact) atomicAdd(g.ws + kPointExact, exact);
    }
}

// 10 bits of v spread to every third bit
__device__ __forceinline__ unsigned long long spread10(unsigned v) {
    unsigned long long r = 0;
#pragma unroll
    for (int b = 0; b < 10; ++b) r |= (unsigned long long)((v >> b) & 1u) << (3 * b);
    return r;
}

// Morton key of each point in the mesh's frame, quantised in the root box
// (points outside clamp to its faces: the key only orders the work)
__global__ void k_point_keys(PointArgs g, unsigned long long* keys, unsigned* vals) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
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
    vals[i] = (unsigned)i;
}

__global__ void k_point_init(unsigned long long* ws) {
    if (threadIdx.x < kPointWords) ws[threadIdx.x] = 0ull;
}

}  // namespace

int sort_points(const PointArgs& g, unsigned long long* const keys[2], unsigned* const vals[2], unsigned* hist,
                cudaStream_t st) {
    k_point_keys<<<(unsigned)((g.n + 255) / 256), 256, 0, st>>>(g, keys[0], vals[0]);
    return radix_sort_pairs(keys, vals, g.n, 30, hist, st);
}

cudaError_t launch_point(const PointArgs& g, int sms, cudaStream_t st) {
    k_point_init<<<1, 32, 0, st>>>(g.ws);
    if (g.n > 0) {
        const long long warps = (long long)sms * kPointCtas * kPointWarps;
        // a warp's next points in chunks of up to 4: their float64 mapping
        // then costs a quarter, and the last chunks still even out
        const long long chunk = std::max(1ll, std::min(4ll, g.n / (8 * warps)));
        const long long ctas = std::min((long long)sms * kPointCtas, (g.n + chunk * kPointWarps - 1) / (chunk * kPointWarps));
        k_point<<<(unsigned)ctas, kPointThreads, 0, st>>>(g, (unsigned)chunk);
    }
    return cudaGetLastError();
}

}  // namespace gd
