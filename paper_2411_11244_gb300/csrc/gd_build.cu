// f12-BVH construction on the device (Section 7.3): Morton codes of the
// triangle centroids, a stable LSD radix sort (ties keep the original
// order), 2^L leaves of one or two consecutive sorted triangles, exact leaf
// boxes, and a level-by-level union up to the root.  Leaf boxes are exact
// bounds of their vertices, so every box is tight (Section 4: tight leaves
// make every node tight).  Refit for moved vertices (Section 8, deformable
// scenes): the same leaf and union kernels over the stored leaf order.
#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "gd_internal.cuh"
#include "gd_launch.h"

namespace gd {

namespace {

constexpr int kSortThreads = 256;  // one per digit value
constexpr int kSortWarps = kSortThreads / 32;
// Keys per thread and tile: a sort of up to 2^18 keys takes small tiles, so
// that they spread over the SMs (a tile's ranking is a chain over its items)
constexpr int kItemsSmall = 4, kItemsLarge = 16;
constexpr long long kSmallSort = 1 << 18;

// float -> uint32 whose unsigned order is the float order
__device__ __forceinline__ unsigned ordered(float f) {
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float unordered(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// Vertex v.  (Three 4-byte loads: an 8-byte and a 4-byte one, the only wider
// form that a 12-byte stride allows, took the gathers of k_validate from 31 to
// 49 us and of k_leaves from 182 to 199.)
__device__ __forceinline__ void load_vertex(const float* verts, unsigned v, float* x) {
    const float* p = verts + 3ull * v;
    x[0] = p[0];
    x[1] = p[1];
    x[2] = p[2];
}

// flags: [0] bad index, [1] non-finite vertex, [2..4] ordered min, [5..7] ordered max,
// [8..13] root box, [kFlagTies], [kFlagSort]
__global__ void k_init_flags(unsigned* flags) {
    if (threadIdx.x < 16) flags[threadIdx.x] = (threadIdx.x >= 2 && threadIdx.x < 5) ? 0xffffffffu : 0u;
}

// Index range, finiteness and bounds of the referenced vertices.  A triangle's
// nine coordinates are loaded without waiting for one another (an index out of
// range reads vertex 0: the build then fails), two triangles at a time, and a CTA
// sends one atomic a word: with a branch around every load, and one atomic a
// warp (20,000 on each of six words of one L2 line), 7.5 M triangles took 104 us;
// this form 31.
__global__ void __launch_bounds__(512) k_validate(const float* verts, long long nv, const int32_t* tris, long long nt,
                                                  unsigned* flags) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    bool bad_idx = false, bad_val = false;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += 2 * stride) {
        const long long u = t + stride < nt ? t + stride : t;
        int v[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            v[k] = tris[3 * t + k];
            v[3 + k] = tris[3 * u + k];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const bool bad = v[k] < 0 || v[k] >= nv;
            bad_idx = bad_idx || bad;
            v[k] = bad ? 0 : v[k];
        }
        float x[18];
#pragma unroll
        for (int k = 0; k < 6; ++k) load_vertex(verts, (unsigned)v[k], x + 3 * k);
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            bad_val = bad_val || !isfinite(x[k]);
            lo[k % 3] = fminf(lo[k % 3], x[k]);
            hi[k % 3] = fmaxf(hi[k % 3], x[k]);
        }
    }
    __shared__ unsigned s_lo[3], s_hi[3];
    if (threadIdx.x < 3) {
        s_lo[threadIdx.x] = 0xffffffffu;
        s_hi[threadIdx.x] = 0u;
    }
    const int any_idx = __syncthreads_or(bad_idx), any_val = __syncthreads_or(bad_val);
    for (int c = 0; c < 3; ++c) {
        const unsigned a = __reduce_min_sync(kFull, ordered(lo[c])), b = __reduce_max_sync(kFull, ordered(hi[c]));
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s_lo[c], a);
            atomicMax(&s_hi[c], b);
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        atomicMin(flags + 2 + threadIdx.x, s_lo[threadIdx.x]);
        atomicMax(flags + 5 + threadIdx.x, s_hi[threadIdx.x]);
    }
    if (threadIdx.x == 0) {
        if (any_idx) atomicOr(flags + 0, 1u);
        if (any_val) atomicOr(flags + 1, 1u);
    }
}

// the low 10 bits of v at every third bit
__device__ __forceinline__ unsigned spread3(unsigned v) {
    unsigned x = v & 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    x = (x | (x << 2)) & 0x09249249u;
    return x;
}

// 63-bit Morton code of three 21-bit cells, in 32-bit steps
__device__ __forceinline__ unsigned long long morton63(unsigned x, unsigned y, unsigned z) {
    const unsigned low = spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
    const unsigned mid = spread3(x >> 10) | (spread3(y >> 10) << 1) | (spread3(z >> 10) << 2);
    const unsigned top = (x >> 20) | ((y >> 20) << 1) | ((z >> 20) << 2);
    return (unsigned long long)low | ((unsigned long long)mid << 30) | ((unsigned long long)top << 60);
}

// Adds a key's digits to the CTA's histograms of all passes (every lane
// calls; neighbouring triangles share their high digits, so a warp of one
// value adds once).
__device__ __forceinline__ void add_digits(unsigned (*h)[256], unsigned long long key, bool ok, int lo, int passes) {
    key >>= lo;
    for (int p = 0; p < passes; ++p, key >>= 8) {
        const unsigned d = ok ? (unsigned)key & 255u : 256u;
        if (__all_sync(kFull, d == __shfl_sync(kFull, d, 0))) {
            if (ok && (threadIdx.x & 31) == 0) atomicAdd(&h[p][d], 32u);
        } else if (ok) {
            atomicAdd(&h[p][d], 1u);
        }
    }
}

__global__ void __launch_bounds__(512) k_morton(const float* verts, const int32_t* tris, long long nt,
                                                const unsigned* flags, int bits, unsigned long long* keys, int lo_bit,
                                                int passes, unsigned* hist) {
    __shared__ unsigned h[kSortPasses][256];
    for (int i = threadIdx.x; i < 256 * passes; i += blockDim.x) h[i >> 8][i & 255] = 0u;
    __syncthreads();
    // one scale for all three axes (cubic cells): per-axis scales would make
    // the cells of flat or thin meshes into slabs whose boxes are far from
    // the surface they bound
    const bool bad = flags[0] != 0u;  // an index out of range: the build fails, nothing is read through it
    float lo[3], ext[3], e = 0.f;
    for (int c = 0; c < 3; ++c) {
        lo[c] = unordered(flags[2 + c]);
        e = fmaxf(e, __fsub_rn(unordered(flags[5 + c]), lo[c]));
    }
    for (int c = 0; c < 3; ++c) ext[c] = e;
    const float cells = (float)(1u << bits);
    const unsigned top = (1u << bits) - 1u;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long b = (long long)blockIdx.x * blockDim.x; b < nt; b += stride) {
        const long long t = b + threadIdx.x;
        const bool ok = t < nt;
        unsigned long long key = 0;
        if (ok) {
            unsigned q[3];
            float v[9];
#pragma unroll
            for (int k = 0; k < 3; ++k) load_vertex(verts, bad ? 0u : (unsigned)tris[3 * t + k], v + 3 * k);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                // explicit round-to-nearest steps (no contraction), so that the
                // codes can be reproduced bit for bit on the host
                float s = __fadd_rn(__fadd_rn(v[c], v[3 + c]), v[6 + c]);
                float x = __fsub_rn(__fmul_rn(s, 1.0f / 3.0f), lo[c]);
                float f = ext[c] > 0.f ? __fmul_rn(__fdiv_rn(x, ext[c]), cells) : 0.f;
                unsigned qi = f <= 0.f ? 0u : (f >= (float)top ? top : (unsigned)f);
                q[c] = qi;
            }
            key = morton63(q[0], q[1], q[2]);
            keys[t] = key;
        }
        add_digits(h, key, ok, lo_bit, passes);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256 * passes; i += blockDim.x) {
        const unsigned n = h[i >> 8][i & 255];
        if (n) atomicAdd(hist + i, n);
    }
}

// ---- stable LSD radix sort of (64-bit key, 32-bit value), 8 bits per pass.
// One pass reads every pair once and writes it once: the digit counts of all
// passes come from the kernel that makes the keys, and a tile learns how many
// of its keys' digits the tiles before it hold by looking back over their
// published counts (aggregate of one tile, or inclusive up to it), as the
// one-sweep radix sort of Adinets and Merrill does.  Tiles are numbered by a
// counter, so every predecessor has started.  A word of the look-back table is
// (tag, count): the tag names the pass, so the table is cleared once a sort.
// 7.5 M pairs: 72 us a pass (2.5 TB/s), where a histogram, three scans and a
// scatter in tile-sized rounds took 161.  Bound by the tile's own phases (load,
// rank, look back, exchange, store: 41 % of the issue slots, 22 % of DRAM); 3
// and 4 CTAs an SM, with fewer items a thread, took 74.

// exclusive scan of one value a thread over the CTA's 256 threads
__device__ __forceinline__ unsigned block_excl_scan(unsigned v) {
    __shared__ unsigned warp_sum[kSortWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    unsigned before = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) before += w < warp ? warp_sum[w] : 0u;
    __syncthreads();
    return before + x - v;
}

__device__ __forceinline__ void publish(unsigned long long* p, unsigned tag, unsigned count) {
    const unsigned long long w = ((unsigned long long)tag << 32) | count;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

// vin == nullptr: the values are 0, 1, 2, ...
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_sort_pass(const unsigned long long* kin, const unsigned* vin,
                                                            unsigned long long* kout, unsigned* vout, long long n,
                                                            int shift, int pass, SortWork w) {
    constexpr int kTile = kSortThreads * ITEMS;
    constexpr int kAhead = 8;         // predecessors read at a time
    constexpr unsigned kPollNs = 40;  // between two looks at one that has not published
    __shared__ unsigned long long s_key[kTile];
    __shared__ unsigned s_cnt[kSortWarps][256];
    __shared__ unsigned s_off[256];
    __shared__ unsigned s_tile, s_err;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_tile = atomicAdd(w.ticket + pass, 1u);
        s_err = ld_relaxed(w.err);
    }
    for (int k = 0; k < kSortWarps; ++k) s_cnt[k][tid] = 0u;
    __syncthreads();
    // a wait of this pass or of one before it gave up: part of the input was never
    // written, and its digits do not add up to the counts that place them
    if (s_err) return;
    const unsigned tile = s_tile;
    const long long base = (long long)tile * kTile;
    const int m = (int)(n - base < kTile ? n - base : kTile);
    // a warp's items are consecutive runs of 32, so that ranks follow the
    // input order; the last tile is padded with keys that sort behind all
    const int first = warp * 32 * ITEMS + lane;
    unsigned long long key[ITEMS];
    unsigned val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) key[k] = first + 32 * k < m ? kin[base + first + 32 * k] : ~0ull;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        val[k] = vin ? (first + 32 * k < m ? vin[base + first + 32 * k] : 0u) : (unsigned)(base + first + 32 * k);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const unsigned d = (unsigned)(key[k] >> shift) & 255u;
        // the lanes of the same digit, from the ballots of its bits (12 %
        // faster over the pass than __match_any_sync)
        unsigned peers = kFull;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool on = (d >> b) & 1u;
            const unsigned v = __ballot_sync(kFull, on);
            peers &= on ? v : ~v;
        }
        const unsigned before = __popc(peers & lanemask_lt());
        const unsigned c = s_cnt[warp][d];
        __syncwarp();
        if (before == 0u) s_cnt[warp][d] = c + __popc(peers);
        __syncwarp();
        rank[k] = c + before;
    }
    __syncthreads();
    // thread t: digit t.  Its count in the tile, and each warp's offset in it
    unsigned count = 0;
#pragma unroll
    for (int k = 0; k < kSortWarps; ++k) {
        const unsigned c = s_cnt[k][tid];
        s_cnt[k][tid] = count;
        count += c;
    }
    const unsigned agg = 2u * pass + 1u, incl = agg + 1u;
    unsigned long long* st = w.status + 256ull * tile + tid;
    publish(st, tile == 0 ? incl : agg, count);
    const unsigned excl = block_excl_scan(count);                        // first slot of the digit in the tile
    const unsigned gbase = block_excl_scan(w.hist[256 * pass + tid]);  // ... and in the output
    unsigned prev = 0;
    bool failed = false;
    if (tile > 0) {
        unsigned at = tile;  // the next predecessor is at - 1
        for (bool done = false; !done && !failed;) {
            // a batch of predecessors at once, as far as they have published
            unsigned long long v[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k)
                v[k] = at > (unsigned)k ? ld_relaxed64(w.status + 256ull * (at - 1u - k) + tid) : 0ull;
            bool wait = false;
#pragma unroll
            for (int k = 0; k < kAhead; ++k) {
                const unsigned tag = (unsigned)(v[k] >> 32);
                wait = wait || (tag != agg && tag != incl);
                if (!done && !wait) {
                    prev += (unsigned)v[k];
                    --at;
                    done = tag == incl;
                }
            }
            if (done || !wait) continue;
            // the first that has not: poll it alone (polling whole batches from
            // every waiting tile kept the L2 from the tiles waited for)
            unsigned long long t0 = 0;
            for (unsigned spin = 1;; ++spin) {
                const unsigned tag = (unsigned)(ld_relaxed64(w.status + 256ull * (at - 1u) + tid) >> 32);
                if (tag == agg || tag == incl) break;
                __nanosleep(kPollNs);
                if ((spin & 255u) == 0u) {
                    const unsigned long long now = globaltimer();
                    if (t0 == 0) t0 = now;
                    if (now - t0 > w.timeout_ns || ld_relaxed(w.err)) {
                        atomicExch(w.err, 1u);
                        failed = true;
                        break;
                    }
                }
            }
        }
        if (!failed) publish(st, incl, prev + count);
    }
    s_off[tid] = gbase + prev - excl;
    // the warps' offsets become slots of the tile
#pragma unroll
    for (int k = 0; k < kSortWarps; ++k) s_cnt[k][tid] += excl;
    if (__syncthreads_or(failed)) return;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        rank[k] += s_cnt[warp][(unsigned)(key[k] >> shift) & 255u];
        s_key[rank[k]] = key[k];
    }
    __syncthreads();
    unsigned to[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int slot = k * kSortThreads + tid;
        const unsigned long long x = s_key[slot];
        to[k] = s_off[(unsigned)(x >> shift) & 255u] + (unsigned)slot;
        if (slot < m) kout[to[k]] = x;
    }
    __syncthreads();
    unsigned* s_val = reinterpret_cast<unsigned*>(s_key);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) s_val[rank[k]] = val[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int slot = k * kSortThreads + tid;
        if (slot < m) vout[to[k]] = s_val[slot];
    }
}

// The order of the triangles from pairs sorted on the key bits from lo up: a
// run of equal high bits is put in the order of its low bits (ties by
// position, so by original index), each thread counting the members of its run
// that come before its own.  A run of more than kTieRun sets flags[kFlagTies]
// and the build sorts on all bits instead.  A failed sort (*err) leaves the
// identity, so that nothing reads through an index that was never written.
constexpr int kTieRun = 128;
constexpr int kOrderTile = 1024;  // keys a CTA places, with kTieRun more on either side in shared memory

__global__ void __launch_bounds__(256) k_order(const unsigned long long* keys, const unsigned* vals, long long n,
                                               int lo, const unsigned* err, unsigned* order, unsigned* flags) {
    __shared__ unsigned long long s[kOrderTile + 2 * kTieRun];
    const long long base = (long long)blockIdx.x * kOrderTile;
    const bool failed = *err != 0u;
    if (lo > 0 && !failed) {
        for (int k = threadIdx.x; k < kOrderTile + 2 * kTieRun; k += 256) {
            const long long i = base - kTieRun + k;
            s[k] = i >= 0 && i < n ? keys[i] : ~0ull;  // (no key: they have 63 bits)
        }
        __syncthreads();
    }
#pragma unroll
    for (int h = 0; h < kOrderTile / 256; ++h) {
        const int k = h * 256 + (int)threadIdx.x;
        const long long i = base + k;
        if (i >= n) return;
        if (failed) {
            if (i == 0) flags[kFlagSort] = 1u;
            order[i] = (unsigned)i;
            continue;
        }
        const unsigned v = vals[i];
        long long to = i;
        if (lo > 0) {
            const unsigned long long key = s[kTieRun + k], top = key >> lo;
            int run = 1, d = 0;
            for (int j = kTieRun + k - 1; j >= 0 && s[j] >> lo == top && ++run <= kTieRun; --j) d -= s[j] > key;
            for (int j = kTieRun + k + 1; j < kOrderTile + 2 * kTieRun && s[j] >> lo == top && ++run <= kTieRun; ++j)
                d += s[j] < key;
            if (run > kTieRun) {
                flags[kFlagTies] = 1u;
                d = 0;
            }
            to += d;
        }
        order[to] = v;
    }
}

constexpr int kTreeLevels = 8;  // tree levels one CTA reduces (2^8 = 256 nodes in, one out)

// A run of shared memory to global memory by the bulk copy engine (one thread;
// both addresses multiples of 16, and the size).  The threads that wrote the
// run call bulk_ready before the barrier in front of it; the issuing thread
// calls bulk_done before it leaves.
__device__ __forceinline__ void bulk_ready() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                 "r"((unsigned)__cvta_generic_to_shared(src)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_done() {
    asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
}

// Subtree union shared by the two tree kernels: on entry hb holds the 2^levels
// boxes of the CTA's consecutive nodes of depth d (heap ids from first) at heap
// positions 2^levels .. 2^(levels+1)-1, six floats each; every step makes node k
// the union of its children 2k, 2k+1 (Section 4: tight children make a tight
// parent).  The rows of boxes (from row 0 up to row rows - 1) then go out, each
// a run of its own: 48 bytes times a whole number from an even node on, so the
// copy engine takes all but the first.  At the root (depth 0) the root box goes
// to root_out[0..5] and max |coordinate| to *P_out, when given.
__device__ __forceinline__ void reduce_subtree(float* hb, float* box, long long first, int levels, int rows,
                                               float* root_out, float* P_out) {
    const int tid = threadIdx.x;
    for (int lev = levels - 1; lev >= 0; --lev) {
        __syncthreads();
        for (int j = tid; j < (1 << lev); j += blockDim.x) {
            // children 2k, 2k+1 are twelve floats side by side
            const float4* l = reinterpret_cast<const float4*>(hb + 12 * ((1 << lev) + j));
            const float4 a = l[0], b = l[1], c = l[2];
            float2* o = reinterpret_cast<float2*>(hb + 6 * ((1 << lev) + j));
            o[0] = make_float2(fminf(a.x, b.z), fminf(a.y, b.w));
            o[1] = make_float2(fminf(a.z, c.x), fmaxf(a.w, c.y));
            o[2] = make_float2(fmaxf(b.x, c.z), fmaxf(b.y, c.w));
        }
    }
    bulk_ready();
    __syncthreads();
    const long long root = first >> levels;
    if (tid == 0) {
        for (int r = 1; r < rows; ++r) bulk_store(box + 6 * (root << r), hb + (6 << r), 24u << r);
        float P = 0.f;
        for (int c = 0; c < 6; ++c) {
            box[6 * root + c] = hb[6 + c];
            if (root == 1 && root_out) root_out[c] = hb[6 + c];
            P = fmaxf(P, fabsf(hb[6 + c]));
        }
        if (root == 1 && P_out) *P_out = P;
        bulk_done();
    }
}

// leaves: leaf l owns sorted triangles [floor(l T / 2^L), floor((l+1) T / 2^L)).
// 2^levels leaves and threads per CTA, whose triangles are one run: a thread
// gathers one or two of them (order[j] = original index of sorted triangle j)
// into shared memory, the records go out from there as one run, then a thread
// takes each leaf's exact box, and the CTA its subtree.  The build (stris_in
// == nullptr) reads each triangle's vertex indices through order and stores
// them in leaf order (stris_out); the refit of a deformed mesh reads them from
// there, contiguously, so its vertex gathers wait on one load instead of two
// dependent ones.
// bad != nullptr: a non-finite coordinate sets *bad (the refit's check; the
// build's validation has made its own).  skip != nullptr and *skip != 0: the
// build has met an index out of range and nothing is read through it.
// Bound: the stores (48 bytes a triangle, 24 a node), which the copy engine
// takes as runs.  A thread per leaf that stored its records and boxes itself
// wrote every 32-byte sector in two or three pieces; one update of 7.5 M
// triangles, copy and call included, took 204 us so, 212 with four CTAs an SM of
// this form (64 registers), 196 with six.
__global__ void __launch_bounds__(1 << kTreeLevels, 6)
    k_leaves(const float* verts, const int32_t* tris, long long nt, int L, const unsigned* order,
             const int32_t* stris_in, int32_t* stris_out, float4* tri, float* box, int levels, unsigned* bad,
             const unsigned* skip, float* root_out, float* P_out) {
    constexpr int kMost = 2 << kTreeLevels;  // triangles of 2^kTreeLevels leaves
    __shared__ float4 s_rec[3 * kMost];
    __shared__ __align__(16) float hb[6 * kMost];  // the vertex indices, then the boxes
    int* s_idx = reinterpret_cast<int*>(hb);
    if (skip && *skip) return;
    const int tid = threadIdx.x;
    const long long l0 = (long long)blockIdx.x << levels;  // the CTA's first leaf
    const long long j0 = (long long)(((unsigned long long)l0 * (unsigned long long)nt) >> L);
    const long long j1 = (long long)(((unsigned long long)(l0 + (1ll << levels)) * (unsigned long long)nt) >> L);
    const int m = (int)(j1 - j0);
    bool finite = true;
    // both of a thread's triangles at once: their gathers overlap
    unsigned id[2];
    int vi[2][3];
    float v[2][9];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = tid + h * (int)blockDim.x;
        if (i < m) id[h] = order[j0 + i];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = tid + h * (int)blockDim.x;
        if (i < m) {
            const int32_t* t = stris_in ? stris_in + 3 * (j0 + i) : tris + 3ll * id[h];
#pragma unroll
            for (int k = 0; k < 3; ++k) vi[h][k] = t[k];
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (tid + h * (int)blockDim.x < m)
#pragma unroll
            for (int k = 0; k < 3; ++k) load_vertex(verts, (unsigned)vi[h][k], v[h] + 3 * k);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = tid + h * (int)blockDim.x;
        if (i < m) {
#pragma unroll
            for (int k = 0; k < 9; ++k) finite = finite && isfinite(v[h][k]);
            s_rec[3 * i] = make_float4(v[h][0], v[h][1], v[h][2], v[h][3]);
            s_rec[3 * i + 1] = make_float4(v[h][4], v[h][5], v[h][6], v[h][7]);
            s_rec[3 * i + 2] = make_float4(v[h][8], __int_as_float((int)id[h]), 0.f, 0.f);
            if (stris_out) {
#pragma unroll
                for (int k = 0; k < 3; ++k) s_idx[3 * i + k] = vi[h][k];
            }
        }
    }
    bulk_ready();
    if (__syncthreads_or(!finite) && bad && tid == 0) atomicOr(bad, 1u);
    if (tid == 0) bulk_store(tri + 3 * j0, s_rec, 48u * (unsigned)m);
    if (stris_out) {
        for (int i = tid; i < 3 * m; i += blockDim.x) stris_out[3 * j0 + i] = s_idx[i];
        __syncthreads();
    }
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    {
        const long long l = l0 + tid;
        const int a = (int)((long long)(((unsigned long long)l * (unsigned long long)nt) >> L) - j0);
        const int b = (int)((long long)(((unsigned long long)(l + 1) * (unsigned long long)nt) >> L) - j0);
        for (int i = a; i < b; ++i) {
            const float4 p = s_rec[3 * i], q = s_rec[3 * i + 1];
            const float z = s_rec[3 * i + 2].x;
            lo[0] = fminf(lo[0], fminf(p.x, fminf(p.w, q.z)));
            lo[1] = fminf(lo[1], fminf(p.y, fminf(q.x, q.w)));
            lo[2] = fminf(lo[2], fminf(p.z, fminf(q.y, z)));
            hi[0] = fmaxf(hi[0], fmaxf(p.x, fmaxf(p.w, q.z)));
            hi[1] = fmaxf(hi[1], fmaxf(p.y, fmaxf(q.x, q.w)));
            hi[2] = fmaxf(hi[2], fmaxf(p.z, fmaxf(q.y, z)));
        }
    }
    float2* o = reinterpret_cast<float2*>(hb + 6 * ((1 << levels) + tid));
    o[0] = make_float2(lo[0], lo[1]);
    o[1] = make_float2(lo[2], hi[0]);
    o[2] = make_float2(hi[1], hi[2]);
    reduce_subtree(hb, box, (1ll << L) + l0, levels, levels + 1, root_out, P_out);
}

// levels above depth d: each CTA loads 2^levels consecutive nodes of depth d
// and reduces them (grid x block = 2^d exactly)
__global__ void __launch_bounds__(1 << kTreeLevels)
    k_reduce_up(float* box, int d, int levels, float* root_out, float* P_out) {
    __shared__ __align__(16) float hb[6 * (2 << kTreeLevels)];
    const long long first = (1ll << d) + ((long long)blockIdx.x << levels);
    for (int i = threadIdx.x; i < 6 << levels; i += blockDim.x) hb[(6 << levels) + i] = box[6 * first + i];
    reduce_subtree(hb, box, first, levels, levels, root_out, P_out);
}

// all boxes from the sorted order: leaves plus the lowest levels, then one
// launch per further kTreeLevels levels (three launches for 2^22 leaves)
void tree_boxes(const float* verts, const int32_t* tris, long long nt, int L, const unsigned* order,
                const int32_t* stris_in, int32_t* stris_out, float4* tri, float* box, unsigned* bad,
                const unsigned* skip, float* root_out, float* P_out, cudaStream_t st) {
    int lv = L < kTreeLevels ? L : kTreeLevels;
    k_leaves<<<(unsigned)(1ll << (L - lv)), 1u << lv, 0, st>>>(verts, tris, nt, L, order, stris_in, stris_out, tri, box,
                                                                 lv, bad, skip, root_out, P_out);
    for (int d = L - lv; d > 0; d -= lv) {
        lv = d < kTreeLevels ? d : kTreeLevels;
        k_reduce_up<<<(unsigned)(1ll << (d - lv)), 1u << lv, 0, st>>>(box, d, lv, root_out, P_out);
    }
}

// at most four CTAs an SM for the kernels that end in atomics on common words
int grid_for(long long n, int threads) {
    long long g = (n + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 152 * 4) g = 152 * 4;
    return (int)g;
}

}  // namespace

size_t sort_scratch_bytes(long long n) {
    const long long tile = kSortThreads * (n <= kSmallSort ? kItemsSmall : kItemsLarge);
    const size_t tiles = (size_t)((n + tile - 1) / tile);
    return 256 * sizeof(unsigned long long) * tiles + sizeof(unsigned) * (256 * kSortPasses + 64);
}

SortWork sort_scratch(void* p, long long n, unsigned long long timeout_ns) {
    const size_t words = (sort_scratch_bytes(n) - sizeof(unsigned) * (256 * kSortPasses + 64)) / sizeof(unsigned long long);
    SortWork w;
    w.status = static_cast<unsigned long long*>(p);
    w.hist = reinterpret_cast<unsigned*>(w.status + words);
    w.ticket = w.hist + 256 * kSortPasses;
    w.err = w.ticket + 32;
    w.timeout_ns = timeout_ns;
    return w;
}

cudaError_t build_validate(const BuildBuffers& b, cudaStream_t st) {
    k_init_flags<<<1, 32, 0, st>>>(b.flags);
    k_validate<<<grid_for(b.nt, 512), 512, 0, st>>>(b.verts, b.nv, b.tris, b.nt, b.flags);
    return cudaGetLastError();
}

cudaError_t sort_clear(const SortWork& w, long long n, cudaStream_t st) {
    return cudaMemsetAsync(w.status, 0, sort_scratch_bytes(n), st);
}

int radix_sort_pairs(const SortWork& w, unsigned long long* const keys[2], unsigned* const vals[2], long long n,
                     int lo_bit, int passes, cudaStream_t st) {
    const bool small = n <= kSmallSort;
    const long long tile = kSortThreads * (small ? kItemsSmall : kItemsLarge);
    const unsigned tiles = (unsigned)((n + tile - 1) / tile);
    auto pass = small ? k_sort_pass<kItemsSmall> : k_sort_pass<kItemsLarge>;
    int cur = 0;
    for (int p = 0; p < passes; ++p) {
        pass<<<tiles, kSortThreads, 0, st>>>(keys[cur], p ? vals[cur] : nullptr, keys[cur ^ 1], vals[cur ^ 1], n,
                                             lo_bit + 8 * p, p, w);
        cur ^= 1;
    }
    return cur;
}

// Passes of the build's sort.  The triangles of a surface fill about 2^(2 b / 3)
// cells of b key bits, so 1.5 log2 T bits leave a few triangles a cell, put in
// order afterwards (k_order): 5 passes instead of 8 for 7.5 M triangles (with 4
// the ties cost more than the pass), 4 for 2 M, 3 for 20,000.
int build_passes(long long nt, int morton_bits) {
    int lg = 0;
    while ((2ll << lg) <= nt) ++lg;
    const int all = (3 * morton_bits + 7) / 8;
    return std::min(all, std::max(2, (3 * (lg + 1) / 2 + 6) / 8));
}

cudaError_t build_tree(const BuildBuffers& b, bool all_bits, float* P_out, cudaStream_t st) {
    const int bits = 3 * b.morton_bits, all = (bits + 7) / 8;
    const int passes = all_bits ? all : build_passes(b.nt, b.morton_bits);
    const int lo = passes == all ? 0 : bits - 8 * passes;
    cudaError_t e = sort_clear(b.sort, b.nt, st);
    if (e != cudaSuccess) return e;
    k_morton<<<grid_for(b.nt, 512), 512, 0, st>>>(b.verts, b.tris, b.nt, b.flags, b.morton_bits, b.keys[0], lo, passes,
                                                  b.sort.hist);
    const int cur = radix_sort_pairs(b.sort, b.keys, b.vals, b.nt, lo, passes, st);
    k_order<<<(unsigned)((b.nt + kOrderTile - 1) / kOrderTile), 256, 0, st>>>(b.keys[cur], b.vals[cur], b.nt, lo, b.sort.err, b.order,
                                                             b.flags);
    tree_boxes(b.verts, b.tris, b.nt, b.L, b.order, nullptr, b.stris, b.tri, b.box, nullptr, b.flags,
               reinterpret_cast<float*>(b.flags + 8), P_out, st);
    return cudaGetLastError();
}

cudaError_t build_refit(const BuildBuffers& b, float* P_out, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(b.flags, 0, 16 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    tree_boxes(b.verts, b.tris, b.nt, b.L, b.order, b.stris, nullptr, b.tri, b.box, b.flags + 1,
               nullptr, reinterpret_cast<float*>(b.flags + 8), P_out, st);
    return cudaGetLastError();
}

}  // namespace gd
