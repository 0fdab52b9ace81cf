// Host-side entry points of the engine's kernels (shared by the C ABI file).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "gd_internal.cuh"

namespace gd {

// ---- BVH build (gd_build.cu)
constexpr int kSortPasses = 8;  // 64-bit keys, 8 bits a pass
constexpr int kFlagTies = 14, kFlagSort = 15;

struct SortWork {
    unsigned long long* status;  // look-back table, 256 words a tile
    unsigned* hist;              // digit counts, 256 a pass
    unsigned* ticket;            // next tile of each pass
    unsigned* err;               // a wait gave up
    unsigned long long timeout_ns;  // a tile's longest wait for one before it
};

struct BuildBuffers {
    const float* verts;   // nv x 3, device
    const int32_t* tris;  // nt x 3, device
    long long nv, nt;
    int L;
    int morton_bits;
    float* box;           // 6 * 2^(L+1) floats, device
    float4* tri;          // 3 * nt float4, device
    unsigned* order;      // nt, device: original index of each sorted triangle (kept for refits)
    int32_t* stris;       // nt x 3, device: the sorted triangles' vertex indices (written by the
                          // build, read by refits; may be nullptr for a build that keeps none)
    unsigned* flags;      // device, 16 words: [0] bad index, [1] non-finite vertex, [2..7] bounds of the
                          // vertices, [8..13] the root box, [kFlagTies] more equal keys than the shortened
                          // sort can order, [kFlagSort] a wait of the sort gave up
    unsigned long long* keys[2];  // nt each, device
    unsigned* vals[2];            // nt each, device
    SortWork sort;
};

// Stable LSD radix sort of n (key, value) pairs on the 8 passes key bits from
// lo_bit up; the keys start in keys[0], their values are 0, 1, 2, ...; returns
// the index of the buffers that hold the sorted pairs.  Before it, sort_clear,
// then a kernel that adds the keys' digits to w.hist (256 words a pass).
// scratch: sort_scratch_bytes(n) bytes, 8-byte aligned.  A bounded wait that gave
// up sets *w.err (device): the pass leaves the rest of its output as it was, the
// passes after it do nothing, and nothing outside the buffers is written.
size_t sort_scratch_bytes(long long n);
SortWork sort_scratch(void* p, long long n, unsigned long long timeout_ns);
cudaError_t sort_clear(const SortWork& w, long long n, cudaStream_t stream);
int radix_sort_pairs(const SortWork& w, unsigned long long* const keys[2], unsigned* const vals[2], long long n,
                     int lo_bit, int passes, cudaStream_t stream);
// checks indices and finiteness, and bounds the referenced vertices (flags)
cudaError_t build_validate(const BuildBuffers& b, cudaStream_t stream);
// the rest of the build, after build_validate (its kernels read nothing through
// an index that is out of range).  The sort takes as many key bits as the
// triangle count calls for; flags[kFlagTies] != 0 afterwards: too many triangles
// share those, build again with all_bits.  *P_out: max |coordinate| of the root box
cudaError_t build_tree(const BuildBuffers& b, bool all_bits, float* P_out, cudaStream_t stream);
// refit of a built tree after its vertices moved (verts, tris, L, order, tri,
// box, flags): stored triangles and leaf boxes from the new vertices, then the
// unions up to the root.  flags[1] != 0 afterwards: a referenced coordinate is
// not finite; flags[8..13]: the root box (float bits); *P_out (device, may be
// null): max |coordinate| of the root box.
cudaError_t build_refit(const BuildBuffers& b, float* P_out, cudaStream_t stream);

// ---- naive comparator (gd_naive.cu)
// words of its device scratch (uint64 each)
enum : int {
    kNaiveU = 0,         // running bound: float bits of a squared distance (low 32 bits)
    kNaiveTests = 1,     // node boxes tested
    kNaiveLeaves = 2,    // triangle pairs evaluated
    kNaiveMaxTests = 3,  // most boxes tested by one thread
    kNaiveT0 = 4,        // globaltimer stamp of the first thread to start
    kNaiveTimeout = 5,   // some thread passed the deadline and stopped
    kNaiveBad = 6,       // a walk outgrew its stack (never, for at most 31 levels)
    kNaiveWords = 8,
};

struct NaiveArgs {
    const float4* triA;   // A's triangles in leaf order
    long long TA;
    const float* boxB;    // B's tree
    const float4* triB;
    long long TB;
    int LB;
    float R[9], t[3];     // A-local -> B-local, float32
    float E;              // widening of each mapped triangle's box
    unsigned long long* ws;
    long long timeout_ns;
};

cudaError_t launch_naive(int kind, const NaiveArgs& g, cudaStream_t stream);

// ---- point-to-mesh queries (gd_point.cu)
enum : int {
    kPointTests = 0,     // node boxes tested
    kPointExact = 1,     // float64 point-triangle distances
    kPointT0 = 2,        // globaltimer stamp of the first CTA to start
    kPointTimeout = 3,   // some point passed the deadline
    kPointSlots = 4,     // points whose walk is shared
    kPointParts = 5,     // answers of parts of shared walks
    // (words that all warps use, a 128-byte line each)
    kPointTicket = 16,   // points handed out to warps
    kPointHead = 32,     // gifts claimed by idle warps
    kPointTail = 48,     // gifts made
    kPointAnswered = 64, // points answered
    kPointWords = 80,
};

// Shared walks: a warp with a long walk gives parts of its stack to idle
// warps.  Fixed room, reused by every call; when it is full walks are no longer
// divided.  (The tests compile it with little room too.)
#ifndef GD_POINT_SLOTS
#define GD_POINT_SLOTS (1u << 14)
#define GD_POINT_SHARES (1u << 16)
#endif
constexpr unsigned kPointMaxSlots = GD_POINT_SLOTS;    // points with a shared walk
constexpr unsigned kPointMaxShares = GD_POINT_SHARES;  // gifts

struct PointSlot {
    unsigned U;       // least upper bound of all parts (float bits, squared)
    unsigned parts;   // parts still running
    unsigned chain;   // latest answer of a part (index into parts, kNone: none)
    unsigned i;       // the point
    unsigned failed;  // a part ran into the deadline
};

struct PointShare {
    unsigned ready;   // the call's epoch once the gift is complete
    unsigned slot, n, pad;
    unsigned node[32];
};

constexpr unsigned kPartCands = 6;

struct PointPart {
    unsigned n, next;
    unsigned tri[kPartCands];
    float low[kPartCands];
};

constexpr size_t kPointShareBytes = sizeof(PointShare) * kPointMaxShares + sizeof(PointSlot) * kPointMaxSlots +
                                    sizeof(PointPart) * (kPointMaxSlots + kPointMaxShares);

struct PointArgs {
    const float* box;     // the mesh's tree
    const float4* tri;
    long long T;
    int L;
    double x[12];         // mesh local -> world
    const double* pts;    // n x 3 world points, device
    long long n;
    gd_point_result* out; // n results, device
    const unsigned* order;// order of work: the i-th point taken is order[i] (nullptr: point i)
    const unsigned* order_err;  // device: != 0, order was not written (used with order)
    unsigned long long* ws;
    long long timeout_ns;
    unsigned epoch;       // differs from call to call
    unsigned share_steps; // steps of a walk before it gives any of it away (set by launch_point),
    unsigned share_mask;  //   looks for idle warps in steps whose low bits these are zero
    PointShare* shares;   // kPointMaxShares
    PointSlot* slots;     // kPointMaxSlots
    PointPart* parts;     // kPointMaxSlots + kPointMaxShares
};

// order the points along a Morton curve in the mesh's frame so that nearby
// points are walked at the same time: the indices end in vals[returned index]
int sort_points(const PointArgs& g, const SortWork& w, unsigned long long* const keys[2], unsigned* const vals[2],
                cudaStream_t stream);
// sms: the device's SM count
cudaError_t launch_point(PointArgs g, int sms, cudaStream_t stream);

// ---- query (gd_query.cu)
// co-resident CTAs per SM of the query kernel's single-query or batch launch
int query_max_blocks_per_sm(int kind, bool batch = false);
cudaError_t launch_query(int kind, const KArgs& args, int grid, cudaStream_t stream);
// *best (device): the page of the zeroed buffer that CTA 0's atomics reach soonest
cudaError_t launch_near_page(unsigned* base, int pages, unsigned words, unsigned* best, int grid, cudaStream_t stream);
cudaError_t build_query_graph(int kind, const KArgs& args, int grid, cudaGraphExec_t* exec);

}  // namespace gd
