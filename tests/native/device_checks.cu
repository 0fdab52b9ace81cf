// Device code of the engine called beneath its C ABI, for the tests of what the
// ABI cannot reach.  Compiled by the tests together with the sources it calls.
#include <cuda_runtime.h>

#include <chrono>
#include <vector>

#include "gd_launch.h"

#define EXPORT extern "C" __attribute__((visibility("default")))

namespace {
struct Buffer {
    void* p = nullptr;
    explicit Buffer(size_t bytes) { cudaMalloc(&p, bytes); }
    ~Buffer() { cudaFree(p); }
};
}  // namespace

// A sort of n keys (the caller's; n and n + 4096 on one side of 2^18) whose first
// tile is never taken, so that every other tile of the first pass waits for it
// until the wait gives up, after timeout_ns.  The buffers lie as the engine's do,
// keys, values and scratch in one allocation with guard words behind it.  *ms: how
// long the sort took.  Returns 0, or 1 a CUDA error, 2 no error word, 3 the input changed, 4 an output was written,
// 5 a guard word was written.
EXPORT int check_sort_gives_up(const unsigned long long* host, long long n, int passes, unsigned long long timeout_ns,
                               double* ms) {
    using namespace gd;
    constexpr unsigned long long kMark = 0x5aa5c33c5aa5c33cull;
    // (tile numbers run from 1 on: room in the look-back table for one tile more)
    const size_t k = (8 * (size_t)n + 255) / 256 * 256, v = (4 * (size_t)n + 255) / 256 * 256;
    const size_t scratch = (sort_scratch_bytes(n + 4096) + 255) / 256 * 256, guard = 16 * (size_t)n + (1u << 20);
    const size_t total = 2 * (k + v) + scratch + guard;
    Buffer mem(total);
    if (!mem.p) return 1;
    std::vector<unsigned long long> all(total / 8, kMark);
    cudaMemcpy(mem.p, all.data(), total, cudaMemcpyHostToDevice);
    char* base = static_cast<char*>(mem.p);
    unsigned long long* const keys[2] = {reinterpret_cast<unsigned long long*>(base),
                                         reinterpret_cast<unsigned long long*>(base + k)};
    unsigned* const vals[2] = {reinterpret_cast<unsigned*>(base + 2 * k), reinterpret_cast<unsigned*>(base + 2 * k + v)};
    const SortWork w = sort_scratch(base + 2 * (k + v), n + 4096, timeout_ns);
    if (sort_clear(w, n + 4096, nullptr) != cudaSuccess) return 1;
    std::vector<unsigned> hist(256 * passes, 0u);
    for (long long i = 0; i < n; ++i)
        for (int p = 0; p < passes; ++p) ++hist[256 * p + ((host[i] >> (8 * p)) & 255u)];
    const unsigned one = 1u;
    cudaMemcpy(keys[0], host, 8 * (size_t)n, cudaMemcpyHostToDevice);
    cudaMemcpy(w.hist, hist.data(), sizeof(unsigned) * hist.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(w.ticket, &one, sizeof(one), cudaMemcpyHostToDevice);
    cudaDeviceSynchronize();
    const auto t0 = std::chrono::steady_clock::now();
    radix_sort_pairs(w, keys, vals, n, 0, passes, nullptr);
    cudaDeviceSynchronize();
    *ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    unsigned err = 0;
    cudaMemcpy(&err, w.err, sizeof(err), cudaMemcpyDeviceToHost);
    cudaMemcpy(all.data(), mem.p, total, cudaMemcpyDeviceToHost);
    if (cudaGetLastError() != cudaSuccess) return 1;
    if (!err) return 2;
    for (long long i = 0; i < n; ++i)
        if (all[i] != host[i]) return 3;
    for (size_t i = k / 8; i < 2 * (k + v) / 8; ++i)
        if (all[i] != kMark) return 4;
    for (size_t i = (total - guard) / 8; i < total / 8; ++i)
        if (all[i] != kMark) return 5;
    return 0;
}

// Point queries on a mesh, twice over with the same room for shared walks: out
// (2 n records) and the counters of the second call.  Returns 0, or 1 on an error.
EXPORT int check_points(const float* verts, long long nv, const int32_t* tris, long long nt, const double* points,
                        long long n, gd_point_result* out, unsigned long long* slots, unsigned long long* gifts,
                        unsigned long long* parts) {
    using namespace gd;
    int L = 0;
    while ((2ll << L) <= nt) ++L;
    Buffer v(12 * (size_t)nv), t(12 * (size_t)nt), box(24 * (2ull << L)), tri(48 * (size_t)nt), order(4 * (size_t)nt),
        stris(12 * (size_t)nt), flags(64), P(4), k0(8 * (size_t)nt), k1(8 * (size_t)nt), v0(4 * (size_t)nt),
        v1(4 * (size_t)nt), scratch(sort_scratch_bytes(nt)), pts(24 * (size_t)n), res(sizeof(gd_point_result) * n),
        ws(8 * kPointWords), share(kPointShareBytes);
    cudaMemcpy(v.p, verts, 12 * (size_t)nv, cudaMemcpyHostToDevice);
    cudaMemcpy(t.p, tris, 12 * (size_t)nt, cudaMemcpyHostToDevice);
    cudaMemcpy(pts.p, points, 24 * (size_t)n, cudaMemcpyHostToDevice);
    cudaMemset(share.p, 0, kPointShareBytes);
    BuildBuffers b{};
    b.verts = static_cast<float*>(v.p); b.tris = static_cast<int32_t*>(t.p); b.nv = nv; b.nt = nt; b.L = L;
    b.morton_bits = 21;
    b.box = static_cast<float*>(box.p); b.tri = static_cast<float4*>(tri.p);
    b.order = static_cast<unsigned*>(order.p); b.stris = static_cast<int32_t*>(stris.p);
    b.flags = static_cast<unsigned*>(flags.p);
    b.keys[0] = static_cast<unsigned long long*>(k0.p); b.keys[1] = static_cast<unsigned long long*>(k1.p);
    b.vals[0] = static_cast<unsigned*>(v0.p); b.vals[1] = static_cast<unsigned*>(v1.p);
    b.sort = sort_scratch(scratch.p, nt, 2000000000ull);
    if (build_validate(b, nullptr) != cudaSuccess || build_tree(b, true, static_cast<float*>(P.p), nullptr) != cudaSuccess)
        return 1;
    PointArgs g{};
    g.box = b.box; g.tri = b.tri; g.T = nt; g.L = L;
    g.x[0] = g.x[5] = g.x[10] = 1.0;
    g.pts = static_cast<double*>(pts.p);
    g.n = n;
    g.out = static_cast<gd_point_result*>(res.p);
    g.ws = static_cast<unsigned long long*>(ws.p);
    g.timeout_ns = 2000000000ll;
    g.shares = static_cast<PointShare*>(share.p);
    g.parts = reinterpret_cast<PointPart*>(g.shares + kPointMaxShares);
    g.slots = reinterpret_cast<PointSlot*>(g.parts + kPointMaxSlots + kPointMaxShares);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    unsigned long long w[kPointWords];
    for (unsigned call = 0; call < 2; ++call) {
        g.epoch = call + 1;
        cudaMemset(res.p, 0xff, sizeof(gd_point_result) * n);
        if (launch_point(g, sms, nullptr) != cudaSuccess) return 1;
        cudaMemcpy(out + call * n, res.p, sizeof(gd_point_result) * n, cudaMemcpyDeviceToHost);
        cudaMemcpy(w, ws.p, sizeof(w), cudaMemcpyDeviceToHost);
        if (w[kPointTimeout] || w[kPointAnswered] != (unsigned long long)n) return 1;
    }
    *slots = w[kPointSlots];
    *gifts = w[kPointTail];
    *parts = w[kPointParts];
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

// Blocks of device memory filled with a byte, to lie where the engine has freed
// some, and whether they still hold it.
EXPORT void* check_block(size_t bytes, int value) {
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) return nullptr;
    cudaMemset(p, value, bytes);
    return p;
}

// 1: unchanged, 0: changed, -1: a CUDA error; frees it
EXPORT int check_block_kept(void* p, size_t bytes, int value) {
    std::vector<unsigned char> h(bytes);
    cudaDeviceSynchronize();
    if (cudaMemcpy(h.data(), p, bytes, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    cudaFree(p);
    for (unsigned char c : h)
        if (c != (unsigned char)value) return 0;
    return 1;
}
