// gwn_classify_static: gwn_classify without any device allocation.
//
// Some callers cannot allocate device memory on the call path: hosts that
// reserve their whole device-memory budget up front (a fixed pool, another
// framework's caching allocator owning the GPU), and latency-critical loops
// that must not enter the CUDA allocator, whose calls can take locks,
// synchronise or grow a memory pool.  gwn_classify obtains its scratch (the
// crossing numbers, the FP64 re-evaluation list and the boundary-sum partials)
// from the stream-ordered allocator on every call; this entry point instead
// uses one file-scope device array that every GPU loading the library holds
// until the process exits.
#include <algorithm>
#include <mutex>

#include "gwn_internal.cuh"

namespace {

constexpr size_t kScratchBytes = size_t(32) << 20;   // 32 MiB per device
constexpr int64_t kMaxQueries = int64_t(1) << 21;     // 2,097,152 queries per call
constexpr size_t kHeader = 256;                       // the re-evaluation counter, padded

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

std::mutex g_mu;
constexpr int kMaxDevices = 64;
void *g_addr[kMaxDevices] = {};

// Device address of g_scratch on the current device (looked up once per device;
// a host-side reference to g_scratch names a host stand-in, not device memory).
gwn_status scratch_address(int dev, unsigned char **out) {
    if (dev < 0 || dev >= kMaxDevices) return gwn::set_error(GWN_ERR_INVALID_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess)
            return gwn::set_error(GWN_ERR_CUDA, std::string("cudaGetSymbolAddress(static scratch): ") +
                                                    cudaGetErrorString(e));
        g_addr[dev] = p;
    }
    *out = static_cast<unsigned char *>(g_addr[dev]);
    return GWN_OK;
}


// Queries per slice of an ordered call, at most: an order over fewer than 2^20 queries has
// at most 64^3 cells.
constexpr int64_t kSlice = (int64_t(1) << 20) - 256;
// What a slice of n queries needs: 29.125 bytes a query and 1 MiB of cell counts (unordered
// 12.125), with 8 bytes a query and part of the boundary, as many parts as the whole call
// has on gwn_classify's path (so that w is the same to the bit), and the roundings.
int64_t slice_queries(bool ordered, int64_t parts) {
    const size_t bits = (ordered ? 29 * 8 : 12 * 8) + 1 + (parts > 1 ? 64 * (size_t)parts : 0);
    const size_t room = kScratchBytes - kHeader - 1024 - (ordered ? gwn::order_cells_bytes(kSlice) : 0);
    return std::min<int64_t>(kSlice, (int64_t)(room * 8 / bits));
}

// layout: [counter | chi n x int32 | list n x int32 | w n x float | listed (n + 31) / 32 x uint32 |
//          ordered: perm n x uint32 | queries n x 12 | label n | cell counts || FP64 partials ...]
// (the ranks of the order share the crossing numbers' place)
gwn_status run_slice(const gwn_mesh *m, const float *q, int64_t n, uint8_t *label, float *w, bool ordered, bool far,
                     int64_t call_n, int64_t parts, unsigned char *base, cudaStream_t s) {
    auto *len = reinterpret_cast<unsigned long long *>(base);
    auto *chi = reinterpret_cast<int32_t *>(base + kHeader);
    auto *list = chi + n;
    float *ws = reinterpret_cast<float *>(list + n);
    auto *listed = reinterpret_cast<unsigned *>(ws + n);
    const size_t words = (size_t)((n + 31) / 32);
    auto *perm = reinterpret_cast<uint32_t *>(listed + words);
    float *qs = reinterpret_cast<float *>(perm + n);
    auto *cells = reinterpret_cast<uint32_t *>(qs + 3 * n);
    uint8_t *ls = reinterpret_cast<uint8_t *>(cells) + (ordered ? gwn::order_cells_bytes(n) : 0);
    size_t used = ordered ? (size_t)(ls + n - base) : (size_t)(reinterpret_cast<unsigned char *>(perm) - base);
    used = (used + 255) & ~size_t(255);
    const size_t sums = parts > 1 ? sizeof(double) * (size_t)(parts * n) : 0;
    if (used + sums > kScratchBytes) return gwn::set_error(GWN_ERR_INVALID_ARG, "gwn_classify_static: slice beyond the scratch");
    double *partial = reinterpret_cast<double *>(base + used);
    GWN_CUDA_TRY(cudaMemsetAsync(len, 0, sizeof(unsigned long long), s));
    GWN_CUDA_TRY(cudaMemsetAsync(listed, 0, sizeof(unsigned) * words, s));
    if (!ordered)
        return gwn::launch_classify_on_scratch(m, q, n, label, w ? w : ws, chi, list, len, listed, partial, call_n,
                                               false, s);
    gwn_status st = gwn::order_queries_on(m, q, n, reinterpret_cast<uint32_t *>(chi), perm, qs, cells, s);
    if (st == GWN_OK)
        st = gwn::launch_classify_on_scratch(m, qs, n, ls, ws, chi, list, len, listed, partial, call_n, far, s);
    if (st == GWN_OK) st = gwn::scatter_results(perm, n, ws, w, nullptr, nullptr, ls, label, s);
    return st;
}

}  // namespace

extern "C" gwn_status gwn_classify_static(const gwn_mesh *m, const float *q, int64_t n, uint8_t *label,
                                          float *w_or_null, void *stream) {
    gwn::clear_error();
    if (!m) return gwn::set_error(GWN_ERR_INVALID_ARG, "mesh is NULL");
    if (n < 0) return gwn::set_error(GWN_ERR_INVALID_ARG, "negative query count");
    if (n > kMaxQueries)
        return gwn::set_error(GWN_ERR_INVALID_ARG,
                              "gwn_classify_static: n = " + std::to_string(n) +
                                  " exceeds the static scratch limit of 2097152 queries per call");
    if (!m->built) return gwn::set_error(GWN_ERR_NOT_BUILT, "call gwn_build_accel first");
    if (n == 0) return GWN_OK;
    if (!q || !label) return gwn::set_error(GWN_ERR_INVALID_ARG, "q or label is NULL");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != m->device) cudaSetDevice(m->device);
    gwn_status st = GWN_OK;
    const int kq = gwn::pointer_kind(q, m->device), kl = gwn::pointer_kind(label, m->device),
              kw = gwn::pointer_kind(w_or_null, m->device);
    if (kq < 0 || kl < 0 || kw < 0) {
        st = gwn::set_error(GWN_ERR_INVALID_ARG, "gwn_classify_static: a buffer is device memory of another GPU "
                                                 "than the mesh's");
    } else if (kq == 0 || kl == 0 || kw == 0) {
        st = gwn::set_error(GWN_ERR_INVALID_ARG,
                            "gwn_classify_static takes device pointers only (host buffers would need staging)");
    } else {
        unsigned char *base = nullptr;
        st = scratch_address(m->device, &base);
        if (st == GWN_OK && gwn::small_call(m, n)) {
            st = gwn::launch_small(m, q, n, w_or_null, nullptr, label, (cudaStream_t)stream);
        } else if (st == GWN_OK) {
            cudaStream_t s = (cudaStream_t)stream;
            // Large calls run in spatial order like gwn_classify's, in slices that fit the
            // scratch (an order over the slice serves as well); small ones as they come.
            const bool ordered = n >= gwn::kOrderMinQueries, far = ordered && gwn::far_pays(m, n);
            const int64_t parts = gwn::boundary_parts(m, n, far), most = slice_queries(ordered, parts);
            const int64_t slices = (n + most - 1) / most, slice = (n + slices - 1) / slices;
            for (int64_t at = 0; at < n && st == GWN_OK; at += slice)
                st = run_slice(m, q + 3 * at, std::min<int64_t>(slice, n - at), label + at,
                               w_or_null ? w_or_null + at : nullptr, ordered, far, n, parts, base, s);
        }
    }
    if (prev >= 0 && prev != m->device) cudaSetDevice(prev);
    return st;
}
