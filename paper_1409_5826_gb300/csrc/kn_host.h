// kn_host.h -- host-side pieces shared by the runtime's translation units:
// error reporting, the device-buffer helper, a network's host and device
// state, and the table builder's entry points.
#pragma once

#include <cstdarg>
#include <cstdint>
#include <map>
#include <memory>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/kn.h"
#include "kn_internal.h"

namespace kn {
// Record a formatted message for kn_last_error and return s.
kn_status fail(kn_status s, const char* fmt, ...);
const char* last_error();

inline int pad16(int x) { return (x + 15) & ~15; }

// a device buffer that grows on demand
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    ~DevBuf() { release(); }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    cudaError_t ensure(size_t b) {
        if (b <= bytes && p) return cudaSuccess;
        release();
        cudaError_t e = cudaMalloc(&p, b ? b : 16);
        if (e == cudaSuccess) bytes = b;
        return e;
    }
    // Grow to b bytes and copy them from pageable host memory.  Such a copy may return
    // with its last part still on the way, ordered before later work on streams that
    // follow the default stream only; after upload_wait it is there for every stream.
    cudaError_t upload(const void* src, size_t b) {
        const cudaError_t e = ensure(b);
        return e == cudaSuccess ? cudaMemcpy(p, src, b, cudaMemcpyHostToDevice) : e;
    }
    static cudaError_t upload_wait() { return cudaStreamSynchronize(cudaStreamLegacy); }
    template <class T> T* as() const { return (T*)p; }
};

// The gather's summation order: the slices of 32 lanes, each lane's terms in order.
struct GatherOrder {
    struct Slice {
        int len = 0;                  // terms per lane
        std::vector<int> row;         // [32] the lane's row (F+_i: i, k_i: N + i; -1: no row)
        std::vector<uint16_t> terms;  // [len][32] indices into V
    };
    std::vector<Slice> slices;
};

// one of an order's slot tables; blob points into Tables::slot_blob
struct SlotBlob {
    const unsigned char* blob = nullptr;
    SlotTables st{};
    bool fits = false;
};

struct Tables {
    const unsigned char* dev = nullptr;              // in one of kn_network::table_mem
    TableLayout tl{};
    GatherOrder order;                               // mixed form
    std::vector<int> banks;                          // kn_slots.cu: V's values' banks, found on first use
    std::map<std::pair<int, int>, SlotBlob> slots;   // (threads, 8 zones per group + capacities) -> table
    std::unique_ptr<DevBuf> slot_blob;
    bool slots_built = false;
    int L = 0, n_slices = 0, warp_len = 0;  // piece cap, slices, longest warp's terms per lane
};
}  // namespace kn

#define KN_CUDA(call)                                                                      \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess)                                                             \
            return kn::fail(e_ == cudaErrorMemoryAllocation ? KN_ERR_NOMEM : KN_ERR_CUDA,  \
                            "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

struct kn_network {
    int N = 0, R = 0, S_r = 0, S_p = 0;
    std::vector<double> A, lnk0, tn;
    std::vector<int> reac, prod, nr, slot0;  // in the caller's reaction order
    std::vector<int> perm;                   // sorted position -> caller's reaction index
    int R1 = 0, R12 = 0;                     // 1-body reactions [0,R1), 2-body [R1,R12)
    double cmax = 0;
    kn::DevBuf rate0;                            // double2[R] (ln k0, n), sorted order
    double nbar = 0, rbar = 0;
    std::map<std::pair<int, int>, kn::Tables> tables;  // (precision, Q) -> table
    std::vector<std::unique_ptr<kn::DevBuf>> table_mem;
    // zone state
    int Z = 0, capZ = 0;
    kn::DevBuf Y, T0, rho0, tau, ts, te, dtt, tout, dtn, steps, rej, props, status, energy;
    kn::DevBuf bind;            // [N] binding energies, when set
    bool has_bind = false;
    kn::DevBuf key_in, key_out, idx_in, order, cub_tmp, qhead;
    bool has_const = true;  // conservative until zones are known
    bool zones_set = false;
    int trial_Z = 0;        // > 0 during autotune trials: integrate only the first trial_Z zones of the queue
    int tuned_P[3][3] = {};  // [precision][plain, learned, QSS]: autotuned CTA size
    int tuned_G[3][3] = {};  // ... and zone group size
    kn_launch_info launched = {-1, 0, 0, 0, 0, 0};  // the last kn_integrate_batch (kernel < 0: none yet)
};

namespace kn {
// kn_tables.cu: validation and the sorted reaction order (no device work), and
// one network's tables for (precision, threads per zone group), built and
// checked on the host; `blob` is what goes to the device.
kn_status network_host_setup(const kn_network_desc* d, std::unique_ptr<kn_network>& n, std::vector<double>& r0);
kn_status build_tables_host(const kn_network* n, int prec, int Q, std::vector<unsigned char>& blob, Tables& T);
// The slot tables (kn_slots.cu) for groups of T threads and NZ zones with the
// capacities kSlotCaps[cap], from the summation order of `tb`; checked on the host
// like the tables.  fits = false: the network does not fit the capacities or the
// 16-bit offsets.
kn_status build_slots_host(const kn_network* n, Tables& tb, int T, int NZ, int cap, std::vector<unsigned char>& blob,
                           SlotTables& st, bool& fits);
// kn_slots.cu: the threads of a group when a CTA holds ng of them, and the fewest that a
// group needs: the species' warps and the one that decides.  One warp if the order is.
constexpr int kMaxSlotGroups = 3;
inline int slot_threads(bool warp, int ng) { return warp ? 32 : kSlotThreads / ng / 32 * 32; }
inline int slot_min_threads(const kn_network* n, bool warp) { return warp ? 32 : (n->N + 31) / 32 * 32 + 32; }
SlotLayout slot_layout(const kn_network* n, const SlotTables& st, int T, int NZ, bool qss);
}  // namespace kn
