// rewl_host_internal.hpp -- host-side instance record shared by the
// single-instance driver (rewl_host.cu) and the batch engine (rewl_batch.cu).
#pragma once
#include <sys/mman.h>
#include <unistd.h>

#include <cstdint>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "rewl.h"
#include "rewl_internal.cuh"

// Every entry point of the C ABI returns a status and lets no C++ exception
// (a failed host allocation inside a standard container) cross the ABI.
#define REWL_API_TRY try {
#define REWL_API_CATCH                                                                     \
    }                                                                                      \
    catch (const std::bad_alloc &) {                                                       \
        return rewl::host::fail(REWL_ERR_NOMEM, "host memory exhausted");                  \
    }                                                                                      \
    catch (...) {                                                                          \
        return rewl::host::fail(REWL_ERR_STATE, "unexpected host error");                 \
    }

namespace rewl {
namespace host {

// Device memory of a handle, a batch or a server: from the allocator set with
// rewl_set_allocator (else cudaMalloc), returned through the matching free.
struct DevBlock {
    void *ptr = nullptr;
    bool hooked = false;                              // false: cudaMalloc / cudaFree
    void (*free_fn)(void *ptr, void *ctx) = nullptr;  // hooked: nullptr means kept by the allocator
    void *ctx = nullptr;
};
// cudaSuccess, or cudaErrorMemoryAllocation (also for memory not 256-byte aligned).
cudaError_t dev_alloc(DevBlock &b, size_t bytes);
void dev_free(DevBlock &b);
void set_allocator(void *(*alloc)(size_t, void *), void (*free_fn)(void *, void *), void *ctx);

// Fault in every page of [p, p + bytes) for writing, the contents as they are.
// (By the kernel: to read a fresh page and write it back maps the zero page first
// and keeps huge pages away, 189 MB 9 -> 70 ms; a plain write loses the contents.)
// Above 4 MB not if the pages at the quarters are there already: a buffer in use,
// 9 MB read in 63 us instead of 66 for the walk over its pages.  (Smaller buffers
// from a heap are often there in part, and the walk costs under a microsecond.)
inline void fault_in(void *p, size_t bytes) {
#ifndef MADV_POPULATE_WRITE
    constexpr int MADV_POPULATE_WRITE = 23;  // Linux 5.14
#endif
    static const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    if (bytes == 0) return;
    const uintptr_t at = (uintptr_t)p;
    bool there = bytes >= (size_t)(4 << 20);
    for (int i = 1; i <= 3 && there; ++i) {
        unsigned char v = 0;
        there = mincore((void *)((at + bytes / 4 * i) & ~(page - 1)), 1, &v) == 0 && (v & 1);
    }
    if (there) return;
    const uintptr_t from = at & ~(page - 1), to = (at + bytes + page - 1) & ~(page - 1);
    (void)madvise((void *)from, to - from, MADV_POPULATE_WRITE);  // (refused: left to the copy)
}

// Fault in a caller's result buffer that a copy from the device is about to fill.
// Fresh pageable memory that the device reaches through the host's page tables is
// otherwise faulted in by the copy, one page at a time.  Fresh 64 KB pages, left to
// the copy -> faulted in: 330 KB 164 -> 57 us, 1.3 MB 216 -> 97, 9 MB 520 -> 405,
// 60 MB 3.6 -> 2.7 ms; in use already: 330 KB 15 -> 16 us, 9 MB 61 -> 63.
// Only pageable host memory: any other pointer is left to the copy, which takes
// or refuses it.
inline void touch_pages(void *p, size_t bytes) {
    if (bytes < (size_t)(256 << 10)) return;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    if (a.type == cudaMemoryTypeUnregistered) fault_in(p, bytes);
}

// A named range on the host timeline of a profiler (NVTX; free when none is attached).
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
    Range(const Range &) = delete;
    Range &operator=(const Range &) = delete;
};
}  // namespace host
}  // namespace rewl

struct rewl_s {
    rewl_params prm{};
    rewl::Model M{};
    rewl::State S{};
    rewl::SweepPlan plan{};
    int device = 0;
    cudaStream_t own_stream = nullptr;
    cudaStream_t stream = nullptr;
    void *dmem = nullptr;  // base of this instance's device arrays
    rewl::host::DevBlock dblock;  // the allocation behind dmem (stand-alone handles)
    size_t dbytes = 0;
    rewl::Ctl *h_ctl = nullptr;  // pinned mirror of the device control block
    std::vector<int32_t> e_lo;
    cudaGraphExec_t graph = nullptr;
    int sms = 0, smem_optin = 0;
    int lat_mode = 0;  // REWL_OPT_LATTICE: 0 by size, 1 global memory, 2 shared memory
    long long stall_ms = 0;  // REWL_OPT_STALL_MS: rewl_run gives up after this long without progress
    // byte offsets of the state arrays relative to dmem (for save / load); the
    // last part is the control block
    struct Part { size_t off, bytes; };
    std::vector<Part> parts;
    // false for an instance that lives inside a batch: the batch owns its
    // memory, stream and pinned status block, and runs its rounds
    bool owns = true;
    // fixed-weight production (rewl_production_start): H(E, O) and spin counts
    rewl::host::DevBlock prod_block;
};

namespace rewl {
namespace host {


// Checks the parameters, computes the window table and the sizes of the device
// arrays (h->parts, h->dbytes) and plans the sweep.  lanes: lanes per walker of
// the fast sweep (0 = from the walker count).  spin_capacity_bits (0 = the
// packing chosen): the configuration buffers are sized for this packing, so
// that a batch can repack its spins in place.  No device memory is touched.
rewl_status prepare_instance(rewl_s *h, const rewl_params &p, int spin_bits, int lanes, int spin_capacity_bits = 0);
// Points h->S at the arrays of a region of h->dbytes bytes at `base`.
void carve_instance(rewl_s *h, void *base);
// Queues zeroing, the window table, ln f = 1 and the initial configurations.
cudaError_t init_instance_async(rewl_s *h, cudaStream_t s);
// Reads the control block (synchronises h->stream) and maps its error bits.
rewl_status read_status(rewl_s *h);
rewl_status fail(rewl_status st, const char *fmt, ...);
// Joins h window pieces (lw, mw: h x (W + 1), window-major) into out[2N + 1]
// (Sec. 2, Fig. 2): each neighbouring pair meets at the bin of their overlap
// where the pieces' slopes d ln g / dE differ least; -inf where no window
// visited a bin.  REWL_ERR_STATE when a pair has no usable bin.
rewl_status join_windows(int N, int W, const std::vector<int32_t> &e_lo, const std::vector<double> &lw,
                         const std::vector<uint8_t> &mw, double *out);
// Shifts the finite entries of v[nb] so that sum g = q^N.
void normalise_total(int q, int N, double *v, int nb);

}  // namespace host
}  // namespace rewl
