// sw_dslash_schur_noalloc: the Schur operator of sw_dslash (SW_OP_S) for
// callers that must not allocate device memory -- for instance a host
// application or framework that owns every device allocation and forbids
// others, or a real-time loop that may not call into the allocator.
// sw_dslash allocates its work buffers and the B^-1 table on first use; this
// entry point instead keeps all of its scratch in one file-scope device array
// of fixed size.
//
// Scratch layout for N = L0 L1 <= kNoAllocMaxSites (complex128 units):
//   [0, N)      copy of an input that overlaps the output
//   [N, 2N)     intermediate vector of the Schur operator
//   [2N, 6N)    B^-1 table for the requested mass (rebuilt every call)
#include <cmath>
#include <mutex>
#include <string>

#include "sw_internal.h"

namespace {

constexpr long kNoAllocMaxSites = 65536;  // e.g. 256 x 256; 6.3 MB of device memory
static __device__ __align__(256) double2 g_noalloc_scratch[6 * kNoAllocMaxSites];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double2* g_noalloc_ptr[kMaxDevices] = {nullptr};

// Device address of the scratch array on the current device (looked up once
// per device; the name g_noalloc_scratch is only a host-side stand-in).
double2* noalloc_scratch(int device) {
  SW_REQUIRE(device >= 0 && device < kMaxDevices, SW_ERR_ARG, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[device]) {
    void* p = nullptr;
    SW_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    g_noalloc_ptr[device] = (double2*)p;
  }
  return g_noalloc_ptr[device];
}

}  // namespace

extern "C" int sw_dslash_schur_noalloc(sw_gauge* g, double mass, const void* in, void* out) {
  if (!g || !in || !out) return SW_ERR_ARG;
  sw_ctx* c = g->ctx;
  return guarded(c, [&] {
    SW_REQUIRE((long)g->N <= kNoAllocMaxSites, SW_ERR_SHAPE,
               "sw_dslash_schur_noalloc: lattice has " + std::to_string(g->N) +
                   " sites, the fixed scratch holds at most " +
                   std::to_string(kNoAllocMaxSites));
    SW_REQUIRE(std::isfinite(mass) && mass > 0.0, SW_ERR_ARG, "mass must be > 0");
    cudaStream_t s = c->stream;
    long N = g->N;
    double2* base = noalloc_scratch(c->device);
    double2* w = base + N;
    double2* binv = base + 2 * N;
    launch_binv_build(g, mass, binv, s);
    const double2* x = (const double2*)in;
    double2* y = (double2*)out;
    if (x < y + N && y < x + N) {
      SW_CUDA(cudaMemcpyAsync(base, x, N * sizeof(double2), cudaMemcpyDeviceToDevice, s));
      x = base;
    }
    fine_lex_S(g, binv, x, y, w, s);
    return SW_OK;
  });
}
