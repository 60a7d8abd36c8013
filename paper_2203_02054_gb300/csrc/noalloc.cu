// Allocation-free contact check.
//
// casim_contacts_noalloc runs the same spatial-hash broad phase and exact
// narrow phase as a casim_step iteration, but keeps every intermediate buffer
// (packed positions, the query vertices' lists, the pair lists, control words)
// in one file-scope device array instead of memory from cudaMalloc.  It exists
// for callers that cannot allocate device memory while they run: real-time
// controllers that must not allocate inside a control loop, and host programs
// whose own allocator owns the GPU's memory pool and forbids outside cudaMalloc
// calls.  The caller still provides the inputs and the outputs.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <string>

#include "casim.h"
#include "common.cuh"
#include "kernels.h"

namespace casim {
namespace {

constexpr int NA_MAX_VERTS = 32768;
constexpr int NA_MAX_TETS = 65536;
constexpr int NA_MAX_QUERY = 16384;
constexpr unsigned NA_HASH = 65536;  // power of two >= 4 * NA_MAX_QUERY
constexpr int NA_MAX_PAIRS = 16;
constexpr int NA_CAP_ITEMS = 16 * NA_MAX_TETS + 4096;

// Byte offsets of the pieces inside the scratch array (each 256-byte aligned).
// The first ones are zeroed by every call, as far as its hash needs.
constexpr size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t OFF_CTRL = 0;
constexpr size_t OFF_ENTRIES = align256(OFF_CTRL + sizeof(Ctrl));
constexpr size_t OFF_BITS = align256(OFF_ENTRIES + sizeof(unsigned long long));
constexpr size_t OFF_HEAD = align256(OFF_BITS + sizeof(unsigned) * (NA_HASH / 8));
constexpr size_t OFF_X = align256(OFF_HEAD + sizeof(int) * NA_HASH);
constexpr size_t OFF_NEXT = align256(OFF_X + sizeof(R4<float>) * NA_MAX_VERTS);
constexpr size_t OFF_POS = align256(OFF_NEXT + sizeof(int) * NA_MAX_QUERY);
constexpr size_t OFF_COUNT = align256(OFF_POS + sizeof(float4) * NA_MAX_QUERY);
constexpr size_t OFF_PAIRS = align256(OFF_COUNT + sizeof(int) * NA_MAX_QUERY);
constexpr size_t SCRATCH_BYTES = align256(OFF_PAIRS + sizeof(int) * NA_MAX_PAIRS * NA_MAX_QUERY);

// The scratch: about 2.2 MiB, held by every GPU that loads the library until
// the process exits.  Every call uses it, so calls whose GPU work
// overlaps (on different streams or host threads) race with each other.
static __device__ __align__(256) unsigned char g_scratch[SCRATCH_BYTES];

// Device address of g_scratch per device, looked up once per device with that
// device current.  In host code the name g_scratch is only a host-side stand-in
// and must never be passed to a kernel.  The cached address belongs to the
// device's primary context: it does not survive cudaDeviceReset (the module is
// loaded again in the new context).
std::mutex g_mu;
void* g_addr[64] = {nullptr};

// The pair lists into the caller's arrays (a rejected call leaves them alone).
__global__ void k_pairs_out(Dev<float> d, int* __restrict__ count, int* __restrict__ tets) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= d.n_q || (d.ctrl->status & ST_BAD_INPUT)) return;
  const int n = min(d.pair_count[q], d.max_pairs);
  count[q] = n;
  for (int k = 0; k < n; ++k) tets[(size_t)q * d.max_pairs + k] = d.pair_tet[(size_t)q * d.max_pairs + k];
}

// Records the reason of a rejection for casim_last_error(NULL) on this thread.
int fail(int code, const std::string& msg) {
  set_handle_free_error(msg.c_str());
  return code;
}

}  // namespace
}  // namespace casim

using namespace casim;

extern "C" int casim_contacts_noalloc(int32_t n_verts, const float* dev_xyz, int32_t n_tets, const int32_t* dev_tets,
                                      int32_t n_query, const int32_t* dev_query, double cell_size,
                                      int32_t max_pairs, int32_t* dev_pair_count, int32_t* dev_pair_tet,
                                      void* cuda_stream) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (n_verts < 1 || n_verts > NA_MAX_VERTS)
    return fail(CASIM_E_INVALID, "n_verts must be in 1.." + std::to_string(NA_MAX_VERTS));
  if (n_tets < 1 || n_tets > NA_MAX_TETS)
    return fail(CASIM_E_INVALID, "n_tets must be in 1.." + std::to_string(NA_MAX_TETS));
  if (n_query < 0 || n_query > NA_MAX_QUERY)
    return fail(CASIM_E_INVALID, "n_query must be in 0.." + std::to_string(NA_MAX_QUERY));
  if (max_pairs < 1 || max_pairs > 16) return fail(CASIM_E_INVALID, "max_pairs must be in 1..16");
  if (!(cell_size > 0.0) || !(cell_size < 1e300)) return fail(CASIM_E_INVALID, "cell_size must be positive");
  if (!dev_xyz || !dev_tets || (n_query > 0 && (!dev_query || !dev_pair_count || !dev_pair_tet)))
    return fail(CASIM_E_INVALID, "null device pointer");
  if (reinterpret_cast<uintptr_t>(dev_tets) % 16 != 0)
    return fail(CASIM_E_INVALID, "dev_tets must be 16-byte aligned");
  if (n_query == 0) return CASIM_OK;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return fail(CASIM_E_CUDA, "cudaGetDevice failed");
  if (!g_addr[dev]) {
    // first call on this device: look up the scratch's device address (must
    // happen outside stream capture)
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p) return fail(CASIM_E_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_addr[dev] = p;
  }
  unsigned char* base = static_cast<unsigned char*>(g_addr[dev]);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  Ctrl* ctrl = reinterpret_cast<Ctrl*>(base + OFF_CTRL);
  R4<float>* X = reinterpret_cast<R4<float>*>(base + OFF_X);
  Dev<float> d{};
  d.n_v = n_verts;
  d.n_t = n_tets;
  d.n_q = n_query;
  d.X = X;
  d.tet = reinterpret_cast<const int4*>(dev_tets);
  d.q_verts = dev_query;
  d.H_q = 64;
  while (d.H_q < 4u * (unsigned)n_query) d.H_q *= 2;
  d.q_bits = reinterpret_cast<unsigned*>(base + OFF_BITS);
  d.q_head = reinterpret_cast<int*>(base + OFF_HEAD);
  d.q_next = reinterpret_cast<int*>(base + OFF_NEXT);
  d.q_pos = reinterpret_cast<float4*>(base + OFF_POS);
  d.entries = reinterpret_cast<unsigned long long*>(base + OFF_ENTRIES);
  d.cap_items = NA_CAP_ITEMS;
  d.pair_count = reinterpret_cast<int*>(base + OFF_COUNT);
  d.pair_tet = reinterpret_cast<int*>(base + OFF_PAIRS);
  d.max_pairs = max_pairs;
  d.collision = 1;
  d.narrow_threads = 128;  // a few thousand tets: more, smaller blocks
  d.cell = cell_size;
  d.inv_cell = 1.0 / cell_size;
  d.ctrl = ctrl;
  // zero control word, entries, bits and list heads; the vertex ids are tested
  // where they are first used, so one wait at the end serves every check
  cudaError_t e2 = cudaMemsetAsync(base, 0, OFF_HEAD + sizeof(int) * d.H_q, st);
  launch_pack_queries(d, dev_xyz, X, st);
  launch_tets<float>(d, true, st);
  k_pairs_out<<<(n_query + 127) / 128, 128, 0, st>>>(d, dev_pair_count, dev_pair_tet);
  e = e2 == cudaSuccess ? cudaGetLastError() : e2;
  int status = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&status, &ctrl->status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(CASIM_E_CUDA, std::string("contact check: ") + cudaGetErrorString(e));
  if (status & ST_BAD_INPUT) return fail(CASIM_E_INVALID, "a tet or query vertex id is out of range");
  if (status & ST_NONFINITE) return fail(CASIM_E_NONFINITE, "non-finite position");
  if (status & ST_PAIRS_TRUNC)
    return fail(CASIM_E_OVERFLOW, "a query vertex lies in more than max_pairs tets (the smallest ids are kept)");
  if (status & ST_OVERFLOW)
    return fail(CASIM_E_OVERFLOW, "more hash entries than the scratch holds (cell_size too small for the tets)");
  return CASIM_OK;
}
