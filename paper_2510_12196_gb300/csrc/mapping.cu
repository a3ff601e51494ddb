// Mappings between the caller's PE ids (host memory) and the PE codes of the
// device state (common.cuh).  Where every a_i is a power of two the code of a
// PE is its id and a mapping is copied as it stands.  Otherwise, and for the
// range check of a mapping that is set, large mappings are converted by a
// kernel: the loop over a host array cost about 1 ns a vertex (2 ms of
// the 23.7 ms map of a 3D grid of 2^21 vertices; the copy alone 0.3 ms).
#include <algorithm>

#include "engine.h"

namespace gm {
namespace {

constexpr int32_t kHostConvert = 8192;  // mappings up to this size: a host loop is shorter than a launch

__global__ void k_ids_of_codes(int32_t n, const int32_t* __restrict__ code, const int32_t* __restrict__ pe_of_code,
                               int32_t kc, int32_t* __restrict__ id) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = code[v];
    id[v] = x >= 0 && x < kc ? pe_of_code[x] : -1;
  }
}

// In place; *bad is set when an id lies outside [0, k).
__global__ void k_codes_of_ids(int32_t n, int32_t* pi, const int32_t* __restrict__ code_of_pe, int32_t k,
                               int32_t* bad) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = pi[v];
    if (p < 0 || p >= k) *bad = 1;
    else pi[v] = code_of_pe[p];
  }
}

unsigned grid(const Ctx& c, int64_t n) {
  return (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c.num_sms * 8);
}

}  // namespace

// Reads n codes back as PE ids, -1 where there is none: targets that no step
// has set yet are -1 (synchronises).
void download_mapping(Ctx& c, const int32_t* codes, int32_t n, int32_t* out) {
  const bool same = c.k == c.topo.kc;  // every code is a PE, and codes ascend with the ids
  const bool host = !same && n <= kHostConvert;
  if (!same && !host) {
    k_ids_of_codes<<<grid(c, n), 256, 0, c.st>>>(n, codes, c.d_pe_of_code, c.topo.kc, c.dest);  // (rebalancing scratch)
    count_launch();
    GM_CUDA(cudaGetLastError());
    codes = c.dest;
  }
  GM_CUDA(cudaMemcpyAsync(out, codes, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, c.st));
  GM_CUDA(cudaStreamSynchronize(c.st));
  if (host)
    for (int32_t v = 0; v < n; v++) {
      const int32_t x = out[v];
      out[v] = x >= 0 && x < c.topo.kc ? c.pe_of_code[(size_t)x] : -1;
    }
}

// Sets n codes from PE ids; MAP_E_INVALID, and the codes unchanged, when an id
// lies outside [0, k).
void upload_mapping(Ctx& c, const int32_t* pi, int32_t n, int32_t* codes) {
  const char* msg = "mapping entry out of [0, k)";
  if (n <= kHostConvert) {
    std::vector<int32_t> host((size_t)n);
    for (int32_t v = 0; v < n; v++) {
      if (pi[v] < 0 || pi[v] >= c.k) throw ApiError(MAP_E_INVALID, msg);
      host[(size_t)v] = c.code_of_pe[(size_t)pi[v]];
    }
    GM_CUDA(cudaMemcpyAsync(codes, host.data(), host.size() * sizeof(int32_t), cudaMemcpyHostToDevice, c.st));
    GM_CUDA(cudaStreamSynchronize(c.st));
    return;
  }
  int32_t* bad = reinterpret_cast<int32_t*>(c.d_stats);
  GM_CUDA(cudaMemsetAsync(bad, 0, sizeof(int64_t), c.st));
  GM_CUDA(cudaMemcpyAsync(c.dest, pi, (size_t)n * sizeof(int32_t), cudaMemcpyHostToDevice, c.st));
  k_codes_of_ids<<<grid(c, n), 256, 0, c.st>>>(n, c.dest, c.d_code_of_pe, c.k, bad); count_launch();
  GM_CUDA(cudaGetLastError());
  GM_CUDA(cudaMemcpyAsync(c.h_small + 6, bad, sizeof(int64_t), cudaMemcpyDeviceToHost, c.st));
  GM_CUDA(cudaStreamSynchronize(c.st));
  if (c.h_small[6]) throw ApiError(MAP_E_INVALID, msg);
  GM_CUDA(cudaMemcpyAsync(codes, c.dest, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToDevice, c.st));
}

}  // namespace gm
