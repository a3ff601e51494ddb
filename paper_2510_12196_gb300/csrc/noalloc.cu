// Allocation-free evaluation of the objective J and the maximum block weight.
//
// map_objective_noalloc computes the same two numbers as map_objective, but
// without a context and without allocating any device memory: the caller
// passes device pointers to the graph, the mapping and a two-element output,
// and the scratch (J accumulator, block weights, PE code table) lives in one
// file-scope __device__ array.  It serves callers that cannot or must not
// allocate: the CUDA allocation calls (cudaMalloc / cudaFree) may synchronise
// the whole device and stall unrelated streams, and some callers run under a
// fixed device-memory budget owned by their own memory pool, or simply hold a
// graph and a mapping in device memory and want its cost without creating a
// context (whose set-up allocates and validates the whole graph).
//
// Limits and sharing: at most kNoAllocMaxPE = 16384 PEs (code space 2^14).
// Every call on a device shares the single scratch array, which keeps the
// last call's contents; each call clears what must start at zero before it
// uses it.  Calls whose work overlaps on the GPU (different streams, or
// several host threads) race on the array and give wrong results: serialise
// them.  The first call on a device looks up the array's device address
// (cudaGetSymbolAddress, with that device current) and keeps it for the
// process; make that first call before any stream capture on the device.
// A cudaDeviceReset invalidates the kept address: the entry point must not be
// used on a device after it was reset.
#include <mutex>
#include <string>

#include "engine.h"
#include "search.h"

namespace gm {
namespace {

constexpr int kNoAllocMaxPE = 1 << kMaxCodeBits;
constexpr int kNaThreads = 256;

struct NoAllocScratch {
  unsigned long long J;
  long long maxw;
  unsigned int done;                // blocks of the pass that have finished
  long long W[kNoAllocMaxPE];       // block weights by PE code
  int32_t code[kNoAllocMaxPE];      // PE id -> PE code
};

// The scratch of every call on this device (about 192 KiB, held until exit).
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

struct Hier {
  int32_t a[kMaxLevels];
};

// Clears the accumulators and fills the PE id -> code table.
__global__ void k_na_clear(NoAllocScratch* s, Topo t, Hier h) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    s->J = 0;
    s->maxw = 0;
    s->done = 0;
  }
  for (int b = i; b < t.kc; b += gridDim.x * blockDim.x) s->W[b] = 0;
  for (int p = i; p < t.k; p += gridDim.x * blockDim.x) {
    int rem = p, code = 0;
    for (int l = 0; l < t.levels; l++) {
      code |= (rem % h.a[l]) << t.s[l];
      rem /= h.a[l];
    }
    s->code[p] = code;
  }
}

// J and block weights.  The CSR entries are split evenly whatever the degrees:
// a block takes consecutive tiles of kNaTile entries and finds the row of its
// first entry by one 256-way search of xadj.  The rows that start in a tile set
// a bit at their first entry and store their PE there, and an entry takes its
// row's PE from the last bit at or before it.  A warp's entries are 32
// consecutive ones at a time, so that their neighbours' PEs, near one another
// where the ids have locality, come in few cache lines.  The pass streams 8
// bytes an entry and gathers 4.  RGG of 2^20 vertices, 12.6e6 entries: 64-85 us
// whatever the mapping and the code space, R-MAT 2^20 of 31e6 entries 183 us (eight
// consecutive entries per thread 87-135 and 268 us; eight lanes per row 81-614 us
// and 5.5 ms).
// The weights are summed by warp and PE first, then in the block's shared
// memory where it has more vertices than there are PE codes (at most kNaCodes),
// else straight into the global sums.
// Mapping entries or neighbours outside their range are skipped, and only
// entries of [0, xadj[n]) are read, so that a malformed xadj cannot make the
// pass read outside the adjacency arrays.  The last block to finish writes
// the result.
constexpr int kNaItems = 8;
constexpr int kNaTile = kNaThreads * kNaItems;
constexpr int kNaCodes = 2048;
constexpr int64_t kNaVertices = 1024;  // vertices per block at least (blocks past the last one sum no weights)

// Largest v in [0, n) with xadj[v] <= e, -1 if none; all threads call it.
__device__ __forceinline__ int32_t na_row_of(const int64_t* __restrict__ xadj, int32_t n, int64_t e) {
  if (xadj[0] > e) return -1;
  return (int32_t)last_by_probes(n, kNaThreads, [&](int64_t lo, int64_t len, int64_t step) {
    const int64_t at = (int64_t)threadIdx.x * step;
    return __syncthreads_count(at < len && xadj[lo + at] <= e);
  });
}

// The rows of a tile, two tiles in turn.
struct NaRows {
  uint32_t heads[2][kNaTile / 32];  // entries that start a row
  int16_t code[2][kNaTile];         // and its PE code (-1: PE id out of range)
  int16_t carry[2];                 // code of the row that the tile's first entries go on with
  int16_t last[kNaTile / 32];       // last start before each 32 entries (-1: none)
};

// plain: the PE ids are their own codes (every a_i a power of two)
__global__ void __launch_bounds__(kNaThreads, 5) k_na_eval(int32_t n, const int64_t* __restrict__ xadj,
                                                           const int32_t* __restrict__ adj,
                                                           const int32_t* __restrict__ adjw,
                                                           const int32_t* __restrict__ vw,
                                                           const int32_t* __restrict__ pi, NoAllocScratch* s, Topo t,
                                                           int plain, int64_t* out) {
  extern __shared__ __align__(16) unsigned char na_dyn[];
  unsigned long long* sW = reinterpret_cast<unsigned long long*>(na_dyn);  // [kc] when kc <= kNaCodes
  const bool fits = t.kc <= kNaCodes;
  uint16_t* scode = reinterpret_cast<uint16_t*>(na_dyn + (fits ? (size_t)t.kc * 8 : 0));  // [k] unless plain
  __shared__ int32_t sdist[32];
  __shared__ int64_t sm[33];
  __shared__ NaRows R;
  __shared__ unsigned int last;
  static_assert(kNaTile / 32 == 64, "a warp scans the words of a tile, two per lane");
  const int lane = (int)threadIdx.x & 31;
  // consecutive vertices per block
  const int64_t per = max(kNaVertices, ((int64_t)n + gridDim.x - 1) / gridDim.x);
  const int64_t va = min((int64_t)n, blockIdx.x * per), vb = min((int64_t)n, va + per);
  const bool local = fits && per >= t.kc && va < vb;
  load_sdist(sdist, t);
  if (threadIdx.x < 2 * (kNaTile / 32)) R.heads[threadIdx.x / (kNaTile / 32)][threadIdx.x % (kNaTile / 32)] = 0;
  if (local)
    for (int b = threadIdx.x; b < t.kc; b += kNaThreads) sW[b] = 0;
  if (!plain)
    for (int p = threadIdx.x; p < t.k; p += kNaThreads) scode[p] = (uint16_t)s->code[p];
  __syncthreads();
  auto code_of = [&](int32_t p) { return plain ? p : (int32_t)scode[p]; };
  auto code_or_none = [&](int32_t p) { return p >= 0 && p < t.k ? code_of(p) : -1; };
  auto add_weight = [&](int32_t c, int64_t x) {
    atomicAdd(local ? &sW[c] : (unsigned long long*)&s->W[c], (unsigned long long)x);
  };

  for (int64_t v0 = va + (threadIdx.x - lane); v0 < vb; v0 += kNaThreads) {  // (warp-uniform)
    const int64_t v = v0 + lane;
    const int32_t c = v < vb ? code_or_none(pi[v]) : -1;
    warp_add(c, c >= 0 ? vw[v] : 0, add_weight);
  }

  const int64_t m = xadj[n];
  int64_t acc = 0;
  const int64_t tiles = (m + kNaTile - 1) / kNaTile;
  const int64_t t0 = tiles * blockIdx.x / gridDim.x, t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  // the row of the block's first entry (row 0 for entries before the first row)
  int32_t lo = t0 < t1 ? max(na_row_of(xadj, n, t0 * kNaTile), 0) : 0;
  const int first = ((int)threadIdx.x - lane) * kNaItems + lane;  // this thread's entries: first + 32 j
  for (int64_t tile = t0; tile < t1; tile++) {
    const int cur = (int)(tile & 1);
    const int64_t e0 = tile * kNaTile, e1 = min(e0 + kNaTile, m);
    const int span = (int)(e1 - e0);
    int32_t u[kNaItems], w[kNaItems];
#pragma unroll
    for (int j = 0; j < kNaItems; j++) {
      const int x = first + 32 * j;
      u[j] = x < span ? adj[e0 + x] : -1;
      w[j] = x < span ? (adjw ? adjw[e0 + x] : 1) : 0;
    }
    // the rows lo .. lo + nr - 1 start before e1
    int32_t nr = 0;
    bool staged = false;
    while (!staged && nr < kNaTile) {
      const int32_t r = nr + (int32_t)threadIdx.x;
      const int64_t at = (int64_t)lo + r;
      const bool is_row = at < n;
      const int64_t b = is_row ? xadj[at] - e0 : span, e = is_row ? xadj[at + 1] - e0 : span;
      const int32_t p = is_row ? pi[at] : -1;
      if (nr == 0) {  // the neighbours' PEs, in flight with the rows
#pragma unroll
        for (int j = 0; j < kNaItems; j++) u[j] = u[j] >= 0 && u[j] < n ? pi[u[j]] : -1;
      }
      const int16_t c = (int16_t)code_or_none(p);
      if (r == 0) R.carry[cur] = b <= 0 ? c : (int16_t)-1;
      if (is_row && b >= 0 && b < span && e > b) {
        R.code[cur][b] = c;
        atomicOr(&R.heads[cur][b >> 5], 1u << (b & 31));
      }
      const int got = __syncthreads_count(is_row && (r == 0 || b < span));
      nr += got;
      staged = got < kNaThreads;
    }
    if (!staged) nr = max(na_row_of(xadj, n, e1 - 1) - lo + 1, 1);  // long runs of empty rows: searched below
    if (threadIdx.x < 32) {
      const uint32_t a = R.heads[cur][lane], b = R.heads[cur][32 + lane];
      int x = a ? 32 * lane + 31 - __clz(a) : -1, y = b ? 32 * (32 + lane) + 31 - __clz(b) : -1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int p = __shfl_up_sync(0xffffffffu, x, o), q = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) {
          x = max(x, p);
          y = max(y, q);
        }
      }
      const int all = __shfl_sync(0xffffffffu, x, 31);
      const int px = __shfl_up_sync(0xffffffffu, x, 1), py = __shfl_up_sync(0xffffffffu, y, 1);
      R.last[lane] = (int16_t)(lane ? px : -1);
      R.last[32 + lane] = (int16_t)max(all, lane ? py : -1);
    } else if (threadIdx.x < 32 + kNaTile / 32) {
      R.heads[cur ^ 1][threadIdx.x - 32] = 0;  // the next tile's (every thread is done with the last one)
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kNaItems; j++) {
      const int x = first + 32 * j;
      if (x >= span || u[j] < 0 || u[j] >= t.k) continue;
      int32_t cv;
      if (staged) {
        const uint32_t word = R.heads[cur][x >> 5] & (0xffffffffu >> (31 - lane));
        const int pos = word ? (x & ~31) + 31 - __clz(word) : R.last[x >> 5];
        cv = pos >= 0 ? R.code[cur][pos] : R.carry[cur];
      } else {
        const int32_t i = last_by_bisection(0, nr, [&](int32_t r) { return xadj[lo + r] - e0 <= x; });
        cv = xadj[lo + i] - e0 <= x ? code_or_none(pi[lo + i]) : -1;
      }
      if (cv >= 0) acc += (int64_t)w[j] * dcode(sdist, cv, code_of(u[j]));
    }
    lo += nr - 1;  // the last row of this tile may go on in the next
  }
  acc = block_sum(acc, sm);
  if (threadIdx.x == 0 && acc) atomicAdd(&s->J, (unsigned long long)acc);
  if (local)
    for (int b = threadIdx.x; b < t.kc; b += kNaThreads)
      if (sW[b]) atomicAdd((unsigned long long*)&s->W[b], sW[b]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&s->done, 1u) == gridDim.x - 1 ? 1u : 0u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  __shared__ long long smax[kNaThreads / 32];
  long long mx = 0;
  for (int b = threadIdx.x; b < t.kc; b += kNaThreads) mx = max(mx, __ldcg(&s->W[b]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kNaThreads / 32; w++) mx = max(mx, smax[w]);
    s->maxw = mx;
    out[0] = (int64_t)atomicAdd(&s->J, 0ULL);
    out[1] = mx;
  }
}

// Address of the scratch array on each device, looked up once per device.
std::mutex g_na_mutex;
NoAllocScratch* g_na_ptr[256] = {nullptr};

}  // namespace
}  // namespace gm

using namespace gm;

extern "C" GPUMAP_API map_status map_objective_noalloc(const int64_t* xadj, const int32_t* adjncy,
                                                       const int32_t* adjwgt, const int32_t* vwgt, int32_t n,
                                                       const int32_t* pi, const int32_t* hier, const int32_t* dist,
                                                       int32_t levels, int64_t* out, void* stream) {
  last_create_error().clear();
  auto fail = [](map_status s, const std::string& m) {
    last_create_error() = m;  // readable through map_last_error(NULL)
    return s;
  };
  if (n < 1 || !xadj || !vwgt || !pi || !hier || !dist || !out) return fail(MAP_E_INVALID, "null pointer or n < 1");
  if (levels < 1 || levels > kMaxLevels) return fail(MAP_E_INVALID, "levels must be in [1, 16]");
  Topo t{};
  Hier h{};
  t.levels = levels;
  int64_t k = 1;
  int32_t s = 0;
  for (int i = 0; i < levels; i++) {
    if (hier[i] < 1 || dist[i] < 0) return fail(MAP_E_INVALID, "hierarchy factors must be >= 1, distances >= 0");
    int32_t b = 0;
    while ((1 << b) < hier[i]) b++;
    t.s[i] = s;
    s += b;
    if (s > kMaxCodeBits)
      return fail(MAP_E_INVALID, "hierarchy exceeds the 16384-PE code space of map_objective_noalloc");
    k *= hier[i];
    h.a[i] = hier[i];
    t.dist[i] = dist[i];
  }
  t.s[levels] = s;
  t.code_bits = s;
  t.kc = 1 << s;
  t.k = (int32_t)k;
  for (int b = 0; b < 32; b++) t.dist_of_bit[b] = 0;
  for (int i = 0; i < levels; i++)
    for (int b = t.s[i]; b < t.s[i + 1]; b++) t.dist_of_bit[b] = dist[i];

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) {
    cudaGetLastError();
    return fail(MAP_E_CUDA, "cudaGetDevice failed");
  }
  NoAllocScratch* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        cudaGetLastError();
        return fail(MAP_E_CUDA, std::string("cudaGetSymbolAddress of the scratch array failed: ") +
                                    cudaGetErrorString(e));
      }
      g_na_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    scratch = g_na_ptr[dev];
  }
  cudaStream_t st = (cudaStream_t)stream;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 1) sms = 1;
  k_na_clear<<<(t.kc + kNaThreads - 1) / kNaThreads, kNaThreads, 0, st>>>(scratch, t, h); count_launch();
  int plain = 1;
  for (int i = 0; i < levels; i++) plain &= (hier[i] & (hier[i] - 1)) == 0 ? 1 : 0;
  const size_t smem = (t.kc <= kNaCodes ? (size_t)t.kc * 8 : 0) + (plain ? 0 : (size_t)t.k * sizeof(uint16_t));
  // the entry count lies in device memory: one wave of blocks, those without a tile leave at once
  k_na_eval<<<(unsigned)(sms * 5), kNaThreads, smem, st>>>(n, xadj, adjncy, adjwgt, vwgt, pi, scratch, t, plain, out);
  count_launch();
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(MAP_E_CUDA, std::string("launch failed: ") + cudaGetErrorString(e));
  return MAP_OK;
}
