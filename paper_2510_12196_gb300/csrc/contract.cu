// Contraction of large levels: the coarse CSR from one counting sort by the
// coarse target.
//
// The entries are walked by coarse source: the fine vertices are grouped by
// M(v) (a counting sort of n ids), so the entry stream comes in ascending
// order of the coarse source c for free.  The adjacency is symmetric, so the
// entries (c -> d, w), sorted stably by d alone, are the rows d with their
// neighbours c in ascending order and parallel entries next to each other:
// half the key of a sort by (source, target).  Source, target and weight share
// one 64-bit word, so a pass moves 16 bytes an entry:
//   k_ct_gen      gathers M, writes the words in source order (entries inside
//                 a cluster as kDrop) and counts the first digit
//   k_ct_scatter  one stable pass by a digit of at most kCtDigitBits bits; the
//                 first also drops the kDrop words
//   k_ct_heads, k_ct_apply  number the distinct (d, c), sum their weights and
//                 write the coarse rows
// Every block owns a contiguous range of the stream in all of them, so the
// digit counts are kept per block, not per tile, and a block's writes to a
// digit follow one another.  What bounds it is HBM traffic: 8 + 4 (M from L2)
// + 8 bytes in k_ct_gen, 16 per scatter, 8 per count, 16 to number and write.
// R-MAT 2^22, 128 M entries to 84 M, and two more levels of 84 and 80 M: 3.2 ms a
// level (k_ct_gen 0.58, two scatters 1.66, counts 0.17 + 0.12, k_ct_apply 0.53),
// where keys (source, target) with separate weights, five or six 8-bit passes
// with per-tile digit counts and three scans took 11 ms.
#include <algorithm>
#include <atomic>

#include "engine.h"
#include "search.h"

namespace gm {
namespace {

constexpr uint64_t kDrop = ~0ULL;
constexpr int kCtDigitBits = 10;
constexpr int kCtDigits = 1 << kCtDigitBits;
constexpr int kGenThreads = 256;
constexpr int kGenItems = 8;
constexpr int kGenTile = kGenThreads * kGenItems;
constexpr int kScThreads = 512;
constexpr int kScItems = 16;
constexpr int kScTile = kScThreads * kScItems;
constexpr int kScWarps = kScThreads / 32;
constexpr int kSplit = 4;  // k_ct_gen / k_ct_hist blocks per scatter block (they hold less state)
static_assert(kScTile % (kSplit * kGenTile) == 0, "a quarter of a block's range is whole gen tiles");
constexpr int kApThreads = 256;
constexpr int kApItems = 16;
constexpr int kApTile = kApThreads * kApItems;

// Entries of the stream per scatter block (whole tiles).
__host__ __device__ __forceinline__ int64_t block_range(int64_t n, int blocks) {
  const int64_t per = (n + blocks - 1) / blocks;
  return (per + kScTile - 1) / kScTile * kScTile;
}

// --- grouping of the fine vertices by coarse vertex -------------------------
__global__ void k_ct_count(int32_t n, const int64_t* __restrict__ xadj, const int32_t* __restrict__ M,
                           const int32_t* __restrict__ vw, int32_t* cnt, int32_t* vwc) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = M[v];
    atomicAdd(&vwc[c], vw[v]);
    if (xadj[v + 1] > xadj[v]) atomicAdd(&cnt[c], 1);
  }
}
__global__ void k_ct_place(int32_t n, const int64_t* __restrict__ xadj, const int32_t* __restrict__ M, int32_t* cur,
                           int32_t* perm) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (xadj[v + 1] > xadj[v]) perm[atomicAdd(&cur[M[v]], 1)] = (int32_t)v;  // any order inside a group
}
struct LoadCnt {
  const int32_t* a;
  __device__ int64_t operator()(int64_t i) const { return a[i]; }
};
struct StoreCnt {
  int32_t* a;
  __device__ void operator()(int64_t i, int64_t e, int64_t) const { a[i] = (int32_t)e; }
};
struct LoadRowDeg {
  const int32_t* perm;
  const int64_t* xadj;
  __device__ int64_t operator()(int64_t i) const {
    const int32_t v = perm[i];
    return xadj[v + 1] - xadj[v];
  }
};
__global__ void k_ct_copy(const int64_t* src, int64_t* dst) { *dst = *src; }

// Largest i in [0, n) with a[i] <= x (a[0] <= x); all kGenThreads threads call it.
__device__ __forceinline__ int64_t find_row(const int64_t* __restrict__ a, int64_t n, int64_t x) {
  return last_by_probes(n, kGenThreads, [&](int64_t lo, int64_t len, int64_t step) {
    const int64_t at = (int64_t)threadIdx.x * step;
    return __syncthreads_count(at < len && a[lo + at] <= x);
  });
}

// The words of the stream, in coarse source order.  A tile's rows are looked
// up together (non-empty, so at most one per entry); an entry finds its row by
// the count of row starts up to it in a bit mask.
__global__ void __launch_bounds__(kGenThreads) k_ct_gen(const int64_t* __restrict__ xadj,
                                                        const int32_t* __restrict__ adj,
                                                        const int32_t* __restrict__ adjw,
                                                        const int32_t* __restrict__ M,
                                                        const int32_t* __restrict__ perm,
                                                        const int64_t* __restrict__ pre, const int64_t* d_rows,
                                                        int64_t m, int bits, int wbits, int digit_bits,
                                                        uint64_t* __restrict__ key, int32_t* bhist, int blocks) {
  __shared__ int64_t rbase[kGenTile + 1];  // CSR position of stream position f of row r: rbase[r] + f
  __shared__ int32_t rc[kGenTile + 1];     // its coarse source
  __shared__ uint32_t heads[kGenTile / 32];
  __shared__ int32_t before[kGenTile / 32];
  __shared__ int32_t hist[kCtDigits];
  static_assert(kGenTile / 32 == 64, "two warps number the row starts");
  const int64_t rows = *d_rows;
  const int64_t range = block_range(m, blocks), part = range / kSplit;
  const int own = blockIdx.x / kSplit;
  const int64_t f0 = (int64_t)own * range + (blockIdx.x % kSplit) * part, f1 = min(f0 + part, m);
  if (f0 >= f1) return;
  const int ndig = 1 << digit_bits;
  for (int i = threadIdx.x; i < ndig; i += kGenThreads) hist[i] = 0;
  int64_t lo = find_row(pre, rows, f0);
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = f0; e0 < f1; e0 += kGenTile) {
    const int64_t e1 = min(e0 + kGenTile, f1);
    __syncthreads();  // the previous tile's rows have been read
    if (threadIdx.x < kGenTile / 32) heads[threadIdx.x] = 0;
    __syncthreads();
    int nr = 0, got;
    do {
      const int r = nr + (int)threadIdx.x;
      const int64_t at = lo + r;
      const int64_t f = at < rows ? pre[at] : m;
      const bool in = at < rows && f < e1;
      if (in) {
        const int32_t v = perm[at];
        rc[r] = M[v];
        rbase[r] = xadj[v] - f;
        if (r > 0) atomicOr(&heads[(f - e0) >> 5], 1u << ((f - e0) & 31));  // (f >= e0: row lo holds e0 or ends there)
      }
      got = __syncthreads_count(in);
      nr += got;
    } while (got == kGenThreads);
    if (threadIdx.x < 32) {  // row starts before each 32-entry word
      const int a = __popc(heads[lane]), b = __popc(heads[32 + lane]);
      int x = a, y = b;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int p = __shfl_up_sync(0xffffffffu, x, o), q = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) {
          x += p;
          y += q;
        }
      }
      before[lane] = x - a;
      before[32 + lane] = __shfl_sync(0xffffffffu, x, 31) + y - b;
    }
    __syncthreads();
    // entries x = warp * 256 + 32 j + lane of the tile
    const int first = (threadIdx.x >> 5) * (32 * kGenItems) + lane;
    int32_t c[kGenItems], d[kGenItems], w[kGenItems];
#pragma unroll
    for (int j = 0; j < kGenItems; j++) {
      const int x = first + 32 * j;
      c[j] = -1;
      d[j] = 0;
      w[j] = 0;
      if (e0 + x < e1) {
        const int r = before[x >> 5] + __popc(heads[x >> 5] & (0xffffffffu >> (31 - lane)));
        c[j] = rc[r];
        const int64_t e = rbase[r] + e0 + x;
        d[j] = adj[e];
        w[j] = adjw[e];
      }
    }
#pragma unroll
    for (int j = 0; j < kGenItems; j++)
      if (c[j] >= 0) d[j] = M[d[j]];
#pragma unroll
    for (int j = 0; j < kGenItems; j++) {
      if (c[j] < 0) continue;
      const bool keep = c[j] != d[j];
      key[e0 + first + 32 * j] =
          keep ? (((((uint64_t)(uint32_t)d[j]) << bits) | (uint32_t)c[j]) << wbits) | (uint32_t)w[j] : kDrop;
      if (keep) atomicAdd(&hist[d[j] & (ndig - 1)], 1);
    }
    lo += nr - 1;  // the last row may go on in the next tile
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ndig; i += kGenThreads)
    if (hist[i]) atomicAdd(&bhist[(int64_t)i * blocks + own], hist[i]);
}

// Digit counts per block of the words [0, *d_n).
__global__ void __launch_bounds__(kGenThreads) k_ct_hist(const uint64_t* __restrict__ key, const int64_t* d_n,
                                                         int shift, int digit_bits, int32_t* bhist, int blocks) {
  __shared__ int32_t hist[kCtDigits];
  const int64_t n = *d_n;
  const int64_t range = block_range(n, blocks), part = range / kSplit;
  const int own = blockIdx.x / kSplit;
  const int64_t f0 = (int64_t)own * range + (blockIdx.x % kSplit) * part, f1 = min(f0 + part, n);
  if (f0 >= f1) return;
  const int ndig = 1 << digit_bits;
  for (int i = threadIdx.x; i < ndig; i += kGenThreads) hist[i] = 0;
  __syncthreads();
  for (int64_t f = f0; f < f1; f += kGenTile) {
#pragma unroll
    for (int j = 0; j < kGenItems; j++) {
      const int64_t x = f + j * kGenThreads + threadIdx.x;
      if (x < f1) atomicAdd(&hist[(int)(key[x] >> shift) & (ndig - 1)], 1);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ndig; i += kGenThreads)
    if (hist[i]) atomicAdd(&bhist[(int64_t)i * blocks + own], hist[i]);
}

// One digit per CTA: its blocks' counts to offsets, and its total.
__global__ void __launch_bounds__(128) k_ct_dscan(int32_t* bhist, int blocks, int32_t* total) {
  __shared__ int32_t sm[33];
  int32_t* row = bhist + (int64_t)blockIdx.x * blocks;
  int32_t carry = 0;
  for (int base = 0; base < blocks; base += 128) {
    const int i = base + (int)threadIdx.x;
    const int32_t x = i < blocks ? row[i] : 0;
    int32_t tot;
    const int32_t e = block_exclusive_scan(x, sm, &tot);
    if (i < blocks) row[i] = carry + e;
    carry += tot;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

struct ScSmem {
  uint64_t key[kScTile];             // a tile in digit order
  uint16_t cnt[kScWarps][kCtDigits]; // per warp: a digit's count, then its offset within the digit
  int32_t run[kCtDigits];            // the block's next position of each digit
  int32_t start[kCtDigits];          // a digit's first slot in the tile
};

// One stable counting-sort pass.  A block walks its range tile by tile (512
// threads x 16 words, two blocks per SM): ranks within the tile in (warp,
// step, lane) order, which is stream order, the tile placed in digit order in
// shared memory, then written out in runs.
__global__ void __launch_bounds__(kScThreads, 2) k_ct_scatter(const uint64_t* __restrict__ kin,
                                                              uint64_t* __restrict__ kout, int64_t max_n,
                                                              const int64_t* d_n, int shift, int digit_bits,
                                                              const int32_t* __restrict__ bhist,
                                                              const int32_t* __restrict__ total, int blocks,
                                                              int64_t* d_out) {
  extern __shared__ __align__(16) unsigned char sc_raw[];
  ScSmem& S = *reinterpret_cast<ScSmem*>(sc_raw);
  __shared__ int32_t sm[33];
  const int64_t n = d_n ? *d_n : max_n;
  const int64_t range = block_range(n, blocks);
  const int64_t f0 = (int64_t)blockIdx.x * range, f1 = min(f0 + range, n);
  const int ndig = 1 << digit_bits;
  const uint32_t dmask = ndig - 1;
  static_assert(kCtDigits == 2 * kScThreads, "two digits per thread");
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int g0 = 2 * (int)threadIdx.x;
  {  // first position of every digit, then of this block's part of it
    const int32_t a = g0 < ndig ? total[g0] : 0, b = g0 + 1 < ndig ? total[g0 + 1] : 0;
    int32_t all;
    const int32_t e = block_exclusive_scan(a + b, sm, &all);
    if (g0 < ndig) S.run[g0] = e + bhist[(int64_t)g0 * blocks + blockIdx.x];
    if (g0 + 1 < ndig) S.run[g0 + 1] = e + a + bhist[(int64_t)(g0 + 1) * blocks + blockIdx.x];
    if (d_out && blockIdx.x == 0 && threadIdx.x == 0) *d_out = all;
  }
  const unsigned lt = (1u << l) - 1u;
  for (int64_t base = f0; base < f1; base += kScTile) {
    for (int i = threadIdx.x; i < kScWarps * kCtDigits / 2; i += kScThreads)
      reinterpret_cast<uint32_t*>(&S.cnt[0][0])[i] = 0;
    uint64_t k[kScItems];
    const int64_t wbase = base + (int64_t)w * 32 * kScItems;
#pragma unroll
    for (int j = 0; j < kScItems; j++) {
      const int64_t x = wbase + j * 32 + l;
      k[j] = x < f1 ? kin[x] : kDrop;
    }
    __syncthreads();
    uint32_t rank2[kScItems / 2];  // two 16-bit ranks per word
#pragma unroll
    for (int j = 0; j < kScItems; j++) {
      const bool valid = k[j] != kDrop;
      const uint32_t d = (uint32_t)(k[j] >> shift) & dmask;
      // the lanes of the same digit, one ballot per bit (0.83 ms a
      // pass of R-MAT 2^22, with __match_any_sync 0.89)
      unsigned peers = __ballot_sync(0xffffffffu, valid);
      for (int b = 0; b < digit_bits; b++) {
        const bool on = (d >> b) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, on);
        peers &= on ? m : ~m;
      }
      const uint32_t r = valid ? S.cnt[w][d] + __popc(peers & lt) : 0;
      __syncwarp();
      if (valid && (peers & lt) == 0) S.cnt[w][d] = (uint16_t)(r + __popc(peers));
      __syncwarp();
      if (j & 1) rank2[j / 2] |= r << 16;
      else rank2[j / 2] = r;
    }
    __syncthreads();
    // the warps' offsets within each digit, and the digit's count
    int32_t c0 = 0, c1 = 0;
    if (g0 < ndig) {
#pragma unroll
      for (int ww = 0; ww < kScWarps; ww++) {
        uint32_t& both = *reinterpret_cast<uint32_t*>(&S.cnt[ww][g0]);
        const uint32_t x = both;
        both = (uint32_t)c0 | ((uint32_t)c1 << 16);
        c0 += x & 0xffffu;
        c1 += x >> 16;
      }
    }
    int32_t cnt;
    const int32_t e = block_exclusive_scan(c0 + c1, sm, &cnt);
    if (g0 < ndig) {
      S.start[g0] = e;
      S.start[g0 + 1] = e + c0;  // (ndig is even)
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kScItems; j++) {
      if (k[j] == kDrop) continue;
      const uint32_t d = (uint32_t)(k[j] >> shift) & dmask;
      const uint32_t r = (j & 1) ? rank2[j / 2] >> 16 : rank2[j / 2] & 0xffffu;
      S.key[S.start[d] + S.cnt[w][d] + r] = k[j];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += kScThreads) {
      const uint64_t key = S.key[i];
      const uint32_t d = (uint32_t)(key >> shift) & dmask;
      kout[S.run[d] + (i - S.start[d])] = key;
    }
    __syncthreads();
    if (g0 < ndig) {
      S.run[g0] += c0;
      S.run[g0 + 1] += c1;
    }
  }
}

// Distinct (d, c) per tile of the sorted words.
__global__ void __launch_bounds__(kApThreads) k_ct_heads(const uint64_t* __restrict__ key, const int64_t* d_n,
                                                         int wbits, int64_t* tile_sums) {
  __shared__ int32_t sm[33];
  const int64_t n = *d_n;
  const int64_t base = (int64_t)blockIdx.x * kApTile;
  int32_t cnt = 0;
  if (base < n) {
#pragma unroll
    for (int j = 0; j < kApItems; j++) {
      const int64_t x = base + j * kApThreads + threadIdx.x;
      if (x < n) cnt += (x == 0 || (key[x] >> wbits) != (key[x - 1] >> wbits)) ? 1 : 0;
    }
  }
  cnt = block_sum(cnt, sm);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = cnt;
}

// Writes the coarse rows: a warp takes 512 consecutive words, 32 at a time.
// The distinct pairs that begin and end within a step are stored, the pieces
// of a pair that crosses a step are added (adjw starts at zero).  The first
// pair of a row also writes the row's start (the empty rows stay at -1).
__global__ void __launch_bounds__(kApThreads) k_ct_apply(const uint64_t* __restrict__ key, const int64_t* d_n,
                                                         int bits, int wbits, const int64_t* __restrict__ tile_off,
                                                         int32_t* __restrict__ adjc, int32_t* adjwc, int64_t* xadjc) {
  __shared__ int32_t wsum[kApThreads / 32];
  const int64_t n = *d_n;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int64_t first = (int64_t)blockIdx.x * kApTile + (int64_t)w * 32 * kApItems;
  uint64_t k[kApItems];
#pragma unroll
  for (int j = 0; j < kApItems; j++) {
    const int64_t x = first + 32 * j + l;
    k[j] = x < n ? key[x] : kDrop;
  }
  // the pair before this warp's words (none before the first)
  const uint64_t none = kDrop;
  uint64_t prev = (first > 0 && first < n) ? key[first - 1] >> wbits : none;
  const uint64_t prev0 = prev;
  int32_t heads = 0;
#pragma unroll
  for (int j = 0; j < kApItems; j++) {
    const uint64_t p = k[j] >> wbits;
    uint64_t q = __shfl_up_sync(0xffffffffu, p, 1);
    if (l == 0) q = prev;
    prev = __shfl_sync(0xffffffffu, p, 31);
    heads += __popc(__ballot_sync(0xffffffffu, k[j] != kDrop && p != q));
  }
  if (l == 0) wsum[w] = heads;
  __syncthreads();
  int64_t at = tile_off[blockIdx.x];  // distinct pairs before the current step
  for (int i = 0; i < w; i++) at += wsum[i];
  prev = prev0;
  const uint64_t wmask = (1ULL << wbits) - 1ULL, cmask = (1ULL << bits) - 1ULL;
#pragma unroll
  for (int j = 0; j < kApItems; j++) {
    const bool valid = k[j] != kDrop;
    const uint64_t p = k[j] >> wbits;
    uint64_t q = __shfl_up_sync(0xffffffffu, p, 1);
    if (l == 0) q = prev;
    prev = __shfl_sync(0xffffffffu, p, 31);
    const bool head = valid && p != q;
    const unsigned hb = __ballot_sync(0xffffffffu, head);
    int32_t sum = valid ? (int32_t)(k[j] & wmask) : 0;  // inclusive prefix of the step's weights
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, sum, o);
      if (l >= o) sum += y;
    }
    // a piece: the words from lane l to the one before the next head
    const unsigned later = l < 31 ? hb & (0xffffffffu << (l + 1)) : 0u;
    const int end = later ? __ffs(later) - 2 : 31;
    int32_t piece = __shfl_sync(0xffffffffu, sum, end);
    const int32_t below = __shfl_up_sync(0xffffffffu, sum, 1);
    if (l > 0) piece -= below;
    const int64_t pos = at + __popc(hb & ((1u << l) - 1u));  // this lane's pair when it is a head
    if (head) {
      adjc[pos] = (int32_t)(p & cmask);
      if (later) adjwc[pos] = piece;
      else atomicAdd(&adjwc[pos], piece);  // may go on in the next step
      const int32_t d = (int32_t)(p >> bits);
      if (q == none || (int32_t)(q >> bits) != d) xadjc[d] = pos;
    } else if (l == 0 && valid) {
      atomicAdd(&adjwc[at - 1], piece);  // goes on from the step before
    }
    at += __popc(hb);
  }
}

// Row starts of the empty coarse rows (-1 so far): that of the next non-empty
// row, found in the sorted words.
__global__ void k_ct_xadj(int32_t nc, int64_t mc, const uint64_t* __restrict__ key, const int64_t* d_n, int shift,
                          int64_t* xadjc) {
  const int64_t n = *d_n;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= nc; r += (int64_t)gridDim.x * blockDim.x) {
    if (r < nc && xadjc[r] >= 0) continue;
    int64_t lo = 0, hi = n;
    if (r == nc) lo = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((int64_t)(key[mid] >> shift) < r) lo = mid + 1;
      else hi = mid;
    }
    xadjc[r] = lo < n ? xadjc[key[lo] >> shift] : mc;
  }
}

inline unsigned ct_grid(const Ctx& c, int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)c.num_sms * 8));
}

}  // namespace

bool contract_fits(const Level& F, int bits, int wbits) { return F.m > kCtMinEntries && 2 * bits + wbits <= 64; }

ContractSort contract_sort(Ctx& c, const Level& F, int32_t nc, int bits, int wbits, int32_t* vwc) {
  cudaStream_t st = c.st;
  ContractSort s;
  s.bits = bits;
  s.wbits = wbits;
  int64_t* d_n = c.counters + 7;
  s.d_n = d_n;
  int64_t* d_rows = c.counters + 6;
  int32_t* cnt = c.rank;   // members per coarse vertex, then their next place
  int32_t* perm = c.req;   // the fine vertices with entries, by coarse vertex
  int64_t* pre = c.P64b;   // first stream position of each
  const unsigned gn = ct_grid(c, F.n);
  GM_CUDA(cudaMemsetAsync(cnt, 0, (size_t)nc * sizeof(int32_t), st));
  k_ct_count<<<gn, 256, 0, st>>>(F.n, F.xadj, F.M, F.vw, cnt, vwc); count_launch();
  scan(LoadCnt{cnt}, StoreCnt{cnt}, nc, nullptr, c.scan, st);
  k_ct_copy<<<1, 1, 0, st>>>(c.scan.tile_sums + std::max<int64_t>(1, scan_tiles(nc)), d_rows); count_launch();
  k_ct_place<<<gn, 256, 0, st>>>(F.n, F.xadj, F.M, cnt, perm); count_launch();
  scan(LoadRowDeg{perm, F.xadj}, StoreExcl{pre}, F.n, d_rows, c.scan, st);
  const int passes = (bits + kCtDigitBits - 1) / kCtDigitBits;
  const int db = (bits + passes - 1) / passes;
  const int blocks = (int)std::min<int64_t>(2 * (int64_t)c.num_sms, (F.m + kScTile - 1) / kScTile);
  int32_t* total = reinterpret_cast<int32_t*>(c.P64);
  int32_t* bhist = total + kCtDigits;
  static std::atomic<unsigned long long> attr_done{0};  // one bit per device
  const unsigned long long bit = 1ULL << (c.dev & 63);
  if (!(attr_done.load() & bit)) {
    GM_CUDA(cudaFuncSetAttribute(k_ct_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScSmem)));
    attr_done.fetch_or(bit);
  }
  int cur = 0;
  for (int p = 0; p < passes; p++) {
    const int nb = std::min(db, bits - p * db), ndig = 1 << nb, shift = wbits + bits + p * db;
    GM_CUDA(cudaMemsetAsync(bhist, 0, (size_t)ndig * blocks * sizeof(int32_t), st));
    if (p == 0)
      k_ct_gen<<<blocks * kSplit, kGenThreads, 0, st>>>(F.xadj, F.adj, F.adjw, F.M, perm, pre, d_rows, F.m, bits,
                                                        wbits, nb, c.sort.key[0], bhist, blocks);
    else
      k_ct_hist<<<blocks * kSplit, kGenThreads, 0, st>>>(c.sort.key[cur], s.d_n, shift, nb, bhist, blocks);
    count_launch();
    k_ct_dscan<<<ndig, 128, 0, st>>>(bhist, blocks, total); count_launch();
    k_ct_scatter<<<blocks, kScThreads, sizeof(ScSmem), st>>>(c.sort.key[cur], c.sort.key[cur ^ 1], F.m,
                                                             p == 0 ? nullptr : s.d_n, shift, nb, bhist, total, blocks,
                                                             p == 0 ? d_n : nullptr); count_launch();
    cur ^= 1;
  }
  s.key = c.sort.key[cur];
  s.tiles = (F.m + kApTile - 1) / kApTile;
  k_ct_heads<<<(unsigned)s.tiles, kApThreads, 0, st>>>(s.key, s.d_n, wbits, c.scan.tile_sums); count_launch();
  k_scan_tile_sums<<<1, 1024, 0, st>>>(c.scan.tile_sums, s.tiles); count_launch();
  GM_CUDA(cudaMemcpyAsync(c.h_small + 6, c.scan.tile_sums + s.tiles, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  GM_CUDA(cudaStreamSynchronize(st));
  s.mc = c.h_small[6];
  return s;
}

void contract_rows(Ctx& c, const ContractSort& s, int32_t nc, int64_t* xadj, int32_t* adj, int32_t* adjw) {
  cudaStream_t st = c.st;
  GM_CUDA(cudaMemsetAsync(xadj, 0xFF, ((size_t)nc + 1) * sizeof(int64_t), st));
  if (s.mc > 0) {
    GM_CUDA(cudaMemsetAsync(adjw, 0, (size_t)s.mc * sizeof(int32_t), st));
    k_ct_apply<<<(unsigned)s.tiles, kApThreads, 0, st>>>(s.key, s.d_n, s.bits, s.wbits, c.scan.tile_sums, adj, adjw,
                                                         xadj); count_launch();
  }
  k_ct_xadj<<<ct_grid(c, (int64_t)nc + 1), 256, 0, st>>>(nc, s.mc, s.key, s.d_n, s.bits + s.wbits, xadj);
  count_launch();
  GM_CUDA(cudaGetLastError());
}

}  // namespace gm
