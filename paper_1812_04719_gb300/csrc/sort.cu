// Stable LSD radix sort of (64-bit key, int32 value) pairs, digits of at most 8
// bits.
//
// Replaces the distributed hypercube quicksort of Alg. 1's check-point sort (Sec. 3.3.1,
// Table 3) on one GPU: equal keys keep their input order, so the payload is
// "scattered" exactly as in Table 3.  The item count may live on the device
// (n_dev); the host passes an upper bound for the launch shapes.
//
// Per digit pass: (1) per-tile digit histograms [digit][tile], (2) one CTA per
// digit scans its row over the tiles (exclusive, coalesced) and writes the
// digit's total, (3) a stable scatter.  The scatter bounds a pass: a tile's warps
// rank their own consecutive items against counters of their own (no barrier
// between the rounds), one scan over the warps places them, and the tile leaves
// sorted through shared memory, so that runs of one digit are written together.
// One million 48-bit keys (6 passes): 22 -> 14 us per scatter against rounds
// of 256 items with five barriers each, 226 -> 132 us the whole call, which no
// longer copies its input (the passes alternate between two buffers so that the
// last one writes the output).
#include "stiv_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;                    // items per thread per tile
constexpr int kTile = kThreads * kItems;     // 2048 items per tile
constexpr int kRadix = 256;
constexpr int kWarps = kThreads / 32;
static_assert(kThreads == kRadix, "the scatter scans the digit totals one per thread");

// Exclusive scan of one value per thread over the CTA (kThreads), in a fixed
// order; *total gets the sum.  wsum: kWarps ints of shared memory.
__device__ __forceinline__ int32_t cta_exclusive_scan(int32_t v, int32_t* wsum, int32_t* total) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = v;
  for (int off = 1; off < 32; off <<= 1) {
    int32_t y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  int32_t pre = 0, tot = 0;
  for (int q = 0; q < kWarps; ++q) {
    int32_t s = wsum[q];
    pre += q < w ? s : 0;
    tot += s;
  }
  __syncthreads();
  *total = tot;
  return pre + x - v;
}

__device__ __forceinline__ int64_t load_n(const int64_t* n_dev, int64_t n_max) {
  if (!n_dev) return n_max;
  int64_t n = *n_dev;
  return n < n_max ? n : n_max;
}
__device__ __forceinline__ int tiles_of(int64_t n) { return (int)((n + kTile - 1) / kTile); }

// The histogram rows are as long as the items need (known on the device), so
// tiles past the count cost nothing.
__global__ void __launch_bounds__(kThreads) hist_kernel(const uint64_t* keys, const int64_t* n_dev, int64_t n_max,
                                                         int shift, unsigned mask, int32_t* hist) {
  __shared__ int32_t h[kRadix];
  int64_t n = load_n(n_dev, n_max);
  const int nt = tiles_of(n);
  for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    int64_t base = (int64_t)tile * kTile;
    uint64_t k[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      int64_t idx = base + q * kThreads + threadIdx.x;
      k[q] = idx < n ? keys[idx] : 0;
    }
    h[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kItems; ++q)
      if (base + q * kThreads + threadIdx.x < n) atomicAdd(&h[(unsigned)(k[q] >> shift) & mask], 1);
    __syncthreads();
    hist[(int64_t)threadIdx.x * nt + tile] = h[threadIdx.x];
    __syncthreads();
  }
}

// CTA d: exclusive scan of hist[d][0 .. tiles) in place; totals[d] = the sum.
__global__ void __launch_bounds__(kThreads) scan_kernel(int32_t* hist, const int64_t* n_dev, int64_t n_max,
                                                         int32_t* totals) {
  __shared__ int32_t wsum[kWarps];
  const int nt = tiles_of(load_n(n_dev, n_max));
  int32_t* row = hist + (int64_t)blockIdx.x * nt;
  int32_t carry = 0;
  for (int base = 0; base < nt; base += kThreads) {
    int i = base + threadIdx.x;
    int32_t v = i < nt ? row[i] : 0, tot;
    int32_t ex = cta_exclusive_scan(v, wsum, &tot);
    if (i < nt) row[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(kThreads) scatter_kernel(const uint64_t* kin, const int32_t* vin, uint64_t* kout,
                                                            int32_t* vout, const int64_t* n_dev, int64_t n_max,
                                                            int shift, unsigned mask, const int32_t* hist,
                                                            const int32_t* totals) {
  __shared__ uint64_t skey[kTile];
  __shared__ int32_t sval[kTile];
  __shared__ int32_t cnt[kWarps][kRadix];   // per warp: items of each digit, then their first place in the tile
  __shared__ int32_t gbase[kRadix];         // output place of the tile's first item of a digit, less its place in the tile
  __shared__ int32_t wsum[kWarps];
  const int64_t n = load_n(n_dev, n_max);
  const int nt = tiles_of(n);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d = threadIdx.x;
  int32_t tot;
  if ((int)blockIdx.x >= nt) return;
  const int32_t dbase = cta_exclusive_scan(totals[d], wsum, &tot);   // digit d = threadIdx.x
  for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    const int64_t base = (int64_t)tile * kTile;
    const int here = (int)(n - base < kTile ? n - base : kTile);
    uint64_t key[kItems];
    int32_t val[kItems];
    int rank[kItems];
    // warp w: items [w * 256, w * 256 + 256) of the tile, lanes in order
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      int i = w * (32 * kItems) + q * 32 + lane;
      key[q] = i < here ? kin[base + i] : ~0ull;
      val[q] = i < here ? vin[base + i] : 0;
    }
    for (int q = lane; q < kRadix; q += 32) cnt[w][q] = 0;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      const bool valid = w * (32 * kItems) + q * 32 + lane < here;
      const unsigned dig = (unsigned)(key[q] >> shift) & mask;
      const unsigned peers = digit_peers<8>(dig, valid), below = peers & ((1u << lane) - 1u);
      const int c = valid ? cnt[w][dig] : 0;
      __syncwarp();
      if (valid && !below) cnt[w][dig] = c + __popc(peers);
      rank[q] = c + __popc(below);
      __syncwarp();
    }
    __syncthreads();
    int32_t run = 0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) { int32_t c = cnt[q][d]; cnt[q][d] = run; run += c; }
    const int32_t first = cta_exclusive_scan(run, wsum, &tot);   // place of the digit's first item in the tile
#pragma unroll
    for (int q = 0; q < kWarps; ++q) cnt[q][d] += first;
    gbase[d] = dbase + hist[(int64_t)d * nt + tile] - first;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kItems; ++q)
      if (w * (32 * kItems) + q * 32 + lane < here) {
        const int at = cnt[w][(unsigned)(key[q] >> shift) & mask] + rank[q];
        skey[at] = key[q];
        sval[at] = val[q];
      }
    __syncthreads();
    for (int i = threadIdx.x; i < here; i += kThreads) {
      const uint64_t k = skey[i];
      const int64_t pos = (int64_t)gbase[(unsigned)(k >> shift) & mask] + i;
      kout[pos] = k;
      vout[pos] = sval[i];
    }
    __syncthreads();
  }
}

}  // namespace

size_t stiv_sort_scratch_impl(int64_t n) {
  int64_t ntiles = (n + kTile - 1) / kTile;
  if (ntiles < 1) ntiles = 1;
  return sizeof(int32_t) * (size_t)(kRadix * ntiles + kRadix) + 256;
}

// Sorts n (or *n_dev if given, <= n) pairs of kin/vin into kout/vout, through
// ktmp/vtmp (n each, distinct from both; may be kin/vin themselves for an odd
// number of passes).  kin/vin are only read when they are not the temporaries.
int stiv_sort_pairs_impl(cudaStream_t st, int64_t n, int key_bits, const uint64_t* kin, const int32_t* vin,
                         uint64_t* kout, int32_t* vout, uint64_t* ktmp, int32_t* vtmp, void* scratch,
                         size_t scratch_bytes, const int64_t* n_dev) {
  if (n < 0 || key_bits < 0 || key_bits > 64) return STIV_ERR_ARG;
  int64_t ntiles = (n + kTile - 1) / kTile;
  if (ntiles < 1) ntiles = 1;
  if (scratch_bytes < stiv_sort_scratch_impl(n)) return STIV_ERR_ARG;
  int32_t* hist = (int32_t*)scratch;
  int32_t* totals = hist + (size_t)kRadix * ntiles;
  int passes = (key_bits + 7) / 8;
  if (passes == 0) {
    if (n > 0) {
      STIV_CUDA(STIV_NO_HANDLE, cudaMemcpyAsync(kout, kin, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, st));
      STIV_CUDA(STIV_NO_HANDLE, cudaMemcpyAsync(vout, vin, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, st));
    }
    return STIV_OK;
  }
  if (passes % 2 == 0 && (ktmp == kin || vtmp == vin)) return STIV_ERR_ARG;   // the first pass would write its input
  const int bits = (key_bits + passes - 1) / passes;
  // an upper bound n may be far above the count on the device: at most four CTAs
  // per SM, each taking the tiles of its stride
  const unsigned grid = (unsigned)(ntiles < 4 * 152 ? ntiles : 4 * 152);
  const uint64_t* ka = kin;
  const int32_t* va = vin;
  for (int ps = 0; ps < passes; ++ps) {
    const int shift = bits * ps;
    const int left = key_bits - shift;
    const unsigned mask = (1u << (left < bits ? left : bits)) - 1u;
    uint64_t* kb = (passes - 1 - ps) % 2 == 0 ? kout : ktmp;
    int32_t* vb = (passes - 1 - ps) % 2 == 0 ? vout : vtmp;
    hist_kernel<<<grid, kThreads, 0, st>>>(ka, n_dev, n, shift, mask, hist);
    STIV_LAUNCH(STIV_NO_HANDLE);
    scan_kernel<<<kRadix, kThreads, 0, st>>>(hist, n_dev, n, totals);
    STIV_LAUNCH(STIV_NO_HANDLE);
    scatter_kernel<<<grid, kThreads, 0, st>>>(ka, va, kb, vb, n_dev, n, shift, mask, hist, totals);
    STIV_LAUNCH(STIV_NO_HANDLE);
    ka = kb;
    va = vb;
  }
  return STIV_OK;
}

// The sort of a caller's arrays, which may overlap (sorting in place): with an odd
// number of passes the first one writes the output, and with none (key_bits 0) the
// keys' copy does, so an overlapping input is copied to the temporaries before.
int stiv_sort_user_impl(cudaStream_t st, int64_t n, int key_bits, const uint64_t* kin, const int32_t* vin,
                        uint64_t* kout, int32_t* vout, uint64_t* kt, int32_t* vt, void* scratch, size_t scratch_bytes) {
  if (key_bits < 0 || key_bits > 64) return STIV_ERR_ARG;
  const char* in[2] = {(const char*)kin, (const char*)vin};
  const char* out[2] = {(const char*)kout, (const char*)vout};
  const size_t len[2] = {sizeof(uint64_t) * (size_t)n, sizeof(int32_t) * (size_t)n};
  bool overlap = false;
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 2; ++b) overlap = overlap || (in[a] < out[b] + len[b] && out[b] < in[a] + len[a]);
  const int passes = (key_bits + 7) / 8;
  if (overlap && (passes % 2 == 1 || passes == 0)) {
    STIV_CUDA(STIV_NO_HANDLE, cudaMemcpyAsync(kt, kin, len[0], cudaMemcpyDeviceToDevice, st));
    STIV_CUDA(STIV_NO_HANDLE, cudaMemcpyAsync(vt, vin, len[1], cudaMemcpyDeviceToDevice, st));
    kin = kt;
    vin = vt;
  }
  return stiv_sort_pairs_impl(st, n, key_bits, kin, vin, kout, vout, kt, vt, scratch, scratch_bytes, nullptr);
}

extern "C" size_t stiv_sort_scratch_bytes(int64_t n) {
  if (n < 0) n = 0;
  return ((stiv_sort_scratch_impl(n) + 15) & ~(size_t)15) + sizeof(uint64_t) * (size_t)n + sizeof(int32_t) * (size_t)n + 64;
}

extern "C" int stiv_sort_pairs(void* stream, int64_t n, int32_t key_bits, const uint64_t* keys_in,
                               const int32_t* vals_in, uint64_t* keys_out, int32_t* vals_out,
                               void* scratch, size_t scratch_bytes) {
  if (n < 0 || (n > 0 && (!keys_in || !vals_in || !keys_out || !vals_out || !scratch))) return STIV_ERR_ARG;
  if (n == 0) return STIV_OK;
  size_t need = stiv_sort_scratch_impl(n);
  if (scratch_bytes < stiv_sort_scratch_bytes(n)) return STIV_ERR_ARG;
  uint64_t* kt = (uint64_t*)((char*)scratch + ((need + 15) & ~(size_t)15));
  int32_t* vt = (int32_t*)(kt + n);
  return stiv_sort_user_impl((cudaStream_t)stream, n, key_bits, keys_in, vals_in, keys_out, vals_out, kt, vt, scratch,
                             need);
}
