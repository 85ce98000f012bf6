// Device-wide primitives: exclusive scan, stable LSD radix sort of 128-bit
// determinant keys, content hash and sortedness check of key arrays.
#include <cooperative_groups.h>

#include "hci_internal.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int SCAN_BLOCK = 256;
constexpr int SCAN_ITEMS = 16;
constexpr int SCAN_TILE = SCAN_BLOCK * SCAN_ITEMS;

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns the exclusive
// prefix and writes the block total to *total.
__device__ int64_t block_excl_scan(int64_t v, int64_t* total) {
  __shared__ int64_t wsum[32];
  __shared__ int64_t btot;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int64_t inc = warp_incl_scan(v);
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < nw ? wsum[lane] : 0;
    int64_t wi = warp_incl_scan(w);
    if (lane < nw) wsum[lane] = wi - w;
    if (lane == nw - 1) btot = wi;
  }
  __syncthreads();
  int64_t res = inc - v + wsum[warp];
  if (total) *total = btot;
  __syncthreads();
  return res;
}

__global__ void k_scan_reduce(const int64_t* __restrict__ in, int64_t n, int64_t* __restrict__ bsum) {
  int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  int64_t acc = 0;
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    int64_t i = base + (int64_t)k * SCAN_BLOCK + threadIdx.x;
    if (i < n) acc += in[i];
  }
  int64_t tot;
  block_excl_scan(acc, &tot);
  if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// single block: exclusive scan of m block sums in place, total to *total
__global__ void k_scan_sums(int64_t* bsum, int64_t m, int64_t* total) {
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t b = 0; b < m; b += blockDim.x) {
    int64_t i = b + threadIdx.x;
    int64_t v = i < m ? bsum[i] : 0;
    int64_t tot;
    int64_t ex = block_excl_scan(v, &tot);
    if (i < m) bsum[i] = ex + carry;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// bsum: the blocks' sums, or with `raw` set the sums not yet scanned: every
// block then adds up those before its own, and the last one writes the total
__global__ void k_scan_final(const int64_t* __restrict__ in, int64_t* __restrict__ out, int64_t n,
                             const int64_t* __restrict__ bsum, int raw, int64_t* __restrict__ total) {
  int64_t before = 0;
  if (raw) {
    int64_t part = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += SCAN_BLOCK) part += bsum[b];
    block_excl_scan(part, &before);
  } else {
    before = bsum[blockIdx.x];
  }
  // each thread owns SCAN_ITEMS consecutive elements
  int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int64_t v[SCAN_ITEMS];
  int64_t acc = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    int64_t i = base + k;
    v[k] = i < n ? in[i] : 0;
    acc += v[k];
  }
  int64_t tot;
  int64_t ex = block_excl_scan(acc, &tot) + before;
  if (raw && total && threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) *total = before + tot;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    int64_t i = base + k;
    if (i < n) out[i] = ex;
    ex += v[k];
  }
}

// The whole scan by one block, SCAN_ONE_TILE elements at a time, the next
// tile's loads issued before this one's sums: 4.0, 6.3 and 10.4 us for 100,
// 2000 and 8192 elements, 16.7 us for 20000, where two launches take 12.5.
constexpr int SCAN_ONE_ITEMS = 8;
constexpr int SCAN_ONE_TILE = 1024 * SCAN_ONE_ITEMS;
constexpr int64_t SCAN_ONE = 2 * SCAN_ONE_TILE;
constexpr int64_t SCAN_RAW = 4096;   // block sums that every block may add up itself

__global__ void __launch_bounds__(1024) k_scan_one(const int64_t* in, int64_t* out, int n, int64_t* total) {
  int64_t v[SCAN_ONE_ITEMS], w[SCAN_ONE_ITEMS], carry = 0;
  const int at = (int)threadIdx.x * SCAN_ONE_ITEMS;
#pragma unroll
  for (int k = 0; k < SCAN_ONE_ITEMS; ++k) v[k] = at + k < n ? in[at + k] : 0;
  for (int t0 = 0; t0 < n; t0 += SCAN_ONE_TILE) {
    const int i0 = t0 + at;
    int64_t acc = 0, all = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ONE_ITEMS; ++k) {
      const int i = i0 + SCAN_ONE_TILE + k;
      w[k] = i < n ? in[i] : 0;
      acc += v[k];
    }
    int64_t ex = block_excl_scan(acc, &all) + carry;
    carry += all;
#pragma unroll
    for (int k = 0; k < SCAN_ONE_ITEMS; ++k) {
      if (i0 + k < n) out[i0 + k] = ex;
      ex += v[k];
      v[k] = w[k];
    }
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// ---------------------------------------------------------------------------
// radix sort of 128-bit keys, 8-bit digits, stable per pass
// ---------------------------------------------------------------------------
constexpr int RS_BLOCK = 256;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_BLOCK * RS_ITEMS;

__device__ __forceinline__ int digit_of(ulonglong2 k, int word, int shift) {
  // word 0 = low (beta) word, 1 = high (alpha), 2 = hash of both
  const uint64_t w = word == 0 ? k.y : word == 1 ? k.x : group_hash(k);
  return (int)((w >> shift) & 0xFFu);
}

__global__ void k_rs_hist(const ulonglong2* __restrict__ keys, int64_t n, int word, int shift,
                          int64_t* __restrict__ hist, int64_t ntiles, unsigned long long* __restrict__ total) {
  __shared__ int h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * RS_TILE;
  for (int k = 0; k < RS_ITEMS; ++k) {
    int64_t i = base + (int64_t)k * RS_BLOCK + threadIdx.x;
    if (i < n) atomicAdd(&h[digit_of(keys[i], word, shift)], 1);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
  if (h[threadIdx.x]) atomicAdd(&total[threadIdx.x], (unsigned long long)h[threadIdx.x]);
}

// hist[digit][tile] -> the place of the tile's first entry of the digit, in
// place: one block per digit scans its row from the lower digits' totals.
// One launch where a scan of the whole table takes three (9.1 us of kernels
// and three gaps per pass on a selection's 213 tiles, 2.7 us and one so).
__global__ void __launch_bounds__(RS_BLOCK) k_rs_offs(int64_t* __restrict__ hist, int64_t ntiles,
                                                      const unsigned long long* __restrict__ total) {
  const int d = blockIdx.x;
  int64_t below = 0;
  block_excl_scan((int)threadIdx.x < d ? (int64_t)total[threadIdx.x] : 0, &below);
  int64_t* row = hist + (int64_t)d * ntiles;
  for (int64_t t0 = 0; t0 < ntiles; t0 += RS_BLOCK * 4) {
    const int64_t t = t0 + (int64_t)threadIdx.x * 4;
    int64_t v[4], sum = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = t + u < ntiles ? row[t + u] : 0;
      sum += v[u];
    }
    int64_t all = 0;
    int64_t ex = below + block_excl_scan(sum, &all);
    below += all;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (t + u < ntiles) row[t + u] = ex;
      ex += v[u];
    }
  }
}

// One tile to its places, in digit order.  Warp w ranks the 512 consecutive
// entries of its share among the entries of the same digit (one vote per 32
// entries, counters of its own), the tile is put in digit order in shared
// memory, and every digit's run is written as one stretch: written entry by
// entry a tile of random digits touches a sector per entry (8e7 entries of
// 28 bytes: 3.39 ms per pass, 1.07 ms so).
constexpr int RS_WARPS = RS_BLOCK / 32;
constexpr size_t RS_SMEM = (size_t)RS_TILE * 16 + RS_TILE + 256 * 8 + (size_t)RS_WARPS * 256 * 4 + 256 * 4;

__global__ void __launch_bounds__(RS_BLOCK) k_rs_scatter(const ulonglong2* __restrict__ in, ulonglong2* __restrict__ out,
                                                         int64_t n, int word, int shift, const int64_t* __restrict__ offs,
                                                         int64_t ntiles, const double* __restrict__ pin,
                                                         double* __restrict__ pout, const int32_t* __restrict__ qin,
                                                         int32_t* __restrict__ qout) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  ulonglong2* s_key = reinterpret_cast<ulonglong2*>(s_raw);
  int64_t* gbase = reinterpret_cast<int64_t*>(s_raw + (size_t)RS_TILE * 16);   // place of a digit's run less its start here
  int* wcnt = reinterpret_cast<int*>(gbase + 256);                             // [warp][digit]
  int* start = wcnt + RS_WARPS * 256;
  unsigned char* s_dig = reinterpret_cast<unsigned char*>(start + 256);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  const int cnt = n - base < RS_TILE ? (int)(n - base) : RS_TILE;
  for (int k = tid; k < RS_WARPS * 256; k += RS_BLOCK) wcnt[k] = 0;
  __syncthreads();
  int pos[RS_ITEMS];        // rank within the warp's share, then place in the tile
  ulonglong2 key[RS_ITEMS];
  int* mine = wcnt + warp * 256;
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    const int k = warp * (RS_ITEMS * 32) + r * 32 + lane;
    key[r] = k < cnt ? in[base + k] : make_ulonglong2(0, 0);
  }
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    const int k = warp * (RS_ITEMS * 32) + r * 32 + lane;
    const bool valid = k < cnt;
    const int d = valid ? digit_of(key[r], word, shift) : 256;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int before = valid ? mine[d] : 0;
    pos[r] = before + __popc(peers & lt);
    __syncwarp();
    if (valid && (peers & lt) == 0) mine[d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {
    // digit tid: its counts over the warps, its start in the tile
    int run = 0;
    for (int w = 0; w < RS_WARPS; ++w) {
      const int c = wcnt[w * 256 + tid];
      wcnt[w * 256 + tid] = run;
      run += c;
    }
    const int st = (int)block_excl_scan(run, nullptr);
    start[tid] = st;
    gbase[tid] = offs[(int64_t)tid * ntiles + blockIdx.x] - st;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; ++r) {
    const int k = warp * (RS_ITEMS * 32) + r * 32 + lane;
    if (k < cnt) {
      const int d = digit_of(key[r], word, shift);
      pos[r] += start[d] + wcnt[warp * 256 + d];
      s_key[pos[r]] = key[r];
      s_dig[pos[r]] = (unsigned char)d;
    }
  }
  __syncthreads();
  for (int k = tid; k < cnt; k += RS_BLOCK) out[gbase[s_dig[k]] + k] = s_key[k];
  if (pin) {
    double* s_val = reinterpret_cast<double*>(s_raw);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
      const int k = warp * (RS_ITEMS * 32) + r * 32 + lane;
      if (k < cnt) s_val[pos[r]] = pin[base + k];
    }
    __syncthreads();
    for (int k = tid; k < cnt; k += RS_BLOCK) pout[gbase[s_dig[k]] + k] = s_val[k];
  }
  if (qin) {
    int32_t* s_idx = reinterpret_cast<int32_t*>(s_raw);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; ++r) {
      const int k = warp * (RS_ITEMS * 32) + r * 32 + lane;
      if (k < cnt) s_idx[pos[r]] = qin[base + k];
    }
    __syncthreads();
    for (int k = tid; k < cnt; k += RS_BLOCK) qout[gbase[s_dig[k]] + k] = s_idx[k];
  }
}

// lanes whose digit is this lane's, among the `valid` ones, by nine votes
__device__ __forceinline__ unsigned same_digit(int d, bool valid) {
  unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1);
    peers &= (d >> b) & 1 ? m : ~m;
  }
  return peers;
}

// Up to 65536 keys sorted in place in one launch: one thread-block cluster,
// each CTA holding RC_TILE keys in shared memory.  A pass reads the CTA's
// keys into registers, ranks them as k_rs_scatter does, exchanges the CTAs'
// digit counts over distributed shared memory and writes every key straight
// to its place in the CTA that holds it (to global memory in the last pass).
// Two cluster barriers and no launch per pass.  Bound by the latency of a
// pass's dependent steps, about 4 us and 1.3 us more per key that a thread
// holds, so small sets are spread over the CTAs as thinly as they go.  Six
// passes over 48 bits: 2000 keys 115 -> 27 us, 8192 139 -> 31, 65536 139 ->
// 84; past that the passes of whole tiles are as fast.
constexpr int RC_BLOCK = 1024, RC_ITEMS = 8, RC_WARPS = RC_BLOCK / 32;
constexpr int RC_TILE = RC_BLOCK * RC_ITEMS;
constexpr int RC_MAXCTA = 8;                 // the portable cluster size
constexpr int64_t RC_MAX = (int64_t)RC_TILE * RC_MAXCTA;
constexpr size_t RC_SMEM = (size_t)RC_TILE * 16 + (size_t)RC_WARPS * 256 * 2 + 256 * 4 * 2;

__global__ void __launch_bounds__(RC_BLOCK) k_rs_cluster(ulonglong2* __restrict__ keys, int n, int items_log, int bits_b,
                                                         int bits_a) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  ulonglong2* s_key = reinterpret_cast<ulonglong2*>(s_raw);
  uint16_t* wcnt = reinterpret_cast<uint16_t*>(s_raw + (size_t)RC_TILE * 16);   // [warp][digit]
  int* hist = reinterpret_cast<int*>(wcnt + RC_WARPS * 256);                    // this CTA's keys per digit
  int* base = hist + 256;                                                       // place of its first key of a digit
  const cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), nc = (int)cl.num_blocks();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int items = 1 << items_log, tile_log = 10 + items_log, tile = 1 << tile_log;
  const int cnt = max(0, min(n - rank * tile, tile));
  const int npb = (bits_b + 7) / 8, npass = npb + (bits_a + 7) / 8;
  const int k0 = warp * (items * 32) + lane;
  uint16_t* mine = wcnt + warp * 256;
  for (int pass = 0; pass < npass; ++pass) {
    const int word = pass < npb ? 0 : 1, shift = (pass < npb ? pass : pass - npb) * 8;
    ulonglong2 key[RC_ITEMS];
    int pos[RC_ITEMS];
    const ulonglong2* src = pass == 0 ? keys + (int64_t)rank * tile : s_key;
#pragma unroll
    for (int r = 0; r < RC_ITEMS; ++r)
      if (r < items) key[r] = k0 + r * 32 < cnt ? src[k0 + r * 32] : make_ulonglong2(0, 0);
    for (int k = tid; k < RC_WARPS * 128; k += RC_BLOCK) reinterpret_cast<unsigned*>(wcnt)[k] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RC_ITEMS; ++r) {
      if (r >= items) break;
      const bool valid = k0 + r * 32 < cnt;
      const int d = digit_of(key[r], word, shift);
      const unsigned peers = same_digit(d, valid);
      const int before = valid ? mine[d] : 0;
      pos[r] = before + __popc(peers & lt);
      __syncwarp();
      if (valid && (peers & lt) == 0) mine[d] = (uint16_t)(before + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    if (tid < 256) {
      int run = 0;
#pragma unroll 8
      for (int w = 0; w < RC_WARPS; ++w) {
        const int c = wcnt[w * 256 + tid];
        wcnt[w * 256 + tid] = (uint16_t)run;
        run += c;
      }
      hist[tid] = run;
    }
    cl.sync();     // counts of every CTA, and every CTA's keys in registers
    int below = 0, all = 0;
    if (tid < 256) {
      for (int q = 0; q < nc; ++q) {
        const int c = cl.map_shared_rank(hist, q)[tid];
        if (q < rank) below += c;
        all += c;
      }
    }
    const int first = (int)block_excl_scan(all, nullptr);
    if (tid < 256) base[tid] = first + below;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RC_ITEMS; ++r) {
      if (r < items && k0 + r * 32 < cnt) {
        const int d = digit_of(key[r], word, shift);
        const int p = base[d] + mine[d] + pos[r];
        if (pass == npass - 1) keys[p] = key[r];
        else cl.map_shared_rank(s_key, p >> tile_log)[p & (tile - 1)] = key[r];
      }
    }
    cl.sync();     // every key in its place, every count read
  }
}

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x ^= x >> 33; x *= 0xff51afd7ed558ccdull; x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ull; x ^= x >> 33;
  return x;
}

__global__ void k_hash(const ulonglong2* __restrict__ keys, int64_t n, unsigned long long* out) {
  uint64_t hx = 0, hs = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 k = keys[i];
    uint64_t m = mix64(k.x * 0x9E3779B97F4A7C15ull ^ mix64(k.y + (uint64_t)i));
    hx ^= m;
    hs += m;
  }
  for (int o = 16; o; o >>= 1) {
    hx ^= __shfl_xor_sync(0xffffffffu, hx, o);
    hs += __shfl_xor_sync(0xffffffffu, hs, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicXor(&out[0], (unsigned long long)hx);
    atomicAdd(&out[1], (unsigned long long)hs);
  }
}

__global__ void k_check_sorted(const ulonglong2* __restrict__ keys, int64_t n, int* bad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i + 1 < n; i += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 a = keys[i], b = keys[i + 1];
    bool ok = (a.x < b.x) || (a.x == b.x && a.y < b.y);
    if (!ok) atomicOr(bad, 1);
  }
}

}  // namespace

hci_status scan_i64(hci_ctx* ctx, const int64_t* in, int64_t* out, int64_t n, int64_t* total_dev) {
  if (n <= 0) {
    if (total_dev) HCI_CUDA(ctx, cudaMemsetAsync(total_dev, 0, sizeof(int64_t), ctx->st));
    return HCI_OK;
  }
  if (n <= SCAN_ONE) {
    HCI_LAUNCH(k_scan_one, 1, 1024, 0, ctx->st)(in, out, (int)n, total_dev);
    HCI_CUDA(ctx, cudaGetLastError());
    return HCI_OK;
  }
  int64_t nb = (n + SCAN_TILE - 1) / SCAN_TILE;
  HCI_TRY(ensure_buf(ctx, ctx->s_scan, (size_t)nb * sizeof(int64_t)));
  int64_t* bsum = bp<int64_t>(ctx->s_scan);
  const int raw = nb <= SCAN_RAW;
  HCI_LAUNCH(k_scan_reduce, (unsigned)nb, SCAN_BLOCK, 0, ctx->st)(in, n, bsum);
  if (!raw) HCI_LAUNCH(k_scan_sums, 1, 1024, 0, ctx->st)(bsum, nb, total_dev);
  HCI_LAUNCH(k_scan_final, (unsigned)nb, SCAN_BLOCK, 0, ctx->st)(in, out, n, bsum, raw, total_dev);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

hci_status sort_keys(hci_ctx* ctx, uint64_t* keys, uint64_t* tmp, int64_t n, int bits_a, int bits_b) {
  if (n <= 1 || bits_a + bits_b <= 0) return HCI_OK;
  if (n > RC_MAX) return sort_pairs(ctx, keys, tmp, nullptr, nullptr, nullptr, nullptr, n, bits_a, bits_b);
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_rs_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RC_SMEM));
  unsigned ctas = 1;
  int items_log = 0;
  while ((int)ctas < RC_MAXCTA && (int64_t)ctas * RC_BLOCK < n) ctas *= 2;
  while ((int64_t)ctas * (RC_BLOCK << items_log) < n) ++items_log;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(RC_BLOCK);
  cfg.dynamicSmemBytes = RC_SMEM;
  cfg.stream = ctx->st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  hci_count_launch();
  HCI_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_rs_cluster, reinterpret_cast<ulonglong2*>(keys), (int)n, items_log, bits_b,
                                   bits_a));
  return HCI_OK;
}

// stable passes over the digits of `bits[word]` bits of words w0 .. w1
static hci_status radix_passes(hci_ctx* ctx, uint64_t* keys, uint64_t* tmp, double* vals, double* vtmp, int32_t* idx,
                               int32_t* itmp, int64_t n, int w0, int w1, const int* bits) {
  if (n <= 1) return HCI_OK;
  int64_t ntiles = (n + RS_TILE - 1) / RS_TILE;
  int npass = 0;
  for (int word = w0; word <= w1; ++word) npass += (bits[word] + 7) / 8;
  // every pass's digit totals, then the table of one pass
  HCI_TRY(ensure_buf(ctx, ctx->s_hist, (size_t)(ntiles + npass) * 256 * sizeof(int64_t)));
  unsigned long long* total = bp<unsigned long long>(ctx->s_hist);
  int64_t* hist = bp<int64_t>(ctx->s_hist) + (int64_t)npass * 256;
  HCI_CUDA(ctx, cudaMemsetAsync(total, 0, (size_t)npass * 256 * 8, ctx->st));
  ulonglong2* a = reinterpret_cast<ulonglong2*>(keys);
  ulonglong2* b = reinterpret_cast<ulonglong2*>(tmp);
  double* va = vals;
  double* vb = vtmp;
  int32_t* ia = idx;
  int32_t* ib = itmp;
  int passes = 0;
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_rs_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RS_SMEM));
  for (int word = w0; word <= w1; ++word) {
    for (int shift = 0; shift < bits[word]; shift += 8) {
      HCI_LAUNCH(k_rs_hist, (unsigned)ntiles, RS_BLOCK, 0, ctx->st)(a, n, word, shift, hist, ntiles, total + passes * 256);
      HCI_LAUNCH(k_rs_offs, 256, RS_BLOCK, 0, ctx->st)(hist, ntiles, total + passes * 256);
      HCI_LAUNCH(k_rs_scatter, (unsigned)ntiles, RS_BLOCK, RS_SMEM, ctx->st)(a, b, n, word, shift, hist, ntiles, va, vb,
                                                                       ia, ib);
      ulonglong2* t = a; a = b; b = t;
      double* tv = va; va = vb; vb = tv;
      int32_t* ti = ia; ia = ib; ib = ti;
      ++passes;
    }
  }
  HCI_CUDA(ctx, cudaGetLastError());
  if (passes & 1) {
    HCI_CUDA(ctx, cudaMemcpyAsync(keys, tmp, (size_t)n * 16, cudaMemcpyDeviceToDevice, ctx->st));
    if (vals) HCI_CUDA(ctx, cudaMemcpyAsync(vals, vtmp, (size_t)n * 8, cudaMemcpyDeviceToDevice, ctx->st));
    if (idx) HCI_CUDA(ctx, cudaMemcpyAsync(idx, itmp, (size_t)n * 4, cudaMemcpyDeviceToDevice, ctx->st));
  }
  return HCI_OK;
}

hci_status sort_pairs(hci_ctx* ctx, uint64_t* keys, uint64_t* tmp, double* vals, double* vtmp, int32_t* idx,
                      int32_t* itmp, int64_t n, int bits_a, int bits_b) {
  const int bits[3] = {bits_b, bits_a, 0};
  return radix_passes(ctx, keys, tmp, vals, vtmp, idx, itmp, n, 0, 1, bits);
}

// Grouping needs the order of the keys' hash only: 4 passes over 32 bits
// where the keys of (44e,44o) determinants take 12 over 88.  Bits: at least
// 16 times as many hashes as pairs, so that runs of several keys are rare
// (2e7 targets: one in 200), and an even number of passes, so that the last
// one ends in `keys`.
hci_status group_pairs(hci_ctx* ctx, uint64_t* keys, uint64_t* tmp, double* vals, double* vtmp, int32_t* idx,
                       int32_t* itmp, int64_t n, int* bits) {
  *bits = n <= (1 << 12) ? 16 : n <= ((int64_t)1 << 28) ? 32 : 48;
  const int b[3] = {0, 0, *bits};
  return radix_passes(ctx, keys, tmp, vals, vtmp, idx, itmp, n, 2, 2, b);
}

hci_status hash_keys(hci_ctx* ctx, const uint64_t* keys, int64_t n, uint64_t* hash_host) {
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  unsigned long long* d = bp<unsigned long long>(ctx->s_counter);
  HCI_CUDA(ctx, cudaMemsetAsync(d, 0, 16, ctx->st));
  if (n > 0)
    HCI_LAUNCH(k_hash, grid_for(n, 256, ctx->nsm * 8), 256, 0, ctx->st)(reinterpret_cast<const ulonglong2*>(keys), n, d);
  unsigned long long hv[2];
  HCI_CUDA(ctx, cudaMemcpyAsync(hv, d, 16, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  *hash_host = (uint64_t)hv[0] * 31ull + (uint64_t)hv[1] + (uint64_t)n * 0x9E3779B97F4A7C15ull;
  return HCI_OK;
}

hci_status check_sorted(hci_ctx* ctx, const uint64_t* keys, int64_t n, int* ok_host) {
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  int* d = reinterpret_cast<int*>(bp<char>(ctx->s_counter) + 32);
  HCI_CUDA(ctx, cudaMemsetAsync(d, 0, sizeof(int), ctx->st));
  if (n > 1)
    HCI_LAUNCH(k_check_sorted, grid_for(n, 256, ctx->nsm * 8), 256, 0, ctx->st)(reinterpret_cast<const ulonglong2*>(keys), n, d);
  int bad = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&bad, d, sizeof(int), cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  *ok_host = bad ? 0 : 1;
  return HCI_OK;
}
