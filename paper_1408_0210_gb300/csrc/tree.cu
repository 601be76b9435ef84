// tree.cu -- octree bin/sort of the points (Section 3.3: uniform 2^D-tree
// with kappa + 1 levels; leaves are the 8^kappa boxes of level kappa).
//
// Leaf coordinate floor((x - lo) * (2^kappa / L)) clamped to [0, 2^kappa - 1],
// Morton key with the x bit lowest, then a stable LSD radix sort of the keys
// (8-bit digits; a block ranks its tile warp by warp with __match_any_sync so
// that equal digits keep their input order), leaf offsets from the sorted
// keys and the gather of sorted FP64 coordinates plus FP32 coordinates
// relative to the leaf centre.
#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>

#include "internal.h"

namespace eifmm {
namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;  // 2048 keys per block

// The sort moves (key, index) pairs through LSD passes of at most 8 bits, the
// 3 depth bits spread evenly.  A pass is three launches: digit counts per tile of
// RS_TILE keys (the first pass's come with the keys), the scan of each digit's
// row of counts, and the scatter, which ranks its tile in shared memory and
// writes it in digit order (runs of neighbours instead of single words).
// The passes alternate between an array of 8-byte pairs and the output arrays
// (keys and indices apart), which the last one writes; the first takes the
// indices as positions.  2^20 points, depth 5: the sort into kept arrays 174 ->
// 153 us with its launches and its one read-back (separate words, 13 launches
// before), 127 us with the keys below.
constexpr int RS_DIGITS = 256;
enum RsFormat { kRsKeys = 0, kRsPairs = 1, kRsSplit = 2 };

// Order of doubles as integers; a NaN lies beyond the infinities.  Bounds are
// made with the zero that is nearer to the outside.
inline __host__ __device__ long long ordered(long long bits) { return bits ^ ((bits >> 63) & 0x7fffffffffffffffll); }
struct KeyBox {
  double lo[3], scale;
  long long olo[3], ohi[3];  // ordered bounds
  int shift;                 // scale = 2^shift, |shift| <= 1000 (so that denormals give 0), or INT_MIN
  bool origin;               // lo = 0
};
KeyBox key_box(const double lo[3], double L, int depth) {
  KeyBox b;
  b.scale = ldexp(1.0, depth) / L;
  b.origin = true;
  for (int a = 0; a < 3; ++a) {
    const double l = lo[a] == 0.0 ? -0.0 : lo[a], hi = lo[a] + L, h = hi == 0.0 ? 0.0 : hi;
    b.lo[a] = lo[a];
    long long u;
    memcpy(&u, &l, 8);
    b.olo[a] = ordered(u);
    memcpy(&u, &h, 8);
    b.ohi[a] = ordered(u);
    b.origin = b.origin && lo[a] == 0.0;
  }
  int e;
  b.shift = frexp(b.scale, &e) == 0.5 && abs(e) < 1000 ? e - 1 : INT_MIN;
  return b;
}

// Keys of a tile of points and the tile's counts of the first digit.  The FP64
// pipe (two lanes a cycle and SM) bounds it as soon as it takes part: the bounds
// are compared as integers, the truncation takes the upper words, and the
// difference and the product are left out where they change nothing (a cube at
// the origin, an edge that is a power of two).  2^20 points: 39 us
// before, the whole sort 153 -> 127 us.
__global__ void __launch_bounds__(RS_THREADS)
k_keys(const double* __restrict__ xyz, int64_t n, const __grid_constant__ KeyBox box, int depth, uint32_t mask,
       uint32_t* __restrict__ keys, uint32_t* __restrict__ counts, int nblocks, int* __restrict__ bad) {
  __shared__ uint32_t h[RS_DIGITS];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int nmax = (1 << depth) - 1;
#pragma unroll 4
  for (int j = 0; j < RS_ITEMS; ++j) {
    const int64_t i = (int64_t)blockIdx.x * RS_TILE + j * RS_THREADS + threadIdx.x;
    if (i >= n) break;
    int c[3];
    bool out = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double x = xyz[3 * i + a];
      const long long o = ordered(__double_as_longlong(x));
      out = out || o < box.olo[a] || o > box.ohi[a];
      // (x - lo) * scale: a subtraction then a product, never fused, truncated
      // toward zero and clamped to [0, nmax] (NaN gives 0); truncation equals
      // floor wherever the clamp leaves the value unchanged.
      int up = box.shift;
      if (!box.origin) x = __dsub_rn(x, box.lo[a]);
      if (box.shift == INT_MIN) {
        x = __dmul_rn(x, box.scale);
        up = 0;
      }
      // the 20 leading fraction bits hold the integer part of anything below 2^20
      const bool nan = (__double_as_longlong(x) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
      const int hw = __double2hiint(x), e = ((hw >> 20) & 0x7ff) - 1023 + up;
      const int v = ((hw & 0xfffff) | 0x100000) >> (20 - min(max(e, 0), 20));
      c[a] = hw < 0 || e < 0 || nan ? 0 : (e > 19 ? nmax : min(v, nmax));
    }
    if (out) atomicAdd(bad, 1);
    const uint32_t k = (uint32_t)morton_encode(c[0], c[1], c[2], depth);
    keys[i] = k;
    atomicAdd(&h[k & mask], 1u);
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

template <int IN>
__global__ void __launch_bounds__(RS_THREADS)
k_rs_count(const uint32_t* __restrict__ kin, const uint2* __restrict__ pin, int64_t n, int shift, uint32_t mask,
           uint32_t* __restrict__ counts, int nblocks) {
  __shared__ uint32_t h[RS_DIGITS];
  h[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j) {
    const int64_t p = (int64_t)blockIdx.x * RS_TILE + j * RS_THREADS + threadIdx.x;
    if (p < n) atomicAdd(&h[((IN == kRsPairs ? pin[p].x : kin[p]) >> shift) & mask], 1u);
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of one value per thread over the block; *total receives the
// block's sum.
template <int THREADS>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();  // ws may still be read by a previous call
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t u = lane < THREADS / 32 ? ws[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, u, o);
      if (lane >= o) u += y;
    }
    ws[lane] = u;
  }
  __syncthreads();
  *total = ws[THREADS / 32 - 1];
  return x - v + (w > 0 ? ws[w - 1] : 0u);
}

// Exclusive scan of a digit's counts over the tiles, one block per digit; the
// digit's total goes to total[digit] (the scatter scans the 256 totals itself).
constexpr int SC_THREADS = 1024;
__global__ void __launch_bounds__(SC_THREADS)
k_rs_rows(uint32_t* __restrict__ counts, int nblocks, uint32_t* __restrict__ total) {
  uint32_t* row = counts + (int64_t)blockIdx.x * nblocks;
  uint32_t run = 0;
  for (int b0 = 0; b0 < nblocks; b0 += SC_THREADS) {
    const int b = b0 + threadIdx.x;
    const uint32_t v = b < nblocks ? row[b] : 0u;
    uint32_t t;
    const uint32_t x = block_excl_scan<SC_THREADS>(v, &t);
    if (b < nblocks) row[b] = run + x;
    run += t;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = run;
}

template <int IN, int OUT>
__global__ void __launch_bounds__(RS_THREADS)
k_rs_scatter(const uint32_t* __restrict__ kin, const int32_t* __restrict__ vin, const uint2* __restrict__ pin,
             uint2* __restrict__ pout,
             uint32_t* __restrict__ kout, int32_t* __restrict__ vout, int64_t n, int shift, uint32_t mask,
             const uint32_t* __restrict__ rows, const uint32_t* __restrict__ total, int nblocks) {
  __shared__ uint32_t wc[RS_WARPS][RS_DIGITS + 1];
  __shared__ uint32_t s_pos[RS_DIGITS];  // global position of the tile's position 0 in a digit's order
  __shared__ uint32_t s_loc[RS_DIGITS];  // first tile position of a digit
  __shared__ uint2 s_pair[RS_TILE];
  for (int i = threadIdx.x; i < RS_WARPS * (RS_DIGITS + 1); i += RS_THREADS) (&wc[0][0])[i] = 0;
  uint32_t all;
  const uint32_t base = block_excl_scan<RS_THREADS>(total[threadIdx.x], &all);
  const uint32_t row = rows[(int64_t)threadIdx.x * nblocks + blockIdx.x];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t wbase = (int64_t)blockIdx.x * RS_TILE + (int64_t)w * (32 * RS_ITEMS);
  uint2 e[RS_ITEMS];
  uint32_t rank[RS_ITEMS];
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j) {
    const int64_t p = wbase + j * 32 + lane;
    e[j] = make_uint2(0u, 0u);
    if (p < n) e[j] = IN == kRsPairs ? pin[p] : make_uint2(kin[p], IN == kRsSplit ? (uint32_t)vin[p] : (uint32_t)p);
  }
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j) {
    const bool valid = wbase + j * 32 + lane < n;
    const int d = valid ? (int)((e[j].x >> shift) & mask) : RS_DIGITS;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const uint32_t old = wc[w][d];
    __syncwarp();
    if (lane == __ffs(peers) - 1) wc[w][d] = old + __popc(peers);
    __syncwarp();
    rank[j] = old + __popc(peers & lt);
  }
  __syncthreads();
  {
    const int d = threadIdx.x;
    uint32_t run = 0;
    for (int ww = 0; ww < RS_WARPS; ++ww) {
      const uint32_t t = wc[ww][d];
      wc[ww][d] = run;
      run += t;
    }
    uint32_t cnt;
    const uint32_t loc = block_excl_scan<RS_THREADS>(run, &cnt);
    s_loc[d] = loc;
    s_pos[d] = base + row - loc;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < RS_ITEMS; ++j)
    if (wbase + j * 32 + lane < n) {
      const int d = (int)((e[j].x >> shift) & mask);
      s_pair[s_loc[d] + wc[w][d] + rank[j]] = e[j];
    }
  __syncthreads();
  const int64_t left = n - (int64_t)blockIdx.x * RS_TILE;
  const int cnt = left < RS_TILE ? (int)left : RS_TILE;
  for (int i = threadIdx.x; i < cnt; i += RS_THREADS) {
    const uint2 q = s_pair[i];
    const uint32_t pos = s_pos[(q.x >> shift) & mask] + (uint32_t)i;
    if (OUT == kRsPairs) {
      pout[pos] = q;
    } else {
      kout[pos] = q.x;
      vout[pos] = (int32_t)q.y;
    }
  }
}

// Scratch of the sort of n points: an array of pairs, counts, totals.
struct SortBuffers {
  uint2* pairs;
  uint32_t* counts;
  uint32_t* total;
};

// keys, perm: the sorted keys and input positions of the points xyz.
eifmm_status sort_points(const double* xyz, int64_t n, const double lo[3], double L, int depth, uint32_t* keys,
                         int32_t* perm, const SortBuffers& b, int* bad, cudaStream_t s) {
  const int nb = (int)((n + RS_TILE - 1) / RS_TILE), T = RS_THREADS;
  const int bits = 3 * depth, passes = (bits + 7) / 8;
  // pass p writes the output arrays when an even number of passes follows it;
  // the unsorted keys start where the first pass does not write
  auto to_split = [&](int p) { return (passes - 1 - p) % 2 == 0; };
  uint32_t* k0 = to_split(0) ? (uint32_t*)b.pairs : keys;
  int shift = 0;
  for (int p = 0; p < passes; ++p) {
    const int w = bits / passes + (p < bits % passes ? 1 : 0);
    const uint32_t mask = (1u << w) - 1u;
    const bool split = to_split(p);
    if (p == 0)
      k_keys<<<nb, T, 0, s>>>(xyz, n, key_box(lo, L, depth), depth, mask, k0, b.counts, nb, bad);
    else if (split)
      k_rs_count<kRsPairs><<<nb, T, 0, s>>>(nullptr, b.pairs, n, shift, mask, b.counts, nb);
    else
      k_rs_count<kRsSplit><<<nb, T, 0, s>>>(keys, nullptr, n, shift, mask, b.counts, nb);
    EIFMM_CHECK_LAUNCH();
    k_rs_rows<<<RS_DIGITS, SC_THREADS, 0, s>>>(b.counts, nb, b.total);
    EIFMM_CHECK_LAUNCH();
    if (p == 0 && split)
      k_rs_scatter<kRsKeys, kRsSplit><<<nb, T, 0, s>>>(k0, nullptr, nullptr, nullptr, keys, perm, n, shift, mask,
                                                      b.counts, b.total, nb);
    else if (p == 0)
      k_rs_scatter<kRsKeys, kRsPairs><<<nb, T, 0, s>>>(k0, nullptr, nullptr, b.pairs, nullptr, nullptr, n, shift, mask,
                                                      b.counts, b.total, nb);
    else if (split)
      k_rs_scatter<kRsPairs, kRsSplit><<<nb, T, 0, s>>>(nullptr, nullptr, b.pairs, nullptr, keys, perm, n, shift, mask,
                                                       b.counts, b.total, nb);
    else
      k_rs_scatter<kRsSplit, kRsPairs><<<nb, T, 0, s>>>(keys, perm, nullptr, b.pairs, nullptr, nullptr, n, shift, mask,
                                                       b.counts, b.total, nb);
    EIFMM_CHECK_LAUNCH();
    shift += w;
  }
  return EIFMM_OK;
}

// off[b] = first sorted position whose key is at least b (b = 0..nleaf;
// off[nleaf] = n): one thread per leaf, a binary search over the sorted
// keys, so runs of empty leaves cost no more than full ones.
__global__ void k_leaf_off(const uint32_t* __restrict__ skeys, int64_t n,
                           int64_t nleaf, int32_t* __restrict__ off) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b > nleaf) return;
  int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(skeys + mid) < b) lo = mid + 1;
    else hi = mid;
  }
  off[b] = (int32_t)lo;
}

// Leaf-centre coordinates lo_a + (2 c + 1) l_kappa of the 2^depth cells
// per axis are formed once per block in shared memory ([3][2^depth]).
__global__ void k_gather_points(const double* __restrict__ xyz,
                                const int32_t* __restrict__ perm,
                                const uint32_t* __restrict__ skeys, int64_t n,
                                double lo0, double lo1, double lo2, double lk,
                                int depth, double* __restrict__ x,
                                double* __restrict__ y, double* __restrict__ z,
                                float* __restrict__ lx, float* __restrict__ ly,
                                float* __restrict__ lz) {
  extern __shared__ double s_ctr[];
  const int nc = 1 << depth;
  for (int t = threadIdx.x; t < 3 * nc; t += blockDim.x) {
    const int a = t >> depth, c = t & (nc - 1);
    const double lo = a == 0 ? lo0 : (a == 1 ? lo1 : lo2);
    s_ctr[t] = lo + (2.0 * c + 1.0) * lk;
  }
  __syncthreads();
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int64_t i = perm[p];
  const double px = xyz[3 * i], py = xyz[3 * i + 1], pz = xyz[3 * i + 2];
  int c[3];
  morton_decode(skeys[p], depth, c);
  x[p] = px;
  y[p] = py;
  z[p] = pz;
  lx[p] = (float)(px - s_ctr[c[0]]);
  ly[p] = (float)(py - s_ctr[nc + c[1]]);
  lz[p] = (float)(pz - s_ctr[2 * nc + c[2]]);
}

// cnt[0]: their number, cnt[kFullest]: the points of the fullest, in a cache line of
// its own, which an SM reads from L1; next to the counter every read went to L2
// between the additions.  Tree build of 2^20 points in 2^27 leaves: 3.75 ms; next to
// the counter 4.18, with a reduction in every warp, empty ones too, 4.69.
constexpr int kFullest = 32;
constexpr int kCounters = 2 + kFullest;  // points outside the cube, then cnt
__global__ void k_nonempty(const int32_t* __restrict__ off, int64_t nleaf,
                           int32_t* __restrict__ list, int32_t* __restrict__ cnt) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int n = b < nleaf ? off[b + 1] - off[b] : 0;
  if (n == 0) return;
  list[atomicAdd(cnt, 1)] = (int32_t)b;
  if (n > cnt[kFullest]) atomicMax(cnt + kFullest, n);  // an old count only costs an atomic more
}

struct SortScratch {
  std::mutex m;
  unsigned char* p = nullptr;
  size_t cap = 0;
};
SortScratch& sort_scratch(int dev) {
  static SortScratch s[64];
  return s[dev & 63];
}

}  // namespace

eifmm_status build_pointset(const double* xyz, int64_t n, const double lo[3],
                            double L, int depth, cudaStream_t s, PointSet* ps) {
  ps->n = n;
  const int64_t nleaf = (int64_t)1 << (3 * depth);
  const int64_t nn = n > 0 ? n : 1;
  // one slab for the point set, one for the sort's scratch (256-byte aligned parts)
  auto take = [](size_t& off, size_t bytes) { const size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  size_t off = 0;
  const size_t o_perm = take(off, nn * 4), o_keys = take(off, nn * 4), o_loff = take(off, (nleaf + 1) * 4),
               o_ne = take(off, nleaf * 4), o_x = take(off, nn * 8), o_y = take(off, nn * 8),
               o_z = take(off, nn * 8), o_lx = take(off, nn * 4), o_ly = take(off, nn * 4),
               o_lz = take(off, nn * 4);
  unsigned char* slab = nullptr;
  EIFMM_TRY(dalloc(&slab, off));
  ps->slab = slab;
  ps->perm = (int32_t*)(slab + o_perm);
  ps->keys = (uint32_t*)(slab + o_keys);
  ps->leaf_off = (int32_t*)(slab + o_loff);
  ps->nonempty = (int32_t*)(slab + o_ne);
  ps->x = (double*)(slab + o_x);
  ps->y = (double*)(slab + o_y);
  ps->z = (double*)(slab + o_z);
  ps->lx = (float*)(slab + o_lx);
  ps->ly = (float*)(slab + o_ly);
  ps->lz = (float*)(slab + o_lz);

  const int nblocks = (int)((n + RS_TILE - 1) / RS_TILE);
  const int nb1 = nblocks > 0 ? nblocks : 1;
  size_t soff = 0;
  const size_t o_pairs = take(soff, nn * 8), o_cnt = take(soff, (size_t)RS_DIGITS * nb1 * 4),
               o_tot = take(soff, RS_DIGITS * 4), o_bad = take(soff, kCounters * sizeof(int));
  // The sort's scratch is kept per device between builds (grown on demand,
  // held until the process exits); builds on one device take turns on it.
  int dev = 0;
  EIFMM_CUDA(cudaGetDevice(&dev));
  SortScratch& sc = sort_scratch(dev);
  std::unique_lock<std::mutex> hold(sc.m);
  if (sc.cap < soff) {
    dfree(sc.p);
    sc.p = nullptr;
    sc.cap = 0;
    EIFMM_TRY(dalloc(&sc.p, soff));
    sc.cap = soff;
  }
  unsigned char* scratch = sc.p;
  const SortBuffers sb{(uint2*)(scratch + o_pairs), (uint32_t*)(scratch + o_cnt), (uint32_t*)(scratch + o_tot)};
  int* dbad = (int*)(scratch + o_bad);
  EIFMM_CUDA(cudaMemsetAsync(dbad, 0, kCounters * sizeof(int), s));

  if (n > 0) EIFMM_TRY(sort_points(xyz, n, lo, L, depth, ps->keys, ps->perm, sb, dbad, s));
  k_leaf_off<<<(unsigned)((nleaf + 1 + 255) / 256), 256, 0, s>>>(ps->keys, n, nleaf, ps->leaf_off);
  EIFMM_CHECK_LAUNCH();
  if (n > 0) {
    const double lk = L * ldexp(1.0, -(depth + 1));
    k_gather_points<<<(unsigned)((n + 255) / 256), 256, (size_t)3 * sizeof(double) << depth, s>>>(
        xyz, ps->perm, ps->keys, n, lo[0], lo[1], lo[2], lk, depth, ps->x, ps->y,
        ps->z, ps->lx, ps->ly, ps->lz);
    EIFMM_CHECK_LAUNCH();
  }
  k_nonempty<<<(unsigned)((nleaf + 255) / 256), 256, 0, s>>>(ps->leaf_off, nleaf, ps->nonempty, dbad + 1);
  EIFMM_CHECK_LAUNCH();
  int hb[kCounters] = {};
  EIFMM_CUDA(cudaMemcpyAsync(hb, dbad, kCounters * sizeof(int), cudaMemcpyDeviceToHost, s));
  EIFMM_CUDA(cudaStreamSynchronize(s));
  ps->n_nonempty = hb[1];
  ps->max_leaf = hb[1 + kFullest];
  if (hb[0] != 0) {
    set_error("eifmm_tree_build: " + std::to_string(hb[0]) +
              " coordinates lie outside the cube [lo, lo + L]^3");
    return EIFMM_EINVAL;
  }
  return EIFMM_OK;
}

void free_pointset(PointSet* ps) {
  dfree(ps->slab);
  *ps = PointSet();
}

}  // namespace eifmm

// ---------------------------------------------------------------------------
// Allocation-free variant of the bin/sort (eifmm_tree_sort_static).  Its
// radix-sort scratch lives in a file-scope device array: the pairs of the
// passes between (8 bytes per point), the digit counts of the tiles (256 x 4
// bytes per 2048 points), their totals and an error counter.
// ---------------------------------------------------------------------------
namespace eifmm {
namespace {
constexpr int64_t kStaticMax = EIFMM_STATIC_SORT_MAX_POINTS;
constexpr int64_t kStaticBlocks = (kStaticMax + RS_TILE - 1) / RS_TILE;
constexpr size_t kOffPairs = 0;
constexpr size_t kOffCounts = kOffPairs + (size_t)kStaticMax * 8;
constexpr size_t kOffTotal = kOffCounts + (size_t)RS_DIGITS * kStaticBlocks * 4;
constexpr size_t kOffBad = kOffTotal + RS_DIGITS * 4;
constexpr size_t kStaticBytes = kOffBad + 256;
static_assert(kStaticBytes == EIFMM_STATIC_SORT_SCRATCH_BYTES, "scratch size of the header");

__device__ __align__(256) unsigned char g_sort_scratch[kStaticBytes];

constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices] = {};
std::mutex g_scratch_mu;

// Device address of the scratch on the current device, looked up once per
// device (the host-side symbol is only a stand-in, never a device address).
eifmm_status static_scratch(unsigned char** out) {
  int dev = 0;
  EIFMM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("eifmm_tree_sort_static: device ordinal out of range");
    return EIFMM_EUNSUPPORTED;
  }
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_sort_scratch);
    if (e != cudaSuccess || p == nullptr) {
      set_error(std::string("eifmm_tree_sort_static: cudaGetSymbolAddress failed: ") +
                cudaGetErrorString(e));
      return EIFMM_ECUDA;
    }
    g_scratch_addr[dev] = p;
  }
  *out = (unsigned char*)g_scratch_addr[dev];
  return EIFMM_OK;
}
}  // namespace
}  // namespace eifmm

using namespace eifmm;

extern "C" eifmm_status eifmm_tree_sort_static(const double* xyz, int64_t n, const double lo[3],
                                               double L, int depth, uint32_t* keys_out,
                                               int32_t* perm_out, int32_t* leaf_off_out,
                                               eifmm_stream stream) {
  if (!lo || !leaf_off_out || n < 0 || (n > 0 && (!xyz || !keys_out || !perm_out)) || depth < 2 ||
      depth > kMaxLevel || !(L > 0.0)) {
    set_error("eifmm_tree_sort_static: invalid argument");
    return EIFMM_EINVAL;
  }
  if (n > kStaticMax) {
    set_error("eifmm_tree_sort_static: n = " + std::to_string(n) + " exceeds the static scratch limit of " +
              std::to_string(kStaticMax) + " points (EIFMM_STATIC_SORT_MAX_POINTS)");
    return EIFMM_EINVAL;
  }
  unsigned char* base = nullptr;
  EIFMM_TRY(static_scratch(&base));
  cudaStream_t s = (cudaStream_t)stream;
  const SortBuffers sb{(uint2*)(base + kOffPairs), (uint32_t*)(base + kOffCounts), (uint32_t*)(base + kOffTotal)};
  int* bad = (int*)(base + kOffBad);
  // the error counter must start at zero on every call
  EIFMM_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
  const int64_t nleaf = (int64_t)1 << (3 * depth);
  if (n > 0) EIFMM_TRY(sort_points(xyz, n, lo, L, depth, keys_out, perm_out, sb, bad, s));
  k_leaf_off<<<(unsigned)((nleaf + 1 + 255) / 256), 256, 0, s>>>(keys_out, n, nleaf, leaf_off_out);
  EIFMM_CHECK_LAUNCH();
  int hbad = 0;
  EIFMM_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  EIFMM_CUDA(cudaStreamSynchronize(s));
  if (hbad != 0) {
    set_error("eifmm_tree_sort_static: " + std::to_string(hbad) +
              " coordinates lie outside the cube [lo, lo + L]^3");
    return EIFMM_EINVAL;
  }
  return EIFMM_OK;
}
