// m2l_crt.cu -- the dense products of Algorithm 3 (M2M, M2L, L2L and the Delta^t
// of step 6) in FP64 accuracy on the tcgen05 tensor cores.  The M2L (step 4):
//
//   g^I_{m'} = sum_{J in I(I)} sum_l T^delta_{m'l} W^J_l
//
// The FP64 pipes of this GPU run at 1/72 of the FP32 rate, the tensor cores
// 25 times above the latter.  The sum is therefore formed exactly in integers by
// residues (K. Ozaki, Y. Uchino, T. Imamura, "Ozaki Scheme II", 2025): W is
// rounded to 59-bit integers with a power-of-two scale (M2L: one per level and
// right-hand side), row m' of every T^delta with one scale per row, chosen so
// that the whole sum over offsets and l stays below M / 2 in magnitude, M the
// product of 14 pairwise coprime moduli up to 513 (125.2 bits).  Modulo m_i
// both operands are integers in [-256, 256], exact in BF16; a product is at
// most 2^16, so 240 terms are summed exactly in the FP32 accumulator (below
// 2^24, every partial sum an integer).  The running sums are kept modulo m_i
// in FP32 registers, and the Chinese remainder theorem gives the exact integer
// sum, rounded once to FP64.
//
// Accuracy: the sum of |T| over a row and all offsets has 66 bits, the largest
// |W| of a level 58, and the sum itself adds no rounding.  Against quad
// precision g errs by 1.0e-16 to 6e-16 (2-norm; 1/r at eps 1e-4 to 1e-7, levels
// 2 to 4, uniform and clustered points), the FP64 sum on the FP64 pipes by
// 1.2e-15 to 6.8e-15 and the FP32 pairs by about 2e-12; for the config-3 kernel
// (eps 1e-6) 4.2e-13 against 6.6e-12 in FP64.
// Uneven problems keep their digits (weak_bits): 1/r, 2,000 charges
// of order 1 that cancel in one corner and 1e-12 elsewhere, depth 7: f differs from
// the FP64 pipes' by 4e-16 in the median; with one part by 1.8e-14.
//
// Seven launches cover all levels: largest |W| per level, box and column; the
// residue planes of W; those of the second part (weak_bits), if any; the residue
// GEMMs; those of the second part; the reconstruction; the weak boxes.  At 2^20 points,
// depth 5: eps 1e-6 (d = 193) 4.65 + 0.2 ms, where the FP32 pairs took 144 ms; eps
// 1e-4 (d = 126) 2.3 ms, where the FP64 pipes took 195 ms; eps 1e-7 (d = 256)
// 8.0 ms (202 ms in FP32 pairs).  The GEMM issues 14 times the method's products,
// 13% of them zero (189 offsets for 165 pairs per box), 1.8 PFLOP/s at d = 193 and 1.45
// at d = 126.  It is bound by shared memory: the operands of an MMA (4 KB of W, 32
// bytes per column), the operator residues written there and the windows take 1,870
// cycles per offset at 128 bytes a cycle (d = 193; 1,790 measured), 830 at d = 126
// (860 measured); the MMAs take 1,350 and 510.
//
// M2M, L2L and Delta^t are the same sums over the 8 children, the parent and the
// box itself, without shifts.  A sum stays within one parent or box, and so does
// its scale: a weak box next to strong ones keeps all its bits.  Delta^t is formed
// explicitly in double-double and takes 18 moduli (160.5 bits): its entries reach
// 2^34 / |A| at eps 1e-7, and the product cancels by as much.  K(x, X) Delta^t l then errs by 1.6e-16 to 9e-16
// (1/r, eps 1e-4 to 1e-7) where the FP64 triangular solves err by 2.3e-16 to 2.7e-15
// (config-3 at 1e-6: 1.4e-12 and 7.2e-12).  At 2^20 points, depth 5, d = 193, on
// the FP64 pipes before: M2M 3.0 -> 0.27 ms, L2L 5.1 -> 0.33 ms, Delta^t 3.5 -> 0.36
// ms; 512 leaves: Delta^t 1.73 -> 0.037 ms.  They are bound by their passes over
// the residues (28 bytes an entry) and, for small levels, by their launches.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "m2l_crt.h"
#include "tc_ptx.cuh"

namespace eifmm {
namespace {

constexpr int kMods = 14;     // M2L, M2M, L2L: 125.2 bits
constexpr int kBoxMods = 18;  // Delta^t: 160.5 bits
__host__ __device__ constexpr int crt_mod(int i) {
  return i == 0 ? 513 : i == 1 ? 512 : i == 2 ? 511 : i == 3 ? 509 : i == 4 ? 505 : i == 5 ? 503 : i == 6 ? 499
       : i == 7 ? 491 : i == 8 ? 487 : i == 9 ? 481 : i == 10 ? 479 : i == 11 ? 473 : i == 12 ? 467 : i == 13 ? 463
       : i == 14 ? 461 : i == 15 ? 457 : i == 16 ? 449 : 443;
}
// |W| 2^b < 2^wbits; sum over offsets and l of |T| 2^a < 2^rowbits; wbits +
// rowbits + 1 (the sign) is the size of the product of the moduli.
constexpr int kWBits = 58, kRowBits = 66, kEntryBits = 60;  // |T| 2^a < 2^60
// The M2L's scale is the level's, so a target box all of whose sources are far
// weaker than the level's strongest box would get them in few bits.  A box is weak
// where the exponent of the largest |W| of its interaction list lies more than
// weak_bits(d) below that of the level's.  Up to there the rounding of W, 2^-58 of
// the level's largest, adds less to the sum than FP64 rounds its d terms and more to
// (exact sums, clustered points, lists of one or two occupied boxes: 0.76 of the FP64
// pipes' error at the limit for d = 17, 0.44 for d = 64, 0.21 for d = 128).
//
// The weak boxes of a tile with kTileWork or more occupied sources take a second
// part: the same sum over what the rounding left of W, in units 2^-kRestBits times
// smaller, added in FP64.  Fewer sources, and boxes weaker than kMaxWeak, are summed
// on the FP64 pipes source by source: most weak boxes lie at the rim of a cluster
// and have one or two (2^20 points of a mixture of 8 Gaussians, d = 193: 308 boxes on 112 of
// the 256 tiles of level 5).  Even problems have no weak box; the second part then
// has no items, and its three kernels end at once.
__host__ __device__ __forceinline__ int weak_bits(int d) {
  int b = 4;
  while (d >= 4) ++b, d >>= 2;
  return b;
}
constexpr int kRestBits = 59, kMaxWeak = 60;
constexpr unsigned kTileWork = 128;
constexpr int kBoxWBits = 55, kBoxRowBits = 104;
constexpr int kMaxSteps = 15;  // k-steps of 16 terms in one accumulation: 240 terms

// Target tile of a CTA: 8 x 4 x 4 boxes of one parity class (128 rows of the
// MMA).  The sources of class c' for one y-shift and all x- and z-shifts lie
// in a window of 10 x 4 x 6 boxes of that class's grid, kept in shared memory
// as [k8][z][y][x][8 terms]: the canonical K-major layout without swizzle,
// where a shift by one box is a shift of the start address by 16 bytes (x) or
// 640 bytes (z), and the 8-row groups (y, z) lie 160 bytes apart.  One window
// serves the 5 to 9 offsets of its class and y-shift, so that W is read from
// L2 3.6 times less often than with one tile per offset.
constexpr int kTX = 8, kTY = 4, kTZ = 4;
constexpr int kWinRows = (kTX + 2) * kTY * (kTZ + 2);       // 240
constexpr uint32_t kWinStep = 2u * kWinRows * 16u;          // bytes of one k-step of a window
constexpr int kWins = 2;
constexpr int kMaxStages = 8;
constexpr int kDrainWarps = 8;
constexpr int kThreads = 32 * (kDrainWarps + 3);
constexpr int kAccCols = 256;  // TMEM columns of an accumulator
constexpr uint32_t kSmemMax = 227u * 1024u;
constexpr uint32_t kSmemBars = 512;

// One level (or one slab and column range of it) of a launch.
struct CrtLv {
  CrtMode mode;
  int slevel, ds, ncs;       // source boxes: level, rank, parity classes (8, or 1: the whole grid)
  int tlevel, d, nct;        // target boxes: level, rank, classes
  int K, Nt, NT;             // padded terms, columns per tile, column tiles
  int nw, nslots;            // windows per target class, operators of the stack
  int wbits;                 // size of the integers of W
  int h;                     // boxes per axis of a class (of source and target alike)
  int z0, nz, sz0, snz;      // planes of target boxes, planes of source boxes held
  int r0, Rc, R, G;          // columns r0 .. r0 + Rc of R, offset groups
  int nchunk, n0, ks0, ks1;  // chunks of K: n0 of ks0 k-steps, then ks1 k-steps each
  uint16_t ng[8][8];         // accumulations of a tile of class [ct], group [grp]
  unsigned pinv;             // 2^32 over the pairs of coefficients of a row, rounded up
  unsigned item0, pl0, rc0, mx0;  // first block of this level in each of the launches
  const double* W;
  double* g;
  const double* add;         // added to the sum, same layout as g (may be null)
  __nv_bfloat16* planes;     // [mod][r][class][k8][z][y][x][8]
  int16_t* res;              // [mod][group][r][class][z][y][x][NT Nt]
  const __nv_bfloat16* img;  // [mod][slot][column tile][k8][Nt][8]
  const double* colscale;    // per column m': M 2^(-96 - a)
  // [unit][R] bits of the largest |W| of a unit, the boxes that share a scale:
  // source box J is in unit J >> sshift, target box I takes unit I >> tshift
  unsigned long long* wmax;
  int sshift, tshift;
  // weak boxes of the M2L: null elsewhere
  unsigned long long* bmax;  // [box][R] bits of the largest |W| of a box
  unsigned char* weak;       // [box][R] 1 or, beyond kMaxWeak, 2 for a weak target box
  unsigned* need;            // [r][class][tile z, y, x] occupied sources of the tile's weak boxes (1)
  const double* T;           // the operators, [slot][l < ds][m' < d]
  int pstep;                 // class grids of the first part in `planes`
  int64_t rstep;             // entries of the first part in `res`
};
constexpr int kMaxLv = kMaxLevel - 1;
struct CrtArgs {
  int nlev, stages;
  unsigned items, plane_blocks, rebuild_blocks;
  // [0] some tile takes the second part, [1] weak boxes in `list` (null: not the M2L)
  unsigned* any;
  uint2* list;  // (level << 16 | column, box)
  uint32_t stage_b, win_b;
  int* err;
  CrtLv lv[kMaxLv];
};
struct CrtMaps {
  CUtensorMap m[kMaxLv];
};
// 2^(32 NW) y_i / m_i, y_i the inverse of M / m_i modulo m_i, for NM moduli
template <int NM, int NW>
struct CrtK {
  uint32_t k[NM][NW];
};

// K / 16 k-steps in chunks of five and three: three chunks of five or five of
// three fill an accumulation (kMaxSteps), and a chunk of five keeps the MMAs of
// a step (5 x 104 cycles at N = 208) above the cost of its wait and commit.
void split_chunks(CrtLv* v) {
  const int n = v->K / 16;
  int a = n / 5;
  if (n < 8) {
    v->ks0 = n <= 5 ? n : n - 3;
    v->ks1 = 3;
    v->n0 = 1;
    v->nchunk = n <= 5 ? 1 : 2;
    return;
  }
  while ((n - 5 * a) % 3) --a;  // reaches a = 2 n mod 3 at the latest, and 10 <= n where that is 2
  v->ks0 = 5;
  v->ks1 = 3;
  v->n0 = a;
  v->nchunk = a + (n - 5 * a) / 3;
}
__host__ __device__ __forceinline__ int chunk_ksteps(const CrtLv& v, int c) { return c < v.n0 ? v.ks0 : v.ks1; }

// bits of shifts s + 1 in {0, 1, 2} along one axis whose child offset
// 2 s + cs - ct is at most one box (the near field)
__host__ __device__ __forceinline__ int near_bits(int cs, int ct) { return cs == ct ? 2 : (cs > ct ? 3 : 6); }

// The (sz, sx) shifts of class cs and y-shift sy + 1 that belong to the
// interaction list of class ct: bit 3 (sz + 1) + sx + 1.
__host__ __device__ __forceinline__ int combo_mask(int ct, int cs, int sy1) {
  if (!((near_bits((cs >> 1) & 1, (ct >> 1) & 1) >> sy1) & 1)) return 0x1ff;
  const int nx = near_bits(cs & 1, ct & 1), nz = near_bits((cs >> 2) & 1, (ct >> 2) & 1);
  const int m = ((nz & 1) ? nx : 0) | ((nz & 2) ? nx << 3 : 0) | ((nz & 4) ? nx << 6 : 0);
  return 0x1ff & ~m;
}

// Window w of target class ct: source class, y-shift + 1, mask of (sz, sx)
// shifts (bit 3 (sz + 1) + sx + 1) and the operator of the shift (0, 0).
struct Win {
  int cs, sy1, mask, slot;
};
__host__ __device__ __forceinline__ Win window_of(const CrtLv& v, int ct, int w) {
  Win o;
  if (v.mode == kCrtM2L) {
    // by the parity of the offset: the CTAs of all target classes read (nearly)
    // the same operators at the same time
    o.cs = ct ^ (w / 3);
    o.sy1 = w % 3;
    o.mask = combo_mask(ct, o.cs, o.sy1);
    o.slot = (2 * (o.sy1 - 1) + ((o.cs >> 1) & 1) - ((ct >> 1) & 1) + 3) * 7 + (o.cs & 1) - (ct & 1) + 3 +
             ((o.cs >> 2) - (ct >> 2) + 3) * 49;
  } else {  // no shift: the 8 children of a box (M2M), its parent (L2L), itself (box)
    o.cs = v.mode == kCrtM2M ? w : (v.mode == kCrtL2L ? 0 : ct);
    o.slot = v.mode == kCrtM2M ? w : (v.mode == kCrtL2L ? ct : 0);
    o.sy1 = 1;
    o.mask = 0x10;
  }
  return o;
}

// Accumulations of kMaxSteps k-steps at most that the windows of a tile fill.
int accumulations(const CrtLv& v, int ct, int grp) {
  int n = 1, acc = 0;
  for (int w = grp * v.nw / v.G; w < (grp + 1) * v.nw / v.G; ++w)
    for (int c = 0; c < v.nchunk; ++c)
      for (int m = window_of(v, ct, w).mask; m; m &= m - 1) {
        const int ks = chunk_ksteps(v, c);
        if (acc + ks > kMaxSteps) ++n, acc = 0;
        acc += ks;
      }
  return n;
}

// Morton key of box (x, y, z) of class c of nc
__device__ __forceinline__ int64_t class_box(int nc, int c, int x, int y, int z) {
  const int64_t m = morton_encode(x, y, z, 0);
  return nc == 1 ? m : 8 * m + c;
}

// scale exponent of a column from the bits of its largest |W|
__device__ __forceinline__ bool w_finite(unsigned long long bits) { return bits < 0x7ff0000000000000ull; }
__device__ __forceinline__ int w_exp(unsigned long long bits, int wbits) {
  return wbits - ((int)(bits >> 52) - 1022);
}
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// W 2^b rounded to an integer, |W| 2^b <= 2^58
__device__ __forceinline__ long long w_int(double w, int b) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(w) & 0x7fffffffffffffffull;
  const int e = (int)(u >> 52);
  unsigned long long m = u & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = (e ? e : 1) - 1075 + b;  // at most 6
  if (sh >= 0) m <<= sh;
  else m = sh < -54 ? 0 : (m + (1ull << (-sh - 1))) >> -sh;
  return w < 0.0 ? -(long long)m : (long long)m;
}

// What the rounding left, (w 2^b - v) 2^kRestBits rounded to an integer, at most
// 2^58 in magnitude; the terms are formed modulo 2^64.
__device__ __forceinline__ long long w_rest(double w, int b, long long v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(w) & 0x7fffffffffffffffull;
  const int e = (int)(u >> 52);
  unsigned long long m = u & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int sh = (e ? e : 1) - 1075 + b + kRestBits;  // at most 65
  if (sh >= 0) m = sh < 64 ? m << sh : 0;
  else m = sh < -54 ? 0 : (m + (1ull << (-sh - 1))) >> -sh;
  return (long long)((w < 0.0 ? 0 - m : m) - ((unsigned long long)v << kRestBits));
}

// 2^(12 j) modulo crt_mod(i), in [-m/2, m/2]
__host__ __device__ constexpr int limb_res(int i, int j) {
  int r = 1;
  for (int k = 0; k < 12 * j; ++k) r = 2 * r % crt_mod(i);
  return r > crt_mod(i) / 2 ? r - crt_mod(i) : r;
}

// Two integers, |v| <= 2^60, as FP32 limbs of 12 bits, the last one signed.
struct Limbs {
  float2 l[5];
};
__device__ __forceinline__ Limbs limbs_of(long long v0, long long v1) {
  Limbs o;
#pragma unroll
  for (int j = 0; j < 5; ++j)
    o.l[j] = j < 4 ? make_float2((float)((int)(v0 >> (12 * j)) & 0xfff), (float)((int)(v1 >> (12 * j)) & 0xfff))
                   : make_float2((float)(int)(v0 >> 48), (float)(int)(v1 >> 48));
  return o;
}
// Residues of both modulo crt_mod(I), in [-m/2, m/2], as two BF16.  The sum of
// the limbs' residues is exact (below 2^22.1); its quotient by m is off by less
// than 6e-4 before it is rounded, and a multiple of 1 / m for odd m comes no
// nearer to a half than 1 / 2m >= 9.7e-4 (for m = 512 it is exact).  Residues up to
// 256 are exact in BF16, whose bits are the upper half of FP32's.
template <int I>
__device__ __forceinline__ uint32_t residue2(const Limbs& v) {
  constexpr float fm = (float)crt_mod(I), inv = 1.0f / fm;
  float2 u = v.l[0];
  u = __ffma2_rn(v.l[1], make_float2(limb_res(I, 1), limb_res(I, 1)), u);
  u = __ffma2_rn(v.l[2], make_float2(limb_res(I, 2), limb_res(I, 2)), u);
  u = __ffma2_rn(v.l[3], make_float2(limb_res(I, 3), limb_res(I, 3)), u);
  u = __ffma2_rn(v.l[4], make_float2(limb_res(I, 4), limb_res(I, 4)), u);
  const float2 k = __fadd2_rn(__ffma2_rn(u, make_float2(inv, inv), make_float2(12582912.0f, 12582912.0f)),
                              make_float2(-12582912.0f, -12582912.0f));
  const float2 r = __ffma2_rn(k, make_float2(-fm, -fm), u);
  return __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632);
}

__device__ __forceinline__ int find_level(const CrtArgs& a, unsigned CrtLv::*first, unsigned b) {
  int q = 0;
  while (q + 1 < a.nlev && b >= a.lv[q + 1].*first) ++q;
  return q;
}

// ---------------------------------------------------------- largest |W| --
// A block takes 32 boxes of a column, eight lanes a box with eight loads in flight
// (one box after the other by a warp took 34 us at any size).  One maximum per
// unit: the whole level (M2L, and each box), eight children or one box.
constexpr int kMaxBoxes = 32;
__device__ __forceinline__ unsigned long long max_over(unsigned long long m, int lanes) {
  for (int o = 1; o < lanes; o <<= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, o);
    m = x > m ? x : m;
  }
  return m;
}
__global__ void __launch_bounds__(256) k_crt_max(const __grid_constant__ CrtArgs a) {
  const CrtLv& v = a.lv[find_level(a, &CrtLv::mx0, blockIdx.x)];
  const unsigned b = blockIdx.x - v.mx0, q = b / (unsigned)v.Rc;
  const int r = v.r0 + (int)(b - q * v.Rc), ds = v.ds, t = threadIdx.x;
  const int64_t first = (int64_t)q * kMaxBoxes;  // the boxes of a level are a multiple of 32
  const double* w = v.W + ((first + (t >> 3)) * v.R + r) * ds;
  unsigned long long m = 0;
#pragma unroll 8
  for (int l = t & 7; l < ds; l += 8) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(w[l]) & 0x7fffffffffffffffull;
    m = x > m ? x : m;
  }
  m = max_over(m, 8);
  __shared__ unsigned long long sm[kMaxBoxes];
  if ((t & 7) == 0) sm[t >> 3] = m;
  __syncthreads();
  if (t >= kMaxBoxes) return;
  m = sm[t];
  if (v.bmax) v.bmax[(first + t) * v.R + r] = m;
  const int per = v.sshift >= 5 ? kMaxBoxes : 1 << v.sshift;
  m = max_over(m, per);
  if (t % per != 0) return;
  unsigned long long* out = v.wmax + ((first + t) >> v.sshift) * v.R + r;
  if (v.sshift <= 5) *out = m;
  else if (m > *(volatile unsigned long long*)out) atomicMax(out, m);
}

// ------------------------------------------------------- residue planes --
// A block takes 8 boxes along x of one class, z, y and column, a warp each: their
// W is rounded to integers once, and every thread writes 8 terms of one box for
// all moduli (16-byte stores, 128 contiguous bytes per 8 threads).  Both the
// rounding and the residues stay off the FP64 and the conversion units: 262,144
// points, 7 columns, d = 193, the leaf level 694 -> 455 us (3.5 TB/s).
template <int I, int NM>
__device__ __forceinline__ void store_residues(const Limbs (&v)[4], __nv_bfloat16* dst, int64_t step) {
  if constexpr (I < NM) {
    *reinterpret_cast<uint4*>(dst) =
        make_uint4(residue2<I>(v[0]), residue2<I>(v[1]), residue2<I>(v[2]), residue2<I>(v[3]));
    store_residues<I + 1, NM>(v, dst + step, step);
  }
}
// Index in `need` of the tile of target box (x, y, z) of class ct, column r.
__device__ __forceinline__ int need_index(const CrtLv& v, int r, int ct, int z, int y, int x) {
  const int nx = (v.h + kTX - 1) / kTX, ny = (v.h + kTY - 1) / kTY, nz = (v.nz + kTZ - 1) / kTZ;
  return (((r * v.nct + ct) * nz + (z - v.z0) / kTZ) * ny + y / kTY) * nx + x / kTX;
}
// Whether box (x, y, z) of class ct is weak, by its warp.  The
// boxes of its interaction list are the children of the 27 neighbours of its
// parent (x, y, z) but its own neighbours.
__device__ __forceinline__ void mark_weak(const CrtArgs& a, const CrtLv& v, int r, int ct, int z, int y, int x,
                                          int64_t box, unsigned long long level) {
  // by the exponents (subnormals count as the smallest one); most boxes have a
  // strong source among the first 32 looked at
  const int top = (int)(level >> 52), enough = top - weak_bits(v.ds);
  int most = -1;
  unsigned occupied = 0;
  bool strong = !w_finite(level);
  for (int i = threadIdx.x & 31; i < 224 && !strong; i += 32) {
    const int n = i >> 3, c = i & 7, dx = n % 3 - 1, dy = n / 3 % 3 - 1, dz = n / 9 - 1;
    const bool in = i < 216 && x + dx >= 0 && y + dy >= 0 && z + dz >= 0 && x + dx < v.h && y + dy < v.h &&
                    z + dz < v.h;
    const int ox = 2 * dx + (c & 1) - (ct & 1), oy = 2 * dy + ((c >> 1) & 1) - ((ct >> 1) & 1),
              oz = 2 * dz + (c >> 2) - (ct >> 2);
    unsigned long long m = 0;
    if (in && (abs(ox) > 1 || abs(oy) > 1 || abs(oz) > 1))
      m = v.bmax[class_box(8, c, x + dx, y + dy, z + dz) * v.R + r];
    occupied += __popc(__ballot_sync(0xffffffffu, m > 0));
    if (m > 0) most = max(most, (int)(m >> 52));
    strong = __any_sync(0xffffffffu, most >= enough);
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) != 0) return;
  const bool weak = !strong && occupied > 0;
  v.weak[box * v.R + r] = !weak ? 0 : top - most > kMaxWeak ? 2 : 1;
  if (!weak) return;
  a.list[atomicAdd(a.any + 1, 1u)] = make_uint2((unsigned)(&v - a.lv) << 16 | (unsigned)r, (unsigned)box);
  if (top - most > kMaxWeak) return;
  const unsigned old = atomicAdd(v.need + need_index(v, r - v.r0, ct, z, y, x), occupied);
  if (old < kTileWork && old + occupied >= kTileWork) *a.any = 1;
}
// One block of the planes; REST: of the second part.
template <int NM, bool REST>
__device__ __forceinline__ void planes_block(const CrtArgs& a, unsigned block, long long* s_w) {
  const CrtLv& v = a.lv[find_level(a, &CrtLv::pl0, block)];
  unsigned b = block - v.pl0;
  const int h = v.h, nxs = (h + 7) / 8;
  const int xs = (int)(b % nxs);
  b /= nxs;
  const int y = (int)(b % h);
  b /= h;
  const int zs = (int)(b % v.snz);
  b /= v.snz;
  const int cls = (int)(b % v.ncs), r = (int)(b / v.ncs);
  const int z = v.sz0 + zs, K = v.K, ld = K + 1;
  {
    const int bx = threadIdx.x >> 5, x = 8 * xs + bx;
    const int64_t box = x < h ? class_box(v.ncs, cls, x, y, z) : 0;
    const unsigned long long bits = v.wmax[(box >> v.sshift) * v.R + v.r0 + r];
    const bool fin = w_finite(bits);
    const int e = w_exp(fin ? bits : 0, v.wbits);
    const double* w = x < h && fin ? v.W + (box * v.R + v.r0 + r) * v.ds : nullptr;
#pragma unroll 4
    for (int l = threadIdx.x & 31; l < K; l += 32) {
      const long long q = w && l < v.ds ? w_int(w[l], e) : 0;
      s_w[bx * ld + l] = REST && w && l < v.ds ? w_rest(w[l], e, q) : q;
    }
    if (!REST && v.bmax && x < h && z >= v.z0 && z < v.z0 + v.nz) mark_weak(a, v, v.r0 + r, cls, z, y, x, box, bits);
  }
  __syncthreads();
  const int64_t plane = (int64_t)(K / 8) * v.snz * h * h * 8;  // elements of one (mod, r, class)
  for (int u = threadIdx.x; u < K; u += 256) {
    const int bx = u & 7, k8 = u >> 3, x = 8 * xs + bx;
    if (x >= h) continue;
    const long long* q = s_w + bx * ld + 8 * k8;
    Limbs w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = limbs_of(q[2 * j], q[2 * j + 1]);
    __nv_bfloat16* dst = v.planes + (int64_t)((REST ? v.pstep : 0) + r * v.ncs + cls) * plane +
                         ((((int64_t)k8 * v.snz + zs) * h + y) * h + x) * 8;
    store_residues<0, NM>(w, dst, (int64_t)v.Rc * v.ncs * plane);
  }
}
template <int NM>
__global__ void __launch_bounds__(256) k_crt_planes(const __grid_constant__ CrtArgs a) {
  extern __shared__ long long s_w[];  // [8][K + 1]
  planes_block<NM, false>(a, blockIdx.x, s_w);
}
template <int NM>
__global__ void __launch_bounds__(256) k_crt_planes_rest(const __grid_constant__ CrtArgs a) {
  extern __shared__ long long s_w[];
  if (*a.any == 0) return;
  for (unsigned b = blockIdx.x; b < a.plane_blocks; b += gridDim.x) {
    planes_block<NM, true>(a, b, s_w);
    __syncthreads();
  }
}

// -------------------------------------------------------- residue GEMMs --
// Shared-memory descriptor: K-major, no swizzle, version 1.  lbo: bytes from
// the first 8 terms of a k-step to the next 8; sbo: bytes between 8-row groups.
__device__ __forceinline__ uint64_t desc_k(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// D = F32, A and B BF16, both K-major, M = 128
__device__ __forceinline__ uint32_t idesc_bf16(uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
// the KS k-steps of one offset's chunk; n2: descriptor units between k-steps of B
template <int KS>
__device__ __forceinline__ void mma_steps(uint32_t dst, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                          uint32_t n2, uint32_t id, uint32_t acc, uint32_t el) {
#pragma unroll
  for (int kk = 0; kk < KS; ++kk)
    mma_f16_el(dst, alo + kk * (kWinStep >> 4), ahi, blo + kk * n2, bhi, id, kk ? 1u : acc, el);
}

struct Item {
  int q, x0, y0, z0, ct, nt, r, grp, mod, w_beg, w_end;
};
__device__ __forceinline__ Item item_of(const CrtArgs& a, unsigned i) {
  Item o;
  o.q = find_level(a, &CrtLv::item0, i);
  const CrtLv& v = a.lv[o.q];
  unsigned b = i - v.item0;
  auto digit = [&](int n) {
    const unsigned q = b / (unsigned)n, r = b - q * (unsigned)n;
    b = q;
    return (int)r;
  };
  o.x0 = kTX * digit((v.h + kTX - 1) / kTX);
  o.y0 = kTY * digit((v.h + kTY - 1) / kTY);
  o.z0 = v.z0 + kTZ * digit((v.nz + kTZ - 1) / kTZ);
  o.ct = digit(v.nct);
  o.nt = digit(v.NT);
  o.r = digit(v.Rc);
  o.grp = digit(v.G);
  o.mod = (int)b;
  o.w_beg = o.grp * v.nw / v.G;
  o.w_end = (o.grp + 1) * v.nw / v.G;
  return o;
}

// An item of the second part is left out where its tile does not take that.
__device__ __forceinline__ bool left_out(const CrtLv& v, const Item& t) {
  return !__any_sync(0xffffffffu, v.need[need_index(v, t.r, t.ct, t.z0, t.y0, t.x0)] >= kTileWork);
}

// One item: one modulus, one target tile (128 boxes of a class), one column
// tile, one right-hand side, one group of (source class, y-shift) windows.  A
// CTA per SM takes every gridDim-th; each role runs on into the next item, so
// that its operands load and its first sums form while the last one's are
// reduced and written.  Against a CTA per item, 2^20 points: L2L 0.39 -> 0.33 and
// Delta^t 0.45 -> 0.36 ms at d = 193, 0.32 -> 0.27 and 0.34 -> 0.28 at d = 126; the M2L
// about the same there, 0.40 -> 0.36 with 512 leaves.
// Warps 0-7 drain the accumulators, warp 8 streams the operator residues
// (K-chunk of one offset per stage), warp 9 issues the MMAs, warp 10 loads the
// windows.  M = 128 boxes, N = Nt columns m', K in chunks of at most 64 terms.
// Two TMEM accumulators of Nt columns: while one is filled (15 k-steps at
// most), the other is added to the register sums modulo m.
// REST: the second part of the M2L, for the tiles that take it (a launch of its own,
// which ends at once where none does; as more items of one launch their checks took
// 1.2% of the M2L and 6% of the L2L).
template <bool REST>
__global__ void __launch_bounds__(kThreads, 1)
k_crt_gemm(const __grid_constant__ CrtMaps maps, const __grid_constant__ CrtArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // uniform for the compiler: the roles of warps 8 to 10 run converged
  const int wu = (int)__reduce_or_sync(0xffffffffu, (unsigned)warp);
  const int S = a.stages;
  if (REST && *a.any == 0) return;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t s_stage = sbase + kWins * a.win_b;
  uint64_t* bars = (uint64_t*)(smem + kWins * a.win_b + (uint32_t)S * a.stage_b);
  // bfull[8] bempty[8] wfull[kWins] wempty[kWins] afull[2] aempty[2]
  auto bfull = [&](int i) { return smem_u32(&bars[i]); };
  auto bempty = [&](int i) { return smem_u32(&bars[kMaxStages + i]); };
  auto wfull = [&](int i) { return smem_u32(&bars[2 * kMaxStages + i]); };
  auto wempty = [&](int i) { return smem_u32(&bars[2 * kMaxStages + kWins + i]); };
  auto afull = [&](int i) { return smem_u32(&bars[2 * kMaxStages + 2 * kWins + i]); };
  auto aempty = [&](int i) { return smem_u32(&bars[2 * kMaxStages + 2 * kWins + 2 + i]); };
  uint32_t* tslot = (uint32_t*)(bars + 2 * kMaxStages + 2 * kWins + 4);
  volatile int* abort = (volatile int*)(tslot + 1);

  if (tid == 0) {
    for (int i = 0; i < kMaxStages; ++i) {
      mbar_init(bfull(i), 1);
      mbar_init(bempty(i), 1);
    }
    for (int i = 0; i < kWins; ++i) {
      mbar_init(wfull(i), 1);
      mbar_init(wempty(i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(afull(i), 1);
      mbar_init(aempty(i), kDrainWarps);
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __reduce_or_sync(0xffffffffu, *tslot);

  if (wu == 8) {
    // ----------------------------------------- operator residues (B) --
    const uint32_t el = elect_one();
    const uint32_t stage_b = a.stage_b;
    int it = 0, st = 0;
    uint32_t ph = 0, dst = s_stage;
    bool ok = true;
    for (unsigned i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
      const Item t = item_of(a, i);
      const CrtLv& v = a.lv[t.q];
      if (REST && left_out(v, t)) continue;
      const int64_t tile_b = (int64_t)v.K * v.Nt * 2, slot_b = v.NT * tile_b;  // bytes of a column tile, of a slot
      const char* img = (const char*)v.img + (int64_t)t.mod * v.nslots * slot_b + t.nt * tile_b;
      const int n0 = v.n0, ks0 = v.ks0, ks1 = v.ks1, nchunk = v.nchunk;
      for (int w = t.w_beg; w < t.w_end && ok; ++w) {
        const Win wn = window_of(v, t.ct, w);
        const int mask = wn.mask;
        const char* src = img + wn.slot * slot_b;
        for (int c = 0; c < nchunk && ok; ++c) {
          const uint32_t bytes = (uint32_t)(c < n0 ? ks0 : ks1) * 32u * (uint32_t)v.Nt;
#pragma unroll 1
          for (int left = mask; left && ok; left &= left - 1) {
            const int m = __ffs(left) - 1, mz = (11 * m) >> 5;
            const char* from = src + (2 * (m - 3 * mz - 1) + 98 * (mz - 1)) * slot_b;
            if (it >= S) ok = mbar_wait_u(bempty(st), ph ^ 1u, a.err, 11, abort);
            if (ok) {
              if (el) {
                mbar_expect_tx(bfull(st), bytes);
                bulk_g2s(dst, from, bytes, bfull(st));
              }
              __syncwarp();
              ++it;
              dst += stage_b;
              if (++st == S) st = 0, ph ^= 1u, dst = s_stage;
            }
          }
          src += bytes;
        }
      }
    }
    drain_fills(it, S, bars, a.err);
  } else if (wu == 10) {
    // ------------------------------------------------- windows of W (A) --
    const uint32_t el = elect_one();
    int wi = 0, s = 0;
    uint32_t wph = 0;
    bool ok = true;
    for (unsigned i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
      const Item t = item_of(a, i);
      const CrtLv& v = a.lv[t.q];
      if (REST && left_out(v, t)) continue;
      for (int w = t.w_beg; w < t.w_end && ok; ++w) {
        const Win wn = window_of(v, t.ct, w);
        int k0 = 0;
        for (int c = 0; c < v.nchunk; ++c, ++wi) {
          const int ks = chunk_ksteps(v, c);
          if (wi >= kWins && !mbar_wait_u(wempty(s), wph ^ 1u, a.err, 12, abort)) {
            ok = false;
            break;
          }
          if (el) {
            mbar_expect_tx(wfull(s), (uint32_t)ks * kWinStep);
            for (int kk = 0; kk < ks; ++kk)
              tma_load_5d(sbase + (uint32_t)s * a.win_b + (uint32_t)kk * kWinStep, &maps.m[t.q], 8 * (t.x0 - 1),
                          t.y0 + wn.sy1 - 1, t.z0 - 1 - v.sz0, 2 * (k0 + kk),
                          (REST ? v.pstep : 0) + (t.mod * v.Rc + t.r) * v.ncs + wn.cs, wfull(s));
          }
          __syncwarp();
          k0 += ks;
          if (++s == kWins) s = 0, wph ^= 1u;
        }
      }
    }
    drain_fills(wi, kWins, bars + 2 * kMaxStages, a.err);
  } else if (wu == 9) {
    // ----------------------------------------------------- MMA issuer --
    const uint32_t el = elect_one();
    const uint64_t dA = desc_k(sbase, kWinRows * 16u, (kTX + 2) * 16u);
    const uint32_t ahi = (uint32_t)(dA >> 32), stage16 = a.stage_b >> 4, win16 = a.win_b >> 4;
    int st = 0, s = 0, g = 0, acc = 0;
    uint32_t ph = 0, wph = 0, dst = tmem, id = 0, n2 = 0, bhi = 0;
    const uint32_t blo0 = (uint32_t)desc_k(s_stage, 0u, 128u);
    uint32_t blo = blo0;  // with the item's LBO in the upper half
    uint32_t lbo = 0;
    bool ok = true;
    // accumulator g, when the sums of g - 2 have been taken from it
    auto open_acc = [&]() {
      acc = 0;
      dst = tmem + (uint32_t)((g & 1) * kAccCols);
      if (g >= 2) ok = ok && mbar_wait_u(aempty(g & 1), ((g >> 1) - 1) & 1, a.err, 14, abort);
    };
    // the steps of one window whose chunk has KS k-steps.  A loop, not
    // unrolled over the shifts: one warp runs through this code once per window,
    // and fetching it took longer than the MMAs (M2L of 2^20 points, unrolled and
    // so: d = 193 5.14 and 4.86 ms, d = 126 3.29 and 2.33)
    auto window = [&](auto ksc, int mask, uint32_t awin) {
      constexpr int KS = decltype(ksc)::value;
#pragma unroll 1
      for (int left = mask; left; left &= left - 1) {
        const int m = __ffs(left) - 1, mz = (11 * m) >> 5;
        if (acc + KS > kMaxSteps) {  // this accumulator is full
          mma_commit_el(afull(g & 1), el);
          ++g;
          open_acc();
        }
        ok = ok && mbar_wait_u(bfull(st), ph, a.err, 15, abort);
        if (!ok) return;
        tc_fence_after();
        mma_steps<KS>(dst, awin + (uint32_t)(mz * ((kTX + 2) * kTY - 3) + m), ahi, blo | lbo, bhi, n2, id,
                      acc > 0 ? 1u : 0u, el);
        acc += KS;
        mma_commit_el(bempty(st), el);
        blo += stage16;
        if (++st == S) st = 0, ph ^= 1u, blo = blo0;
      }
    };
    for (unsigned i = blockIdx.x; i < a.items && ok; i += gridDim.x) {
      const Item t = item_of(a, i);
      const CrtLv& v = a.lv[t.q];
      if (REST && left_out(v, t)) continue;
      const int n0 = v.n0, ks0 = v.ks0, ks1 = v.ks1, nchunk = v.nchunk;
      const uint64_t dB = desc_k(0, (uint32_t)v.Nt * 16u, 128u);
      lbo = (uint32_t)dB;
      bhi = (uint32_t)(dB >> 32);
      n2 = 2u * (uint32_t)v.Nt;
      id = idesc_bf16((uint32_t)v.Nt);
      open_acc();
      for (int w = t.w_beg; w < t.w_end && ok; ++w) {
        const int mask = window_of(v, t.ct, w).mask;
        for (int c = 0; c < nchunk && ok; ++c) {
          const int ks = c < n0 ? ks0 : ks1;
          ok = mbar_wait_u(wfull(s), wph, a.err, 13, abort);
          if (!ok) break;
          const uint32_t awin = (uint32_t)dA + (uint32_t)s * win16;
          if (ks == 5) window(std::integral_constant<int, 5>(), mask, awin);
          else if (ks == 4) window(std::integral_constant<int, 4>(), mask, awin);
          else if (ks == 3) window(std::integral_constant<int, 3>(), mask, awin);
          else if (ks == 2) window(std::integral_constant<int, 2>(), mask, awin);
          else window(std::integral_constant<int, 1>(), mask, awin);
          if (ok) mma_commit_el(wempty(s), el);
          if (++s == kWins) s = 0, wph ^= 1u;
        }
      }
      if (ok) mma_commit_el(afull(g & 1), el);
      ++g;
    }
  } else if (warp < kDrainWarps) {
    // -------------------------------------------------- residue sums --
    // warp w reads TMEM lanes 32 (w % 4) .. and half w / 4 of the columns
    const int quad = warp & 3, half = warp >> 2;
    const float2 mg = make_float2(12582912.0f, 12582912.0f), ng2 = make_float2(-12582912.0f, -12582912.0f);
    int g = 0;
    bool have = true;
    for (unsigned it = blockIdx.x; it < a.items && have; it += gridDim.x) {
      const Item t = item_of(a, it);
      const CrtLv& v = a.lv[t.q];
      if (REST && left_out(v, t)) continue;
      const int Nt = v.Nt, nh = Nt / 2;
      const float fm = (float)crt_mod(t.mod);
      const float2 inv2 = make_float2(1.0f / fm, 1.0f / fm), m2 = make_float2(-fm, -fm);
      float2 sum[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) sum[j] = make_float2(0.f, 0.f);
      for (int n = v.ng[t.ct][t.grp]; n > 0; --n, ++g) {
        have = mbar_wait_ab(afull(g & 1), (g >> 1) & 1, a.err, 16, abort);
        have = __all_sync(0xffffffffu, have);
        if (!have) break;
        tc_fence_after();
        const uint32_t t0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)((g & 1) * kAccCols + half * nh);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (16 * j < nh) {
            float x[16];
            tmem_ld16(t0 + 16u * j, x);
            // |x| <= 240 2^16 and |sum| < 2^9: x + sum is an exact integer
            // below 2^24; minus the nearest multiple of m (1.5 2^23 rounds to
            // the nearest integer), again exact
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float2 u = __fadd2_rn(make_float2(x[2 * i], x[2 * i + 1]), sum[8 * j + i]);
              const float2 k = __fadd2_rn(__ffma2_rn(u, inv2, mg), ng2);
              sum[8 * j + i] = __ffma2_rn(k, m2, u);
            }
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(aempty(g & 1)) : "memory");
      }
      // row = (z, y, x) of the tile: TMEM lane 32 quad + lane
      const int row = 32 * quad + lane, h = v.h;
      const int x = t.x0 + (row & 7), y = t.y0 + ((row >> 3) & 3), z = t.z0 + (row >> 5);
      if (have && x < h && y < h && z < v.z0 + v.nz) {
        const int N = v.NT * Nt;
        int16_t* out = v.res + (REST ? v.rstep : 0) +
                       ((((((int64_t)t.mod * v.G + t.grp) * v.Rc + t.r) * v.nct + t.ct) * v.nz + (z - v.z0)) * h + y) *
                           (int64_t)h * N +
                       (int64_t)x * N + t.nt * Nt + half * nh;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (8 * j < nh) {
            uint32_t p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              p[i] = ((uint32_t)(int)sum[4 * j + i].x & 0xffffu) | ((uint32_t)(int)sum[4 * j + i].y << 16);
            *reinterpret_cast<uint4*>(out + 8 * j) = make_uint4(p[0], p[1], p[2], p[3]);
          }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

// -------------------------------------------------------- reconstruction --
// G / M modulo 1 = sum_i s_i y_i / m_i modulo 1, in fixed point of NW words (the
// constants' rounding adds at most 2^(14 - 32 NW) of M; G itself is about 2^-10
// of M, 2^-40 for Delta^t, whose terms cancel, with one word more, and down to
// 2^-74 for the first part of a weak target, with two more).
// A thread takes two coefficients; the result is rounded in integers, once (the
// FP64 pipe, at 1/64 of the integer rate, took two thirds of the time: the M2L's 45
// million sums at 262,144 points, 7 columns 1,677 -> 626 us).
constexpr int kRebuild = 128;

// +-(H 2^64 + L) 2^(e - 128) times c, rounded to FP64; c normal and positive
__device__ __forceinline__ double fixed_times(bool neg, unsigned long long H, unsigned long long L, int e, double c) {
  if (H == 0) {
    H = L;
    L = 0;
    e -= 64;
  }
  if (H == 0) return 0.0;
  const int z = __clzll((long long)H);
  if (z) H = (H << z) | (L >> (64 - z));
  const unsigned long long cb = (unsigned long long)__double_as_longlong(c);
  unsigned long long P = __umul64hi(H, (cb << 11) | (1ull << 63));
  // P 2^(e - z) (c's exponent in units of 2^-63): normalise its top bit
  const int up = (long long)P >= 0;
  P <<= up;
  const unsigned long long m = (P >> 11) + ((P >> 10) & 1);
  // value P 2^-64 2^(e - z - up) 2^(ec + 1), ec the exponent of c: P 2^-63 in [1, 2)
  const int E = e - z - up + (int)(cb >> 52) - 1023;
  double y;
  if (E > -1022 && E < 1023) y = __longlong_as_double((long long)(((unsigned long long)(E + 1022) << 52) + m));
  else y = scalbn((double)(long long)m, E - 52);
  return neg ? -y : y;
}

// The signed fraction p (NW words of 32 bits, the lowest first) times 2^e c.
template <int NW>
__device__ __forceinline__ double fraction_times(const unsigned long long (&p)[NW], int e, double c) {
  if constexpr (NW <= 4) {
    unsigned long long H = (p[NW - 1] << 32) | (p[NW - 2] & 0xffffffffull);
    unsigned long long L = (p[NW - 3] << 32) | (NW == 4 ? p[0] & 0xffffffffull : 0ull);
    const bool neg = (long long)H < 0;
    if (neg) {
      L = ~L + 1;
      H = ~H + (L == 0);
    }
    return fixed_times(neg, H, L, e, c);
  } else {  // the four words from the first one that counts
    const bool neg = (p[NW - 1] >> 31) & 1;
    unsigned w[NW + 3] = {};  // w[3] the lowest
    unsigned long long carry = neg ? 1 : 0;
    int t = 3;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      carry += neg ? ~(unsigned)p[i] : (unsigned)p[i];
      w[i + 3] = (unsigned)carry;
      carry >>= 32;
      if (w[i + 3]) t = i + 3;
    }
    unsigned long long H = 0, L = 0;
#pragma unroll
    for (int i = 3; i < NW + 3; ++i)
      if (i == t) {
        H = (unsigned long long)w[i] << 32 | w[i - 1];
        L = (unsigned long long)w[i - 2] << 32 | w[i - 3];
      }
    return fixed_times(neg, H, L, e + 32 * (t - (NW + 2)), c);
  }
}

constexpr int kMaxGroups = 8;
// Residues of coefficients c and c + 1, the offset groups added.
template <int NM, bool GROUPS>
__device__ __forceinline__ void load_pair(const CrtLv& v, const int16_t* __restrict__ res, int64_t step, int (&s0)[NM],
                                          int (&s1)[NM]) {
  const int64_t mod = GROUPS ? v.G * step : step;
  int u[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) u[i] = *reinterpret_cast<const int*>(res + i * mod);
#pragma unroll
  for (int i = 0; i < NM; ++i) asm volatile("" : "+r"(u[i]));  // every load is on its way before the first use
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    s0[i] = (int16_t)u[i];
    s1[i] = u[i] >> 16;
  }
  if (GROUPS && v.G > 1) {
    for (int k = 1; k < v.G; ++k)
#pragma unroll
      for (int i = 0; i < NM; ++i) {
        const short2 u = *reinterpret_cast<const short2*>(res + ((int64_t)i * v.G + k) * step);
        s0[i] += u.x;
        s1[i] += u.y;
      }
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      s0[i] %= crt_mod(i);
      s1[i] %= crt_mod(i);
    }
  }
}
// The sums from their residues.
template <int NM, int NW>
__device__ __forceinline__ void rebuild_pair(const CrtLv& v, const CrtK<NM, NW>& kc, const int (&s0)[NM],
                                             const int (&s1)[NM], int c, int e, bool fin, double* y) {
  unsigned long long p[2][NW] = {};
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    // non-negative, and zero for zero: a sum of nothing is exactly 0
    const unsigned u0 = (unsigned)(s0[i] + (s0[i] < 0 ? crt_mod(i) : 0));
    const unsigned u1 = (unsigned)(s1[i] + (s1[i] < 0 ? crt_mod(i) : 0));
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      p[0][w] += (unsigned long long)u0 * kc.k[i][w];
      p[1][w] += (unsigned long long)u1 * kc.k[i][w];
    }
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    y[k] = 0.0;
    if (c + k >= v.d) break;
#pragma unroll
    for (int w = 1; w < NW; ++w) p[k][w] += p[k][w - 1] >> 32;
    y[k] = fin ? fraction_times<NW>(p[k], e, v.colscale[c + k]) : __longlong_as_double(0x7ff8000000000000ll);
  }
}

// One block of coefficient pairs; WEAK: both parts of the weak targets among them.
template <int NM, int NW, bool GROUPS, bool WEAK>
__device__ __forceinline__ void rebuild_block(const CrtArgs& a, const CrtK<NM, NW>& kc, unsigned block) {
  const CrtLv& v = a.lv[find_level(a, &CrtLv::rc0, block)];
  const unsigned P = (unsigned)(v.d + 1) / 2;  // pairs of a row
  const unsigned cells = (unsigned)(v.nz * v.h * v.h), rows = cells * (unsigned)(v.nct * v.Rc);
  // the block's first pair, then a thread's within 2^16: one multiplication
  const int64_t first = (int64_t)(block - v.rc0) * kRebuild;
  const unsigned row0 = (unsigned)(first / P), t = (unsigned)(first - (int64_t)row0 * P) + threadIdx.x;
  const unsigned dr = __umulhi(t, v.pinv), row = row0 + dr;
  if (row >= rows) return;
  const int c = 2 * (int)(t - dr * P);
  const int N = v.NT * v.Nt;
  const int64_t step = (int64_t)rows * N;
  const int16_t* res = v.res + (int64_t)row * N + c;
  int s0[NM], s1[NM];
  if (!GROUPS) load_pair<NM, GROUPS>(v, res, step, s0, s1);
  const unsigned rr = v.Rc == 1 ? 0u : row / (cells * (unsigned)v.nct), in = row - rr * cells * (unsigned)v.nct;
  const int r = v.r0 + (int)rr;
  const int lh = 31 - __clz(v.h);  // h is a power of two
  const unsigned cz = in >> (2 * lh), cls = v.nct == 1 ? 0u : cz / (unsigned)v.nz;
  const int64_t I = class_box(v.nct, (int)cls, (int)(in & (v.h - 1)), (int)((in >> lh) & (v.h - 1)),
                              v.z0 + (int)(cz - cls * v.nz));
  if (WEAK) {
    const int x = (int)(in & (v.h - 1)), y = (int)((in >> lh) & (v.h - 1)), z = v.z0 + (int)(cz - cls * v.nz);
    if (v.weak[I * v.R + r] != 1 || v.need[need_index(v, (int)rr, (int)cls, z, y, x)] < kTileWork) return;
  }
  double* g = v.g + (I * v.R + r) * v.d + c;
  const unsigned long long bits = v.wmax[(I >> v.tshift) * v.R + r];
  const bool fin = w_finite(bits);
  // colscale is in units of 2^(-32 NW), NW of the mode
  const int e = (NM == kMods ? 96 : 128) - w_exp(bits, v.wbits);
  const double* add = v.add ? v.add + (I * v.R + r) * v.d + c : nullptr;
  double y[2];
  if (GROUPS) load_pair<NM, GROUPS>(v, res, step, s0, s1);
  rebuild_pair<NM, NW>(v, kc, s0, s1, c, e, fin, y);
  if (WEAK) {
    double z[2];
    load_pair<NM, GROUPS>(v, res + v.rstep, step, s0, s1);
    rebuild_pair<NM, NW>(v, kc, s0, s1, c, e - kRestBits, fin, z);
    y[0] += z[0];
    y[1] += z[1];
  }
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (c + k < v.d) g[k] = add ? add[k] + y[k] : y[k];
}
template <int NM, int NW, bool GROUPS>
__global__ void __launch_bounds__(kRebuild)
k_crt_rebuild(const __grid_constant__ CrtArgs a, const __grid_constant__ CrtK<NM, NW> kc) {
  rebuild_block<NM, NW, GROUPS, false>(a, kc, blockIdx.x);
}
// A weak box on the FP64 pipes: a block takes 32 coefficients, a warp every fourth
// occupied source; the warps' sums are added in order.
__device__ __forceinline__ void weak_box(const CrtLv& v, int r, int64_t box, int c0, double* s_sum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, mp = c0 + lane;
  int b[3];
  morton_decode(box, v.tlevel, b);
  const int n = 1 << v.tlevel;
  double sum = 0.0;
  int turn = 0;
  for (int k = 0; k < 224; k += 32) {  // the children of the 27 neighbours of its parent
    const int i = k + lane, x = (b[0] & ~1) - 2 + i % 6, y = (b[1] & ~1) - 2 + i / 6 % 6, z = (b[2] & ~1) - 2 + i / 36;
    const int dx = x - b[0], dy = y - b[1], dz = z - b[2];
    const bool in = i < 216 && x >= 0 && y >= 0 && z >= 0 && x < n && y < n && z < n &&
                    (abs(dx) > 1 || abs(dy) > 1 || abs(dz) > 1);
    const int J = in ? (int)morton_encode(x, y, z, v.tlevel) : 0, slot = (dz + 3) * 49 + (dy + 3) * 7 + dx + 3;
    for (unsigned left = __ballot_sync(0xffffffffu, in && v.bmax[(int64_t)J * v.R + r] != 0); left; left &= left - 1) {
      const int from = __ffs(left) - 1;
      const int64_t Js = __shfl_sync(0xffffffffu, J, from);
      const int sl = __shfl_sync(0xffffffffu, slot, from);
      if ((turn++ & 3) != warp || mp >= v.d) continue;
      const double* T = v.T + (int64_t)sl * v.ds * v.d + mp;
      const double* w = v.W + (Js * v.R + r) * v.ds;
#pragma unroll 8
      for (int l = 0; l < v.ds; ++l) sum = fma(T[(int64_t)l * v.d], w[l], sum);
    }
  }
  __syncthreads();
  s_sum[threadIdx.x] = sum;
  __syncthreads();
  if (warp == 0 && mp < v.d)
    v.g[(box * v.R + r) * v.d + mp] = s_sum[lane] + s_sum[32 + lane] + s_sum[64 + lane] + s_sum[96 + lane];
}
// The weak boxes: by the second part, or on the FP64 pipes.
__global__ void __launch_bounds__(kRebuild)
k_crt_weak(const __grid_constant__ CrtArgs a, const __grid_constant__ CrtK<kMods, 5> kc) {
  __shared__ double s_sum[kRebuild];
  const unsigned n = a.any[1];
  if (n == 0) return;
  if (a.any[0])
    for (unsigned b = blockIdx.x; b < a.rebuild_blocks; b += gridDim.x) rebuild_block<kMods, 5, true, true>(a, kc, b);
  const unsigned chunks = (kMaxD + 31) / 32;
  for (unsigned u = blockIdx.x; u < n * chunks; u += gridDim.x) {
    const uint2 e = a.list[u / chunks];
    const CrtLv& v = a.lv[e.x >> 16];
    const int r = (int)(e.x & 0xffffu), c0 = 32 * (int)(u % chunks);
    if (c0 >= v.d) continue;
    const int64_t box = e.y;
    int b[3];
    morton_decode(box, v.tlevel, b);
    const int ct = (b[0] & 1) | (b[1] & 1) << 1 | (b[2] & 1) << 2;
    if (v.weak[box * v.R + r] == 1 &&
        v.need[need_index(v, r - v.r0, ct, b[2] >> 1, b[1] >> 1, b[0] >> 1)] >= kTileWork)
      continue;
    weak_box(v, r, box, c0, s_sum);
  }
}

// ---------------------------------------------------------- the images --
// Largest entry and sum of |T| over slots and l for 32 rows m' and one of the
// kRowParts shares of the (slot, l) per block: part[share][0 or 1][m'].
constexpr int kRowParts = 64;
__global__ void __launch_bounds__(256) k_crt_rowsum(const double* __restrict__ kdT, int nslots, int dl, int d,
                                                    double* __restrict__ part) {
  const int mp = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y;
  const int64_t n = (int64_t)nslots * dl, i0 = n * y / kRowParts, i1 = n * (y + 1) / kRowParts;
  double s = 0.0, m = 0.0;
  if (mp < d)
    for (int64_t i = i0 + threadIdx.y; i < i1; i += 8) {
      const int slot = (int)(i / dl);
      const int dx = slot % 7 - 3, dy = (slot / 7) % 7 - 3, dz = slot / 49 - 3;
      if (nslots == kNumSlots && abs(dx) <= 1 && abs(dy) <= 1 && abs(dz) <= 1) continue;  // the near field
      const double t = fabs(kdT[i * d + mp]);
      s += t;
      m = fmax(m, t);
    }
  __shared__ double ss[8][33], sm[8][33];
  ss[threadIdx.y][threadIdx.x] = s;
  sm[threadIdx.y][threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.y == 0 && mp < d) {
    for (int k = 1; k < 8; ++k) {
      s += ss[k][threadIdx.x];
      m = fmax(m, sm[k][threadIdx.x]);
    }
    part[(int64_t)(2 * y) * d + mp] = m;
    part[(int64_t)(2 * y + 1) * d + mp] = s;
  }
}

// Exponents a of the rows: l1 2^a < 2^rowbits and mx 2^a < 2^entrybits.
__global__ void k_crt_rowscale(const double* __restrict__ part, int d, double mscale, int rowbits, int entrybits,
                               double* __restrict__ up, double* __restrict__ colscale) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= d) return;
  double mx = 0.0, l1 = 0.0;
  for (int y = 0; y < kRowParts; ++y) {
    mx = fmax(mx, part[(int64_t)(2 * y) * d + m]);
    l1 += part[(int64_t)(2 * y + 1) * d + m];
  }
  int e = 0, e1 = 0;
  // the sum itself carries rounding; 2^-40 relative covers it
  frexp(l1 * (1.0 + 0x1p-40), &e);
  frexp(mx, &e1);
  int s = min(rowbits - e, entrybits - e1);
  s = l1 > 0.0 ? max(-900, min(900, s)) : 0;
  up[m] = pow2(s);
  colscale[m] = ldexp(mscale, -s);
}

// One thread per (slot, column tile, k8, n): 8 terms of one row for every modulus.
__global__ void __launch_bounds__(256) k_crt_image(const double* __restrict__ kdT, int nslots, int dl, int d, int K,
                                                   int Nt, int NT, const double* __restrict__ up,
                                                   __nv_bfloat16* __restrict__ img) {
  const int slot = blockIdx.y;
  const int64_t tile_e = (int64_t)K * Nt;
  const int units = NT * (K / 8) * Nt;
  for (int u = blockIdx.x * 256 + threadIdx.x; u < units; u += gridDim.x * 256) {
    const int n = u % Nt, k8 = (u / Nt) % (K / 8), nt = u / (Nt * (K / 8));
    const int mp = nt * Nt + n;
    long long w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int l = 8 * k8 + j;
      w[j] = (mp < d && l < dl) ? __double2ll_rn(kdT[((int64_t)slot * dl + l) * d + mp] * up[mp]) : 0;
    }
    __nv_bfloat16* dst = img + ((int64_t)slot * NT + nt) * tile_e + ((int64_t)k8 * Nt + n) * 8;
    Limbs q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = limbs_of(w[2 * j], w[2 * j + 1]);
    store_residues<0, kMods>(q, dst, (int64_t)nslots * NT * tile_e);
  }
}

// ------------------------------------------------- Delta^t, explicitly --
// Delta^t = Gamma^-t B^-1 in double-double (106 bits), a warp per column j: B z
// = e_j forward, Gamma^t w = z backward, the dot products over the lanes.
struct Dd {
  double h, l;
};
__device__ __forceinline__ Dd dd_norm(double a, double b) {  // |a| >= |b| or a = 0
  const double s = __dadd_rn(a, b);
  return {s, __dadd_rn(b, -__dadd_rn(s, -a))};
}
__device__ __forceinline__ Dd dd_add(Dd a, Dd b) {
  const double s = __dadd_rn(a.h, b.h), sb = __dadd_rn(s, -a.h);
  const double e = __dadd_rn(__dadd_rn(a.h, -__dadd_rn(s, -sb)), __dadd_rn(b.h, -sb));
  const double t = __dadd_rn(a.l, b.l), tb = __dadd_rn(t, -a.l);
  const double f = __dadd_rn(__dadd_rn(a.l, -__dadd_rn(t, -tb)), __dadd_rn(b.l, -tb));
  const Dd x = dd_norm(s, __dadd_rn(e, t));
  return dd_norm(x.h, __dadd_rn(x.l, f));
}
__device__ __forceinline__ Dd dd_mul(Dd a, double b) {
  const double p = __dmul_rn(a.h, b), e = __fma_rn(a.h, b, -p);
  return dd_norm(p, __fma_rn(a.l, b, e));
}
__device__ __forceinline__ Dd dd_div(Dd a, double b) {
  const double q1 = __ddiv_rn(a.h, b);
  const Dd r1 = dd_add(a, dd_mul({b, 0.0}, -q1));
  const double q2 = __ddiv_rn(r1.h, b);
  const Dd r2 = dd_add(r1, dd_mul({b, 0.0}, -q2));
  return dd_add(dd_norm(q1, q2), {__ddiv_rn(r2.h, b), 0.0});
}
__device__ __forceinline__ Dd dd_warp_sum(Dd v) {
  for (int o = 16; o > 0; o >>= 1)
    v = dd_add(v, {__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
  return v;
}
// hi, lo: [j][i] = Delta^t_{ij}
__global__ void __launch_bounds__(32) k_delta_t_dd(int d, const double* __restrict__ G, const double* __restrict__ B,
                                                   double* __restrict__ hi, double* __restrict__ lo) {
  __shared__ double zh[kMaxD], zl[kMaxD];
  const int j = blockIdx.x, lane = threadIdx.x;
  for (int i = lane; i < d; i += 32) zh[i] = zl[i] = 0.0;
  for (int i = j; i < d; ++i) {
    __syncwarp();
    Dd s = {0.0, 0.0};
    for (int m = j + lane; m < i; m += 32) s = dd_add(s, dd_mul({zh[m], zl[m]}, -B[(int64_t)i * d + m]));
    s = dd_warp_sum(s);
    if (lane == 0) {
      if (i == j) s = {1.0, 0.0};  // the sum is empty
      zh[i] = s.h;
      zl[i] = s.l;
    }
  }
  for (int i = d - 1; i >= 0; --i) {
    __syncwarp();
    Dd s = {0.0, 0.0};
    for (int m = i + 1 + lane; m < d; m += 32) s = dd_add(s, dd_mul({zh[m], zl[m]}, -G[(int64_t)m * d + i]));
    s = dd_warp_sum(s);
    if (lane == 0) {
      s = dd_div(dd_add({zh[i], zl[i]}, s), G[(int64_t)i * d + i]);
      zh[i] = s.h;
      zl[i] = s.l;
    }
  }
  __syncwarp();
  for (int i = lane; i < d; i += 32) {
    hi[(int64_t)j * d + i] = zh[i];
    lo[(int64_t)j * d + i] = zl[i];
  }
}

// x 2^s toward zero, for |x| 2^s < 2^126.
__device__ __int128 scaled_int(double x, int s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e == 0) return 0;
  const __int128 m = (__int128)((b & 0xfffffffffffffull) | (1ull << 52));
  const int t = e - 1075 + s;
  const __int128 q = t >= 0 ? (t < 74 ? m << t : 0) : (t > -64 ? m >> -t : 0);
  return b >> 63 ? -q : q;
}
// As k_crt_image for one operator given as hi + lo; up: 2^a of the rows.
__global__ void __launch_bounds__(256) k_crt_image_dd(const double* __restrict__ hi, const double* __restrict__ lo,
                                                      int d, int K, int Nt, int NT, const double* __restrict__ up,
                                                      __nv_bfloat16* __restrict__ img) {
  const int64_t tile_e = (int64_t)K * Nt;
  const int u = blockIdx.x * 256 + threadIdx.x;
  if (u >= NT * K * Nt) return;
  const int n = u % Nt, l = (u / Nt) % K, nt = u / (Nt * K), mp = nt * Nt + n;
  __int128 w = 0;
  if (mp < d && l < d) {
    const int s = (int)(((unsigned long long)__double_as_longlong(up[mp]) >> 52) & 0x7ff) - 1023;
    w = scaled_int(hi[(int64_t)l * d + mp], s) + scaled_int(lo[(int64_t)l * d + mp], s);
  }
  __nv_bfloat16* dst = img + (int64_t)nt * tile_e + ((int64_t)(l / 8) * Nt + n) * 8 + (l & 7);
  for (int i = 0; i < kBoxMods; ++i) {
    const int m = crt_mod(i);
    int r = (int)(w % m);
    if (2 * r > m) r -= m;
    if (2 * r < -m) r += m;
    dst[(int64_t)i * NT * tile_e] = __float2bfloat16_rn((float)r);
  }
}

// out[slot]: the ratio of crt_kappa for one offset (0 in the near field).
__global__ void __launch_bounds__(128) k_crt_kappa(int kern, int d, double lk, const double* __restrict__ X,
                                                   const double* __restrict__ Y, const double* __restrict__ kdT,
                                                   double* __restrict__ out) {
  __shared__ double w[kMaxD];
  __shared__ double red[2][4];
  const int slot = blockIdx.x;
  const int dx = slot % 7 - 3, dy = (slot / 7) % 7 - 3, dz = slot / 49 - 3;
  for (int l = threadIdx.x; l < d; l += 128)
    w[l] = fabs(kern_f64(kern, X[3 * l] - Y[0], X[3 * l + 1] - Y[1], X[3 * l + 2] - Y[2]));
  __syncthreads();
  double num = 0.0, den = 0.0;
  const bool far = abs(dx) > 1 || abs(dy) > 1 || abs(dz) > 1;
  for (int m = threadIdx.x; far && m < d; m += 128) {
    double s = 0.0;
    for (int l = 0; l < d; ++l) s += fabs(kdT[((int64_t)slot * d + l) * d + m]) * w[l];
    num = fmax(num, s);
    den = fmax(den, fabs(kern_f64(kern, Y[3 * m] - (Y[0] + 2.0 * dx * lk), Y[3 * m + 1] - (Y[1] + 2.0 * dy * lk),
                                  Y[3 * m + 2] - (Y[2] + 2.0 * dz * lk))));
  }
  for (int o = 16; o > 0; o >>= 1) {
    num = fmax(num, __shfl_xor_sync(0xffffffffu, num, o));
    den = fmax(den, __shfl_xor_sync(0xffffffffu, den, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = num;
    red[1][threadIdx.x >> 5] = den;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 4; ++i) {
      num = fmax(num, red[0][i]);
      den = fmax(den, red[1][i]);
    }
    out[slot] = num > 0.0 ? num / den : 0.0;
  }
}

// Product of the first n moduli times 2^-shift.
double crt_product_scaled(int n, int shift) {
  unsigned __int128 m = 1;  // exact to 125 bits, then the moduli beyond in FP64
  double rest = 1.0;
  for (int i = 0; i < n; ++i) {
    if (i < kMods) m *= (unsigned)crt_mod(i);
    else rest *= crt_mod(i);
  }
  return std::ldexp((double)m * rest, -shift);
}

template <int NM, int NW>
CrtK<NM, NW> crt_constants() {
  CrtK<NM, NW> c;
  for (int i = 0; i < NM; ++i) {
    const uint64_t m = (uint64_t)crt_mod(i);
    uint64_t p = 1;  // M / m_i modulo m_i
    for (int j = 0; j < NM; ++j)
      if (j != i) p = p * (uint64_t)crt_mod(j) % m;
    uint64_t y = 1;
    while (p * y % m != 1) ++y;
    // y / m to NW words by long division, rounded to nearest
    uint64_t r = y;
    for (int w = NW - 1; w >= 0; --w) {
      r <<= 32;
      c.k[i][w] = (uint32_t)(r / m);
      r %= m;
    }
    if (2 * r >= m)
      for (int w = 0; w < NW && ++c.k[i][w] == 0; ++w) {
      }
  }
  return c;
}

// The scratch of a level is split into columns and slabs of planes beyond this.
constexpr size_t kScratchLimit = (size_t)4 << 30;

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }
// Class grid of a job whose target boxes have level `level`.
int mode_mods(CrtMode m) { return m == kCrtBox ? kBoxMods : kMods; }
int mode_ncs(CrtMode m) { return m == kCrtL2L ? 1 : 8; }
int mode_nct(CrtMode m) { return m == kCrtM2M ? 1 : 8; }
int mode_h(CrtMode m, int level) { return m == kCrtM2M ? 1 << level : 1 << (level - 1); }
int mode_parts(CrtMode m) { return m == kCrtM2L ? 2 : 1; }
size_t planes_bytes(CrtMode m, int K, int h, int snz, int Rc) {
  return align256((size_t)mode_parts(m) * mode_mods(m) * Rc * mode_ncs(m) * snz * h * h * K * 2);
}
size_t res_bytes(CrtMode m, int N, int h, int nz, int Rc, int G) {
  return align256((size_t)mode_parts(m) * mode_mods(m) * G * Rc * mode_nct(m) * nz * h * h * N * 2);
}
// offset groups are used only by M2L and M2M launches of few tiles: levels below this one
constexpr int kGroupLevel = 4;
int max_groups(CrtMode m, int level) {
  return (m == kCrtM2L || m == kCrtM2M) && level < kGroupLevel ? kMaxGroups : 1;
}
size_t job_bytes(CrtMode m, const CrtImage& im, int level, int nz, int Rc) {
  const int h = mode_h(m, level);
  const int snz = std::min(h, nz + 2);
  return planes_bytes(m, im.K, h, snz, Rc) + res_bytes(m, im.NT * im.Nt, h, nz, Rc, max_groups(m, level));
}
int64_t need_tiles(int h, int nz, int Rc) {
  return (int64_t)((h + kTX - 1) / kTX) * ((h + kTY - 1) / kTY) * ((nz + kTZ - 1) / kTZ) * 8 * Rc;
}
// columns and planes of one slab of a level within `limit` bytes
void slab_shape(CrtMode m, const CrtImage& im, int level, int R, size_t limit, int* Rc, int* nz) {
  *Rc = R;
  *nz = mode_h(m, level);
  while (*Rc > 1 && job_bytes(m, im, level, *nz, *Rc) > limit) *Rc = (*Rc + 1) / 2;
  while (*nz > kTZ && job_bytes(m, im, level, *nz, *Rc) > limit) *nz = std::max(kTZ, (*nz / 2 + kTZ - 1) / kTZ * kTZ);
}

}  // namespace

size_t crt_scratch_bytes(int njobs, const CrtJob* jobs, int R) {
  size_t total = 0, most = 0;
  for (int j = 0; j < njobs; ++j) {
    int Rc, nz;
    slab_shape(jobs[j].mode, *jobs[j].img, jobs[j].level, R, kScratchLimit, &Rc, &nz);
    const size_t n = job_bytes(jobs[j].mode, *jobs[j].img, jobs[j].level, nz, Rc);
    if (jobs[j].mode == kCrtM2L) total += n;  // the levels of the M2L share a launch
    most = std::max(most, n);
  }
  return std::max(most, std::min(total, kScratchLimit));
}

bool crt_steep(int kern, double L, int level) {
  const double w = L * std::ldexp(1.0, -level);
  double near = 0.0, far = 0.0;
  for (int a = 0; a < 3; ++a)
    near = std::max(near, std::fabs(kern_f64(kern, a == 0 ? w : 0.0, a == 1 ? w : 0.0, a == 2 ? w : 0.0)));
  for (int i = 0; i < 32; ++i) {  // several distances: the kernel may oscillate
    const double z = 4.0 * w * (0.9 + 0.1 * i / 31.0);
    far = std::max(far, std::fabs(kern_f64(kern, z, z, z)));
  }
  return !(near > 0.0 && far >= 0x1p-7 * near);
}

bool crt_ready(CrtMode mode, int level, const CrtImage& im, int R, size_t bytes) {
  if (!im.img || bytes == 0) return false;
  const CrtJob job{mode, level, &im, nullptr, nullptr, nullptr};
  return crt_scratch_bytes(1, &job, R) <= bytes;
}

// [kMaxLevel + 1][R] maxima of the M2L's levels, the word `any`, the tiles' `need`,
// the boxes' maxima, their list, their `weak`; or the maxima of another mode's units
size_t crt_max_words(int depth, int R) {
  size_t boxes = 0, tiles = 0;
  for (int k = 2; k <= depth; ++k) {
    boxes += (size_t)1 << (3 * k);
    tiles += need_tiles(1 << (k - 1), 1 << (k - 1), R);
  }
  return (size_t)(kMaxLevel + 1) * R + 1 + (tiles + 1) / 2 + 2 * boxes * R + (boxes * R + 7) / 8;
}

void free_crt_image(CrtImage* im) {
  dfree(im->img);
  dfree(im->colscale);
  *im = CrtImage();
}

eifmm_status build_crt_image(const double* kdT, int nslots, int dl, int d, CrtImage* im, cudaStream_t s) {
  im->T = kdT;
  im->d = d;
  im->dl = dl;
  im->nslots = nslots;
  im->K = (dl + 15) / 16 * 16;
  im->NT = (d + 255) / 256;
  im->Nt = (((d + 15) / 16 + im->NT - 1) / im->NT) * 16;
  double* tmp = nullptr;  // 2^a of each row, then the shares of its largest entry and sum
  eifmm_status rc = dalloc(&tmp, (size_t)(2 * kRowParts + 1) * d);
  if (rc == EIFMM_OK) rc = dalloc(&im->colscale, d);
  const size_t e = (size_t)kMods * nslots * im->NT * im->K * im->Nt;
  if (rc == EIFMM_OK) rc = dmalloc(&im->img, e * sizeof(__nv_bfloat16));
  if (rc == EIFMM_OK) {
    k_crt_rowsum<<<dim3((d + 31) / 32, kRowParts), dim3(32, 8), 0, s>>>(kdT, nslots, dl, d, tmp + d);
    count_launch();
    const double mscale = crt_product_scaled(kMods, 96);
    k_crt_rowscale<<<(d + 127) / 128, 128, 0, s>>>(tmp + d, d, mscale, kRowBits, kEntryBits, tmp, im->colscale);
    count_launch();
    const int units = im->NT * (im->K / 8) * im->Nt;
    k_crt_image<<<dim3((units + 255) / 256, nslots), 256, 0, s>>>(kdT, nslots, dl, d, im->K, im->Nt, im->NT,
                                                                  tmp, (__nv_bfloat16*)im->img);
    count_launch();
    // other streams may read the image as soon as this returns
    if (cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
      set_error("building the residue images of the M2L operators failed");
      rc = EIFMM_ECUDA;
    }
  }
  dfree(tmp);
  if (rc != EIFMM_OK) free_crt_image(im);
  return rc;
}

eifmm_status build_crt_delta_image(const LevelOps& v, CrtImage* im, cudaStream_t s) {
  const int d = v.d;
  im->d = im->dl = d;
  im->nslots = 1;
  im->K = (d + 15) / 16 * 16;
  im->NT = (d + 255) / 256;
  im->Nt = (((d + 15) / 16 + im->NT - 1) / im->NT) * 16;
  double* tmp = nullptr;  // Delta^t hi and lo, then as in build_crt_image
  const size_t dd = (size_t)d * d;
  eifmm_status rc = dalloc(&tmp, 2 * dd + (size_t)(2 * kRowParts + 1) * d);
  if (rc == EIFMM_OK) rc = dalloc(&im->colscale, d);
  if (rc == EIFMM_OK) rc = dmalloc(&im->img, (size_t)kBoxMods * im->NT * im->K * im->Nt * sizeof(__nv_bfloat16));
  bool fine = false;
  if (rc == EIFMM_OK) {
    double *hi = tmp, *lo = tmp + dd, *row = tmp + 2 * dd;
    k_delta_t_dd<<<d, 32, 0, s>>>(d, v.G_rm, v.B_rm, hi, lo);
    count_launch();
    k_crt_rowsum<<<dim3((d + 31) / 32, kRowParts), dim3(32, 8), 0, s>>>(hi, 1, d, d, row + d);
    count_launch();
    k_crt_rowscale<<<(d + 127) / 128, 128, 0, s>>>(row + d, d, crt_product_scaled(kBoxMods, 128), kBoxRowBits,
                                                   kBoxRowBits, row, im->colscale);
    count_launch();
    k_crt_image_dd<<<(im->NT * im->K * im->Nt + 255) / 256, 256, 0, s>>>(hi, lo, d, im->K, im->Nt, im->NT, row,
                                                                         (__nv_bfloat16*)im->img);
    count_launch();
    std::vector<double> up(d);
    double g11 = 0.0;
    if (cudaMemcpyAsync(up.data(), row, d * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(&g11, v.G_rm, sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
      set_error("building the residue image of Delta^t failed");
      rc = EIFMM_ECUDA;
    } else {
      // the entries are rounded to 2^-a: times |A| <= |Gamma_11| and d terms
      // that is the backward error of the product, which stays below 2^-52 as
      // the triangular solves' does (1/r at eps 1e-7: 2^-55)
      double q = 0.0;
      for (double u : up) q = std::max(q, 1.0 / u);
      fine = q * std::fabs(g11) * d <= 0x1p-52;
    }
  }
  dfree(tmp);
  if (rc != EIFMM_OK || !fine) {
    free_crt_image(im);
    im->refused = rc == EIFMM_OK;
  }
  return rc;
}

eifmm_status crt_kappa(int kern, const LevelOps& v, double lk, double* kappa, cudaStream_t s) {
  double* out = nullptr;
  EIFMM_TRY(dalloc(&out, kNumSlots));
  k_crt_kappa<<<kNumSlots, 128, 0, s>>>(kern, v.d, lk, v.X, v.Y, v.kdT, out);
  count_launch();
  double h[kNumSlots];
  const bool ok = cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
                  cudaStreamSynchronize(s) == cudaSuccess;
  dfree(out);
  if (!ok) {
    set_error("the amplification of the M2L operators could not be computed");
    return EIFMM_ECUDA;
  }
  *kappa = *std::max_element(h, h + kNumSlots);
  return EIFMM_OK;
}

eifmm_status launch_crt(int njobs, const CrtJob* jobs, int R, void* buf, size_t buf_bytes,
                            unsigned long long* wmax, int nsm, int* err, cudaStream_t s) {
  auto encode = encode_fn();
  if (!encode) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return EIFMM_ECUDA;
  }
  static const CrtK<kMods, 3> kc = crt_constants<kMods, 3>();
  static const CrtK<kMods, 5> kweak = crt_constants<kMods, 5>();
  static const CrtK<kBoxMods, 4> kcb = crt_constants<kBoxMods, 4>();
  static bool attr[64] = {};
  int dev = 0;
  EIFMM_CUDA(cudaGetDevice(&dev));
  if (dev >= 64 || !attr[dev]) {
    EIFMM_CUDA(cudaFuncSetAttribute(k_crt_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
    EIFMM_CUDA(cudaFuncSetAttribute(k_crt_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
    if (dev < 64) attr[dev] = true;
  }
  const bool m2l = njobs > 0 && jobs[0].mode == kCrtM2L;
  unsigned *any = nullptr, *need = nullptr;
  uint2* list = nullptr;
  unsigned char* weak[kMaxLevel + 1] = {};
  unsigned long long* bmax[kMaxLevel + 1] = {};
  if (m2l) {
    unsigned long long* p = wmax + (size_t)(kMaxLevel + 1) * R;
    any = (unsigned*)p++;
    need = (unsigned*)p;
    size_t boxes = 0, tiles = 0;
    for (int j = 0; j < njobs; ++j) tiles += need_tiles(1 << (jobs[j].level - 1), 1 << (jobs[j].level - 1), R);
    p += (tiles + 1) / 2;
    EIFMM_CUDA(cudaMemsetAsync(wmax, 0, (char*)p - (char*)wmax, s));
    for (int j = 0; j < njobs; ++j) {
      bmax[jobs[j].level] = p + boxes * R;
      boxes += (size_t)1 << (3 * jobs[j].level);
    }
    list = (uint2*)(p + boxes * R);
    unsigned char* c = (unsigned char*)(p + 2 * boxes * R);
    for (int j = 0; j < njobs; ++j) {
      weak[jobs[j].level] = c;
      c += ((size_t)1 << (3 * jobs[j].level)) * R;
    }
  }
  // slabs of all jobs, largest levels first; consecutive ones that fit the
  // scratch together share their launches
  std::vector<CrtLv> todo;
  for (int j = njobs - 1; j >= 0; --j) {
    const CrtJob& b = jobs[j];
    int Rc, nz;
    slab_shape(b.mode, *b.img, b.level, R, kScratchLimit, &Rc, &nz);
    const int h = mode_h(b.mode, b.level);
    for (int r0 = 0; r0 < R; r0 += Rc)
      for (int z0 = 0; z0 < h; z0 += nz) {
        CrtLv v = {};
        v.mode = b.mode;
        v.tlevel = b.level;
        v.slevel = b.mode == kCrtM2M ? b.level + 1 : b.mode == kCrtL2L ? b.level - 1 : b.level;
        v.ncs = mode_ncs(b.mode);
        v.nct = mode_nct(b.mode);
        v.nw = b.mode == kCrtM2L ? 24 : b.mode == kCrtM2M ? 8 : 1;
        v.nslots = b.img->nslots;
        v.wbits = b.mode == kCrtBox ? kBoxWBits : kWBits;
        v.d = b.img->d;
        v.ds = b.img->dl;
        v.K = b.img->K;
        v.Nt = b.img->Nt;
        v.NT = b.img->NT;
        v.h = h;
        v.z0 = z0;
        v.nz = std::min(nz, h - z0);
        v.sz0 = std::max(0, z0 - 1);
        v.snz = std::min(h, z0 + v.nz + 1) - v.sz0;
        v.r0 = r0;
        v.Rc = std::min(Rc, R - r0);
        v.R = R;
        split_chunks(&v);
        v.W = b.W;
        v.g = b.g;
        v.add = b.add;
        v.img = (const __nv_bfloat16*)b.img->img;
        v.colscale = b.img->colscale;
        v.sshift = b.mode == kCrtM2L ? 3 * b.level : b.mode == kCrtM2M ? 3 : 0;
        v.tshift = b.mode == kCrtM2L ? 3 * b.level : b.mode == kCrtL2L ? 3 : 0;
        v.wmax = b.mode == kCrtM2L ? wmax + (size_t)b.level * R : wmax;
        if (m2l) {
          v.bmax = bmax[b.level];
          v.weak = weak[b.level];
          v.need = need;
          v.T = b.img->T;
          need += need_tiles(h, v.nz, v.Rc);
        }
        todo.push_back(v);
      }
  }
  for (size_t i0 = 0; i0 < todo.size();) {
    CrtArgs a = {};
    CrtMaps maps = {};
    a.err = err;
    a.any = any;
    a.list = list;
    if (m2l && i0 > 0) EIFMM_CUDA(cudaMemsetAsync(any, 0, 2 * sizeof(unsigned), s));
    size_t off = 0, i1 = i0;
    int64_t items = 0;
    auto tiles = [](const CrtLv& v) {
      return (int64_t)((v.h + kTX - 1) / kTX) * ((v.h + kTY - 1) / kTY) * ((v.nz + kTZ - 1) / kTZ) * v.nct * v.NT *
             v.Rc * mode_mods(v.mode);
    };
    for (; i1 < todo.size() && a.nlev < kMaxLv; ++i1) {
      const CrtLv& v = todo[i1];
      const size_t need = planes_bytes(v.mode, v.K, v.h, v.snz, v.Rc) +
                          res_bytes(v.mode, v.NT * v.Nt, v.h, v.nz, v.Rc, max_groups(v.mode, v.tlevel));
      if (a.nlev > 0 && (off + need > buf_bytes || mode_mods(v.mode) != mode_mods(a.lv[0].mode))) break;
      if (need > buf_bytes) {
        set_error("residue M2L: scratch too small");
        return EIFMM_EINVAL;
      }
      off += need;
      items += tiles(v);
      a.lv[a.nlev++] = v;
    }
    off = 0;
    unsigned it = 0, pl = 0, rb = 0, mx = 0;
    uint32_t stage = 0, win = 0;
    size_t pl_smem = 0;
    bool groups = false;
    for (int q = 0; q < a.nlev; ++q) {
      CrtLv& v = a.lv[q];
      // a launch of few tiles: the windows of the coarse levels' tiles are
      // split into groups until the CTAs cover four waves (M2L), or as long as
      // they stay within one (M2M, whose CTAs have 8 short windows: 14 CTAs 29
      // us, 112 CTAs 14 us; but 98 CTAs 31 us, 784 CTAs 51 us)
      v.G = 1;
      const int64_t most = (v.mode == kCrtM2M ? nsm : 8 * (int64_t)nsm - 1) / 2;
      while (v.G < max_groups(v.mode, v.tlevel) && items * v.G <= most) v.G *= 2;
      groups = groups || v.G > 1;
      for (int ct = 0; ct < v.nct; ++ct)
        for (int p = 0; p < v.G; ++p) v.ng[ct][p] = (uint16_t)accumulations(v, ct, p);
      v.pstep = mode_mods(v.mode) * v.Rc * v.ncs;
      v.rstep = (int64_t)mode_mods(v.mode) * v.G * v.Rc * v.nct * v.nz * v.h * v.h * v.NT * v.Nt;
      v.planes = (__nv_bfloat16*)((char*)buf + off);
      off += planes_bytes(v.mode, v.K, v.h, v.snz, v.Rc);
      v.res = (int16_t*)((char*)buf + off);
      off += res_bytes(v.mode, v.NT * v.Nt, v.h, v.nz, v.Rc, v.G);
      v.item0 = it;
      v.pl0 = pl;
      v.rc0 = rb;
      v.mx0 = mx;
      it += (unsigned)(tiles(v) * v.G);
      pl += (unsigned)((int64_t)((v.h + 7) / 8) * v.h * v.snz * v.ncs * v.Rc);
      const unsigned pairs = (unsigned)(v.d + 1) / 2;
      v.pinv = (unsigned)((0xffffffffull + pairs) / pairs);
      rb += (unsigned)(((int64_t)v.nz * v.h * v.h * v.nct * v.Rc * pairs + kRebuild - 1) / kRebuild);
      mx += (unsigned)((((int64_t)1 << (3 * v.slevel)) + kMaxBoxes - 1) / kMaxBoxes * v.Rc);
      const uint32_t ks = (uint32_t)std::max(v.ks0, v.nchunk > v.n0 ? v.ks1 : 0);
      stage = std::max(stage, ks * 32u * (uint32_t)v.Nt);
      win = std::max(win, ks * kWinStep);
      pl_smem = std::max(pl_smem, (size_t)8 * (v.K + 1) * sizeof(long long));
      const cuuint64_t hh = (cuuint64_t)v.h;
      cuuint64_t dims[5] = {8 * hh, hh, (cuuint64_t)v.snz, (cuuint64_t)v.K / 8,
                            (cuuint64_t)mode_parts(v.mode) * v.pstep};
      cuuint64_t strides[4] = {16 * hh, 16 * hh * hh, 16 * hh * hh * v.snz, 16 * hh * hh * v.snz * (v.K / 8)};
      cuuint32_t box[5] = {8 * (kTX + 2), kTY, kTZ + 2, 2, 1};
      cuuint32_t estr[5] = {1, 1, 1, 1, 1};
      const CUresult r = encode(&maps.m[q], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, v.planes, dims, strides, box, estr,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
        return EIFMM_ECUDA;
      }
    }
    a.stage_b = stage;
    a.win_b = win;
    a.stages = (int)std::min<uint32_t>(kMaxStages, (kSmemMax - 1024 - kSmemBars - kWins * win) / stage);
    const uint32_t smem = 1024 + kSmemBars + kWins * win + (uint32_t)a.stages * stage;
    // a level that runs in several slabs needs its maximum once; repeating it
    // per slab gives the same value
    k_crt_max<<<mx, 256, 0, s>>>(a);
    EIFMM_CHECK_LAUNCH();
    const bool box = a.lv[0].mode == kCrtBox;
    if (box) k_crt_planes<kBoxMods><<<pl, 256, pl_smem, s>>>(a);
    else k_crt_planes<kMods><<<pl, 256, pl_smem, s>>>(a);
    EIFMM_CHECK_LAUNCH();
    a.items = it;
    a.plane_blocks = pl;
    a.rebuild_blocks = rb;
    if (m2l) {
      k_crt_planes_rest<kMods><<<std::min(pl, 4 * (unsigned)nsm), 256, pl_smem, s>>>(a);
      EIFMM_CHECK_LAUNCH();
    }
    k_crt_gemm<false><<<std::min(it, (unsigned)nsm), kThreads, smem, s>>>(maps, a);
    if (m2l) {
      EIFMM_CHECK_LAUNCH();
      k_crt_gemm<true><<<std::min(it, (unsigned)nsm), kThreads, smem, s>>>(maps, a);
    }
    EIFMM_CHECK_LAUNCH();
    if (box) k_crt_rebuild<kBoxMods, 4, false><<<rb, kRebuild, 0, s>>>(a, kcb);
    else if (groups) k_crt_rebuild<kMods, 3, true><<<rb, kRebuild, 0, s>>>(a, kc);
    else k_crt_rebuild<kMods, 3, false><<<rb, kRebuild, 0, s>>>(a, kc);
    EIFMM_CHECK_LAUNCH();
    if (m2l) {
      k_crt_weak<<<8 * (unsigned)nsm, kRebuild, 0, s>>>(a, kweak);
      EIFMM_CHECK_LAUNCH();
    }
    i0 = i1;
  }
  return EIFMM_OK;
}

}  // namespace eifmm
