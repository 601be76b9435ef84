// point64.cu -- the point kernels of the FP64 far field and near field for
// K = 1/r and the config-3 kernel: P2M (step 1), L2P (step 7 with the sum and the un-permute) and the
// direct sum over the 27 neighbouring leaves, with the kernel from integer
// coordinate differences (inv_fx.cuh) and the sums in FP64.
//
// Their bound is the integer and FP32 issue: about 75 instructions per kernel
// value, of which one FP64 FMA per right-hand side; on the FP64 pipe alone a
// value takes 20 operations at 2 per clock and SM.  A loop of values reaches
// 2.2e11/s against 3.6e10/s in FP64.  2^20 points, depth 5 (FP64 before): near
// field 34.0 -> 4.1 ms (8.5e8 pairs), P2M 6.3 -> 1.3 and L2P 7.9 -> 1.0 ms at d =
// 193.
//
// A distance below 2^54 units (L / 64 to L / 128 of box-relative coordinates, 1 / 128
// of two leaf widths between points) is formed in FP64.  From depth 7 on the nearest
// nodes are that close, from depth 8 on most; the mapping of the threads still pays:
// 200,000 points, P2M and L2P in FP64 before and now, depth 7, d = 126, 4.05 -> 1.95
// and 20.7 -> 1.69 ms; depth 8, d = 32, 3.90 -> 1.44 and 5.87 -> 1.01 ms; 20,000
// points within 1e-4, all pairs that close, near field 1,840 -> 52 ms.
#include <algorithm>
#include <cmath>

#include "inv_fx.cuh"
#include "internal.h"

namespace eifmm {
namespace {

constexpr int FX_THREADS = 128;

__global__ void k_to_fx(const double* __restrict__ x, int64_t n, int K, long long* __restrict__ q) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    q[i] = to_fx(x[i], K);
}

// Coordinates relative to the leaf centre c in units of 2^-K2 from the point's
// coordinate q in units of 2^-K (both modulo 2^64; the difference is small).
__device__ __forceinline__ long long local_fx(long long q, long long cq, int shift) {
  return (q - cq + (1ll << (shift - 1))) >> shift;
}

// The kernel value of an integer difference; false where the integers do not
// reach (points closer than 2^54 units).
template <int KERN>
__device__ __forceinline__ bool fx_value(long long dx, long long dy, long long dz, int kb, const FxConfig3& c3,
                                         double* kv) {
  if (KERN == EIFMM_KERNEL_CONFIG3) return config3_fx(dx, dy, dz, kb, c3, kv);
  return inv_fx(dx, dy, dz, kb, kv);
}
// There, in FP64.
template <int KERN>
__device__ __noinline__ double fx_slow(double z0, double z1, double z2) {
  return kern_f64(KERN, z0, z1, z2);
}

struct FxLeaf {
  double lo[3], lk;  // corner of the cube, half width of a leaf
  int depth, K, K2;  // units 2^-K of the points, 2^-K2 of box-relative coordinates
  FxConfig3 c3, c32;  // constants of the config-3 kernel in units of the points and of the boxes
};
__device__ __forceinline__ void leaf_centre(const FxLeaf& f, int b, double* c) {
  int ic[3];
  morton_decode(b, f.depth, ic);
  for (int a = 0; a < 3; ++a) c[a] = f.lo[a] + (2.0 * ic[a] + 1.0) * f.lk;
}

// Step 1: W_m^I = sum_j sigma_j / |x_m - (y_j - c_I)|.  One CTA per non-empty
// leaf, one thread per coefficient (in passes), the leaf's points staged as
// integers; RCT right-hand sides share a kernel value.
template <int KERN, int RCT>
__global__ void __launch_bounds__(256)
k_p2m_fx(FxLeaf lf, const int32_t* __restrict__ leaves, const int32_t* __restrict__ off,
         const double* __restrict__ px, const double* __restrict__ py, const double* __restrict__ pz,
         const long long* __restrict__ qx, const long long* __restrict__ qy, const long long* __restrict__ qz,
         const double* __restrict__ sig, int64_t n, int R, const double* __restrict__ X,
         const long long* __restrict__ Xq, int d, double* __restrict__ W) {
  constexpr int NP = 64;
  __shared__ longlong2 s_xy[NP];
  __shared__ long long s_z[NP];
  __shared__ double s_s[NP][RCT];
  const int b = leaves[blockIdx.x];
  double c[3];
  leaf_centre(lf, b, c);
  const long long cq0 = to_fx(c[0], lf.K), cq1 = to_fx(c[1], lf.K), cq2 = to_fx(c[2], lf.K);
  const int shift = lf.K - lf.K2, kb = lf.K2 + 958;
  const int beg = off[b], end = off[b + 1];
  for (int r0 = 0; r0 < R; r0 += RCT) {
    for (int m0 = 0; m0 < d; m0 += blockDim.x) {
      const int m = m0 + threadIdx.x;
      long long x0 = 0, x1 = 0, x2 = 0;
      if (m < d) {
        x0 = Xq[3 * m];
        x1 = Xq[3 * m + 1];
        x2 = Xq[3 * m + 2];
      }
      double acc[RCT];
#pragma unroll
      for (int rr = 0; rr < RCT; ++rr) acc[rr] = 0.0;
      for (int j0 = beg; j0 < end; j0 += NP) {
        const int cnt = min(NP, end - j0);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
          const int j = j0 + t;
          s_xy[t] = make_longlong2(local_fx(qx[j], cq0, shift), local_fx(qy[j], cq1, shift));
          s_z[t] = local_fx(qz[j], cq2, shift);
#pragma unroll
          for (int rr = 0; rr < RCT; ++rr) s_s[t][rr] = r0 + rr < R ? sig[j + (r0 + rr) * n] : 0.0;
        }
        __syncthreads();
        if (m < d)
#pragma unroll 2
          for (int t = 0; t < cnt; ++t) {
            const longlong2 xy = s_xy[t];
            double kv;
            if (!fx_value<KERN>(x0 - xy.x, x1 - xy.y, x2 - s_z[t], kb, lf.c32, &kv))
              kv = fx_slow<KERN>(X[3 * m] - (px[j0 + t] - c[0]), X[3 * m + 1] - (py[j0 + t] - c[1]),
                            X[3 * m + 2] - (pz[j0 + t] - c[2]));
#pragma unroll
            for (int rr = 0; rr < RCT; ++rr) acc[rr] += s_s[t][rr] * kv;
          }
      }
      if (m < d)
#pragma unroll
        for (int rr = 0; rr < RCT; ++rr)
          if (r0 + rr < R) W[((int64_t)b * R + r0 + rr) * d + m] = acc[rr];
    }
  }
}

// Step 7 + sum + un-permute.  One CTA per non-empty leaf; a thread takes one
// point of the pass and one slice of the l (32 points: 4 slices), the slices are
// added in order.
template <int KERN, int RCT>
__global__ void __launch_bounds__(FX_THREADS)
k_l2p_fx(FxLeaf lf, const int32_t* __restrict__ leaves, const int32_t* __restrict__ off,
         const int32_t* __restrict__ perm, const double* __restrict__ px, const double* __restrict__ py,
         const double* __restrict__ pz, const long long* __restrict__ qx, const long long* __restrict__ qy,
         const long long* __restrict__ qz, int64_t n, int R, const double* __restrict__ X,
         const long long* __restrict__ Xq, int d, const double* __restrict__ lh, const double* __restrict__ fnear,
         double* __restrict__ ffar, double* __restrict__ f, int64_t ld_f) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  longlong2* s_xy = reinterpret_cast<longlong2*>(fx_smem);  // [d]
  long long* s_z = reinterpret_cast<long long*>(s_xy + d);  // [d]
  double* s_l = reinterpret_cast<double*>(s_z + d);         // [d][RCT]
  __shared__ double s_red[RCT][FX_THREADS];
  const int tid = threadIdx.x;
  const int b = leaves[blockIdx.x];
  double c[3];
  leaf_centre(lf, b, c);
  const long long cq0 = to_fx(c[0], lf.K), cq1 = to_fx(c[1], lf.K), cq2 = to_fx(c[2], lf.K);
  const int shift = lf.K - lf.K2, kb = lf.K2 + 958;
  const int beg = off[b], end = off[b + 1];
  for (int l = tid; l < d; l += FX_THREADS) {
    s_xy[l] = make_longlong2(Xq[3 * l], Xq[3 * l + 1]);
    s_z[l] = Xq[3 * l + 2];
  }
  for (int r0 = 0; r0 < R; r0 += RCT) {
    __syncthreads();
    for (int t = tid; t < RCT * d; t += FX_THREADS) {
      const int rr = t / d, l = t - rr * d;
      s_l[l * RCT + rr] = r0 + rr < R ? lh[((int64_t)b * R + r0 + rr) * d + l] : 0.0;
    }
    __syncthreads();
    for (int t0 = beg, P = 0; t0 < end; t0 += P) {
      const int m = end - t0;
      P = m >= FX_THREADS ? FX_THREADS : (m > 32 ? 32 : m);
      const int S = min(FX_THREADS / P, 32);
      const int ti = tid % P, si = tid / P;
      const bool act = si < S;
      const int p = t0 + ti;
      double acc[RCT];
#pragma unroll
      for (int rr = 0; rr < RCT; ++rr) acc[rr] = 0.0;
      if (act) {
        const long long z0 = local_fx(qx[p], cq0, shift), z1 = local_fx(qy[p], cq1, shift),
                        z2 = local_fx(qz[p], cq2, shift);
        const int l0 = si * d / S, l1 = (si + 1) * d / S;
#pragma unroll 2
        for (int l = l0; l < l1; ++l) {
          const longlong2 xy = s_xy[l];
          double kv;
          if (!fx_value<KERN>(z0 - xy.x, z1 - xy.y, z2 - s_z[l], kb, lf.c32, &kv))
            kv = fx_slow<KERN>((px[p] - c[0]) - X[3 * l], (py[p] - c[1]) - X[3 * l + 1], (pz[p] - c[2]) - X[3 * l + 2]);
#pragma unroll
          for (int rr = 0; rr < RCT; ++rr) acc[rr] += kv * s_l[l * RCT + rr];
        }
      }
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < RCT; ++rr) s_red[rr][tid] = acc[rr];
      __syncthreads();
      for (int t = tid; t < P * RCT; t += FX_THREADS) {
        const int rr = t / P, q = t - rr * P, rg = r0 + rr;
        if (rg >= R) continue;
        double s = 0.0;
        for (int k = 0; k < S; ++k) s += s_red[rr][q + k * P];
        const int64_t pp = t0 + q;
        if (ffar) ffar[pp + rg * n] = s;
        f[perm[pp] + rg * ld_f] = s + fnear[pp + rg * n];
      }
    }
  }
}

// Near field f_N(x_i) = sum over the 27 neighbouring leaves of sigma_j / r.  One
// CTA per non-empty target leaf; the sources of the neighbourhood are staged in
// chunks of FX_SRC as integers; a thread takes one target of the pass and one
// slice of the chunk, and a target's slices are added in order.
constexpr int FX_SRC = 512;
template <int KERN, int RCT>
__global__ void __launch_bounds__(FX_THREADS)
k_p2p_fx(FxLeaf lf, const int32_t* __restrict__ leaves, const int32_t* __restrict__ toff,
         const double* __restrict__ tx, const double* __restrict__ ty, const double* __restrict__ tz,
         const long long* __restrict__ tqx, const long long* __restrict__ tqy, const long long* __restrict__ tqz,
         int64_t nt, const int32_t* __restrict__ soff, const double* __restrict__ sx, const double* __restrict__ sy,
         const double* __restrict__ sz, const long long* __restrict__ sqx, const long long* __restrict__ sqy,
         const long long* __restrict__ sqz, const double* __restrict__ sig, int64_t ns, int R, int exclude_self,
         double* __restrict__ fnear) {
  __shared__ longlong2 s_xy[FX_SRC];
  __shared__ long long s_z[FX_SRC];
  __shared__ double s_s[FX_SRC * RCT];
  __shared__ int s_j[FX_SRC];
  __shared__ double s_red[RCT][FX_THREADS];
  __shared__ int s_pos[28], s_beg[27];
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = leaves[blockIdx.x], kb = lf.K + 958;
  const int beg = toff[b], end = toff[b + 1];
  if ((int)blockIdx.y >= near_passes(end - beg)) return;
  if (tid < 32) {
    int c[3];
    morton_decode(b, lf.depth, c);
    const int n = 1 << lf.depth;
    int beg = 0, len = 0;
    if (lane < 27) {
      const int jx = c[0] + lane % 3 - 1, jy = c[1] + (lane / 3) % 3 - 1, jz = c[2] + lane / 9 - 1;
      if (jx >= 0 && jy >= 0 && jz >= 0 && jx < n && jy < n && jz < n) {
        const int64_t J = morton_encode(jx, jy, jz, lf.depth);
        beg = soff[J];
        len = soff[J + 1] - beg;
      }
      s_beg[lane] = beg;
    }
    int x = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < 28) s_pos[lane] = x - len;  // exclusive; lane 27: the total
  }
  __syncthreads();
  const int total = s_pos[27];
  for (int r0 = 0; r0 < R; r0 += RCT) {
    int staged = -1, pass = 0;
    for (int t0 = beg, P = 0; t0 < end; t0 += P) {
      const int m = end - t0;
      P = m >= FX_THREADS ? FX_THREADS : (m > 32 ? 32 : m);
      if (pass++ % (int)gridDim.y != (int)blockIdx.y) continue;
      const int S = min(FX_THREADS / P, 32);
      const int ti = tid % P, si = tid / P;
      const bool act = si < S;
      const int p = t0 + ti;
      double acc[RCT];
#pragma unroll
      for (int rr = 0; rr < RCT; ++rr) acc[rr] = 0.0;
      const long long x0 = tqx[p], x1 = tqy[p], x2 = tqz[p];
      for (int c0 = 0; c0 < total; c0 += FX_SRC) {
        const int cn = min(FX_SRC, total - c0);
        if (staged != c0) {
          __syncthreads();
          for (int i = tid; i < cn; i += FX_THREADS) {
            const int pos = c0 + i;
            int sg = 0;  // the last segment that starts at or before pos
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
              if (sg + step < 27 && s_pos[sg + step] <= pos) sg += step;
            const int j = s_beg[sg] + (pos - s_pos[sg]);
            s_j[i] = j;
            s_xy[i] = make_longlong2(sqx[j], sqy[j]);
            s_z[i] = sqz[j];
#pragma unroll
            for (int rr = 0; rr < RCT; ++rr) s_s[i * RCT + rr] = r0 + rr < R ? sig[j + (r0 + rr) * ns] : 0.0;
          }
          __syncthreads();
          staged = c0;
        }
        if (act) {
          const int i0 = si * cn / S, i1 = (si + 1) * cn / S;
#pragma unroll 2
          for (int i = i0; i < i1; ++i) {
            const longlong2 xy = s_xy[i];
            double kv;
            if (!fx_value<KERN>(x0 - xy.x, x1 - xy.y, x2 - s_z[i], kb, lf.c3, &kv)) {
              const int j = s_j[i];
              if (exclude_self && j == p) continue;
              kv = fx_slow<KERN>(tx[p] - sx[j], ty[p] - sy[j], tz[p] - sz[j]);
            }
#pragma unroll
            for (int rr = 0; rr < RCT; ++rr) acc[rr] += s_s[i * RCT + rr] * kv;
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < RCT; ++rr) s_red[rr][tid] = acc[rr];
      __syncthreads();
      for (int t = tid; t < P * RCT; t += FX_THREADS) {
        const int rr = t / P, q = t - rr * P;
        if (r0 + rr >= R) continue;
        double s = 0.0;
        for (int k = 0; k < S; ++k) s += s_red[rr][q + k * P];
        fnear[t0 + q + (int64_t)(r0 + rr) * nt] = s;
      }
    }
  }
}

FxLeaf fx_leaf(const Tree* t) {
  FxLeaf f;
  for (int a = 0; a < 3; ++a) f.lo[a] = t->lo[a];
  f.lk = t->L * std::ldexp(1.0, -(t->depth + 1));
  f.depth = t->depth;
  f.K = fx_point_exponent(t->L, t->depth);
  f.K2 = fx_box_exponent(t->L);
  const FxConfig3* c[2] = {&f.c3, &f.c32};
  for (int i = 0; i < 2; ++i) {
    // 1e-3 (53 bits) times 2^(2 K), 2 K <= 134
    int e = 0;
    const double m = std::ldexp(std::frexp(1e-3, &e), 53);
    const int sh = e - 53 + 2 * (i == 0 ? f.K : f.K2);
    const unsigned __int128 m128 = (unsigned __int128)m;
    const unsigned __int128 v = sh >= 0 && sh < 75 ? m128 << sh : sh < 0 && sh > -53 ? m128 >> -sh : 0;
    const_cast<FxConfig3*>(c[i])->e_hi = (unsigned long long)(v >> 64);
    const_cast<FxConfig3*>(c[i])->e_lo = (unsigned long long)v;
  }
  return f;
}

}  // namespace

// Differences of points of neighbouring leaves (up to two leaf widths) and of a
// box-relative point and an interpolation point (up to L) stay within 2^61.
int fx_point_exponent(double L, int depth) {
  int e = 0;
  std::frexp(L * std::ldexp(1.0, 1 - depth), &e);
  return 61 - e;
}
int fx_box_exponent(double L) {
  int e = 0;
  std::frexp(L, &e);
  return 61 - e;
}
// 1/r: the exponent field of the results stays in range (any L but extreme
// ones).  config-3, whose constants set a scale: r below 700 and 1e-3 in the 126
// bits of a square (depth 0: the box-relative coordinates alone).
bool fx_usable(int kern, double L, int depth) {
  int e = 0;
  std::frexp(L, &e);
  if (kern == EIFMM_KERNEL_INV_R) return e > -800 && e < 800;
  if (kern == EIFMM_KERNEL_CONFIG3)
    return e <= 8 && fx_box_exponent(L) <= 67 && (depth == 0 || fx_point_exponent(L, depth) <= 67);
  return false;
}

eifmm_status launch_to_fx(const double* x, int64_t n, int K, long long* q, cudaStream_t s) {
  if (n <= 0) return EIFMM_OK;
  k_to_fx<<<(unsigned)std::min<int64_t>((n + 255) / 256, 8192), 256, 0, s>>>(x, n, K, q);
  EIFMM_CHECK_LAUNCH();
  return EIFMM_OK;
}

// Integer coordinates of the tree's points into ws.fx_src and ws.fx_tgt (x, y, z
// one after the other).
eifmm_status launch_fx_points(const Tree* t, cudaStream_t s) {
  const Workspace& ws = t->ws;
  const int K = fx_point_exponent(t->L, t->depth);
  const PointSet* sets[2] = {&t->src, &t->tgt};
  for (int i = 0; i < (t->same ? 1 : 2); ++i) {
    const PointSet& p = *sets[i];
    long long* q = i == 0 ? ws.fx_src : ws.fx_tgt;
    const double* c[3] = {p.x, p.y, p.z};
    for (int a = 0; a < 3; ++a) EIFMM_TRY(launch_to_fx(c[a], p.n, K, q + a * p.n, s));
  }
  return EIFMM_OK;
}

eifmm_status launch_p2m_fx(const Tree* t, int kern, const LevelOps& v, int R, double* W, cudaStream_t s) {
  const PointSet& S = t->src;
  if (S.n_nonempty == 0) return EIFMM_OK;
  const FxLeaf f = fx_leaf(t);
  const long long* q = t->ws.fx_src;
  // passes of equal size over the coefficients, at most 256 threads
  const int passes = (v.d + 255) / 256, threads = (((v.d + passes - 1) / passes) + 31) / 32 * 32;
#define EIFMM_P2M_FX(K, RCT)                                                                                           \
  k_p2m_fx<K, RCT><<<S.n_nonempty, threads, 0, s>>>(f, S.nonempty, S.leaf_off, S.x, S.y, S.z, q, q + S.n, q + 2 * S.n, \
                                                 t->ws.sig, S.n, R, v.X, v.Xq, v.d, W)
  if (kern == EIFMM_KERNEL_CONFIG3) {
    if (R == 1) EIFMM_P2M_FX(EIFMM_KERNEL_CONFIG3, 1);
    else EIFMM_P2M_FX(EIFMM_KERNEL_CONFIG3, 4);
  } else if (R == 1) EIFMM_P2M_FX(EIFMM_KERNEL_INV_R, 1);
  else if (R <= 4) EIFMM_P2M_FX(EIFMM_KERNEL_INV_R, 4);
  else EIFMM_P2M_FX(EIFMM_KERNEL_INV_R, 8);
#undef EIFMM_P2M_FX
  EIFMM_CHECK_LAUNCH();
  return EIFMM_OK;
}

eifmm_status launch_l2p_fx(const Tree* t, int kern, const LevelOps& v, int R, double* f, int64_t ld_f, cudaStream_t s) {
  const PointSet& T = t->tgt;
  if (T.n_nonempty == 0) return EIFMM_OK;
  const FxLeaf lf = fx_leaf(t);
  const long long* q = t->same ? t->ws.fx_src : t->ws.fx_tgt;
  // d = 512 with 4 columns: 28 KB (8 columns would pass 48 KB with the sums)
#define EIFMM_L2P_FX(K, RCT)                                                                                        \
  k_l2p_fx<K, RCT><<<T.n_nonempty, FX_THREADS, (size_t)v.d * (24 + 8 * RCT), s>>>(                                  \
      lf, T.nonempty, T.leaf_off, T.perm, T.x, T.y, T.z, q, q + T.n, q + 2 * T.n, T.n, R, v.X, v.Xq, v.d, t->ws.lh, \
      t->ws.fnear, t->ws.ffar, f, ld_f)
  if (kern == EIFMM_KERNEL_CONFIG3) {
    if (R == 1) EIFMM_L2P_FX(EIFMM_KERNEL_CONFIG3, 1);
    else EIFMM_L2P_FX(EIFMM_KERNEL_CONFIG3, 4);
  } else if (R == 1) EIFMM_L2P_FX(EIFMM_KERNEL_INV_R, 1);
  else EIFMM_L2P_FX(EIFMM_KERNEL_INV_R, 4);
#undef EIFMM_L2P_FX
  EIFMM_CHECK_LAUNCH();
  return EIFMM_OK;
}

eifmm_status launch_p2p_fx(const Tree* t, int kern, int R, double* fnear, cudaStream_t s) {
  const PointSet &T = t->tgt, &S = t->src;
  if (T.n_nonempty == 0) return EIFMM_OK;
  const FxLeaf f = fx_leaf(t);
  const long long* sq = t->ws.fx_src;
  const long long* tq = t->same ? sq : t->ws.fx_tgt;
#define EIFMM_P2P_FX(K, RCT)                                                                                      \
  k_p2p_fx<K, RCT><<<dim3(T.n_nonempty, near_split(T.max_leaf)), FX_THREADS, 0, s>>>(                             \
      f, T.nonempty, T.leaf_off, T.x, T.y, T.z, tq, tq + T.n, tq + 2 * T.n, T.n, S.leaf_off, S.x, S.y, S.z, sq, \
      sq + S.n, sq + 2 * S.n, t->ws.sig, S.n, R, t->exclude_self, fnear)
  if (kern == EIFMM_KERNEL_CONFIG3) {
    if (R == 1) EIFMM_P2P_FX(EIFMM_KERNEL_CONFIG3, 1);
    else EIFMM_P2P_FX(EIFMM_KERNEL_CONFIG3, 4);
  } else if (R == 1) EIFMM_P2P_FX(EIFMM_KERNEL_INV_R, 1);
  else EIFMM_P2P_FX(EIFMM_KERNEL_INV_R, 4);
#undef EIFMM_P2P_FX
  EIFMM_CHECK_LAUNCH();
  return EIFMM_OK;
}

}  // namespace eifmm
