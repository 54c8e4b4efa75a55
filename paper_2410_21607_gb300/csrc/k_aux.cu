// Criterion, diagnostics and coordinate kernels.
//
//   adapt_column<N, EQ>: Sec. 3.1 threshold criterion.  One CTA per leaf
//     column; per element the criterion variables at every local node
//     (hanging nodes interpolated as in the modified DSS), their element
//     maxima, and the flag
//       +1 if max C^(lvl+1) > threshold(lvl+1) and lvl < lvl_max,
//       -1 if max C^lvl <= threshold(lvl) and lvl > 0, else 0,
//     with C^l the variable chosen for level l (speed by default; vertical
//     vorticity or dry Ertel potential vorticity from element-local
//     derivatives).  adapt_speed<N, EQ> is the same criterion where every level
//     uses the speed (not on small thin meshes).  The speed is evaluated with explicitly rounded float64
//     operations (sqrt(U U + V V + W W) / rho in that order, no contraction
//     into FMA) so that the decision is taken in float64 exactly as written.
//   diag_partial, diag_level: Sec. 4.2 diagnostics per vertical level: maximum
//     horizontal speed and the mass-weighted mean speed over the horizontal
//     sub-domain |x|, |y| <= half_width, reduced in a fixed order.
#include <algorithm>

#include "sem_internal.h"

namespace sem {

__constant__ double a_D[kMaxN + 1][(kMaxN + 1) * (kMaxN + 1)];  // [i][m] = h_m'(xi_i)

static int upload_aux_constants_now() {
  double D[kMaxN + 1][(kMaxN + 1) * (kMaxN + 1)] = {};
  for (int N = 2; N <= kMaxN; ++N) {
    const Basis1D& B = basis(N);
    for (int k = 0; k < (N + 1) * (N + 1); ++k) D[N][k] = B.D[k];
  }
  SEM_CUDA_TRY(cudaMemcpyToSymbol(a_D, D, sizeof(D)));
  return SEM_OK;
}

// the tables of the current device (uploaded on its first use)
static int upload_aux_constants() {
  static DeviceOnce once;
  return device_once(once, upload_aux_constants_now);
}

struct AdaptArgs {
  const double* q;
  const int* hmap;
  const int* hang_h;
  const double* hang_w;
  const int* col_level;
  const double* ref;
  const double* refG;             // warped layers: reference rows per node and hanging line, else null
  const double* refH;
  int8_t* flags;
  double* cmax;
  int nz, NZ;
  long long NG;
  int lvl_max;
  int need_grad;                  // 1: vorticity, 2: also potential vorticity
  double f;
  double thr[SEM_MAX_THRESHOLDS];
  int var[SEM_MAX_THRESHOLDS];    // SEM_CRIT_* per threshold
  double gx[16], gy[16];          // 2 / h per level
  const double* hzk;              // [nz] layer thicknesses
  // level the rule is evaluated for: per element (elem_level, [Ne]), or one
  // level for every element (level_all >= 0), else the column's own level;
  // the geometry always uses the column's level
  const int8_t* elem_level;
  int level_all;
  // warped layers: z_xi, z_eta, z_zeta per node of each column line
  // ([Ncol][Nq][nz][N+1][3]), else null
  const double* metric;
};

template <int N, int EQ>
__global__ void __launch_bounds__(((N + 1) * (N + 1) * (N + 1) + 31) / 32 * 32)
adapt_column(const AdaptArgs A) {
  constexpr int n1 = N + 1, Nq = n1 * n1, P = n1 * n1 * n1;
  constexpr int NW = (P + 31) / 32;
  __shared__ double red[3][NW];
  __shared__ double sQ[4][P];     // u, v, w, theta at the element's nodes
  const int col = blockIdx.x, t = threadIdx.x;
  const bool act = t < P;
  const int i = t % n1, j = (t / n1) % n1, c = t / Nq;
  const int ab = i + n1 * j;
  const int hm = act ? A.hmap[(long long)col * Nq + ab] : 0;
  const int geo_lev = A.col_level[col];
  for (int k = 0; k < A.nz; ++k) {
    double s = 0.0, zeta = 0.0, pv = 0.0, rho = 1.0;
    if (act) {
      const int kz = k * N + c;
      double v[kFields] = {0, 0, 0, 0, 0};
      if (hm >= 0) {
        const double* p = A.q + (long long)hm * A.NZ + kz;
        for (int f = 0; f < kFields; ++f) v[f] = p[(long long)f * A.NG];
      } else {
        const int h = -1 - hm;
        for (int m = 0; m <= N; ++m) {
          const double w = A.hang_w[h * n1 + m];
          const double* p = A.q + (long long)A.hang_h[h * n1 + m] * A.NZ + kz;
          for (int f = 0; f < kFields; ++f) v[f] = __dadd_rn(v[f], __dmul_rn(w, p[(long long)f * A.NG]));
        }
      }
      double ss = __dadd_rn(__dadd_rn(__dmul_rn(v[1], v[1]), __dmul_rn(v[2], v[2])), __dmul_rn(v[3], v[3]));
      s = __dsqrt_rn(ss);
      const double* rf = !A.refG ? A.ref + (long long)kz * kRef
                         : (hm >= 0 ? A.refG + ((long long)hm * A.NZ + kz) * kRef
                                    : A.refH + ((long long)(-1 - hm) * A.NZ + kz) * kRef);
      rho = rf[3] + v[0];
      if (EQ == 0) s = __ddiv_rn(s, __dadd_rn(rf[3], v[0]));
      if (A.need_grad) {
        if (EQ == 0) {
          sQ[0][t] = v[1] / rho;
          sQ[1][t] = v[2] / rho;
          sQ[2][t] = v[3] / rho;
          sQ[3][t] = (rf[4] + v[4]) / rho;
        } else {
          sQ[0][t] = v[1];
          sQ[1][t] = v[2];
          sQ[2][t] = v[3];
          sQ[3][t] = rf[0] + v[4];
        }
      }
    }
    if (A.need_grad) {
      __syncthreads();
      if (act) {
        // element-local derivatives d/dx (along i), d/dy (along j), d/dz (along c)
        double d[4][3] = {};
        for (int m = 0; m < n1; ++m) {
          const double Di = a_D[N][i * n1 + m], Dj = a_D[N][j * n1 + m], Dc = a_D[N][c * n1 + m];
          const int lx = m + n1 * j + Nq * c, ly = i + n1 * m + Nq * c, lz = i + n1 * j + Nq * m;
          for (int qv = 0; qv < 4; ++qv) {
            d[qv][0] += Di * sQ[qv][lx];
            d[qv][1] += Dj * sQ[qv][ly];
            d[qv][2] += Dc * sQ[qv][lz];
          }
        }
        const double gx = A.gx[geo_lev], gy = A.gy[geo_lev];
        if (A.metric) {
          // warped layers: derivatives at constant height through the node's
          // metric, d/dx = (2/hx) (d/dxi - (z_xi / z_zeta) d/dzeta), d/dz = d/dzeta / z_zeta
          const double* mt = A.metric + ((((long long)col * Nq + ab) * A.nz + k) * n1 + c) * 3;
          const double zx = mt[0], zy = mt[1], zz = mt[2];
          for (int qv = 0; qv < 4; ++qv) {
            const double dz = d[qv][2] / zz;
            d[qv][0] = gx * (d[qv][0] - zx * dz);
            d[qv][1] = gy * (d[qv][1] - zy * dz);
            d[qv][2] = dz;
          }
        } else {
          const double gz = 2.0 / A.hzk[k];
          for (int qv = 0; qv < 4; ++qv) {
            d[qv][0] *= gx;
            d[qv][1] *= gy;
            d[qv][2] *= gz;
          }
        }
        const double wz = d[1][0] - d[0][1];
        zeta = fabs(wz);
        if (A.need_grad > 1) {
          const double wx = d[2][1] - d[1][2], wy = d[0][2] - d[2][0];
          pv = fabs(wx * d[3][0] + wy * d[3][1] + (wz + A.f) * d[3][2]) / rho;
        }
      }
    }
    // block maxima over the element's nodes
    double mv[3] = {s, zeta, pv};
    for (int cv = 0; cv < 3; ++cv) {
      double x = mv[cv];
      for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
      if ((t & 31) == 0) red[cv][t >> 5] = x;
    }
    __syncthreads();
    if (t == 0) {
      double mx[3];
      for (int cv = 0; cv < 3; ++cv) {
        mx[cv] = red[cv][0];
        for (int w = 1; w < NW; ++w) mx[cv] = fmax(mx[cv], red[cv][w]);
      }
      const long long e = (long long)col * A.nz + k;
      const int lev = A.elem_level ? (int)A.elem_level[e] : (A.level_all >= 0 ? A.level_all : geo_lev);
      int flag = 0;
      if (lev < A.lvl_max && mx[A.var[lev]] > A.thr[lev]) flag = 1;
      else if (lev > 0 && mx[A.var[lev - 1]] <= A.thr[lev - 1]) flag = -1;
      A.flags[e] = (int8_t)flag;
      if (A.cmax) {
        const int test = lev < A.lvl_max ? lev : lev - 1;
        A.cmax[e] = mx[(test >= 0 && test < SEM_MAX_THRESHOLDS) ? A.var[test] : A.var[0]];
      }
    }
    __syncthreads();
  }
}


// The speed criterion (no derivatives).  What it needs per element is the
// maximum over the nodes of s = sqrt(U U + V V + W W) / rho in float64, and
// a float64 square root and divide at every node is what the general kernel
// above spends its time on (float64 pipe; 64x64x16, N = 4: 672 us for 137 MB of
// state, here 59 us).  Here a thread owns a level of a column and first bounds s at the
// level's (N+1)^2 nodes in float32; only nodes whose upper bound reaches the
// largest lower bound of a layer they belong to can hold its maximum, and
// only those are evaluated in float64, with the same rounded operations in
// the same order, so the maxima and the flags are those of the general kernel
// bit for bit.  A layer whose bounds are of no use (a density that is not
// positive, values outside float32's range, a tiny maximum) evaluates all of
// its nodes; a plane of exact zeros has the maximum 0.  A level that two
// layers share is bounded once.  Lanes run along z, so the loads are
// contiguous; what is left is instruction issue and the loads' latency.
template <int N, int EQ>
__device__ __forceinline__ void criterion_node(const AdaptArgs& A, const int hm, const int kz, double (&v)[4]) {
  // rho', U, V, W as the general kernel forms them
  if (hm >= 0) {
    const double* p = A.q + (long long)hm * A.NZ + kz;
#pragma unroll
    for (int f = EQ == 0 ? 0 : 1; f < 4; ++f) v[f] = __ldg(p + (long long)f * A.NG);
  } else {
    const int h = -1 - hm;
#pragma unroll
    for (int f = 0; f < 4; ++f) v[f] = 0.0;
    for (int m = 0; m <= N; ++m) {
      const double w = A.hang_w[h * (N + 1) + m];
      const double* p = A.q + (long long)A.hang_h[h * (N + 1) + m] * A.NZ + kz;
#pragma unroll
      for (int f = EQ == 0 ? 0 : 1; f < 4; ++f) v[f] = __dadd_rn(v[f], __dmul_rn(w, __ldg(p + (long long)f * A.NG)));
    }
  }
}
__device__ __forceinline__ double ref_rho(const AdaptArgs& A, const int hm, const int kz) {
  const double* rf = !A.refG ? A.ref + (long long)kz * kRef
                     : (hm >= 0 ? A.refG + ((long long)hm * A.NZ + kz) * kRef
                                : A.refH + ((long long)(-1 - hm) * A.NZ + kz) * kRef);
  return rf[3];
}
template <int N, int EQ>
__device__ __noinline__ double exact_speed(const AdaptArgs& A, const int hm, const int kz) {
  double v[4];
  criterion_node<N, EQ>(A, hm, kz, v);
  const double ss = __dadd_rn(__dadd_rn(__dmul_rn(v[1], v[1]), __dmul_rn(v[2], v[2])), __dmul_rn(v[3], v[3]));
  double s = __dsqrt_rn(ss);
  if (EQ == 0) s = __ddiv_rn(s, __dadd_rn(ref_rho(A, hm, kz), v[0]));
  return s;
}
// |x| as float32 by its bits (significand truncated).  Values below 2^-100
// give 0; `u` is the magnitude's upper half, for the caller's range checks.
constexpr unsigned kTinyHi = (1023u - 100u) << 20, kHugeHi = (1023u + 100u) << 20, kZeroHi = (1023u - 540u) << 20;
__device__ __forceinline__ float mag_f32(double x, unsigned& u) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  u = hi & 0x7fffffffu;
  // the 11-bit exponent less 896 is its low 8 bits with the top one flipped
  const float f = __uint_as_float((__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u);
  return u < kTinyHi ? 0.f : f;
}
__device__ __forceinline__ float near_f32(double x, unsigned& u) {
  return copysignf(mag_f32(x, u), __int_as_float(__double2hiint(x)));
}
// What a thread collects over its plane: ranges of the magnitudes' upper
// halves and of the density, from which the plane's bounds are judged once.
struct PlaneRange {
  unsigned top = 0u, low = 0u;   // largest magnitude; largest one that counted as 0
  float rmin = 1e30f, rmax = -1e30f;
};
// s^2 at a node in float32 and the factor-free excess e by which a hanging
// node's s may be larger.  Every operand is within 2^-23 of its value, the
// density (checked to stay within 1/4 .. 4 of its reference) within 7 2^-23,
// and the products, sums and the reciprocal add a few units: s^2 is within
// 6e-6 of its value, for which kSlack = 1e-5 is taken.  A hanging node is a
// weighted sum of nodes: its terms are bounded by their absolute sums.
constexpr float kSlack = 1e-5f;
template <int N, int EQ>
__device__ __forceinline__ float speed2(const AdaptArgs& A, const int hm, const int kz, const float rho0,
                                        PlaneRange& R, float& e) {
  float r = 1.f, s2;
  unsigned u;
  e = 0.f;
  if (hm >= 0) {
    const double* p = A.q + (long long)hm * A.NZ + kz;
    double d[4];
#pragma unroll
    for (int f = EQ == 0 ? 0 : 1; f < 4; ++f) d[f] = __ldg(p + (long long)f * A.NG);
    if (EQ == 0) {
      r = rho0 + near_f32(d[0], u);
      R.top = max(R.top, u);
    }
    s2 = 0.f;
#pragma unroll
    for (int f = 1; f < 4; ++f) {
      const float x = mag_f32(d[f], u);
      R.top = max(R.top, u);
      R.low = max(R.low, u < kTinyHi ? u : 0u);
      s2 = fmaf(x, x, s2);
    }
  } else {
    const int h = -1 - hm;
    float x[3] = {0.f, 0.f, 0.f}, a = 0.f, ar = 0.f;
    r = EQ == 0 ? 0.f : 1.f;
    for (int m = 0; m <= N; ++m) {
      const float w = near_f32(A.hang_w[h * (N + 1) + m], u);
      const double* p = A.q + (long long)A.hang_h[h * (N + 1) + m] * A.NZ + kz;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const float t = w * near_f32(__ldg(p + (long long)(f + 1) * A.NG), u);
        R.top = max(R.top, u);
        R.low = max(R.low, u < kTinyHi ? u : 0u);
        x[f] += t;
        a += fabsf(t);
      }
      if (EQ == 0) {
        const float t = w * near_f32(__ldg(p), u);
        R.top = max(R.top, u);
        r += t;
        ar += fabsf(t);
      }
    }
    if (EQ == 0) r += rho0;
    // a density that is too uncertain for the bounds: none
    if (EQ == 0 && !(ar * 4e-6f < 1e-7f * r)) r = -1.f;
    e = __fdividef(4e-6f * a, r);
    s2 = fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2]));
  }
  if (EQ == 0) {
    R.rmin = fminf(R.rmin, r);
    R.rmax = fmaxf(R.rmax, r);
    const float inv = __fdividef(1.f, r);
    s2 *= inv * inv;
  }
  return s2;
}
// the upper bound on s^2 from it
__device__ __forceinline__ float upper2(float s2, float e) {
  if (e > 0.f) {
    const float s = sqrtf(s2) + e;
    s2 = s * s;
  }
  return s2 * (1.f + kSlack);
}

constexpr int kSpeedThreads = 256;
template <int N, int EQ>
__global__ void __launch_bounds__(kSpeedThreads)
adapt_speed(const AdaptArgs A, const int ncol, const int cols, const int KL) {
  constexpr int n1 = N + 1, Nq = n1 * n1;
  extern __shared__ double s_ex[];                      // [items] exact maximum of a level, NaN: not needed
  const int LV = KL * N + 1;                            // levels of a chunk of KL layers
  float* s_lo = reinterpret_cast<float*>(s_ex + cols * LV);   // [items] largest lower bound on s^2
  float* s_hi = s_lo + cols * LV;                       // [items] largest upper bound; infinity: none
  for (int k0 = blockIdx.y * KL; k0 < A.nz; k0 += gridDim.y * KL) {
    const int kl = min(KL, A.nz - k0), nlev = kl * N + 1;
    const int c0 = blockIdx.x * cols, nc = min(cols, ncol - c0), items = nc * nlev;
    const int t = threadIdx.x;
    const bool act = t < items;
    const int lc = act ? t / nlev : 0, lv = act ? t - lc * nlev : 0, kz = k0 * N + lv;
    const int* hmap = A.hmap + (long long)(c0 + lc) * Nq;
    float lo = 0.f, hi = 0.f, hi2 = 0.f;
    int arg = 0;
    const float inf = __int_as_float(0x7f800000);
    if (act) {
      const float rho0 = EQ == 0 ? (float)A.ref[(long long)kz * kRef + 3] : 1.f;
      PlaneRange R;
      bool fits = rho0 > 1e-6f && rho0 < 1e18f;   // 1 / rho^2 is a normal number up to 9e18
#pragma unroll 5
      for (int ab = 0; ab < Nq; ++ab) {
        const int hm = hmap[ab];
        float r0 = rho0, e;
        if (EQ == 0 && A.refG) {
          // warped layers: the node's own reference density, taken relative to rho0's range
          r0 = (float)ref_rho(A, hm, kz);
          fits = fits && r0 > 0.5f * rho0 && r0 < 2.f * rho0;
        }
        const float s2 = speed2<N, EQ>(A, hm, kz, r0, R, e), u2 = upper2(s2, e);
        if (e == 0.f) lo = fmaxf(lo, s2);
        if (u2 > hi) {
          hi2 = hi;
          hi = u2;
          arg = ab;
        } else {
          hi2 = fmaxf(hi2, u2);
        }
      }
      lo *= 1.f - kSlack;
      // a plane whose bounds say nothing: infinity
      if (EQ == 0) fits = fits && R.rmin > 0.5f * rho0 && R.rmax < 2.f * rho0;
      fits = fits && R.top < kHugeHi && hi < 1e34f && !(R.low > kZeroHi && hi < 1e-24f);
      s_lo[t] = lo;
      s_hi[t] = fits ? hi : inf;
    }
    __syncthreads();
    if (act) {
      // the smaller of the layers' lower bounds that this level has to reach;
      // -1 (every node) where a layer holds a plane without bounds
      float need = inf;
      for (int s = 0; s < 2; ++s) {
        const int k = lv / N - s;                      // layers [k N, k N + N] that hold the level
        if (k < 0 || k >= kl || lv > k * N + N) continue;
        float m = 0.f, h = 0.f;
        for (int c = 0; c <= N; ++c) {
          m = fmaxf(m, s_lo[lc * nlev + k * N + c]);
          h = fmaxf(h, s_hi[lc * nlev + k * N + c]);
        }
        // a maximum below 1e-12 (s^2 below 1e-24): squares near float32's
        // underflow, no bound, except planes of zeros (hi = 0)
        if (!(h < 1e34f) || (h > 0.f && m < 1e-24f)) m = -1.f;
        need = fminf(need, m);
      }
      double ex = __longlong_as_double(0x7ff8000000000000ll);   // fmax ignores it
      if (need < 0.f || hi2 >= need) {
        if (need == 0.f && hi == 0.f) {
          ex = 0.0;                                    // zeros throughout
        } else {
          for (int ab = 0; ab < Nq; ++ab) {
            const int hm = hmap[ab];
            if (need >= 0.f) {
              PlaneRange R;
              float e;
              const float s2 = speed2<N, EQ>(A, hm, kz, EQ == 0 ? (float)ref_rho(A, hm, kz) : 1.f, R, e);
              if (upper2(s2, e) < need) continue;
            }
            ex = fmax(ex, exact_speed<N, EQ>(A, hm, kz));
          }
        }
      } else if (hi >= need) {
        ex = exact_speed<N, EQ>(A, hmap[arg], kz);
      }
      s_ex[t] = ex;
    }
    __syncthreads();
    for (int el = t; el < nc * kl; el += blockDim.x) {
      const int c = el / kl, k = el - c * kl;
      double mx = s_ex[c * nlev + k * N];
      for (int i = 1; i <= N; ++i) mx = fmax(mx, s_ex[c * nlev + k * N + i]);
      // the general kernel's idle lanes hold 0
      if ((n1 * Nq) % 32 != 0) mx = fmax(mx, 0.0);
      const long long e = (long long)(c0 + c) * A.nz + k0 + k;
      const int lev = A.elem_level ? (int)A.elem_level[e] : (A.level_all >= 0 ? A.level_all : A.col_level[c0 + c]);
      int flag = 0;
      if (lev < A.lvl_max && mx > A.thr[lev]) flag = 1;
      else if (lev > 0 && mx <= A.thr[lev - 1]) flag = -1;
      A.flags[e] = (int8_t)flag;
      if (A.cmax) A.cmax[e] = mx;
    }
    __syncthreads();
  }
}

static int sm_count() {
  int dev = 0, nsm = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  return nsm;
}

template <int N>
static void launch_speed(const AdaptArgs& A, int ncol, int eq, cudaStream_t st) {
  // layers per chunk: as many as the block's threads have levels; columns per
  // block: as many as fill it, one where the mesh has too few of them to give
  // every SM two blocks
  const int nsm = sm_count();
  const int KL = std::min(A.nz, (kSpeedThreads - 1) / N), LV = KL * N + 1;
  const int chunks = (A.nz + KL - 1) / KL;
  int cols = kSpeedThreads / LV;
  while (cols > 1 && (long long)((ncol + cols - 1) / cols) * chunks < 2LL * nsm) --cols;
  const int nt = (cols * LV + 31) / 32 * 32;
  const dim3 grid((unsigned)((ncol + cols - 1) / cols), (unsigned)std::min(chunks, 65535));
  const size_t sm = (size_t)cols * LV * 16;
  if (eq == 0)
    adapt_speed<N, 0><<<grid, nt, sm, st>>>(A, ncol, cols, KL);
  else
    adapt_speed<N, 1><<<grid, nt, sm, st>>>(A, ncol, cols, KL);
}

template <int N>
static void launch_adapt_n(const AdaptArgs& A, int ncol, int eq, cudaStream_t st) {
  constexpr int P = (N + 1) * (N + 1) * (N + 1);
  constexpr int nt = (P + 31) / 32 * 32;
  // The speed at every level: bounded in float32 first, except on small thin
  // meshes.  There a thread's chain over its level's (N+1)^2 nodes (7, 9, 12, 16 and
  // 20 us for N = 2 to 6, whatever the size) is longer than the general
  // kernel's, whose threads have a node per layer.  Microseconds, general and speed kernel: one layer, N = 3,
  // 1024 columns 7.6 and 9.2, 2500 15.5 and 9.1; N = 5, 324 columns 10.9 and 15.8, 600 16.8
  // and 15.8; two layers, N = 4, 144 columns 7.1 and 12.1, 600 14.8 and 12.2; N = 6, 144 columns
  // 13.9 and 20.1, 196 21.0 and 20.2; three layers, N = 4, 144 columns 9.9 and 12.1, 196 13.1
  // and 12.2; N = 2 8.0 and 6.8; four layers, N = 5 17.6 and 16.1.
  bool speed = true;
  for (int k = 0; k < SEM_MAX_THRESHOLDS; ++k) speed = speed && A.var[k] == SEM_CRIT_SPEED;
  const long long nsm = sm_count();
  const bool thin = A.nz <= 2 ? ncol <= nsm || (long long)ncol * A.nz * std::max(nt, 64) <= 600 * nsm
                              : A.nz == 3 && N >= 3 && ncol <= nsm;
  if (speed && !thin) return launch_speed<N>(A, ncol, eq, st);
  if (eq == 0)
    adapt_column<N, 0><<<ncol, nt, 0, st>>>(A);
  else
    adapt_column<N, 1><<<ncol, nt, 0, st>>>(A);
}

int launch_adapt(Mesh& m, const sem_params& p, const double* q, int8_t* flags, double* cmax,
                 cudaStream_t st, const int8_t* elem_level, int level_all) {
  DeviceTables& D = *m.dev;
  AdaptArgs A;
  A.elem_level = elem_level;
  A.level_all = level_all;
  A.q = q;
  A.hmap = D.hmap;
  A.hang_h = D.hang_h;
  A.hang_w = D.hang_w;
  A.col_level = D.col_level;
  A.ref = D.ref;
  A.refG = m.warped() ? D.refG : nullptr;
  A.refH = m.warped() ? D.refH : nullptr;
  A.flags = flags;
  A.cmax = cmax;
  A.nz = m.nz;
  A.NZ = m.NZ;
  A.NG = m.NG;
  A.lvl_max = p.lvl_max;
  A.need_grad = 0;
  for (int k = 0; k < SEM_MAX_THRESHOLDS; ++k) {
    A.thr[k] = p.thresholds[k];
    A.var[k] = p.criterion[k];
    // only the thresholds the levels use decide whether derivatives are needed
    if (k < p.n_thresholds && k < std::max(p.lvl_max, 1))
      A.need_grad = std::max(A.need_grad, p.criterion[k] == SEM_CRIT_PV ? 2 : (p.criterion[k] == SEM_CRIT_VORTICITY ? 1 : 0));
  }
  A.f = p.f;
  for (int l = 0; l < 16; ++l) {
    A.gx[l] = 2.0 / m.hx(l);
    A.gy[l] = 2.0 / m.hy(l);
  }
  A.hzk = D.hzk;
  A.metric = m.warped() ? D.metric : nullptr;
  if (A.need_grad) {
    int rc = upload_aux_constants();
    if (rc) return rc;
  }
  const int nc = (int)m.Ncol();
  switch (m.N) {
    case 2: launch_adapt_n<2>(A, nc, p.eqset, st); break;
    case 3: launch_adapt_n<3>(A, nc, p.eqset, st); break;
    case 4: launch_adapt_n<4>(A, nc, p.eqset, st); break;
    case 5: launch_adapt_n<5>(A, nc, p.eqset, st); break;
    case 6: launch_adapt_n<6>(A, nc, p.eqset, st); break;
    default: return fail(SEM_ERR_UNSUPPORTED, "order N not compiled");
  }
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

// ---------------------------------------------------------------------------
// Wind diagnostics in two passes.  diag_partial: one CTA per 8 to 32 horizontal
// nodes (diag_lines) lists those inside the sub-domain (most CTAs have none and end there)
// and, lanes along z so that the loads are contiguous, reduces each level over
// the list, dealt out to as many groups of warps as fit (a node costs a float64
// root and a divide, in a serial chain per level), the groups' values added in
// order; diag_level: one CTA per level reduces the CTAs' partial values in a
// fixed order.  64x64x16, N = 4, 100 km: 28 + 7 us; 135 us as one CTA per level
// walking all horizontal nodes with loads NZ apart.
constexpr int kDiagThreads = 384;
// Horizontal nodes per CTA of diag_partial.  More levels leave fewer groups, and
// the nodes of a small sub-domain, which lie side by side, fall on few SMs: with
// 32 nodes a CTA and 129 levels, 9216 nodes and 100 km took 62 us (48 as one
// launch), with 8 nodes 48.  On larger meshes the CTAs outside the sub-domain cost
// more than that: 65536 nodes, 65 levels, 20 km: 38 us with 32.
static int diag_lines(long long NH, int NZ) {
  return NZ <= 32 || NH >= 50000 ? 32 : (NH < 20000 ? 8 : 16);
}
__global__ void __launch_bounds__(kDiagThreads)
diag_partial(const double* __restrict__ q, const double* __restrict__ xh, const double* __restrict__ yh,
             const double* __restrict__ Mh, const double* __restrict__ ref, long long NH, int NZ, long long NG,
             double hw, int eq, const double* __restrict__ refG, const double* __restrict__ Minv_g, int lines,
             double* __restrict__ part /*[chunks][NZ][3]*/, int* __restrict__ count) {
  __shared__ int s_h[32];
  const long long h0 = (long long)blockIdx.x * lines;
  const int lane = threadIdx.x & 31;
  const bool in = lane < lines && h0 + lane < NH && fabs(xh[h0 + lane]) <= hw + 1e-6 && fabs(yh[h0 + lane]) <= hw + 1e-6;
  const unsigned mask = __ballot_sync(0xffffffffu, in);
  const int n = __popc(mask);
  if (threadIdx.x == 0) count[blockIdx.x] = n;
  if (n == 0) return;
  if (threadIdx.x < 32 && in) s_h[__popc(mask & ((1u << lane) - 1u))] = lane;
  __shared__ double s_v[3][kDiagThreads];
  const int LVT = min((NZ + 31) & ~31, kDiagThreads);   // threads of a group: one per level
  const int groups = kDiagThreads / LVT, gr = threadIdx.x / LVT, lt = threadIdx.x - gr * LVT;
  for (int k0 = 0; k0 < NZ; k0 += LVT) {
    __syncthreads();
    const int kz = k0 + lt;
    double mx = 0.0, num = 0.0, den = 0.0;
    if (kz < NZ && gr < groups) {
      const double rho0 = ref[(long long)kz * kRef + 3];
#pragma unroll 2
      for (int i = gr; i < n; i += groups) {
        const long long h = h0 + s_h[i], g = h * NZ + kz;
        const double U = q[NG + g], V = q[2 * NG + g];
        double s = sqrt(U * U + V * V);
        // warped layers: the node's own reference density and lumped mass (the
        // level means are then over a grid level, not a height)
        if (eq == 0) s = s / ((refG ? refG[g * kRef + 3] : rho0) + q[g]);
        const double wm = Minv_g ? 1.0 / Minv_g[g] : Mh[h];
        mx = fmax(mx, s);
        num += wm * s;
        den += wm;
      }
    }
    s_v[0][threadIdx.x] = mx;
    s_v[1][threadIdx.x] = num;
    s_v[2][threadIdx.x] = den;
    __syncthreads();
    if (gr == 0 && kz < NZ) {
      for (int i = 1; i < groups; ++i) {
        mx = fmax(mx, s_v[0][i * LVT + lt]);
        num += s_v[1][i * LVT + lt];
        den += s_v[2][i * LVT + lt];
      }
      double* o = part + ((long long)blockIdx.x * NZ + kz) * 3;
      o[0] = mx;
      o[1] = num;
      o[2] = den;
    }
  }
}

// a block's 256 values in a fixed order
__device__ __forceinline__ void diag_reduce(double mx, double num, double den, double* s_max, double* s_num,
                                            double* s_den, double* out) {
  s_max[threadIdx.x] = mx;
  s_num[threadIdx.x] = num;
  s_den[threadIdx.x] = den;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      s_max[threadIdx.x] = fmax(s_max[threadIdx.x], s_max[threadIdx.x + o]);
      s_num[threadIdx.x] += s_num[threadIdx.x + o];
      s_den[threadIdx.x] += s_den[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = s_max[0];
    out[1] = s_num[0];
    out[2] = s_den[0];
    out[3] = 0.0;
  }
}
__global__ void __launch_bounds__(256)
diag_level(const double* __restrict__ part, const int* __restrict__ count, int chunks, int NZ,
           double* __restrict__ out /*[NZ][4]*/) {
  __shared__ double s_max[256], s_num[256], s_den[256];
  const int kz = blockIdx.x;
  double mx = 0.0, num = 0.0, den = 0.0;
  for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
    if (count[c] == 0) continue;
    const double* p = part + ((long long)c * NZ + kz) * 3;
    mx = fmax(mx, p[0]);
    num += p[1];
    den += p[2];
  }
  diag_reduce(mx, num, den, s_max, s_num, s_den, out + kz * 4);
}
// Small meshes: one CTA per level walks all horizontal nodes, in one launch.
__global__ void __launch_bounds__(256)
diag_level_small(const double* __restrict__ q, const double* __restrict__ xh, const double* __restrict__ yh,
                 const double* __restrict__ Mh, const double* __restrict__ ref, long long NH, int NZ, long long NG,
                 double hw, int eq, const double* __restrict__ refG, const double* __restrict__ Minv_g,
                 double* __restrict__ out /*[NZ][4]*/) {
  __shared__ double s_max[256], s_num[256], s_den[256];
  const int kz = blockIdx.x;
  const double rho0 = ref[(long long)kz * kRef + 3];
  double mx = 0.0, num = 0.0, den = 0.0;
  for (long long h = threadIdx.x; h < NH; h += blockDim.x) {
    if (!(fabs(xh[h]) <= hw + 1e-6 && fabs(yh[h]) <= hw + 1e-6)) continue;
    const long long g = h * NZ + kz;
    const double U = q[NG + g], V = q[2 * NG + g];
    double s = sqrt(U * U + V * V);
    // warped layers: the node's own reference density and lumped mass (the
    // level means are then over a grid level, not a height)
    if (eq == 0) s = s / ((refG ? refG[g * kRef + 3] : rho0) + q[g]);
    const double wm = Minv_g ? 1.0 / Minv_g[g] : Mh[h];
    mx = fmax(mx, s);
    num += wm * s;
    den += wm;
  }
  diag_reduce(mx, num, den, s_max, s_num, s_den, out + kz * 4);
}

// doubles of D.diag_buf: the levels' results, the partial values, the counts
size_t diag_doubles(const Mesh& m) {
  const int lines = diag_lines(m.NH, m.NZ);
  const size_t chunks = (size_t)((m.NH + lines - 1) / lines);
  return (size_t)m.NZ * 4 + chunks * m.NZ * 3 + (chunks + 1) / 2;
}

int launch_diag(Mesh& m, const sem_params& p, const double* q, double hw, sem_diag_out* out,
                cudaStream_t st) {
  DeviceTables& D = *m.dev;
  const int lines = diag_lines(m.NH, m.NZ), chunks = (int)((m.NH + lines - 1) / lines);
  double* part = D.diag_buf + (size_t)m.NZ * 4;
  int* count = reinterpret_cast<int*>(part + (size_t)chunks * m.NZ * 3);
  const double *refG = m.warped() ? D.refG : nullptr, *Minv_g = m.warped() ? D.Minv_g : nullptr;
  // One launch up to 4096 nodes (16 per thread), and up to 8192 where about one
  // node per thread lies in the sub-domain (as if the nodes were spread evenly);
  // it walks all nodes and costs a root and a divide per 256 inside.  N = 4,
  // 17 levels, one launch and two: 4624 nodes, 20 km 32 and 35 us, 100 km 44 and 37, all
  // 60 and 36; 9216 nodes, 20 km 35 and 35; 65536 nodes, 100 km 94 and 46 (with the copy
  // to the host).  With many levels one launch fills the SMs by itself and stays
  // the faster one longer (129 levels, 100 km: 6400 nodes 45 and 53, 25600 58 and 53).
  const long long one = m.NZ > 80 ? std::min(128LL * m.NZ, 16384LL) : 4096;
  const double inside = (double)m.NH * std::min(1.0, 2.0 * hw / m.Lx) * std::min(1.0, 2.0 * hw / m.Ly);
  if (m.NH <= one || (m.NH <= 8192 && inside <= 256.0)) {
    diag_level_small<<<m.NZ, 256, 0, st>>>(q, D.xh, D.yh, D.Mh, D.ref, m.NH, m.NZ, m.NG, hw, p.eqset, refG, Minv_g,
                                           D.diag_buf);
  } else {
    diag_partial<<<chunks, kDiagThreads, 0, st>>>(q, D.xh, D.yh, D.Mh, D.ref, m.NH, m.NZ, m.NG, hw, p.eqset, refG,
                                                  Minv_g, lines, part, count);
    diag_level<<<m.NZ, 256, 0, st>>>(part, count, chunks, m.NZ, D.diag_buf);
  }
  SEM_CUDA_TRY(cudaGetLastError());
  std::vector<double> buf((size_t)m.NZ * 4);
  SEM_CUDA_TRY(cudaMemcpyAsync(buf.data(), D.diag_buf, buf.size() * sizeof(double),
                               cudaMemcpyDeviceToHost, st));
  SEM_CUDA_TRY(cudaStreamSynchronize(st));
  double mx = 0.0, mm = -1.0;
  for (int k = 0; k < m.NZ; ++k) {
    mx = std::max(mx, buf[k * 4]);
    if (buf[k * 4 + 2] > 0) mm = std::max(mm, buf[k * 4 + 1] / buf[k * 4 + 2]);
  }
  if (mm < 0) return fail(SEM_ERR_ARG, "no node inside the diagnostic sub-domain");
  out->max_wind = mx;
  out->max_mean_wind = mm;
  return SEM_OK;
}

// ---------------------------------------------------------------------------
// Criterion flags merged with a predictor's flags (the learned schedule, the
// criterion kept as the fallback): refine when either asks, coarsen only when
// both do, keep otherwise; a request the element's level cannot take (refine
// at lvl_max, coarsen at level 0) counts as keep.
__global__ void merge_flags_kernel(const int8_t* crit, const int8_t* pred, const int8_t* level, int lvl_max,
                                   long long n, int8_t* out) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int L = level[e];
    int c = crit[e], p = pred[e];
    if (L >= lvl_max) { c = c > 0 ? 0 : c; p = p > 0 ? 0 : p; }
    if (L <= 0) { c = c < 0 ? 0 : c; p = p < 0 ? 0 : p; }
    out[e] = (int8_t)((c > 0 || p > 0) ? 1 : ((c < 0 && p < 0) ? -1 : 0));
  }
}

int launch_merge_flags(const int8_t* crit, const int8_t* pred, const int8_t* level, int lvl_max, long long n,
                       int8_t* out, cudaStream_t st) {
  const long long blocks = std::max<long long>(1, std::min<long long>((n + 255) / 256, 152 * 8));
  merge_flags_kernel<<<(int)blocks, 256, 0, st>>>(crit, pred, level, lvl_max, n, out);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

// ---------------------------------------------------------------------------
__global__ void coords_kernel(const double* xh, const double* yh, const double* zk, long long NH,
                              int NZ, const double* zG, double* xyz) {
  const long long NG = NH * NZ;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < NG;
       g += (long long)gridDim.x * blockDim.x) {
    const long long h = g / NZ;
    const int k = (int)(g - h * NZ);
    xyz[g] = xh[h];
    xyz[NG + g] = yh[h];
    xyz[2 * NG + g] = zG ? zG[g] : zk[k];
  }
}

int launch_coords(Mesh& m, double* xyz, cudaStream_t st) {
  DeviceTables& D = *m.dev;
  long long blocks = std::min<long long>((m.NG + 255) / 256, 152 * 16);
  coords_kernel<<<(int)blocks, 256, 0, st>>>(D.xh, D.yh, D.zk, m.NH, m.NZ, m.warped() ? D.zG : nullptr, xyz);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace sem
