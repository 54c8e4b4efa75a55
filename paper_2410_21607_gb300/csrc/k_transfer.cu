// Solution transfer to an adapted mesh (Algorithm 3, "refine and coarsen
// marked elements").  The paper does not state the transfer operator; the
// one used:
//   1. new element values: unchanged columns copy theirs; a refined column's
//      children evaluate the parent polynomial at their nodes (horizontal
//      child interpolation P_a (x) P_b, z unchanged); a coarsened column takes
//      the exact L2 projection of its four children,
//      q = 1/4 sum_{a,b} (R_a (x) R_b) q_ab,  R_c = M^-1 P_c^T M  (M the exact
//      1-D mass matrix; the z direction is common to parent and children);
//   2. projection onto the continuous, hanging-node-constrained space,
//      (Q^T W Q) q_G = Q^T W q_L with W the LGL quadrature weights times the
//      Jacobian.  Q^T W Q = A_h (x) M_z: diagonal (the lumped mass) except on
//      the coarse-side nodes that hanging rows couple; those small coupled
//      blocks are solved by float64 iterative refinement whose corrections
//      come from a Jacobi-preconditioned float32 conjugate gradient, with
//      bounded iteration counts.
// The float64 pipe of this part is narrow (1/64 of the float32 rate): even a
// weight per copied value would bound a copy, so unchanged values are moved,
// not multiplied.
// The projection keeps every continuous field (refinement changes nothing)
// and the lumped total of every field.
#include <algorithm>
#include <numeric>

#include "sem_internal.h"

namespace sem {

__constant__ double c_P[kMaxN + 1][2][(kMaxN + 1) * (kMaxN + 1)];  // child interpolation
__constant__ double c_R[kMaxN + 1][2][(kMaxN + 1) * (kMaxN + 1)];  // child L2 projection, halved
__constant__ double c_tw[kMaxN + 1][kMaxN + 1];                     // LGL weights

static int upload_transfer_constants_now() {
  static double P[kMaxN + 1][2][(kMaxN + 1) * (kMaxN + 1)] = {};
  static double R[kMaxN + 1][2][(kMaxN + 1) * (kMaxN + 1)] = {};
  static double W[kMaxN + 1][kMaxN + 1] = {};
  for (int N = 2; N <= kMaxN; ++N) {
    const Basis1D& B = basis(N);
    const int n = N + 1;
    // inverse of the exact mass matrix (Gauss-Jordan, SPD, tiny)
    std::vector<double> M = B.Mex, Mi(n * n, 0.0);
    for (int i = 0; i < n; ++i) Mi[i * n + i] = 1.0;
    for (int col = 0; col < n; ++col) {
      int piv = col;
      for (int r = col + 1; r < n; ++r)
        if (std::fabs(M[r * n + col]) > std::fabs(M[piv * n + col])) piv = r;
      for (int q = 0; q < n; ++q) {
        std::swap(M[col * n + q], M[piv * n + q]);
        std::swap(Mi[col * n + q], Mi[piv * n + q]);
      }
      double d = M[col * n + col];
      for (int q = 0; q < n; ++q) {
        M[col * n + q] /= d;
        Mi[col * n + q] /= d;
      }
      for (int r = 0; r < n; ++r) {
        if (r == col) continue;
        double f = M[r * n + col];
        for (int q = 0; q < n; ++q) {
          M[r * n + q] -= f * M[col * n + q];
          Mi[r * n + q] -= f * Mi[col * n + q];
        }
      }
    }
    for (int c = 0; c < 2; ++c) {
      // R_c = M^-1 P_c^T M
      std::vector<double> T(n * n, 0.0);
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j)
          for (int q = 0; q < n; ++q) T[i * n + j] += B.P[c][q * n + i] * B.Mex[q * n + j];
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) {
          double s = 0.0;
          for (int q = 0; q < n; ++q) s += Mi[i * n + q] * T[q * n + j];
          R[N][c][i * n + j] = 0.5 * s;   // with the 1/4 of the four children
          P[N][c][i * n + j] = B.P[c][i * n + j];
        }
    }
    for (int i = 0; i < n; ++i) W[N][i] = B.w[i];
  }
  SEM_CUDA_TRY(cudaMemcpyToSymbol(c_P, P, sizeof(P)));
  SEM_CUDA_TRY(cudaMemcpyToSymbol(c_R, R, sizeof(R)));
  SEM_CUDA_TRY(cudaMemcpyToSymbol(c_tw, W, sizeof(W)));
  return SEM_OK;
}

// the tables of the current device (uploaded on its first use)
static int upload_transfer_constants() {
  static DeviceOnce once;
  return device_once(once, upload_transfer_constants_now);
}

struct TrArgs {
  const double* qold;
  const int* old_hmap;
  const int* old_hang_h;
  const double* old_hang_w;
  long long old_NG;
  const int* org;      // [Ncol][6]
  const int* new_level;
  double* out;         // new scratch [Ncol][Nq][5][NZ], mapped columns only
  int N, NZ;
  double hxy;          // Lx Ly / (nx ny) / 4: J of a level-0 column per unit w_a w_b
};

// New values of the refined and coarsened columns, out[col][ab][f][kz].  One
// CTA per new column (those of unchanged columns end at once); a thread owns
// one level of one field and holds the level's (N+1)^2 nodes in registers, so
// the two directions are contracted one after the other (per node and field
// 2 (N+1) FMAs for a refined column, 6 (N+1) for a coarsened one, where the
// 2-D operators applied node by node take (N+1)^2 and 4 (N+1)^2 and their
// weights), the operators are read as uniform constants and the lanes run
// along z.  Bound by the float64 pipe.  No factor of the vertical direction
// enters: parent and children share the levels, and the layers' weights
// cancel against the vertical lumped mass.  Remesh of 113 k elements, N = 4:
// 468 us, and 147 us for transfer_gather, which moves the unchanged lines
// itself; 2348 and 204 us when every column was mapped node by node and every
// value weighted.
// Values of one field and level on N + 1 lines of a source column.  The loads
// of all lines are issued before any is looked at (a hanging one's from line 0,
// then replaced): behind a branch per line they wait for one another, 100 times for a
// coarsened column of order 4, which thin meshes cannot hide (2 layers, order 4, 64
// columns: a coarsening 60 us, now 54).
template <int N>
__device__ __forceinline__ void old_values(const TrArgs& A, const int* hm, const int f, const int kz, double (&r)[N + 1]) {
  const double* q = A.qold + (long long)f * A.old_NG + kz;
  int h[N + 1];
#pragma unroll
  for (int m = 0; m <= N; ++m) h[m] = hm[m];
#pragma unroll
  for (int m = 0; m <= N; ++m) r[m] = __ldg(q + (long long)max(h[m], 0) * A.NZ);
#pragma unroll
  for (int m = 0; m <= N; ++m)
    if (h[m] < 0) {
      const int k = -1 - h[m];
      r[m] = 0.0;
#pragma unroll
      for (int n = 0; n <= N; ++n)
        r[m] += A.old_hang_w[k * (N + 1) + n] * __ldg(q + (long long)A.old_hang_h[k * (N + 1) + n] * A.NZ);
    }
}
// One (field, level) of a new column from its source columns.  The operator
// tables are indexed directly (not through a selected pointer, which would make
// their loads generic), c and d being the same for the whole CTA.
template <int N, bool COARSE>
__device__ __forceinline__ void new_plane(const TrArgs& A, const int* o, const int f, const int kz,
                                          double (&acc)[(N + 1) * (N + 1)]) {
  constexpr int n1 = N + 1, Nq = n1 * n1;
#pragma unroll
  for (int ab = 0; ab < Nq; ++ab) acc[ab] = 0.0;
#pragma unroll 1
  for (int b = 0; b < (COARSE ? 2 : 1); ++b) {
    double v[Nq];   // contracted along x
#pragma unroll
    for (int ab = 0; ab < Nq; ++ab) v[ab] = 0.0;
#pragma unroll 1
    for (int a = 0; a < (COARSE ? 2 : 1); ++a) {
      const int ca = COARSE ? a : (o[5] & 1);
      const int* hm = A.old_hmap + (long long)o[1 + a + 2 * b] * Nq;
#pragma unroll
      for (int j = 0; j < n1; ++j) {
        double r[n1];
        old_values<N>(A, hm + n1 * j, f, kz, r);
#pragma unroll
        for (int i = 0; i < n1; ++i)
#pragma unroll
          for (int m = 0; m < n1; ++m)
            v[i + n1 * j] = fma(COARSE ? c_R[N][ca][i * n1 + m] : c_P[N][ca][i * n1 + m], r[m], v[i + n1 * j]);
      }
    }
    const int cb = COARSE ? b : (o[5] >> 1);
#pragma unroll
    for (int j = 0; j < n1; ++j)
#pragma unroll
      for (int n = 0; n < n1; ++n) {
        const double y = COARSE ? c_R[N][cb][j * n1 + n] : c_P[N][cb][j * n1 + n];
#pragma unroll
        for (int i = 0; i < n1; ++i) acc[i + n1 * j] = fma(y, v[i + n1 * n], acc[i + n1 * j]);
      }
  }
}

constexpr int kTrThreads = 192;
template <int N>
__global__ void __launch_bounds__(kTrThreads, N <= 4 ? 2 : 1)
transfer_local(const TrArgs A) {
  constexpr int Nq = (N + 1) * (N + 1);
  const int col = blockIdx.x;
  const int* o = A.org + (long long)col * 6;
  const int kind = o[0];
  if (kind == 0) return;
  const long long ld = (long long)kFields * A.NZ;
  for (int it = threadIdx.x; it < kFields * A.NZ; it += blockDim.x) {
    const int f = it / A.NZ, kz = it - f * A.NZ;
    double acc[Nq];
    if (kind == 1) new_plane<N, false>(A, o, f, kz, acc);
    else new_plane<N, true>(A, o, f, kz, acc);
    double* dst = A.out + ((long long)col * Nq * kFields + f) * A.NZ + kz;
#pragma unroll
    for (int ab = 0; ab < Nq; ++ab) dst[ab * ld] = acc[ab];
  }
}

// Where the new line h comes from: meta[h] >= 0: every source is an unchanged
// column's node of the same old line, whose weighted mean is that line (a
// copy); meta[h] <= -2: the only source is node -2 - meta[h] of a mapped
// column; -1: the weighted sum over the sources.
__global__ void transfer_meta(const TrArgs A, const int4* __restrict__ rec_unit, const int* __restrict__ coupled,
                              int NH, int* __restrict__ meta) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= NH) return;
  const int Nq = (A.N + 1) * (A.N + 1);
  const int4 r = rec_unit[h];
  int m = -1;
  if (r.x >= 0 && !coupled[h]) {
    const int src[4] = {r.x, r.y, r.z, r.w};
    const int* o = A.org + (long long)(r.x / Nq) * 6;
    if (o[0] != 0) {
      if (r.y < 0) m = -2 - r.x;
    } else {
      m = A.old_hmap[(long long)o[1] * Nq + r.x % Nq];
      for (int e = 1; e < 4 && src[e] >= 0 && m >= 0; ++e) {
        const int* oe = A.org + (long long)(src[e] / Nq) * 6;
        if (oe[0] != 0 || A.old_hmap[(long long)oe[1] * Nq + src[e] % Nq] != m) m = -1;
      }
      if (m < 0) m = -1;
    }
  }
  meta[h] = m;
}

__global__ void __launch_bounds__(256)
transfer_gather(const TrArgs A, const int* __restrict__ meta, const int* __restrict__ qt_ptr,
                const int* __restrict__ qt_src, const double* __restrict__ qt_w,
                const double* __restrict__ Minv_h, const int* __restrict__ coupled, unsigned NG,
                double* __restrict__ q) {
  const unsigned NZ = (unsigned)A.NZ;
  for (unsigned g = blockIdx.x * blockDim.x + threadIdx.x; g < NG; g += gridDim.x * blockDim.x) {
    const unsigned h = g / NZ, kz = g - h * NZ;
    const int m = __ldg(meta + h);
    double v[kFields];
    if (m != -1) {
      const double* p = m >= 0 ? A.qold + (long long)m * NZ + kz
                               : A.out + (long long)(-2 - m) * kFields * NZ + kz;
      const long long ld = m >= 0 ? A.old_NG : (long long)NZ;
#pragma unroll
      for (int f = 0; f < kFields; ++f) v[f] = __ldg(p + f * ld);
    } else {
      const int n1 = A.N + 1, Nq = n1 * n1;
#pragma unroll
      for (int f = 0; f < kFields; ++f) v[f] = 0.0;
      const int end = qt_ptr[h + 1];
      for (int e = qt_ptr[h]; e < end; ++e) {
        const int src = qt_src[e], col = src / Nq, ab = src - col * Nq;
        const int* o = A.org + (long long)col * 6;
        // w_a w_b hx hy / 4 of the source's column, times the entry's weight
        const double w = qt_w[e] * (c_tw[A.N][ab % n1] * c_tw[A.N][ab / n1] *
                                    (A.hxy / (double)(1ll << (2 * A.new_level[col]))));
        if (o[0] != 0) {
          const double* p = A.out + (long long)src * kFields * NZ + kz;
#pragma unroll
          for (int f = 0; f < kFields; ++f) v[f] = fma(w, __ldg(p + f * (long long)NZ), v[f]);
          continue;
        }
        const int hm = A.old_hmap[(long long)o[1] * Nq + ab];
        if (hm >= 0) {
          const double* p = A.qold + (long long)hm * NZ + kz;
#pragma unroll
          for (int f = 0; f < kFields; ++f) v[f] = fma(w, __ldg(p + f * A.old_NG), v[f]);
        } else {
          const int k = -1 - hm;
          double u[kFields] = {0, 0, 0, 0, 0};
          for (int i = 0; i < n1; ++i) {
            const double wi = A.old_hang_w[k * n1 + i];
            const double* p = A.qold + (long long)A.old_hang_h[k * n1 + i] * NZ + kz;
#pragma unroll
            for (int f = 0; f < kFields; ++f) u[f] += wi * __ldg(p + f * A.old_NG);
          }
#pragma unroll
          for (int f = 0; f < kFields; ++f) v[f] = fma(w, u[f], v[f]);
        }
      }
      // coupled nodes keep b as the right-hand side of their block solve
      if (!coupled[h]) {
#pragma unroll
        for (int f = 0; f < kFields; ++f) v[f] *= Minv_h[h];
      }
    }
#pragma unroll
    for (int f = 0; f < kFields; ++f) q[(size_t)f * NG + g] = v[f];
  }
}

// Sums over the block of NR values per thread, the same in every thread.
template <typename T, int NR>
__device__ __forceinline__ void block_sums(T (&v)[NR], T* red) {
#pragma unroll
  for (int i = 0; i < NR; ++i)
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int i = 0; i < NR; ++i) red[(threadIdx.x >> 5) * NR + i] = v[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    T s = (T)0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w * NR + i];
    v[i] = s;
  }
}

// Coupled blocks, A x = b for NR right-hand sides (field, level) of one block
// at a time.  As a float64 conjugate gradient, one CTA per right-hand side,
// this was bound by the float64 pipe (84 % busy, 489 us on 113 k elements with
// 4 blocks of about 780 nodes and 165 right-hand sides; 396 us now, bound by the
// latency of the inner iteration).  Now the float64 work
// is the residual alone: with the symmetrically scaled matrix S A S (S =
// diag(A)^-1/2, entries of order 1, float32) a float32 conjugate gradient finds
// the correction to 1e-5, x and r are updated in float64 (r by r -= A d, so that
// its rounding shrinks with the corrections), and the residual falls by that factor per pass
// (S A S of a 2:1 block has a condition number below 2) until it is below 1e-15
// of the right-hand side, which takes four of the passes allowed; what has not
// got there by then is reported in the status word.  The matrix is read once
// for NR right-hand sides.
constexpr int kCgThreads = 512, kCgOuter = 12, kCgInner = 200;
template <int NR>
__global__ void __launch_bounds__(kCgThreads)
transfer_cg(const int* __restrict__ comp_ptr, const int* __restrict__ nodes, const int* __restrict__ A_ptr,
            const int* __restrict__ A_col, const double* __restrict__ A_val, const float* __restrict__ A32,
            const double* __restrict__ S, long long NG, int NZ, double* q, int* status) {
  extern __shared__ double sm[];
  __shared__ double red64[kCgThreads / 32 * NR];
  float* red = reinterpret_cast<float*>(red64);
  const int beg = comp_ptr[blockIdx.x], n = comp_ptr[blockIdx.x + 1] - beg;
  const int rhs0 = blockIdx.y * NR, nrhs = kFields * NZ;
  double* x = sm;                                  // [n][NR]
  double* r = x + (size_t)n * NR;
  float* p = reinterpret_cast<float*>(r + (size_t)n * NR);
  float* Ap = p + (size_t)n * NR;
  double* d = reinterpret_cast<double*>(p);        // the correction, over p and Ap
  float* z = Ap + (size_t)n * NR;                  // scaled residual of the inner iteration
  float* y = z + (size_t)n * NR;                   // its solution
  const int t = threadIdx.x, nt = blockDim.x;
  auto at = [&](int a, int i) {
    const int rhs = rhs0 + i, f = rhs / NZ, kz = rhs - f * NZ;
    return (long long)f * NG + (long long)nodes[beg + a] * NZ + kz;
  };
  // r -= A v
  auto residual = [&](const double* v) {
    for (int a = t; a < n; a += nt) {
      double s[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i) s[i] = r[a * NR + i];
      for (int e = A_ptr[beg + a]; e < A_ptr[beg + a + 1]; ++e) {
        const double w = -A_val[e];
        const int c = A_col[e];
#pragma unroll
        for (int i = 0; i < NR; ++i) s[i] = fma(w, v[c * NR + i], s[i]);
      }
#pragma unroll
      for (int i = 0; i < NR; ++i) r[a * NR + i] = s[i];
    }
  };
  auto norms = [&](double (&v)[NR]) {
#pragma unroll
    for (int i = 0; i < NR; ++i) v[i] = 0.0;
    for (int a = t; a < n; a += nt) {
      const double s = S[beg + a];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const double u = r[a * NR + i] * s;
        v[i] = fma(u, u, v[i]);
      }
    }
    block_sums<double, NR>(v, red64);
  };
  for (int a = t; a < n; a += nt) {
    const double s = S[beg + a];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const double b = rhs0 + i < nrhs ? q[at(a, i)] : 0.0;
      r[a * NR + i] = b;
      x[a * NR + i] = b * s * s;
    }
  }
  __syncthreads();
  double bb[NR], rr[NR];
  norms(bb);
  residual(x);
  __syncthreads();
  bool done = false;
  for (int outer = 0; outer <= kCgOuter; ++outer) {
    norms(rr);
    done = true;
    double up[NR], dn[NR];   // scale of the inner right-hand side, and back
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const bool ok = rr[i] <= 1e-30 * bb[i];
      done = done && ok;
      dn[i] = ok ? 0.0 : sqrt(rr[i]);
      up[i] = ok ? 0.0 : 1.0 / dn[i];
    }
    if (done || outer == kCgOuter) break;
    float rz[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) rz[i] = 0.f;
    for (int a = t; a < n; a += nt) {
      const double s = S[beg + a];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const float u = (float)(r[a * NR + i] * s * up[i]);
        z[a * NR + i] = p[a * NR + i] = u;
        y[a * NR + i] = 0.f;
        rz[i] = fmaf(u, u, rz[i]);
      }
    }
    block_sums<float, NR>(rz, red);
    for (int it = 0; it < kCgInner; ++it) {
      float pap[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i) pap[i] = 0.f;
      for (int a = t; a < n; a += nt) {
        float s[NR];
#pragma unroll
        for (int i = 0; i < NR; ++i) s[i] = 0.f;
        for (int e = A_ptr[beg + a]; e < A_ptr[beg + a + 1]; ++e) {
          const float w = A32[e];
          const int c = A_col[e];
#pragma unroll
          for (int i = 0; i < NR; ++i) s[i] = fmaf(w, p[c * NR + i], s[i]);
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          Ap[a * NR + i] = s[i];
          pap[i] = fmaf(p[a * NR + i], s[i], pap[i]);
        }
      }
      block_sums<float, NR>(pap, red);
      float rz2[NR], alpha[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        alpha[i] = pap[i] > 0.f ? rz[i] / pap[i] : 0.f;
        rz2[i] = 0.f;
      }
      for (int a = t; a < n; a += nt) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          y[a * NR + i] = fmaf(alpha[i], p[a * NR + i], y[a * NR + i]);
          const float u = fmaf(-alpha[i], Ap[a * NR + i], z[a * NR + i]);
          z[a * NR + i] = u;
          rz2[i] = fmaf(u, u, rz2[i]);
        }
      }
      block_sums<float, NR>(rz2, red);
      float worst = 0.f;
#pragma unroll
      for (int i = 0; i < NR; ++i) worst = fmaxf(worst, rz2[i]);
      if (!(worst > 1e-10f)) break;   // the inner right-hand side has norm 1 (or 0)
      for (int a = t; a < n; a += nt) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          const float beta = rz[i] > 0.f ? rz2[i] / rz[i] : 0.f;
          p[a * NR + i] = fmaf(beta, p[a * NR + i], z[a * NR + i]);
        }
      }
#pragma unroll
      for (int i = 0; i < NR; ++i) rz[i] = rz2[i];
      __syncthreads();
    }
    __syncthreads();
    for (int a = t; a < n; a += nt) {
      const double s = S[beg + a];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const double u = (double)y[a * NR + i] * (s * dn[i]);
        d[a * NR + i] = u;
        x[a * NR + i] += u;
      }
    }
    __syncthreads();
    residual(d);
    __syncthreads();
  }
  if (!done && t == 0) atomicOr(status, 2);
  for (int a = t; a < n; a += nt) {
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (rhs0 + i < nrhs) q[at(a, i)] = x[a * NR + i];
  }
}

// Build the coupled blocks of A_h = Q_h^T W_h Q_h on the host (once per mesh).
static int build_coupled_blocks(Mesh& m) {
  DeviceTables& D = *m.dev;
  if (D.tr_coupled) return SEM_OK;
  const int n1 = m.N + 1;
  const Basis1D& B = basis(m.N);
  const long long nh = m.NH;
  std::vector<int> parent(nh);
  std::iota(parent.begin(), parent.end(), 0);
  auto find = [&](int x) {
    while (parent[x] != x) x = parent[x] = parent[parent[x]];
    return x;
  };
  std::vector<char> coupled(nh, 0);
  const long long nhang = (long long)m.hang_h.size() / n1;
  for (long long k = 0; k < nhang; ++k) {
    int first = -1, cnt = 0;
    for (int q = 0; q < n1; ++q)
      if (m.hang_w[k * n1 + q] != 0.0) ++cnt;
    if (cnt < 2) continue;
    for (int q = 0; q < n1; ++q) {
      if (m.hang_w[k * n1 + q] == 0.0) continue;
      int h = m.hang_h[k * n1 + q];
      coupled[h] = 1;
      if (first < 0) first = h;
      else parent[find(h)] = find(first);
    }
  }
  // components in order of their smallest node
  std::vector<int> comp_of(nh, -1), order;
  std::vector<std::vector<int>> comps;
  for (long long h = 0; h < nh; ++h) {
    if (!coupled[h]) continue;
    int r = find((int)h);
    if (comp_of[r] < 0) {
      comp_of[r] = (int)comps.size();
      comps.emplace_back();
    }
    comps[comp_of[r]].push_back((int)h);
  }
  std::vector<int> local(nh, -1), cid(nh, -1);
  std::vector<int> comp_ptr(1, 0), nodes;
  for (size_t c = 0; c < comps.size(); ++c) {
    for (size_t a = 0; a < comps[c].size(); ++a) {
      local[comps[c][a]] = (int)a;
      cid[comps[c][a]] = (int)c;
      nodes.push_back(comps[c][a]);
    }
    comp_ptr.push_back((int)nodes.size());
  }
  // assemble rows of A_h for the coupled nodes
  std::vector<std::vector<std::pair<int, double>>> rows(nodes.size());
  auto row_of = [&](int h) { return comp_ptr[cid[h]] + local[h]; };
  auto add = [&](int h, int g, double v) {
    auto& R = rows[row_of(h)];
    int lc = local[g];
    for (auto& e : R)
      if (e.first == lc) { e.second += v; return; }
    R.push_back({lc, v});
  };
  for (long long c = 0; c < m.Ncol(); ++c) {
    const int l = m.leaves[c].l;
    for (int ab = 0; ab < m.Nq; ++ab) {
      const double W = B.w[ab % n1] * B.w[ab / n1] * m.hx(l) * m.hy(l) * 0.25;
      const int v = m.hmap[c * m.Nq + ab];
      if (v >= 0) {
        if (coupled[v]) add(v, v, W);
      } else {
        const int k = -1 - v;
        for (int q = 0; q < n1; ++q) {
          const double wq = m.hang_w[(size_t)k * n1 + q];
          if (wq == 0.0) continue;
          const int hq = m.hang_h[(size_t)k * n1 + q];
          if (!coupled[hq]) continue;  // delta rows only touch uncoupled nodes
          for (int r = 0; r < n1; ++r) {
            const double wr = m.hang_w[(size_t)k * n1 + r];
            if (wr == 0.0) continue;
            add(hq, m.hang_h[(size_t)k * n1 + r], wq * wr * W);
          }
        }
      }
    }
  }
  std::vector<int> A_ptr(1, 0), A_col;
  std::vector<double> A_val;
  for (auto& R : rows) {
    std::sort(R.begin(), R.end());
    for (auto& e : R) {
      A_col.push_back(e.first);
      A_val.push_back(e.second);
    }
    A_ptr.push_back((int)A_col.size());
  }
  // S = diag(A)^-1/2 and S A S in float32
  std::vector<double> sd(rows.size());
  for (size_t a = 0; a < rows.size(); ++a)
    for (auto& e : rows[a])
      if (comp_ptr[cid[nodes[a]]] + e.first == (int)a) sd[a] = 1.0 / std::sqrt(e.second);
  std::vector<float> A32(A_val.size());
  for (size_t a = 0; a < rows.size(); ++a)
    for (int e = A_ptr[a]; e < A_ptr[a + 1]; ++e)
      A32[e] = (float)(A_val[e] * sd[a] * sd[comp_ptr[cid[nodes[a]]] + A_col[e]]);
  std::vector<int> cpl(nh);
  for (long long h = 0; h < nh; ++h) cpl[h] = coupled[h];
  D.n_comp = (int)comps.size();
  D.max_comp = 0;
  for (auto& c : comps) D.max_comp = std::max<int>(D.max_comp, (int)c.size());
  auto up = [](auto*& dst, const auto& v) -> int {
    using T = typename std::decay<decltype(v[0])>::type;
    size_t n = v.empty() ? 1 : v.size();
    SEM_CUDA_TRY(cudaMalloc((void**)&dst, n * sizeof(T)));
    if (!v.empty()) SEM_CUDA_TRY(cudaMemcpy(dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
    return SEM_OK;
  };
  // tr_coupled last: it marks the tables as complete
  int rc;
  const std::vector<int> meta(nh, -1);
  if ((rc = up(D.tr_comp_ptr, comp_ptr)) || (rc = up(D.tr_nodes, nodes)) || (rc = up(D.tr_A_ptr, A_ptr)) ||
      (rc = up(D.tr_A_col, A_col)) || (rc = up(D.tr_A_val, A_val)) || (rc = up(D.tr_A32, A32)) ||
      (rc = up(D.tr_S, sd)) || (rc = up(D.tr_meta, meta)) || (rc = up(D.tr_coupled, cpl)))
    return rc;
  return SEM_OK;
}

template <int N>
static void launch_local(const TrArgs& A, int ncol, cudaStream_t st) {
  // as few passes of at most kTrThreads threads over a column's (field, level)
  // pairs as fit, of equal size
  const int items = kFields * A.NZ, passes = (items + kTrThreads - 1) / kTrThreads;
  const int nt = ((items + passes - 1) / passes + 31) / 32 * 32;
  transfer_local<N><<<ncol, nt, 0, st>>>(A);
}

template <int NR>
static int launch_cg(Mesh& m, double* q, cudaStream_t st) {
  DeviceTables& D = *m.dev;
  const size_t smem = (size_t)32 * NR * D.max_comp;
  SEM_CUDA_TRY(cudaFuncSetAttribute(transfer_cg<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const dim3 grid(D.n_comp, (kFields * m.NZ + NR - 1) / NR);
  transfer_cg<NR><<<grid, kCgThreads, smem, st>>>(D.tr_comp_ptr, D.tr_nodes, D.tr_A_ptr, D.tr_A_col, D.tr_A_val,
                                                  D.tr_A32, D.tr_S, m.NG, m.NZ, q, D.status);
  return SEM_OK;
}

int launch_transfer(Mesh& o, Mesh& m, const double* qold, double* qnew, cudaStream_t st) {
  int rc = upload_transfer_constants();
  if (rc) return rc;
  if ((rc = build_coupled_blocks(m))) return rc;
  DeviceTables& D = *m.dev;
  DeviceTables& Do = *o.dev;
  if (m.NG >= (1ll << 31)) return fail(SEM_ERR_ARG, "mesh too large for 32-bit node indexing");
  if (o.NZ != m.NZ || o.N != m.N) return fail(SEM_ERR_ARG, "meshes differ in N or layering");
  TrArgs A;
  A.qold = qold;
  A.old_hmap = Do.hmap;
  A.old_hang_h = Do.hang_h;
  A.old_hang_w = Do.hang_w;
  A.old_NG = o.NG;
  A.org = D.org;
  A.new_level = D.col_level;
  A.out = (double*)D.scratch;
  A.N = m.N;
  A.NZ = m.NZ;
  A.hxy = m.hx(0) * m.hy(0) * 0.25;
  const int nc = (int)m.Ncol();
  switch (m.N) {
    case 2: launch_local<2>(A, nc, st); break;
    case 3: launch_local<3>(A, nc, st); break;
    case 4: launch_local<4>(A, nc, st); break;
    case 5: launch_local<5>(A, nc, st); break;
    case 6: launch_local<6>(A, nc, st); break;
    default: return fail(SEM_ERR_UNSUPPORTED, "order N not compiled");
  }
  SEM_CUDA_TRY(cudaGetLastError());
  transfer_meta<<<(unsigned)((m.NH + 255) / 256), 256, 0, st>>>(
      A, reinterpret_cast<const int4*>(D.qt_rec_unit), D.tr_coupled, (int)m.NH, D.tr_meta);
  long long blocks = std::min<long long>((m.NG + 255) / 256, 152 * 64);
  transfer_gather<<<(int)blocks, 256, 0, st>>>(A, D.tr_meta, D.qt_ptr, D.qt_src, D.qt_w, D.Minv_h, D.tr_coupled,
                                              (unsigned)m.NG, qnew);
  SEM_CUDA_TRY(cudaGetLastError());
  if (D.n_comp > 0) {
    // four right-hand sides per CTA where their vectors fit its shared memory
    // and the blocks still give every SM one
    if ((size_t)40 * D.max_comp > 200 * 1024) return fail(SEM_ERR_UNSUPPORTED, "coupled 2:1 block too large for one CTA");
    int dev = 0, nsm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const bool four = (size_t)128 * D.max_comp <= 200 * 1024 && (long long)D.n_comp * kFields * m.NZ >= 4LL * nsm;
    if ((rc = four ? launch_cg<4>(m, qnew, st) : launch_cg<1>(m, qnew, st))) return rc;
    SEM_CUDA_TRY(cudaGetLastError());
  }
  return SEM_OK;
}

}  // namespace sem
