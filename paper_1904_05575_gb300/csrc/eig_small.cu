// Lowest eigenpairs of the small Hermitian matrices of the Davidson projection.
//
// The projected problem of an iteration is m x m with m up to a few hundred, of
// which the k = 2 nev lowest pairs are used.  A library eigensolve spends its
// time between launches (5.3 ms at m = 32 to 192, 128 of 170 ms of a solve of
// N = 2,560, nev = 8).  Here:
//   1. k_hetrd      Householder reduction to a real tridiagonal T (the
//                   algorithm of Golub and Van Loan, Matrix Computations, 8.3.1,
//                   complex Hermitian form), one cooperative launch: every block
//                   keeps a cyclic set of rows in shared memory, two grid
//                   barriers per column
//   2. host         the k lowest eigenvalues of T by bisection on Sturm counts
//                   (all k in lock step) and their vectors by inverse iteration,
//                   close ones orthogonalised; O(k m) each
//   3. k_back       the reflectors applied to the k vectors, one block per vector
// The result is checked (residual and orthogonality in T); the caller falls
// back on the library where it fails or m is too large.  Bound by the latency
// of the reduction's chain per column (two grid exchanges, a square root, two
// divisions and three block sums, about 7 us): the projected problems of that
// solve take 2.6 instead of 6.4 ms per iteration, the solve 95 to 97 instead of
// 166 (72.5 with the tall-skinny products of davidson.cu).
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "bse_internal.h"

namespace bse {
namespace {

constexpr int kTrdThreads = 256, kTrdBlocks = 64, kTrdMaxM = 512;
constexpr int kTrdMaxK = 64;   // (orthogonalising k close vectors costs k^2 m on the host)

struct TrdArgs {
  int m, lds;
  const double2* S;     // column-major, the lower triangle is read
  double2 *V, *tau;     // reflector j: V[j m + i], i > j (V[j m + j + 1] = 1)
  double *d, *e;
  double2 *col, *p;     // [2][m] exchange buffers
  int *arrived, *gave_up;
  long long wait;       // clock budget of a grid barrier
};

__device__ __forceinline__ bool trd_barrier(const TrdArgs& a, int target, int* ok_s) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.arrived) : "memory");
    const long long t0 = clock64();
    for (int spin = 1;; ++spin) {
      int seen;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(a.arrived) : "memory");
      if (seen >= target) break;
      int stop = clock64() - t0 > a.wait;
      if (!stop && (spin & 63) == 0)
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(stop) : "l"(a.gave_up) : "memory");
      if (stop) {
        atomicExch(a.gave_up, 1);
        ok = 0;
        break;
      }
    }
    *ok_s = ok;
  }
  __syncthreads();
  return *ok_s != 0;
}

__device__ __forceinline__ double warp_add(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// sum of (x, y) over the block, in every thread
template <int TH>
__device__ __forceinline__ double2 block_add(double2 v, double2* red) {
  v = make_double2(warp_add(v.x), warp_add(v.y));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double2 t = red[0];
#pragma unroll
  for (int w = 1; w < TH / 32; ++w) {
    t.x += red[w].x;
    t.y += red[w].y;
  }
  return t;
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

__global__ void __launch_bounds__(kTrdThreads, 1) k_hetrd(TrdArgs a) {
  extern __shared__ double2 trd_smem[];
  __shared__ double2 red[kTrdThreads / 32], tau_s, scale_s;
  __shared__ int ok_s;
  const int m = a.m, nb = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nrows = (m - (int)blockIdx.x + nb - 1) / nb;   // rows blockIdx.x + r nb
  double2* v = trd_smem;           // [m]
  double2* w = v + m;              // [m]
  double2* A = w + m;              // [nrows][m]
  for (int t = tid; t < nrows * m; t += kTrdThreads) {
    const int r = t / m, l = t - r * m, i = blockIdx.x + r * nb;
    double2 x = l <= i ? a.S[i + (int64_t)l * a.lds] : a.S[l + (int64_t)i * a.lds];
    if (l > i) x.y = -x.y;
    if (l == i) x.y = 0.0;
    A[t] = x;
  }
  __syncthreads();
  for (int r = tid; r < nrows; r += kTrdThreads) {
    const int i = blockIdx.x + r * nb;
    __stcg(a.col + i, A[r * m]);
    if (i == 0) a.d[0] = A[r * m].x;
  }
  int arrived = 0;
#pragma unroll 1
  for (int j = 0; j + 1 < m; ++j) {
    double2 *col = a.col + (int64_t)(j & 1) * m, *next = a.col + (int64_t)((j + 1) & 1) * m;
    double2* p = a.p + (int64_t)(j & 1) * m;
    if (!trd_barrier(a, arrived += nb, &ok_s)) return;
    // the reflector of column j (every block: the same bits); a column whose
    // squares fall out of the range of FP64 (below 1e-154) gives an infinite scale,
    // T is not finite and the library serves the matrix
    double s2 = 0.0;
    for (int i = j + 1 + tid; i < m; i += kTrdThreads) {
      const double2 x = __ldcg(col + i);
      v[i] = x;
      if (i > j + 1) s2 = fma(x.x, x.x, fma(x.y, x.y, s2));
    }
    s2 = block_add<kTrdThreads>(make_double2(s2, 0.0), red).x;   // (syncs: v is complete)
    if (tid == 0) {
      const double2 al = v[j + 1];
      double beta = al.x;
      double2 tau = make_double2(0.0, 0.0), sc = tau;
      if (s2 > 0.0 || al.y != 0.0) {
        beta = -copysign(sqrt(fma(al.x, al.x, fma(al.y, al.y, s2))), al.x);
        const double ib = 1.0 / beta;
        tau = make_double2((beta - al.x) * ib, -al.y * ib);
        const double2 q = make_double2(al.x - beta, al.y);
        const double iq = 1.0 / fma(q.x, q.x, q.y * q.y);
        sc = make_double2(q.x * iq, -q.y * iq);
      }
      tau_s = tau;
      scale_s = sc;
      if (blockIdx.x == 0) {
        a.e[j] = beta;
        a.tau[j] = tau;
      }
    }
    __syncthreads();
    const double2 tau = tau_s, sc = scale_s;
    for (int i = j + 1 + tid; i < m; i += kTrdThreads) {
      const double2 x = i == j + 1 ? make_double2(1.0, 0.0) : cmul(v[i], sc);
      v[i] = x;
      if (blockIdx.x == 0) a.V[(int64_t)j * m + i] = x;
    }
    __syncthreads();
    // p = tau A v on the own rows, one warp per row
#pragma unroll 1
    for (int r = warp; r < nrows; r += kTrdThreads / 32) {
      const int i = blockIdx.x + r * nb;
      if (i <= j) continue;
      double2 t = make_double2(0.0, 0.0);
      for (int l = j + 1 + lane; l < m; l += 32) {
        const double2 x = A[r * m + l], y = v[l];
        t.x = fma(x.x, y.x, fma(-x.y, y.y, t.x));
        t.y = fma(x.x, y.y, fma(x.y, y.x, t.y));
      }
      t = make_double2(warp_add(t.x), warp_add(t.y));
      if (lane == 0) __stcg(p + i, cmul(tau, t));
    }
    if (!trd_barrier(a, arrived += nb, &ok_s)) return;
    // w = p - (tau / 2) (p^H v) v
    double2 dot = make_double2(0.0, 0.0);
    for (int i = j + 1 + tid; i < m; i += kTrdThreads) {
      const double2 x = __ldcg(p + i), y = v[i];
      w[i] = x;
      dot.x = fma(x.x, y.x, fma(x.y, y.y, dot.x));
      dot.y = fma(x.x, y.y, fma(-x.y, y.x, dot.y));
    }
    dot = block_add<kTrdThreads>(dot, red);
    double2 al = cmul(tau, dot);
    al = make_double2(-0.5 * al.x, -0.5 * al.y);
    for (int i = j + 1 + tid; i < m; i += kTrdThreads) {
      const double2 y = cmul(al, v[i]);
      w[i] = make_double2(w[i].x + y.x, w[i].y + y.y);
    }
    __syncthreads();
    // A -= v w^H + w v^H on the own rows
    const int nl = m - j - 1;
#pragma unroll 1
    for (int t = tid; t < nrows * nl; t += kTrdThreads) {
      const int r = t / nl, l = j + 1 + t - r * nl, i = blockIdx.x + r * nb;
      if (i <= j) continue;
      const double2 vi = v[i], wi = w[i], vl = v[l], wl = w[l];
      double2 x = A[r * m + l];
      x.x -= fma(vi.x, wl.x, fma(vi.y, wl.y, fma(wi.x, vl.x, wi.y * vl.y)));
      x.y -= fma(vi.y, wl.x, fma(-vi.x, wl.y, fma(wi.y, vl.x, -wi.x * vl.y)));
      A[r * m + l] = x;
    }
    __syncthreads();
    for (int r = tid; r < nrows; r += kTrdThreads) {
      const int i = blockIdx.x + r * nb;
      if (i > j + 1) __stcg(next + i, A[r * m + j + 1]);
      if (i == j + 1) a.d[i] = A[r * m + i].x;
    }
  }
}

// x = H_0 ... H_{m-2} z for one eigenvector of T per block
constexpr int kBackThreads = 128;
__global__ void __launch_bounds__(kBackThreads) k_back(int m, const double2* V, const double2* tau,
                                                       const double* Z, double2* X, int ldx) {
  __shared__ double2 x[kTrdMaxM], red[kBackThreads / 32];
  const int tid = threadIdx.x;
  for (int i = tid; i < m; i += kBackThreads)
    x[i] = make_double2(Z[(int64_t)blockIdx.x * m + i], 0.0);
  __syncthreads();
#pragma unroll 1
  for (int j = m - 2; j >= 0; --j) {
    double2 v[kTrdMaxM / kBackThreads], dot = make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < kTrdMaxM / kBackThreads; ++q) {
      const int i = j + 1 + tid + q * kBackThreads;
      v[q] = i < m ? V[(int64_t)j * m + i] : make_double2(0.0, 0.0);
      if (i < m) {
        dot.x = fma(v[q].x, x[i].x, fma(v[q].y, x[i].y, dot.x));
        dot.y = fma(v[q].x, x[i].y, fma(-v[q].y, x[i].x, dot.y));
      }
    }
    dot = cmul(tau[j], block_add<kBackThreads>(dot, red));
#pragma unroll
    for (int q = 0; q < kTrdMaxM / kBackThreads; ++q) {
      const int i = j + 1 + tid + q * kBackThreads;
      if (i < m) {
        const double2 t = cmul(dot, v[q]);
        x[i] = make_double2(x[i].x - t.x, x[i].y - t.y);
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < m; i += kBackThreads) X[(int64_t)blockIdx.x * ldx + i] = x[i];
}

}  // namespace

// The k lowest eigenpairs of the real symmetric tridiagonal (d, e): bisection on
// Sturm counts, inverse iteration.  False if a residual or an overlap is larger
// than a library eigensolve leaves them: vectors of eigenvalues kTriCluster |T|
// apart are not orthogonalised and overlap by rounding / kTriCluster, residuals are
// one or two units of rounding (up to 23 within groups of equal eigenvalues whose
// shifts had to be moved apart; hundreds where such a shift met another eigenvalue,
// which the library gets right).
constexpr double kTriCluster = 1e-3, kTriOverlap = DBL_EPSILON / kTriCluster,
                 kTriResidual = 32.0 * DBL_EPSILON;
bool tridiagonal_lowest(int m, const double* d, const double* e, int k, double* lam, double* Z) {
  double lo = DBL_MAX, hi = -DBL_MAX, e2max = 0.0;
  for (int i = 0; i < m; ++i) {
    const double r = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i + 1 < m ? std::fabs(e[i]) : 0.0);
    if (!std::isfinite(d[i]) || !std::isfinite(r)) return false;
    lo = std::min(lo, d[i] - r);
    hi = std::max(hi, d[i] + r);
    if (i + 1 < m) e2max = std::max(e2max, e[i] * e[i]);
  }
  const double norm = std::max(std::fabs(lo), std::fabs(hi));
  if (!(norm > 0.0) || norm > 1e150 || norm < 1e-150) return false;
  const double pivmin = DBL_MIN * std::max(1.0, e2max) * 4.0;
  lo -= 4.0 * DBL_EPSILON * norm;
  hi += 4.0 * DBL_EPSILON * norm;
  std::vector<double> l(k, lo), h(k, hi), x(k), q(k);
  std::vector<int> cnt(k);
  for (int it = 0; it < 64; ++it) {
    double widest = 0.0;
    for (int c = 0; c < k; ++c) {
      x[c] = 0.5 * (l[c] + h[c]);
      q[c] = 1.0;
      cnt[c] = 0;
      widest = std::max(widest, h[c] - l[c]);
    }
    if (widest <= DBL_EPSILON * norm) break;
    for (int i = 0; i < m; ++i) {
      const double e2 = i > 0 ? e[i - 1] * e[i - 1] : 0.0, di = d[i];
      for (int c = 0; c < k; ++c) {
        double t = di - x[c] - e2 / q[c];
        t = std::fabs(t) < pivmin ? -pivmin : t;
        q[c] = t;
        cnt[c] += t < 0.0;
      }
    }
    for (int c = 0; c < k; ++c) (cnt[c] > c ? h[c] : l[c]) = x[c];
  }
  for (int c = 0; c < k; ++c) lam[c] = 0.5 * (l[c] + h[c]);
  // inverse iteration: T - lam by Gaussian elimination with partial pivoting
  std::vector<double> u0(m), u1(m), u2(m), mul(m), b(m);
  std::vector<char> swapped(m);
  const double tiny = DBL_EPSILON * norm;
  double shift_prev = 0.0;
  uint64_t seed = 88172645463325252ull;
  int cluster = 0;   // first vector of the current group of close eigenvalues
  for (int c = 0; c < k; ++c) {
    if (c > 0 && lam[c] - lam[c - 1] > kTriCluster * norm) cluster = c;
    double shift = lam[c];   // (equal eigenvalues: shifts a few ulp apart)
    if (c > cluster && shift - shift_prev < 10.0 * tiny) shift = shift_prev + 10.0 * tiny;
    shift_prev = shift;
    double a0 = d[0] - shift, a1 = m > 1 ? e[0] : 0.0, a2 = 0.0;
    for (int i = 0; i + 1 < m; ++i) {
      const double s = e[i], n0 = d[i + 1] - shift, n1 = i + 2 < m ? e[i + 1] : 0.0;
      if (std::fabs(s) > std::fabs(a0)) {
        swapped[i] = 1;
        mul[i] = a0 / s;
        u0[i] = s; u1[i] = n0; u2[i] = n1;
        a0 = a1 - mul[i] * n0;
        a1 = a2 - mul[i] * n1;
      } else {
        swapped[i] = 0;
        if (a0 == 0.0) a0 = tiny;
        mul[i] = s / a0;
        u0[i] = a0; u1[i] = a1; u2[i] = a2;
        a0 = n0 - mul[i] * a1;
        a1 = n1 - mul[i] * a2;
      }
      a2 = 0.0;
    }
    u0[m - 1] = std::fabs(a0) < tiny ? (a0 < 0.0 ? -tiny : tiny) : a0;
    u1[m - 1] = u2[m - 1] = 0.0;
    double* z = Z + (size_t)c * m;
    for (int i = 0; i < m; ++i) {   // xorshift64 (Marsaglia 2003): a start vector with no pattern
      seed ^= seed << 13;
      seed ^= seed >> 7;
      seed ^= seed << 17;
      b[i] = (double)(int64_t)seed * 0x1p-63;
    }
    for (int it = 0; it < 4; ++it) {
      if (it > 0)   // (the first solve takes the start vector as already eliminated)
        for (int i = 0; i + 1 < m; ++i) {
          if (swapped[i]) std::swap(b[i], b[i + 1]);
          b[i + 1] -= mul[i] * b[i];
        }
      for (int i = m - 1; i >= 0; --i) {
        double t = b[i];
        if (i + 1 < m) t -= u1[i] * b[i + 1];
        if (i + 2 < m) t -= u2[i] * b[i + 2];
        b[i] = t / u0[i];
      }
      double big = 0.0;
      for (int i = 0; i < m; ++i) big = std::max(big, std::fabs(b[i]));
      if (!(big > 0.0) || !std::isfinite(big)) return false;
      for (int i = 0; i < m; ++i) b[i] /= big;
      for (int pass = 0; pass < (it == 3 ? 2 : 1); ++pass)
        for (int g = cluster; g < c; ++g) {
          const double* y = Z + (size_t)g * m;
          double t = 0.0;
          for (int i = 0; i < m; ++i) t += y[i] * b[i];
          for (int i = 0; i < m; ++i) b[i] -= t * y[i];
        }
      double n2 = 0.0;
      for (int i = 0; i < m; ++i) n2 += b[i] * b[i];
      if (!(n2 > 0.0)) return false;
      const double f = 1.0 / std::sqrt(n2);
      for (int i = 0; i < m; ++i) b[i] *= f;
    }
    // residual of the pair, and overlaps with every vector before it
    double res = 0.0;
    for (int i = 0; i < m; ++i) {
      double t = (d[i] - lam[c]) * b[i];
      if (i > 0) t += e[i - 1] * b[i - 1];
      if (i + 1 < m) t += e[i] * b[i + 1];
      res = std::max(res, std::fabs(t));
      z[i] = b[i];
    }
    if (!(res < kTriResidual * norm)) return false;
    for (int g = 0; g < c; ++g) {
      const double* y = Z + (size_t)g * m;
      double t = 0.0;
      for (int i = 0; i < m; ++i) t += y[i] * z[i];
      if (!(std::fabs(t) < kTriOverlap)) return false;
    }
  }
  return true;
}

size_t eig_lowest_workspace(int m) {
  const size_t mm = (size_t)std::min(m, kTrdMaxM);
  // V, tau, col, p, d, e, Z (at most m vectors), control words
  return mm * mm * 16 + mm * 16 * 5 + mm * 8 * 2 + mm * mm * 8 + 64;
}

// The k lowest eigenpairs of the Hermitian m x m S (device, column-major, lower
// triangle): eigenvalues to the host array lam, vectors over the first k columns
// of S.  False (S untouched): not served, take the library.  Syncs.
bool eig_lowest(int m, double2* S, int lds, int k, double* lam, void* work, cudaStream_t s) {
  if (m < 3 || m > kTrdMaxM || k < 1 || k > std::min(m, kTrdMaxK)) return false;
  char* w = static_cast<char*>(work);
  auto take = [&](size_t bytes) {
    char* p = w;
    w += bytes;
    return p;
  };
  double2* V = reinterpret_cast<double2*>(take((size_t)m * m * 16));
  double2* tau = reinterpret_cast<double2*>(take((size_t)m * 16));
  double2* col = reinterpret_cast<double2*>(take((size_t)m * 32));
  double2* p = reinterpret_cast<double2*>(take((size_t)m * 32));
  double* de = reinterpret_cast<double*>(take((size_t)m * 16));
  double* Z = reinterpret_cast<double*>(take((size_t)m * k * 8));
  int* ctl = reinterpret_cast<int*>((reinterpret_cast<uintptr_t>(w) + 15) & ~static_cast<uintptr_t>(15));
  BSE_CUDA(cudaMemsetAsync(ctl, 0, 2 * sizeof(int), s));
  const int blocks = std::min(kTrdBlocks, m), rows = (m + blocks - 1) / blocks;
  const size_t smem = ((size_t)rows + 2) * m * sizeof(double2);
  BSE_CUDA(cudaFuncSetAttribute(k_hetrd, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
  TrdArgs a{m, lds, S, V, tau, de, de + m, col, p, ctl, ctl + 1, call_wait_cycles()};
  void* args[] = {&a};
  BSE_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_hetrd), dim3(blocks),
                                       dim3(kTrdThreads), args, smem, s));
  note_launches(1);
  std::vector<double> h(2 * (size_t)m), z((size_t)m * k);
  int gave_up = 0;
  BSE_CUDA(cudaMemcpyAsync(h.data(), de, (size_t)m * 16, cudaMemcpyDeviceToHost, s));
  BSE_CUDA(cudaMemcpyAsync(&gave_up, ctl + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
  BSE_CUDA(cudaStreamSynchronize(s));
  if (gave_up) throw Error(BSE_ERR_TIMEOUT, "projected eigensolve: a bounded grid-barrier wait expired");
  if (!tridiagonal_lowest(m, h.data(), h.data() + m, k, lam, z.data())) return false;
  BSE_CUDA(cudaMemcpyAsync(Z, z.data(), (size_t)m * k * 8, cudaMemcpyHostToDevice, s));
  k_back<<<k, kBackThreads, 0, s>>>(m, V, tau, Z, S, lds);
  BSE_CUDA(cudaGetLastError());
  note_launches(1);
  BSE_CUDA(cudaStreamSynchronize(s));   // z (host) has been read
  return true;
}

}  // namespace bse
