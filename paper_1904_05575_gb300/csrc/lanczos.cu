// eps_M on a frequency grid without the eigensolve: a Lanczos recursion on
// the product form and a continued fraction.
//
// The spectrum of Eqs. chir / osci / epsmtensor sums over the excitons,
//   eps(w) = 1 - c_Q Ha sum_l |t_l|^2 [1/(w - E_l + i d) - 1/(w + E_l + i d)],
// with |t_l|^2 = |u_l|^2 / (E_l V_c), u = Z^T L^T rho, S Z = Z E^2 and
// S = L^H (A+B) L, A-B = L L^H (Eq. auxham).  Since 1/(z - E) - 1/(z + E) =
// 2E/(z^2 - E^2), the sum is (2 / V_c) w^H (z^2 - S)^-1 w with w = L^H conj(rho),
// and with K = (A-B)(A+B) = L S L^-1 it becomes
//   Q(z^2) = conj(rho)^H (z^2 - K)^-1 (A-B) conj(rho),   z = w + i d.
// K is self-adjoint in the inner product <a, b> = a^H (A-B)^-1 b, and
// Q = <v, (z^2 - K)^-1 v> for v = (A-B) conj(rho), <v, v> = conj(rho)^H (A-B)
// conj(rho).  Lanczos in that inner product keeps, beside each vector v_j,
// y_j = (A-B)^-1 v_j, so that no inverse or factorisation is needed:
//   u = (A+B) v_j,  alpha_j = v_j^H u,
//   y = u - alpha_j y_j - beta_{j-1} y_{j-1},  x = (A-B) y,  beta_j^2 = y^H x,
//   v_{j+1} = x / beta_j,  y_{j+1} = y / beta_j,
// two Hermitian matrix-vector products per step.  Q is then <v, v> over the
// continued fraction z^2 - alpha_0 - beta_0^2 / (z^2 - alpha_1 - ...) of the
// tridiagonal matrix (the recursion-method form of a resolvent element).
// The recursion stops when eps on the grid changes by less than tol (relative
// to its largest value) between checks.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <vector>

#include "bits.cuh"
#include "bse_internal.h"
#include "lanczos.h"

namespace bse {
namespace {

// ---------------------------------------------------------------------------
// FP64 products: many steps in one cooperative launch
// ---------------------------------------------------------------------------
// One block per SM owns a contiguous range of rows; a step is two row-range
// products with a grid-wide exchange after each, nothing else crosses blocks:
//   u = (A+B) x             x = beta_{j-1} v_j, left unnormalised (f = 1/beta_{j-1});
//                           partial sums of x^H u = alpha_j / f^2
//   x = (A-B) y             y = f u - alpha f y_j' - beta f' y_{j-1}' (y' unnormalised)
//                           formed by every block for all columns while it
//                           stages them in shared memory (6 FMAs per column,
//                           against 4 per column and owned row); partial sums
//                           of beta_j^2 = y^H x
// Every block adds the per-block partials in one fixed order, so all blocks
// hold the same scalars and a run repeats bit for bit.
//
// Bound by the FP64 pipe (1.8 FMAs per clock and SM: 15 us of products per
// step at N = 1,024) and around them by latencies: a dependent FP64 add takes
// 67 clocks, one behind a shuffle 104, a division 435, an exchange about 2,000.
// So the reciprocal root runs in a warp of its own during the next product,
// a row is summed by one warp, and both halves of a step share one body of
// code: written out per half it grew to 82 KB, and fetching it cost as much
// as the products.  Measured per step, checks included: N = 1,024 32 us (51
// as seven launches per step: column-chunk products, partial sums,
// recurrence, scaling), N = 256 15 us, N = 2,000 82 us.
constexpr int kLzThreads = 512;          // 15 warps of products, 1 of scalars
constexpr int kLzProd = kLzThreads - 32;
constexpr int kLzCols = 1024;            // columns staged in shared memory at a time
constexpr int kLzMaxBlocks = 160;

struct LzArgs {
  int n;
  const double2 *C, *D;     // A+B, A-B (column-major, ld)
  int64_t ld;
  double2 *x, *u;           // beta v_j, product u (finite before the first launch)
  double2* y[3];            // unnormalised y_j, ring: step j reads j % 3, (j + 2) % 3, writes (j + 1) % 3
  double* coef;             // alpha_j at 2j, beta_j^2 at 2j + 1
  int nv2_slot;             // <v_0, v_0> of the start vector
  double* part;             // [2][kLzMaxBlocks] per-block partial sums (of even and odd exchanges)
  int* arrived;             // arrivals at the exchanges, zeroed before the launch
  int* gave_up;             // a bounded wait expired
  long long wait;           // clock budget of one exchange
  int rows;                 // rows per block
  int j0, steps;            // first step, number of steps; steps = 0: x = (A-B) y[0] and <v, v> only
};

struct LzSmem {
  double2 xs[kLzCols];
  double2 red[kLzProd];
  double sums[kLzThreads / 32];
  double fu, ca, cb;        // y = fu u - ca y_j' - cb y_{j-1}'
  int ok;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __noinline__ double lz_inv_root(double v) { return v > 0.0 ? rsqrt(v) : 0.0; }

// The scalar warp's half of an exchange: publishes the block's partial sum
// (the warps' sums in sm.sums), waits until every block has (bounded; false:
// gave up) and leaves the sum of all partials in *total (same bits in every
// block).  What the blocks wrote before is visible after it.
__device__ __forceinline__ bool lz_exchange(const LzArgs& a, LzSmem& sm, int phase, double* total) {
  const int lane = threadIdx.x & 31, nb = gridDim.x;
  double t = warp_sum(lane < kLzProd / 32 ? sm.sums[lane] : 0.0);
  double* part = a.part + (phase & 1) * kLzMaxBlocks;
  int ok = 1;
  if (lane == 0) {
    __stcg(part + blockIdx.x, t);
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.arrived) : "memory");
    const int target = (phase + 1) * nb;
    const long long t0 = clock64();
#pragma unroll 1
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
  }
  __syncwarp();   // lane 0's acquire orders the other lanes' reads below (a shuffle orders no memory)
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) return false;
  double p[kLzMaxBlocks / 32];
#pragma unroll
  for (int q = 0; q < kLzMaxBlocks / 32; ++q)
    p[q] = lane + 32 * q < nb ? __ldcg(part + lane + 32 * q) : 0.0;
  t = p[0];
#pragma unroll
  for (int q = 1; q < kLzMaxBlocks / 32; ++q) t += p[q];
  *total = warp_sum(t);
  return true;
}

__global__ void __launch_bounds__(kLzThreads, 1) k_lanczos_steps(LzArgs a) {
  __shared__ LzSmem sm;
  const int n = a.n, r0 = blockIdx.x * a.rows, rn = min(a.rows, n - r0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool scalar = tid >= kLzProd;
  const bool start = a.steps == 0;   // only x = (A-B) y_0: the second half with y = y[0]
  // (scalar warp) beta^2 before step j: coef[2j - 1], or <v_0, v_0> before the first
  double b2 = 0.0, f = 0.0, f_prev = 0.0;
  if (scalar && !start) {
    b2 = a.coef[a.j0 > 0 ? 2 * a.j0 - 1 : a.nv2_slot];
    if (a.j0 > 0) f_prev = lz_inv_root(a.coef[a.j0 > 1 ? 2 * a.j0 - 3 : a.nv2_slot]);
  }
  if (tid == 0) {
    sm.fu = sm.cb = 0.0;
    sm.ca = -1.0;
  }
  const int last = start ? 2 : 2 * a.steps;
#pragma unroll 1
  for (int half = start ? 1 : 0, phase = 0; half < last; ++half, ++phase) {
    const int j = a.j0 + (half >> 1);
    const bool second = half & 1;   // x = (A-B) y, else u = (A+B) x
    const double2* M = second ? a.D : a.C;
    const double2* y1 = j % 3 == 0 ? a.y[0] : j % 3 == 1 ? a.y[1] : a.y[2];
    const double2* y0 = j % 3 == 0 ? a.y[2] : j % 3 == 1 ? a.y[0] : a.y[1];
    double2* y2 = j % 3 == 0 ? a.y[1] : j % 3 == 1 ? a.y[2] : a.y[0];
    __syncthreads();   // sm.fu, ca, cb of the exchange before; sm.sums read
    const double fu = sm.fu, ca = sm.ca, cb = sm.cb;
    auto operand = [&](int c) {
      if (!second) return __ldcg(a.x + c);
      const double2 u = __ldcg(a.u + c), p = __ldcg(y1 + c), q = __ldcg(y0 + c);
      return make_double2(fma(-cb, q.x, fma(-ca, p.x, fu * u.x)),
                          fma(-cb, q.y, fma(-ca, p.y, fu * u.y)));
    };
    double d = 0.0;
#pragma unroll 1
    for (int rs = 0; rs < rn; rs += kLzProd) {
      // rb rows at a time; product thread t holds row t % rb of the column
      // group t / rb (lanes on consecutive rows of a column)
      const int rb = min(kLzProd, rn - rs);
      const int ngroups = kLzProd / rb, r = tid % rb, g = tid / rb;
      double ax = 0.0, ay = 0.0;
#pragma unroll 1
      for (int c0 = 0; c0 < n; c0 += kLzCols) {
        const int cn = min(kLzCols, n - c0);
        __syncthreads();
#pragma unroll 1
        for (int c = tid; c < cn; c += kLzThreads) sm.xs[c] = operand(c0 + c);
        __syncthreads();
        if (scalar) {
          if (c0 == 0 && rs == 0 && !second) {   // f = 1 / beta_{j-1} during the first product
            f = lz_inv_root(b2);
            if (lane == 0) {
              sm.fu = f;
              sm.cb = b2 * f * f_prev;   // beta_{j-1} / beta_{j-2} (0 at the first step)
            }
          }
        } else if (g < ngroups) {
          // the next four columns' loads are issued before this four's products
          const double2 none = make_double2(0.0, 0.0);
          const int64_t step = (int64_t)ngroups * a.ld;
          const double2* pc = M + (int64_t)(c0 + g) * a.ld + r0 + rs + r;
          double2 m[4], nx[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) m[q] = g + q * ngroups < cn ? __ldg(pc + q * step) : none;
#pragma unroll 1
          for (int c = g; c < cn; c += 4 * ngroups) {
            pc += 4 * step;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              nx[q] = c + (4 + q) * ngroups < cn ? __ldg(pc + q * step) : none;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (c + q * ngroups < cn) {
                const double2 xv = sm.xs[c + q * ngroups];
                ax = fma(m[q].x, xv.x, fma(-m[q].y, xv.y, ax));
                ay = fma(m[q].x, xv.y, fma(m[q].y, xv.x, ay));
              }
              m[q] = nx[q];
            }
          }
        }
      }
      if (!scalar) sm.red[tid] = make_double2(ax, ay);
      __syncthreads();
      if (!scalar) {
#pragma unroll 1
        for (int row = warp; row < rb; row += kLzProd / 32) {   // one warp adds a row's groups
          double2 s = make_double2(0.0, 0.0);
#pragma unroll 1
          for (int q = lane; q < ngroups; q += 32) {
            const double2 v = sm.red[q * rb + row];
            s.x += v.x;
            s.y += v.y;
          }
          s = make_double2(warp_sum(s.x), warp_sum(s.y));
          if (lane == 0) {
            const int i = r0 + rs + row;
            const double2 v = operand(i);
            __stcg((second ? a.x : a.u) + i, s);
            if (second) __stcg(y2 + i, v);
            d += v.x * s.x + v.y * s.y;
          }
        }
      }
    }
    if (lane == 0) sm.sums[warp] = d;
    __syncthreads();
    if (scalar) {
      double t = 0.0;
      const bool ok = lz_exchange(a, sm, phase, &t);
      if (second) {
        b2 = t;
        f_prev = f;
      } else {
        t *= f * f;   // alpha_j
      }
      if (lane == 0) {
        sm.ok = ok;
        if (!second) sm.ca = t * f;
        if (ok && blockIdx.x == 0) a.coef[start ? a.nv2_slot : 2 * j + (second ? 1 : 0)] = t;
      }
    }
    __syncthreads();
    if (!sm.ok) return;
  }
}

// ---------------------------------------------------------------------------
// tensor-core products (see TcMatvec): the kernels between the two GEMMs of a
// step, each a fusion of what the next GEMM needs.  q is the step's place in
// the captured graph, *jbase the step the graph starts at.
// ---------------------------------------------------------------------------
// element i of the vector split into the planes of the products' B operand
__device__ __forceinline__ void split_into_planes(const TcMatvecIo& io, int i, double2 v) {
  const uint64_t bx = (uint64_t)__double_as_longlong(v.x), by = (uint64_t)__double_as_longlong(v.y);
  uint32_t hr[3], hi[3];
  const uint32_t fr = f64w_to_f32_bits((uint32_t)bx, (uint32_t)(bx >> 32));
  const uint32_t fi = f64w_to_f32_bits((uint32_t)by, (uint32_t)(by >> 32));
  if (io.pieces == 3) {
    split_f32_bf16<3>(fr, hr);
    split_f32_bf16<3>(fi, hi);
  } else {
    split_f32_bf16<2>(fr, hr);
    split_f32_bf16<2>(fi, hi);
  }
  uint16_t* out = reinterpret_cast<uint16_t*>(io.vplanes) + i;
#pragma unroll
  for (int p = 0; p < 3; ++p)
    if (p < io.pieces) {
      out[(3 * p) * io.vplane] = (uint16_t)(hi[p] ^ 0x8000u);
      out[(3 * p + 1) * io.vplane] = (uint16_t)hr[p];
      out[(3 * p + 2) * io.vplane] = (uint16_t)hi[p];
    }
}

// out = the product of v: its K segments' partial sums added in segment order
// (FP32) plus the FP64 diagonal term; wsum[block] = the block's part of
// Re(conj(v) out).  32 rows per block: eight warps stage the segments in shared memory (all loads in
// flight at once), then one warp adds them in order; one thread per row
// walking the segments itself took 13 us at N = 4,860 (38 dependent rounds on
// 19 blocks).
constexpr int kRedSegs = 64;   // segments staged at a time
__global__ void __launch_bounds__(256) k_tc_reduce_dot(int n, TcMatvecIo io, const double2* v,
                                                       double2* out, double* wsum) {
  __shared__ float2 st[kRedSegs][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 32 + lane;
  double2 w = make_double2(0.0, 0.0), dg = w;
  if (warp == 0 && i < n) {
    w = v[i];
    if (io.diag) dg = io.diag[i * (io.diag_ld + 1)];
  }
  float re = 0.f, im = 0.f;
  for (int s0 = 0; s0 < io.nseg; s0 += kRedSegs) {
    const int ns = min(kRedSegs, io.nseg - s0);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kRedSegs / 8; ++q) {
      const int sgm = warp + 8 * q;
      if (sgm < ns && i < n) st[sgm][lane] = __ldg(io.part + (int64_t)(s0 + sgm) * n + i);
    }
    __syncthreads();
    if (warp == 0 && i < n)
      for (int sgm = 0; sgm < ns; ++sgm) {
        re += st[sgm][lane].x;
        im += st[sgm][lane].y;
      }
  }
  if (warp != 0) return;
  double d = 0.0;
  if (i < n) {
    double2 o = make_double2(f32_to_f64_bits(re), f32_to_f64_bits(im));
    if (io.diag) {
      o.x += dg.x * w.x - dg.y * w.y;
      o.y += dg.x * w.y + dg.y * w.x;
    }
    out[i] = o;
    d = w.x * o.x + w.y * o.y;
  }
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  if (lane == 0) wsum[blockIdx.x] = d;
}

// The dot product from its per-block parts, in every thread of a block of 128:
// groups of eight parts (256 rows) by a tree, the groups in order.  One order,
// so that a run repeats bit for bit (with atomic additions eps changed by up to
// 1e-9 from run to run: the recursion amplifies the last bits).
__device__ __forceinline__ double tc_dot(const double* wsum, int parts) {
  __shared__ double gs[128];
  __shared__ double total;
  double acc = 0.0;
  const int groups = (parts + 7) / 8;
  for (int g0 = 0; g0 < groups; g0 += 128) {
    const int g = g0 + threadIdx.x;
    if (g < groups) {
      double w[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q] = 8 * g + q < parts ? __ldg(wsum + 8 * g + q) : 0.0;
      gs[threadIdx.x] = ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int q = 0; q < min(128, groups - g0); ++q) acc += gs[q];
    __syncthreads();
  }
  if (threadIdx.x == 0) total = acc;
  __syncthreads();
  return total;
}
__global__ void __launch_bounds__(128) k_tc_total(const double* wsum, int parts, double* out) {
  const double t = tc_dot(wsum, parts);
  if (threadIdx.x == 0) *out = t;
}

// alpha_j and y_{j+1} (unnormalised) = u - alpha_j y_j - beta_{j-1} y_{j-1}, split for the
// next product
__global__ void __launch_bounds__(128) k_tc_y(int n, TcMatvecIo io, const double2* u, const double2* y,
                                              const double2* yprev, const double* wsum, int parts,
                                              double* coef, const int* jbase, int q, double2* ynew) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = *jbase + q;
  const double a = tc_dot(wsum, parts);
  if (i == 0) coef[2 * j] = a;
  if (i >= n) return;
  const double b = j > 0 ? sqrt(fmax(coef[2 * j - 1], 0.0)) : 0.0;
  const double2 uy = u[i], y1 = y[i], y0 = yprev[i];
  const double2 o = make_double2(uy.x - a * y1.x - b * y0.x, uy.y - a * y1.y - b * y0.y);
  ynew[i] = o;
  split_into_planes(io, i, o);
}

// beta_{j-1}^2 (<v_0, v_0> before step 0) and v = x / beta, y_prev <- y <- y_new / beta, v
// split for the next product
__global__ void __launch_bounds__(128) k_tc_scale(int n, TcMatvecIo io, const double* wsum, int parts,
                                                  double* coef, const int* jbase, int q,
                                                  const double2* x, double2* v, const double2* ynew,
                                                  double2* y, double2* yprev) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = *jbase + q;
  const double b2 = tc_dot(wsum, parts);
  if (i == 0 && j > 0) coef[2 * j - 1] = b2;
  if (i >= n) return;
  const double f = b2 > 0.0 ? 1.0 / sqrt(b2) : 0.0;
  const double2 xv = x[i], yv = ynew[i];
  const double2 o = make_double2(xv.x * f, xv.y * f);
  yprev[i] = y[i];
  y[i] = make_double2(yv.x * f, yv.y * f);
  v[i] = o;
  split_into_planes(io, i, o);
}

// the step a captured graph starts at: one thread, after the graph's last kernel
__global__ void k_step_add(int* jbase, int by) { *jbase += by; }

// C = A + B, D = A - B (n x n, C and D with leading dimension n)
__global__ void k_form_pm(int n, const double2* A, const double2* B, int64_t ld, double2* C,
                          double2* D) {
  const int64_t total = (int64_t)n * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / n, i = e - j * n;
    const double2 a = A[i + j * ld], b = B[i + j * ld];
    C[e] = make_double2(a.x + b.x, a.y + b.y);
    D[e] = make_double2(a.x - b.x, a.y - b.y);
  }
}

// y = scale conj(rho), split for the first product where that runs on the tensor cores
__global__ void k_conj(int n, TcMatvecIo io, const double2* rho, double scale, double2* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 o = make_double2(scale * rho[i].x, -scale * rho[i].y);
  y[i] = o;
  if (io.vplanes) split_into_planes(io, i, o);
}

// eps(w) = 1 - pref <v,v> / (z^2 - alpha_0 - beta_0^2/(z^2 - alpha_1 - ...)),
// m coefficients (alpha_0 .. alpha_{m-1}, beta_0^2 .. beta_{m-2}^2); one thread
// per frequency.  The tail of the fraction is kept as num / den, so that a
// level is two dependent FMAs (num' = (z^2 - alpha) num - beta^2 den, den' =
// num) instead of a division (11 dependent FP64 operations of about 115 clocks
// each).  A power of two is taken out every 8 levels; where num leaves the range
// of FP64 within them (z^2 beyond 1e38 or below 1e-38: the tail of a recursion
// that has ended has alpha = 0) the 8 are done again with one after each level.
struct LzTail {
  double nr, ni, dr, di;   // num, den
  __device__ __forceinline__ int exponent() const {   // of the larger part of num, biased
    return max((__double2hiint(nr) >> 20) & 0x7FF, (__double2hiint(ni) >> 20) & 0x7FF);
  }
  __device__ __forceinline__ void rescale() {
    const int e = max(exponent(), 1);
    if (e >= 0x7FE || (nr == 0.0 && ni == 0.0)) return;
    const double sc = __longlong_as_double((long long)(2046 - e) << 52);
    nr *= sc;
    ni *= sc;
    dr *= sc;
    di *= sc;
  }
  // one level up: num' = (zr - alpha + i zi) num - b2 den, den' = num
  __device__ __forceinline__ void level(double zr, double zi, double alpha, double b2) {
    const double a = zr - alpha;
    const double tr = fma(a, nr, fma(-zi, ni, -b2 * dr));
    const double ti = fma(a, ni, fma(zi, nr, -b2 * di));
    dr = nr;
    di = ni;
    nr = tr;
    ni = ti;
  }
};
__global__ void k_lanczos_eps(int m, const double* coef, double nv2, int n_omega,
                              const double* omega, double delta, double pref, double2* eps) {
  const int iw = blockIdx.x * blockDim.x + threadIdx.x;
  if (iw >= n_omega) return;
  const double w = omega[iw];
  const double zr = w * w - delta * delta, zi = 2.0 * w * delta;   // (w + i d)^2
  LzTail t{zr - coef[2 * (m - 1)], zi, 1.0, 0.0};
  for (int j0 = m - 2; j0 >= 0; j0 -= 8) {
    t.rescale();
    const LzTail before = t;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (j0 - u >= 0) t.level(zr, zi, coef[2 * (j0 - u)], coef[2 * (j0 - u) + 1]);
    const int e = t.exponent();
    if (e == 0 || e == 0x7FF) {
      t = before;
#pragma unroll 1
      for (int j = j0; j >= 0 && j > j0 - 8; --j) {
        t.level(zr, zi, coef[2 * j], coef[2 * j + 1]);
        t.rescale();
      }
    }
  }
  t.rescale();   // |num|^2 below
  const double g = pref * nv2 / fma(t.nr, t.nr, t.ni * t.ni);   // 1 / (num / den) = den conj(num) / |num|^2
  eps[iw] = make_double2(1.0 - g * fma(t.dr, t.nr, t.di * t.ni), -g * fma(t.di, t.nr, -t.dr * t.ni));
}

// diff[0] = max |a - b|, diff[1] = max |b| over the grid (one block)
__global__ void __launch_bounds__(256) k_eps_change(int n_omega, const double2* a, const double2* b,
                                                    double* diff) {
  __shared__ double r0[256], r1[256];
  double d = 0.0, m = 0.0;
  for (int i = threadIdx.x; i < n_omega; i += 256) {
    d = fmax(d, hypot(a[i].x - b[i].x, a[i].y - b[i].y));
    m = fmax(m, hypot(b[i].x, b[i].y));
  }
  r0[threadIdx.x] = d;
  r1[threadIdx.x] = m;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      r0[threadIdx.x] = fmax(r0[threadIdx.x], r0[threadIdx.x + h]);
      r1[threadIdx.x] = fmax(r1[threadIdx.x], r1[threadIdx.x + h]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    diff[0] = r0[0];
    diff[1] = r1[0];
  }
}

}  // namespace


// eps on the grid from the recursion above; returns the steps taken.
//
// FP64 products: every step between two convergence checks in one cooperative
// launch of k_lanczos_steps.  Tensor-core products: a step is two split-K
// GEMM launches and four element-wise kernels; ten steps are captured once as
// a CUDA graph and replayed (the step index lives on the device, the vectors
// stay in place), so that no launch waits for the host and the products are
// bound by reading the 12 N^2 bytes of planes.  A step at N = 4,860 takes
// 140 us; it took 430 us when each product uploaded its tile list and
// synchronised and ran on 38 blocks (one per 128 rows, all of K each).
int spectrum_lanczos(int n, const bse_c128* A, const bse_c128* B, int64_t ld, const bse_c128* rho,
                     double c_q, double vc, int n_omega, const double* omega, double delta,
                     double tol, int max_steps, int matvec_precision, bse_c128* eps_out,
                     cudaStream_t s) {
  const double2* A2 = reinterpret_cast<const double2*>(A);
  const double2* B2 = reinterpret_cast<const double2*>(B);
  int dev = 0, sms = 0;
  BSE_CUDA(cudaGetDevice(&dev));
  BSE_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const bool tc = matvec_precision != BSE_PREC_FP64;
  const size_t vb = (size_t)n * sizeof(double2);
  // <v_0, v_0> is kept in the last coefficient slot
  const int ncoef = 2 * max_steps + 2, nv2_slot = 2 * max_steps + 1;
  DeviceBuffer bv(tc ? vb : 0, s), bx(vb, s), by0(vb, s), by1(vb, s), by2(vb, s), bu(vb, s),
      coef((size_t)ncoef * sizeof(double), s),
      ea((size_t)std::max(n_omega, 1) * sizeof(double2), s), diff(2 * sizeof(double), s),
      ctl(4 * sizeof(int), s), part((size_t)2 * kLzMaxBlocks * sizeof(double), s),
      dots(tc ? (size_t)((n + 31) / 32) * sizeof(double) : 0, s);
  double* cf = coef.as<double>();
  int* ct = ctl.as<int>();   // [0] first step of the captured graph; [2], [3] grid exchange
  const int eb = (n + 127) / 128, rb = (n + 31) / 32;
  int launches = 0;
  // A+B and A-B formed once (each product then reads one matrix: 4 instead
  // of 6 FP64 FMAs and 16 instead of 32 bytes per element); B = NULL: both A
  std::unique_ptr<DeviceBuffer> pm;
  const double2 *Cp = A2, *Dp = A2;
  int64_t ldp = ld;
  if (B) {
    pm.reset(new DeviceBuffer(2 * (size_t)n * n * sizeof(double2), s));
    k_form_pm<<<sms * 8, 256, 0, s>>>(n, A2, B2, ld, pm->as<double2>(),
                                      pm->as<double2>() + (size_t)n * n);
    ++launches;
    Cp = pm->as<double2>();
    Dp = Cp + (size_t)n * n;
    ldp = n;
  }
  // split-precision products: A+B and A-B split once into BF16 pieces, the
  // products on the tensor cores (the diagonal in FP64), FP64 results
  std::unique_ptr<TcMatvec, void (*)(TcMatvec*)> tcp(nullptr, tc_matvec_destroy);
  std::unique_ptr<TcMatvec, void (*)(TcMatvec*)> tcd(nullptr, tc_matvec_destroy);
  TcMatvecIo iop{}, iod{};
  if (tc) {
    tcp.reset(tc_matvec_create(n, reinterpret_cast<const bse_c128*>(Cp), nullptr, ldp,
                               matvec_precision, 1, s));
    if (B)
      tcd.reset(tc_matvec_create(n, reinterpret_cast<const bse_c128*>(Dp), nullptr, ldp,
                                 matvec_precision, 1, s));
    iop = tc_matvec_io(tcp.get());
    iod = tcd ? tc_matvec_io(tcd.get()) : iop;
  }
  TcMatvec* mp = tcp.get();
  TcMatvec* md = tcd ? tcd.get() : tcp.get();

  Phase ph("spectrum_lanczos", s);
  BSE_CUDA(cudaMemsetAsync(cf, 0, (size_t)ncoef * sizeof(double), s));
  BSE_CUDA(cudaMemsetAsync(ct, 0, 4 * sizeof(int), s));
  if (!tc) {   // y_{-1} and the product read by the start
    BSE_CUDA(cudaMemsetAsync(by2.ptr, 0, vb, s));
    BSE_CUDA(cudaMemsetAsync(bu.ptr, 0, vb, s));
  }

  // FP64 steps [j0, j0 + steps) (steps = 0: the start vector)
  const int rows = (n + std::min(sms, kLzMaxBlocks) - 1) / std::min(sms, kLzMaxBlocks);
  const int blocks = (n + rows - 1) / rows;
  LzArgs lz{n, Cp, Dp, ldp, bx.as<double2>(), bu.as<double2>(),
            {by0.as<double2>(), by1.as<double2>(), by2.as<double2>()}, cf, nv2_slot,
            part.as<double>(), ct + 2, ct + 3, call_wait_cycles(), rows, 0, 0};
  auto fp64_steps = [&](int j0, int steps) {
    lz.j0 = j0;
    lz.steps = steps;
    BSE_CUDA(cudaMemsetAsync(ct + 2, 0, sizeof(int), s));
    void* args[] = {&lz};
    BSE_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_lanczos_steps), dim3(blocks),
                                         dim3(kLzThreads), args, 0, s));
    ++launches;
  };
  // one tensor-core step (place q of a captured graph) on stream st
  double2 *V = bv.as<double2>(), *X = bx.as<double2>(), *U = bu.as<double2>(),
          *Y = by0.as<double2>(), *Yp = by1.as<double2>(), *Yn = by2.as<double2>();
  double* ws = dots.as<double>();
  auto tc_step = [&](cudaStream_t st, int q) {
    k_tc_scale<<<eb, 128, 0, st>>>(n, iop, ws, rb, cf, ct, q, X, V, Yn, Y, Yp);
    tc_matvec_products(mp, st);                                  // u = (A+B) v_j
    k_tc_reduce_dot<<<rb, 256, 0, st>>>(n, iop, V, U, ws);       // alpha_j
    k_tc_y<<<eb, 128, 0, st>>>(n, iod, U, Y, Yp, ws, rb, cf, ct, q, Yn);
    tc_matvec_products(md, st);                                  // x = (A-B) y
    k_tc_reduce_dot<<<rb, 256, 0, st>>>(n, iod, Yn, X, ws);      // beta_j^2
    BSE_CUDA(cudaGetLastError());
  };
  auto step_add = [&](cudaStream_t st, int by) { k_step_add<<<1, 1, 0, st>>>(ct, by); };
  // a bounded wait that expired in any launch so far
  auto check_waits = [&] {
    int gave_up = 0;
    BSE_CUDA(cudaMemcpyAsync(&gave_up, ct + 3, sizeof(int), cudaMemcpyDeviceToHost, s));
    BSE_CUDA(cudaStreamSynchronize(s));
    if (gave_up) throw Error(BSE_ERR_TIMEOUT, "Lanczos: a bounded wait between blocks expired");
    if (tc) tc_matvec_check(mp, s);
    if (tcd) tc_matvec_check(md, s);
  };

  // start: y_0 = conj(rho), v_0 = (A-B) y_0, <v_0, v_0> = y_0^H v_0
  auto conj_rho = [&](double scale) {
    k_conj<<<eb, 128, 0, s>>>(n, iod, reinterpret_cast<const double2*>(rho), scale,
                              tc ? Yn : by0.as<double2>());
    ++launches;
  };
  conj_rho(1.0);
  if (tc) {
    BSE_CUDA(cudaMemsetAsync(Y, 0, vb, s));   // becomes y_{-1}
    tc_matvec_products(md, s);
    k_tc_reduce_dot<<<rb, 256, 0, s>>>(n, iod, Yn, X, ws);
    k_tc_total<<<1, 128, 0, s>>>(ws, rb, cf + nv2_slot);
    launches += 2;
  } else {
    fp64_steps(0, 0);
  }
  double nv2 = 0.0;
  BSE_CUDA(cudaMemcpyAsync(&nv2, cf + nv2_slot, sizeof(double), cudaMemcpyDeviceToHost, s));
  check_waits();
  if (!(nv2 > 0.0)) {
    note_launches(launches);
    throw Error(nv2 == 0.0 ? BSE_ERR_ARG : BSE_ERR_NOT_PD,
                nv2 == 0.0 ? "rho is zero" : "conj(rho)^H (A-B) conj(rho) <= 0: A-B is not positive definite");
  }

  // The FP64 steps leave x_j = beta v_j unnormalised, so alpha_0 comes from sums of
  // the size of <v_0, v_0> alpha_0 (and of its inverse): a start vector near the
  // ends of the FP64 range is brought to about 1 by a power of two (the fraction
  // does not depend on it).
  if (!tc && (nv2 < 1e-200 || nv2 > 1e200) && std::isfinite(nv2)) {
    conj_rho(std::ldexp(1.0, -std::ilogb(nv2) / 2));
    fp64_steps(0, 0);
  }

  // ten tensor-core steps as one graph
  constexpr int kGraphSteps = 10;
  struct GraphGuard {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t e = nullptr;
    cudaStream_t cs = nullptr;
    ~GraphGuard() {
      if (e) cudaGraphExecDestroy(e);
      if (g) cudaGraphDestroy(g);
      if (cs) cudaStreamDestroy(cs);
    }
  } gg;
  if (tc && max_steps >= kGraphSteps) {
    BSE_CUDA(cudaStreamCreateWithFlags(&gg.cs, cudaStreamNonBlocking));
    BSE_CUDA(cudaStreamBeginCapture(gg.cs, cudaStreamCaptureModeThreadLocal));
    for (int q = 0; q < kGraphSteps; ++q) tc_step(gg.cs, q);
    step_add(gg.cs, kGraphSteps);
    BSE_CUDA(cudaStreamEndCapture(gg.cs, &gg.g));
    BSE_CUDA(cudaGraphInstantiate(&gg.e, gg.g, 0));
    note_launches(-2 * kGraphSteps);   // the products captured, not launched
  }
  const double pref = c_q * kHartreeEv * 2.0 / vc;
  // eps is compared every `check` steps; at least min_steps are taken (past
  // n steps the recursion only repeats what the Krylov space already holds)
  const int check = !tc && max_steps >= 6 ? std::max(6, std::min(48, (n / 6) * 6))
                                          : std::max(10, std::min(50, n));
  const int min_steps = std::min(100, 2 * n);
  int steps = 0;
  bool have_prev = false, converged = false;
  while (steps < max_steps) {
    const int upto = std::min(max_steps, (steps / check + 1) * check);
    if (!tc) {
      fp64_steps(steps, upto - steps);
      steps = upto;
    }
    while (steps < upto) {
      if (gg.e && upto - steps >= kGraphSteps) {
        BSE_CUDA(cudaGraphLaunch(gg.e, s));
        launches += kGraphSteps * 6 + 1;   // products and element-wise kernels of the graph
        steps += kGraphSteps;
      } else {
        tc_step(s, 0);
        step_add(s, 1);
        launches += 5;                     // (products count themselves outside the graph)
        steps += 1;
      }
    }
    double2* cur = have_prev ? ea.as<double2>() : reinterpret_cast<double2*>(eps_out);
    k_lanczos_eps<<<(n_omega + 63) / 64, 64, 0, s>>>(steps, cf, nv2, n_omega, omega, delta, pref,
                                                     cur);
    ++launches;
    if (have_prev) {
      k_eps_change<<<1, 256, 0, s>>>(n_omega, reinterpret_cast<double2*>(eps_out), cur,
                                     diff.as<double>());
      BSE_CUDA(cudaMemcpyAsync(eps_out, cur, (size_t)n_omega * sizeof(double2),
                               cudaMemcpyDeviceToDevice, s));
      ++launches;
      double hd[2];
      BSE_CUDA(cudaMemcpyAsync(hd, diff.ptr, sizeof(hd), cudaMemcpyDeviceToHost, s));
      check_waits();
      if (steps >= min_steps && hd[0] <= tol * hd[1]) {
        converged = true;
        break;
      }
    }
    have_prev = true;
  }
  BSE_CUDA(cudaGetLastError());
  note_launches(launches);
  check_waits();
  if (!converged)
    throw Error(BSE_ERR_NO_CONV, "eps changed by more than tol after " + std::to_string(steps) +
                                     " Lanczos steps");
  return steps;
}

}  // namespace bse
