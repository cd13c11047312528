// ddlr_gmres.cuh -- restarted GMRES(m), right-preconditioned (Sec. 5: the
// accelerator for the indefinite problems, GMRES(40)), and the inverse of an
// indefinite I - K for DDLR-2 in the indefinite mode.
//
// One Arnoldi step on A M^-1: z_j = M^-1 v_j (kept, so x += Z y needs no
// further apply), w = A z_j, two classical Gram-Schmidt passes against
// v_0..v_j (the Hessenberg column is the sum of both passes' coefficients:
// the generic CGS kernels of ddlr_lbd.cuh with k_gm_reduce_acc),
// h_{j+1,j} = ||w||, v_{j+1} = w / h_{j+1,j}, then one Givens step.  H is
// column-major with leading dimension m + 1; all scalars stay on the device.
#pragma once
#include "ddlr_lbd.cuh"

namespace ddlr {

// c[col] = sum_g partials[g][col] (a warp per column, fixed order), and the
// Hessenberg column hcol[col] = c[col] (first pass) or += c[col]
__global__ void k_gm_reduce_acc(int G, int ncol, const double *partials, double *c, double *hcol, int first) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, l = threadIdx.x & 31;
  if (w >= ncol) return;
  double s = 0;
  for (int g = l; g < G; g += 32) s += partials[(long long)g * ncol + w];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (l == 0) {
    c[w] = s;
    hcol[w] = first ? s : hcol[w] + s;
  }
}

// sqrt of the sum of G dot partials into *o1 and *o2 (a NaN stays a NaN)
__global__ void k_gm_norm(int G, const double *partials, double *o1, double *o2) {
  const double v = warp_sum_partials(partials, G);
  if (threadIdx.x == 0) {
    const double r = v >= 0.0 ? sqrt(v) : v;
    *o1 = r;
    *o2 = r;
  }
}

// g = (beta, 0, ..., 0), m + 1 entries
__global__ void k_gm_ginit(int m, const double *beta, double *g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i <= m) g[i] = i == 0 ? *beta : 0.0;
}

// Givens step j (one thread): the rotations 0..j-1 applied to column j of H,
// then the rotation that zeroes h_{j+1,j}; g updated; *res = |g_{j+1}|, the
// residual norm of the current iterate
__global__ void k_gm_givens(int j, double *hcol, double *cs, double *sn, double *g, double *res) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int i = 0; i < j; i++) {
    const double t = cs[i] * hcol[i] + sn[i] * hcol[i + 1];
    hcol[i + 1] = -sn[i] * hcol[i] + cs[i] * hcol[i + 1];
    hcol[i] = t;
  }
  const double d = hypot(hcol[j], hcol[j + 1]);
  cs[j] = d > 0.0 ? hcol[j] / d : 1.0;
  sn[j] = d > 0.0 ? hcol[j + 1] / d : 0.0;
  hcol[j] = d;
  hcol[j + 1] = 0.0;
  g[j + 1] = -sn[j] * g[j];
  g[j] = cs[j] * g[j];
  *res = fabs(g[j + 1]);
}

// R y = g, R the leading j x j upper triangle of H (one thread)
__global__ void k_gm_backsolve(int j, const double *H, int ld, const double *g, double *y) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int i = j - 1; i >= 0; i--) {
    double t = g[i];
    for (int l = i + 1; l < j; l++) t -= H[i + (long long)l * ld] * y[l];
    y[i] = t / H[i + (long long)i * ld];
  }
}

// x += Z y (Z n x j column-major), a thread per row, y in shared memory
__global__ void k_gm_update(long long n, int j, const double *Z, const double *y, double *x) {
  extern __shared__ double ys[];
  for (int l = threadIdx.x; l < j; l += blockDim.x) ys[l] = y[l];
  __syncthreads();
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  double t = 0;
  for (int l = 0; l < j; l++) t += Z[(long long)l * n + r] * ys[l];
  x[r] += t;
}

// r = b - q
__global__ void k_gm_resid(long long n, const double *b, const double *q, double *r) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = b[i] - q[i];
}

// Indefinite mode, DDLR-2: H_k = (I - K)^-1 with K the summed products
// (k_hk_reduce), symmetrised as for the Cholesky path, inverted by Gauss-Jordan
// elimination with partial pivoting (the first of equal magnitudes).  A pivot
// of magnitude <= 1e-14 times the largest entry sets *singular.  Hk row-major.
// One CTA: the row operations of a step run over all threads (one thread's
// serial elimination took about as long as the Cholesky form, 20 ms at
// k = 32); every entry sees the operations of the serial elimination.
constexpr int kGjThreads = 512;
__global__ void __launch_bounds__(kGjThreads) k_hk_finalize_gj(int k, double *M, double *Hk, int *singular) {
  __shared__ double fs[256], s_amax[kGjThreads / 32];
  __shared__ int s_piv;
  __shared__ double s_pmax;
  const int tid = threadIdx.x, wi = tid >> 5, l = tid & 31;
  double am = 0.0;
  for (int o = tid; o < k * k; o += kGjThreads) {
    const int a = o / k, b = o - a * k;
    Hk[o] = a == b ? 1.0 : 0.0;
    if (b > a) continue;
    const double v = (a == b ? 1.0 : 0.0) - 0.5 * (M[a * k + b] + M[b * k + a]);
    M[a * k + b] = v;
    M[b * k + a] = v;
    am = fmax(am, fabs(v));
  }
  for (int d = 16; d > 0; d >>= 1) am = fmax(am, __shfl_xor_sync(0xffffffffu, am, d));
  if (l == 0) s_amax[wi] = am;
  __syncthreads();
  am = 0.0;
  for (int w = 0; w < kGjThreads / 32; w++) am = fmax(am, s_amax[w]);
  for (int j = 0; j < k; j++) {
    if (wi == 0) {
      double best = -1.0;
      int at = k;
      for (int r = j + l; r < k; r += 32) {
        const double v = fabs(M[r * k + j]);
        if (v > best) { best = v; at = r; }
      }
      for (int d = 16; d > 0; d >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, d);
        const int oa = __shfl_xor_sync(0xffffffffu, at, d);
        if (ob > best || (ob == best && oa < at)) { best = ob; at = oa; }
      }
      if (l == 0) { s_piv = at; s_pmax = best; }
    }
    __syncthreads();
    const int piv = s_piv;
    if (!(s_pmax > 1e-14 * am)) {
      if (tid == 0) *singular = 1;
      return;
    }
    const double d = M[piv * k + j];
    __syncthreads();
    // rows j and piv change places, row j divided by the pivot
    for (int c = tid; c < k; c += kGjThreads) {
      const double mp = M[piv * k + c], hp = Hk[piv * k + c];
      if (piv != j) {
        M[piv * k + c] = M[j * k + c];
        Hk[piv * k + c] = Hk[j * k + c];
      }
      M[j * k + c] = mp / d;
      Hk[j * k + c] = hp / d;
    }
    __syncthreads();
    for (int r = tid; r < k; r += kGjThreads) fs[r] = M[r * k + j];
    __syncthreads();
    for (int r = wi; r < k; r += kGjThreads / 32) {
      const double f = fs[r];
      if (r == j || f == 0.0) continue;
      for (int c = l; c < k; c += 32) {
        M[r * k + c] -= f * M[j * k + c];
        Hk[r * k + c] -= f * Hk[j * k + c];
      }
    }
    __syncthreads();
  }
}

}  // namespace ddlr
