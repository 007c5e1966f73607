// CUDA kernels of the periodic FM-BEM (sm_103a).
//
// Operator (paper eq. 9) applied to Psi = (phi_e, varphi_e) per element:
//   y_2e   = phi_e - V_e + U_e
//   y_2e+1 = varphi_e + c2 (dU_e - rho dV_e),      c2 = 2 / (i eta (1 + rho))
// with V = D1 phi - i eta S1 varphi, dV = T1 phi - i eta K1 varphi (same fiber,
// wavenumber k1, eq. 5) and U = D2b phi - i eta S2b varphi, dU = T2b phi - i eta
// K2b varphi (all fibers and their images, wavenumber k, eqs. 7-8).  U and dU
// come from the periodic FMM of Sec. 3 (near field + P2M/M2M/M2L/L2L/L2P +
// lattice-sum root translation), V and dV from a fiber-local direct sum.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "internal.h"
#include "side_chain.h"

// Gauss-Legendre rules g = 1..16 on [-1, 1]: node q of rule g at [g-1][q].
__constant__ double c_glx[PF_GLMAX][PF_GLMAX];
__constant__ double c_glw[PF_GLMAX][PF_GLMAX];
__constant__ float c_glxf[PF_GLMAX][PF_GLMAX];
__constant__ float c_glwf[PF_GLMAX][PF_GLMAX];
// q-thresholds (distance / element length) above which rule g meets the
// quadrature tolerance; [0] for the FP64 path, [1] for the FP32 path.
__constant__ double c_glthr[2][PF_GLMAX + 1];

// Rule size for a source element at distance ratio q = |x - c| / h.
__device__ __forceinline__ int gl_order(double q, int which) {
  int g = 1;
#pragma unroll 1
  while (g < PF_GLMAX && q < c_glthr[which][g]) ++g;
  return g;
}

void k_upload_gauss(const double* x, const double* w, const double* thr64, const double* thr32) {
  float xf[PF_GLMAX * PF_GLMAX], wf[PF_GLMAX * PF_GLMAX];
  for (int i = 0; i < PF_GLMAX * PF_GLMAX; ++i) {
    xf[i] = (float)x[i];
    wf[i] = (float)w[i];
  }
  double thr[2][PF_GLMAX + 1];
  for (int i = 0; i <= PF_GLMAX; ++i) {
    thr[0][i] = thr64[i];
    thr[1][i] = thr32[i];
  }
  cudaMemcpyToSymbol(c_glx, x, sizeof(double) * PF_GLMAX * PF_GLMAX);
  cudaMemcpyToSymbol(c_glw, w, sizeof(double) * PF_GLMAX * PF_GLMAX);
  cudaMemcpyToSymbol(c_glxf, xf, sizeof(xf));
  cudaMemcpyToSymbol(c_glwf, wf, sizeof(wf));
  cudaMemcpyToSymbol(c_glthr, thr, sizeof(thr));
}

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ cplx cexp_d(cplx z) {
  double s, c;
  sincos(z.im, &s, &c);
  double e = exp(z.re);
  return cplx{e * c, e * s};
}
__device__ __forceinline__ cplx clog_d(cplx z) { return cplx{log(hypot(z.re, z.im)), atan2(z.im, z.re)}; }
__device__ __forceinline__ cplx csqrt_d(cplx z) {
  double r = hypot(z.re, z.im);
  double a = sqrt(fmax(0.0, 0.5 * (r + z.re)));
  double b = sqrt(fmax(0.0, 0.5 * (r - z.re)));
  return cplx{a, z.im < 0 ? -b : b};
}
__device__ __forceinline__ cplx shfl_down(cplx v, int o) {
  return cplx{__shfl_down_sync(0xffffffffu, v.re, o), __shfl_down_sync(0xffffffffu, v.im, o)};
}
__device__ __forceinline__ cplx warp_sum(cplx v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += shfl_down(v, o);
  return v;
}
__device__ __forceinline__ cplx ipow_phase(cplx alpha, int m) {
  // alpha^m for any image m by |m| products; |alpha| = 1, so alpha^{-1} = conj(alpha)
  cplx r{1, 0};
  for (int i = 0; i < (m < 0 ? -m : m); ++i) r = r * alpha;
  return m < 0 ? conj(r) : r;
}

// ---------------------------------------------------------------- profiling
void prof_begin(pfmbem* h, int ph) {
  h->prof.launches[ph]++;
  if (!h->prof.on) return;
  if (h->prof.ev.empty()) {
    h->prof.ev.resize(4096);
    for (auto& e : h->prof.ev) cudaEventCreate(&e);
  }
  if (h->prof.used + 2 > (int)h->prof.ev.size()) prof_fold(h);
  cudaEventRecord(h->prof.ev[h->prof.used++], h->stream);
}

void prof_end(pfmbem* h, int ph) {
  if (!h->prof.on) return;
  cudaEventRecord(h->prof.ev[h->prof.used++], h->stream);
  h->prof.phase_of_pair.push_back(ph);
}

cudaError_t prof_fold(pfmbem* h) {
  Prof& P = h->prof;
  if (P.used == 0) return cudaSuccess;
  cudaError_t e = cudaEventSynchronize(P.ev[P.used - 1]);
  if (e != cudaSuccess) return e;
  for (size_t i = 0; i < P.phase_of_pair.size(); ++i) {
    float ms = 0;
    cudaEventElapsedTime(&ms, P.ev[2 * i], P.ev[2 * i + 1]);
    P.ms[P.phase_of_pair[i]] += ms;
  }
  P.used = 0;
  P.phase_of_pair.clear();
  return cudaSuccess;
}

void prof_release(pfmbem* h) {
  for (auto& e : h->prof.ev) cudaEventDestroy(e);
  h->prof.ev.clear();
}

// ---------------------------------------------------------------- translation tables
// Built on the device from the level's weights w_n (already resident), one
// block per translation vector; thread 0 evaluates J_0..J_N (Miller) and
// Y_0..Y_N (CUDA y0/y1 and forward recurrence) of k|v| into shared memory.
__device__ void bessel_jy_block(double x, int N, double* J, double* Y) {
  if (threadIdx.x == 0) {
    bessel_j_array(x, N, J);
    Y[0] = y0(x);
    if (N >= 1) Y[1] = y1(x);
    for (int n = 1; n < N; ++n) Y[n + 1] = (2.0 * n / x) * Y[n] - Y[n - 1];
  }
  __syncthreads();
}

// M2L operators of level l = blockIdx.y + 1 (Sec. 3.2): T[o][a][n] = w_a H^+_{n-a}(k v_o) w_n,
// H^+_j = H_j(k|v|) e^{i j theta_v}, H_{-j} = (-1)^j H_j, for the offsets
// v_o = (dx, dy) d, o = (dx + 3) 7 + (dy + 3) = blockIdx.x; offsets with
// max(|dx|, |dy|) <= 1 are never used and are written as zeros.  Also the
// transposed copy [o][n][a] and FP32 copies.
__global__ void m2l_tables_kernel(TableLevels tl, double k, int* __restrict__ bad) {
  const int l = blockIdx.y + 1, o = blockIdx.x, dx = o / 7 - 3, dy = o % 7 - 3;
  const int p = tl.p[l], P = 2 * p + 1;
  const double* w = tl.w[l];
  cplx* T = tl.T[l] + (size_t)o * P * P;
  cplxf* Tf = tl.Tf[l] + (size_t)o * P * P;
  cplx* Tt = tl.Tt[l] + (size_t)o * P * P;
  cplxf* Ttf = tl.Ttf[l] + (size_t)o * P * P;
  cplxf* Ttl = tl.Ttl[l] + (size_t)o * P * P;
  if (abs(dx) <= 1 && abs(dy) <= 1) {
    for (int t = threadIdx.x; t < P * P; t += blockDim.x) {
      T[t] = Tt[t] = cplx{0, 0};
      Tf[t] = Ttf[t] = Ttl[t] = cplxf{0, 0};
    }
    return;
  }
  __shared__ double J[4 * PF_PMAX + 2], Y[4 * PF_PMAX + 2];
  __shared__ cplx hv[4 * PF_PMAX + 1];
  const double vx = dx * tl.d[l], vy = dy * tl.d[l];
  const double r = sqrt(vx * vx + vy * vy), th = atan2(vy, vx);
  bessel_jy_block(k * r, 2 * p, J, Y);
  for (int j = threadIdx.x - 2 * p; j <= 2 * p; j += blockDim.x) {
    const int aj = abs(j);
    const double sg = (j < 0 && (aj & 1)) ? -1.0 : 1.0;
    double sn, cs;
    sincos(j * th, &sn, &cs);
    const double hr = sg * J[aj], hi = sg * Y[aj];
    hv[j + 2 * p] = cplx{hr * cs - hi * sn, hr * sn + hi * cs};
  }
  __syncthreads();
  for (int t = threadIdx.x; t < P * P; t += blockDim.x) {
    const int a = t / P, n = t % P;                 // a: target coefficient + p, n: source + p
    const cplx hj = hv[n - a + 2 * p];
    const double sc = w[a] * w[n];
    const cplx v{sc * hj.re, sc * hj.im};
    if (!isfinite(v.re) || !isfinite(v.im)) atomicExch(bad, 1);
    T[t] = v;
    Tf[t] = to_f(v);
    Tt[(size_t)n * P + a] = v;
    Ttf[(size_t)n * P + a] = to_f(v);
    Ttl[(size_t)n * P + a] = split_lo(v);
  }
}

// M2M (children of level l+1 -> level l) and L2L (level l -> children), l =
// blockIdx.y, for the child quadrant q = blockIdx.x, v = O_child - O_parent:
//   A[q][m][n] = J^-_{n-m}(k v) w^c_m / w^p_n,  J^-_j = J_j e^{-i j theta}
//   B[q][m][n] = w^c_n J^+_{m-n}(k v) / w^p_m,  J^+_j = J_j e^{+i j theta}
// (m child and n parent coefficient in A, m parent and n child in B).
__global__ void m2m_tables_kernel(TableLevels tl, double k) {
  const int l = blockIdx.y, q = blockIdx.x, cx = q & 1, cy = (q >> 1) & 1;
  const int p = tl.p[l], pc = tl.p[l + 1], P = 2 * p + 1, Pc = 2 * pc + 1;
  const double* wp = tl.w[l];
  const double* wc = tl.w[l + 1];
  __shared__ double J[2 * PF_PMAX + 2], Y[2 * PF_PMAX + 2];
  __shared__ cplx ej[4 * PF_PMAX + 3];            // J_j e^{i j theta}, j = -(p + pc) .. p + pc
  const double dc = tl.d[l + 1];
  const double vx = (cx - 0.5) * dc, vy = (cy - 0.5) * dc;
  const double r = sqrt(vx * vx + vy * vy), th = atan2(vy, vx);
  bessel_jy_block(k * r, p + pc, J, Y);
  {
    // the entries depend on j = n - m only: one sincos per j instead of per entry
    const int jm = p + pc;
    for (int j = (int)threadIdx.x - jm; j <= jm; j += blockDim.x) {
      const int aj = abs(j);
      const double Jj = (j < 0 && (aj & 1)) ? -J[aj] : J[aj];
      double sn, cs;
      sincos(j * th, &sn, &cs);
      ej[j + jm] = cplx{Jj * cs, Jj * sn};
    }
    __syncthreads();
  }
  cplx* A = tl.A[l] + (size_t)q * Pc * P;
  cplxf* Af = tl.Af[l] + (size_t)q * Pc * P;
  cplxf* Al = tl.Al[l] + (size_t)q * Pc * P;
  cplx* B = tl.B[l] + (size_t)q * P * Pc;
  cplxf* Bf = tl.Bf[l] + (size_t)q * P * Pc;
  cplxf* Bl = tl.Bl[l] + (size_t)q * P * Pc;
  for (int t = threadIdx.x; t < P * Pc; t += blockDim.x) {
    {
      const int m = t / P - pc, n = t % P - p;       // A: [q][m + pc][n + p]
      const cplx e = ej[n - m + p + pc];              // J_j e^{i j theta}; A takes J_j e^{-i j theta}
      const double sc = wc[m + pc] / wp[n + p];
      const cplx v{sc * e.re, -sc * e.im};
      A[t] = v;
      Af[t] = to_f(v);
      Al[t] = split_lo(v);
    }
    {
      const int m = t / Pc - p, n = t % Pc - pc;     // B: [q][m + p][n + pc]
      const cplx e = ej[m - n + p + pc];
      const double sc = wc[n + pc] / wp[m + p];
      const cplx v{sc * e.re, sc * e.im};
      B[t] = v;
      Bf[t] = to_f(v);
      Bl[t] = split_lo(v);
    }
  }
}

cudaError_t k_tables(pfmbem* h, const TableLevels& tl, cudaStream_t st) {
  if (h->D >= 1) {
    m2l_tables_kernel<<<dim3(49, h->D), 256, 0, st>>>(tl, h->k, h->tab_err);
    m2m_tables_kernel<<<dim3(4, h->D), 256, 0, st>>>(tl, h->k);
  }
  return cudaGetLastError();
}

// Triangle tree (Sec. 3.1, Fig. 5): the cells' centres are not on one grid, so
// the operators are built for the list of offsets that occur, per level.
// M2L, one block per offset v_o = target - source centre:
//   T[o][a][n] = w_a H^+_{n-a}(k v_o) w_n   (the square tree's formula above).
__global__ void tri_m2l_tables_kernel(const double2* __restrict__ v, int p, const double* __restrict__ w, double k,
                                      cplx* __restrict__ T, int* __restrict__ bad) {
  const int o = blockIdx.x, P = 2 * p + 1;
  __shared__ double J[4 * PF_PMAX + 2], Y[4 * PF_PMAX + 2];
  __shared__ cplx hv[4 * PF_PMAX + 1];
  const double vx = v[o].x, vy = v[o].y;
  const double r = sqrt(vx * vx + vy * vy), th = atan2(vy, vx);
  bessel_jy_block(k * r, 2 * p, J, Y);
  for (int j = threadIdx.x - 2 * p; j <= 2 * p; j += blockDim.x) {
    const int aj = abs(j);
    const double sg = (j < 0 && (aj & 1)) ? -1.0 : 1.0;
    double sn, cs;
    sincos(j * th, &sn, &cs);
    const double hr = sg * J[aj], hi = sg * Y[aj];
    hv[j + 2 * p] = cplx{hr * cs - hi * sn, hr * sn + hi * cs};
  }
  __syncthreads();
  cplx* To = T + (size_t)o * P * P;
  for (int t = threadIdx.x; t < P * P; t += blockDim.x) {
    const int a = t / P, n = t % P;
    const cplx hj = hv[n - a + 2 * p];
    const double sc = w[a] * w[n];
    const cplx val{sc * hj.re, sc * hj.im};
    if (!isfinite(val.re) || !isfinite(val.im)) atomicExch(bad, 1);
    To[t] = val;
  }
}

// M2M and L2L, one block per child offset v_q = O_child - O_parent (zero for the
// middle child of a triangle, whose centroid is its parent's):
//   A[q][m][n] = J^-_{n-m}(k v) w^c_m / w^p_n,  B[q][m][n] = w^c_n J^+_{m-n}(k v) / w^p_m
// (m child and n parent coefficient in A, m parent and n child in B).
__global__ void tri_shift_tables_kernel(const double2* __restrict__ v, int p, int pc, const double* __restrict__ wp,
                                        const double* __restrict__ wc, double k, cplx* __restrict__ A,
                                        cplx* __restrict__ B) {
  const int q = blockIdx.x, P = 2 * p + 1, Pc = 2 * pc + 1;
  __shared__ double J[2 * PF_PMAX + 2], Y[2 * PF_PMAX + 2];
  __shared__ cplx ej[4 * PF_PMAX + 3];            // J_j e^{i j theta}, j = -(p + pc) .. p + pc
  const double vx = v[q].x, vy = v[q].y;
  const double r = sqrt(vx * vx + vy * vy), th = r > 0 ? atan2(vy, vx) : 0.0;
  bessel_jy_block(k * r, p + pc, J, Y);          // r = 0: J_n = delta_n0 (Y is not used)
  const int jm = p + pc;
  for (int j = (int)threadIdx.x - jm; j <= jm; j += blockDim.x) {
    const int aj = abs(j);
    const double Jj = (j < 0 && (aj & 1)) ? -J[aj] : J[aj];
    double sn, cs;
    sincos(j * th, &sn, &cs);
    ej[j + jm] = cplx{Jj * cs, Jj * sn};
  }
  __syncthreads();
  cplx* Aq = A + (size_t)q * Pc * P;
  cplx* Bq = B + (size_t)q * P * Pc;
  for (int t = threadIdx.x; t < P * Pc; t += blockDim.x) {
    {
      const int m = t / P - pc, n = t % P - p;       // A: [q][m + pc][n + p]
      const cplx e = ej[n - m + jm];
      const double sc = wc[m + pc] / wp[n + p];
      Aq[t] = cplx{sc * e.re, -sc * e.im};
    }
    {
      const int m = t / Pc - p, n = t % Pc - pc;     // B: [q][m + p][n + pc]
      const cplx e = ej[m - n + jm];
      const double sc = wc[n + pc] / wp[m + p];
      Bq[t] = cplx{sc * e.re, sc * e.im};
    }
  }
}

cudaError_t k_tri_tables(pfmbem* h, int l, const double2* m2l_v, int nm2l, const double2* shift_v, int nshift) {
  Level& L = h->lev[l];
  if (nm2l > 0) tri_m2l_tables_kernel<<<nm2l, 256, 0, h->stream>>>(m2l_v, L.p, L.w_dev, h->k, L.m2l, h->tab_err);
  if (nshift > 0)
    tri_shift_tables_kernel<<<nshift, 256, 0, h->stream>>>(shift_v, L.p, h->lev[l + 1].p, L.w_dev,
                                                           h->lev[l + 1].w_dev, h->k, L.m2m, L.l2l);
  return cudaGetLastError();
}

// Periodic root translation (Sec. 3.3): R[a][n] = w_a S_{|n-a|} w_n, S_{-j} = S_j.
__global__ void root_operator_kernel(int p0, const double* __restrict__ w, const cplx* __restrict__ S,
                                     cplx* __restrict__ R, cplxf* __restrict__ Rf, int* __restrict__ bad) {
  const int P = 2 * p0 + 1;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < P * P; t += gridDim.x * blockDim.x) {
    const int a = t / P, n = t % P;
    const cplx sj = S[abs(n - a)];
    const double sc = w[a] * w[n];
    const cplx v{sc * sj.re, sc * sj.im};
    if (!isfinite(v.re) || !isfinite(v.im)) atomicExch(bad, 1);
    R[t] = v;
    if (Rf) Rf[t] = to_f(v);
  }
}

cudaError_t k_root_operator(pfmbem* h, int p0, const double* w0, const cplx* S) {
  const int P = 2 * p0 + 1;
  prof_begin(h, PH_SETUP);
  root_operator_kernel<<<(P * P + 255) / 256, 256, 0, h->stream>>>(p0, w0, S, h->root, h->rootf, h->tab_err);
  prof_end(h, PH_SETUP);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- blocks wider than H
// A row of nr root squares (centres c_i, level-0 order p0) is closed at the top by a
// super root: the centre C of the row, radius R_s, order ps.  The images |m| >= m0 of
// the whole row reach every root through C: M2M from each root to C, the lattice
// sums of Sec. 3.3 taken from image m0 on, L2L from C back to each root.  The images
// |m| < m0 of the root pairs that are not neighbours (|i - j| > 1 or |m| > 1) go by
// explicit root-to-root M2L; the neighbours are the tree lists' (Sec. 3.1).  With
// the translation tables' conventions (A[child m][parent n], B[parent m][child n],
// T[target a][source n] = w_a H^+_{n-a}(k v) w_n, v = target - source centre):
//   TOP[(i,a)][(j,n)] = sum_c B_i[c][a] sum_b R_s[c][b] A_j[n][b]
//                      + sum_{explicit m} alpha^m w_a H^+_{n-a}(k (c_i - c_j - m h)) w_n.
// One root (nr = 1, m0 = 2, C = c_0) gives TOP = R.

// A_j and B_j of root j = blockIdx.x, v = c_j - C.
__global__ void wide_shift_kernel(int p0, int ps, double k, const double2* __restrict__ v, const double* __restrict__ w0,
                                  const double* __restrict__ ws, cplx* __restrict__ A, cplx* __restrict__ B) {
  const int j = blockIdx.x, P0 = 2 * p0 + 1, Ps = 2 * ps + 1;
  __shared__ double J[2 * PF_PMAX + 2], Y[2 * PF_PMAX + 2];
  const double vx = v[j].x, vy = v[j].y;
  const double r = sqrt(vx * vx + vy * vy), th = r > 0 ? atan2(vy, vx) : 0.0;
  bessel_jy_block(k * r, p0 + ps, J, Y);          // r = 0 (a root at C): J_n = delta_n0; Y is not used
  cplx* Aj = A + (size_t)j * P0 * Ps;
  cplx* Bj = B + (size_t)j * Ps * P0;
  for (int t = threadIdx.x; t < P0 * Ps; t += blockDim.x) {
    {
      const int m = t / Ps - p0, n = t % Ps - ps;      // A: [m + p0 (root)][n + ps (super)]
      const int jj = n - m, aj = abs(jj);
      const double Jj = (jj < 0 && (aj & 1)) ? -J[aj] : J[aj];
      const double sc = w0[m + p0] / ws[n + ps];
      double sn, cs;
      sincos(jj * th, &sn, &cs);
      Aj[t] = cplx{sc * Jj * cs, -sc * Jj * sn};
    }
    {
      const int m = t / P0 - ps, n = t % P0 - p0;      // B: [m + ps (super)][n + p0 (root)]
      const int jj = m - n, aj = abs(jj);
      const double Jj = (jj < 0 && (aj & 1)) ? -J[aj] : J[aj];
      const double sc = w0[n + p0] / ws[m + ps];
      double sn, cs;
      sincos(jj * th, &sn, &cs);
      Bj[t] = cplx{sc * Jj * cs, sc * Jj * sn};
    }
  }
}

// X_j[c][n] = sum_b R_s[c][b] A_j[n][b], one thread per (j, c, n).
__global__ void wide_x_kernel(int nr, int P0, int Ps, const cplx* __restrict__ Rs, const cplx* __restrict__ A,
                              cplx* __restrict__ X) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (size_t)nr * Ps * P0) return;
  const int j = (int)(t / ((size_t)Ps * P0)), c = (int)(t / P0 % Ps), n = (int)(t % P0);
  const cplx* Ar = A + ((size_t)j * P0 + n) * Ps;
  const cplx* Rr = Rs + (size_t)c * Ps;
  cplx acc{0, 0};
  for (int b = 0; b < Ps; ++b) acc += Rr[b] * Ar[b];
  X[t] = acc;
}

// TOP tile (i, j) = blockIdx.x / nr, blockIdx.x % nr.
__global__ void wide_top_kernel(int nr, int p0, int Ps, int m0, double k, double H, cplx alpha,
                                const double2* __restrict__ ctr, const double* __restrict__ w0,
                                const cplx* __restrict__ B, const cplx* __restrict__ X, cplx* __restrict__ TOP,
                                int* __restrict__ bad, const unsigned char* __restrict__ nbr) {
  const int i = blockIdx.x / nr, j = blockIdx.x % nr, P0 = 2 * p0 + 1, RS = nr * P0;
  const cplx* Bi = B + (size_t)i * Ps * P0;
  const cplx* Xj = X + (size_t)j * Ps * P0;
  for (int t = threadIdx.x; t < P0 * P0; t += blockDim.x) {
    const int a = t / P0, n = t % P0;
    cplx acc{0, 0};
    for (int c = 0; c < Ps; ++c) acc += Bi[(size_t)c * P0 + a] * Xj[(size_t)c * P0 + n];
    TOP[(size_t)(i * P0 + a) * RS + j * P0 + n] = acc;
  }
  __shared__ double J[4 * PF_PMAX + 2], Y[4 * PF_PMAX + 2];
  __shared__ cplx hv[4 * PF_PMAX + 1];
  for (int m = -(m0 - 1); m <= m0 - 1; ++m) {
    // neighbours: the tree's lists (a row of squares: adjacent indices; otherwise
    // the mask nbr[i][j][m + 1] over the images |m| <= 1)
    if (abs(m) <= 1 && (nbr ? nbr[((size_t)i * nr + j) * 3 + m + 1] != 0 : abs(i - j) <= 1)) continue;
    const double vx = ctr[i].x - ctr[j].x, vy = ctr[i].y - ctr[j].y - m * H;
    const double r = sqrt(vx * vx + vy * vy), th = atan2(vy, vx);
    __syncthreads();
    bessel_jy_block(k * r, 2 * p0, J, Y);
    for (int q = threadIdx.x - 2 * p0; q <= 2 * p0; q += blockDim.x) {
      const int aq = abs(q);
      const double sg = (q < 0 && (aq & 1)) ? -1.0 : 1.0;
      double sn, cs;
      sincos(q * th, &sn, &cs);
      const double hr = sg * J[aq], hi = sg * Y[aq];
      hv[q + 2 * p0] = cplx{hr * cs - hi * sn, hr * sn + hi * cs};
    }
    __syncthreads();
    const cplx am = ipow_phase(alpha, m);
    for (int t = threadIdx.x; t < P0 * P0; t += blockDim.x) {
      const int a = t / P0, n = t % P0;
      const cplx h = am * hv[n - a + 2 * p0];
      const double sc = w0[a] * w0[n];
      cplx* o = TOP + (size_t)(i * P0 + a) * RS + j * P0 + n;
      *o = *o + cplx{sc * h.re, sc * h.im};
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < P0 * P0; t += blockDim.x) {
    const cplx v = TOP[(size_t)(i * P0 + t / P0) * RS + j * P0 + t % P0];
    if (!isfinite(v.re) || !isfinite(v.im)) atomicExch(bad, 1);
  }
}

// The super root's expansions for the field: M_C = sum_j A_j^T M_j over the
// non-empty roots, L_C = R_s M_C.  One block.
__global__ void wide_local_kernel(int nne0, const int* __restrict__ ne0, int P0, int Ps, const cplx* __restrict__ A,
                                  const cplx* __restrict__ Rs, const cplx* __restrict__ M0, cplx* __restrict__ ML) {
  cplx* Ms = ML;
  cplx* Ls = ML + Ps;
  for (int b = threadIdx.x; b < Ps; b += blockDim.x) {
    cplx acc{0, 0};
    for (int r = 0; r < nne0; ++r) {
      const int j = ne0[r];
      const cplx* Aj = A + (size_t)j * P0 * Ps;
      for (int n = 0; n < P0; ++n) acc += Aj[(size_t)n * Ps + b] * M0[(size_t)j * P0 + n];
    }
    Ms[b] = acc;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < Ps; c += blockDim.x) {
    cplx acc{0, 0};
    for (int b = 0; b < Ps; ++b) acc += Rs[(size_t)c * Ps + b] * Ms[b];
    Ls[c] = acc;
  }
}

// dv: [2 nr] device: the roots' centres, then their shifts c_j - C; S [2 ps + 1] and
// X [nr][Ps][P0] device scratch; the super root's weights, A, B, R_s and the
// expansions' buffer are the handle's (allocated by the caller).
cudaError_t k_wide_top(pfmbem* h, const double2* dv, cplx* S, cplx* X, const unsigned char* nbr) {
  const int nr = h->nroot, p0 = h->lev[0].p, P0 = 2 * p0 + 1, ps = h->wide_ps, Ps = 2 * ps + 1;
  cudaStream_t st = h->stream;
  prof_begin(h, PH_SETUP);
  // lattice sums of the super root from image m0 on
  cudaError_t e = k_lattice_sums(h, 2 * ps, std::max(h->lattice_q, h->wide_m0 + 4), S, h->wide_m0);
  if (e != cudaSuccess) return e;
  root_operator_kernel<<<(Ps * Ps + 255) / 256, 256, 0, st>>>(ps, h->wide_w, S, h->wide_Rs, nullptr, h->tab_err);
  wide_shift_kernel<<<nr, 256, 0, st>>>(p0, ps, h->k, dv + nr, h->lev[0].w_dev, h->wide_w, h->wide_A, h->wide_B);
  const size_t nx = (size_t)nr * Ps * P0;
  wide_x_kernel<<<(unsigned)((nx + 255) / 256), 256, 0, st>>>(nr, P0, Ps, h->wide_Rs, h->wide_A, X);
  wide_top_kernel<<<nr * nr, 256, 0, st>>>(nr, p0, Ps, h->wide_m0, h->k, h->H, h->alpha, dv, h->lev[0].w_dev,
                                           h->wide_B, X, h->root, h->tab_err, nbr);
  prof_end(h, PH_SETUP);
  return cudaGetLastError();
}

cudaError_t k_wide_local(pfmbem* h) {
  const Level& r = h->lev[0];
  const int Ps = 2 * h->wide_ps + 1;
  wide_local_kernel<<<1, 256, 0, h->stream>>>(r.nne, r.ne, r.P, Ps, h->wide_A, h->wide_Rs, r.M, h->wide_ML);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- self terms
// S_ee = (i/2)(1/kappa) I(x), T_ee = (i/2) kappa [I(x) - H1(x)], x = kappa h/2,
// I(x) = int_0^x H0(t) dt by term-wise integration of the ascending series of
// J0 and Y0 (Y0 = (2/pi)(ln(t/2) + gamma) J0 + (2/pi) sum (-1)^{m+1} H_m (t/2)^{2m}/(m!)^2).
__device__ void self_pair(double kap, double h, cplx& S, cplx& T) {
  const double x = 0.5 * kap * h;
  const double hx2 = 0.25 * x * x;
  const double lnh = log(0.5 * x);
  const double EG = 0.57721566490153286061;
  double base = x;     // x (x/2)^{2m} / (m!)^2
  double IJ = 0.0, IYa = 0.0, IYb = 0.0, Hm = 0.0;
  for (int m = 0; m < 60; ++m) {
    double term = base / (2 * m + 1);
    double sg = (m & 1) ? -1.0 : 1.0;
    IJ += sg * term;
    IYa += sg * term * (lnh + EG - 1.0 / (2 * m + 1));
    if (m >= 1) IYb += -sg * Hm * term;
    if (fabs(term) < 1e-18 * fabs(IJ)) break;
    base *= hx2 / ((double)(m + 1) * (m + 1));
    Hm += 1.0 / (m + 1);
  }
  const double IY = (2.0 / M_PI) * (IYa + IYb);
  const double J1 = j1(x), Y1 = y1(x);
  S = cplx{-IY / (2.0 * kap), IJ / (2.0 * kap)};
  T = cplx{-0.5 * kap * (IY - Y1), 0.5 * kap * (IJ - J1)};
}

__global__ void self_terms_kernel(int E, double k, double k1, const double* __restrict__ hlen, cplx* __restrict__ out) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  cplx s, t;
  self_pair(k, hlen[e], s, t);
  out[4 * e + 0] = s;
  out[4 * e + 1] = t;
  self_pair(k1, hlen[e], s, t);
  out[4 * e + 2] = s;
  out[4 * e + 3] = t;
}

cudaError_t k_self_terms(pfmbem* h) {
  prof_begin(h, PH_SETUP);
  self_terms_kernel<<<(h->E + 127) / 128, 128, 0, h->stream>>>(h->E, h->k, h->k1, h->o_h, h->self4);
  prof_end(h, PH_SETUP);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- lattice sums
// S_j = sum_{2<=|m|<=q} alpha^m H_j(k|m|H) e^{i j theta} + tail_+ + tail_-,
// tails from the spectral form of the image sums (Sec. 3.3, eq. 17) on the
// contour t = +-sqrt(u^2 - 2iku) of eq. 18 with u = v^2, where mu = u - ik and
// dt / mu = du / sqrt(u^2 - 2iku) (the Jacobian), so that
//   tail_+(n) = (1/(i pi)) int_0^inf (-i/k)^n [w^n + (-k^2/w)^n] e^{iq beta - qH mu}
//               / (e^{H mu - i beta} - 1) * 2 / sqrt(v^2 - 2ik) dv,   w = mu + sqrt(u^2 - 2iku)
//   tail_-(n) = the same with beta -> -beta and (-i/k)^n -> (i/k)^n.
// One block per order j >= 0 (S_-j = S_j); nodes: composite 16-point Gauss on
// geometrically graded panels [V 2^-(P-1-i)...], given by the host.
#define LS_PANELS 12
__global__ void lattice_sum_kernel(int jmax, int q, double k, double H, double beta, double V,
                                   cplx* __restrict__ out, int mlo = 2) {
  const int j = blockIdx.x;
  __shared__ double red[2][256];
  cplx acc{0, 0};
  const int nq = LS_PANELS * 16;
  for (int t = threadIdx.x; t < nq; t += blockDim.x) {
    int pnl = t / 16, node = t % 16;
    double a = (pnl == 0) ? 0.0 : V * ldexp(1.0, pnl - LS_PANELS);
    double b = V * ldexp(1.0, pnl + 1 - LS_PANELS);
    double v = 0.5 * (a + b) + 0.5 * (b - a) * c_glx[15][node];
    double om = 0.5 * (b - a) * c_glw[15][node];
    double u = v * v;
    cplx mu{u, -k};
    cplx sq = csqrt_d(cplx{u, -2.0 * k});            // sqrt(v^2 - 2ik), 4th quadrant
    cplx s = v * sq;                                 // sqrt(u^2 - 2iku)
    cplx w = mu + s;
    cplx F = cdiv(cplx{2.0 * om, 0}, sq);
    // e^{-qH mu} = e^{-qHu} e^{iqHk}
    cplx eq = cexp_d(cplx{-q * H * u, q * H * k});
    cplx base = cdiv(F * eq, cplx{0, M_PI});         // / (i pi)
    cplx ehu = cexp_d(cplx{H * u, -H * k});         // e^{H mu}
    cplx dp = ehu * cexp_d(cplx{0, -beta}) - cplx{1, 0};
    cplx dm = ehu * cexp_d(cplx{0, beta}) - cplx{1, 0};
    cplx Ap = cdiv(cexp_d(cplx{0, q * beta}), dp);
    cplx Am = cdiv(cexp_d(cplx{0, -q * beta}), dm);
    cplx lw = clog_d(w);
    double lk = log(k);
    // (-i w / k)^n, (i k / w)^n, (i w / k)^n, (-i k / w)^n in log form
    cplx l1 = cplx{lw.re - lk, lw.im - 0.5 * M_PI};
    cplx l2 = cplx{lk - lw.re, 0.5 * M_PI - lw.im};
    cplx l3 = cplx{lw.re - lk, lw.im + 0.5 * M_PI};
    cplx l4 = cplx{lk - lw.re, -0.5 * M_PI - lw.im};
    cplx lbp = clog_d(base * Ap);
    cplx lbm = clog_d(base * Am);
    double n = (double)j;
    acc += cexp_d(n * l1 + lbp) + cexp_d(n * l2 + lbp) + cexp_d(n * l3 + lbm) + cexp_d(n * l4 + lbm);
  }
  // direct rows mlo <= |m| <= q (mlo = 2: every image beyond the adjacent ones)
  for (int m = mlo + threadIdx.x; m <= q; m += blockDim.x) {
    double x = k * m * H;
    double Jv[2 * PF_PMAX + 2];
    bessel_j_array(x, j, Jv);
    double y0v = ::y0(x), y1v = ::y1(x), Y = y0v;
    if (j >= 1) {
      double ym = y0v, yc = y1v;
      for (int n = 1; n < j; ++n) {
        double yn = (2.0 * n / x) * yc - ym;
        ym = yc;
        yc = yn;
      }
      Y = yc;
    }
    cplx Hj{Jv[j], Y};
    // i^j and (-i)^j
    cplx ij{1, 0};
    for (int r = 0; r < (j & 3); ++r) ij = mul_i(ij);
    cplx mij = conj(ij);
    // alpha^m = e^{i m beta}
    cplx am = cexp_d(cplx{0, m * beta});
    acc += Hj * (am * mij + conj(am) * ij);
  }
  red[0][threadIdx.x] = acc.re;
  red[1][threadIdx.x] = acc.im;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      red[0][threadIdx.x] += red[0][threadIdx.x + s];
      red[1][threadIdx.x] += red[1][threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) out[j] = cplx{red[0][0], red[1][0]};
}

// host: upper limit V of the v-integral where every order's integrand has
// dropped by e^-40 below its peak.
static double lattice_vmax(int jmax, int q, double k, double H) {
  double V = sqrt(40.0 / (q * H));
  for (int n = 0; n <= jmax; n += (jmax > 8 ? jmax / 8 : 1)) {
    double peak = -1e300, vpk = 0;
    // the peak of the log-integrand, on a grid of step 0.04 in v (an estimate
    // low by a little moves the cut-off below out by a little: safe)
    for (int i = 1; i < 500; ++i) {
      double v = 0.04 * i;
      double u = v * v;
      double wabs = hypot(u, k) + sqrt(hypot(u * u, 2 * k * u));
      double f = n * log(wabs / k) - q * H * u;
      if (f > peak) { peak = f; vpk = v; }
    }
    for (double v = vpk; v < 200; v *= 1.02) {
      double u = v * v;
      double wabs = hypot(u, k) + sqrt(hypot(u * u, 2 * k * u));
      double f = n * log(wabs / k) - q * H * u;
      if (f < peak - 42.0) { if (v > V) V = v; break; }
    }
  }
  return V;
}

cudaError_t k_lattice_sums(pfmbem* h, int jmax, int q, cplx* out_dev, int mlo) {
  double V = lattice_vmax(jmax, q, h->k, h->H);
  prof_begin(h, PH_SETUP);
  lattice_sum_kernel<<<jmax + 1, 256, 0, h->stream>>>(jmax, q, h->k, h->H, h->beta, V, out_dev, mlo);
  prof_end(h, PH_SETUP);
  return cudaGetLastError();
}

// ---------------------------------------------------- lattice sums, allocation-free variant
// Same kernel as above, but its device results land in a fixed array that lives
// in this library's device image instead of in memory the caller or a handle
// allocates.  Every GPU that loads the library holds the array until exit.
#define PF_NOALLOC_JMAX 128
static __device__ __align__(256) cplx g_lattice_scratch[PF_NOALLOC_JMAX + 1];
// Device address of the array per device ordinal, published with release order
// once that device's set-up is complete (null until then); the mutex makes two
// host threads that call first on one device run the set-up once.
static std::atomic<cplx*> g_lattice_scratch_dev[64];
static std::mutex g_lattice_scratch_mutex;

__global__ void symmetric_expand_kernel(const cplx* __restrict__ half, int jmax, cplx* __restrict__ full) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i <= 2 * jmax) full[i] = half[abs(i - jmax)];
}

extern "C" pfmbem_status pfmbem_lattice_sums_noalloc(double k, double H, double theta, int jmax, void* cuda_stream,
                                                     double* S) {
  if (!S || !(k > 0) || !(H > 0) || !isfinite(theta)) return PFMBEM_EINVAL;
  if (jmax < 0 || jmax > PF_NOALLOC_JMAX) return PFMBEM_EINVAL;   // beyond the fixed array
  {
    const double s = sin(theta);
    double dmin = 1e300;
    for (double v : {k * H * (1 + s), k * H * (1 - s)}) dmin = fmin(dmin, fabs(v - 2 * M_PI * round(v / (2 * M_PI))));
    if (dmin < 1e-3) return PFMBEM_EWOOD;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return PFMBEM_ECUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // A device output must live on the current device: the kernels below run there.
  cudaPointerAttributes a;
  const bool attr_ok = cudaPointerGetAttributes(&a, S) == cudaSuccess;
  cudaGetLastError();
  const bool sdev = attr_ok && (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
  if (attr_ok && a.type == cudaMemoryTypeDevice && a.device != dev) return PFMBEM_EINVAL;
  cplx* scratch = g_lattice_scratch_dev[dev].load(std::memory_order_acquire);
  if (!scratch) {
    // one-time set-up on this device: Gauss rules for the contour integral and
    // the device address of the fixed array (host code may not use its name)
    std::lock_guard<std::mutex> lock(g_lattice_scratch_mutex);
    scratch = g_lattice_scratch_dev[dev].load(std::memory_order_acquire);
    if (!scratch) {
      double x[PF_GLMAX * PF_GLMAX] = {0}, w[PF_GLMAX * PF_GLMAX] = {0};
      for (int g = 1; g <= PF_GLMAX; ++g) gauss_legendre(g, &x[(g - 1) * PF_GLMAX], &w[(g - 1) * PF_GLMAX]);
      if (cudaMemcpyToSymbol(c_glx, x, sizeof(x)) != cudaSuccess) return PFMBEM_ECUDA;
      if (cudaMemcpyToSymbol(c_glw, w, sizeof(w)) != cudaSuccess) return PFMBEM_ECUDA;
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_lattice_scratch) != cudaSuccess || !p) return PFMBEM_ECUDA;
      scratch = static_cast<cplx*>(p);
      g_lattice_scratch_dev[dev].store(scratch, std::memory_order_release);
    }
  }
  const int q = 8;
  const double beta = k * H * sin(theta);
  const double V = lattice_vmax(jmax, q, k, H);
  if (cudaMemsetAsync(scratch, 0, sizeof(cplx) * (jmax + 1), st) != cudaSuccess) return PFMBEM_ECUDA;
  lattice_sum_kernel<<<jmax + 1, 256, 0, st>>>(jmax, q, k, H, beta, V, scratch);
  if (cudaGetLastError() != cudaSuccess) return PFMBEM_ECUDA;
  if (sdev) {
    symmetric_expand_kernel<<<(2 * jmax + 1 + 127) / 128, 128, 0, st>>>(scratch, jmax, reinterpret_cast<cplx*>(S));
    if (cudaGetLastError() != cudaSuccess) return PFMBEM_ECUDA;
    return PFMBEM_OK;
  }
  cplx half[PF_NOALLOC_JMAX + 1];
  if (cudaMemcpyAsync(half, scratch, sizeof(cplx) * (jmax + 1), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return PFMBEM_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return PFMBEM_ECUDA;
  for (int j = -jmax; j <= jmax; ++j) {
    S[2 * (j + jmax)] = half[abs(j)].re;
    S[2 * (j + jmax) + 1] = half[abs(j)].im;
  }
  return PFMBEM_OK;
}

// ---------------------------------------------------------------- J0, J1, Y0, Y1
// All four at once, each within 1e-15 of the modulus sqrt(J^2 + Y^2):
// x <= 3  the ascending series of J_0, J_1 / x and of the entire parts of Y_0 and
//         Y_1 / x in x^2 (Abramowitz & Stegun 9.1.10, 9.1.11, 9.1.13: Y_0 = (2/pi)
//         ln(x/2) J_0 + entire, Y_1 = (2/pi) ln(x/2) J_1 - 2/(pi x) + entire);
// x <= 8  Chebyshev interpolants of the same functions on 4 <= x^2 <= 68, in
//         powers of s = (x^2 - 36) / 32 (a mapping without rounding: the errors
//         of neighbouring elements then do not add up);
// x > 8   H_n = sqrt(2/(pi x)) (P_n + i Q_n / x) e^{i(x - n pi/2 - pi/4)} with the
//         interpolants of P_n and Q_n in s = 2 (8/x)^2 - 1.
// The interpolants were sampled with 50 digits.  The element integrals, most of a
// block's set-up and the field sums, are bound by the FP64 pipe (one warp
// instruction per 16 cycles and SM), so the number of FP64 instructions is their
// time: about 100 in each range.  The forms before took up to 27 terms of six
// (series, x <= 4) or CUDA's four functions, each with its own amplitude, phase
// and sine.  A create of the 24-fiber round-square crystal (512 x 512 blocks) took
// 7.2 instead of 9.6 ms with them.
__constant__ double c_bes_lo[4][15] = {
    {1.0, -0.25, 0.015625, -0.00043402777777777775, 6.781684027777777e-06, -6.781684027777778e-08,
     4.709502797067901e-10, -2.4028075495244395e-12, 9.385966990329842e-15, -2.896903392077112e-17,
     7.242258480192779e-20, -1.4963343967340453e-22, 2.5978027721077174e-25, -3.842903509035085e-28,
     4.9016626390753635e-31},
    {0.5, -0.0625, 0.0026041666666666665, -5.425347222222222e-05, 6.781684027777778e-07, -5.651403356481481e-09,
     3.363930569334215e-11, -1.5017547184527747e-13, 5.214426105738801e-16, -1.4484516960385557e-18,
     3.2919356728148996e-21, -6.234726653058522e-24, 9.991549123491221e-27, -1.3724655389411017e-29,
     1.6338875463584545e-32},
    {0.36746690519661596, 0.06728821679274134, -0.009179105521168063, 0.00034707870839581153, -6.502443354192743e-06,
     7.365914182599293e-08, -5.614911948799596e-10, 3.083275965031416e-12, -1.2790958259508146e-14,
     4.1527406208644286e-17, -1.0842908046669823e-19, 2.326869899670465e-22, -4.177522404380815e-25,
     6.367956744012936e-28, -8.345286331389722e-31},
    {0.024578509506412646, 0.026769238141428797, -0.0018061615852847733, 4.77021926915092e-05,
     -6.934178768396019e-07, 6.43807807869613e-09, -4.1636188715218474e-11, 1.9868003998329693e-13,
     -7.290510519752471e-16, 2.1224759598830894e-18, -5.0238541729715624e-21, 9.860672509570446e-24,
     -1.6312040698718383e-26, 2.305475219254014e-29, -2.8164342810578055e-32}};
__constant__ double c_bes_mid[4][18] = {
    {0.15064525725099692, 0.7378236216735082, -0.8635491909695483, -0.36272477177924045, 0.7535493684273741,
     -0.40688852091573613, 0.1227797948288713, -0.02465533220134352, 0.003585284432299863, -0.00039772279081992586,
     3.48964997321362e-05, -2.4878193679695065e-06, 1.471659663747625e-07, -7.34668883355121e-09,
     3.138569904238356e-10, -1.1610145099432411e-11, 3.7686127751646765e-13, -1.0751696350115894e-14},
    {-0.046113976354594265, 0.10794364887119354, 0.06801089470860758, -0.18838734210684352, 0.12715266278616752,
     -0.04604242306082677, 0.01078670783808779, -0.0017926422161496942, 0.00022371906983621186,
     -2.181031233344214e-05, 1.7103758154708207e-06, -1.1037447303587369e-07, 5.96918468771569e-09,
     -2.746268803110627e-10, 1.088450413709229e-11, -3.7563388539058014e-13, 1.142551567215672e-14,
     -3.068480314718871e-16},
    {-0.39355572157911856, -0.0919622276302254, 1.231419952971538, -0.4578484462337575, -0.3731829868697732,
     0.3428807844534468, -0.12715227640166488, 0.028898442425832806, -0.004586237521220281, 0.0005440982503465963,
     -5.040270987700256e-05, 3.7602179232539514e-06, -2.3126562508795542e-07, 1.1944392479749037e-08,
     -5.258845422628135e-10, 1.998606892001458e-11, -6.648898528715865e-13, 1.9396153891496335e-14},
    {0.020767528754338974, -0.18032609331465363, 0.12458290765677417, 0.06527784099599758, -0.09557111859474952,
     0.04458491554123203, -0.01206123593726682, 0.00221193620518041, -0.00029729474319291355, 3.074784557724527e-05,
     -2.532168227724288e-06, 1.70348770486391e-07, -9.551333319901538e-09, 4.536390295374432e-10,
     -1.8497265031831036e-11, 6.549098430060115e-13, -2.03917336866426e-14, 5.594327278751556e-16}};
__constant__ double c_bes_hi[4][15] = {
    {0.9994572757882519, -0.0005363673192130047, 6.137416080163085e-06, -2.0527448156307146e-07,
     1.2803760583405539e-08, -1.2121182069774233e-09, 1.5501079933860844e-10, -2.4882702786880542e-11,
     4.772297614846628e-12, -1.0636861151667625e-12, 2.668750992381705e-13, -6.416781008015415e-14,
     1.7716435634547776e-14, -1.180002783020184e-14, 4.479453416045804e-15},
    {-0.12444091103610815, 0.0005466519279475266, -1.1817110661200976e-05, 5.684971881753781e-07,
     -4.534972837363434e-08, 5.146231602705606e-09, -7.5763304988972e-10, 1.3623497617833053e-10,
     -2.8707211071105146e-11, 6.951785915752245e-12, -1.873640743543296e-12, 4.605060470396763e-13,
     -1.3137515498826537e-13, 1.0185094098694355e-13, -4.0574096424030336e-14},
    {1.0009070262780821, 0.0008988049416705579, -7.95969469849487e-06, 2.4536766222672443e-07,
     -1.4708512086159542e-08, 1.3603058049468316e-09, -1.7131617922370612e-10, 2.720406848040165e-11,
     -5.1756417352379415e-12, 1.1462229852806783e-12, -2.861148018572335e-13, 6.864486664846182e-14,
     -1.8904930097426227e-14, 1.2489929194563941e-14, -4.728767819765722e-15},
    {0.3742149922195918, -0.0007697167057643706, 1.4569614809851411e-05, -6.633568561050814e-07,
     5.136105997071193e-08, -5.720890888840857e-09, 8.316077350038262e-10, -1.4816588916791194e-10,
     3.100364837230575e-11, -7.465104477698295e-12, 2.002728774766585e-12, -4.91574062967655e-13,
     1.3996264453471973e-13, -1.0759215471978615e-13, 4.275621822194818e-14}};

template <int DEG, int N>
__device__ __forceinline__ double poly(const double (&c)[N], double s) {
  double a = c[DEG];
#pragma unroll
  for (int i = DEG - 1; i >= 0; --i) a = fma(a, s, c[i]);
  return a;
}

__device__ __forceinline__ void bessel01(double x, double& J0, double& J1, double& Y0, double& Y1) {
  constexpr double TPI = 0.63661977236758134308, TPI_LO = -3.935735335036497e-17;   // 2/pi
  if (x <= 8.0) {
    const double t = x * x;
    double b1, e0, e1;
    if (x <= 3.0) {
      J0 = poly<14>(c_bes_lo[0], t);
      b1 = poly<13>(c_bes_lo[1], t);
      e0 = poly<14>(c_bes_lo[2], t);
      e1 = poly<13>(c_bes_lo[3], t);
    } else {
      const double s = (t - 36.0) * 0.03125;
      J0 = poly<17>(c_bes_mid[0], s);
      b1 = poly<16>(c_bes_mid[1], s);
      e0 = poly<17>(c_bes_mid[2], s);
      e1 = poly<16>(c_bes_mid[3], s);
    }
    const double lg = log(0.5 * x), L = fma(TPI_LO, lg, TPI * lg);
    J1 = x * b1;
    Y0 = fma(L, J0, e0);
    Y1 = fma(x, e1, fma(L, J1, -TPI / x));
    return;
  }
  const double ix = 1.0 / x, s = fma(ix * ix, 128.0, -1.0);
  const double P0 = poly<14>(c_bes_hi[0], s), Q0 = ix * poly<14>(c_bes_hi[1], s);
  const double P1 = poly<14>(c_bes_hi[2], s), Q1 = ix * poly<14>(c_bes_hi[3], s);
  double sn, cs;
  sincos(x, &sn, &cs);
  const double a = 0.56418958354775628695 * sqrt(ix);       // sqrt(2/(pi x)) / sqrt 2
  const double c = a * (cs + sn), d = a * (sn - cs);        // e^{i(x - pi/4)} scaled
  J0 = P0 * c - Q0 * d;
  Y0 = P0 * d + Q0 * c;
  J1 = P1 * d + Q1 * c;
  Y1 = Q1 * d - P1 * c;
}

// The same four by the ascending series with psi(m+1) = H_m - gamma to x = 4 and CUDA's
// functions above, for the scattered field itself: where a density radiates almost
// nothing u cancels to 1e-8 of its terms, and another rounding of these functions shows
// at 1e-8 of u (the joint interpolants take half the time).  Per-term constants of the
// series, m = 1..39: 1/m^2, 1/(m(m+1)), H_m and 2 H_m + 1/(m+1) - 2 gamma, a term's four
// together: as four arrays beside the interpolants' tables they cost field maps of few
// points 3 to 5 % (one warp an SM sub-partition, and its constant loads in the chain).
struct alignas(16) SerTerm {
  double im2, imm1, H, y1;
};
__constant__ SerTerm c_ser[40];

void k_upload_series() {
  SerTerm t[40] = {};
  const double EG = 0.57721566490153286061;
  double Hm = 0.0;
  for (int m = 1; m < 40; ++m) {
    Hm += 1.0 / m;
    t[m] = SerTerm{1.0 / ((double)m * m), 1.0 / ((double)m * (m + 1)), Hm, 2.0 * Hm + 1.0 / (m + 1) - 2.0 * EG};
  }
  cudaMemcpyToSymbol(c_ser, t, sizeof(t));
}

__device__ __forceinline__ void bessel01_series(double x, double& J0, double& J1, double& Y0, double& Y1) {
  if (x > 4.0) {
    J0 = j0(x); J1 = j1(x); Y0 = y0(x); Y1 = y1(x);
    return;
  }
  const double h = 0.5 * x, h2 = h * h;
  const double EG = 0.57721566490153286061;
  // a_m = (-1)^m (x/2)^{2m} / (m!)^2,  b_m = (-1)^m (x/2)^{2m} / (m! (m+1)!)
  double a = 1.0, b = 1.0;
  double sJ0 = 1.0, sJ1 = 1.0, sY0 = 0.0, sY1 = -(2.0 * (-EG) + 1.0);  // m = 0 terms
  // Y1 series term: (psi(m+1) + psi(m+2)) b_m with psi(m+1) = H_m - gamma
  // the number of terms for |term| < 1e-17 grows with x; bound it from x
  const int mmax = x < 0.5 ? 10 : (x < 1.5 ? 15 : (x < 3.0 ? 21 : 27));
#pragma unroll 1
  for (int m = 1; m < mmax; ++m) {
    const SerTerm t = c_ser[m];
    a *= -h2 * t.im2;
    b *= -h2 * t.imm1;
    sJ0 += a;
    sJ1 += b;
    sY0 = fma(-t.H, a, sY0);           // (-1)^{m+1} H_m (x/2)^{2m}/(m!)^2
    sY1 = fma(-t.y1, b, sY1);
  }
  const double L = log(h);
  J0 = sJ0;
  J1 = h * sJ1;
  Y0 = (2.0 / M_PI) * ((L + EG) * J0 + sY0);
  // Y1 = -2/(pi x) + (2/pi) ln(x/2) J1 - (1/pi) sum (psi(m+1) + psi(m+2)) b_m (x/2)
  Y1 = -2.0 / (M_PI * x) + (2.0 / M_PI) * L * J1 + (1.0 / M_PI) * h * sY1;
}

// ---------------------------------------------------------------- pair integrals
// Element integrals of (i/4)H0(kap|x-y|) (S), its d/dnu_y (D), d/dnu_x (K) and
// d2/dnu_x dnu_y (T) over the flat element c + s t, |s| <= h/2, by g-point
// Gauss-Legendre; the factor i/4 is applied by the caller.  Nodes q0, q0 + qs,
// ... only (a share of the rule, for callers that split it over lanes); SER: the Bessel
// functions by bessel01_series.
template <bool SER = false>
__device__ __forceinline__ void pair4_f64(double kap, double2 x, double2 nx, double2 c, double2 t, double2 ny,
                                          double h, int g, cplx& S, cplx& D, cplx& K, cplx& T, int q0 = 0,
                                          int qs = 1) {
  const double nn = nx.x * ny.x + nx.y * ny.y;
#pragma unroll 1
  for (int q = q0; q < g; q += qs) {
    double s = 0.5 * h * c_glx[g - 1][q];
    double wq = 0.5 * h * c_glw[g - 1][q];
    double z1 = x.x - (c.x + s * t.x);
    double z2 = x.y - (c.y + s * t.y);
    double r = sqrt(z1 * z1 + z2 * z2);
    double ir = 1.0 / r;
    double kr = kap * r;
    double J0, J1, Y0, Y1;
    if (SER) bessel01_series(kr, J0, J1, Y0, Y1);
    else bessel01(kr, J0, J1, Y0, Y1);
    double zy = (z1 * ny.x + z2 * ny.y) * ir;
    double zx = (z1 * nx.x + z2 * nx.y) * ir;
    S += wq * cplx{J0, Y0};
    D += (wq * kap * zy) * cplx{J1, Y1};
    K += (-wq * kap * zx) * cplx{J1, Y1};
    double a = kap * zx * zy;
    double b = ir * (nn - 2.0 * zx * zy);
    T += (wq * kap) * cplx{a * J0 + b * J1, a * Y0 + b * Y1};
  }
}

// A near-field block from S, D, K, T (without i/4) at the matrix wavenumber:
// (i/4) {D, -i eta S, T, -i eta K} = {(i/4) D, (eta/4) S, (i/4) T, (eta/4) K},
// the form in which the tables keep them (FP64 and FP32).
__device__ __forceinline__ void near_block_form(double eta, cplx S, cplx D, cplx K, cplx T, cplx* o, cplxf* of,
                                                cplxf* ol) {
  const double e4 = 0.25 * eta;
  const cplx b[4] = {cplx{-0.25 * D.im, 0.25 * D.re}, cplx{e4 * S.re, e4 * S.im}, cplx{-0.25 * T.im, 0.25 * T.re},
                     cplx{e4 * K.re, e4 * K.im}};
  for (int q = 0; q < 4; ++q) {
    o[q] = b[q];
    of[q] = cplxf{(float)b[q].re, (float)b[q].im};
    ol[q] = split_lo(b[q]);
  }
}

// ---------------------------------------------------------------- permute
__global__ void gather_dens_kernel(int E, const int* __restrict__ perm, const cplx* __restrict__ ph,
                                   const cplx* __restrict__ x, cplx* __restrict__ dens) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= E) return;
  int e = perm[s];
  cplx p = ph[s];
  dens[2 * s] = p * x[2 * e];
  dens[2 * s + 1] = p * x[2 * e + 1];
}

// ---------------------------------------------------------------- P2M (FP64)
// M_n(O_C) = sum_elements sum_g w_g h/2 [phi' dJ^-_n/dnu_y - i eta varphi' J^-_n](k(y_g - O_C)),
// J^-_n(v) = J_n(|v|) e^{-i n theta_v}, dJ^-_n/dnu = (k/2)(-nu J^-_{n+1} + conj(nu) J^-_{n-1})
// with nu = nu_x + i nu_y (Sec. 3.2, the moments of S2b and D2b); stored scaled by 1/w_n.
__global__ void p2m_f64_kernel(const int* __restrict__ ne, const int* __restrict__ bb, const int* __restrict__ be,
                               int D, double d, int p, const double* __restrict__ wgt, int g,
                               double k, double eta, double x0, double y0,
                               const double2* __restrict__ sc, const double2* __restrict__ st,
                               const double2* __restrict__ snu, const double* __restrict__ sh,
                               const cplx* __restrict__ dens, cplx* __restrict__ Mout,
                               const double2* __restrict__ ctr, bool turn) {
  const int box = ne[blockIdx.x];
  const int P = 2 * p + 1;
  const size_t row = wgt ? box : blockIdx.x;      // no weights: unscaled, a row per listed box
  __shared__ double acc[2 * PF_NCOEF];
  for (int i = threadIdx.x; i < 2 * P; i += blockDim.x) acc[i] = 0.0;
  __syncthreads();
  // box centre: given (triangle tree), else from the Morton code
  int ix = (box >> (2 * D)) << D, iy = 0;       // root squares in a row along x, root-major
  for (int b = 0; b < D; ++b) {
    ix |= ((box >> (2 * b)) & 1) << b;
    iy |= ((box >> (2 * b + 1)) & 1) << b;
  }
  const double ox = ctr ? ctr[box].x : x0 + (ix + 0.5) * d, oy = ctr ? ctr[box].y : y0 + (iy + 0.5) * d;
  const int lb = bb[box], le = be[box];
  const int npts = (le - lb) * g;
  for (int t = threadIdx.x; t < npts; t += blockDim.x) {
    int f = lb + t / g, q = t % g;
    double2 c = sc[f], tt = st[f], nu = snu[f];
    double hh = sh[f];
    double s = 0.5 * hh * c_glx[g - 1][q];
    double cw = 0.5 * hh * c_glw[g - 1][q];
    double vx = c.x + s * tt.x - ox, vy = c.y + s * tt.y - oy;
    double r = sqrt(vx * vx + vy * vy);
    cplx z = r > 0 ? cplx{vx / r, -vy / r} : cplx{1, 0};   // e^{-i theta}
    double J[PF_PMAX + 2];
    bessel_j_array(k * r, p + 1, J);
    cplx Jm[2 * PF_PMAX + 3];                               // J^-_n, n = -p-1..p+1
    cplx zp{1, 0};
    for (int n = 0; n <= p + 1; ++n) {
      Jm[p + 1 + n] = J[n] * zp;
      double sg = (n & 1) ? -1.0 : 1.0;
      Jm[p + 1 - n] = (sg * J[n]) * conj(zp);
      zp = zp * z;
    }
    cplx ph = dens[2 * f], va = dens[2 * f + 1];
    cplx a = (cw * 0.5 * k) * ph;
    cplx bcoef = (-eta * cw) * mul_i(va);
    cplx nuc{nu.x, nu.y};
    // turn: every thread begins at another coefficient, for in step they all add to one word
    // (887 -> 346 us a launch on 16384 elements)
    for (int i = 0, j = turn ? threadIdx.x % P : 0; i < P; ++i, j = j + 1 < P ? j + 1 : 0) {
      cplx v = a * (conj(nuc) * Jm[j] - nuc * Jm[j + 2]) + bcoef * Jm[j + 1];
      double iw = wgt ? 1.0 / wgt[j] : 1.0;
      atomicAdd(&acc[2 * j], v.re * iw);
      atomicAdd(&acc[2 * j + 1], v.im * iw);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < P; i += blockDim.x) Mout[row * P + i] = cplx{acc[2 * i], acc[2 * i + 1]};
}

// ---------------------------------------------------------------- M2M (FP64)
// M(parent) = sum_children A_q M(child), A_q[n][m] = J^-_{n-m}(k(O_child - O_parent)) w^c_m / w^p_n.
// Children nch box + q, q < nch; the child's operator is q, or aidx[child] where
// the children's offsets vary (triangle tree).  SPLIT groups of 64 threads
// share the children's coefficients: one thread's chain of 4 Pc operator loads
// is the kernel's time (the block has little else to overlap it with).  Four of
// them, M2M_SPLIT, but for the field u, whose sums keep one order (upward_f64).
constexpr int M2M_SPLIT = 4;
template <int SPLIT>
__global__ void __launch_bounds__(64 * SPLIT) m2m_f64_kernel(
    const int* __restrict__ ne, int P, int Pc, const cplx* __restrict__ A, const int* __restrict__ cbb,
    const int* __restrict__ cbe, const cplx* __restrict__ Mc, cplx* __restrict__ Mp, int nch,
    const int* __restrict__ aidx) {
  const int box = ne[blockIdx.x];
  __shared__ cplx sm[6 * PF_NCOEF], red[SPLIT][64];
  for (int i = threadIdx.x; i < nch * Pc; i += blockDim.x) sm[i] = Mc[(size_t)nch * box * Pc + i];
  __syncthreads();
  const int part = threadIdx.x >> 6, lane = threadIdx.x & 63;
  for (int n0 = 0; n0 < P; n0 += 64) {
    const int n = n0 + lane;
    cplx acc{0, 0};
    for (int q = 0; n < P && q < nch; ++q) {
      const int ch = nch * box + q;
      if (cbb[ch] >= cbe[ch]) continue;   // empty child (uniform across the block)
      const int op = aidx ? aidx[ch] : q;
      const cplx* col = A + (size_t)op * Pc * P + n;              // transposed [op][m][n]
      const cplx* mc = sm + q * Pc;
#pragma unroll 4
      for (int m = part; m < Pc; m += SPLIT) acc += col[(size_t)m * P] * mc[m];
    }
    if (SPLIT == 1) {
      if (n < P) Mp[(size_t)box * P + n] = acc;
      continue;
    }
    red[part][lane] = acc;
    __syncthreads();
    if (part == 0 && n < P) {
      for (int i = 1; i < SPLIT; ++i) acc += red[i][lane];
      Mp[(size_t)box * P + n] = acc;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------- L2L + M2L (FP64)
// L(box) = B_q L(parent) + sum_{(C, o, m) in IL(box)} alpha^m T_o M(C)
// (Sec. 3.2: M2L with the Toeplitz H^+_{n-l} operators shared by all boxes at
// the same offset o, and L2L with J^+_{l-n}); at the root, L = R M(root) with
// the lattice-sum operator R (Sec. 3.3).
__global__ void local_f64_kernel(const int* __restrict__ ne, int D_unused, int P, int Pp,
                                 const cplx* __restrict__ B, const cplx* __restrict__ Lp,
                                 const int* __restrict__ ilp, const int* __restrict__ ils,
                                 const int* __restrict__ ilo, const int* __restrict__ ilm,
                                 const cplx* __restrict__ T, const cplx* __restrict__ Mlev,
                                 const cplx* __restrict__ root, cplx alpha, cplx* __restrict__ Lout,
                                 int nchp, const int* __restrict__ pidx) {
  const int ti = blockIdx.x;
  const int box = ne[ti];
  __shared__ cplx sm[PF_NCOEF];
  cplx acc{0, 0};
  const int l = threadIdx.x;
  if (root) {   // level 0
    for (int i = threadIdx.x; i < P; i += blockDim.x) sm[i] = Mlev[i];
    __syncthreads();
    if (l < P)
      for (int n = 0; n < P; ++n) acc += root[(size_t)l * P + n] * sm[n];
    if (l < P) Lout[l] = acc;
    return;
  }
  // L2L from the parent (nchp children per parent; the box's operator q, or
  // pidx[box] where the children's offsets vary)
  {
    int par = box / nchp, q = pidx ? pidx[box] : box % nchp;
    for (int i = threadIdx.x; i < Pp; i += blockDim.x) sm[i] = Lp[(size_t)par * Pp + i];
    __syncthreads();
    if (l < P) {
      const cplx* col = B + (size_t)q * Pp * P + l;               // transposed [q][m][n]
      for (int m = 0; m < Pp; ++m) acc += col[(size_t)m * P] * sm[m];
    }
  }
  // M2L (none without lists: the caller adds it by offset groups)
  for (int e = ilp ? ilp[ti] : 0; ilp && e < ilp[ti + 1]; ++e) {
    int src = ils[e], off = ilo[e];
    cplx ph = ipow_phase(alpha, ilm[e]);
    __syncthreads();
    for (int i = threadIdx.x; i < P; i += blockDim.x) sm[i] = ph * Mlev[(size_t)src * P + i];
    __syncthreads();
    if (l < P) {
      const cplx* row = T + ((size_t)off * P + l) * P;
      for (int n = 0; n < P; ++n) acc += row[n] * sm[n];
    }
  }
  if (l < P) Lout[(size_t)box * P + l] = acc;
}

// ---------------------------------------------------------------- L2P (FP64)
// U'(x) = (i/4) sum_l L_l J^+_l(k(x - O_D)),
// dU'(x) = (i/4)(k/2) sum_l L_l (-conj(nu) J^+_{l+1} + nu J^+_{l-1}).
__global__ void l2p_f64_kernel(const int* __restrict__ ne, const int* __restrict__ bb, const int* __restrict__ be,
                               int D, double d, int p, const double* __restrict__ wgt, double k,
                               double x0, double y0, const double2* __restrict__ sc, const double2* __restrict__ snu,
                               const cplx* __restrict__ L, cplx* __restrict__ U, const double2* __restrict__ ctr) {
  const int box = ne[blockIdx.x];
  const int P = 2 * p + 1;
  __shared__ cplx sl[PF_NCOEF];
  for (int i = threadIdx.x; i < P; i += blockDim.x) sl[i] = (1.0 / wgt[i]) * L[(size_t)box * P + i];
  __syncthreads();
  int ix = (box >> (2 * D)) << D, iy = 0;       // root squares in a row along x, root-major
  for (int b = 0; b < D; ++b) {
    ix |= ((box >> (2 * b)) & 1) << b;
    iy |= ((box >> (2 * b + 1)) & 1) << b;
  }
  const double ox = ctr ? ctr[box].x : x0 + (ix + 0.5) * d, oy = ctr ? ctr[box].y : y0 + (iy + 0.5) * d;
  for (int s = bb[box] + threadIdx.x; s < be[box]; s += blockDim.x) {
    double2 c = sc[s], nu = snu[s];
    double vx = c.x - ox, vy = c.y - oy;
    double r = sqrt(vx * vx + vy * vy);
    cplx z = r > 0 ? cplx{vx / r, vy / r} : cplx{1, 0};    // e^{+i theta}
    double J[PF_PMAX + 2];
    bessel_j_array(k * r, p + 1, J);
    cplx nuc{nu.x, nu.y};
    cplx u{0, 0}, du{0, 0};
    // J^+_l = J_l z^l (l >= 0), J^+_{-l} = (-1)^l J_l conj(z)^l
    cplx zp{1, 0};
    for (int l = 0; l <= p + 1; ++l) {
      cplx jp = J[l] * zp;                                 // J^+_l
      cplx jn = ((l & 1) ? -J[l] : J[l]) * conj(zp);       // J^+_{-l}
      if (l <= p) {
        u += sl[p + l] * jp;
        if (l > 0) u += sl[p - l] * jn;
      }
      // coefficient L_m contributes -conj(nu) J^+_{m+1} + nu J^+_{m-1}
      //   J^+_l appears as J^+_{m+1} for m = l - 1 and as J^+_{m-1} for m = l + 1
      if (l - 1 >= -p && l - 1 <= p) du -= conj(nuc) * (sl[p + l - 1] * jp);
      if (l + 1 <= p) du += nuc * (sl[p + l + 1] * jp);
      if (l > 0) {
        // J^+_{-l}: as J^+_{m+1} for m = -l - 1, as J^+_{m-1} for m = -l + 1
        if (-l - 1 >= -p) du -= conj(nuc) * (sl[p - l - 1] * jn);
        if (-l + 1 <= p) du += nuc * (sl[p - l + 1] * jn);
      }
      zp = zp * z;
    }
    U[2 * s] = mul_i(0.25 * u);
    U[2 * s + 1] = mul_i((0.125 * k) * du);
  }
}

// ---------------------------------------------------------------- near field (FP64)
// Direct element integrals over the <= 9 neighbouring leaves (with their
// periodic images m = -1, 0, 1 and phases alpha^m); the self element is skipped
// (its integrals are added in the combine step).  One warp per target.
__global__ void near_f64_kernel(const int* __restrict__ ne, const int* __restrict__ bb, const int* __restrict__ be,
                                const int* __restrict__ nlp, const int* __restrict__ nls, const int* __restrict__ nlm,
                                double k, double eta, double H, cplx alpha,
                                const double2* __restrict__ sc, const double2* __restrict__ st,
                                const double2* __restrict__ snu, const double* __restrict__ sh,
                                const cplx* __restrict__ dens, cplx* __restrict__ U) {
  const int li = blockIdx.x;
  const int box = ne[li];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int s = bb[box] + warp; s < be[box]; s += nw) {
    double2 x = sc[s], nx = snu[s];
    cplx u{0, 0}, du{0, 0};
    for (int e = nlp[li]; e < nlp[li + 1]; ++e) {
      int src = nls[e], m = nlm[e];
      cplx ph = ipow_phase(alpha, m);
      double shift = m * H;
      cplx uu{0, 0}, dd{0, 0};
      for (int f = bb[src] + lane; f < be[src]; f += 32) {
        if (f == s && m == 0) continue;
        double2 c = sc[f];
        c.y += shift;
        double hh = sh[f];
        double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / hh;
        int g = gl_order(q, 0);
        cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
        pair4_f64(k, x, nx, c, st[f], snu[f], hh, g, S, Dv, K, T);
        cplx phi = dens[2 * f], vphi = dens[2 * f + 1];
        // (i/4)(D phi - i eta S varphi), (i/4)(T phi - i eta K varphi)
        uu += Dv * phi - eta * mul_i(S * vphi);
        dd += T * phi - eta * mul_i(K * vphi);
      }
      u += ph * uu;
      du += ph * dd;
    }
    u = warp_sum(u);
    du = warp_sum(du);
    if (lane == 0) {
      U[2 * s] += mul_i(0.25 * u);
      U[2 * s + 1] += mul_i(0.25 * du);
    }
  }
}

// ------------------------------------------------- fiber-local k1 + combine (FP64)
// V, dV over the target's own fiber (free-space k1 kernel, eq. 5), then eq. 9.
__global__ void fiber_combine_f64_kernel(int E, const int* __restrict__ fib, const int* __restrict__ foff,
                                         double k1, double eta, double rho, cplx c2,
                                         const double2* __restrict__ oc, const double2* __restrict__ ot,
                                         const double2* __restrict__ onu, const double* __restrict__ oh,
                                         const int* __restrict__ opos, const cplx* __restrict__ sph,
                                         const cplx* __restrict__ self4, const cplx* __restrict__ x,
                                         const cplx* __restrict__ U, cplx* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (e >= E) return;
  const int fb = fib[e];
  const double2 xe = oc[e], nxe = onu[e];
  cplx v{0, 0}, dv{0, 0};
  for (int f = foff[fb] + lane; f < foff[fb + 1]; f += 32) {
    if (f == e) continue;
    double2 c = oc[f];
    double hh = oh[f];
    double q = sqrt((xe.x - c.x) * (xe.x - c.x) + (xe.y - c.y) * (xe.y - c.y)) / hh;
    int g = gl_order(q, 0);
    cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
    pair4_f64(k1, xe, nxe, c, ot[f], onu[f], hh, g, S, Dv, K, T);
    cplx phi = x[2 * f], vphi = x[2 * f + 1];
    v += Dv * phi - eta * mul_i(S * vphi);
    dv += T * phi - eta * mul_i(K * vphi);
  }
  v = warp_sum(v);
  dv = warp_sum(dv);
  if (lane == 0) {
    v = mul_i(0.25 * v);
    dv = mul_i(0.25 * dv);
    const cplx phi = x[2 * e], vphi = x[2 * e + 1];
    const int s = opos[e];
    const cplx po = cdiv(cplx{1, 0}, sph[s]);   // alpha^{m0}
    cplx u = po * U[2 * s], du = po * U[2 * s + 1];
    const cplx Sk = self4[4 * e], Tk = self4[4 * e + 1], Sk1 = self4[4 * e + 2], Tk1 = self4[4 * e + 3];
    u += -eta * mul_i(Sk * vphi);
    du += Tk * phi;
    v += -eta * mul_i(Sk1 * vphi);
    dv += Tk1 * phi;
    y[2 * e] = phi - v + u;
    y[2 * e + 1] = vphi + c2 * (du - rho * dv);
  }
}

// ------------------------------------------------------------ cached near field
// Build: for leaf li with targets s in [bb, be) and the concatenated source list
// (f, m) of its neighbour leaves, block (t, j) holds (i/4) alpha^m times
// {D, -i eta S, T, -i eta K} of source f at target s (zero for f = s, m = 0).
// Two launches: near_build_kernel fills every block read from a table (k table
// of a regular polygon, fiber-pair table) and queues the rest, which
// near_direct_kernel integrates one pair per thread, so that the Gauss ladder's
// cost is spread evenly over the GPU instead of over one leaf's warps.
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Integrals shared by translated copies of a fiber pair: table t holds S, D, K,
// T (without i/4) at the matrix wavenumber of every element a of fiber A_t
// against every element b of fiber B_t shifted by m_t periods, for the pair
// (A_t, B_t, m_t) that represents the class (true coordinates).  Every fiber
// pair in the class is a rigid translate of it.  One thread per entry.
__global__ void pair_table_kernel(int ntab, const int* __restrict__ tA, const int* __restrict__ tB,
                                  const int* __restrict__ tm, const int64_t* __restrict__ tbase,
                                  const int64_t* __restrict__ tstart, const int* __restrict__ foff, double k,
                                  double H, const double2* __restrict__ oc, const double2* __restrict__ ot,
                                  const double2* __restrict__ onu, const double* __restrict__ oh, double eta,
                                  cplx* __restrict__ tval, cplxf* __restrict__ tvalf, cplxf* __restrict__ tvall,
                                  unsigned long long* __restrict__ stat) {
  const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long np = 0, nq = 0;
  if (gi < tstart[ntab]) {
    int lo = 0, hi = ntab - 1;                       // table of entry gi
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (tstart[mid] <= gi) lo = mid; else hi = mid - 1;
    }
    const int t = lo;
    const int A = tA[t], B = tB[t];
    const int nb = foff[B + 1] - foff[B];
    const int64_t local = gi - tstart[t];
    const int a = (int)(local / nb), b = (int)(local % nb);
    const int e = foff[A] + a, f = foff[B] + b;
    const double2 x = oc[e], nx = onu[e];
    double2 c = oc[f];
    c.y += tm[t] * H;
    const double hh = oh[f];
    const double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / hh;
    const int g = gl_order(q, 0);
    cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
    pair4_f64(k, x, nx, c, ot[f], onu[f], hh, g, S, Dv, K, T);
    near_block_form(eta, S, Dv, K, T, tval + 4 * (tbase[t] + local), tvalf + 4 * (tbase[t] + local),
                    tvall + 4 * (tbase[t] + local));
    np = 1;
    nq = g;
  }
  if (stat) {
    np = warp_sum_u64(np);
    nq = warp_sum_u64(nq);
    if ((threadIdx.x & 31) == 0 && np) {
      atomicAdd(&stat[0], np);
      atomicAdd(&stat[1], nq);
    }
  }
}

// Table lookup of one near pair (target fiber fs, source fiber ff, true image
// shift mt): -2 = the k table of fs (same fiber, same image, regular polygon),
// >= 0 = a fiber-pair table, -1 = none (integrate).
__device__ __forceinline__ int near_lookup(int fs, int ff, int mt, int64_t kb, const int* __restrict__ pl_ptr,
                                           const int* __restrict__ pl_fib, const int* __restrict__ pl_img,
                                           const int* __restrict__ pl_tab) {
  if (ff == fs && mt == 0) return kb >= 0 ? -2 : -1;
  if (pl_ptr)
    for (int q = pl_ptr[fs]; q < pl_ptr[fs + 1]; ++q)
      if (pl_fib[q] == ff && pl_img[q] == mt) return pl_tab[q];
  return -1;
}

constexpr int NB_RUNS = 8;       // target runs per leaf whose lookups are shared through shared memory

// Phase 1 of the near-field build, one block per leaf.  The leaf's sources and
// targets are described once in shared memory, and the table of every
// (target run, source) pair is looked up once: a run is a stretch of targets of
// one fiber and one wrap shift m0 (the sort by leaf key is stable and the
// input is fiber-major, so a leaf holds few).  Then every block (t, j) that a
// table covers is copied and scaled by (i/4) alpha^m; the others are queued for
// near_direct_kernel.
__global__ void near_build_kernel(const int* __restrict__ ne, const int* __restrict__ bb, const int* __restrict__ be,
                                  const int64_t* __restrict__ base, const int* __restrict__ sbase,
                                  const int* __restrict__ srcf, const int* __restrict__ srcm, double eta, cplx alpha,
                                  const int* __restrict__ perm, const int* __restrict__ ofib,
                                  const int* __restrict__ foff, const int* __restrict__ sm0,
                                  const int64_t* __restrict__ kbase, const cplx* __restrict__ kval,
                                  const cplxf* __restrict__ kvalf, const cplxf* __restrict__ kvall,
                                  const int* __restrict__ pl_ptr, const int* __restrict__ pl_fib,
                                  const int* __restrict__ pl_img, const int* __restrict__ pl_tab,
                                  const int64_t* __restrict__ tab_base, const int* __restrict__ tab_nb,
                                  const cplx* __restrict__ tab_val, const cplxf* __restrict__ tab_valf,
                                  const cplxf* __restrict__ tab_vall, cplx* __restrict__ val,
                                  cplxf* __restrict__ valf, cplxf* __restrict__ vall,
                                  unsigned long long* __restrict__ queue, unsigned* __restrict__ qlen,
                                  unsigned qcap) {
  extern __shared__ int nbs[];
  const int li = blockIdx.x;
  const int box = ne[li];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int s0 = bb[box], nt = be[box] - s0;
  const int j0 = sbase[li], ns = sbase[li + 1] - j0;
  int* s_f = nbs;                    // [ns] source element (sorted)
  int* s_ef = s_f + ns;              // [ns] its original index
  int* s_ff = s_ef + ns;             // [ns] its fiber
  int* s_dm = s_ff + ns;             // [ns] image m minus the source's wrap shift m0
  int* s_m = s_dm + ns;              // [ns] image m
  int* t_run = s_m + ns;             // [nt] run of the target (-1: beyond NB_RUNS)
  int* t_es = t_run + nt;            // [nt] original index, fiber and wrap shift of the target
  int* t_fs = t_es + nt;
  int* t_ms = t_fs + nt;
  int* r_fs = t_ms + nt;             // [NB_RUNS] fiber and wrap shift of each run
  int* r_ms = r_fs + NB_RUNS;
  int* r_tab = r_ms + NB_RUNS;       // [NB_RUNS][ns] table per (run, source)
  __shared__ int s_nrun;
  for (int j = threadIdx.x; j < ns; j += blockDim.x) {
    const int f = srcf[j0 + j], m = srcm[j0 + j], ef = perm[f];
    s_f[j] = f;
    s_ef[j] = ef;
    s_ff[j] = ofib[ef];
    s_dm[j] = m - sm0[f];
    s_m[j] = m;
  }
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    const int es = perm[s0 + t];
    t_es[t] = es;
    t_fs[t] = ofib[es];
    t_ms[t] = sm0[s0 + t];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int nr = 0, pf = -1, pm = 0;
    for (int t = 0; t < nt; ++t) {
      const int fs = t_fs[t], ms = t_ms[t];
      if (t == 0 || fs != pf || ms != pm) {
        if (nr < NB_RUNS) {
          r_fs[nr] = fs;
          r_ms[nr] = ms;
        }
        ++nr;
        pf = fs;
        pm = ms;
      }
      t_run[t] = nr - 1 < NB_RUNS ? nr - 1 : -1;
    }
    s_nrun = nr < NB_RUNS ? nr : NB_RUNS;
  }
  __syncthreads();
  const int nr = s_nrun;
  for (int q = threadIdx.x; q < nr * ns; q += blockDim.x) {
    const int r = q / ns, j = q - r * ns;
    const int fs = r_fs[r];
    r_tab[q] = near_lookup(fs, s_ff[j], s_dm[j] + r_ms[r], kbase[fs], pl_ptr, pl_fib, pl_img, pl_tab);
  }
  __syncthreads();
  for (int t = warp; t < nt; t += nw) {
    const int s = s0 + t;
    const int es = t_es[t], fs = t_fs[t], ms = t_ms[t];
    const int64_t kb = kbase[fs];
    const int fN = foff[fs + 1] - foff[fs], fo = foff[fs];
    const int r = t_run[t];
    cplx* row = val ? val + base[li] + (int64_t)t * ns * 4 : nullptr;
    cplxf* rowf = valf ? valf + base[li] + (int64_t)t * ns * 4 : nullptr;
    cplxf* rowl = vall + base[li] + (int64_t)t * ns * 4;
    // four lanes per source j, one complex value each, so that a warp writes
    // 8 whole blocks (512 contiguous bytes in FP64) per store
    const int q = lane & 3;
    for (int j = lane >> 2; j < ns; j += 8) {
      const int m = s_m[j];
      if (s_f[j] == s && m == 0) {
        if (row) row[4 * j + q] = cplx{0, 0};
        if (rowf) rowf[4 * j + q] = cplxf{0.f, 0.f};
        rowl[4 * j + q] = cplxf{0.f, 0.f};
        continue;
      }
      const int ef = s_ef[j], ff = s_ff[j];
      const int tab = r >= 0 ? r_tab[r * ns + j] : near_lookup(fs, ff, s_dm[j] + ms, kb, pl_ptr, pl_fib, pl_img, pl_tab);
      int64_t at;
      const cplx* tv;
      const cplxf* tvf;
      const cplxf* tvl;
      if (tab == -2) {
        // same fiber and, in true coordinates, the same image: a rotation of the k table
        int dl = ef - es;
        if (dl < 0) dl += fN;
        at = 4 * (kb + dl);
        tv = kval;
        tvf = kvalf;
        tvl = kvall;
      } else if (tab >= 0) {
        // a translated copy of a fiber pair whose integrals are tabulated
        at = 4 * (tab_base[tab] + (int64_t)(es - fo) * tab_nb[tab] + (ef - foff[ff]));
        tv = tab_val;
        tvf = tab_valf;
        tvl = tab_vall;
      } else {
        if (q == 0) {
          const unsigned at2 = atomicAdd(qlen, 1u);
          if (at2 < qcap)
            queue[at2] = ((unsigned long long)li << 40) | ((unsigned long long)t << 24) | (unsigned long long)j;
        }
        continue;
      }
      // the tables hold the blocks of image 0; image m adds the factor alpha^m
      if (m == 0) {
        if (row) row[4 * j + q] = tv[at + q];
        if (rowf) rowf[4 * j + q] = tvf[at + q];
        rowl[4 * j + q] = tvl[at + q];
      } else {
        const cplx b = ipow_phase(alpha, m) * tv[at + q];
        if (row) row[4 * j + q] = b;
        if (rowf) rowf[4 * j + q] = cplxf{(float)b.re, (float)b.im};
        rowl[4 * j + q] = split_lo(b);
      }
    }
  }
}

// The near-field pairs that no table covers, one thread each: the element
// integrals by the Gauss ladder (as above), written into their blocks.  A block sorts
// its batch by the rule, the largest first, so that the threads of a warp take equally
// many nodes: the FP64 pipe bounds it, and in the queue's order a warp took as long as
// its nearest pair.
constexpr int ND_NT = 128, ND_MAX = 1024;
__global__ void __launch_bounds__(ND_NT) near_direct_kernel(
    const unsigned long long* __restrict__ queue, const unsigned* __restrict__ qlen, unsigned qcap,
    const int* __restrict__ ne, const int* __restrict__ bb, const int64_t* __restrict__ base,
    const int* __restrict__ sbase, const int* __restrict__ srcf, const int* __restrict__ srcm, double k, double eta,
    double H, cplx alpha, const double2* __restrict__ sc, const double2* __restrict__ st,
    const double2* __restrict__ snu, const double* __restrict__ sh, cplx* __restrict__ val, cplxf* __restrict__ valf,
    cplxf* __restrict__ vall, unsigned long long* __restrict__ stat) {
  __shared__ unsigned long long s_w[ND_MAX];
  __shared__ unsigned char s_g[ND_MAX];
  __shared__ int s_cnt[PF_GLMAX + 1], s_off[PF_GLMAX + 1];
  const unsigned n = min(*qlen, qcap);
  // pairs of a batch: the block's share, in whole passes of the block
  const unsigned share = (n + gridDim.x - 1) / gridDim.x;
  const int batch = (int)min((unsigned)ND_MAX, max(1u, (share + ND_NT - 1) / ND_NT) * ND_NT);
  unsigned long long npair = 0, nquad = 0;
  for (int64_t b0 = (int64_t)blockIdx.x * batch; b0 < n; b0 += (int64_t)gridDim.x * batch) {
    const int m0 = (int)min((int64_t)batch, n - b0);
    if (threadIdx.x <= PF_GLMAX) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long wr[ND_MAX / ND_NT];
    int key[ND_MAX / ND_NT];           // rule and place among its like
#pragma unroll
    for (int r = 0; r < ND_MAX / ND_NT; ++r) {
      const int e = r * ND_NT + (int)threadIdx.x;
      if (e >= m0) continue;
      const unsigned long long w = queue[b0 + e];
      const int li = (int)(w >> 40), t = (int)((w >> 24) & 0xFFFF), j = (int)(w & 0xFFFFFF);
      const int f = srcf[sbase[li] + j];
      const double2 x = sc[bb[ne[li]] + t];
      double2 c = sc[f];
      c.y += srcm[sbase[li] + j] * H;
      const int g = gl_order(sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / sh[f], 0);
      wr[r] = w;
      key[r] = (g << 16) | atomicAdd(&s_cnt[g], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int g = PF_GLMAX, o = 0; g >= 0; --g) {
        s_off[g] = o;
        o += s_cnt[g];
      }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ND_MAX / ND_NT; ++r)
      if (r * ND_NT + (int)threadIdx.x < m0) {
        const int g = key[r] >> 16, o = s_off[g] + (key[r] & 0xFFFF);
        s_w[o] = wr[r];
        s_g[o] = (unsigned char)g;
      }
    __syncthreads();
    for (int e = threadIdx.x; e < m0; e += ND_NT) {
      const unsigned long long w = s_w[e];
      const int li = (int)(w >> 40), t = (int)((w >> 24) & 0xFFFF), j = (int)(w & 0xFFFFFF);
      const int s = bb[ne[li]] + t;
      const int j0 = sbase[li], ns = sbase[li + 1] - j0;
      const int f = srcf[j0 + j], m = srcm[j0 + j];
      const double2 x = sc[s], nx = snu[s];
      double2 c = sc[f];
      c.y += m * H;
      const double hh = sh[f];
      const int g = s_g[e];
      ++npair;
      nquad += g;
      cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
      pair4_f64(k, x, nx, c, st[f], snu[f], hh, g, S, Dv, K, T);
      const cplx ph = mul_i(0.25 * ipow_phase(alpha, m));      // (i/4) alpha^m
      const cplx b[4] = {ph * Dv, (-eta) * mul_i(ph * S), ph * T, (-eta) * mul_i(ph * K)};
      const int64_t o = base[li] + ((int64_t)t * ns + j) * 4;
      for (int q2 = 0; q2 < 4; ++q2) {
        if (val) val[o + q2] = b[q2];
        if (valf) valf[o + q2] = cplxf{(float)b[q2].re, (float)b[q2].im};
        vall[o + q2] = split_lo(b[q2]);
      }
    }
    __syncthreads();
  }
  if (stat) {
    npair = warp_sum_u64(npair);
    nquad = warp_sum_u64(nquad);
    if ((threadIdx.x & 31) == 0 && npair) {
      atomicAdd(&stat[0], npair);
      atomicAdd(&stat[1], nquad);
    }
  }
}

// ------------------------------------------------------------ cached fiber blocks
// Row pair (2e, 2e+1) of fiber i's diagonal block of (I - A) without the
// periodic k part:  [1 - D1, i eta S1; -c2 rho T1, 1 + i eta c2 rho K1] over the
// same-fiber sources (k1, eq. 5), plus on the diagonal the self terms of both
// wavenumbers (-i eta S_ee(k) and c2 T_ee(k) of the k part, whose remainder
// comes from the FMM).  rows lists the elements whose row pairs are stored (the
// first element of a circulant fiber, every element of the others).  For a
// regular-polygon fiber (kbase >= 0) the launch's second plane (blockIdx.z = 1)
// writes the fiber's k table: S, D, K, T (without i/4) at the matrix
// wavenumber k of the first element's midpoint against element f0 + dl,
// dl = f - f0 (zero for dl = 0).  Rotating the fiber by one element maps it onto
// itself, so element pair (e, e + dl) has the integrals of (f0, f0 + dl) and the
// near-field build reads same-fiber pairs from this table.
// SP consecutive lanes share one (row element e, source f) pair and take every SP-th
// Gauss node; the partial sums meet by shuffles.  Four where the rows are few (regular
// polygons keep one: a pair's chain of nodes is then the time), one elsewhere: the FP64
// pipe bounds it, a rule of three nodes left a lane of four idle, and the end of a pair
// (the sums' shuffles and the products by c2) costs a warp the same for 8 pairs as for 32.
// A regular polygon is also symmetric under the reflection through the
// midpoint of its first element and the centre: it maps source f0 + dl onto
// f0 + N - dl and keeps both normals outward, and the Gauss rule is symmetric,
// so the first element's row (both planes) takes the integrals of dl <= N/2
// and writes each also at N - dl.

template <int SP>
__device__ __forceinline__ void group_sum(cplx& v) {
#pragma unroll
  for (int o = 1; o < SP; o <<= 1) {
    v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
    v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
  }
}

template <int SP>
__global__ void fiber_build_kernel(const int* __restrict__ rows, const int* __restrict__ fib,
                                   const int* __restrict__ foff, const int64_t* __restrict__ fbase, double k,
                                   double k1, double eta, double rho, cplx c2, const double2* __restrict__ oc,
                                   const double2* __restrict__ ot, const double2* __restrict__ onu,
                                   const double* __restrict__ oh, const cplx* __restrict__ self4,
                                   const int64_t* __restrict__ kbase, cplx* __restrict__ kval,
                                   cplx* __restrict__ ksval, cplxf* __restrict__ ksvalf, cplxf* __restrict__ ksvall,
                                   cplx* __restrict__ val, cplxf* __restrict__ valf,
                                   unsigned long long* __restrict__ stat, int zoff) {
  const int e = rows[blockIdx.x];
  const int fb = fib[e], f0 = foff[fb], N = foff[fb + 1] - f0, el = e - f0;
  const bool ktab = blockIdx.z + zoff == 1;
  const int64_t kb = kbase[fb];
  if (ktab && kb < 0) return;                      // uniform over the block
  const bool mir = kb >= 0 && el == 0;             // mirrored half row (regular polygon)
  if (mir && (int)blockIdx.y * (int)(blockDim.x / SP) > N / 2) return;   // uniform over the block
  const int part = threadIdx.x % SP;
  const int fl = blockIdx.y * (blockDim.x / SP) + threadIdx.x / SP;
  const bool lead = part == 0;
  unsigned long long np = 0, nq = 0;
  const bool on = fl < N && !(mir && fl > N / 2);
  const int fm = mir && fl > 0 && 2 * fl != N ? N - fl : -1;   // mirror entry, if any
  const int f = f0 + (on ? fl : 0);
  const bool self = on && f == e;
  cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
  const double2 xe = oc[e], nxe = onu[e];
  if (on && !self) {
    const double2 c = oc[f], tf = ot[f], nf = onu[f];
    const double hh = oh[f];
    const double q = sqrt((xe.x - c.x) * (xe.x - c.x) + (xe.y - c.y) * (xe.y - c.y)) / hh;
    const int g = gl_order(q, 0);
    if (lead) {
      np = fm >= 0 ? 2 : 1;
      nq = fm >= 0 ? 2 * g : g;
    }
    pair4_f64(ktab ? k : k1, xe, nxe, c, tf, nf, hh, g, S, Dv, K, T, part, SP);
  }
  group_sum<SP>(S);
  group_sum<SP>(Dv);
  group_sum<SP>(K);
  group_sum<SP>(T);
  if (on && lead) {
    if (ktab) {
      cplx* tv = kval + 4 * (kb + fl);
      tv[0] = S;
      tv[1] = Dv;
      tv[2] = K;
      tv[3] = T;
      near_block_form(eta, S, Dv, K, T, ksval + 4 * (kb + fl), ksvalf + 4 * (kb + fl), ksvall + 4 * (kb + fl));
      if (fm >= 0) {
        cplx* tm = kval + 4 * (kb + fm);
        tm[0] = S;
        tm[1] = Dv;
        tm[2] = K;
        tm[3] = T;
        near_block_form(eta, S, Dv, K, T, ksval + 4 * (kb + fm), ksvalf + 4 * (kb + fm), ksvall + 4 * (kb + fm));
      }
    } else {
      const int64_t r0 = fbase[fb] + (int64_t)(2 * el) * (2 * N), r1 = r0 + 2 * N;
      const cplx c2r = rho * c2;
      cplx a00, a01, a10, a11;
      if (self) {
        const cplx Sk = self4[4 * e], Tk = self4[4 * e + 1], Sk1 = self4[4 * e + 2], Tk1 = self4[4 * e + 3];
        a00 = cplx{1, 0};
        a01 = eta * mul_i(Sk1) - eta * mul_i(Sk);
        a10 = c2 * Tk - c2r * Tk1;
        a11 = cplx{1, 0};
      } else {
        S = mul_i(0.25 * S);
        Dv = mul_i(0.25 * Dv);
        K = mul_i(0.25 * K);
        T = mul_i(0.25 * T);
        a00 = -Dv;
        a01 = eta * mul_i(S);
        a10 = -(c2r * T);
        a11 = eta * mul_i(c2r * K);
      }
      for (int w = 0; w < 2; ++w) {
        const int q = w == 0 ? fl : fm;
        if (q < 0) break;
        val[r0 + 2 * q] = a00;
        val[r0 + 2 * q + 1] = a01;
        val[r1 + 2 * q] = a10;
        val[r1 + 2 * q + 1] = a11;
        if (valf) {
          valf[r0 + 2 * q] = cplxf{(float)a00.re, (float)a00.im};
          valf[r0 + 2 * q + 1] = cplxf{(float)a01.re, (float)a01.im};
          valf[r1 + 2 * q] = cplxf{(float)a10.re, (float)a10.im};
          valf[r1 + 2 * q + 1] = cplxf{(float)a11.re, (float)a11.im};
        }
      }
    }
  }
  if (stat) {
    np = warp_sum_u64(np);
    nq = warp_sum_u64(nq);
    if ((threadIdx.x & 31) == 0 && np) {
      atomicAdd(&stat[ktab ? 0 : 2], np);
      atomicAdd(&stat[ktab ? 1 : 3], nq);
    }
  }
}

// Tree-ordered copies of the element arrays (one thread per sorted element s,
// original e = perm[s]): midpoint wrapped into the root cell along y (the
// product and the subtraction rounded separately, as the host does when it
// builds the tree), tangent, normal, length, the input phase alpha^{-m0}
// (alpha = e^{i beta}), the wrap shift m0 and the leaf key.
__global__ void sort_elements_kernel(int E, const int* __restrict__ perm, const double2* __restrict__ oc,
                                     const double2* __restrict__ ot, const double2* __restrict__ onu,
                                     const double* __restrict__ oh, const int* __restrict__ om0,
                                     const int* __restrict__ okey, double H, double beta, double2* __restrict__ sc,
                                     double2* __restrict__ st, double2* __restrict__ snu, double* __restrict__ sh,
                                     cplx* __restrict__ sph, int* __restrict__ sm0, int* __restrict__ sleaf) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= E) return;
  const int e = perm[s], m = om0[e];
  const double2 c = oc[e];
  sc[s] = double2{c.x, __dsub_rn(c.y, __dmul_rn((double)m, H))};
  st[s] = ot[e];
  snu[s] = onu[e];
  sh[s] = oh[e];
  double sn, cs;
  sincos(__dmul_rn((double)(-m), beta), &sn, &cs);
  sph[s] = cplx{cs, sn};
  sm0[s] = m;
  sleaf[s] = okey[e];
}

cudaError_t k_sort_elements(pfmbem* h) {
  sort_elements_kernel<<<(h->E + 255) / 256, 256, 0, h->stream>>>(
      h->E, h->s_perm, h->o_c, h->o_t, h->o_nu, h->o_h, h->o_m0, h->o_key, h->H, h->beta, h->s_c, h->s_t, h->s_nu,
      h->s_h, h->s_ph, h->s_m0, h->s_leaf);
  return cudaGetLastError();
}

// Concatenated source list of every leaf (sorted element, image m): the
// elements of the leaf's near-list boxes in list order.  One block per leaf.
__global__ void near_sources_kernel(const int* __restrict__ nl_ptr, const int* __restrict__ nl_src,
                                    const int* __restrict__ nl_img, const int* __restrict__ bb,
                                    const int* __restrict__ be, const int* __restrict__ sbase, int* __restrict__ src,
                                    int* __restrict__ img) {
  const int li = blockIdx.x;
  int o = sbase[li];
  for (int e = nl_ptr[li]; e < nl_ptr[li + 1]; ++e) {
    const int sb = nl_src[e], m = nl_img[e], f0 = bb[sb], n = be[sb] - f0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      src[o + t] = f0 + t;
      img[o + t] = m;
    }
    o += n;
  }
}

// Launches one plane of fiber_build_kernel: the k tables (ktab) or the same-fiber blocks.
static void fiber_build_plane(pfmbem* h, bool ktab, cudaStream_t st) {
  cplx c2{h->c2re, h->c2im};
  prof_begin(h, PH_BUILD);
  const int sp = (int64_t)h->nfb_rows * h->max_fiber >= PF_SMS * 2048 ? 1 : 4;   // pairs for every resident thread
  auto kern = sp == 1 ? fiber_build_kernel<1> : fiber_build_kernel<4>;
  kern<<<dim3(h->nfb_rows, (h->max_fiber + 128 / sp - 1) / (128 / sp), 1), 128, 0, st>>>(
      h->fb_rows, h->o_fiber, h->fib_off, h->fb_base, h->k, h->k1, h->eta, h->rho, c2, h->o_c, h->o_t, h->o_nu,
      h->o_h, h->self4, h->kt_base, h->kt_val, h->kt_sval, h->kt_svalf, h->kt_svall, h->fb_val, h->fb_valf,
      h->stat_dev, ktab ? 1 : 0);
  prof_end(h, PH_BUILD);
}

// The same-fiber blocks (fiber_build_kernel's first plane), apart from the
// near-field chain, which needs only the k tables.
cudaError_t k_build_fiber_blocks(pfmbem* h) {
  fiber_build_plane(h, false, h->stream);
  return cudaGetLastError();
}

// The near-field chain: near sources, the fibers' k tables (recorded in
// ktab_done when given), the pair tables and the near-field blocks.
cudaError_t k_build_caches(pfmbem* h, cudaEvent_t ktab_done) {
  cudaStream_t st = h->stream;
  Level& leaf = h->lev[h->D];
  near_sources_kernel<<<leaf.nne, 128, 0, st>>>(h->nl_ptr, h->nl_src, h->nl_img, leaf.box_begin, leaf.box_end,
                                                h->nc_sbase, h->nc_src, h->nc_img);
  // the near-field build reads the k tables
  fiber_build_plane(h, true, st);
  if (ktab_done) {
    cudaError_t e = cudaEventRecord(ktab_done, st);
    if (e != cudaSuccess) return e;
  }
  trace(h, st, "near: k tables done");
  if (h->ntab > 0) {
    prof_begin(h, PH_BUILD);
    pair_table_kernel<<<(unsigned)((h->tab_entries + 255) / 256), 256, 0, st>>>(
        h->ntab, h->tab_A, h->tab_B, h->tab_m, h->tab_start, h->tab_start, h->fib_off, h->k, h->H, h->o_c, h->o_t,
        h->o_nu, h->o_h, h->eta, h->tab_val, h->tab_valf, h->tab_vall, h->stat_dev);
    prof_end(h, PH_BUILD);
  }
  cudaMemsetAsync(h->nq_len, 0, sizeof(unsigned), st);
  prof_begin(h, PH_BUILD);
  {
    // per-source arrays, the run and description of every target, the runs and their lookups
    const size_t smem = sizeof(int) * (5 * (size_t)h->nc_maxns + 4 * (size_t)h->leaf_maxn + 2 * NB_RUNS +
                                       (size_t)NB_RUNS * h->nc_maxns);
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(near_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    near_build_kernel<<<leaf.nne, 256, smem, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, h->nc_base, h->nc_sbase,
                                                   h->nc_src, h->nc_img, h->eta, h->alpha, h->s_perm, h->o_fiber,
                                                   h->fib_off, h->s_m0, h->kt_base, h->kt_sval, h->kt_svalf,
                                                   h->kt_svall, h->ntab > 0 ? h->pl_ptr : nullptr, h->pl_fib,
                                                   h->pl_img, h->pl_tab, h->tab_start, h->tab_nb, h->tab_val,
                                                   h->tab_valf, h->tab_vall, h->nc_val, h->nc_valf, h->nc_vall, h->nq,
                                                   h->nq_len, h->nq_cap);
  }
  prof_end(h, PH_BUILD);
  trace(h, st, "near: near_build done");
  prof_begin(h, PH_BUILD);
  near_direct_kernel<<<1216, ND_NT, 0, st>>>(h->nq, h->nq_len, h->nq_cap, leaf.ne, leaf.box_begin, h->nc_base,
                                           h->nc_sbase, h->nc_src, h->nc_img, h->k, h->eta, h->H, h->alpha, h->s_c,
                                           h->s_t, h->s_nu, h->s_h, h->nc_val, h->nc_valf, h->nc_vall,
                                           h->stat_dev);
  prof_end(h, PH_BUILD);
  trace(h, st, "near: near_direct done");
  return cudaGetLastError();
}

// ------------------------------------------------------------ cached P2M / L2P
__device__ __forceinline__ void morton_centre(int box, int D, double d, double x0, double y0, double& ox, double& oy) {
  int ix = (box >> (2 * D)) << D, iy = 0;       // root squares in a row along x, root-major
  for (int b = 0; b < D; ++b) {
    ix |= ((box >> (2 * b)) & 1) << b;
    iy |= ((box >> (2 * b + 1)) & 1) << b;
  }
  ox = x0 + (ix + 0.5) * d;
  oy = y0 + (iy + 0.5) * d;
}

// P2M coefficients of element s (the moments of Sec. 3.2 per unit density):
//   c[s][0][n] = sum_g w_g h/2 (k/2)(conj(nu) J^-_{n-1} - nu J^-_{n+1}) / w_n   (phi')
//   c[s][1][n] = sum_g w_g h/2 (-i eta) J^-_n / w_n                             (varphi')
// One thread per (element s, Gauss node q): the node's share of c[s][.][n] is
// added atomically into out, which the launcher clears first.
__global__ void p2m_coef_kernel(int E, const int* __restrict__ sleaf, int D, double d, int p,
                                const double* __restrict__ iwgt, int g, double k, double eta, double x0, double y0,
                                const double2* __restrict__ sc, const double2* __restrict__ st,
                                const double2* __restrict__ snu, const double* __restrict__ sh,
                                cplx* __restrict__ out, const double2* __restrict__ ctr) {
  // one thread per (element, Gauss node), its terms added atomically (measured
  // faster on GB300 than warp-shuffle sums over the nodes, 214 against 305 us
  // on the 8x8 hexagon block, and than J^-_m carried in a window of three)
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= E * g) return;
  const int s = t / g, q = t - s * g;
  const int P = 2 * p + 1;
  double ox, oy;
  morton_centre(sleaf[s], D, d, x0, y0, ox, oy);
  if (ctr) {                                       // leaf centres given (triangle tree)
    ox = ctr[sleaf[s]].x;
    oy = ctr[sleaf[s]].y;
  }
  const double2 c = sc[s], tt = st[s], nu = snu[s];
  const double hh = sh[s];
  const cplx nuc{nu.x, nu.y};
  cplx* o = out + (size_t)s * 2 * P;
  const double sp = 0.5 * hh * c_glx[g - 1][q];
  const double cw = 0.5 * hh * c_glw[g - 1][q];
  const double vx = c.x + sp * tt.x - ox, vy = c.y + sp * tt.y - oy;
  const double r = sqrt(vx * vx + vy * vy);
  const cplx z = r > 0 ? cplx{vx / r, -vy / r} : cplx{1, 0};   // e^{-i theta}
  double J[PF_PMAX + 2];
  bessel_j_array(k * r, p + 1, J);
  cplx Jm[2 * PF_PMAX + 3];                  // J^-_n = J_n z^n, n = -p-1 .. p+1
  cplx zp{1, 0};
  for (int n = 0; n <= p + 1; ++n) {
    Jm[p + 1 + n] = J[n] * zp;
    Jm[p + 1 - n] = (((n & 1) ? -1.0 : 1.0) * J[n]) * conj(zp);
    zp = zp * z;
  }
  for (int n = -p; n <= p; ++n) {
    const double iw = iwgt[n + p];
    const cplx a = (cw * 0.5 * k * iw) * (conj(nuc) * Jm[p + n] - nuc * Jm[p + n + 2]);
    const cplx b = (-eta * cw * iw) * mul_i(Jm[p + n + 1]);
    atomicAdd(&o[n + p].re, a.re);
    atomicAdd(&o[n + p].im, a.im);
    atomicAdd(&o[P + n + p].re, b.re);
    atomicAdd(&o[P + n + p].im, b.im);
  }
}

// FP32 copy (the hi part) and, with lo, the lo part of each value.
__global__ void to_f32_kernel(size_t n, const cplx* __restrict__ a, cplxf* __restrict__ b, cplxf* __restrict__ lo) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    b[i] = to_f(a[i]);
    if (lo) lo[i] = split_lo(a[i]);
  }
}

// L2P coefficients of target s (stored coefficient-major: [2][P][E]):
//   c[s][0][l] = (i/4) J^+_l(k(x - O)) / w_l
//   c[s][1][l] = (i/4)(k/2)(-conj(nu) J^+_{l+1} + nu J^+_{l-1}) / w_l
__global__ void l2p_coef_kernel(int E, const int* __restrict__ sleaf, int D, double d, int p,
                                const double* __restrict__ iwgt, double k, double x0, double y0,
                                const double2* __restrict__ sc, const double2* __restrict__ snu,
                                cplx* __restrict__ out, cplxf* __restrict__ outf, const double2* __restrict__ ctr,
                                size_t es, size_t cs) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= E) return;
  const int P = 2 * p + 1;
  double ox, oy;
  morton_centre(sleaf[s], D, d, x0, y0, ox, oy);
  if (ctr) {                                       // leaf centres given (triangle tree)
    ox = ctr[sleaf[s]].x;
    oy = ctr[sleaf[s]].y;
  }
  const double2 c = sc[s], nu = snu[s];
  const double vx = c.x - ox, vy = c.y - oy;
  const double r = sqrt(vx * vx + vy * vy);
  const cplx z = r > 0 ? cplx{vx / r, vy / r} : cplx{1, 0};
  double J[PF_PMAX + 2];
  bessel_j_array(k * r, p + 1, J);
  cplx Jp[2 * PF_PMAX + 3];                  // J^+_n = J_n z^n, n = -p-1 .. p+1
  cplx zp{1, 0};
  for (int n = 0; n <= p + 1; ++n) {
    Jp[p + 1 + n] = J[n] * zp;
    Jp[p + 1 - n] = (((n & 1) ? -1.0 : 1.0) * J[n]) * conj(zp);
    zp = zp * z;
  }
  const cplx nuc{nu.x, nu.y};
  // entry (q, l) of element s at s es + (q P + l) cs
  for (int l = -p; l <= p; ++l) {
    const double iw = iwgt[l + p];
    const cplx v = mul_i((0.25 * iw) * Jp[p + 1 + l]);
    const cplx dv = mul_i((0.125 * k * iw) * (nuc * Jp[p + l] - conj(nuc) * Jp[p + l + 2]));
    const size_t i0 = s * es + (l + p) * cs, i1 = s * es + (P + l + p) * cs;
    out[i0] = v;
    out[i1] = dv;
    if (outf) {
      outf[i0] = to_f(v);
      outf[i1] = to_f(dv);
    }
  }
}

// ------------------------------------------------ precision-generic matvec pieces
template <class C>
__global__ void gather_t_kernel(int E, const int* __restrict__ perm, const cplx* __restrict__ ph,
                                const cplx* __restrict__ x, C* __restrict__ dens) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= E) return;
  int e = perm[s];
  cplx p = ph[s];
  dens[2 * s] = from_d<C>(p * x[2 * e]);
  dens[2 * s + 1] = from_d<C>(p * x[2 * e + 1]);
}

// M(leaf)_n = sum_f c[f][0][n] phi'_f + c[f][1][n] varphi'_f; one block per leaf.
// Clears L(leaf) where Lz is given (the triangle tree's M2L adds to it).
template <class C>
__global__ void p2m_apply_t_kernel(const int* __restrict__ ne, const int* __restrict__ bb,
                                   const int* __restrict__ be, int P, const C* __restrict__ coef,
                                   const C* __restrict__ dens, C* __restrict__ Mout, C* __restrict__ Lz = nullptr) {
  const int box = ne[blockIdx.x];
  const int n = threadIdx.x;
  if (n >= P) return;
  if (Lz) Lz[(size_t)box * P + n] = C{0, 0};
  C acc{0, 0};
  for (int f = bb[box]; f < be[box]; ++f) {
    const C* cf = coef + (size_t)f * 2 * P;
    acc += cf[n] * dens[2 * f] + cf[P + n] * dens[2 * f + 1];
  }
  Mout[(size_t)box * P + n] = acc;
}

template <class C>
__global__ void m2m_t_kernel(const int* __restrict__ ne, int P, int Pc, const C* __restrict__ A,
                             const int* __restrict__ cbb, const int* __restrict__ cbe, const C* __restrict__ Mc,
                             C* __restrict__ Mp) {
  const int box = ne[blockIdx.x];
  __shared__ C sm[PF_NCOEF];
  C acc{0, 0};
  for (int q = 0; q < 4; ++q) {
    int ch = 4 * box + q;
    if (cbb[ch] >= cbe[ch]) continue;
    __syncthreads();
    for (int i = threadIdx.x; i < Pc; i += blockDim.x) sm[i] = Mc[(size_t)ch * Pc + i];
    __syncthreads();
    if (threadIdx.x < P) {
      const C* col = A + (size_t)q * Pc * P + threadIdx.x;        // transposed [q][m][n]
      for (int m = 0; m < Pc; ++m) acc += col[(size_t)m * P] * sm[m];
    }
  }
  if (threadIdx.x < P) Mp[(size_t)box * P + threadIdx.x] = acc;
}

// L(box) = B_q L(parent) + sum_{IL} alpha^m T_o M(src); at the root L = R M(root).
template <class C>
__global__ void local_t_kernel(const int* __restrict__ ne, int P, int Pp, const C* __restrict__ B,
                               const C* __restrict__ Lp, const int* __restrict__ ilp, const int* __restrict__ ils,
                               const int* __restrict__ ilo, const int* __restrict__ ilm, const C* __restrict__ T,
                               const C* __restrict__ Mlev, const C* __restrict__ root, cplx alpha,
                               C* __restrict__ Lout) {
  const int ti = blockIdx.x;
  const int box = ne[ti];
  __shared__ C sm[PF_NCOEF];
  C acc{0, 0};
  const int l = threadIdx.x;
  if (root) {
    for (int i = threadIdx.x; i < P; i += blockDim.x) sm[i] = Mlev[i];
    __syncthreads();
    if (l < P) {
      for (int n = 0; n < P; ++n) acc += root[(size_t)l * P + n] * sm[n];
      Lout[l] = acc;
    }
    return;
  }
  {
    int par = box >> 2, q = box & 3;
    for (int i = threadIdx.x; i < Pp; i += blockDim.x) sm[i] = Lp[(size_t)par * Pp + i];
    __syncthreads();
    if (l < P) {
      const C* col = B + (size_t)q * Pp * P + l;                  // transposed [q][m][n]
      for (int m = 0; m < Pp; ++m) acc += col[(size_t)m * P] * sm[m];
    }
  }
  for (int e = ilp[ti]; e < ilp[ti + 1]; ++e) {
    const int src = ils[e], off = ilo[e];
    const C ph = from_d<C>(ipow_phase(alpha, ilm[e]));
    __syncthreads();
    for (int i = threadIdx.x; i < P; i += blockDim.x) sm[i] = ph * Mlev[(size_t)src * P + i];
    __syncthreads();
    if (l < P) {
      const C* row = T + ((size_t)off * P + l) * P;
      for (int n = 0; n < P; ++n) acc += row[n] * sm[n];
    }
  }
  if (l < P) Lout[(size_t)box * P + l] = acc;
}

// L2L only (level >= 1): L(box) = B_q L(parent).
template <class C>
__global__ void l2l_t_kernel(const int* __restrict__ ne, int P, int Pp, const C* __restrict__ B,
                             const C* __restrict__ Lp, C* __restrict__ Lout) {
  const int box = ne[blockIdx.x];
  __shared__ C sm[PF_NCOEF];
  const int par = box >> 2, q = box & 3;
  for (int i = threadIdx.x; i < Pp; i += blockDim.x) sm[i] = Lp[(size_t)par * Pp + i];
  __syncthreads();
  for (int l = threadIdx.x; l < P; l += blockDim.x) {
    const C* col = B + (size_t)q * Pp * P + l;                    // transposed [q][m][n]
    C acc{0, 0};
    for (int m = 0; m < Pp; ++m) acc += col[(size_t)m * P] * sm[m];
    Lout[(size_t)box * P + l] = acc;
  }
}

__device__ __forceinline__ void atomic_add_c(cplx* p, cplx v) {
  atomicAdd(&p->re, v.re);
  atomicAdd(&p->im, v.im);
}
__device__ __forceinline__ void atomic_add_c(cplxf* p, cplxf v) {
  atomicAdd(&p->re, v.re);
  atomicAdd(&p->im, v.im);
}

// M2L grouped by translation offset (Sec. 3.2: the operator H^+_{n-l}(k(O_D - O_C))
// depends only on the offset, so all pairs with offset o share T_o).  Block b
// takes a chunk of the pairs of one offset: T_o is staged in shared memory once,
// each warp applies it to one pair at a time (lanes over output rows) and adds
// alpha^m T_o M(src) into L(target) atomically.
template <class C>
__global__ void m2l_offset_t_kernel(int P, const int* __restrict__ chunk_off, const int* __restrict__ chunk_beg,
                                    const int* __restrict__ chunk_end, const int* __restrict__ ptgt,
                                    const int* __restrict__ psrc, const int* __restrict__ pimg,
                                    const C* __restrict__ T, const C* __restrict__ M, cplx alpha,
                                    C* __restrict__ L) {
  extern __shared__ unsigned char smraw[];
  C* sT = reinterpret_cast<C*>(smraw);             // [P][P+1] (padded rows)
  C* sM = sT + (size_t)P * (P + 1);                 // [warps][P]
  const int o = chunk_off[blockIdx.x];
  const int pb = chunk_beg[blockIdx.x], pe = chunk_end[blockIdx.x];
  const C* To = T + (size_t)o * P * P;
  for (int i = threadIdx.x; i < P * P; i += blockDim.x) sT[(i / P) * (P + 1) + (i % P)] = To[i];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  C* mw = sM + (size_t)warp * P;
  __syncthreads();
  for (int pi = pb + warp; pi < pe; pi += nw) {
    const int src = psrc[pi], tgt = ptgt[pi];
    const C ph = from_d<C>(ipow_phase(alpha, pimg[pi]));
    for (int n = lane; n < P; n += 32) mw[n] = ph * M[(size_t)src * P + n];
    __syncwarp();
    for (int l = lane; l < P; l += 32) {
      const C* row = sT + (size_t)l * (P + 1);
      C acc0{0, 0}, acc1{0, 0};            // two independent chains
      int n = 0;
      for (; n + 1 < P; n += 2) {
        acc0 += row[n] * mw[n];
        acc1 += row[n + 1] * mw[n + 1];
      }
      if (n < P) acc0 += row[n] * mw[n];
      atomic_add_c(&L[(size_t)tgt * P + l], acc0 + acc1);
    }
    __syncwarp();
  }
}

// U'_s = sum_l c[s][0][l] L_l, dU'_s = sum_l c[s][1][l] L_l; one warp per target.
template <class C>
__global__ void l2p_apply_t_kernel(const int* __restrict__ ne, const int* __restrict__ bb,
                                   const int* __restrict__ be, int P, int E, const C* __restrict__ coef,
                                   const C* __restrict__ L, C* __restrict__ U) {
  const int box = ne[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const C* Lb = L + (size_t)box * P;
  for (int s = bb[box] + warp; s < be[box]; s += nw) {
    // coefficient-major cache: entry (q, l) of element s at (q P + l) E + s
    const C* cs = coef + s;
    C u{0, 0}, du{0, 0};
    for (int l = lane; l < P; l += 32) {
      const C Ll = Lb[l];
      u += cs[(size_t)l * E] * Ll;
      du += cs[(size_t)(P + l) * E] * Ll;
    }
    for (int o = 16; o > 0; o >>= 1) {
      u.re += __shfl_down_sync(0xffffffffu, u.re, o);
      u.im += __shfl_down_sync(0xffffffffu, u.im, o);
      du.re += __shfl_down_sync(0xffffffffu, du.re, o);
      du.im += __shfl_down_sync(0xffffffffu, du.im, o);
    }
    if (lane == 0) {
      U[2 * s] = u;
      U[2 * s + 1] = du;
    }
  }
}

template <class C>
__device__ __forceinline__ C warp_sum_t(C v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.re += __shfl_down_sync(0xffffffffu, v.re, o);
    v.im += __shfl_down_sync(0xffffffffu, v.im, o);
  }
  return v;
}

// The leaf's source densities (shared by all its targets) are staged in shared
// memory once; each row then streams only its cached 2x2 blocks, with two
// independent accumulator pairs per lane to keep more loads in flight.
#define NEAR_SMEM_SRC 1536
template <class C>
__global__ void near_apply_t_kernel(const int* __restrict__ ne, const int* __restrict__ bb,
                                    const int* __restrict__ be, const int64_t* __restrict__ base,
                                    const int* __restrict__ sbase, const int* __restrict__ srcf,
                                    const C* __restrict__ val, const C* __restrict__ dens, C* __restrict__ U) {
  __shared__ C sd[2 * NEAR_SMEM_SRC];
  const int li = blockIdx.x;
  const int box = ne[li];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int s0 = bb[box], nt = be[box] - s0;
  const int j0 = sbase[li], ns = sbase[li + 1] - j0;
  const bool staged = ns <= NEAR_SMEM_SRC;
  if (staged) {
    for (int j = threadIdx.x; j < ns; j += blockDim.x) {
      const int f = srcf[j0 + j];
      sd[2 * j] = dens[2 * f];
      sd[2 * j + 1] = dens[2 * f + 1];
    }
  }
  __syncthreads();
  for (int t = warp; t < nt; t += nw) {
    const C* row = val + base[li] + (int64_t)t * ns * 4;
    C u0{0, 0}, d0{0, 0}, u1{0, 0}, d1{0, 0};
    int j = lane;
    for (; j + 32 < ns; j += 64) {
      C p0, v0, p1, v1;
      if (staged) {
        p0 = sd[2 * j]; v0 = sd[2 * j + 1]; p1 = sd[2 * j + 64]; v1 = sd[2 * j + 65];
      } else {
        const int f0 = srcf[j0 + j], f1 = srcf[j0 + j + 32];
        p0 = dens[2 * f0]; v0 = dens[2 * f0 + 1]; p1 = dens[2 * f1]; v1 = dens[2 * f1 + 1];
      }
      const C a0 = row[4 * j], a1 = row[4 * j + 1], a2 = row[4 * j + 2], a3 = row[4 * j + 3];
      const C b0 = row[4 * j + 128], b1 = row[4 * j + 129], b2 = row[4 * j + 130], b3 = row[4 * j + 131];
      u0 += a0 * p0 + a1 * v0;
      d0 += a2 * p0 + a3 * v0;
      u1 += b0 * p1 + b1 * v1;
      d1 += b2 * p1 + b3 * v1;
    }
    for (; j < ns; j += 32) {
      C p, v;
      if (staged) { p = sd[2 * j]; v = sd[2 * j + 1]; }
      else { const int f = srcf[j0 + j]; p = dens[2 * f]; v = dens[2 * f + 1]; }
      u0 += row[4 * j] * p + row[4 * j + 1] * v;
      d0 += row[4 * j + 2] * p + row[4 * j + 3] * v;
    }
    C u = warp_sum_t(u0 + u1);
    C du = warp_sum_t(d0 + d1);
    if (lane == 0) {
      U[2 * (s0 + t)] += u;
      U[2 * (s0 + t) + 1] += du;
    }
  }
}

template <class C>
__global__ void fiber_apply_t_kernel(const int* __restrict__ chunk, const int* __restrict__ foff,
                                     const int64_t* __restrict__ fbase, const C* __restrict__ val,
                                     const int* __restrict__ opos, const cplx* __restrict__ sph, cplx c2,
                                     const cplx* __restrict__ x, const C* __restrict__ U, cplx* __restrict__ y,
                                     const int* __restrict__ circ) {
  __shared__ C xs[2 * 1024];
  const int fb = chunk[3 * blockIdx.x], rb = chunk[3 * blockIdx.x + 1], re = chunk[3 * blockIdx.x + 2];
  const int f0 = foff[fb], N = foff[fb + 1] - f0, n2 = 2 * N;
  const bool cir = circ[fb] != 0;
  for (int i = threadIdx.x; i < n2; i += blockDim.x) xs[i] = from_d<C>(x[2 * f0 + i]);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  // a warp takes the row pair (2e, 2e+1) of one element; four independent
  // accumulators per row keep eight loads in flight per lane.  A circulant
  // block is read from its generating row pair with x rotated by 2e:
  // sum_c R[(c - 2e) mod 2N] x[c] = sum_c R[c] x[(c + 2e) mod 2N].
  for (int r = rb + 2 * warp; r < re; r += 2 * nw) {
    const C* row0 = val + fbase[fb] + (cir ? 0 : (int64_t)r * n2);
    const C* row1 = row0 + n2;
    const int sh = cir ? r : 0;
    const bool two = r + 1 < re;
    C a0{0, 0}, a1{0, 0}, b0{0, 0}, b1{0, 0};
    int c = lane;
    for (; c + 32 < n2; c += 64) {
      int i0 = c + sh, i1 = c + 32 + sh;
      if (i0 >= n2) i0 -= n2;
      if (i1 >= n2) i1 -= n2;
      const C x0 = xs[i0], x1 = xs[i1];
      const C r00 = row0[c], r01 = row0[c + 32];
      a0 += r00 * x0;
      a1 += r01 * x1;
      if (two) {
        const C r10 = row1[c], r11 = row1[c + 32];
        b0 += r10 * x0;
        b1 += r11 * x1;
      }
    }
    for (; c < n2; c += 32) {
      int i0 = c + sh;
      if (i0 >= n2) i0 -= n2;
      a0 += row0[c] * xs[i0];
      if (two) b0 += row1[c] * xs[i0];
    }
    const C s0 = warp_sum_t(a0 + a1);
    const C s1 = warp_sum_t(b0 + b1);
    if (lane == 0) {
      for (int q = 0; q < (two ? 2 : 1); ++q) {
        const int rr = r + q;
        const int e = f0 + (rr >> 1);
        const int s = opos[e];
        const cplx po = cdiv(cplx{1, 0}, sph[s]);
        const cplx u = po * to_d(U[2 * s + (rr & 1)]);
        y[2 * f0 + rr] = to_d(q == 0 ? s0 : s1) + ((rr & 1) ? c2 * u : u);
      }
    }
  }
}

// Pointers of one precision for the cached matvec.
template <class C>
struct Ops {
  C* dens;
  C* U;
  C* p2m;
  C* l2p;
  C* near;
  C* fiber;
  C* root;
  C* M[PF_MAXLEVEL + 1];
  C* L[PF_MAXLEVEL + 1];
  C* m2m[PF_MAXLEVEL + 1];
  C* l2l[PF_MAXLEVEL + 1];
  C* m2l[PF_MAXLEVEL + 1];
};

static Ops<cplx> ops64(pfmbem* h) {
  Ops<cplx> o{};
  o.dens = h->dens; o.U = h->U; o.p2m = h->p2m_c; o.l2p = h->l2p_c; o.near = h->nc_val; o.fiber = h->fb_val;
  o.root = h->root;
  for (int l = 0; l <= h->D; ++l) {
    o.M[l] = h->lev[l].M; o.L[l] = h->lev[l].L; o.m2m[l] = h->lev[l].m2m; o.l2l[l] = h->lev[l].l2l;
    o.m2l[l] = h->lev[l].m2l;
  }
  return o;
}

static Ops<cplxf> ops32(pfmbem* h) {
  Ops<cplxf> o{};
  o.dens = h->densf; o.U = h->Uf; o.p2m = h->p2m_cf; o.l2p = h->l2p_cf; o.near = h->nc_valf; o.fiber = h->fb_valf;
  o.root = h->rootf;
  for (int l = 0; l <= h->D; ++l) {
    o.M[l] = h->lev[l].Mf; o.L[l] = h->lev[l].Lf; o.m2m[l] = h->lev[l].m2mf; o.l2l[l] = h->lev[l].l2lf;
    o.m2l[l] = h->lev[l].m2lf;
  }
  return o;
}

static inline int round32(int n) { return ((n + 31) / 32) * 32; }

// The cached matvec: every operator application is plain linear algebra on
// tables built once at create.
// FP32 launches are profiled under phase + 16.
template <class C>
static cudaError_t matvec_cached(pfmbem* h, const cplx* x, cplx* y, const Ops<C>& o) {
  cudaStream_t st = h->stream;
  const int E = h->E, D = h->D;
  const int po = sizeof(C) == sizeof(cplxf) ? 16 : 0;
  Level& leaf = h->lev[D];
  prof_begin(h, PH_GATHER + po);
  gather_t_kernel<C><<<(E + 255) / 256, 256, 0, st>>>(E, h->s_perm, h->s_ph, x, o.dens);
  prof_end(h, PH_GATHER + po);
  prof_begin(h, PH_P2M + po);
  p2m_apply_t_kernel<C><<<leaf.nne, round32(leaf.P), 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, leaf.P, o.p2m,
                                                              o.dens, o.M[D]);
  prof_end(h, PH_P2M + po);
  for (int l = D - 1; l >= 0; --l) {
    Level& a = h->lev[l];
    Level& c = h->lev[l + 1];
    prof_begin(h, PH_M2M + po);
    m2m_t_kernel<C><<<a.nne, round32(a.P), 0, st>>>(a.ne, a.P, c.P, o.m2m[l], c.box_begin, c.box_end, o.M[l + 1],
                                                    o.M[l]);
    prof_end(h, PH_M2M + po);
  }
  {
    Level& r = h->lev[0];
    prof_begin(h, PH_LOCAL + po);
    local_t_kernel<C><<<1, round32(r.P), 0, st>>>(r.ne, r.P, 0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                                  nullptr, o.M[0], o.root, h->alpha, o.L[0]);
    prof_end(h, PH_LOCAL + po);
  }
  for (int l = 1; l <= D; ++l) {
    Level& a = h->lev[l];
    Level& pa = h->lev[l - 1];
    const int nwarp = 8;
    const size_t smem = sizeof(C) * ((size_t)a.P * (a.P + 1) + (size_t)nwarp * a.P);
    prof_begin(h, PH_LOCAL + po);
    const bool tensor = sizeof(C) == sizeof(cplxf) && a.tc_ntile > 0 && a.tc_B != nullptr && h->tc_err != nullptr;
    if (tensor) {
      l2l_t_kernel<C><<<a.nne, round32(a.P), 0, st>>>(a.ne, a.P, pa.P, o.l2l[l - 1], o.L[l - 1], o.L[l]);
      k_m2l_tc(h, l, reinterpret_cast<const cplxf*>(o.M[l]), reinterpret_cast<cplxf*>(o.L[l]));
    } else if (smem <= 200 * 1024) {
      l2l_t_kernel<C><<<a.nne, round32(a.P), 0, st>>>(a.ne, a.P, pa.P, o.l2l[l - 1], o.L[l - 1], o.L[l]);
      if (a.nchunk > 0) {
        if (smem > 48 * 1024)
          cudaFuncSetAttribute(m2l_offset_t_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        m2l_offset_t_kernel<C><<<a.nchunk, 32 * nwarp, smem, st>>>(a.P, a.ch_off, a.ch_beg, a.ch_end, a.pr_tgt,
                                                                    a.pr_src, a.pr_img, o.m2l[l], o.M[l], h->alpha,
                                                                    o.L[l]);
      }
    } else {   // operator too large for shared memory: per-target kernel
      local_t_kernel<C><<<a.nne, round32(a.P), 0, st>>>(a.ne, a.P, pa.P, o.l2l[l - 1], o.L[l - 1], a.il_ptr, a.il_src,
                                                        a.il_off, a.il_img, o.m2l[l], o.M[l], nullptr, h->alpha,
                                                        o.L[l]);
    }
    prof_end(h, PH_LOCAL + po);
  }
  prof_begin(h, PH_L2P + po);
  l2p_apply_t_kernel<C><<<leaf.nne, 256, 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, leaf.P, h->E, o.l2p, o.L[D],
                                                  o.U);
  prof_end(h, PH_L2P + po);
  prof_begin(h, PH_NEAR + po);
  near_apply_t_kernel<C><<<leaf.nne, 256, 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, h->nc_base, h->nc_sbase,
                                                   h->nc_src, o.near, o.dens, o.U);
  prof_end(h, PH_NEAR + po);
  cplx c2{h->c2re, h->c2im};
  prof_begin(h, PH_FIBER + po);
  fiber_apply_t_kernel<C><<<h->nchunk, 256, 0, st>>>(h->fb_chunk, h->fib_off, h->fb_base, o.fiber, h->o_pos, h->s_ph,
                                                     c2, x, o.U, y, h->fb_circ);
  prof_end(h, PH_FIBER + po);
  return cudaGetLastError();
}

cudaError_t k_build_fmm_caches(pfmbem* h) {
  Level& leaf = h->lev[h->D];
  const size_t nc = (size_t)h->E * 2 * leaf.P;
  cudaError_t e = cudaMemsetAsync(h->p2m_c, 0, nc * sizeof(cplx), h->stream);
  if (e != cudaSuccess) return e;
  prof_begin(h, PH_SETUP);
  p2m_coef_kernel<<<(h->E * h->g_far + 127) / 128, 128, 0, h->stream>>>(
      h->E, h->s_leaf, h->D, leaf.d, leaf.p, leaf.iw_dev, h->g_far, h->k, h->eta, h->x0, h->y0, h->s_c, h->s_t,
      h->s_nu, h->s_h, h->p2m_c, nullptr);
  prof_end(h, PH_SETUP);
  prof_begin(h, PH_SETUP);
  to_f32_kernel<<<std::min<size_t>((nc + 255) / 256, 4096), 256, 0, h->stream>>>(nc, h->p2m_c, h->p2m_cf,
                                                                                 h->p2m_cl);
  prof_end(h, PH_SETUP);
  prof_begin(h, PH_SETUP);
  l2p_coef_kernel<<<(h->E + 127) / 128, 128, 0, h->stream>>>(h->E, h->s_leaf, h->D, leaf.d, leaf.p, leaf.iw_dev, h->k,
                                                             h->x0, h->y0, h->s_c, h->s_nu, h->l2p_c, h->l2p_cf,
                                                             nullptr, 1, h->E);
  if (h->l2p_cl)
    to_f32_kernel<<<std::min<size_t>((nc + 255) / 256, 4096), 256, 0, h->stream>>>(nc, h->l2p_c, h->l2p_cf,
                                                                                   h->l2p_cl);
  prof_end(h, PH_SETUP);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- matvec driver

// Gather the densities into tree order and run the upward pass (P2M, M2M)
// and the periodic root translation.  Triangle tree: P2M at the leaf
// triangles' centroids and M2M up to the hexagonal cells (six children each at
// level 0); their local expansions come from the operator between the cells
// (top_apply_kernel, in the product).
// one_sum (the field u): the multipoles by the elements' integrals and M2M in one sum a
// coefficient, the threads of P2M in step.  Where a density radiates almost nothing, the
// field from the far images is what other terms of the size of 1 cancel to 1e-8, and the
// cached coefficients and M2M in shares, each as accurate, moved u by 1e-9 to 6e-9 of
// itself; P2M's threads out of step by 0.4e-9 to 0.7e-9.
static void upward_f64(pfmbem* h, const cplx* x, bool one_sum = false) {
  cudaStream_t st = h->stream;
  const int E = h->E, D = h->D;
  prof_begin(h, PH_GATHER);
  gather_dens_kernel<<<(E + 255) / 256, 256, 0, st>>>(E, h->s_perm, h->s_ph, x, h->dens);
  prof_end(h, PH_GATHER);
  Level& leaf = h->lev[D];
  prof_begin(h, PH_P2M);
  if ((h->cached || h->tri_cache) && !one_sum)       // the coefficients are there
    p2m_apply_t_kernel<cplx><<<leaf.nne, round32(leaf.P), 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, leaf.P,
                                                                   h->p2m_c, h->dens, leaf.M);
  else
    p2m_f64_kernel<<<leaf.nne, 128, 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, D, leaf.d, leaf.p, leaf.w_dev,
                                              h->g_far, h->k, h->eta, h->x0, h->y0, h->s_c, h->s_t, h->s_nu, h->s_h,
                                              h->dens, leaf.M, leaf.ctr, !one_sum);
  prof_end(h, PH_P2M);
  for (int l = D - 1; l >= 0; --l) {
    Level& a = h->lev[l];
    Level& c = h->lev[l + 1];
    prof_begin(h, PH_M2M);
    const int nch = h->tree == 1 && l == 0 ? 6 : 4;
    if (one_sum)
      m2m_f64_kernel<1><<<a.nne, 64, 0, st>>>(a.ne, a.P, c.P, a.m2m, c.box_begin, c.box_end, c.M, a.M, nch, c.pidx);
    else
      m2m_f64_kernel<M2M_SPLIT><<<a.nne, 64 * M2M_SPLIT, 0, st>>>(a.ne, a.P, c.P, a.m2m, c.box_begin, c.box_end, c.M,
                                                                  a.M, nch, c.pidx);
    prof_end(h, PH_M2M);
  }
  if (h->tree == 1) return;
  cplx alpha = h->alpha;
  if (h->nroot > 1) {
    // a row of roots: the super root's local expansion of the images |m| >= m0
    prof_begin(h, PH_LOCAL);
    k_wide_local(h);
    prof_end(h, PH_LOCAL);
    return;
  }
  {
    Level& r = h->lev[0];
    prof_begin(h, PH_LOCAL);
    local_f64_kernel<<<1, round32(r.P), 0, st>>>(r.ne, 0, r.P, 0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                                                 nullptr, r.M, h->root, alpha, r.L, 4, nullptr);
    prof_end(h, PH_LOCAL);
  }
}

// Local expansions of all top cells at once: L0 = TOP M0, TOP [n P0][n P0] the
// operator between every pair of top cells (explicit M2L of the images the
// tree's lists leave out, and the super root's lattice sums for the rest).
// One warp per row.
__global__ void top_apply_kernel(int rows, const cplx* __restrict__ TOP, const cplx* __restrict__ M0,
                                 cplx* __restrict__ L0) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (row >= rows) return;
  const cplx* t = TOP + (size_t)row * rows;
  // four independent sums per lane: four loads of the row in flight at a time
  cplx a0{0, 0}, a1{0, 0}, a2{0, 0}, a3{0, 0};
  int c = lane;
  for (; c + 96 < rows; c += 128) {
    const cplx t0 = t[c], t1 = t[c + 32], t2 = t[c + 64], t3 = t[c + 96];
    a0 += t0 * M0[c];
    a1 += t1 * M0[c + 32];
    a2 += t2 * M0[c + 64];
    a3 += t3 * M0[c + 96];
  }
  for (; c < rows; c += 32) a0 += t[c] * M0[c];
  cplx acc = warp_sum((a0 + a1) + (a2 + a3));
  if (lane == 0) L0[row] = acc;
}

// FP64 near-field blocks as hi + lo of the double-float pair: the set-up keeps
// only the pair (the single-launch FP64 product works on it directly), and the
// paths that read FP64 blocks form them here once, on first use.
__global__ void near64_kernel(size_t n, const cplxf* __restrict__ hi, const cplxf* __restrict__ lo,
                              cplx* __restrict__ out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const cplxf a = hi[i], b = lo[i];
    out[i] = cplx{(double)a.re + (double)b.re, (double)a.im + (double)b.im};
  }
}

cudaError_t k_near64(pfmbem* h) {
  if (h->nc_val || !h->nc_valf || !h->nc_vall) return cudaSuccess;
  const size_t n = 4 * (size_t)h->nc_blocks;
  void* p = nullptr;
  cudaError_t e = cudaMallocAsync(&p, std::max<size_t>(n, 1) * sizeof(cplx), h->stream);
  if (e != cudaSuccess) return e;
  h->allocs.push_back(p);
  h->nc_val = static_cast<cplx*>(p);
  if (n > 0)
    near64_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, 4096), 256, 0, h->stream>>>(n, h->nc_valf, h->nc_vall,
                                                                                           h->nc_val);
  return cudaGetLastError();
}

// Triangle tree, cached FP64 product: the square tree's cached tables where they
// are tree-independent (P2M/L2P coefficients at the leaves' centroids, near-field
// and same-fiber blocks, M2L by offset groups), and M2M/L2L with the per-box
// operators of the triangles.
// Two chains that meet at the end.  The tree's translations keep the FP32 pipes
// busy (double-float M2M, M2L, L2L); the near-field and same-fiber blocks and the
// operator between the cells are FP64 sums and table reads, and run beside them on
// the handle's second stream: near sums and same-fiber rows (which write y) while the
// tree works upward and across, the cells' operator after the M2M; the L2L and L2P
// (which adds to y) wait for that stream.  So M2L comes before L2L and adds
// to expansions that the upward pass cleared.  16384 elements, p = 30: 1.78 ms as
// one chain.
static cudaError_t tri_chains(pfmbem* h, const cplx* x, cplx* y, bool fork) {
  cudaStream_t st = h->stream, st2 = fork ? h->aux[0] : st;
  const int E = h->E, D = h->D;
  Level& leaf = h->lev[D];
  const cplx alpha = h->alpha;
  cudaError_t e = cudaSuccess;
  prof_begin(h, PH_GATHER);
  gather_dens_kernel<<<(E + 255) / 256, 256, 0, st>>>(E, h->s_perm, h->s_ph, x, h->dens);
  prof_end(h, PH_GATHER);
  if (fork) {
    if ((e = cudaEventRecord(h->fork_ev, st)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(st2, h->fork_ev, 0)) != cudaSuccess) return e;
  }
  prof_begin(h, PH_NEAR);
  if ((e = cudaMemsetAsync(h->U, 0, 2 * sizeof(cplx) * (size_t)E, st2)) != cudaSuccess) return e;
  near_apply_t_kernel<cplx><<<leaf.nne, 256, 0, st2>>>(leaf.ne, leaf.box_begin, leaf.box_end, h->nc_base, h->nc_sbase,
                                                       h->nc_src, h->nc_val, h->dens, h->U);
  prof_end(h, PH_NEAR);
  prof_begin(h, PH_FIBER);
  if ((e = k_tri_fiber(h, x, y, st2)) != cudaSuccess) return e;
  prof_end(h, PH_FIBER);
  prof_begin(h, PH_P2M);
  p2m_apply_t_kernel<cplx><<<leaf.nne, round32(leaf.P), 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, leaf.P,
                                                                 h->p2m_c, h->dens, leaf.M, leaf.L);
  prof_end(h, PH_P2M);
  // M2M, L2L and M2L in double-float arithmetic on the FP32 pipes
  // (PFMBEM_TRI_M2L64=1: FP64 instructions, for measurement)
  static const bool m2l64 = std::getenv("PFMBEM_TRI_M2L64") != nullptr;
  for (int l = D - 1; l >= 0; --l) {
    Level& a = h->lev[l];
    Level& c = h->lev[l + 1];
    prof_begin(h, PH_M2M);
    if (!m2l64) {
      e = k_tri_m2m_dd(h, l);
      if (e != cudaSuccess) return e;
    } else {
      m2m_f64_kernel<M2M_SPLIT><<<a.nne, 64 * M2M_SPLIT, 0, st>>>(a.ne, a.P, c.P, a.m2m, c.box_begin, c.box_end, c.M,
                                                                  a.M, l == 0 ? 6 : 4, c.pidx);
    }
    prof_end(h, PH_M2M);
  }
  if (fork) {
    if ((e = cudaEventRecord(h->side_ev, st)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(st2, h->side_ev, 0)) != cudaSuccess) return e;
  }
  prof_begin(h, PH_LOCAL);
  if ((e = k_tri_top(h, st2)) != cudaSuccess) return e;
  prof_end(h, PH_LOCAL);
  if (fork && (e = cudaEventRecord(h->aux_ev[0], st2)) != cudaSuccess) return e;
  // M2L by offset groups; where a group's operator does not fit shared memory,
  // per target over its list, with L2L
  auto grouped = [&](int l) { return !m2l64 && k_tri_m2l_smem(h->lev[l].P) <= TRI_M2L_SMEM; };
  if (!m2l64) {
    prof_begin(h, PH_M2L);
    if ((e = k_tri_m2l_dd(h)) != cudaSuccess) return e;
    prof_end(h, PH_M2L);
  }
  if (fork && (e = cudaStreamWaitEvent(st, h->aux_ev[0], 0)) != cudaSuccess) return e;
  for (int l = 1; l <= D; ++l) {
    Level& a = h->lev[l];
    Level& pa = h->lev[l - 1];
    const int nwarp = 8;
    const size_t smem = sizeof(cplx) * ((size_t)a.P * (a.P + 1) + (size_t)nwarp * a.P);
    const bool lists = !m2l64 || smem > 200 * 1024;
    prof_begin(h, PH_LOCAL);
    if (grouped(l)) {
      e = k_tri_l2l_dd(h, l);
      if (e != cudaSuccess) return e;
    } else {
      local_f64_kernel<<<a.nne, round32(a.P), 0, st>>>(a.ne, 0, a.P, pa.P, pa.l2l, pa.L, lists ? a.il_ptr : nullptr,
                                                       a.il_src, a.il_off, a.il_img, a.m2l, a.M, nullptr, alpha, a.L,
                                                       l == 1 ? 6 : 4, a.pidx);
    }
    prof_end(h, PH_LOCAL);
    if (lists || a.nchunk == 0) continue;
    prof_begin(h, PH_M2L);
    if (smem > 48 * 1024)
      cudaFuncSetAttribute(m2l_offset_t_kernel<cplx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    m2l_offset_t_kernel<cplx><<<a.nchunk, 32 * nwarp, smem, st>>>(a.P, a.ch_off, a.ch_beg, a.ch_end, a.pr_tgt,
                                                                   a.pr_src, a.pr_img, a.m2l, a.M, alpha, a.L);
    prof_end(h, PH_M2L);
  }
  prof_begin(h, PH_L2P);
  if ((e = k_tri_l2p(h, y)) != cudaSuccess) return e;
  prof_end(h, PH_L2P);
  return cudaGetLastError();
}

static cudaError_t matvec_tri_cached(pfmbem* h, const cplx* x, cplx* y) {
  cudaError_t e = k_near64(h);
  if (e != cudaSuccess) return e;
  // one chain where phases are timed, for their events lie on one stream
  const bool fork = h->aux[0] && h->aux_ev[0] && h->fork_ev && h->side_ev && !h->prof.on;
  if (!fork) return tri_chains(h, x, y, false);
  return run_with_side(h->stream, h->aux[0], h->aux_ev[0], [&] { return tri_chains(h, x, y, true); });
}

cudaError_t k_tri_caches(pfmbem* h) {
  cudaStream_t st = h->stream;
  Level& leaf = h->lev[h->D];
  const size_t nc = (size_t)h->E * 2 * leaf.P;
  cudaError_t e = cudaMemsetAsync(h->p2m_c, 0, nc * sizeof(cplx), st);
  if (e != cudaSuccess) return e;
  prof_begin(h, PH_SETUP);
  p2m_coef_kernel<<<(h->E * h->g_far + 127) / 128, 128, 0, st>>>(
      h->E, h->s_leaf, h->D, leaf.d, leaf.p, leaf.iw_dev, h->g_far, h->k, h->eta, h->x0, h->y0, h->s_c, h->s_t,
      h->s_nu, h->s_h, h->p2m_c, leaf.ctr);
  l2p_coef_kernel<<<(h->E + 127) / 128, 128, 0, st>>>(h->E, h->s_leaf, h->D, leaf.d, leaf.p, leaf.iw_dev, h->k, h->x0,
                                                      h->y0, h->s_c, h->s_nu, h->l2p_c, nullptr, leaf.ctr, 2 * leaf.P, 1);
  prof_end(h, PH_SETUP);
  e = k_build_caches(h, nullptr);
  if (e != cudaSuccess) return e;
  return k_build_fiber_blocks(h);
}

cudaError_t k_matvec(pfmbem* h, const cplx* x, cplx* y, int precision) {
  if (h->tree == 1 && h->tri_cache) return matvec_tri_cached(h, x, y);
  if (h->cached && h->fused) return k_matvec_fused(h, x, y, precision);
  if (h->cached) {
    if (precision == PFMBEM_MIXED) return matvec_cached(h, x, y, ops32(h));
    cudaError_t e = k_near64(h);
    if (e != cudaSuccess) return e;
    return matvec_cached(h, x, y, ops64(h));
  }
  // on-the-fly path (no cached operators): FP64 element integrals in every product
  cudaStream_t st = h->stream;
  const int E = h->E, D = h->D;
  Level& leaf = h->lev[D];
  const cplx alpha = h->alpha;
  upward_f64(h, x);
  if (h->tree == 1) {
    // the hexagonal cells' local expansions from all cells' multipoles
    const int rows = h->nroot * h->lev[0].P;
    prof_begin(h, PH_LOCAL);
    top_apply_kernel<<<(rows * 32 + 255) / 256, 256, 0, st>>>(rows, h->root, h->lev[0].M, h->lev[0].L);
    prof_end(h, PH_LOCAL);
  }
  for (int l = 1; l <= D; ++l) {
    Level& a = h->lev[l];
    Level& pa = h->lev[l - 1];
    prof_begin(h, PH_LOCAL);
    local_f64_kernel<<<a.nne, round32(a.P), 0, st>>>(a.ne, 0, a.P, pa.P, pa.l2l, pa.L, a.il_ptr, a.il_src, a.il_off,
                                                     a.il_img, a.m2l, a.M, nullptr, alpha, a.L,
                                                     h->tree == 1 && l == 1 ? 6 : 4, a.pidx);
    prof_end(h, PH_LOCAL);
  }
  prof_begin(h, PH_L2P);
  l2p_f64_kernel<<<leaf.nne, 64, 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, D, leaf.d, leaf.p, leaf.w_dev, h->k,
                                          h->x0, h->y0, h->s_c, h->s_nu, leaf.L, h->U, leaf.ctr);
  prof_end(h, PH_L2P);
  cplx c2{h->c2re, h->c2im};
  prof_begin(h, PH_NEAR);
  near_f64_kernel<<<leaf.nne, 256, 0, st>>>(leaf.ne, leaf.box_begin, leaf.box_end, h->nl_ptr, h->nl_src, h->nl_img,
                                            h->k, h->eta, h->H, alpha, h->s_c, h->s_t, h->s_nu, h->s_h, h->dens, h->U);
  prof_end(h, PH_NEAR);
  prof_begin(h, PH_FIBER);
  fiber_combine_f64_kernel<<<(E * 32 + 255) / 256, 256, 0, st>>>(E, h->o_fiber, h->fib_off, h->k1, h->eta, h->rho, c2,
                                                                 h->o_c, h->o_t, h->o_nu, h->o_h, h->o_pos, h->s_ph,
                                                                 h->self4, x, h->U, y);
  prof_end(h, PH_FIBER);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- rhs
__global__ void rhs_kernel(int E, double k, double dx, double dy, cplx c2, const double2* __restrict__ oc,
                           const double2* __restrict__ onu, cplx* __restrict__ B) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  double2 c = oc[e], nu = onu[e];
  double ph = k * (c.x * dx + c.y * dy);
  double s, co;
  sincos(ph, &s, &co);
  cplx u{co, s};
  cplx dn = mul_i((k * (nu.x * dx + nu.y * dy)) * u);
  B[2 * e] = -u;
  B[2 * e + 1] = -(c2 * dn);
}

cudaError_t k_rhs(pfmbem* h, cplx* B) {
  cplx c2{h->c2re, h->c2im};
  prof_begin(h, PH_OUT);
  rhs_kernel<<<(h->E + 255) / 256, 256, 0, h->stream>>>(h->E, h->k, cos(h->theta), sin(h->theta), c2, h->o_c, h->o_nu, B);
  prof_end(h, PH_OUT);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- BLAS-1 for GMRES
// out[c] = sum_t conj(V[c][t]) w[t] for c < ncol (out zeroed by the caller).
__global__ void multidot_kernel(const cplx* __restrict__ V, int n, const cplx* __restrict__ w, cplx* __restrict__ out) {
  const int c = blockIdx.y;
  const cplx* v = V + (size_t)c * n;
  cplx acc{0, 0};
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) acc += conj(v[t]) * w[t];
  acc = warp_sum(acc);
  __shared__ cplx red[32];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = acc;
  __syncthreads();
  if (wid == 0) {
    acc = lane < (blockDim.x >> 5) ? red[lane] : cplx{0, 0};
    acc = warp_sum(acc);
    if (lane == 0) {
      atomicAdd(&out[c].re, acc.re);
      atomicAdd(&out[c].im, acc.im);
    }
  }
}

cudaError_t k_multidot(pfmbem* h, const cplx* V, int ncol, const cplx* w, int n, cplx* out) {
  cudaMemsetAsync(out, 0, sizeof(cplx) * ncol, h->stream);
  int bx = (n + 255) / 256;
  if (bx > 64) bx = 64;
  dim3 grid(bx, ncol);
  prof_begin(h, PH_BLAS);
  multidot_kernel<<<grid, 256, 0, h->stream>>>(V, n, w, out);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}

__global__ void gemv_kernel(const cplx* __restrict__ V, int ncol, int n, const cplx* __restrict__ coef, double sign,
                            cplx* __restrict__ w) {
  __shared__ cplx cs[256];
  for (int i = threadIdx.x; i < ncol; i += blockDim.x) cs[i] = coef[i];
  __syncthreads();
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    cplx acc{0, 0};
    for (int c = 0; c < ncol; ++c) acc += V[(size_t)c * n + t] * cs[c];
    w[t] += sign * acc;
  }
}

cudaError_t k_gemv_sub(pfmbem* h, const cplx* V, int ncol, const cplx* coef, cplx* w, int n) {
  prof_begin(h, PH_BLAS);
  gemv_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(V, ncol, n, coef, -1.0, w);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}
cudaError_t k_gemv_add(pfmbem* h, const cplx* V, int ncol, const cplx* coef, cplx* y, int n) {
  prof_begin(h, PH_BLAS);
  gemv_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(V, ncol, n, coef, 1.0, y);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}

__global__ void norm2_kernel(const cplx* __restrict__ v, int n, double* __restrict__ out) {
  double acc = 0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) acc += abs2(v[t]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  __shared__ double red[32];
  int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = acc;
  __syncthreads();
  if (wid == 0) {
    acc = lane < (blockDim.x >> 5) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) atomicAdd(out, acc);
  }
}

cudaError_t k_norm2(pfmbem* h, const cplx* v, int n, double* out) {
  cudaMemsetAsync(out, 0, sizeof(double), h->stream);
  int bx = (n + 255) / 256;
  if (bx > 128) bx = 128;
  prof_begin(h, PH_BLAS);
  norm2_kernel<<<bx, 256, 0, h->stream>>>(v, n, out);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}

__global__ void scale_copy_kernel(const cplx* __restrict__ s, cplx a, cplx* __restrict__ d, int n) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) d[t] = a * s[t];
}
cudaError_t k_scale_copy(pfmbem* h, const cplx* src, cplx s, cplx* dst, int n) {
  prof_begin(h, PH_BLAS);
  scale_copy_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(src, s, dst, n);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}
__global__ void axpy_kernel(cplx a, const cplx* __restrict__ x, cplx* __restrict__ y, int n) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) y[t] += a * x[t];
}
cudaError_t k_axpy(pfmbem* h, cplx a, const cplx* x, cplx* y, int n) {
  prof_begin(h, PH_BLAS);
  axpy_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(a, x, y, n);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}
__global__ void sub_kernel(const cplx* __restrict__ a, const cplx* __restrict__ b, cplx* __restrict__ o, int n) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) o[t] = a[t] - b[t];
}
cudaError_t k_sub(pfmbem* h, const cplx* a, const cplx* b, cplx* out, int n) {
  prof_begin(h, PH_BLAS);
  sub_kernel<<<(n + 255) / 256, 256, 0, h->stream>>>(a, b, out, n);
  prof_end(h, PH_BLAS);
  return cudaGetLastError();
}

// sum_n c_n J_n(kr) e^{i n theta} at v, c_n = L_n / w_n, and its x1-derivative
// (k/2) sum_m J_m(kr) e^{i m theta} (c_{m+1} - c_{m-1}).
__device__ void local_field(double k, double vx, double vy, int p0, const double* __restrict__ w0,
                            const cplx* __restrict__ L0, cplx& loc, cplx& dloc) {
  const double r = sqrt(vx * vx + vy * vy);
  const cplx z = r > 0 ? cplx{vx / r, vy / r} : cplx{1, 0};
  double J[PF_PMAX + 2];
  bessel_j_array(k * r, p0 + 1, J);
  cplx zp{1, 0};
  loc = dloc = cplx{0, 0};
  auto coef = [&](int n) -> cplx {
    if (n < -p0 || n > p0) return cplx{0, 0};
    return (1.0 / w0[p0 + n]) * L0[p0 + n];
  };
  for (int l = 0; l <= p0 + 1; ++l) {
    const cplx Bp = J[l] * zp;                                      // B_l
    const cplx Bm = ((l & 1) ? -J[l] : J[l]) * conj(zp);            // B_-l
    if (l <= p0) {
      loc += coef(l) * Bp;
      if (l > 0) loc += coef(-l) * Bm;
    }
    dloc += (coef(l + 1) - coef(l - 1)) * Bp;
    if (l > 0) dloc += (coef(-l + 1) - coef(-l - 1)) * Bm;
    zp = zp * z;
  }
  dloc = (0.5 * k) * dloc;
}

// alpha^{mp}: back from the period's copy of a point to the point itself
__device__ __forceinline__ cplx point_phase(cplx alpha, int mp) {
  return cplx{cos(mp * atan2(alpha.im, alpha.re)), sin(mp * atan2(alpha.im, alpha.re))};
}

// The local expansions at point pi: its part nsl.
__device__ __forceinline__ void local_part(int pi, int npts, const double2* __restrict__ pts, int nsl, double k,
                                           double H, double ox, double oy, double y0, int p0,
                                           const double* __restrict__ w0, const cplx* __restrict__ L0,
                                           cplx* __restrict__ part) {
  if (pi >= npts) return;
  double2 x = pts[pi];
  x.y -= floor((x.y - y0) / H) * H;
  cplx* o = part + 2 * ((size_t)pi * (nsl + 1) + nsl);
  local_field(k, x.x - ox, x.y - oy, p0, w0, L0, o[0], o[1]);
}

// u and du/dx1 of every point from its parts, back at the point's own period:
// u^s(x) = (i/4) alpha^{mp} (sum of the parts).
__global__ void field_finish_kernel(int npts, const double2* __restrict__ pts, int nsl, double H, double y0,
                                    cplx alpha, const cplx* __restrict__ part, cplx* __restrict__ u,
                                    cplx* __restrict__ dudx1) {
  const int pi = blockIdx.x * blockDim.x + threadIdx.x;
  if (pi >= npts) return;
  cplx acc{0, 0}, dacc{0, 0};
  for (int q = 0; q <= nsl; ++q) {
    const cplx* o = part + 2 * ((size_t)pi * (nsl + 1) + q);
    acc += o[0];
    dacc += o[1];
  }
  const cplx am = point_phase(alpha, (int)floor((pts[pi].y - y0) / H));
  if (u) u[pi] = am * mul_i(0.25 * acc);
  if (dudx1) dudx1[pi] = am * mul_i(0.25 * dacc);
}

// ---------------------------------------------------------------- field
// u^s(x) = sum_e (D2b phi - i eta S2b varphi)(x) (eq. 7): the point is moved
// into the root cell (u^s(x + m h) = alpha^m u^s(x), eq. 3), images m = -1, 0, 1
// of every element are integrated directly, and the images |m| >= 2 enter
// through the root local expansion built from the lattice sums (Sec. 3.3).
// Scattered field u^s (eq. 7) and its x1-derivative at points outside the
// fibers.  Images m = -1, 0, 1 of every element by Gauss quadrature (the target
// "normal" (1, 0) turns the K and T integrals into d/dx1 of the single- and
// double-layer integrals); images |m| >= 2 through the root local expansion
// sum_n c_n J_n(kr) e^{i n theta}, c_n = L_n / w_n, whose x1-derivative is
// (k/2) sum_m J_m(kr) e^{i m theta} (c_{m+1} - c_{m-1}).
// With a row of roots the direct images are |m| <= mdir = m0 - 1 and the local
// expansion is the super root's (centre (ox, oy)); one root: mdir = 1, the root's.
// One warp and block per (point, slice), so that few points spread over the SMs and many
// even out (634 points on 3350 elements 28.7 -> 19.2 ms, 11 points on 1296 4.47 -> 4.11
// against blocks of four): slice q of nsl takes every nsl-th group of 32 of
// the (element, image) pairs and leaves its sums in part[point][q]; the local
// expansions are separate threads (the last blocks) and go to part[point][nsl];
// field_finish_kernel adds a point's parts in order.  Bound by the FP64 pipe.  The
// derivative alone takes slices, for one warp per point leaves most of the chip idle
// below some thousand points.  u takes one slice and the series' Bessel functions: its
// terms are of the size of 1 where it may be 1e-8, so that another order of the sum
// shows at 2e-9 to 7e-9 of u (1024 points on 16384 elements: 104 ms; in blocks of four
// warps 117 ms, with the joint interpolants 74 ms, with slices too 64 ms).
template <bool WU, bool WD>
__global__ void __launch_bounds__(32) field_direct_kernel(
    int npts, const double2* __restrict__ pts, int nsl, int E, double k, double eta, double H, double ox, double oy,
    double y0, int mdir, cplx alpha, const double2* __restrict__ sc, const double2* __restrict__ st,
    const double2* __restrict__ snu, const double* __restrict__ sh, const cplx* __restrict__ dens, int p0,
    const double* __restrict__ w0, const cplx* __restrict__ L0, cplx* __restrict__ part) {
  const int lane = threadIdx.x, w = blockIdx.x;
  if (w >= npts * nsl) {
    local_part((w - npts * nsl) * 32 + lane, npts, pts, nsl, k, H, ox, oy, y0, p0, w0, L0, part);
    return;
  }
  const int pi = w / nsl, sl = w - pi * nsl;
  double2 x = pts[pi];
  x.y -= floor((x.y - y0) / H) * H;
  const double2 nx{1.0, 0.0};
  cplx acc{0, 0}, dacc{0, 0};
  const int nim = 2 * mdir + 1;
  for (int t = 32 * sl + lane; t < nim * E; t += 32 * nsl) {
    const int f = t / nim, m = t % nim - mdir;
    double2 c = sc[f];
    c.y += m * H;
    const double hh = sh[f];
    const double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / hh;
    const int g = gl_order(q, 0);
    cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
    pair4_f64<WU>(k, x, nx, c, st[f], snu[f], hh, g, S, Dv, K, T);
    const cplx ph = ipow_phase(alpha, m);
    if (WU) acc += ph * (Dv * dens[2 * f] - eta * mul_i(S * dens[2 * f + 1]));
    if (WD) dacc += ph * (T * dens[2 * f] - eta * mul_i(K * dens[2 * f + 1]));
  }
  if (WU) acc = warp_sum(acc);
  if (WD) dacc = warp_sum(dacc);
  if (lane == 0) {
    cplx* o = part + 2 * ((size_t)pi * (nsl + 1) + sl);
    o[0] = acc;
    o[1] = dacc;
  }
}

// The x1-derivative through the multipoles of the tree (the ETC of Sec. 4): every
// image |m| <= mdir of every box far enough from the point enters by its multipole
// expansion, sum_n M_n d/dx1 H^+_n(k(x - O)), d/dx1 H^+_n = (k/2)(H^+_{n-1} -
// H^+_{n+1}), and only the elements of the remaining leaves by quadrature.  A box
// is far enough when its radius (half an element length added: elements stick out
// of their box) is at most theta_l of its distance, theta_l = min(0.26,
// 10^{-18/(p+1)}): the remainder of a monopole falls like theta^(p+1), that of a
// dipole's derivative is (p + 1) / theta times as large, 2e-16 of the box's field
// (at 10^{-14.7/(p+1)} it was 2e-13 at p = 20; a point costs a tenth more).
// The field itself stays directly summed (field_direct_kernel).
// One block per point walks the levels; the boxes that are too near are listed in
// shared memory and their children tested at the next level.  FT_CAP holds every
// list: the boxes of one level are disjoint and a listed one lies within (R + h/2)
// / theta + R of the point, which at the smallest theta of the rule (0.139 at
// p = 20) and the longest element (a quarter of a leaf) is the area of 141 squares,
// 242 triangles or 121 hexagonal cells (a box that found no room would be summed by
// its elements at once).  The blocks from npts on evaluate the local
// expansions, one point per thread.
// FP64 arithmetic bounds it, about 0.5 million FP64 operations a point (some 300
// expansions of 600 and the near elements); the direct sum has 3 E pairs of about
// 400, 20 million on 16384 elements.  ETC with 256 points on 6144 elements: 25.5 ->
// 0.93 ms.
constexpr int FT_CAP = 256, FT_NT = 256;
struct FieldTree {
  int D, nroot, nch0;
  int p[PF_MAXLEVEL + 1];
  double d[PF_MAXLEVEL + 1];
  double far2[PF_MAXLEVEL + 1];        // (radius / theta)^2: squared distance from which a box is far
  const double* w[PF_MAXLEVEL + 1];
  const int* bb[PF_MAXLEVEL + 1];
  const int* be[PF_MAXLEVEL + 1];
  const cplx* M[PF_MAXLEVEL + 1];
  const double2* ctr[PF_MAXLEVEL + 1]; // box centres (triangle tree), null: from the Morton code
};

// x1-derivative of sum_{|n| <= q} c_n H^+_n(k v), c_n = w_n M_n, or M_n without weights;
// q <= p, the order of M.
__device__ __forceinline__ cplx multipole_dx1(double k, double vx, double vy, int p, int q,
                                              const double* __restrict__ w, const cplx* __restrict__ M) {
  const double r2 = vx * vx + vy * vy, ir = rsqrt(r2), x = k * r2 * ir;
  const cplx z{vx * ir, vy * ir};
  double J0, J1, Y0, Y1;
  bessel01(x, J0, J1, Y0, Y1);
  cplx hm{J0, Y0}, h{J1, Y1}, zp{1, 0};
  const double ix2 = 2.0 / x;
  auto coef = [&](int n) -> cplx {
    if (n > q || n < -q) return cplx{0, 0};
    return w ? w[p + n] * M[p + n] : M[p + n];
  };
  // coefficients around +-n: a_n = c_n, b_n = c_-n
  const cplx c0 = coef(0);
  cplx am = c0, a = coef(1), b = c0, bn = coef(-1);    // am = c_{n-1}, a = c_n, b = c_{-(n-1)}, bn = c_{-n}
  cplx d = hm * (a - bn);                      // m = 0: c_1 - c_-1
  double sg = -1.0;
  for (int n = 1; n <= q + 1; ++n) {
    zp = zp * z;
    const cplx hp = h * zp, hn = sg * (h * conj(zp));   // H^+_n, H^+_-n
    const cplx a2 = coef(n + 1), b2 = coef(-n - 1);      // c_{n+1}, c_{-(n+1)}
    d += hp * (a2 - am) + hn * (b - b2);
    am = a;
    a = a2;
    b = bn;
    bn = b2;
    sg = -sg;
    const cplx hnext{n * ix2 * h.re - hm.re, n * ix2 * h.im - hm.im};
    hm = h;
    h = hnext;
  }
  return (0.5 * k) * d;
}

// The x1-derivative at x of elements f0 .. f1 by quadrature, y moved by m periods.
__device__ __noinline__ cplx elements_dx1(double2 x, int f0, int f1, double my, double k, double eta,
                                          const double2* __restrict__ sc, const double2* __restrict__ st,
                                          const double2* __restrict__ snu, const double* __restrict__ sh,
                                          const cplx* __restrict__ dens) {
  cplx d{0, 0};
  for (int f = f0; f < f1; ++f) {
    double2 c = sc[f];
    c.y += my;
    const double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / sh[f];
    cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
    pair4_f64(k, x, double2{1.0, 0.0}, c, st[f], snu[f], sh[f], gl_order(q, 0), S, Dv, K, T);
    d += T * dens[2 * f] - eta * mul_i(K * dens[2 * f + 1]);
  }
  return d;
}

__global__ void __launch_bounds__(FT_NT) field_tree_kernel(
    const __grid_constant__ FieldTree ft, int npts, const double2* __restrict__ pts, double k, double eta, double H,
    double ox, double oy, double x0, double y0, int mdir, cplx alpha, const double2* __restrict__ sc,
    const double2* __restrict__ st, const double2* __restrict__ snu, const double* __restrict__ sh,
    const cplx* __restrict__ dens, int p0, const double* __restrict__ w0, const cplx* __restrict__ L0,
    cplx* __restrict__ part) {
  if ((int)blockIdx.x >= npts) {
    local_part(((int)blockIdx.x - npts) * FT_NT + threadIdx.x, npts, pts, 1, k, H, ox, oy, y0, p0, w0, L0, part);
    return;
  }
  __shared__ int s_box[2][FT_CAP], s_img[2][FT_CAP], s_n[2], s_off[FT_CAP + 1];
  __shared__ cplx s_red[FT_NT / 32];
  const int tid = threadIdx.x, pi = blockIdx.x;
  double2 x = pts[pi];
  x.y -= floor((x.y - y0) / H) * H;
  cplx dacc{0, 0};
  if (tid < 2) s_n[tid] = 0;
  __syncthreads();
  for (int l = 0; l <= ft.D; ++l) {
    const int cur = l & 1, prv = cur ^ 1;
    const int nch = l == 0 ? ft.nroot : l == 1 ? ft.nch0 : 4;
    const int ntest = l == 0 ? ft.nroot * (2 * mdir + 1) : min(s_n[prv], FT_CAP) * nch;
    for (int i = tid; i < ntest; i += FT_NT) {
      const int q = i / nch, r = i - q * nch;
      const int box = l == 0 ? r : nch * s_box[prv][q] + r;
      const int m = l == 0 ? q - mdir : s_img[prv][q];
      if (ft.bb[l][box] >= ft.be[l][box]) continue;
      double cx, cy;
      if (ft.ctr[l]) {
        cx = ft.ctr[l][box].x;
        cy = ft.ctr[l][box].y;
      } else {
        morton_centre(box, l, ft.d[l], x0, y0, cx, cy);
      }
      const double vx = x.x - cx, vy = x.y - (cy + m * H);
      if (vx * vx + vy * vy >= ft.far2[l]) {
        dacc += ipow_phase(alpha, m) *
                multipole_dx1(k, vx, vy, ft.p[l], ft.p[l], ft.w[l], ft.M[l] + (size_t)box * (2 * ft.p[l] + 1));
      } else {
        const int o = atomicAdd(&s_n[cur], 1);
        if (o < FT_CAP) {
          s_box[cur][o] = box;
          s_img[cur][o] = m;
        } else {
          dacc += ipow_phase(alpha, m) *
                  elements_dx1(x, ft.bb[l][box], ft.be[l][box], m * H, k, eta, sc, st, snu, sh, dens);
        }
      }
    }
    __syncthreads();
    if (tid == 0) s_n[prv] = 0;
    __syncthreads();
  }
  // the elements of the near leaves
  const int cur = ft.D & 1, nl = min(s_n[cur], FT_CAP);
  if (tid == 0) {
    int o = 0;
    for (int i = 0; i < nl; ++i) {
      s_off[i] = o;
      o += ft.be[ft.D][s_box[cur][i]] - ft.bb[ft.D][s_box[cur][i]];
    }
    s_off[nl] = o;
  }
  __syncthreads();
  const double2 nx{1.0, 0.0};
  for (int t = tid; t < s_off[nl]; t += FT_NT) {
    int lo = 0, hi = nl - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_off[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    const int f = ft.bb[ft.D][s_box[cur][lo]] + t - s_off[lo], m = s_img[cur][lo];
    double2 c = sc[f];
    c.y += m * H;
    const double hh = sh[f];
    const double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / hh;
    const int g = gl_order(q, 0);
    cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
    pair4_f64(k, x, nx, c, st[f], snu[f], hh, g, S, Dv, K, T);
    dacc += ipow_phase(alpha, m) * (T * dens[2 * f] - eta * mul_i(K * dens[2 * f + 1]));
  }
  dacc = warp_sum(dacc);
  if ((tid & 31) == 0) s_red[tid >> 5] = dacc;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < FT_NT / 32; ++i) dacc += s_red[i];
    part[4 * (size_t)pi] = cplx{0, 0};
    part[4 * (size_t)pi + 1] = dacc;
  }
}

// The x1-derivative at many points through the multipoles of the leaves, of the same
// quadrature as the direct sum: a leaf enters as a whole where the ladder gives all its
// elements one rule g = 2, 3 or 4 (54 h <= r for g = 3, 790 h for 2; other leaves, and
// those nearer than the expansion allows, go element by element), by the multipoles of
// that rule's nodes, taken once per call (field_rules).  The expansion ends at the order
// q with (R / r)^q and (k R / 2)^q / q! below 10^-18: a dipole's remainder is q r / R
// times that, 10^-16 of the leaf's field.  The field u stays directly summed: where a
// density radiates almost nothing it cancels to 1e-8 of its terms, and any other rounding
// of these shows at 3e-9 to 9e-9 of u (of the derivative at 1e-10).
// A block takes slice sl of nsl of a point's (leaf, image) pairs; the pairs that go by
// elements are collected in shared memory and summed together when the list fills.
// Bound by the FP64 pipe: some 500 instructions a leaf, against 500 to 700 an element.
constexpr int FL_NT = 256, FL_CAP = 1024;
struct FieldLeaf {
  int nleaf, D, p, nmin;                 // nmin: order from which (k R / 2)^n / n! is below 1e-18
  double d, R, far2;                     // leaf side, radius, squared distance from which a leaf is far
  const int *ne, *bb, *be;
  const double2* ctr;
  const double2* hr;                     // [nleaf] shortest and longest element
  const cplx* M;                         // [3][nleaf][2p+1] multipoles of the rules 2, 3, 4
};

__global__ void leaf_lengths_kernel(int nleaf, const int* __restrict__ ne, const int* __restrict__ bb,
                                    const int* __restrict__ be, const double* __restrict__ sh,
                                    double2* __restrict__ hr) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nleaf) return;
  double lo = 1e300, hi = 0;
  for (int f = bb[ne[i]]; f < be[ne[i]]; ++f) {
    lo = fmin(lo, sh[f]);
    hi = fmax(hi, sh[f]);
  }
  hr[i] = double2{lo, hi};
}

__global__ void __launch_bounds__(FL_NT) field_leaf_kernel(
    const __grid_constant__ FieldLeaf fl, int npts, const double2* __restrict__ pts, int nsl, double k, double eta,
    double H, double ox, double oy, double x0, double y0, int mdir, cplx alpha, const double2* __restrict__ sc,
    const double2* __restrict__ st, const double2* __restrict__ snu, const double* __restrict__ sh,
    const cplx* __restrict__ dens, int p0, const double* __restrict__ w0, const cplx* __restrict__ L0,
    cplx* __restrict__ part) {
  if ((int)blockIdx.x >= npts * nsl) {
    local_part(((int)blockIdx.x - npts * nsl) * FL_NT + threadIdx.x, npts, pts, nsl, k, H, ox, oy, y0, p0, w0, L0,
               part);
    return;
  }
  __shared__ int s_li[FL_CAP], s_img[FL_CAP], s_off[FL_CAP + 1], s_n;
  __shared__ cplx s_red[FL_NT / 32];
  const int tid = threadIdx.x, lane = tid & 31, pi = blockIdx.x / nsl, sl = blockIdx.x - pi * nsl;
  const int nim = 2 * mdir + 1, jobs = fl.nleaf * nim, P = 2 * fl.p + 1;
  double2 x = pts[pi];
  x.y -= floor((x.y - y0) / H) * H;
  cplx dacc{0, 0};
  if (tid == 0) s_n = 0;
  __syncthreads();
  for (int base = sl * FL_NT; base < jobs; base += nsl * FL_NT) {
    const int t = base + tid;
    if (t < jobs) {
      const int li = t / nim, m = t - li * nim - mdir, box = fl.ne[li];
      double cx, cy;
      if (fl.ctr) {
        cx = fl.ctr[box].x;
        cy = fl.ctr[box].y;
      } else {
        morton_centre(box, fl.D, fl.d, x0, y0, cx, cy);
      }
      const double vx = x.x - cx, vy = x.y - (cy + m * H), r2 = vx * vx + vy * vy;
      const double2 hr = fl.hr[li];
      const double r = sqrt(r2), lo = (r - fl.R) * (1.0 - 1e-12), hi = (r + fl.R) * (1.0 + 1e-12);
      int g = 0;
      if (r2 >= fl.far2)
        for (int q = 2; q <= 4; ++q)
          if (lo >= c_glthr[0][q] * hr.y && hi < c_glthr[0][q - 1] * hr.x) g = q;
      if (g) {
        const int q = (int)ceilf(18.0f / log10f((float)(r / (fl.R + 0.5 * hr.y))));
        dacc += ipow_phase(alpha, m) * multipole_dx1(k, vx, vy, fl.p, min(fl.p, max(fl.nmin, q)), nullptr,
                                                     fl.M + ((size_t)(g - 2) * fl.nleaf + li) * P);
      } else {
        const int o = atomicAdd(&s_n, 1);          // below FL_CAP: a list of more than FL_CAP - FL_NT was emptied
        s_li[o] = li;
        s_img[o] = m;
      }
    }
    __syncthreads();
    const int nl = s_n;
    if (nl > 0 && (nl > FL_CAP - FL_NT || base + nsl * FL_NT >= jobs)) {
      if (tid < 32) {                              // first element of every entry
        int run = 0;
        for (int i0 = 0; i0 < nl; i0 += 32) {
          const int i = i0 + lane, box = i < nl ? fl.ne[s_li[i]] : 0;
          const int c = i < nl ? fl.be[box] - fl.bb[box] : 0;
          int v = c;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += n;
          }
          if (i < nl) s_off[i] = run + v - c;
          run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) s_off[nl] = run;
      }
      __syncthreads();
      const double2 nx{1.0, 0.0};
      for (int e = tid; e < s_off[nl]; e += FL_NT) {
        int lo = 0, hi = nl - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (s_off[mid] <= e) lo = mid;
          else hi = mid - 1;
        }
        const int f = fl.bb[fl.ne[s_li[lo]]] + e - s_off[lo], m = s_img[lo];
        double2 c = sc[f];
        c.y += m * H;
        const double hh = sh[f];
        const double q = sqrt((x.x - c.x) * (x.x - c.x) + (x.y - c.y) * (x.y - c.y)) / hh;
        cplx S{0, 0}, Dv{0, 0}, K{0, 0}, T{0, 0};
        pair4_f64(k, x, nx, c, st[f], snu[f], hh, gl_order(q, 0), S, Dv, K, T);
        dacc += ipow_phase(alpha, m) * (T * dens[2 * f] - eta * mul_i(K * dens[2 * f + 1]));
      }
      __syncthreads();
      if (tid == 0) s_n = 0;
    }
    __syncthreads();
  }
  dacc = warp_sum(dacc);
  if (lane == 0) s_red[tid >> 5] = dacc;
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < FL_NT / 32; ++i) dacc += s_red[i];
    cplx* o = part + 2 * ((size_t)pi * (nsl + 1) + sl);
    o[0] = cplx{0, 0};
    o[1] = dacc;
  }
}

// Whether the field goes by leaves: orders of the default rule and elements of at most a
// quarter of a leaf, as in field_tree, and points enough to pay for three rules'
// multipoles (nine nodes an element, the work of about seven points' direct sums).
static bool field_leaf(const pfmbem* h, int npts, FieldLeaf& fl) {
  const Level& L = h->lev[h->D];
  if (npts < 32 || h->hmax > 0.25 * L.d) return false;
  fl.R = (h->tree == 1 ? 0.5 : 0.5 * sqrt(2.0)) * L.d;
  const double kd = 2.0 * h->k * fl.R;
  if (kd < 1e-6 || L.p < 20 || L.p < kd + 1.8 * pow(10.0, 2.0 / 3.0) * cbrt(kd)) return false;
  const double far = (fl.R + 0.5 * h->hmax) / fmin(0.26, pow(10.0, -18.0 / (L.p + 1)));
  fl.far2 = far * far;
  fl.nleaf = L.nne;
  fl.D = h->D;
  fl.p = L.p;
  fl.d = L.d;
  fl.ne = L.ne;
  fl.bb = L.box_begin;
  fl.be = L.box_end;
  fl.ctr = L.ctr;
  double t = 1.0;
  for (fl.nmin = 0; fl.nmin < L.p && t > 1e-18; ++fl.nmin) t *= 0.25 * kd / (fl.nmin + 1);
  return true;
}

// Multipoles of the leaves by the rules 2, 3 and 4, and the leaves' element lengths.
static void field_rules(pfmbem* h, FieldLeaf& fl, cplx* M, double2* hr) {
  const Level& L = h->lev[h->D];
  leaf_lengths_kernel<<<(fl.nleaf + 127) / 128, 128, 0, h->stream>>>(fl.nleaf, fl.ne, fl.bb, fl.be, h->s_h, hr);
  for (int g = 2; g <= 4; ++g)
    p2m_f64_kernel<<<fl.nleaf, 128, 0, h->stream>>>(fl.ne, fl.bb, fl.be, h->D, L.d, L.p, nullptr, g, h->k, h->eta,
                                                    h->x0, h->y0, h->s_c, h->s_t, h->s_nu, h->s_h, h->dens,
                                                    M + (size_t)(g - 2) * fl.nleaf * L.P, L.ctr, true);
  fl.M = M;
  fl.hr = hr;
}

// The tree's levels for the derivative at theta_l, or false where the direct sum is
// kept: an order below 20 (whose theta would open nearly every box) or below
// the rule of the default orders (fixed orders; the expansion then need not
// converge at its distance), or elements longer than a quarter of a leaf.
static bool field_tree(const pfmbem* h, FieldTree& ft) {
  ft.D = h->D;
  ft.nroot = h->nroot;
  ft.nch0 = h->tree == 1 ? 6 : 4;
  if (h->hmax > 0.25 * h->lev[h->D].d) return false;
  for (int l = 0; l <= h->D; ++l) {
    const Level& L = h->lev[l];
    const double R = (h->tree == 1 ? 0.5 : 0.5 * sqrt(2.0)) * L.d, kd = 2.0 * h->k * R;
    if (L.p < 20 || L.p < kd + 1.8 * pow(10.0, 2.0 / 3.0) * cbrt(kd)) return false;
    const double far = (R + 0.5 * h->hmax) / fmin(0.26, pow(10.0, -18.0 / (L.p + 1)));
    ft.p[l] = L.p;
    ft.d[l] = L.d;
    ft.far2[l] = far * far;
    ft.w[l] = L.w_dev;
    ft.bb[l] = L.box_begin;
    ft.be[l] = L.box_end;
    ft.M[l] = L.M;
    ft.ctr[l] = L.ctr;
  }
  return true;
}

// with_u: the field itself is asked for (upward_f64's one_sum).
cudaError_t k_field_prepare(pfmbem* h, const cplx* psi, bool with_u) {
  upward_f64(h, psi, with_u);
  if (h->tree == 1) {
    // the super root's local expansion of the images |m| >= m0
    prof_begin(h, PH_LOCAL);
    k_wide_local(h);
    prof_end(h, PH_LOCAL);
  }
  return cudaGetLastError();
}

// Field at npts points; u and dudx1 hold npts values each (either may be null).
// by_tree: the derivative alone, through the tree where its orders allow it.
cudaError_t k_field(pfmbem* h, int npts, const double2* pts, cplx* u, cplx* dudx1, bool by_tree) {
  Level& r = h->lev[0];
  // the images beyond mdir: the root's local expansion, or the super root's
  const bool wide = h->nroot > 1;
  const double ox = wide ? h->wide_cx : h->x0 + 0.5 * h->H, oy = wide ? h->wide_cy : h->y0 + 0.5 * h->H;
  const int mdir = wide ? h->wide_m0 - 1 : 1, p0 = wide ? h->wide_ps : r.p;
  const double* w0 = wide ? h->wide_w : r.w_dev;
  const cplx* L0 = wide ? h->wide_ML + 2 * h->wide_ps + 1 : r.L;
  FieldTree ft;
  const bool tree = by_tree && !u && field_tree(h, ft);
  FieldLeaf fl;
  bool leaf = !tree && !u && field_leaf(h, npts, fl);
  // slices of a point's sum: about 32 warps per SM in all, at least 8 terms a lane; by
  // leaves about eight blocks per SM, at least a pair a thread
  auto slices = [&]() -> int {
    if (tree || u) return 1;      // u: one order of its sum (field_direct_kernel)
    const int64_t terms = (int64_t)(2 * mdir + 1) * (leaf ? fl.nleaf : h->E);
    return (int)std::max<int64_t>(1, std::min<int64_t>((PF_SMS * (leaf ? 8 : 32) + npts - 1) / npts, terms / 256));
  };
  int nsl = slices();
  void* buf = nullptr;
  size_t npart = 2 * (size_t)npts * (nsl + 1);
  const size_t nrule = leaf ? 3 * (size_t)fl.nleaf * (2 * fl.p + 1) : 0;
  cudaError_t e = cudaMallocAsync(&buf, sizeof(cplx) * (npart + nrule + (leaf ? fl.nleaf : 0)), h->stream);
  if (e == cudaErrorMemoryAllocation && leaf) {     // no room for the multipoles: element by element
    cudaGetLastError();
    leaf = false;
    nsl = slices();
    npart = 2 * (size_t)npts * (nsl + 1);
    e = cudaMallocAsync(&buf, sizeof(cplx) * npart, h->stream);
  }
  if (e != cudaSuccess) return e;
  cplx* part = static_cast<cplx*>(buf);
  prof_begin(h, PH_OUT);
  if (tree) {
    field_tree_kernel<<<npts + (npts + FT_NT - 1) / FT_NT, FT_NT, 0, h->stream>>>(
        ft, npts, pts, h->k, h->eta, h->H, ox, oy, h->x0, h->y0, mdir, h->alpha, h->s_c, h->s_t, h->s_nu, h->s_h,
        h->dens, p0, w0, L0, part);
  } else if (leaf) {
    field_rules(h, fl, part + npart, reinterpret_cast<double2*>(part + npart + nrule));
    field_leaf_kernel<<<npts * nsl + (npts + FL_NT - 1) / FL_NT, FL_NT, 0, h->stream>>>(
        fl, npts, pts, nsl, h->k, h->eta, h->H, ox, oy, h->x0, h->y0, mdir, h->alpha, h->s_c, h->s_t, h->s_nu, h->s_h,
        h->dens, p0, w0, L0, part);
  } else {
    const unsigned grid = (unsigned)((int64_t)npts * nsl + (npts + 31) / 32);
    auto launch = [&](auto kern) {
      kern<<<grid, 32, 0, h->stream>>>(npts, pts, nsl, h->E, h->k, h->eta, h->H, ox, oy, h->y0, mdir, h->alpha,
                                        h->s_c, h->s_t, h->s_nu, h->s_h, h->dens, p0, w0, L0, part);
    };
    if (u && dudx1) launch(field_direct_kernel<true, true>);
    else if (u) launch(field_direct_kernel<true, false>);
    else launch(field_direct_kernel<false, true>);
  }
  field_finish_kernel<<<(npts + 127) / 128, 128, 0, h->stream>>>(npts, pts, nsl, h->H, h->y0, h->alpha, part, u, dudx1);
  prof_end(h, PH_OUT);
  e = cudaGetLastError();
  const cudaError_t ef = cudaFreeAsync(buf, h->stream);
  return e != cudaSuccess ? e : ef;
}

// ---------------------------------------------------------------- Bragg coefficients
// Rayleigh amplitudes of the scattered field left/right of the block (from the
// spectral form of G_qp): with w = (+-k_n, kappa_n), kappa_n = k sin(theta) + 2 pi n/H,
// k_n = sqrt(k^2 - kappa_n^2),
//   u_n^+- = (i / (2 H k_n)) sum_e int_e [d/dnu_y e^{-i w.y} phi_e - i eta e^{-i w.y} varphi_e] ds,
// where the element integral of e^{-i w.y} over c + s t is e^{-i w.c} h sinc(w.t h / 2).
// Block (b, slice): order b / 2, side b % 2 (0: transmitted, 1: reflected); the
// blocks of one (order, side) split the elements and add their partial sums
// into out (zeroed by the caller).
__global__ void coeff_kernel(int E, double k, double eta, double H, double ks, const int* __restrict__ orders,
                             const double2* __restrict__ oc, const double2* __restrict__ ot,
                             const double2* __restrict__ onu, const double* __restrict__ oh,
                             const cplx* __restrict__ psi, cplx* __restrict__ out) {
  const int o = blockIdx.x >> 1, side = blockIdx.x & 1;
  const double kap = ks + 2.0 * M_PI * orders[o] / H;
  const double kn = sqrt(fmax(k * k - kap * kap, 0.0));
  const double wx = side == 0 ? kn : -kn, wy = kap;
  cplx acc{0, 0};
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < E; e += gridDim.y * blockDim.x) {
    const double2 c = oc[e], t = ot[e], nu = onu[e];
    const double hh = oh[e];
    const double a = 0.5 * hh * (wx * t.x + wy * t.y);
    const double sinc = fabs(a) < 1e-4 ? 1.0 - a * a / 6.0 : sin(a) / a;
    double s, co;
    sincos(wx * c.x + wy * c.y, &s, &co);
    const cplx ph{co, -s};
    const double wn = wx * nu.x + wy * nu.y;
    // -i (w.nu) phi - i eta varphi
    const cplx bra = mul_i(-(wn * psi[2 * e] + eta * psi[2 * e + 1]));
    acc += (hh * sinc) * (ph * bra);
  }
  acc = warp_sum(acc);
  __shared__ cplx red[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = acc;
  __syncthreads();
  if (wid == 0) {
    acc = lane < (blockDim.x >> 5) ? red[lane] : cplx{0, 0};
    acc = warp_sum(acc);
    if (lane == 0) {
      const cplx v = mul_i((1.0 / (2.0 * H * kn)) * acc);
      atomicAdd(&out[blockIdx.x].re, v.re);
      atomicAdd(&out[blockIdx.x].im, v.im);
    }
  }
}

// ---------------------------------------------------------------- ALU peak probe
// Eight independent FMA chains per thread; 2 flops per FMA.
template <class T>
__global__ void fma_probe_kernel(int iters, T a, T b, T* sink) {
  T x0 = threadIdx.x, x1 = x0 + 1, x2 = x0 + 2, x3 = x0 + 3, x4 = x0 + 4, x5 = x0 + 5, x6 = x0 + 6, x7 = x0 + 7;
#pragma unroll 4
  for (int i = 0; i < iters; ++i) {
    x0 = fma(x0, a, b); x1 = fma(x1, a, b); x2 = fma(x2, a, b); x3 = fma(x3, a, b);
    x4 = fma(x4, a, b); x5 = fma(x5, a, b); x6 = fma(x6, a, b); x7 = fma(x7, a, b);
  }
  T s = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
  if (s == (T)1.2345e-7) sink[0] = s;
}

extern "C" pfmbem_status pfmbem_probe_peak(int dtype, double* tflops) {
  if (!tflops || (dtype != 0 && dtype != 1)) return PFMBEM_EINVAL;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  void* sink = nullptr;
  if (cudaMalloc(&sink, 64) != cudaSuccess) return PFMBEM_ENOMEM;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int threads = 256, blocks = sms * 8;
  const int iters = dtype == 0 ? 1 << 14 : 1 << 16;
  float best = 1e30f;
  for (int rep = 0; rep < 4; ++rep) {
    cudaEventRecord(e0);
    if (dtype == 0) fma_probe_kernel<double><<<blocks, threads>>>(iters, 0.999999, 1e-7, (double*)sink);
    else fma_probe_kernel<float><<<blocks, threads>>>(iters, 0.999999f, 1e-7f, (float*)sink);
    cudaEventRecord(e1);
    cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    if (rep > 0 && ms < best) best = ms;
  }
  cudaError_t err = cudaGetLastError();
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(sink);
  if (err != cudaSuccess) return PFMBEM_ECUDA;
  const double flops = 2.0 * 8.0 * (double)iters * threads * blocks;
  *tflops = flops / (best * 1e-3) / 1e12;
  return PFMBEM_OK;
}

cudaError_t k_coefficients(pfmbem* h, const cplx* psi, int norders, const int* orders_dev, cplx* out_dev) {
  const int slices = std::min(64, (h->E + 255) / 256);
  cudaError_t e = cudaMemsetAsync(out_dev, 0, sizeof(cplx) * 2 * norders, h->stream);
  if (e != cudaSuccess) return e;
  prof_begin(h, PH_OUT);
  coeff_kernel<<<dim3(2 * norders, slices), 256, 0, h->stream>>>(h->E, h->k, h->eta, h->H, h->k * sin(h->theta),
                                                                 orders_dev, h->o_c, h->o_t, h->o_nu, h->o_h, psi,
                                                                 out_dev);
  prof_end(h, PH_OUT);
  return cudaGetLastError();
}
