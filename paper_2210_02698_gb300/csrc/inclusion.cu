// inclusion.cu - scattering by a curve inclusion on the device (Sec. 3.2).
//
// The curve C is cut into N_s straight segments with centres r^s_i, lengths
// w_i and refractive index n_i at the centres.  Eq. sie (the total field
// vanishes on C) enforced at the centres gives the surface system
// K^{s2s} P = K^{v2s} I (Eq. m_sie), and the total field at the cells is
//     U = (K^{v2v} + K^{s2v} (K^{s2s})^{-1} K^{v2s}) I        (Eq. m_v2v_inclu)
// with
//     K^{s2s}_ij = -g(r^s_i, r^s_j) w_j   (i != j)               (Eq. s2s)
//     K^{s2s}_ii = -(i w_i / 4)(1 + (2i/pi)(ln(gamma w n_i w_i / 4) - 1)),
//                  gamma = e^{gamma_E}: minus the integral over the segment
//                  of the small-argument form of (i/4) H0(w n_i |t|)
//     K^{v2s}_ij = g(r^s_i, r_j),   K^{s2v}_ij = g(r_i, r^s_j) w_j   (Eq. m_v2s, Eq. m_s2v)
// and g = v0 f0 + v1 f1 (Eq. babich) with tau^2, v0, v1 interpolated at the
// points from the tables (Eq. chebinterp), as for K^{v2v}.
//
// K^{v2s} and K^{s2v} are stored dense (2 N_s N_v complex values) or, after
// hb_curve_compress, as butterflies (curve_bf.cu); K^{s2s} is factored by
// LU with partial pivoting once per curve and inverted from the factors, so
// an apply is three products (dense, or butterfly - dense - butterfly) on
// top of the K^{v2v} apply (dense or compressed).
//
// Lengths may differ by any factor, and the products hold a factor row and a
// right-hand side to 58 bits of their largest value each (split_fixed.cuh), so
// the lengths' scale is kept out of them: with w_j = m_j p_j, p_j a power of two,
// the stored operators are diag(p) (K^{s2s})^{-1}, whose rows would else scale
// as 1 / w_i, and K^{s2v} diag(1 / p), applied to p P (exact: the same numbers
// otherwise).  Error of the inclusion's field, 200 equal chords of a circle
// with lengths graded by 1e6: 4.0e-11 with the lengths inside and one exponent a
// task, 1.2e-15 like this (equal lengths: 3.1e-15 and 2.7e-15).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "bessel.cuh"
#include "hb_internal.cuh"

namespace hb {

namespace {

constexpr int CMAX_NI = 16;                              // n_I supported (hb_create's limit)
constexpr double GAMMA_EXP = 1.78107241799019798524;     // e^{Euler's constant}
constexpr long long MAX_SEGMENTS = 16384;

struct PointTables {
  const double* nodes;   // nodes_x (n_I) then nodes_y (n_I)
  const double* tab;     // 3 x N_I x N_I forward tables, row = observation node
  int nI, NI;
  double omega;
};

// Lagrange basis l_k(x) of the n_I nodes in barycentric form (weights bw);
// at a node, the basis indicator.
__device__ __forceinline__ void basis_at(const double* nodes, const double* bw, int nI, double x, double* L) {
  int hit = -1;
  for (int k = 0; k < nI; ++k)
    if (x == nodes[k]) hit = k;
  if (hit >= 0) {
    for (int k = 0; k < nI; ++k) L[k] = (k == hit) ? 1.0 : 0.0;
    return;
  }
  double den = 0.0;
  for (int k = 0; k < nI; ++k) {
    L[k] = bw[k] / (x - nodes[k]);
    den += L[k];
  }
  for (int k = 0; k < nI; ++k) L[k] /= den;
}

// ---- the dense curve operators ----
// Every entry is g(seg, cell), g(cell, seg) or g(seg, seg'), so the tables are
// contracted with a segment's basis once, and the cells' tensor structure
// does the rest line by line: 48 FMAs and a tabulated Hankel pair (28) an
// entry.  (Contracting per source cell and evaluating the full basis and the
// recurrences per entry took 28.8 ms of FP64 at 96^2 with 300 segments.)

// lag[p][0..nI) = l_k(x_p), lag[p][16..16 + nI) = l_k(z_p) of segment centre p
__global__ void seg_basis_kernel(PointTables P, const double2* __restrict__ seg, long long ns, double* __restrict__ lag) {
  const long long p = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 1;
  const int d = threadIdx.x & 1;
  if (p >= ns) return;
  const double* nd = P.nodes + d * P.nI;
  double bw[CMAX_NI], L[CMAX_NI];
  for (int k = 0; k < P.nI; ++k) {
    double v = 1.0;
    for (int q = 0; q < P.nI; ++q)
      if (q != k) v *= (nd[k] - nd[q]);
    bw[k] = 1.0 / v;
  }
  basis_at(nd, bw, P.nI, d == 0 ? seg[p].x : seg[p].y, L);
  for (int k = 0; k < CMAX_NI; ++k) lag[(size_t)p * 32 + 16 * d + k] = k < P.nI ? L[k] : 0.0;
}

// G[((t 3 + q) N_I + i) ns + p] = sum_j tab_t[q][i][j] T_j(seg_p), T_j =
// l_{j1}(x) l_{j2}(z); t = 0: the tables (p a source), 1: transposed (p an
// observation point).  blockIdx.y = (t, q, i), lanes over segments.
__global__ void __launch_bounds__(128) seg_contract_kernel(PointTables P, const double* __restrict__ lag, long long ns,
                                                           double* __restrict__ G) {
  __shared__ double row[CMAX_NI * CMAX_NI];
  const int nI = P.nI, NI = P.NI;
  const double* f = P.tab + (size_t)blockIdx.y * NI;
  for (int j = threadIdx.x; j < NI; j += blockDim.x) row[j] = f[j];
  __syncthreads();
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ns) return;
  const double* l = lag + (size_t)p * 32;
  double lx[CMAX_NI];
#pragma unroll
  for (int k = 0; k < CMAX_NI; ++k) lx[k] = l[k];
  double acc = 0.0;
  for (int j2 = 0; j2 < nI; ++j2) {
    double a = 0.0;
#pragma unroll
    for (int j1 = 0; j1 < CMAX_NI; ++j1)
      if (j1 < nI) a = fma(row[j2 * nI + j1], lx[j1], a);
    acc = fma(l[16 + j2], a, acc);
  }
  G[(size_t)blockIdx.y * ns + p] = acc;
}

// g from interpolated tau^2, v0, v1 with the tabulated Hankel pair (as the
// dense apply): i c (v0 H0 - (2 / w^2) v1 x H1)
__device__ __forceinline__ double2 green_tab(const HankelTable& T, double omega, double t2, double v0, double v1) {
  const double c = 0.88622692545275801365;   // sqrt(pi)/2
  const double w2 = omega * omega, w2l = fma(omega, omega, -w2);
  const HankelFG h = hankel_of_t2(T, w2, w2l, t2);
  const double a = c * v0, b = (2.0 * c / w2) * v1;
  return make_double2(fma(-h.F.y, a, h.G.y * b), fma(h.F.x, a, -h.G.x * b));
}

// Segment p (one thread) against the cells [a0, a1) of grid line line0 + blockIdx.y.
// V2S: out[cell ns + p] = g(seg_p, cell) (G: the transposed contractions); else
// out[p Nv + cell] = w_p g(cell, seg_p) (16 bytes a lane at stride Nv: the L2 joins the halves of a
// sector before they leave it).
template <bool V2S>
__global__ void __launch_bounds__(64) seg_line_kernel(EntryParams E, const double* __restrict__ G, long long ns,
                                                      const double* __restrict__ w, int line0, double2* __restrict__ out) {
  const int nI = E.nI;
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ns) return;
  const int b = line0 + blockIdx.y;
  const double* lz = E.LZ + (size_t)b * nI;
  double P[3][CMAX_NI];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k1 = 0; k1 < CMAX_NI; ++k1) {
      double a = 0.0;
      if (k1 < nI)
        for (int k2 = 0; k2 < nI; ++k2) a = fma(lz[k2], G[(size_t)(q * E.NI + k2 * nI + k1) * ns + p], a);
      P[q][k1] = a;
    }
  const int a0 = (int)((long long)E.nx * blockIdx.z / gridDim.z), a1 = (int)((long long)E.nx * (blockIdx.z + 1) / gridDim.z);
  const double wp = V2S ? 1.0 : w[p];
  const long long Nv = (long long)E.nx * E.ny;
  for (int a = a0; a < a1; ++a) {
    const double* lx = E.LX + (size_t)a * nI;
    double f[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < CMAX_NI; ++k) {
      if (k < nI) {
        const double l = lx[k];
#pragma unroll
        for (int q = 0; q < 3; ++q) f[q] = fma(l, P[q][k], f[q]);
      }
    }
    const double2 g = green_tab(E.hank, E.omega, f[0], f[1], f[2]);
    const long long cell = (long long)b * E.nx + a;
    if (V2S) out[cell * ns + p] = g;
    else out[p * Nv + cell] = make_double2(wp * g.x, wp * g.y);
  }
}

// K^{s2s}: entry (i, j) = -w_j g(seg_i, seg_j), the diagonal the segment's own
// term.  One thread per i, blockIdx.y = j (G: the forward contractions).
__global__ void __launch_bounds__(128) seg_seg_kernel(EntryParams E, const double* __restrict__ lag,
                                                      const double* __restrict__ G, long long ns,
                                                      const double* __restrict__ w, const double* __restrict__ nseg,
                                                      double2* __restrict__ out) {
  __shared__ double g[3 * CMAX_NI * CMAX_NI];
  const int nI = E.nI, NI = E.NI;
  const long long j = blockIdx.y;
  for (int k = threadIdx.x; k < 3 * NI; k += blockDim.x) g[k] = G[(size_t)k * ns + j];
  __syncthreads();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ns) return;
  const double wj = w[j];
  double2 v;
  if (i == j) {
    const double c = (2.0 / HB_PI) * (log(GAMMA_EXP * E.omega * nseg[j] * wj / 4.0) - 1.0);
    v = make_double2(0.25 * wj * c, -0.25 * wj);   // -(i w/4)(1 + i c)
  } else {
    const double* l = lag + (size_t)i * 32;
    double lx[CMAX_NI];
#pragma unroll
    for (int k = 0; k < CMAX_NI; ++k) lx[k] = l[k];
    double f[3];
    for (int q = 0; q < 3; ++q) {
      double acc = 0.0;
      for (int i2 = 0; i2 < nI; ++i2) {
        double a = 0.0;
#pragma unroll
        for (int i1 = 0; i1 < CMAX_NI; ++i1)
          if (i1 < nI) a = fma(lx[i1], g[q * NI + i2 * nI + i1], a);
        acc = fma(l[16 + i2], a, acc);
      }
      f[q] = acc;
    }
    const double2 gr = green_tab(E.hank, E.omega, f[0], f[1], f[2]);
    v = make_double2(-wj * gr.x, -wj * gr.y);
  }
  out[(size_t)j * ns + i] = v;
}

// Batched columns of curve-operator blocks: job q (one CTA) writes
// out[J.out_off + a] = J.w g(obs[J.obs0 + a], J.src) for a < J.m - the
// evaluation of one entry at a time, by the recurrences, for sampled blocks
// whose rows are gathered into obs.
__global__ void __launch_bounds__(256) green_jobs_kernel(PointTables P, const double2* __restrict__ obs,
                                                         const GreenCol* __restrict__ jobs,
                                                         double2* __restrict__ out) {
  __shared__ double G[3 * CMAX_NI * CMAX_NI];
  __shared__ double bw[2][CMAX_NI];
  __shared__ double Ls[2][CMAX_NI];
  const int nI = P.nI, NI = P.NI, t = threadIdx.x;
  const GreenCol J = jobs[blockIdx.x];
  if (t < 2 * nI) {
    const int d = t / nI, k = t % nI;
    const double* nd = P.nodes + d * nI;
    double p = 1.0;
    for (int q = 0; q < nI; ++q)
      if (q != k) p *= (nd[k] - nd[q]);
    bw[d][k] = 1.0 / p;
  }
  __syncthreads();
  if (t < 2) basis_at(P.nodes + t * nI, bw[t], nI, t == 0 ? J.src.x : J.src.y, Ls[t]);
  __syncthreads();
  for (int idx = t; idx < 3 * NI; idx += blockDim.x) {
    const int q = idx / NI, i = idx % NI;
    const double* Fr = P.tab + ((size_t)q * NI + i) * NI;
    double acc = 0.0;
    for (int j2 = 0; j2 < nI; ++j2) {
      double a2 = 0.0;
      for (int j1 = 0; j1 < nI; ++j1) a2 = fma(Fr[j2 * nI + j1], Ls[0][j1], a2);
      acc = fma(Ls[1][j2], a2, acc);
    }
    G[idx] = acc;
  }
  __syncthreads();
  for (int a = t; a < J.m; a += blockDim.x) {
    const double2 o = obs[J.obs0 + a];
    double Lx[CMAX_NI], Lz[CMAX_NI];
    basis_at(P.nodes, bw[0], nI, o.x, Lx);
    basis_at(P.nodes + nI, bw[1], nI, o.y, Lz);
    double f[3];
    for (int q = 0; q < 3; ++q) {
      const double* Gq = G + q * NI;
      double acc = 0.0;
      for (int i2 = 0; i2 < nI; ++i2) {
        double a2 = 0.0;
        for (int i1 = 0; i1 < nI; ++i1) a2 = fma(Lx[i1], Gq[i2 * nI + i1], a2);
        acc = fma(Lz[i2], a2, acc);
      }
      f[q] = acc;
    }
    const double2 g = hb_green(f[0], f[1], f[2], P.omega);
    out[J.out_off + a] = make_double2(J.w * g.x, J.w * g.y);
  }
}

// ---- LU with partial pivoting, panels of LU_NB columns ----
// Per panel two launches: one CTA factors the panel (pivot p of column j =
// the row of the largest |A_ij|^2 over i >= j, lowest index on ties; rows
// interchanged, multipliers A_ij /= A_jj), then a CTA per strip of LU_CS other
// columns interchanges their rows and, right of the panel, solves with the
// panel's unit lower triangle and subtracts the products.  Panels are narrow
// because one SM's FP64 unit factors them (2 FMAs a cycle: 16 columns of 300
// rows took 188 us); strips are of 2 columns until they fill the chip.
constexpr int LU_NB = 4;
constexpr int LU_PT = 512;    // threads of the panel kernel
constexpr int LU_SB = 16;     // rows per block of the substitutions
inline int lu_strip(int columns) { return columns < 2 * 608 ? 2 : 8; }

__device__ __forceinline__ double2 csub_mul(double2 a, double2 l, double2 u) {   // a - l u
  a.x = fma(-l.x, u.x, fma(l.y, u.y, a.x));
  a.y = fma(-l.x, u.y, fma(-l.y, u.x, a.y));
  return a;
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__global__ void __launch_bounds__(LU_PT) lu_panel_kernel(double2* __restrict__ A, int n, int k0, int* __restrict__ piv,
                                                         int* __restrict__ singular) {
  __shared__ double wv[LU_PT / 32];
  __shared__ int wi[LU_PT / 32];
  __shared__ int s_p;
  __shared__ double2 urow[LU_NB];
  __shared__ double2 s_inv;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int nb = min(LU_NB, n - k0);
  auto at = [&](int i, int c) -> double2& { return A[(size_t)(k0 + c) * n + i]; };
  double best = -1.0;
  int bi = n;
  for (int i = k0 + t; i < n; i += LU_PT) {
    const double2 v = at(i, 0);
    const double m2 = v.x * v.x + v.y * v.y;
    if (m2 > best) {
      best = m2;
      bi = i;
    }
  }
  for (int j = 0; j < nb; ++j) {
    const int k = k0 + j;
    auto take = [&](double ov, int oi) {
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    };
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, bi, o));
    if (lane == 0) {
      wv[warp] = best;
      wi[warp] = bi;
    }
    __syncthreads();
    if (warp == 0) {
      best = lane < LU_PT / 32 ? wv[lane] : -1.0;
      bi = lane < LU_PT / 32 ? wi[lane] : n;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) take(__shfl_xor_sync(0xffffffffu, best, o), __shfl_xor_sync(0xffffffffu, bi, o));
      const bool zero = !(best > 0.0) || bi >= n;   // an all-zero (or NaN) column
      const int p = bi >= n ? k : bi;
      if (lane == 0) {
        s_p = p;
        piv[k] = p;
        if (zero) *singular = 1;
      }
      // the panel's rows k and p interchanged; row k from the pivot column on is U
      if (lane < nb) {
        const double2 a = at(k, lane), b = at(p, lane);
        if (p != k) {
          at(k, lane) = b;
          at(p, lane) = a;
        }
        urow[lane] = b;
        if (lane == j) {   // one warp divides: 16 of them would hold the FP64 unit for microseconds
          const double dd = b.x * b.x + b.y * b.y;
          s_inv = dd > 0.0 ? make_double2(b.x / dd, -b.y / dd) : make_double2(1.0, 0.0);
        }
      }
    }
    __syncthreads();
    best = -1.0;
    bi = n;
    const double2 inv = s_inv;
    for (int i = k + 1 + t; i < n; i += LU_PT) {
      const double2 l = cmul(at(i, j), inv);
      at(i, j) = l;
      for (int c = j + 1; c < nb; ++c) {
        const double2 v = csub_mul(at(i, c), l, urow[c]);
        at(i, c) = v;
        if (c == j + 1) {
          const double m2 = v.x * v.x + v.y * v.y;
          if (m2 > best) {
            best = m2;
            bi = i;
          }
        }
      }
    }
    __syncthreads();   // row k + 1 .. of the panel complete before the next interchange
  }
}

// Strip blockIdx.x of CS columns outside the panel [k0, k0 + nb).
template <int CS>
__global__ void __launch_bounds__(256) lu_strip_kernel(double2* __restrict__ A, int n, int k0, const int* __restrict__ piv) {
  __shared__ double2 U[LU_NB][CS];
  const int t = threadIdx.x, nb = min(LU_NB, n - k0);
  const int c0 = blockIdx.x * CS, nc = min(CS, n - nb - c0);
  auto col = [&](int c) { return A + (size_t)(c0 + c < k0 ? c0 + c : c0 + c + nb) * n; };   // skips the panel
  if (t < nc) {
    double2* a = col(t);
    for (int j = 0; j < nb; ++j) {
      const int p = piv[k0 + j];
      if (p != k0 + j) {
        const double2 v = a[k0 + j];
        a[k0 + j] = a[p];
        a[p] = v;
      }
    }
    if (c0 + t >= k0) {
      double2 u[LU_NB];
#pragma unroll
      for (int i = 0; i < LU_NB; ++i) {
        u[i] = make_double2(0.0, 0.0);
        if (i < nb) {
          u[i] = a[k0 + i];
#pragma unroll
          for (int j = 0; j < LU_NB; ++j)
            if (j < i) u[i] = csub_mul(u[i], A[(size_t)(k0 + j) * n + k0 + i], u[j]);
          a[k0 + i] = u[i];
        }
        U[i][t] = u[i];
      }
    }
  }
  if (c0 + nc <= k0) return;   // wholly left of the panel: interchanges only
  __syncthreads();
  for (int i = k0 + nb + t; i < n; i += 256) {
    double2 l[LU_NB];
#pragma unroll
    for (int j = 0; j < LU_NB; ++j) l[j] = j < nb ? A[(size_t)(k0 + j) * n + i] : make_double2(0.0, 0.0);
    for (int c = max(0, k0 - c0); c < nc; ++c) {
      double2* a = col(c) + i;
      double2 v = *a;
#pragma unroll
      for (int j = 0; j < LU_NB; ++j)
        if (j < nb) v = csub_mul(v, l[j], U[j][c]);
      *a = v;
    }
  }
}

// D[(2 b + up) SB^2 + c SB + r] = entry (r, c) of the inverse of diagonal
// block b's unit lower (up = 0) or upper triangle.  One warp per (b, up), lane = column.
__global__ void __launch_bounds__(32) lu_diag_kernel(const double2* __restrict__ A, int n, double2* __restrict__ D) {
  __shared__ double2 T[LU_SB][LU_SB];
  const int b0 = (blockIdx.x >> 1) * LU_SB, up = blockIdx.x & 1, nb = min(LU_SB, n - b0), c = threadIdx.x;
  for (int e = c; e < nb * nb; e += 32) T[e % nb][e / nb] = A[(size_t)(b0 + e / nb) * n + b0 + e % nb];
  __syncwarp();
  if (c >= LU_SB) return;
  double2* d = D + (size_t)blockIdx.x * LU_SB * LU_SB + c * LU_SB;
  double2 x[LU_SB];
#pragma unroll
  for (int k = 0; k < LU_SB; ++k) x[k] = make_double2(k == c && c < nb ? 1.0 : 0.0, 0.0);
  if (!up) {
#pragma unroll
    for (int i = 0; i < LU_SB; ++i)
#pragma unroll
      for (int j = 0; j < LU_SB; ++j)
        if (j < i && i < nb) x[i] = csub_mul(x[i], T[i][j], x[j]);
  } else {
#pragma unroll
    for (int i = LU_SB - 1; i >= 0; --i) {
      if (i < nb) {
#pragma unroll
        for (int j = 0; j < LU_SB; ++j)
          if (j > i && j < nb) x[i] = csub_mul(x[i], T[i][j], x[j]);
        const double2 q = T[i][i], v = x[i];
        const double dd = q.x * q.x + q.y * q.y;
        x[i] = make_double2((v.x * q.x + v.y * q.y) / dd, (v.y * q.x - v.x * q.y) / dd);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < LU_SB; ++k) d[k] = x[k];
}

// Y = A^{-1} (Y zero before) with those factors and diagonal inverses, a CTA
// per strip of CS columns of Y (leading dimension n): the unit columns through
// the interchanges, then the unit lower (from the first non-zero block on) and
// the upper triangular substitutions by blocks of LU_SB rows.
template <int CS>
__global__ void __launch_bounds__(256) lu_inverse_kernel(const double2* __restrict__ A, const double2* __restrict__ D,
                                                       const int* __restrict__ piv, int n, double2* __restrict__ Y) {
  __shared__ double2 B[LU_SB][CS];
  __shared__ double2 X[LU_SB][CS];
  const int t = threadIdx.x;
  __shared__ int first;
  const int c0 = blockIdx.x * CS, nc = min(CS, n - c0);
  if (t == 0) first = n;
  __syncthreads();
  if (t < nc) {
    int r = c0 + t;
    for (int k = 0; k < n; ++k) {
      const int p = piv[k];
      r = r == k ? p : r == p ? k : r;
    }
    Y[(size_t)(c0 + t) * n + r] = make_double2(1.0, 0.0);
    atomicMin(&first, r);
  }
  __syncthreads();
  const int blocks = (n + LU_SB - 1) / LU_SB;
  for (int s = first / LU_SB; s < 2 * blocks; ++s) {
    const bool upper = s >= blocks;
    const int bk = upper ? 2 * blocks - 1 - s : s, b0 = LU_SB * bk, nb = min(LU_SB, n - b0);
    const int r = t % LU_SB, c = t / LU_SB;   // entry of the block's solution
    if (c < CS) B[r][c] = (c < nc && r < nb) ? Y[(size_t)(c0 + c) * n + b0 + r] : make_double2(0.0, 0.0);
    __syncthreads();
    if (c < CS) {
      const double2* d = D + (size_t)(2 * bk + (upper ? 1 : 0)) * LU_SB * LU_SB + r;
      double2 v = make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < LU_SB; ++j) v = csub_mul(v, d[j * LU_SB], make_double2(-B[j][c].x, -B[j][c].y));
      X[r][c] = v;
      if (c < nc && r < nb) Y[(size_t)(c0 + c) * n + b0 + r] = v;
    }
    __syncthreads();
    const int i0 = upper ? 0 : b0 + nb, i1 = upper ? b0 : n;
    for (int i = i0 + t; i < i1; i += 256) {
      double2 l[LU_SB];
#pragma unroll
      for (int j = 0; j < LU_SB; ++j) l[j] = j < nb ? A[(size_t)(b0 + j) * n + i] : make_double2(0.0, 0.0);
      for (int q = 0; q < nc; ++q) {
        double2* y = Y + (size_t)(c0 + q) * n + i;
        double2 v = *y;
#pragma unroll
        for (int j = 0; j < LU_SB; ++j) v = csub_mul(v, l[j], X[j][q]);
        *y = v;
      }
    }
    __syncthreads();
  }
}

// row i of the n x n matrix A times p[i]
__global__ void __launch_bounds__(256) scale_rows_kernel(double2* __restrict__ A, long long n, const double* __restrict__ p) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += (long long)gridDim.x * blockDim.x) {
    const double s = p[e % n];
    A[e] = make_double2(s * A[e].x, s * A[e].y);
  }
}

PointTables point_tables(const hb_ctx* c) {
  PointTables P;
  P.nodes = c->d_nodes;
  P.tab = c->d_tab;
  P.nI = c->nI;
  P.NI = c->NI;
  P.omega = c->omega;
  return P;
}

// The three surface operators into column-major outputs (any may be null),
// the columns of K^{s2v} times w_s2v.
void assemble(const hb_ctx* c, double2* k_s2s, double2* k_v2s, double2* k_s2v, const double* w_s2v, cudaStream_t st) {
  const EntryParams E = entry_params(c, 0);
  const long long ns = c->ns_set;
  const double* G0 = c->d_segG;
  const double* G1 = c->d_segG + (size_t)3 * c->NI * ns;
  // lines cut so that a small curve still fills the chip (about 8 warps an SM)
  const long long warps = (ns + 31) / 32 * c->ny;
  const unsigned cut = (unsigned)std::max<long long>(1, std::min<long long>((1216 + warps - 1) / warps, (c->nx + 15) / 16));
  auto lines = [&](int b0) { return dim3((unsigned)((ns + 63) / 64), (unsigned)std::min(65535, c->ny - b0), cut); };
  if (k_s2s) {
    seg_seg_kernel<<<dim3((unsigned)((ns + 127) / 128), (unsigned)ns), 128, 0, st>>>(E, c->d_seglag, G0, ns, c->d_segw,
                                                                                    c->d_segn, k_s2s);
    HB_CHECK_LAUNCH();
  }
  if (k_v2s) {
    for (int b0 = 0; b0 < c->ny; b0 += 65535) {
      seg_line_kernel<true><<<lines(b0), 64, 0, st>>>(E, G1, ns, c->d_segw, b0, k_v2s);
      HB_CHECK_LAUNCH();
    }
  }
  if (k_s2v) {
    for (int b0 = 0; b0 < c->ny; b0 += 65535) {
      seg_line_kernel<false><<<lines(b0), 64, 0, st>>>(E, G0, ns, w_s2v, b0, k_s2v);
      HB_CHECK_LAUNCH();
    }
  }
}

}  // namespace

void green_jobs(const hb_ctx* c, const double2* d_obs, const GreenCol* d_jobs, long long njobs, double2* d_out,
                cudaStream_t st) {
  const PointTables P = point_tables(c);
  for (long long b0 = 0; b0 < njobs; b0 += (1LL << 30)) {
    const unsigned n = (unsigned)std::min<long long>(njobs - b0, 1LL << 30);
    green_jobs_kernel<<<n, 256, 0, st>>>(P, d_obs, d_jobs + b0, d_out);
    HB_CHECK_LAUNCH();
  }
}

void curve_free(hb_ctx* c) {
  for (void* p : {(void*)c->d_seg, (void*)c->d_segw, (void*)c->d_segn, (void*)c->d_lu, (void*)c->d_piv,
                  (void*)c->d_kv2s, (void*)c->d_ks2v, (void*)c->d_cy, (void*)c->d_inv, (void*)c->d_seglag,
                  (void*)c->d_segG, (void*)c->d_pack, (void*)c->d_segm})
    dev_free(p);
  dense_op_free(c->op_v2s);
  dense_op_free(c->op_inv);
  dense_op_free(c->op_s2v);
  c->d_seglag = c->d_segG = nullptr;
  c->d_pack = nullptr;
  c->ns_set = 0;
  c->d_inv = nullptr;
  c->d_seg = nullptr;
  c->d_segw = c->d_segn = c->d_segm = c->d_segp = nullptr;
  c->d_lu = c->d_kv2s = c->d_ks2v = c->d_cy = nullptr;
  c->d_piv = nullptr;
  c->ns = 0;
  c->cy_cap = 0;
  curve_bf_free(c);
}

void curve_set(hb_ctx* c, const double* centers, const double* lengths, const double* n_seg, long long ns) {
  if (!centers || !lengths || !n_seg) throw arg_error("null curve array");
  if (ns < 1 || ns > MAX_SEGMENTS) throw arg_error("segments %lld outside [1, %lld]", ns, MAX_SEGMENTS);
  for (long long i = 0; i < ns; ++i) {
    if (!std::isfinite(centers[2 * i]) || !std::isfinite(centers[2 * i + 1]))
      throw arg_error("segment %lld: centre not finite", i);
    if (!(lengths[i] > 0) || !std::isfinite(lengths[i])) throw arg_error("segment %lld: length must be positive", i);
    if (!(n_seg[i] > 0) || !std::isfinite(n_seg[i])) throw arg_error("segment %lld: n must be positive", i);
  }
  curve_free(c);   // a curve replaces the previous one; on failure the handle has none
  try {
    std::vector<double2> cen((size_t)ns);
    for (long long i = 0; i < ns; ++i) cen[(size_t)i] = make_double2(centers[2 * i], centers[2 * i + 1]);
    c->d_seg = upload(cen);
    c->d_segw = upload(std::vector<double>(lengths, lengths + ns));
    c->d_segn = upload(std::vector<double>(n_seg, n_seg + ns));
    std::vector<double> mp(2 * (size_t)ns);
    for (long long i = 0; i < ns; ++i) {
      mp[(size_t)(ns + i)] = std::ldexp(1.0, std::ilogb(lengths[i]));
      mp[(size_t)i] = lengths[i] / mp[(size_t)(ns + i)];
    }
    c->d_segm = upload(mp);
    c->d_segp = c->d_segm + ns;
    c->ns_set = ns;
    c->d_seglag = dev_alloc<double>((size_t)ns * 32);
    c->d_segG = dev_alloc<double>((size_t)6 * c->NI * ns);
    const PointTables P = point_tables(c);
    seg_basis_kernel<<<(unsigned)((2 * ns + 127) / 128), 128>>>(P, c->d_seg, ns, c->d_seglag);
    HB_CHECK_LAUNCH();
    seg_contract_kernel<<<dim3((unsigned)((ns + 127) / 128), (unsigned)(6 * c->NI)), 128>>>(P, c->d_seglag, ns, c->d_segG);
    HB_CHECK_LAUNCH();
    c->d_lu = dev_alloc<double2>((size_t)ns * ns);
    c->d_piv = dev_alloc<int>((size_t)ns);
    c->d_kv2s = dev_alloc<double2>((size_t)ns * c->Nv);
    c->d_ks2v = dev_alloc<double2>((size_t)ns * c->Nv);
    std::vector<int> zero(1, 0);
    int* d_sing = upload(zero);
    try {
      assemble(c, c->d_lu, c->d_kv2s, c->d_ks2v, c->d_segm, 0);
      const int n = (int)ns;
      for (int k = 0; k < n; k += LU_NB) {
        lu_panel_kernel<<<1, LU_PT>>>(c->d_lu, n, k, c->d_piv, d_sing);
        HB_CHECK_LAUNCH();
        const int others = n - std::min(LU_NB, n - k);
        if (others > 0) {
          if (lu_strip(n) == 2) lu_strip_kernel<2><<<(unsigned)((others + 1) / 2), 256>>>(c->d_lu, n, k, c->d_piv);
          else lu_strip_kernel<8><<<(unsigned)((others + 7) / 8), 256>>>(c->d_lu, n, k, c->d_piv);
          HB_CHECK_LAUNCH();
        }
      }
      HB_CUDA(cudaDeviceSynchronize());
      int sing = 0;
      HB_CUDA(cudaMemcpy(&sing, d_sing, sizeof(int), cudaMemcpyDeviceToHost));
      if (sing) throw Error{HB_ERR_ARG, "K^{s2s} is singular: a zero pivot in its LU factorisation"};
      // the inverse, column by column from the factors (an apply is then one
      // product instead of two sequential triangular solves per column)
      c->d_inv = dev_alloc<double2>((size_t)ns * ns);
      HB_CUDA(cudaMemsetAsync(c->d_inv, 0, sizeof(double2) * (size_t)ns * ns));
      const int diag = 2 * ((n + LU_SB - 1) / LU_SB);
      double2* d_diag = dev_alloc<double2>((size_t)diag * LU_SB * LU_SB);
      lu_diag_kernel<<<(unsigned)diag, 32>>>(c->d_lu, n, d_diag);
      if (lu_strip(n) == 2) lu_inverse_kernel<2><<<(unsigned)((n + 1) / 2), 256>>>(c->d_lu, d_diag, c->d_piv, n, c->d_inv);
      else lu_inverse_kernel<8><<<(unsigned)((n + 7) / 8), 256>>>(c->d_lu, d_diag, c->d_piv, n, c->d_inv);
      scale_rows_kernel<<<(unsigned)std::min<long long>((ns * ns + 255) / 256, 152LL * 16), 256>>>(c->d_inv, ns, c->d_segp);
      const cudaError_t le = cudaGetLastError(), se = cudaDeviceSynchronize();
      dev_free(d_diag);
      HB_CUDA(le);
      HB_CUDA(se);
      c->op_v2s = dense_op(c->d_kv2s, ns, c->Nv, 0);
      c->op_inv = dense_op(c->d_inv, ns, ns, 0);
      c->op_s2v = dense_op(c->d_ks2v, c->Nv, ns, 0);
      size_t rows = 0;
      for (const DenseOp* D : {&c->op_v2s, &c->op_inv, &c->op_s2v})
        rows = std::max(rows, dense_op_rows(*D));
      c->d_pack = dev_alloc<double2>(rows * 16);
    } catch (...) {
      cudaDeviceSynchronize();
      dev_free(d_sing);
      throw;
    }
    dev_free(d_sing);
    c->ns = ns;
  } catch (...) {
    curve_free(c);
    throw;
  }
}

void curve_operators(hb_ctx* c, double2* k_s2s, double2* k_v2s, double2* k_s2v, cudaStream_t st) {
  if (c->ns == 0) throw Error{HB_ERR_STATE, "no curve set (hb_curve_set)"};
  assemble(c, k_s2s, k_v2s, k_s2v, c->d_segw, st);
}

void apply_inclusion(hb_ctx* c, const double2* s, double2* u, int nrhs, int v2v_dense, cudaStream_t st) {
  NvtxRange nr("hb_apply_inclusion");
  if (c->ns == 0) throw Error{HB_ERR_STATE, "no curve set (hb_curve_set)"};
  if (!v2v_dense && !c->built) throw Error{HB_ERR_STATE, "compressed K^{v2v} before hb_build"};
  if (c->cy_cap < nrhs) {
    dev_free(c->d_cy);
    c->d_cy = nullptr;
    c->cy_cap = 0;
    c->d_cy = dev_alloc<double2>((size_t)c->ns * nrhs * 2);
    c->cy_cap = nrhs;
    HB_CUDA(cudaDeviceSynchronize());
  }
  // U = K^{v2v} I
  if (v2v_dense) dense_apply(c, s, u, nrhs, 0, st);
  else apply_bf(c, s, u, nrhs, 0, c->opt.precision, st);
  const long long ns = c->ns;
  auto product = [&](const DenseOp& D, const double2* X, long long ldx, double2* Y, long long ldy, double alpha,
                     int accumulate) {   // 16 columns at a time
    for (int r0 = 0; r0 < nrhs; r0 += 16)
      dense_product(D, X + (size_t)r0 * ldx, ldx, Y + (size_t)r0 * ldy, ldy, std::min(16, nrhs - r0), alpha, accumulate,
                    c->d_pack, c->d_pack + (size_t)D.k * 16, st);
  };
  const bool compressed = c->curve_bf[0] && c->curve_bf[1];
  // Y = K^{v2s} I = h^2 K^{v2s} s
  if (compressed) curve_bf_apply(c, 0, s, c->Nv, c->h * c->h, c->d_cy, ns, 0, nrhs, st);
  else product(c->op_v2s, s, c->Nv, c->d_cy, ns, c->h * c->h, 0);
  // p P = diag(p) (K^{s2s})^{-1} Y
  double2* P = c->d_cy + (size_t)ns * nrhs;
  product(c->op_inv, c->d_cy, ns, P, ns, 1.0, 0);
  // U += K^{s2v} P = (K^{s2v} diag(1 / p)) (p P)
  if (compressed) curve_bf_apply(c, 1, P, ns, 1.0, u, c->Nv, 1, nrhs, st);
  else product(c->op_s2v, P, ns, u, c->Nv, 1.0, 1);
}

}  // namespace hb
