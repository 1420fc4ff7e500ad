// entries.cu - evaluation of the HB matrix entries K_ij on the device
// (Sec. 3.1 Eq. m_v2v; Sec. 4.1 Eq. chebinterp / Eq. chebinterpblock;
// Eq. babich with N = 1; Eq. termf; Appendix A Eq. HankelIntegral2dlemma),
// and the matrix-free dense apply U = K I and its adjoint.
//
// Interpolation layout.  With T_i(r) = l_{i1}(x) l_{i2}(z) and the grid's
// cell coordinates x_a, z_b, the tensor structure of Eq. chebinterp is
// contracted in stages so that each entry costs O(n_I) FP64 FMAs per
// ingredient instead of O(N_I^2):
//   LX[a][k] = l_k(x_a), LZ[b][k] = l_k(z_b)                     (barycentric)
//   H[q][b][i][j1] = sum_{j2} F_q[i][(j2,j1)] LZ[b][j2]          (per source line b)
//   G_j[q][i]      = sum_{j1} H[q][b_j][i][j1] LX[a_j][j1]        (= (F_q T(r_j))_i)
//   P[q][i1]       = sum_{i2} LZ[b_i][i2] G_j[q][(i2,i1)]         (per observation line)
//   f_q(r_i, r_j)  = sum_{i1} LX[a_i][i1] P[q][i1]
// q = 0, 1, 2 for tau^2, v0, v1.  The adjoint uses the transposed tables.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "bessel.cuh"
#include "hb_internal.cuh"

namespace hb {

constexpr int MAX_NI = 16;   // n_I supported by the fused kernels

// ----------------------------------------------------------- helpers ----
// Barycentric Lagrange basis at the coordinates of one grid axis.
__global__ void lagrange_kernel(const double* __restrict__ nodes, int nI, double origin,
                                double h, int count, double* __restrict__ L) {
  int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= count) return;
  double x = origin + (a + 0.5) * h;
  double w[MAX_NI], d[MAX_NI];
  int hit = -1;
  for (int k = 0; k < nI; ++k) {
    double p = 1.0;
    for (int m = 0; m < nI; ++m)
      if (m != k) p *= (nodes[k] - nodes[m]);
    w[k] = 1.0 / p;
    d[k] = x - nodes[k];
    if (d[k] == 0.0) hit = k;
  }
  if (hit >= 0) {
    for (int k = 0; k < nI; ++k) L[(size_t)a * nI + k] = (k == hit) ? 1.0 : 0.0;
    return;
  }
  double den = 0.0;
  for (int k = 0; k < nI; ++k) den += w[k] / d[k];
  for (int k = 0; k < nI; ++k) L[(size_t)a * nI + k] = (w[k] / d[k]) / den;
}

// H[q][b][i][j1] = sum_j2 F_q[i][j2*nI + j1] LZ[b][j2]
__global__ void htable_kernel(const double* __restrict__ F, const double* __restrict__ LZ, int ny,
                              int nI, double* __restrict__ H) {
  const int NI = nI * nI;
  long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long total = 3LL * ny * NI * nI;
  if (idx >= total) return;
  int j1 = idx % nI;
  long long t = idx / nI;
  int i = t % NI;
  t /= NI;
  int b = t % ny;
  int q = (int)(t / ny);
  const double* Fq = F + (size_t)q * NI * NI + (size_t)i * NI;
  double acc = 0.0;
  for (int j2 = 0; j2 < nI; ++j2) acc = fma(Fq[j2 * nI + j1], LZ[(size_t)b * nI + j2], acc);
  H[idx] = acc;
}

// Self term K_ii = (i/4) I / h^2, I = (n0 w)^-2 [8 int_0^{pi/4} R H1(R) dth + 4i],
// R = h n0 w / (2 cos th)  (Appendix A); theta quadrature: Gauss-Legendre.
// A CTA takes SELF_CELLS cells: its threads evaluate the points of the rule, then
// one thread per cell adds them in order (one thread per cell throughout left
// most SMs without work on small grids).
constexpr int SELF_NGL = 64, SELF_CELLS = 4;
__global__ void __launch_bounds__(SELF_NGL * SELF_CELLS) self_kernel(const double* __restrict__ ncell, long long Nv, double h,
                                                                     double omega, const double* __restrict__ glx,
                                                                     const double* __restrict__ glw,
                                                                     double2* __restrict__ out) {
  __shared__ double2 val[SELF_CELLS][SELF_NGL];   // R J1(R), R Y1(R)
  const int cell = threadIdx.x / SELF_NGL, g = threadIdx.x % SELF_NGL;
  const long long i = (long long)blockIdx.x * SELF_CELLS + cell;
  const double n0 = ncell[i < Nv ? i : Nv - 1];
  {
    const double k = 0.5 * h * n0 * omega;
    const double th = (HB_PI / 8.0) * (glx[g] + 1.0);   // map [-1,1] -> [0, pi/4]
    const double R = k / cos(th);
    const Bessel01 b = bessel01(R);
    val[cell][g] = make_double2(R * b.j1, R * b.y1);
  }
  __syncthreads();
  if (g != 0 || i >= Nv) return;
  double re = 0.0, im = 0.0;
  for (int q = 0; q < SELF_NGL; ++q) {
    re = fma(glw[q], val[cell][q].x, re);
    im = fma(glw[q], val[cell][q].y, im);
  }
  re *= HB_PI / 8.0;
  im *= HB_PI / 8.0;
  double s = 1.0 / ((n0 * omega) * (n0 * omega));
  double Ire = s * 8.0 * re;
  double Iim = s * (8.0 * im + 4.0);
  // (i/4)(Ire + i Iim) / h^2
  out[i] = make_double2(-0.25 * Iim / (h * h), 0.25 * Ire / (h * h));
}

// Gauss-Legendre nodes/weights on [-1,1] by Newton iteration on P_n.
static void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(HB_PI * (i + 0.75) / (n + 0.5));
    double dp = 0.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    double p0 = 1.0, p1 = z;
    for (int k = 2; k <= n; ++k) {
      double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    dp = n * (z * p1 - p0) / (z * z - 1.0);
    x[i] = z;
    w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

void setup_tables(hb_ctx* c) {
  const int nI = c->nI, NI = c->NI;
  std::vector<double> nodes(c->nodes_x);
  nodes.insert(nodes.end(), c->nodes_y.begin(), c->nodes_y.end());
  c->d_nodes = upload(nodes);
  std::vector<double> tabs((size_t)6 * NI * NI);
  for (int q = 0; q < 3; ++q)
    for (int i = 0; i < NI; ++i)
      for (int j = 0; j < NI; ++j) {
        tabs[(size_t)q * NI * NI + (size_t)i * NI + j] = c->tab[q][(size_t)i * NI + j];
        tabs[(size_t)(3 + q) * NI * NI + (size_t)i * NI + j] = c->tab[q][(size_t)j * NI + i];
      }
  c->d_tab = upload(tabs);
  c->d_LX = dev_alloc<double>((size_t)c->nx * nI);
  c->d_LZ = dev_alloc<double>((size_t)c->ny * nI);
  lagrange_kernel<<<(c->nx + 127) / 128, 128>>>(c->d_nodes, nI, c->x0, c->h, c->nx, c->d_LX);
  HB_CHECK_LAUNCH();
  lagrange_kernel<<<(c->ny + 127) / 128, 128>>>(c->d_nodes + nI, nI, c->y0, c->h, c->ny, c->d_LZ);
  HB_CHECK_LAUNCH();
  long long htotal = 3LL * c->ny * NI * nI;
  for (int t = 0; t < 2; ++t) {
    c->d_H[t] = dev_alloc<double>(htotal);
    htable_kernel<<<(unsigned)((htotal + 255) / 256), 256>>>(c->d_tab + (size_t)t * 3 * NI * NI,
                                                            c->d_LZ, c->ny, nI, c->d_H[t]);
    HB_CHECK_LAUNCH();
  }
  c->d_ncell = upload(c->n_cells);
  compute_self(c);
}

// At least `need` rows of Hankel expansions.  A row depends on its place alone,
// so an array serves every frequency that it is long enough for; a longer one
// (at least twice, up to HT_CAP: no more than 62 MB in all) takes its place
// and the outgrown one stays until the handle is destroyed, for graphs that
// were captured with it.
static void hankel_rows(hb_ctx* c, int need) {
  if (need <= c->hank_rows) return;
  const int most = (int)std::ceil((HT_CAP - HT_LO) * HT_PER) + 2;
  const int rows = std::max(need, std::min(2 * c->hank_rows, most));
  c->hank_old.reserve(c->hank_old.size() + 1);
  double2* d = dev_alloc<double2>((size_t)rows * HT_ROW);
  hankel_table_kernel<<<(rows + 31) / 32, 32>>>(d, rows);   // one warp an SM: a serial FP64 chain a row
  if (cudaGetLastError() != cudaSuccess) {
    dev_free(d);
    throw Error{HB_ERR_CUDA, "the Hankel expansions could not be computed"};
  }
  if (c->d_hank) c->hank_old.push_back(c->d_hank);
  c->d_hank = d;
  c->hank_rows = rows;
}

// The precomputed entry data that depends on omega (the tables do not): the
// cell-integrated self terms into d_self (allocated on first use) and the
// Hankel expansions of the dense apply.  What can fail for lack of memory
// comes before anything that the handle uses changes.
void compute_self(hb_ctx* c) {
  if (!c->d_self) c->d_self = dev_alloc<double2>(c->Nv);
  if (!c->d_dense_ex) c->d_dense_ex = dev_alloc<int>(17);
  // the expansions of the Hankel pair up to the largest omega tau of the
  // tables (and a tenth of tau^2 more, for cells outside the node hull; past
  // the rows the kernels use the asymptotic series)
  double t2max = 0.0;
  for (double v : c->tab[0]) t2max = std::max(t2max, v);
  const double top = std::min(HT_CAP, c->omega * std::sqrt(1.1 * t2max) + 1.0);
  hankel_rows(c, top > HT_LO ? (int)std::ceil((top - HT_LO) * HT_PER) + 2 : 0);
  std::vector<double> glx, glw;
  gauss_legendre(SELF_NGL, glx, glw);
  // the quadrature rule is scratch: freed on the way out, also when a step throws
  double* d_gl = upload(glx);
  double* d_gw = nullptr;
  try {
    d_gw = upload(glw);
    self_kernel<<<(unsigned)((c->Nv + SELF_CELLS - 1) / SELF_CELLS), SELF_NGL * SELF_CELLS>>>(
        c->d_ncell, c->Nv, c->h, c->omega, d_gl, d_gw, c->d_self);
    HB_CHECK_LAUNCH();
    HB_CUDA(cudaDeviceSynchronize());
  } catch (...) {
    dev_free(d_gl);
    dev_free(d_gw);
    throw;
  }
  dev_free(d_gl);
  dev_free(d_gw);
  c->hank_top = top > HT_LO ? (float)top : 0.0f;
}

EntryParams entry_params(const hb_ctx* c, int transposed) {
  EntryParams p;
  p.nx = c->nx;
  p.ny = c->ny;
  p.nI = c->nI;
  p.NI = c->NI;
  p.omega = c->omega;
  p.LX = c->d_LX;
  p.LZ = c->d_LZ;
  p.H = c->d_H[transposed ? 1 : 0];
  p.self = c->d_self;
  p.hank = HankelTable{c->d_hank, c->hank_top};
  return p;
}

// ------------------------------------------------------- dense apply ----
// The form in plain FP64 FMAs, for values that the digits of dense_split.cu do
// not hold (not finite, or below 2^-960): it runs where that kernel marked a
// right-hand side of the pass (bit bit0 + r of *flag) and writes the marked ones.
//
// One CTA owns the L <= 64 cells of one segment of a grid line (the outputs; a
// line is cut into equal segments) and sweeps the source line segments of L
// cells of its share of the source lines (blockIdx.y of gridDim.y contiguous
// shares; all lines when gridDim.y = 1).  Thread t: output t mod L, group
// t / L takes every (256 / L)-th source of the segment.  RC right-hand sides
// per pass.  FP64 throughout.  With one share the CTA writes u; with several
// it writes its unscaled partial sums to part[share][r][cell] and
// dense_reduce_kernel adds the shares in order.
//
// Bound by the FP64 unit (2 FMAs a cycle and SM).  Per entry: 3 KI for the
// observation contraction (the basis values in registers, the source's P
// broadcast from shared memory), 28 for the Hankel pair (hankel_table.cuh)
// and 4 RC.  sqrt(pi)/2 and the factors of f1 are folded into P.  Measured:
// 64^2, one right-hand side 3.3 ms, 144 x 100 with 16 (adjoint) 62 ms.
constexpr int DT = 64;
constexpr double HB_C0 = 0.88622692545275801365;   // sqrt(pi)/2

template <int RC, bool ADJ, int KI>
__global__ void __launch_bounds__(256, RC <= 4 ? 2 : 1) dense_kernel(EntryParams p, const double2* __restrict__ s,
                                                    double2* __restrict__ u, long long Nv, int L, int r0,
                                                    double scale, double2* __restrict__ part,
                                                    const int* __restrict__ flag, int bit0) {
  extern __shared__ double smem[];
  const int marked = *flag >> bit0 & ((1 << RC) - 1);
  if (!marked) return;   // the digit form (dense_split.cu) holds
  const int nI = p.nI;
  double* M = smem;                           // 3 x KI x KI
  double* P = M + 3 * KI * KI;                // 3 x DT x KI
  double2* S = reinterpret_cast<double2*>(P + 3 * DT * KI);  // DT x RC
  double2* red = S + DT * RC;                 // 256 x RC (partial sums of the groups)

  const int t = threadIdx.x;
  const int ntx = (p.nx + L - 1) / L;
  const int bo = blockIdx.x / ntx;
  const int ao0 = (blockIdx.x % ntx) * L;
  const int olen = min(L, p.nx - ao0);
  const int ngr = 256 / L;
  const int o = t % L;
  const int grp = t / L;
  const bool active = grp < ngr && o < olen;
  const long long onat = (long long)bo * p.nx + ao0 + o;
  const double w2 = p.omega * p.omega, w2l = fma(p.omega, p.omega, -w2);
  const double c1 = 2.0 * HB_C0 / w2;

  double lxo[KI];
#pragma unroll
  for (int k = 0; k < KI; ++k) lxo[k] = (active && k < nI) ? p.LX[(size_t)(ao0 + o) * nI + k] : 0.0;
  double2 acc[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) acc[r] = make_double2(0.0, 0.0);
  const int NI = p.NI;

  const int bq0 = (int)((long long)p.ny * blockIdx.y / gridDim.y);
  const int bq1 = (int)((long long)p.ny * (blockIdx.y + 1) / gridDim.y);
  for (int bq = bq0; bq < bq1; ++bq) {
    __syncthreads();
    // M[q][i1][j1] = sum_i2 LZ[bo][i2] H[q][bq][(i2,i1)][j1], zero past nI
    for (int idx = t; idx < 3 * KI * KI; idx += blockDim.x) {
      const int q = idx / (KI * KI), i1 = (idx / KI) % KI, j1 = idx % KI;
      double a = 0.0;
      if (i1 < nI && j1 < nI) {
        const double* Hq = p.H + (((size_t)q * p.ny + bq) * NI) * nI;
        for (int i2 = 0; i2 < nI; ++i2)
          a = fma(p.LZ[(size_t)bo * nI + i2], Hq[(size_t)(i2 * nI + i1) * nI + j1], a);
        if (q == 1) a *= HB_C0;
        if (q == 2) a *= c1;
      }
      M[idx] = a;
    }
    __syncthreads();
    for (int aq0 = 0; aq0 < p.nx; aq0 += L) {
      const int qlen = min(L, p.nx - aq0);
      // P[q][c][i1] = sum_j1 M[q][i1][j1] LX[a_c][j1]
      for (int idx = t; idx < 3 * qlen * KI; idx += blockDim.x) {
        const int q = idx / (qlen * KI), cc = (idx / KI) % qlen, i1 = idx % KI;
        const double* lx = p.LX + (size_t)(aq0 + cc) * nI;
        double a = 0.0;
        for (int j1 = 0; j1 < nI; ++j1) a = fma(M[(q * KI + i1) * KI + j1], lx[j1], a);
        P[(q * DT + cc) * KI + i1] = a;
      }
      for (int idx = t; idx < qlen * RC; idx += blockDim.x) {
        const int cc = idx % qlen, r = idx / qlen;
        S[cc * RC + r] = s[(size_t)(r0 + r) * Nv + (size_t)bq * p.nx + aq0 + cc];
      }
      __syncthreads();
      if (active) {
        for (int cc = grp; cc < qlen; cc += ngr) {
          double f[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const double2* pq = reinterpret_cast<const double2*>(P + (q * DT + cc) * KI);
            double a = 0.0;
#pragma unroll
            for (int k = 0; k < KI / 2; ++k) {
              const double2 v = pq[k];
              a = fma(lxo[2 * k], v.x, a);
              a = fma(lxo[2 * k + 1], v.y, a);
            }
            f[q] = a;
          }
          const long long qnat = (long long)bq * p.nx + aq0 + cc;
          double2 g;
          if (qnat == onat) {
            g = p.self[onat];
          } else {
            // g = i v0 H0 - i v1 x H1 (the constants are in P)
            const HankelFG h = hankel_of_t2(p.hank, w2, w2l, f[0]);
            g = make_double2(fma(-h.F.y, f[1], h.G.y * f[2]), fma(h.F.x, f[1], -h.G.x * f[2]));
          }
          if (ADJ) g.y = -g.y;
#pragma unroll
          for (int r = 0; r < RC; ++r) {
            double2 x = S[cc * RC + r];
            acc[r].x = fma(g.x, x.x, fma(-g.y, x.y, acc[r].x));
            acc[r].y = fma(g.x, x.y, fma(g.y, x.x, acc[r].y));
          }
        }
      }
      __syncthreads();
    }
  }
  // add the groups' sums in order
  if (active && grp > 0) {
#pragma unroll
    for (int r = 0; r < RC; ++r) red[((grp - 1) * L + o) * RC + r] = acc[r];
  }
  __syncthreads();
  if (active && grp == 0) {
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      if (!(marked >> r & 1)) continue;
      double2 a = acc[r];
      for (int qq = 0; qq < ngr - 1; ++qq) {
        double2 b = red[(qq * L + o) * RC + r];
        a.x += b.x;
        a.y += b.y;
      }
      if (part) part[((size_t)blockIdx.y * RC + r) * Nv + onat] = a;
      else u[(size_t)(r0 + r) * Nv + onat] = make_double2(a.x * scale, a.y * scale);
    }
  }
}

// u[r0 + r][cell] = scale * (sum over the shares, in order, of part[share][r][cell])
// for the columns whose bit (bit0 + r of *flag) equals want: each form of the
// apply has written the shares of its own
__global__ void dense_reduce_kernel(const double2* __restrict__ part, double2* __restrict__ u, long long Nv, int rc,
                                    int nsplit, int r0, double scale, const int* __restrict__ flag, int bit0, int want) {
  const int cols = (want ? *flag : ~*flag) >> bit0 & ((1 << rc) - 1);
  if (!cols) return;
  const long long n = Nv * rc;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / Nv, cell = i - r * Nv;
    if (!(cols >> r & 1)) continue;
    double2 a = make_double2(0.0, 0.0);
    for (int k = 0; k < nsplit; ++k) {
      const double2 b = part[(size_t)k * n + i];
      a.x += b.x;
      a.y += b.y;
    }
    u[(size_t)(r0 + r) * Nv + cell] = make_double2(a.x * scale, a.y * scale);
  }
}

template <int RC, bool ADJ, int KI>
static void launch_dense(const EntryParams& p, const double2* s, double2* u, long long Nv, int L, int r0,
                         double scale, int nsplit, double2* part, const int* flag, int bit0, cudaStream_t st) {
  size_t sm = sizeof(double) * (3 * KI * KI + 3 * DT * KI) + sizeof(double2) * (DT + 256) * RC;
  auto k = dense_kernel<RC, ADJ, KI>;
  HB_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  const int ntx = (p.nx + L - 1) / L;
  k<<<dim3(ntx * p.ny, nsplit), 256, sm, st>>>(p, s, u, Nv, L, r0, scale, nsplit > 1 ? part : nullptr, flag, bit0);
  HB_CHECK_LAUNCH();
  if (nsplit > 1) {
    const long long n = Nv * RC;
    dense_reduce_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 8), 256, 0, st>>>(
        part, u, Nv, RC, nsplit, r0, scale, flag, bit0, 1);
    HB_CHECK_LAUNCH();
  }
}

// the FP64 form for rc right-hand sides from r0 on, in passes of 16, 8, 4, 2 and 1
static void dense_plain(const EntryParams& p, const double2* s, double2* u, long long Nv, int L, int r0, int rc, int adjoint,
                        double scale, int nsplit, double2* part, const int* flag, cudaStream_t st) {
  const int first = r0;
#define HB_DENSE_LAUNCH(R, A, K) launch_dense<R, A, K>(p, s, u, Nv, L, r0, scale, nsplit, part, flag, r0 - first, st)
#define HB_DENSE_CASE(R)                        \
  for (; rc >= R; rc -= R, r0 += R) {           \
    if (p.nI <= 8) {                            \
      if (adjoint) HB_DENSE_LAUNCH(R, true, 8); \
      else HB_DENSE_LAUNCH(R, false, 8);        \
    } else {                                    \
      if (adjoint) HB_DENSE_LAUNCH(R, true, 16);\
      else HB_DENSE_LAUNCH(R, false, 16);       \
    }                                           \
  }
  HB_DENSE_CASE(16)
  HB_DENSE_CASE(8)
  HB_DENSE_CASE(4)
  HB_DENSE_CASE(2)
  HB_DENSE_CASE(1)
#undef HB_DENSE_CASE
#undef HB_DENSE_LAUNCH
}

void dense_apply(hb_ctx* c, const double2* s, double2* u, int nrhs, int adjoint, cudaStream_t st) {
  NvtxRange nr(adjoint ? "hb_apply_dense_adjoint" : "hb_apply_dense");
  EntryParams p = entry_params(c, adjoint);
  const double scale = c->h * c->h;
  // small grids give few output CTAs: split the source lines into shares, up
  // to eight CTAs per SM; of the counts that give, the one that leaves the
  // least of the last wave (one CTA an SM) and of the longest share idle
  int dev = 0, nsm = 0;
  HB_CUDA(cudaGetDevice(&dev));
  HB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // equal segments of at most DT cells: a ragged last segment would idle threads
  const int L = (p.nx + (p.nx + DT - 1) / DT - 1) / ((p.nx + DT - 1) / DT);
  const long long cta = (long long)((p.nx + L - 1) / L) * p.ny;
  const int most = (int)std::max<long long>(1, std::min<long long>(p.ny, (8LL * nsm + cta - 1) / cta));
  int nsplit = 1;
  double best = 0.0;
  for (int k = 1; k <= most; ++k) {
    const double waves = (double)((cta * k + nsm - 1) / nsm), share = (double)((p.ny + k - 1) / k);
    const double eff = (double)(cta * p.ny) / (waves * nsm * (share + 0.1));   // a tenth of a line to set a CTA up
    if (eff > best) {
      best = eff;
      nsplit = k;
    }
  }
  if (nsplit > 1) {
    const size_t need = (size_t)nsplit * 16 * (size_t)c->Nv;
    if (c->dense_part_cap < need) {
      dev_free(c->d_dense_part);
      c->d_dense_part = nullptr;
      c->dense_part_cap = 0;
      c->d_dense_part = dev_alloc<double2>(need);
      c->dense_part_cap = need;
    }
  }
  // passes of up to 16 right-hand sides on the tensor cores; behind each the
  // FP64 kernel, which takes the columns that the digits do not hold
  double2* part = nsplit > 1 ? c->d_dense_part : nullptr;
  const int* flag = c->d_dense_ex + 16;
  for (int r0 = 0; r0 < nrhs; r0 += 16) {
    const int rc = std::min(nrhs - r0, 16);
    dense_split(p, s, u, c->Nv, L, nsplit, r0, rc, adjoint, scale, part, c->d_dense_ex, st);
    if (nsplit > 1) {
      const long long n = c->Nv * rc;
      dense_reduce_kernel<<<(unsigned)std::min<long long>((n + 255) / 256, 152LL * 8), 256, 0, st>>>(
          part, u, c->Nv, rc, nsplit, r0, scale, flag, 0, 0);
      HB_CHECK_LAUNCH();
    }
    dense_plain(p, s, u, c->Nv, L, r0, rc, adjoint, scale, nsplit, part, flag, st);
  }
}

// ------------------------------------------------------ block entries ----
// Work item = (block, one source column).  meta per block (int64 x 6):
//   row_off, m, col_off, n, out_off, seg_off;  nseg = number of row lines.
// Rows of a block are sorted by natural index, so rows of one grid line are
// contiguous; seg array (int64 x 3 per segment): b, first row, count.
// Output: column-major m x n at out_off; row a of the sorted list goes to
// out row rdst[row_off + a] (identity for the build).
// FP64-bound: a warp's FP64 instruction costs the same with few lanes live or on
// the other branch, so a pass takes enough lines that its rows fill the
// threads (with 8 lines it held 40 to 60 rows), and the Hankel pairs are
// evaluated from lists of the near arguments (recurrence) and the far ones
// (asymptotic series), a warp all on one branch.  The lists' order does not
// matter to the values.
constexpr int SEGC = 32;     // row lines per pass
constexpr int ECHUNK = 512;  // rows per round of the lists
constexpr int ETHREADS = 128;

__global__ void __launch_bounds__(ETHREADS) block_entries_kernel(
    EntryParams p, const BlockMeta* __restrict__ meta, const long long* __restrict__ items,
    const long long* __restrict__ rows, const int* __restrict__ rdst, const long long* __restrict__ cols,
    const long long* __restrict__ segs, double2* __restrict__ out) {
  __shared__ double G[3][256];
  __shared__ double P[3][SEGC][MAX_NI];
  __shared__ int s_line[SEGC], s_first[SEGC];
  __shared__ double lt[ECHUNK], l0[ECHUNK], l1[ECHUNK];   // near from the front, far from the back
  __shared__ int lrow[ECHUNK];
  __shared__ int s_near, s_far;
  const int nI = p.nI, NI = p.NI;
  const long long it = items[blockIdx.x];
  const int b = (int)(it >> 20);
  const int jj = (int)(it & 0xFFFFF);
  const BlockMeta bm = meta[b];
  const long long qnat = cols[bm.col_off + jj];
  const int aq = (int)(qnat % p.nx), bq = (int)(qnat / p.nx);
  const int t = threadIdx.x, lane = t & 31;
  // G[q][i] = sum_j1 H[q][bq][i][j1] LX[aq][j1]
  for (int idx = t; idx < 3 * NI; idx += blockDim.x) {
    int q = idx / NI, i = idx % NI;
    const double* Hq = p.H + (((size_t)q * p.ny + bq) * NI + i) * nI;
    const double* lx = p.LX + (size_t)aq * nI;
    double a = 0.0;
    for (int j1 = 0; j1 < nI; ++j1) a = fma(Hq[j1], lx[j1], a);
    G[q][i] = a;
  }
  for (int s0 = 0; s0 < bm.nseg; s0 += SEGC) {
    const int ns = (int)min((long long)SEGC, bm.nseg - s0);
    __syncthreads();
    if (t < ns) {
      s_line[t] = (int)segs[(bm.seg_off + s0 + t) * 3];
      s_first[t] = (int)segs[(bm.seg_off + s0 + t) * 3 + 1];
    }
    __syncthreads();
    for (int idx = t; idx < 3 * ns * nI; idx += blockDim.x) {
      int q = idx / (ns * nI), sl = (idx / nI) % ns, i1 = idx % nI;
      int bo = s_line[sl];
      const double* lz = p.LZ + (size_t)bo * nI;
      double a = 0.0;
      for (int i2 = 0; i2 < nI; ++i2) a = fma(lz[i2], G[q][i2 * nI + i1], a);
      P[q][sl][i1] = a;
    }
    const long long rfirst = segs[(bm.seg_off + s0) * 3 + 1];
    const long long rlast = segs[(bm.seg_off + s0 + ns - 1) * 3 + 1] + segs[(bm.seg_off + s0 + ns - 1) * 3 + 2];
    for (long long rc = rfirst; rc < rlast; rc += ECHUNK) {
      __syncthreads();   // P complete, and the lists of the last round read
      if (t == 0) s_near = s_far = 0;
      __syncthreads();
      const int cnt = (int)min((long long)ECHUNK, rlast - rc);
      for (int r0 = 0; r0 < cnt; r0 += ETHREADS) {
        const bool live = r0 + t < cnt;
        const long long r = rc + (live ? r0 + t : 0);
        // the line of row r: the last one starting at or before it
        int sl = 0;
#pragma unroll
        for (int w = SEGC / 2; w > 0; w >>= 1)
          if (sl + w < ns && s_first[sl + w] <= r) sl += w;
        const long long onat = rows[bm.row_off + r];
        const int ao = (int)(onat % p.nx);
        const double* lx = p.LX + (size_t)ao * nI;
        double f[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          double a = 0.0;
          for (int i1 = 0; i1 < nI; ++i1) a = fma(lx[i1], P[q][sl][i1], a);
          f[q] = a;
        }
        const double tau = sqrt(fmax(f[0], 0.0));
        const bool self = onat == qnat;
        if (live && self) out[bm.out_off + (long long)jj * bm.m + rdst[bm.row_off + r]] = p.self[onat];
        const bool far = hb_green_far(tau, p.omega);
        const unsigned mn = __ballot_sync(0xffffffffu, live && !self && !far);
        const unsigned mf = __ballot_sync(0xffffffffu, live && !self && far);
        int bn = 0, bf = 0;
        if (lane == 0) {
          bn = atomicAdd(&s_near, __popc(mn));
          bf = atomicAdd(&s_far, __popc(mf));
        }
        bn = __shfl_sync(0xffffffffu, bn, 0);
        bf = __shfl_sync(0xffffffffu, bf, 0);
        if (live && !self) {
          const unsigned below = (1u << lane) - 1;
          const int at = far ? ECHUNK - 1 - (bf + __popc(mf & below)) : bn + __popc(mn & below);
          lt[at] = tau;
          l0[at] = f[1];
          l1[at] = f[2];
          lrow[at] = (int)(r - rc);
        }
      }
      __syncthreads();
      // whole warps on one branch: near entries from slot 0, far ones from the next multiple of 32
      const int nn = s_near, nf = s_far, f0 = (nn + 31) / 32 * 32;
      for (int e = t; e < f0 + nf; e += ETHREADS) {
        const int at = e < f0 ? e : ECHUNK - 1 - (e - f0);
        if (e < f0 && e >= nn) continue;
        const double2 g = hb_green_tau(lt[at], l0[at], l1[at], p.omega);
        out[bm.out_off + (long long)jj * bm.m + rdst[bm.row_off + rc + lrow[at]]] = g;
      }
    }
  }
}

// Host side: blocks given as natural-index lists (rows need not be sorted).
void add_block(BlockBatchHost& B, const hb_ctx* c, const long long* rows, long long m,
               const long long* cols, long long n, long long out_off) {
  BlockMeta bm{};
  bm.row_off = (long long)B.rows.size();
  bm.m = m;
  bm.col_off = (long long)B.cols.size();
  bm.n = n;
  bm.out_off = out_off;
  bm.seg_off = (long long)B.segs.size() / 3;
  std::vector<std::pair<long long, int>> order((size_t)m);
  for (long long a = 0; a < m; ++a) order[a] = {rows[a], (int)a};
  std::sort(order.begin(), order.end());
  long long nseg = 0;
  for (long long a = 0; a < m; ++a) {
    long long nat = order[a].first;
    B.rows.push_back(nat);
    B.rdst.push_back(order[a].second);
    long long line = nat / c->nx;
    if (a == 0 || line != order[a - 1].first / c->nx) {
      B.segs.push_back(line);
      B.segs.push_back(a);
      B.segs.push_back(0);
      ++nseg;
    }
    B.segs[B.segs.size() - 1] += 1;
  }
  bm.nseg = nseg;
  B.cols.insert(B.cols.end(), cols, cols + n);
  long long bidx = (long long)B.meta.size();
  for (long long j = 0; j < n; ++j) B.items.push_back((bidx << 20) | j);
  B.meta.push_back(bm);
}

namespace {
// Device scratch of one call, freed when the call returns or throws (after
// the stream has drained, so no launched kernel still reads it).
struct CallScratch {
  cudaStream_t st;
  std::vector<void*> p;
  template <class T>
  T* keep(T* q) {
    p.push_back(q);
    return q;
  }
  ~CallScratch() {
    cudaStreamSynchronize(st);
    for (void* q : p) dev_free(q);
  }
};
}  // namespace

void run_blocks(hb_ctx* c, BlockBatchHost& B, double2* d_out, cudaStream_t st) {
  if (B.items.empty()) return;
  CallScratch sc{st, {}};
  BlockMeta* d_meta = sc.keep(upload(B.meta, st));
  long long* d_items = sc.keep(upload(B.items, st));
  long long* d_rows = sc.keep(upload(B.rows, st));
  int* d_rdst = sc.keep(upload(B.rdst, st));
  long long* d_cols = sc.keep(upload(B.cols, st));
  long long* d_segs = sc.keep(upload(B.segs, st));
  EntryParams p = entry_params(c, 0);
  size_t nitems = B.items.size();
  for (size_t i0 = 0; i0 < nitems; i0 += 1u << 30) {
    unsigned cnt = (unsigned)std::min<size_t>(nitems - i0, 1u << 30);
    block_entries_kernel<<<cnt, ETHREADS, 0, st>>>(p, d_meta, d_items + i0, d_rows, d_rdst, d_cols, d_segs, d_out);
    HB_CHECK_LAUNCH();
  }
  HB_CUDA(cudaStreamSynchronize(st));
}

void eval_entries(hb_ctx* c, const long long* rows, int m, const long long* cols, int n, double2* out,
                  cudaStream_t st) {
  BlockBatchHost B;
  add_block(B, c, rows, m, cols, n, 0);
  run_blocks(c, B, out, st);
}

}  // namespace hb
