// cpqr.cu - batched interpolative decomposition by column-pivoted
// Householder QR, FP64 complex (Sec. 4.2.1, Eq. ID, Eq. proxy).
//
// For each matrix A (m x n, column-major), K(tau_hat, cols) ~ K(tau_hat,
// skel) V with skel the first r pivots and V = [I | R11^-1 R12] P^T:
//  * step k: the trailing column norms over rows >= k are recomputed (fused
//    into the previous step's update, no downdating); the pivot is the
//    lowest position whose norm is at least the largest minus ID_TIE |R_00|
//    (the largest times 1 - ID_TIE at step 0): columns that are mirror
//    images on the grid have norms equal up to rounding, and the window makes
//    the choice among them independent of how the norms were rounded;
//  * the rank is the first k >= 1 with |R_kk| <= eps |R_00| (k = min(m, n)
//    otherwise); an all-zero matrix gets rank 1 with V = e_0^T;
//  * the reflector for column k is H = I - (2/v^H v) v v^H with
//    v = x + e^{i arg x_0} |x| e_0, so R_kk = -e^{i arg x_0} |x|; v is kept in
//    place below the diagonal.
// Outputs: the rank, the full pivot order (first r = skeleton) and, in place
// of R12, T = R11^-1 R12 (rows < r of the columns at pivot positions >= r);
// emit_v_kernel assembles V from them.
// One CTA of 256 threads per matrix, two columns per warp at a time; every
// reduction runs in a fixed order (lane-strided partial sums, then an
// xor-shuffle tree), so results are bitwise reproducible run to run.
//
// Bound by the FP64 unit (2 FMAs a cycle and SM): per trailing column and 32
// rows 4 instructions for v^H x, 6 for the update and 2 for the norm, plus the
// reductions.  Those of a column pair share their steps (the half-warps, then
// the quarters, each carry on with one of the sums: the same additions in
// every tree, 11 instructions instead of 30), and the square roots of the norms are taken
// by all threads at once afterwards (1 / 32 of the instructions).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "hb_internal.cuh"

namespace cg = cooperative_groups;

namespace hb {

constexpr int ID_THREADS = 256;
constexpr int ID_WARPS = ID_THREADS / 32;
constexpr double ID_TIE = 1e-12;   // pivot tie window, relative to |R_00|

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double shfl_xor_d(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// warp_sum of a, b, c, d: lanes 0-7 end with a's, 8-15 b's, 16-23 c's, 24-31 d's
__device__ __forceinline__ double warp_sum4(double a, double b, double c, double d, int lane) {
  const bool up = lane & 16;
  double k0 = up ? c : a, k1 = up ? d : b;
  k0 += shfl_xor_d(up ? a : c, 16);
  k1 += shfl_xor_d(up ? b : d, 16);
  const bool up8 = lane & 8;
  double k = up8 ? k1 : k0;
  k += shfl_xor_d(up8 ? k0 : k1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) k += shfl_xor_d(k, o);
  return k;
}
// warp_sum of a and b: lanes 0-15 end with a's, 16-31 with b's
__device__ __forceinline__ double warp_sum2(double a, double b, int lane) {
  const bool up = lane & 16;
  double k = up ? b : a;
  k += shfl_xor_d(up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) k += shfl_xor_d(k, o);
  return k;
}

// A matrix of at least ID_BIG entries is decomposed by a cluster of cs CTAs
// (CL kernels; the smaller ones of the same launch by the cluster's first CTA
// alone): one CTA has one SM's FP64 unit, and the blocks of the first levels
// (1300 x 64 at 64^2) then outlast the rest of their launch several times
// over.  Clusters of 8, or of 4 where the launch has matrices enough to fill
// the chip (id_cluster).  Decompositions of a 64^2 build, ms: one CTA each 39, the shared
// reductions 36, clusters of 8 from 12288 / 3072 / 1024 entries on 24 / 18 / 16; a whole build at
// 256^2: clusters of 8 2.12 s, of 4 2.06 s.
constexpr long long ID_BIG = 1024;

// Columns never move: position j holds column perm[j] of A.
template <bool CL>
__global__ void __launch_bounds__(ID_THREADS) id_kernel(const int* __restrict__ M, const int* __restrict__ N,
                                                        const long long* __restrict__ aoff, double2* A,
                                                        double eps, int* __restrict__ rank_out,
                                                        int* __restrict__ perm_out,
                                                        const long long* __restrict__ soff, int cs) {
  extern __shared__ unsigned char sm_raw[];
  const int b = CL ? blockIdx.x / cs : blockIdx.x;
  const int m = M[b], n = N[b];
  const bool team = CL && (long long)m * n >= ID_BIG;
  const int cr = team ? blockIdx.x % cs : 0, nc = team ? cs : 1;
  if (CL && !team && blockIdx.x % cs) return;
  double2* a = A + aoff[b];
  double2* rd = reinterpret_cast<double2*>(sm_raw);         // n   R_kk (16-byte aligned first)
  double* nrm0 = reinterpret_cast<double*>(rd + n);         // n   norms of the trailing columns; a team alternates two
  int* perm = reinterpret_cast<int*>(nrm0 + (CL ? 2 : 1) * n);   // n
  __shared__ int s_rank, s_stop;
  __shared__ double s_r00, s_scale;
  __shared__ double2 s_v0;

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the buffer step k reads; a CTA ahead of another writes the next one's
  auto norms = [&](int k) { return nrm0 + ((CL && team && (k & 1)) ? n : 0); };
  // the sums of squares of step k's columns go to every CTA of the team
  auto put = [&](int k, int j, double s, int l) {
    if constexpr (CL) {
      if (team) {
        if (l < cs) cg::this_cluster().map_shared_rank(norms(k), l)[j] = s;
        return;
      }
    }
    if (l == 0) norms(k)[j] = s;
  };
  auto meet = [&]() {
    if constexpr (CL) {
      if (team) {
        __threadfence();
        cg::this_cluster().sync();
        return;
      }
    }
    __syncthreads();
  };
  // columns are written by other SMs of a team: read them from L2
  auto ld = [&](const double2* p) { return CL ? __ldcg(p) : *p; };
  for (int j = threadIdx.x; j < n; j += ID_THREADS) perm[j] = j;
  if (CL && team) cg::this_cluster().sync();   // every CTA of the team runs before its shared memory is written
  // initial column norms over all rows
  for (int j = cr + nc * warp; j < n; j += nc * ID_WARPS) {
    const double2* col = a + (size_t)j * m;
    double s = 0.0;
    for (int i = lane; i < m; i += 32) {
      const double2 x = col[i];
      s = fma(x.x, x.x, fma(x.y, x.y, s));
    }
    put(0, j, warp_sum(s), lane);
  }
  if (threadIdx.x == 0) {
    s_rank = min(m, n);
    s_stop = 0;
  }
  meet();
  const int kmax = min(m, n);
  for (int k = 0; k < kmax; ++k) {
    double* nrm = norms(k);
    for (int j = k + threadIdx.x; j < n; j += ID_THREADS) nrm[j] = sqrt(nrm[j]);
    __syncthreads();
    if (warp == 0) {
      // the largest trailing norm, then the lowest position inside the tie
      // window (both reductions are exact, so their order does not matter)
      double top = 0.0;
      for (int j = k + lane; j < n; j += 32) top = fmax(top, nrm[j]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
      const double thr = (k == 0) ? top * (1.0 - ID_TIE) : top - ID_TIE * s_r00;
      int p = n;
      for (int j = k + lane; j < n; j += 32)
        if (nrm[j] >= thr) {
          p = j;
          break;
        }
      p = __reduce_min_sync(0xffffffffu, p);
      if (lane == 0) {
        if (k == 0) {
          s_r00 = nrm[p];
          if (top == 0.0) { s_rank = 1; s_stop = 2; }
        } else if (top <= eps * s_r00) {
          s_rank = k;
          s_stop = 1;
        }
        if (!s_stop) {
          if (p != k) {
            double t = nrm[k]; nrm[k] = nrm[p]; nrm[p] = t;
            int q = perm[k]; perm[k] = perm[p]; perm[p] = q;
          }
          // Householder vector in column k, rows k..m-1: its first entry is v0
          const double alpha = nrm[k];
          const double2 x0 = ld(a + (size_t)perm[k] * m + k);
          const double ax0 = hypot(x0.x, x0.y);
          double2 ph = (ax0 > 0.0) ? make_double2(x0.x / ax0, x0.y / ax0) : make_double2(1.0, 0.0);
          double2 v0 = make_double2(x0.x + ph.x * alpha, x0.y + ph.y * alpha);
          const double vv = alpha * alpha - ax0 * ax0 + (v0.x * v0.x + v0.y * v0.y);
          s_scale = (vv > 0.0) ? 2.0 / vv : 0.0;
          rd[k] = make_double2(-ph.x * alpha, -ph.y * alpha);
          s_v0 = v0;
        }
      }
    }
    __syncthreads();
    if (s_stop) break;
    const double2* ck = a + (size_t)perm[k] * m;
    const double sc = s_scale;
    const double2 v0 = s_v0;
    // apply to trailing columns and recompute their norms over rows k+1..m-1
    // (sums of squares here; the square roots when the next step begins)
    for (int j = k + 1 + 2 * (cr + nc * warp); j < n; j += 2 * nc * ID_WARPS) {
      const bool two = j + 1 < n;
      double2* c0 = a + (size_t)perm[j] * m;
      double2* c1 = two ? a + (size_t)perm[j + 1] * m : c0;   // alone: the same column twice, stored once
      double wr = 0.0, wi = 0.0, zr = 0.0, zi = 0.0;
      for (int i = k + lane; i < m; i += 32) {
        const double2 v = i == k ? v0 : ld(ck + i), x = ld(c0 + i), y = ld(c1 + i);
        wr = fma(v.x, x.x, fma(v.y, x.y, wr));        // conj(v) x
        wi = fma(v.x, x.y, fma(-v.y, x.x, wi));
        zr = fma(v.x, y.x, fma(v.y, y.y, zr));
        zi = fma(v.x, y.y, fma(-v.y, y.x, zi));
      }
      const double w4 = warp_sum4(wr, wi, zr, zi, lane) * sc;
      wr = __shfl_sync(0xffffffffu, w4, 0);
      wi = __shfl_sync(0xffffffffu, w4, 8);
      zr = __shfl_sync(0xffffffffu, w4, 16);
      zi = __shfl_sync(0xffffffffu, w4, 24);
      double s = 0.0, s1 = 0.0;
      for (int i = k + lane; i < m; i += 32) {
        const double2 v = i == k ? v0 : ld(ck + i);
        double2 x = ld(c0 + i), y = ld(c1 + i);
        x.x -= wr * v.x - wi * v.y;
        x.y -= wr * v.y + wi * v.x;
        y.x -= zr * v.x - zi * v.y;
        y.y -= zr * v.y + zi * v.x;
        c0[i] = x;
        if (two) c1[i] = y;
        if (i > k) {
          s = fma(x.x, x.x, fma(x.y, x.y, s));
          s1 = fma(y.x, y.x, fma(y.y, y.y, s1));
        }
      }
      s = warp_sum2(s, s1, lane);
      if (lane < 16) put(k + 1, j, s, lane);
      else if (two) put(k + 1, j + 1, s, lane - 16);
    }
    meet();
  }
  __syncthreads();
  const int r = s_rank;
  const bool zero = (s_stop == 2);
  // T = R11^-1 R12, one warp per column of R12; R11 diagonal from rd, strict
  // upper part in place; the result overwrites R12.
  if (!zero) {
    for (int j = r + cr + nc * warp; j < n; j += nc * ID_WARPS) {
      double2* cj = a + (size_t)perm[j] * m;
      for (int i = r - 1; i >= 0; --i) {
        double sr = 0.0, si = 0.0;
        for (int l = i + 1 + lane; l < r; l += 32) {
          const double2 R = ld(a + (size_t)perm[l] * m + i), t = ld(cj + l);
          sr = fma(R.x, t.x, fma(-R.y, t.y, sr));
          si = fma(R.x, t.y, fma(R.y, t.x, si));
        }
        sr = warp_sum(sr);
        si = warp_sum(si);
        if (lane == 0) {
          const double2 c = ld(cj + i);
          const double2 num = make_double2(c.x - sr, c.y - si);
          const double2 d = rd[i];
          const double dd = d.x * d.x + d.y * d.y;
          cj[i] = make_double2((num.x * d.x + num.y * d.y) / dd, (num.y * d.x - num.x * d.y) / dd);
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  if (cr) return;
  int* pm = perm_out + soff[b];
  for (int j = threadIdx.x; j < n; j += ID_THREADS) pm[j] = perm[j];
  if (threadIdx.x == 0) rank_out[b] = r;
}

// V[k][perm[j]] = (j < r) ? delta_kj : T[k][j] (in column perm[j] of A); V column-major with leading
// dimension ld = (ld_is_rank ? r : n) at element offset voff[b].
__global__ void emit_v_kernel(const int* __restrict__ M, const int* __restrict__ N,
                              const long long* __restrict__ aoff, const double2* __restrict__ A,
                              const int* __restrict__ rank, const int* __restrict__ perm,
                              const long long* __restrict__ soff, const long long* __restrict__ voff,
                              int ld_is_rank, double2* __restrict__ V64, float2* __restrict__ V32) {
  const int b = blockIdx.x;
  const int m = M[b], n = N[b], r = rank[b];
  const int ld = ld_is_rank ? r : n;
  const double2* a = A + aoff[b];
  const int* pm = perm + soff[b];
  for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
    const int j = idx / r, kk = idx % r;
    // an all-zero input never ran a reflection, so its T entries read as 0
    double2 val = (j < r) ? make_double2(j == kk ? 1.0 : 0.0, 0.0) : a[(size_t)pm[j] * m + kk];
    const size_t o = voff[b] + (size_t)pm[j] * ld + kk;
    if (V64) V64[o] = val;
    if (V32) V32[o] = make_float2((float)val.x, (float)val.y);
  }
}

// CTAs a matrix.  Unequal matrices (a build's levels: a few outlast the rest):
// 8, or 4 past 512 matrices.  Nearly equal ones: one CTA keeps its SM's FP64
// unit busy, so what counts is how evenly the CTAs fill the chip, and what a
// cluster of 2, 4 or 8 loses to its barriers (5, 25, 35 %).  Measured, 400 x 64
// of rank 20, us with 1 / 2 / 4 / 8: 40 matrices 1992 / 1183 / 1079 / 892, 110
// 1997 / 1936 / 1552 / 1829, 228 3671 / 2885 / 3438 / 3495, 304 3681 / 3816 / 4390
// / 4503, 700 9047 / 9271 / 9204 / 9977.
static int id_cluster(int count, const IdSizes& sizes) {
  if (sizes.work < 0.8 * count * sizes.max_work) return count <= 512 ? 8 : 4;
  int dev = 0, nsm = 0;
  HB_CUDA(cudaGetDevice(&dev));
  HB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const double loss[4] = {1.0, 1.05, 1.25, 1.35};
  int best = 1;
  double cost = 0.0;
  for (int k = 0; k < 4; ++k) {
    const long long per = 1 << k, waves = (count * per + nsm - 1) / nsm;
    const double c = (double)waves / (double)per * loss[k];
    if (k == 0 || c < cost) {
      cost = c;
      best = (int)per;
    }
  }
  return best;
}

void id_batch(int count, const int* d_m, const int* d_n, const long long* d_aoff, double2* d_A, double eps,
              int* d_rank, int* d_perm, const long long* d_soff, const IdSizes& sizes, cudaStream_t st) {
  if (count == 0) return;
  // clusters only where a matrix takes one and their second norm buffer fits
  const size_t col = sizeof(double) + sizeof(double2) + sizeof(int);
  const int cs = sizes.max_mn >= ID_BIG && (col + sizeof(double)) * (size_t)sizes.max_n <= (200u << 10)
                     ? id_cluster(count, sizes) : 1;
  const bool cl = cs > 1;
  const size_t sm = std::max<size_t>((size_t)sizes.max_n * (col + (cl ? sizeof(double) : 0)), 1);
  if (cl) HB_CUDA(cudaFuncSetAttribute(id_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  else HB_CUDA(cudaFuncSetAttribute(id_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  const int most = (1 << 30) / cs;
  for (int b0 = 0; b0 < count; b0 += most) {
    const int cnt = std::min(count - b0, most);
    if (cl) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)cnt * (unsigned)cs);
      cfg.blockDim = dim3(ID_THREADS);
      cfg.dynamicSmemBytes = sm;
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)cs;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      HB_CUDA(cudaLaunchKernelEx(&cfg, id_kernel<true>, d_m + b0, d_n + b0, d_aoff + b0, d_A, eps, d_rank + b0, d_perm,
                                 d_soff + b0, cs));
    } else {
      id_kernel<false><<<cnt, ID_THREADS, sm, st>>>(d_m + b0, d_n + b0, d_aoff + b0, d_A, eps, d_rank + b0, d_perm,
                                                    d_soff + b0, 1);
    }
    HB_CHECK_LAUNCH();
  }
}

void emit_v(int count, const int* d_m, const int* d_n, const long long* d_aoff, const double2* d_A,
            const int* d_rank, const int* d_perm, const long long* d_soff, const long long* d_voff,
            int ld_is_rank, double2* V64, float2* V32, cudaStream_t st) {
  for (int b0 = 0; b0 < count; b0 += 1 << 30) {
    int cnt = std::min(count - b0, 1 << 30);
    emit_v_kernel<<<cnt, 128, 0, st>>>(d_m + b0, d_n + b0, d_aoff + b0, d_A, d_rank + b0, d_perm,
                                       d_soff + b0, d_voff + b0, ld_is_rank, V64, V32);
    HB_CHECK_LAUNCH();
  }
}

}  // namespace hb

// ---------------------------------------------------------------------------
// hb_id_batch_noalloc: the same batched decompositions without allocating.
//
// Some callers cannot call cudaMalloc: code running under another
// framework's memory manager (which has reserved the device memory for its
// own pool, so a raw cudaMalloc can fail even though memory is free in that
// pool, or would stall every stream with its implicit synchronisation), and
// latency-critical paths that must not take that synchronisation.  For them
// the per-matrix metadata the kernels read from device memory (sizes and
// offsets) lives in this file-scope array instead of a fresh allocation.
// Every GPU that loads the library holds the array until the process exits.
// The pivot order goes straight into the caller's skel buffer, so nothing
// else is needed.  Every call overwrites the metadata it reads, so nothing
// has to start at zero; calls that overlap on the GPU (different streams or
// host threads without a synchronisation between them) race on the array.
//
// The caller's host arrays m, n, a_off are first copied into a file-scope
// host array (ordinary pageable memory, under a mutex) and the device copies
// read that array.  A copy from pageable memory has consumed its source when
// cudaMemcpyAsync returns, so the caller may reuse its arrays on return even
// when they are page-locked (a copy straight from page-locked memory would
// read them only when the stream reaches it).
#include <algorithm>
#include <cstring>
#include <mutex>

namespace hb {

constexpr int ID_NOALLOC_MAX = 65536;                       // matrices per call
constexpr size_t ID_NOALLOC_BYTES = (size_t)ID_NOALLOC_MAX * 32;   // 2 MiB

static __device__ __align__(256) unsigned char g_id_noalloc_scratch[ID_NOALLOC_BYTES];

namespace {
std::mutex g_noalloc_mu;
void* g_noalloc_addr[256] = {};   // device address of the array, per device ordinal
// host staging of the metadata (pageable; guarded by g_noalloc_mu)
alignas(256) unsigned char g_noalloc_host[(size_t)ID_NOALLOC_MAX * 16];

// Set-up, once per device, with that device current: look up the device
// address of the array (its name in host code is only a host-side stand-in).
// The caller holds g_noalloc_mu.
void* noalloc_scratch() {
  int dev = 0;
  HB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) throw Error{HB_ERR_UNSUPPORTED, "device ordinal above 255"};
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_id_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      throw Error{HB_ERR_CUDA, std::string("cudaGetSymbolAddress(id scratch): ") + cudaGetErrorString(e)};
    }
    g_noalloc_addr[dev] = p;
  }
  return g_noalloc_addr[dev];
}

// s_off[b] = sum_{c<b} n[c], v_off[b] = sum_{c<b} n[c]^2 (one CTA, chunked scan)
__global__ void __launch_bounds__(1024) noalloc_offsets_kernel(const int* __restrict__ n, int count,
                                                                long long* __restrict__ s_off,
                                                                long long* __restrict__ v_off) {
  __shared__ long long ts[1024], tv[1024];
  const int chunk = (count + 1023) / 1024;
  const int b0 = min(count, (int)threadIdx.x * chunk), b1 = min(count, b0 + chunk);
  long long as = 0, av = 0;
  for (int b = b0; b < b1; ++b) {
    as += n[b];
    av += (long long)n[b] * n[b];
  }
  ts[threadIdx.x] = as;
  tv[threadIdx.x] = av;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long rs = 0, rv = 0;
    for (int i = 0; i < 1024; ++i) {
      const long long a = ts[i], v = tv[i];
      ts[i] = rs;
      tv[i] = rv;
      rs += a;
      rv += v;
    }
  }
  __syncthreads();
  as = ts[threadIdx.x];
  av = tv[threadIdx.x];
  for (int b = b0; b < b1; ++b) {
    s_off[b] = as;
    v_off[b] = av;
    as += n[b];
    av += (long long)n[b] * n[b];
  }
}
}  // namespace

void id_batch_noalloc(int count, const int* m, const int* n, const long long* a_off, double2* A, double eps,
                      int* rank, int* skel, double2* V, cudaStream_t st) {
  if (count > ID_NOALLOC_MAX)
    throw arg_error("hb_id_batch_noalloc: count=%d exceeds the static scratch limit of %d matrices", count,
                    ID_NOALLOC_MAX);
  IdSizes sizes;
  for (int b = 0; b < count; ++b) {
    if (m[b] < 1 || n[b] < 1) throw arg_error("matrix %d has an empty dimension", b);
    sizes.add(m[b], n[b]);
  }
  if (count == 0) return;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  unsigned char* base = static_cast<unsigned char*>(noalloc_scratch());
  int* d_m = reinterpret_cast<int*>(base);
  int* d_n = reinterpret_cast<int*>(base + (size_t)ID_NOALLOC_MAX * 4);
  long long* d_a = reinterpret_cast<long long*>(base + (size_t)ID_NOALLOC_MAX * 8);
  long long* d_s = reinterpret_cast<long long*>(base + (size_t)ID_NOALLOC_MAX * 16);
  long long* d_v = reinterpret_cast<long long*>(base + (size_t)ID_NOALLOC_MAX * 24);
  // one host-to-device copy of the staged metadata: m, n, a_off in the
  // array's order (int m[MAX], int n[MAX], long long a_off[MAX]); only the
  // first count entries of each part are copied
  int* h_m = reinterpret_cast<int*>(g_noalloc_host);
  int* h_n = reinterpret_cast<int*>(g_noalloc_host + (size_t)ID_NOALLOC_MAX * 4);
  long long* h_a = reinterpret_cast<long long*>(g_noalloc_host + (size_t)ID_NOALLOC_MAX * 8);
  std::memcpy(h_m, m, sizeof(int) * count);
  std::memcpy(h_n, n, sizeof(int) * count);
  std::memcpy(h_a, a_off, sizeof(long long) * count);
  HB_CUDA(cudaMemcpyAsync(d_m, h_m, sizeof(int) * count, cudaMemcpyHostToDevice, st));
  HB_CUDA(cudaMemcpyAsync(d_n, h_n, sizeof(int) * count, cudaMemcpyHostToDevice, st));
  HB_CUDA(cudaMemcpyAsync(d_a, h_a, sizeof(long long) * count, cudaMemcpyHostToDevice, st));
  noalloc_offsets_kernel<<<1, 1024, 0, st>>>(d_n, count, d_s, d_v);
  HB_CHECK_LAUNCH();
  id_batch(count, d_m, d_n, d_a, A, eps, rank, skel, d_s, sizes, st);
  emit_v(count, d_m, d_n, d_a, A, rank, skel, d_s, d_v, 0, V, nullptr, st);
}

}  // namespace hb
