// dense_split.cu - the matrix-free dense apply U = K I and its adjoint with the
// contractions and the sums on the FP16 tensor cores by integer digits
// (split_fixed.cuh), the entries themselves in FP64 (Sec. 3.1 Eq. m_v2v;
// Sec. 4.1 Eq. chebinterpblock; staged as in entries.cu).
//
// An entry costs 48 FP64 FMAs of interpolation, 12 for the contraction its
// source shares with 64 outputs, 30 for the Hankel pair and the product, and 4
// per right-hand side, on a unit with 2 FMAs a cycle and SM; the tensor cores
// have 1024 FP16 ones.  All but the 30 are contractions:
//   P_q[c][i1] = sum_{j1} LX[c][j1] M_q[i1][j1]       (M per line pair, FP64)
//   f_q(o, c)  = sum_{i1} LX[o][i1] P_q[c][i1]        q = tau^2, v0, v1
//   u[o][r]   += sum_c g(o, c) s[c][r]
// each one k-step of 16 of the error-free digit products, rounded to FP64 once
// per stage.  P and f take the products of a seventh diagonal (26 instead of
// 21): tau^2 of near pairs is small against its own terms, and without them
// tau^2 errs by 3e-17 of the largest, as much as all roundings of plain FP64
// sums.  Root mean square error of an apply against long double sums over
// three media (32^2, 40 x 27, 24^2): 1.6 to 4.8e-15, of the plain FP64 form
// 1.7 to 5.0e-15, with six diagonals only 2.0 to 4.7e-15 and a tenth above it
// on average.
//
// A CTA owns the L <= 64 cells of one segment of a grid line and sweeps segments
// of up to 200 source cells of its share of the source lines.  Warp w works for
// the 16 outputs of m-tile w mod nmt and every (warps / nmt)-th n-tile of 8
// sources.  The accumulator layout of one stage is the operand layout of the
// next: P's (cells, i1) tile is the B fragment of the f stage (its pairs of i1),
// and a lane's four entries g(o, c) are its four words of the A fragment of
// the sum.  Running sums are 64-bit integer pairs at the largest exponent met.
//
// Bound by the FP64 unit still (63 % busy at 64^2 with 8 warps an SM): the Hankel
// pairs.  Measured, evaluation entry by entry through recurrences / plain FP64
// with tabulated pairs (entries.cu) / this: 64^2, one right-hand side 53.4 /
// 3.4 / 1.97 ms; 144 x 100, 16 right-hand sides (adjoint) 435 / 62 / 22.9 ms.
//
// Right-hand sides that are not finite, or too small for the digits
// (split_fixed.cuh), are marked in *flag (bit r), all of them where an operand
// of the entries is so; the FP64 kernel of entries.cu, launched behind this one,
// computes the marked ones instead, so no column depends on another's values.
#include <cuda_runtime.h>

#include <algorithm>

#include "hb_internal.cuh"
#include "split_fixed.cuh"

namespace hb {
namespace {

// n-tiles (8 sources) of a source segment at most: what 227 KB hold beside four
// m-tiles and two tiles of right-hand sides (222.5 KB).  Longer segments share
// their staging and barriers among more entries; 12 / 18 / 25 tiles: 200 x 60 x 4
// 18.2 / 17.7 / 16.7 ms, 144 x 100 x 16 26.6 / 22.8 / 22.8, 120 x 100 17.2 / 14.7 /
// 14.7, 64^2 1.98 each.
constexpr int DS_NT = 25;
constexpr int DS_K = 16;         // interpolation nodes per axis (padded with zeros)
constexpr int DS_DIAGS = 7;      // diagonals of digit products in the contractions (sums: 6)
constexpr double DS_C0 = 0.88622692545275801365;   // sqrt(pi)/2
constexpr uint32_t DS_IM = 0x80000000u;

// ex[r] = largest exponent of right-hand side r
__global__ void __launch_bounds__(256) rhs_exponent_kernel(const double2* __restrict__ s, long long Nv, int* __restrict__ ex) {
  const double2* c = s + (size_t)blockIdx.y * Nv;
  int e = 0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < Nv; i += (long long)gridDim.x * 256)
    e = max(e, block_exponent(c[i]));
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0 && e) atomicMax(&ex[blockIdx.y], e);
}

// the digit products of one 16 x 8 tile, k = 16: acc[i + j] += a_i b_j, i + j < DIAGS
template <int DIAGS, class LoadA, class LoadB>
__device__ __forceinline__ void digit_mma(float (&acc)[DIAGS][4], LoadA&& la, LoadB&& lb) {
#pragma unroll
  for (int d = 0; d < DIAGS; ++d)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[d][e] = 0.f;
  uint2 b[SPLIT_DIGITS];
#pragma unroll
  for (int j = 0; j < SPLIT_DIGITS; ++j) b[j] = lb(j);
#pragma unroll
  for (int i = 0; i < SPLIT_DIGITS; ++i) {
    const uint4 a = la(i);
#pragma unroll
    for (int j = 0; j < SPLIT_DIGITS && i + j < DIAGS; ++j) mma_f16(acc[i + j], a.x, a.y, a.z, a.w, b[j].x, b[j].y);
  }
}

// the sums of one element: hi in units of diagonal 2, lo of diagonal 5 (one
// k-step: diagonal 2's three products stay within 2^24 together); diagonal 6
// goes to its nearest unit of diagonal 5
template <int DIAGS>
__device__ __forceinline__ void digit_sums(const float (&acc)[DIAGS][4], int e, long long& hi, long long& lo) {
  hi = (long long)__float2int_rn(acc[2][e]) + (long long)__float2int_rn(acc[1][e]) * 1024 +
       (long long)__float2int_rn(acc[0][e]) * 1048576;
  lo = (long long)__float2int_rn(acc[5][e]) + (DIAGS > 6 ? __float2int_rn(acc[DIAGS - 1][e] * 0x1p-10f) : 0) + (long long)__float2int_rn(acc[4][e]) * 1024 +
       (long long)__float2int_rn(acc[3][e]) * 1048576;
}

// (hi 2^30 + lo) >> d
__device__ __forceinline__ void shift_sums(long long& hi, long long& lo, int d) {
  if (d >= 60) {
    hi = lo = 0;
    return;
  }
  const long long h = hi >> d, rem = hi - (h << d);
  lo = (lo >> d) + (d <= 30 ? rem << (30 - d) : rem >> (d - 30));
  hi = h;
}

__device__ __forceinline__ int max_xor(int v, int o) { return max(v, __shfl_xor_sync(0xffffffffu, v, o)); }

struct DsLayout {   // dynamic shared memory, in 4-byte words
  int m64, mfrag, mex, lxo, eo, pfrag, ep, sfrag, words;
  __host__ __device__ DsLayout(int nmt, int nt, int rt) {
    int w = 0;
    m64 = w;   w += 3 * DS_K * DS_K * 2;                       // M, FP64
    mfrag = w; w += 3 * 2 * SPLIT_DIGITS * 64;                 // [q][n-tile][digit][lane][2]
    lxo = w;   w += nmt * SPLIT_DIGITS * 128;                  // [m-tile][digit][lane][4]
    pfrag = w; w += nt * 3 * SPLIT_DIGITS * 64;                // [n-tile][q][digit][lane][2]
    sfrag = w; w += nt * rt * SPLIT_DIGITS * 64;               // [n-tile][rhs tile][digit][lane][2]
    mex = w;   w += 3 * DS_K;                                  // exponents of M's rows (q, i1)
    eo = w;    w += nmt * 16;                                  // of the outputs' bases
    ep = w;    w += 3 * nt * 8;                                // of P (q, cell)
    words = w;
  }
};

// RT tiles of 8 right-hand sides.  rc of them are real.
template <int RT, bool ADJ>
__global__ void __launch_bounds__(384) dense_split_kernel(EntryParams p, const double2* __restrict__ s,
                                                          double2* __restrict__ u, long long Nv, int L, int LQ, int nmt,
                                                          int r0, int rc, double scale, double2* __restrict__ part,
                                                          const int* __restrict__ exs, int* __restrict__ flag) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ int s_exs[16];
  const int nI = p.nI, NI = p.NI;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5, g = lane >> 2, t = lane & 3;
  const DsLayout Y(nmt, (LQ + 7) / 8, RT);
  double* M = reinterpret_cast<double*>(sm + Y.m64);
  int* mex = reinterpret_cast<int*>(sm + Y.mex);
  int* eo = reinterpret_cast<int*>(sm + Y.eo);
  int* ep = reinterpret_cast<int*>(sm + Y.ep);
  const int ntx = (p.nx + L - 1) / L;
  const int bo = blockIdx.x / ntx;
  const int ao0 = (blockIdx.x % ntx) * L;
  const int olen = min(L, p.nx - ao0);
  const long long o0 = (long long)bo * p.nx + ao0;
  const double w2 = p.omega * p.omega, w2l = fma(p.omega, p.omega, -w2), c1 = 2.0 * DS_C0 / w2;
  bool bad = false;
  __shared__ unsigned s_left;   // right-hand sides left to the FP64 kernel
  if (tid < 32) {
    const int e = tid < rc ? exs[tid] : 0;
    const unsigned left = __ballot_sync(0xffffffffu, !split_exponent_ok(e));
    if (tid < 16) s_exs[tid] = max(e, SPLIT_MIN_EXP);
    if (tid == 0) {
      s_left = left;
      if (left && blockIdx.x == 0 && blockIdx.y == 0) atomicOr(flag, (int)left);
    }
  }
  __syncthreads();
  if (s_left == (1u << rc) - 1) return;

  // rows of LX as an A fragment: cells base + g and base + 8 + g (below end), row exponents e0, e1
  auto basis_frag = [&](int base, int end, uint32_t (&a)[4][SPLIT_DIGITS], int& e0, int& e1) {
    double2 v[4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int c = base + g + 8 * h, j = 2 * t + 8 * k;
        double2 x = make_double2(0.0, 0.0);
        if (c < end) {
          const double* lx = p.LX + (size_t)c * nI;
          if (j < nI) x.x = lx[j];
          if (j + 1 < nI) x.y = lx[j + 1];
        }
        v[2 * k + h] = x;
      }
    e0 = max(block_exponent(v[0]), block_exponent(v[2]));
    e1 = max(block_exponent(v[1]), block_exponent(v[3]));
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      e0 = max_xor(e0, o);
      e1 = max_xor(e1, o);
    }
    bad = bad || !split_exponent_ok(e0) || !split_exponent_ok(e1);
    e0 = max(e0, SPLIT_MIN_EXP);
    e1 = max(e1, SPLIT_MIN_EXP);
#pragma unroll
    for (int k = 0; k < 4; ++k) split_pair(v[k], (k & 1) ? e1 : e0, 0u, a[k]);
  };

  // the outputs' bases
  if (warp < nmt) {
    uint32_t a[4][SPLIT_DIGITS];
    int e0, e1;
    basis_frag(ao0 + 16 * warp, ao0 + olen, a, e0, e1);
#pragma unroll
    for (int d = 0; d < SPLIT_DIGITS; ++d)
      *reinterpret_cast<uint4*>(sm + Y.lxo + ((warp * SPLIT_DIGITS + d) * 32 + lane) * 4) =
          make_uint4(a[0][d], a[1][d], a[2][d], a[3][d]);
    if (t == 0) {
      eo[16 * warp + g] = e0;
      eo[16 * warp + 8 + g] = e1;
    }
  }

  const int mt = warp % nmt, part_of = warp / nmt, nparts = nwarp / nmt;   // nmt divides the warps (launch)
  // running sums: element e of tile (rt, re / im): output 16 mt + g + 8 (e >> 1), right-hand side 8 rt + 2t + (e & 1)
  long long hi[RT][2][4], lo[RT][2][4];
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
      for (int e = 0; e < 4; ++e) hi[r][z][e] = lo[r][z][e] = 0;
  int erun = SPLIT_MIN_EXP;

  const int bq0 = (int)((long long)p.ny * blockIdx.y / gridDim.y);
  const int bq1 = (int)((long long)p.ny * (blockIdx.y + 1) / gridDim.y);
  for (int bq = bq0; bq < bq1; ++bq) {
    __syncthreads();
    // M[q][i1][j1] = sum_i2 LZ[bo][i2] H[q][bq][(i2,i1)][j1], zero past nI
    for (int idx = tid; idx < 3 * DS_K * DS_K; idx += blockDim.x) {
      const int q = idx / (DS_K * DS_K), i1 = (idx / DS_K) % DS_K, j1 = idx % DS_K;
      double a = 0.0;
      if (i1 < nI && j1 < nI) {
        const double* Hq = p.H + (((size_t)q * p.ny + bq) * NI) * nI;
        for (int i2 = 0; i2 < nI; ++i2)
          a = fma(p.LZ[(size_t)bo * nI + i2], Hq[(size_t)(i2 * nI + i1) * nI + j1], a);
        if (q == 1) a *= DS_C0;
        if (q == 2) a *= c1;
      }
      M[idx] = a;
    }
    __syncthreads();
    // its B fragments: column n = i1 = 8 nt + g, k = j1
    if (warp < 6) {
      const int q = warp >> 1, i1 = 8 * (warp & 1) + g;
      const double* row = M + (q * DS_K + i1) * DS_K;
      const double2 v0 = make_double2(row[2 * t], row[2 * t + 1]), v1 = make_double2(row[2 * t + 8], row[2 * t + 9]);
      int e = max(block_exponent(v0), block_exponent(v1));
      e = max_xor(max_xor(e, 1), 2);
      bad = bad || !split_exponent_ok(e);
      e = max(e, SPLIT_MIN_EXP);
      if (t == 0) mex[q * DS_K + i1] = e;
      uint32_t b0[SPLIT_DIGITS], b1[SPLIT_DIGITS];
      split_pair(v0, e, 0u, b0);
      split_pair(v1, e, 0u, b1);
#pragma unroll
      for (int d = 0; d < SPLIT_DIGITS; ++d)
        *reinterpret_cast<uint2*>(sm + Y.mfrag + ((warp * SPLIT_DIGITS + d) * 32 + lane) * 2) = make_uint2(b0[d], b1[d]);
    }
    __syncthreads();
    for (int aq0 = 0; aq0 < p.nx; aq0 += LQ) {
      const int qlen = min(LQ, p.nx - aq0), ntile = (qlen + 7) / 8;
      if (aq0) __syncthreads();   // the last segment's fragments are read
      // P of 16 cells per warp and turn, as the B fragments of two n-tiles
      for (int mc = warp; 2 * mc < ntile; mc += nwarp) {
        uint32_t a[4][SPLIT_DIGITS];
        int e0, e1;
        basis_frag(aq0 + 16 * mc, aq0 + qlen, a, e0, e1);
#pragma unroll 1
        for (int q = 0; q < 3; ++q) {
          double2 P[2][2];   // [cell half][i1 half]: i1 = 8 nt + 2t, + 1
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) {
            float acc[DS_DIAGS][4];
            const uint32_t* bf = sm + Y.mfrag + ((2 * q + nt) * SPLIT_DIGITS * 32 + lane) * 2;
            digit_mma(acc, [&](int i) { return make_uint4(a[0][i], a[1][i], a[2][i], a[3][i]); },
                      [&](int j) { return *reinterpret_cast<const uint2*>(bf + j * 64); });
            double v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              long long h, l;
              digit_sums(acc, e, h, l);
              v[e] = fixed_to_double(h, l, ((e & 2) ? e1 : e0) + mex[q * DS_K + 8 * nt + 2 * t + (e & 1)] - 2 * SPLIT_EXP_BIAS);
            }
            P[0][nt] = make_double2(v[0], v[1]);
            P[1][nt] = make_double2(v[2], v[3]);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            int e = max(block_exponent(P[h][0]), block_exponent(P[h][1]));
            e = max_xor(max_xor(e, 1), 2);
            bad = bad || !split_exponent_ok(e);
            e = max(e, SPLIT_MIN_EXP);
            const int tile = 2 * mc + h;
            if (tile < ntile) {
              if (t == 0) ep[q * 8 * ((LQ + 7) / 8) + 8 * tile + g] = e;
              uint32_t b0[SPLIT_DIGITS], b1[SPLIT_DIGITS];
              split_pair(P[h][0], e, 0u, b0);
              split_pair(P[h][1], e, 0u, b1);
#pragma unroll
              for (int d = 0; d < SPLIT_DIGITS; ++d)
                *reinterpret_cast<uint2*>(sm + Y.pfrag + (((tile * 3 + q) * SPLIT_DIGITS + d) * 32 + lane) * 2) =
                    make_uint2(b0[d], b1[d]);
            }
          }
        }
      }
      // the sources' B fragments: column n = right-hand side 8 rt + g, inputs 2t and 2t + 1 of the n-tile
      for (int w = warp; w < ntile * RT; w += nwarp) {
        const int tile = w / RT, r = 8 * (w % RT) + g;
        double2 v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int c = 8 * tile + 2 * t + k;
          v[k] = (r < rc && c < qlen) ? s[(size_t)(r0 + r) * Nv + (size_t)bq * p.nx + aq0 + c] : make_double2(0.0, 0.0);
        }
        uint32_t b0[SPLIT_DIGITS], b1[SPLIT_DIGITS];
        split_pair(v[0], s_exs[r], 0u, b0);
        split_pair(v[1], s_exs[r], 0u, b1);
#pragma unroll
        for (int d = 0; d < SPLIT_DIGITS; ++d)
          *reinterpret_cast<uint2*>(sm + Y.sfrag + ((w * SPLIT_DIGITS + d) * 32 + lane) * 2) = make_uint2(b0[d], b1[d]);
      }
      __syncthreads();
      const uint32_t* af = sm + Y.lxo + (mt * SPLIT_DIGITS * 32 + lane) * 4;
      for (int tile = part_of; tile < ntile; tile += nparts) {
        // the entries (o, c): o = 16 mt + g + 8 (e >> 1), c = 8 tile + 2t + (e & 1)
        double f[3][4];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          float acc[DS_DIAGS][4];
          const uint32_t* bf = sm + Y.pfrag + ((tile * 3 + q) * SPLIT_DIGITS * 32 + lane) * 2;
          digit_mma(acc, [&](int i) { return *reinterpret_cast<const uint4*>(af + i * 128); },
                    [&](int j) { return *reinterpret_cast<const uint2*>(bf + j * 64); });
          const int* eq = ep + q * 8 * ((LQ + 7) / 8) + 8 * tile + 2 * t;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            long long h, l;
            digit_sums(acc, e, h, l);
            f[q][e] = fixed_to_double(h, l, eo[16 * mt + g + 8 * (e >> 1)] + eq[e & 1] - 2 * SPLIT_EXP_BIAS);
          }
        }
        double2 gv[4];
        int eg = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int o = 16 * mt + g + 8 * (e >> 1), c = 8 * tile + 2 * t + (e & 1);
          double2 v = make_double2(0.0, 0.0);
          if (o < olen && c < qlen) {
            if ((long long)bq * p.nx + aq0 + c == o0 + o) {
              v = p.self[o0 + o];
            } else {
              // g = i v0 H0 - i v1 x H1 (the constants are in P)
              const HankelFG h = hankel_of_t2(p.hank, w2, w2l, f[0][e]);
              v = make_double2(fma(-h.F.y, f[1][e], h.G.y * f[2][e]), fma(h.F.x, f[1][e], -h.G.x * f[2][e]));
            }
          }
          gv[e] = v;
          eg = max(eg, block_exponent(v));
        }
        eg = __reduce_max_sync(0xffffffffu, eg);
        if (eg == 0) continue;
        bad = bad || !split_exponent_ok(eg);
        eg = max(eg, SPLIT_MIN_EXP);
        uint32_t a[4][SPLIT_DIGITS];
        split_pair(gv[0], eg, ADJ ? DS_IM : 0u, a[0]);
        split_pair(gv[2], eg, ADJ ? DS_IM : 0u, a[1]);
        split_pair(gv[1], eg, ADJ ? DS_IM : 0u, a[2]);
        split_pair(gv[3], eg, ADJ ? DS_IM : 0u, a[3]);
        if (eg > erun) {
          const int d = eg - erun;
          erun = eg;
#pragma unroll
          for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int z = 0; z < 2; ++z)
#pragma unroll
              for (int e = 0; e < 4; ++e) shift_sums(hi[r][z][e], lo[r][z][e], d);
        }
        const int d = erun - eg;
#pragma unroll
        for (int r = 0; r < RT; ++r) {
          const uint32_t* bf = sm + Y.sfrag + ((tile * RT + r) * SPLIT_DIGITS * 32 + lane) * 2;
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            float acc[SPLIT_DIGITS][4];
            digit_mma(acc, [&](int i) { return make_uint4(a[0][i], a[1][i], a[2][i], a[3][i]); },
                      [&](int j) {
                        const uint2 w = *reinterpret_cast<const uint2*>(bf + j * 64);
                        return z == 0 ? make_uint2(w.x ^ DS_IM, w.y ^ DS_IM)
                                      : make_uint2(__byte_perm(w.x, 0, 0x1032), __byte_perm(w.y, 0, 0x1032));
                      });
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              long long h, l;
              digit_sums(acc, e, h, l);
              if (d) shift_sums(h, l, d);
              hi[r][z][e] += h;
              lo[r][z][e] += l;
            }
          }
        }
      }
    }
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) atomicOr(flag, 0xffff);
    return;
  }
  // the parts' sums, added in order: part 0 keeps its own in registers
  double2* red = reinterpret_cast<double2*>(sm);   // [part - 1][m-tile][rt][e][lane]
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int ex = erun + s_exs[8 * r + 2 * t + (e & 1)] - 2 * SPLIT_EXP_BIAS;
      const double2 v = make_double2(fixed_to_double(hi[r][0][e], lo[r][0][e], ex), fixed_to_double(hi[r][1][e], lo[r][1][e], ex));
      red[(((part_of * nmt + mt) * RT + r) * 4 + e) * 32 + lane] = v;
    }
  __syncthreads();
  if (part_of) return;
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int o = 16 * mt + g + 8 * (e >> 1), rr = 8 * r + 2 * t + (e & 1);
      if (o >= olen || rr >= rc || (s_left >> rr & 1)) continue;
      double2 a = make_double2(0.0, 0.0);
      for (int q = 0; q < nparts; ++q) {
        const double2 v = red[(((q * nmt + mt) * RT + r) * 4 + e) * 32 + lane];
        a.x += v.x;
        a.y += v.y;
      }
      if (part) part[((size_t)blockIdx.y * rc + rr) * Nv + o0 + o] = a;
      else u[(size_t)(r0 + rr) * Nv + o0 + o] = make_double2(a.x * scale, a.y * scale);
    }
}

template <int RT, bool ADJ>
void launch(const EntryParams& p, const double2* s, double2* u, long long Nv, int L, int nsplit, int r0, int rc, double scale,
            double2* part, const int* exs, int* flag, cudaStream_t st) {
  const int nmt = (L + 15) / 16;
  const int segs = (p.nx + 8 * DS_NT - 1) / (8 * DS_NT), LQ = (p.nx + segs - 1) / segs;
  // twelve warps (all the registers hold) where the segment has three or four
  // m-tiles: eight leave three m-tiles unevenly spread over the SM's
  // sub-partitions, and 64^2 2.05 -> 1.97 ms, 120 x 100 16.6 -> 14.7, 100 x 80 x 5
  // 9.25 -> 8.45; below that level (24^2), or slower (32^2 x 16: 384 -> 392 us).
  // 1, 2, 3 and 4 divide their count.
  const int warps = nmt >= 3 ? 12 : 8;
  const DsLayout Y(nmt, (LQ + 7) / 8, RT);
  const size_t red = (size_t)(warps / nmt) * nmt * RT * 4 * 32 * sizeof(double2);
  const size_t smem = std::max((size_t)Y.words * 4, red);
  auto k = dense_split_kernel<RT, ADJ>;
  HB_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k<<<dim3((unsigned)((p.nx + L - 1) / L * p.ny), (unsigned)nsplit), 32 * warps, smem, st>>>(
      p, s, u, Nv, L, LQ, nmt, r0, rc, scale, part, exs, flag);
  HB_CHECK_LAUNCH();
}

}  // namespace

// rc <= 16 right-hand sides from r0 on; exs: 16 exponents and, behind them, the flags (all zeroed here)
void dense_split(const EntryParams& p, const double2* s, double2* u, long long Nv, int L, int nsplit, int r0, int rc,
                 int adjoint, double scale, double2* part, int* exs, cudaStream_t st) {
  int* flag = exs + 16;
  HB_CUDA(cudaMemsetAsync(exs, 0, 17 * sizeof(int), st));
  rhs_exponent_kernel<<<dim3((unsigned)std::max<long long>(1, std::min<long long>((Nv + 1023) / 1024, 64)), (unsigned)rc), 256, 0,
                        st>>>(s + (size_t)r0 * Nv, Nv, exs);
  HB_CHECK_LAUNCH();
  if (rc <= 8) {
    if (adjoint) launch<1, true>(p, s, u, Nv, L, nsplit, r0, rc, scale, part, exs, flag, st);
    else launch<1, false>(p, s, u, Nv, L, nsplit, r0, rc, scale, part, exs, flag, st);
  } else {
    if (adjoint) launch<2, true>(p, s, u, Nv, L, nsplit, r0, rc, scale, part, exs, flag, st);
    else launch<2, false>(p, s, u, Nv, L, nsplit, r0, rc, scale, part, exs, flag, st);
  }
}

}  // namespace hb
