// apply.cu - butterfly / HODBF apply and its adjoint on the device
// (Sec. 4.2.1, Eq. butterfly_mat, Eq. butterfly_factors; Sec. 4.2 HODBF).
//
//   x  = h^2 s, gathered into cluster-tree order            (Eq. m_v2v)
//   steps of small dense products over all butterflies      (build.cu plans)
//   u  = y scattered back to natural order
//
// FP64 path: complex128 factors and vectors, the step tasks' products on the
// FP16 tensor cores by integer digits, as accurate as FP64 FMAs as long as a
// factor row and a right-hand side of a task do not hide one another's small
// values (split_fixed.cuh; inclusion.cu keeps the segment lengths out of them
// for that).  Mixed path (HB_MIXED_BF16X3): split-BF16 factors and vectors in
// the MMA-fragment layout of bf_mma.cu, up to 32 right-hand sides per pass.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <tuple>
#include <vector>

#include "hb_internal.cuh"
#include "split_fixed.cuh"

namespace hb {

// x[p][r] = scale * s[r*Nv + perm[p]]   (column-major natural -> row-major tree order)
// for tree positions p in [lo, hi); 0 elsewhere (a shard's share of the
// input).  blockDim.x = R rounded up to a power of two: lane -> right-hand side.
__global__ void gather_kernel(const double2* __restrict__ s, const long long* __restrict__ perm,
                              double2* __restrict__ x, long long Nv, int R, double scale, long long lo, long long hi) {
  const int r = threadIdx.x;
  if (r >= R) return;
  for (long long p = (long long)blockIdx.x * blockDim.y + threadIdx.y; p < Nv; p += (long long)gridDim.x * blockDim.y) {
    const double2 v = (p >= lo && p < hi) ? s[(size_t)r * Nv + perm[p]] : make_double2(0.0, 0.0);
    x[p * R + r] = make_double2(v.x * scale, v.y * scale);
  }
}

// u[r*Nv + perm[p]] = y[p][r] for tree positions p in [lo, hi)
__global__ void scatter_kernel(const double2* __restrict__ y, const long long* __restrict__ perm,
                               double2* __restrict__ u, long long Nv, int R, long long lo, long long hi) {
  const int r = threadIdx.x;
  if (r >= R) return;
  for (long long p = lo + (long long)blockIdx.x * blockDim.y + threadIdx.y; p < hi;
       p += (long long)gridDim.x * blockDim.y)
    u[(size_t)r * Nv + perm[p]] = y[(size_t)p * R + r];
}

// ------------------------------------------------------- step tasks ----
// Y = op(F) X of the step tasks on the FP16 tensor cores by integer digits
// (split_fixed.cuh), in the orientation of the mixed apply: the MMA's M is
// right-hand sides, N outputs, K = 2 x 8 inputs with real and imaginary
// parts interleaved; D_r takes A rows (Re X, -Im X), D_i (Im X, Re X).  Up to
// eight right-hand sides (HALF) both go into one MMA, rows 0-7 and 8-15.
//
// A unit is one n-tile (8 outputs) of one task.  A CTA takes an item: units of
// tasks that read the same inputs (the two transfer blocks of a skeleton, the
// V^0 of every HODBF level and the dense block of a leaf; the tasks of a step
// are kept in input order).  It scales X per right-hand side, splits it into
// digit fragments in shared memory once, TASK_KC k-steps at a time, and every
// warp streams its unit's F from global memory into registers, one k-step
// ahead, scaling it per output row (unit.fe, found when the plan is made) and
// splitting it there: a row far below the others of its task keeps its bits,
// as in a plain FP64 sum.  Long sums (ks k-steps) are dealt over kw(ks) warps and
// the integer sums added.  A unit's sums depend on its task alone, so a
// shard's equal the whole apply's.
//
// Bound by instruction issue: per 8 outputs x 8 inputs 42 (21) MMAs and
// about 250 other instructions of a warp, as many as that to split X where a task's rank
// is near 16, and the epilogue, against 1024 x 4 FP64 FMAs for 16
// right-hand sides (2048 cycles of an SM's FP64 unit).  Measured: 192^2 x 16
// 3.67 ms with one FP64 FMA loop per output, 1.92 with a CTA of 8 warps per
// task, 1.28 with four warps and shared inputs; 120 x 88 adjoint x 5: 601,
// 251, 207 us (205 with one exponent a task, the same in every lane).
constexpr int TASK_KC = 16;              // k-steps of X held at a time
constexpr uint32_t SPLIT_IM_SIGN = 0x80000000u;
// Warps sharing a unit's k-steps: one where a warp's own sums are short beside
// the exchange, more where a step has few long ones.  Measured (us; 192^2 x 16 /
// 120 x 88 adjoint x 5 / 64^2 x 5 / inclusion at 128^2 with 512 segments x 8):
// always one 1270 / 217 / 109 / 366; two and four from 25 and 65 k-steps on
// 1307 / 216 / 109 / 351, from 13 and 33 1315 / 218 / 107 / 294, from 7 and 17
// 1337 / 223 / 104 / 275.
constexpr int task_kw(int ks, int W) {
  const int k = ks <= 12 ? 1 : ks <= 32 ? 2 : 4;
  return k < W ? k : W;
}

// Rows [row0, row1) of a task with plain FP64 FMAs, one warp, for the
// right-hand sides in the mask: those whose inputs the digits do not hold, or
// all when the factors are so (lane -> (row, right-hand side), rows fastest).
__device__ __noinline__ void task_plain(const Task* __restrict__ task, const double2* __restrict__ F, double2* x, double2* y,
                                        double2* xh, int R, int row0, int row1, unsigned mask) {
  const Task& tk = *task;
  double2* bufs[3] = {x, y, xh};
  double2* out = bufs[tk.y_buf] + (size_t)tk.y_off * R;
  const int rows = row1 - row0, total = rows * R;
  for (int idx = threadIdx.x & 31; idx < total; idx += 32) {
    const int row = row0 + idx % rows, rr = idx / rows;
    if (!(mask >> rr & 1)) continue;
    double ar = 0, ai = 0;
    for (int t = 0; t < tk.nterm; ++t) {
      const double2* f = F + tk.f_off[t];
      const double2* xin = bufs[tk.x_buf] + (size_t)tk.x_off[t] * R + rr;
      const int rin = tk.r_in[t];
      if (!tk.conj_t) {
        for (int k = 0; k < rin; ++k) {
          const double2 a = f[(size_t)k * tk.r_out + row];
          const double2 v = xin[(size_t)k * R];
          ar = fma(a.x, v.x, fma(-a.y, v.y, ar));
          ai = fma(a.x, v.y, fma(a.y, v.x, ai));
        }
      } else {
        const double2* fr = f + (size_t)row * rin;
        for (int k = 0; k < rin; ++k) {
          const double2 a = fr[k];
          const double2 v = xin[(size_t)k * R];
          ar = fma(a.x, v.x, fma(a.y, v.y, ar));     // conj(a) v
          ai = fma(a.x, v.y, fma(-a.y, v.x, ai));
        }
      }
    }
    double2* o = out + (size_t)row * R + rr;
    if (tk.accumulate) {
      const double2 prev = *o;
      ar += prev.x;
      ai += prev.y;
    }
    *o = make_double2(ar, ai);
  }
}

template <bool HALF, int W>
__global__ void __launch_bounds__(32 * W, 16 / W)
    task_kernel(const TaskItem* __restrict__ items, const TaskUnit* __restrict__ units,
                const Task* __restrict__ tasks, const double2* __restrict__ F, double2* x, double2* y, double2* xh, int R) {
  constexpr int NR = HALF ? 8 : 16;        // right-hand sides of the MMA rows
  constexpr int NE = HALF ? 4 : 8;         // accumulator elements per lane and digit diagonal
  constexpr int XW = HALF ? 2 : 4;         // X fragment words per lane
  constexpr int XK = 32 * W / NR;          // inputs the CTA's threads take at once
  extern __shared__ __align__(16) uint32_t xs[];   // [k-step][digit][lane][XW]
  __shared__ int s_ex[16];
  __shared__ unsigned s_bad;   // right-hand sides that the digits do not hold
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const TaskItem item = items[blockIdx.x];
  const int rin0 = item.r_in[0], rin1 = item.r_in[1];
  const double2* xin = item.x_buf == 0 ? x : item.x_buf == 1 ? y : xh;
  const double2* xin0 = xin + item.x_off[0] * R;
  const double2* xin1 = xin + item.x_off[1] * R;
  const int ks0 = (rin0 + 7) / 8, ks = ks0 + (rin1 + 7) / 8;
  const int kw = task_kw(ks, W), uw = W / kw;
  const int wt = warp % uw, kp = warp / uw;

  // the warp's unit, and F values (row, k = 2t) and (row, 2t + 1) of its k-step q
  bool work = false, rok = false;
  TaskUnit unit;
  int fe = 0, row = 0;   // of row 8 tile + g
  double2 f0, f1;
  auto load_f = [&](int q) {
    f0 = f1 = make_double2(0.0, 0.0);
    if (!rok || q >= ks) return;
    const bool term = q >= ks0;
    const int rin = term ? rin1 : rin0;
    const int k = 8 * (term ? q - ks0 : q) + 2 * t;
    const double2* f = F + (term ? unit.f_off[1] : unit.f_off[0]);
    const double2* p0 = unit.conj_t ? f + (size_t)row * rin + k : f + (size_t)k * unit.r_out + row;
    const double2* p1 = unit.conj_t ? p0 + 1 : p0 + unit.r_out;
    if (k < rin) f0 = __ldcs(p0);
    if (k + 1 < rin) f1 = __ldcs(p1);
  };
  auto take_unit = [&](int u0) {
    work = u0 + wt < item.units;
    const int at = item.unit0 + (work ? u0 + wt : 0);
    unit = units[at];
    fe = units[at].fe[g];
    row = 8 * unit.tile + g;
    rok = work && row < unit.r_out;
    load_f(kp);
  };
  take_unit(0);

  // value `k` (of the padded, concatenated inputs) of right-hand side xr
  const int xr = tid & (NR - 1), xk = tid / NR;
  auto load_x = [&](int k) {
    const bool term = k >= 8 * ks0;
    const int kin = term ? k - 8 * ks0 : k;
    double2 v = make_double2(0.0, 0.0);
    if (xr < R && kin < (term ? rin1 : rin0)) v = (term ? xin1 : xin0)[(size_t)kin * R + xr];
    return v;
  };

  // the exponent of every right-hand side over the inputs
  if (tid < 16) s_ex[tid] = 0;
  if (tid == 0) s_bad = 0;
  int ex = 0;
  for (int k = xk; k < 8 * ks; k += XK) ex = max(ex, block_exponent(load_x(k)));
  __syncthreads();
  if (ex) atomicMax(&s_ex[xr], ex);
  __syncthreads();
  const int myex = max(s_ex[xr], SPLIT_MIN_EXP);
  if (tid < R && !split_exponent_ok(s_ex[tid])) atomicOr(&s_bad, 1u << tid);   // read after the next barrier

  // X of k-steps [c0, c1) into digit fragments: word j of lane (g, t) is
  // (right-hand side g + 8 (j & 1), input 2t + (j >> 1)); HALF: (g, 2t + j)
  auto split_x = [&](int k, int c0, double2 v) {
    const int q = k >> 3, kk = k & 7;
    uint32_t w[SPLIT_DIGITS];
    split_pair(v, myex, 0u, w);
    const int j = HALF ? (kk & 1) : 2 * (kk & 1) + (xr >> 3);
    uint32_t* dst = xs + (((q - c0) * SPLIT_DIGITS) * 32 + (xr & 7) * 4 + (kk >> 1)) * XW + j;
#pragma unroll
    for (int s = 0; s < SPLIT_DIGITS; ++s) dst[s * 32 * XW] = w[s];
  };

  for (int u0 = 0; u0 < item.units; u0 += uw) {   // several passes only when X is held whole
    if (u0) take_unit(u0);
    const bool fok = __all_sync(0xffffffffu, split_exponent_ok(fe));   // the digits hold every row of the unit
    const int fx = max(fe, SPLIT_MIN_EXP);
    float acc[SPLIT_ACC][NE];
    long long hi[NE], lo[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      hi[e] = lo[e] = 0;
#pragma unroll
      for (int d = 0; d < SPLIT_ACC; ++d) acc[d][e] = 0.f;
    }
    for (int c0 = 0; c0 < ks; c0 += TASK_KC) {
      const int c1 = min(ks, c0 + TASK_KC);
      if (u0 == 0) {
        if (c0) __syncthreads();
        for (int k = 8 * c0 + xk; k < 8 * c1; k += XK) split_x(k, c0, load_x(k));
        __syncthreads();
      }
      if (work && fok) {
        int since = 0;
        for (int q = c0 + kp; q < c1; q += kw) {   // TASK_KC is a multiple of kw
          const double2 a0 = f0, a1 = f1;
          load_f(q + kw);
          uint32_t b0[SPLIT_DIGITS], b1[SPLIT_DIGITS];
          const uint32_t cs = unit.conj_t ? 0x80000000u : 0u;
          split_pair(a0, fx, cs, b0);
          split_pair(a1, fx, cs, b1);
          const uint32_t* xq = xs + ((q - c0) * SPLIT_DIGITS * 32 + lane) * XW;
#pragma unroll
          for (int i = 0; i < SPLIT_DIGITS; ++i) {
            if constexpr (HALF) {
              const uint2 w = *reinterpret_cast<const uint2*>(xq + i * 32 * XW);
              const uint32_t a[4] = {w.x ^ SPLIT_IM_SIGN, __byte_perm(w.x, 0, 0x1032), w.y ^ SPLIT_IM_SIGN,
                                     __byte_perm(w.y, 0, 0x1032)};
#pragma unroll
              for (int j = 0; i + j < SPLIT_DIGITS; ++j)
                mma_f16(acc[i == 2 && j == 0 ? 6 : i + j], a[0], a[1], a[2], a[3], b0[j], b1[j]);
            } else {
              const uint4 w = *reinterpret_cast<const uint4*>(xq + i * 32 * XW);
              const uint32_t r[4] = {w.x ^ SPLIT_IM_SIGN, w.y ^ SPLIT_IM_SIGN, w.z ^ SPLIT_IM_SIGN, w.w ^ SPLIT_IM_SIGN};
              const uint32_t m[4] = {__byte_perm(w.x, 0, 0x1032), __byte_perm(w.y, 0, 0x1032),
                                     __byte_perm(w.z, 0, 0x1032), __byte_perm(w.w, 0, 0x1032)};
#pragma unroll
              for (int j = 0; i + j < SPLIT_DIGITS; ++j) {
                const int d = i == 2 && j == 0 ? 6 : i + j;
                mma_f16(acc[d], r[0], r[1], r[2], r[3], b0[j], b1[j]);
                mma_f16(acc[d] + 4, m[0], m[1], m[2], m[3], b0[j], b1[j]);
              }
            }
          }
          if (++since == 2 || q + kw >= c1) {
            since = 0;
#pragma unroll
            for (int e = 0; e < NE; ++e)
              split_flush(acc[0][e], acc[1][e], acc[2][e], acc[3][e], acc[4][e], acc[5][e], acc[6][e], hi[e], lo[e]);
          }
        }
      }
    }
    // add the shares of the k-steps (kw > 1: one pass)
    if (kw > 1) {
      longlong2* red = reinterpret_cast<longlong2*>(xs);   // [kp - 1][unit][element][lane]
      __syncthreads();
      if (work && kp > 0)
#pragma unroll
        for (int e = 0; e < NE; ++e) red[(((kp - 1) * uw + wt) * NE + e) * 32 + lane] = make_longlong2(hi[e], lo[e]);
      __syncthreads();
      if (kp == 0)
        for (int p = 0; p < kw - 1; ++p)
#pragma unroll
          for (int e = 0; e < NE; ++e) {
            const longlong2 v = red[((p * uw + wt) * NE + e) * 32 + lane];
            hi[e] += v.x;
            lo[e] += v.y;
          }
    }
    if (!work || kp > 0) continue;
    const unsigned plain = fok ? s_bad : 0xffffu;
    double2* out = (unit.y_buf == 0 ? x : unit.y_buf == 1 ? y : xh) + (size_t)unit.y_off * R;
    const int fo[2] = {__shfl_sync(0xffffffffu, fx, 8 * t), __shfl_sync(0xffffffffu, fx, 8 * t + 4)};   // of rows 2t, 2t + 1
    // element e of D: right-hand side g + 8 (e >> 1), output 2t + (e & 1); HALF:
    // elements 0, 1 are D_r and 2, 3 D_i of right-hand side g
#pragma unroll
    for (int e = 0; e < NE / 2; ++e) {
      const int rr = HALF ? g : g + 8 * (e >> 1);
      const int ro = 8 * unit.tile + 2 * t + (e & 1);
      if (rr >= R || ro >= unit.r_out || (plain >> rr & 1)) continue;
      const int sx = fo[e & 1] + max(s_ex[rr], SPLIT_MIN_EXP) - 2 * SPLIT_EXP_BIAS;
      const int ei = HALF ? e + 2 : e + 4;
      double2 v = make_double2(fixed_to_double(hi[e], lo[e], sx), fixed_to_double(hi[ei], lo[ei], sx));
      double2* o = out + (size_t)ro * R + rr;
      if (unit.accumulate) {
        const double2 prev = *o;
        v.x += prev.x;
        v.y += prev.y;
      }
      *o = v;
    }
    if (plain) task_plain(tasks + unit.task, F, x, y, xh, R, 8 * unit.tile, min(unit.r_out, 8 * unit.tile + 8), plain);
  }
}

// units[u].fe[g] = the largest exponent of row g of unit u (0 past the task's rows), one warp a unit
__global__ void __launch_bounds__(256) unit_exponent_kernel(TaskUnit* __restrict__ units, const Task* __restrict__ tasks,
                                                            const double2* __restrict__ F, int n) {
  const int u = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  if (u >= n) return;
  const TaskUnit unit = units[u];
  const Task& tk = tasks[unit.task];
  const int row = 8 * unit.tile + g;
  int e = 0;
  if (row < unit.r_out)
    for (int q = 0; q < tk.nterm; ++q) {
      const int rin = tk.r_in[q];
      const double2* f = F + unit.f_off[q] + (unit.conj_t ? (size_t)row * rin : (size_t)row);
      const size_t step = unit.conj_t ? 1 : (size_t)unit.r_out;
#pragma unroll 4
      for (int k = t; k < rin; k += 4) e = max(e, block_exponent(f[k * step]));
    }
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
  if (t == 0) units[u].fe[g] = (unsigned short)e;
}

void task_exponents(const TaskPlan& P, const Task* d_tasks, const double2* F, cudaStream_t st) {
  if (P.units == 0) return;
  unit_exponent_kernel<<<(unsigned)((P.units + 7) / 8), 256, 0, st>>>(P.d_units, d_tasks, F, P.units);
  HB_CHECK_LAUNCH();
}

bool task_reads_before(const Task& a, const Task& b) {
  auto key = [](const Task& t) {
    return std::make_tuple((int)t.x_buf, t.x_off[0], t.r_in[0], (int)t.nterm, t.nterm > 1 ? t.x_off[1] : -1LL,
                           t.nterm > 1 ? t.r_in[1] : 0);
  };
  return key(a) < key(b);
}

TaskPlan task_plan(const std::vector<Task>& tasks, const std::vector<int>& begin, int W) {
  TaskPlan P;
  P.W = W;
  std::vector<TaskUnit> units;
  std::vector<TaskItem> items;
  for (size_t s = 0; s + 1 < begin.size(); ++s) {
    P.item_begin.push_back((int)items.size());
    int max_ks = 1;
    long long nu = 0;
    for (int i = begin[s]; i < begin[s + 1]; ++i) nu += (tasks[(size_t)i].r_out + 7) / 8;
    for (int i = begin[s]; i < begin[s + 1];) {
      const Task& t = tasks[(size_t)i];
      const int ks = (t.r_in[0] + 7) / 8 + (t.nterm > 1 ? (t.r_in[1] + 7) / 8 : 0);
      max_ks = std::max(max_ks, ks);
      const int first = (int)units.size();
      int j = i;
      for (; j < begin[s + 1] && !task_reads_before(t, tasks[(size_t)j]) && !task_reads_before(tasks[(size_t)j], t); ++j)
        for (int q = 0; q < (tasks[(size_t)j].r_out + 7) / 8; ++q) {
          const Task& tj = tasks[(size_t)j];
          TaskUnit u{};
          u.f_off[0] = tj.f_off[0];
          u.f_off[1] = tj.f_off[1];
          u.y_off = tj.y_off;
          u.task = j;
          u.tile = q;
          u.r_out = tj.r_out;
          u.conj_t = tj.conj_t;
          u.y_buf = tj.y_buf;
          u.accumulate = tj.accumulate;
          units.push_back(u);
        }
      // units per CTA: one pass of its warps; up to three (X split once for
      // all) while the step still has two CTAs for every SM's four
      const int uw = W / task_kw(ks, W);
      const int passes = ks > TASK_KC || task_kw(ks, W) > 1 ? 1 : (int)std::max<long long>(1, std::min<long long>(3, nu / uw / 1216));
      const int per = uw * passes, all = (int)units.size() - first, cut = (all + per - 1) / per;
      for (int c = 0; c < cut; ++c) {   // equal shares
        const int a = (int)((long long)all * c / cut), b = (int)((long long)all * (c + 1) / cut);
        TaskItem it{};
        it.unit0 = first + a;
        it.units = b - a;
        it.x_buf = t.x_buf;
        it.r_in[0] = t.r_in[0];
        it.r_in[1] = t.nterm > 1 ? t.r_in[1] : 0;
        it.x_off[0] = t.x_off[0];
        it.x_off[1] = t.nterm > 1 ? t.x_off[1] : 0;
        items.push_back(it);
      }
      i = j;
    }
    P.max_ks.push_back(max_ks);
  }
  P.item_begin.push_back((int)items.size());
  P.units = (int)units.size();
  P.d_units = upload(units);
  try {
    P.d_items = upload(items);
    HB_CUDA(cudaStreamSynchronize(0));   // the host arrays end here
  } catch (...) {
    task_plan_free(P);
    throw;
  }
  return P;
}

void task_plan_free(TaskPlan& P) {
  dev_free(P.d_units);
  dev_free(P.d_items);
  P = TaskPlan{};
}

void ensure_task_plans(hb_ctx* c) {
  for (int dir = 0; dir < 2; ++dir) {
    if (c->d_tasks[dir]) continue;
    TaskPlan P = task_plan(c->tasks_h[dir], c->step_begin[dir], 4);
    Task* d = nullptr;
    try {
      d = upload(c->tasks_h[dir]);
      task_exponents(P, d, c->d_f64, 0);
      HB_CUDA(cudaStreamSynchronize(0));
    } catch (...) {
      task_plan_free(P);
      dev_free(d);
      throw;
    }
    c->task_plans[dir] = P;
    c->d_tasks[dir] = d;
  }
}

template <bool HALF, int W>
static void launch_tasks(const TaskPlan& P, int step, const Task* tasks, const double2* F, double2* x, double2* y, double2* xh,
                         int R, cudaStream_t st) {
  const int n = P.item_begin[(size_t)step + 1] - P.item_begin[(size_t)step];
  if (n <= 0) return;
  const size_t frag = (size_t)std::min(TASK_KC, P.max_ks[(size_t)step]) * SPLIT_DIGITS * 32 * (HALF ? 2 : 4) * 4;
  const size_t red = (size_t)(W - 1) * 32 * (HALF ? 4 : 8) * sizeof(longlong2);
  const size_t smem = P.max_ks[(size_t)step] > 12 ? std::max(frag, red) : frag;
  HB_CUDA(cudaFuncSetAttribute(task_kernel<HALF, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, 56 << 10));
  task_kernel<HALF, W><<<n, 32 * W, smem, st>>>(P.d_items + P.item_begin[(size_t)step], P.d_units, tasks, F, x, y, xh, R);
  HB_CHECK_LAUNCH();
}

void run_tasks_fp64(const TaskPlan& P, int step, const Task* d_tasks, const double2* F, double2* x, double2* y,
                    double2* xh, int R, cudaStream_t st) {
  if (P.W == 4) {
    if (R <= 8) launch_tasks<true, 4>(P, step, d_tasks, F, x, y, xh, R, st);
    else launch_tasks<false, 4>(P, step, d_tasks, F, x, y, xh, R, st);
  } else {
    if (R <= 8) launch_tasks<true, 8>(P, step, d_tasks, F, x, y, xh, R, st);
    else launch_tasks<false, 8>(P, step, d_tasks, F, x, y, xh, R, st);
  }
}

namespace {

struct TimerScope {
  hb_ctx* c;
  cudaStream_t st;
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev;
  int group(const char* name) {
    for (size_t i = 0; i < c->tnames.size(); ++i)
      if (c->tnames[i] == name) return (int)i;
    c->tnames.push_back(name);
    c->tms.push_back(0);
    c->tcount.push_back(0);
    return (int)c->tnames.size() - 1;
  }
  void begin(const char* name) {
    nvtxRangePushA(name);   // host-side phase marker (matched in end())
    if (!c->timing) return;
    cudaEvent_t a, b;
    HB_CUDA(cudaEventCreate(&a));
    HB_CUDA(cudaEventCreate(&b));
    HB_CUDA(cudaEventRecord(a, st));
    ev.push_back({group(name), {a, b}});
  }
  void end() {
    nvtxRangePop();
    if (!c->timing) return;
    HB_CUDA(cudaEventRecord(ev.back().second.second, st));
  }
  void finish() {
    if (!c->timing) return;
    HB_CUDA(cudaStreamSynchronize(st));
    for (auto& e : ev) {
      float ms = 0;
      HB_CUDA(cudaEventElapsedTime(&ms, e.second.first, e.second.second));
      c->tms[e.first] += ms;
      c->tcount[e.first] += 1;
      cudaEventDestroy(e.second.first);
      cudaEventDestroy(e.second.second);
    }
    ev.clear();
  }
};

// Scratch of the precision in use (allocated on first use, kept); the device
// is synchronised only after an allocation, so applies stay asynchronous.
void ensure_scratch(hb_ctx* c, int nrhs, bool fp64) {
  bool fresh = false;
  if (fp64 && c->cap_rhs < nrhs) {
    fresh = true;
    dev_free(c->d_x);
    dev_free(c->d_y);
    dev_free(c->d_xh);
    c->d_x = c->d_y = c->d_xh = nullptr;
    c->cap_rhs = 0;
    c->d_x = dev_alloc<double2>((size_t)(c->Nv + 1) * nrhs);
    c->d_y = dev_alloc<double2>((size_t)(c->Nv + 1) * nrhs);
    c->d_xh = dev_alloc<double2>((size_t)(std::max<long long>(c->xh_rows, 1) + 1) * nrhs);
    c->cap_rhs = nrhs;
  }
  if (!c->d_perm) {
    fresh = true;
    c->d_perm = upload(c->perm);
  }
  if (!fp64 && (!c->d_mx || !c->d_mxh || !c->d_flags || !c->d_mx_tc)) {
    // native vectors for two m-tiles: 2 KB per row tile, x again in the
    // tensor-core operand layout, and the dataflow launch's flags (all or
    // none: an allocation that failed half way is redone whole on the next
    // call)
    fresh = true;
    for (void* p : {(void*)c->d_mx, (void*)c->d_mxh, (void*)c->d_flags, (void*)c->d_mx_tc}) dev_free(p);
    c->d_mx = c->d_mxh = c->d_mx_tc = nullptr;
    c->d_flags = c->d_epoch = nullptr;
    c->d_mx = dev_alloc<uint4>((size_t)std::max<long long>(c->nv_tiles, 1) * 128);
    c->d_mx_tc = dev_alloc<uint4>((size_t)std::max<long long>(c->nv_tiles, 1) * 128);
    c->d_mxh = dev_alloc<uint4>((size_t)std::max<long long>(c->xh_tiles, 1) * 128);
    // + the dataflow launch's epoch and finish count, the grid barriers' arrival and finish counts
    const size_t nflags = (size_t)(c->nv_tiles + c->xh_tiles) + 4;
    c->d_flags = dev_alloc<unsigned>(nflags);
    HB_CUDA(cudaMemset(c->d_flags, 0, sizeof(unsigned) * nflags));
    c->d_epoch = c->d_flags + (c->nv_tiles + c->xh_tiles);
  }
  if (!c->h_err) {
    fresh = true;
    HB_CUDA(cudaHostAlloc(reinterpret_cast<void**>(&c->h_err), sizeof(int), cudaHostAllocMapped));
    *c->h_err = 0;
    HB_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->d_err), c->h_err, 0));
  }
  if (fresh) HB_CUDA(cudaDeviceSynchronize());
}

}  // namespace

// ------------------------------------------------- dense product ----
// Y = alpha A X (or +=) for a stored column-major A (m x k): step tasks over
// ranges of the inputs (enough CTAs for the chip when m is small; the ranges'
// sums are added in order), X and Y converted between columns and the tasks'
// rows of R values.
__global__ void pack_rows_kernel(const double2* __restrict__ X, long long ldx, long long k, int R, double scale,
                                 double2* __restrict__ x) {
  const int r = threadIdx.x;
  if (r >= R) return;
  for (long long p = (long long)blockIdx.x * blockDim.y + threadIdx.y; p < k; p += (long long)gridDim.x * blockDim.y) {
    const double2 v = X[(size_t)r * ldx + p];
    x[p * R + r] = make_double2(scale * v.x, scale * v.y);
  }
}

__global__ void sum_rows_kernel(const double2* __restrict__ y, long long m, int parts, int R, double2* __restrict__ Y,
                                long long ldy, int accumulate) {
  const int r = threadIdx.x;
  if (r >= R) return;
  for (long long i = (long long)blockIdx.x * blockDim.y + threadIdx.y; i < m; i += (long long)gridDim.x * blockDim.y) {
    double2 a = accumulate ? Y[(size_t)r * ldy + i] : make_double2(0.0, 0.0);
    for (int c = 0; c < parts; ++c) {
      const double2 v = y[((size_t)c * m + i) * R + r];
      a.x += v.x;
      a.y += v.y;
    }
    Y[(size_t)r * ldy + i] = a;
  }
}

DenseOp dense_op(const double2* A, long long m, long long k, cudaStream_t st) {
  if (m > INT32_MAX || k > INT32_MAX) throw Error{HB_ERR_UNSUPPORTED, "stored operator too large"};
  DenseOp D;
  D.A = A;
  D.m = m;
  D.k = k;
  // inputs per task: at least 128 (the exponent scan and the epilogue are per
  // task), and 304 CTAs of 64 outputs in all where that leaves as many
  const long long rb = (m + 63) / 64;
  const long long parts = std::max<long long>(1, std::min<long long>((304 + rb - 1) / rb, (k + 127) / 128));
  const long long kc = ((k + parts - 1) / parts + 7) / 8 * 8;
  std::vector<Task> tasks;
  for (long long k0 = 0; k0 < k; k0 += kc) {
    Task t{};
    t.y_off = (long long)tasks.size() * m;
    t.f_off[0] = k0 * m;
    t.x_off[0] = k0;
    t.r_out = (int)m;
    t.r_in[0] = (int)std::min(kc, k - k0);
    t.nterm = 1;
    t.x_buf = 0;
    t.y_buf = 1;
    tasks.push_back(t);
  }
  D.ntask = (int)tasks.size();
  D.plan = task_plan(tasks, {0, D.ntask}, 8);   // 4 warps: apply with 300 segments at 96^2 338 us, 8: 334
  try {
    D.d_tasks = upload(tasks, st);
    task_exponents(D.plan, D.d_tasks, A, st);
    HB_CUDA(cudaStreamSynchronize(st));
  } catch (...) {
    dense_op_free(D);
    throw;
  }
  return D;
}

void dense_op_free(DenseOp& D) {
  task_plan_free(D.plan);
  dev_free(D.d_tasks);
  D = DenseOp{};
}

namespace {

// launch shape of the vector kernels: lanes over the right-hand sides
struct VecGrid {
  dim3 grid, block;
  VecGrid(long long rows, int R) {
    int rp = 1;
    while (rp < R) rp *= 2;
    block = dim3((unsigned)rp, (unsigned)(256 / rp));
    grid = dim3((unsigned)std::max<long long>(1, std::min<long long>((rows + block.y - 1) / block.y, 152LL * 16)));
  }
};

}  // namespace

void dense_product(const DenseOp& D, const double2* X, long long ldx, double2* Y, long long ldy, int R, double alpha,
                   int accumulate, double2* x, double2* y, cudaStream_t st) {
  const VecGrid in(D.k, R), out(D.m, R);
  pack_rows_kernel<<<in.grid, in.block, 0, st>>>(X, ldx, D.k, R, alpha, x);
  HB_CHECK_LAUNCH();
  run_tasks_fp64(D.plan, 0, D.d_tasks, D.A, x, y, nullptr, R, st);
  sum_rows_kernel<<<out.grid, out.block, 0, st>>>(y, D.m, D.ntask, R, Y, ldy, accumulate);
  HB_CHECK_LAUNCH();
}

namespace {

void run_steps(hb_ctx* c, const double2* F, int nrhs, int dir, cudaStream_t st, TimerScope& ts) {
  const std::vector<int>& sb = c->step_begin[dir];
  for (size_t s = 0; s + 1 < sb.size(); ++s) {
    const int n = sb[s + 1] - sb[s];
    if (n == 0) continue;
    ts.begin(dir ? "bf_step_adjoint" : "bf_step");
    run_tasks_fp64(c->task_plans[dir], (int)s, c->d_tasks[dir], F, (double2*)c->d_x, (double2*)c->d_y, (double2*)c->d_xh,
                   nrhs, st);
    ts.end();
  }
}

}  // namespace

void apply_bf(hb_ctx* c, const double2* s, double2* u, int nrhs, int adjoint, int precision, cudaStream_t st) {
  NvtxRange nr(adjoint ? "hb_apply_adjoint" : "hb_apply");
  if (c->h_err && *reinterpret_cast<volatile int*>(c->h_err)) {
    *reinterpret_cast<volatile int*>(c->h_err) = 0;
    throw Error{HB_ERR_TIMEOUT, "a bounded device wait of an earlier apply gave up"};
  }
  // right-hand sides per pass: the scratch vectors (skeleton rows x pass x 16
  // bytes for FP64) stay bounded for any nrhs
  const int chunk = std::min(nrhs, precision == HB_FP64 ? 16 : 32);
  if (precision == HB_FP64) ensure_task_plans(c);
  ensure_scratch(c, chunk, precision == HB_FP64);
  TimerScope ts{c, st, {}};
  const double scale = c->h * c->h;
  for (int r0 = 0; r0 < nrhs; r0 += chunk) {
    const int R = std::min(chunk, nrhs - r0);
    const double2* sc = s + (size_t)r0 * c->Nv;
    double2* uc = u + (size_t)r0 * c->Nv;
    const VecGrid vg(c->Nv, R);
    if (precision == HB_FP64) {
      ts.begin("gather");
      gather_kernel<<<vg.grid, vg.block, 0, st>>>(sc, c->d_perm, (double2*)c->d_x, c->Nv, R, scale, 0, c->Nv);
      HB_CHECK_LAUNCH();
      ts.end();
      run_steps(c, c->d_f64, R, adjoint, st, ts);
      ts.begin("scatter");
      scatter_kernel<<<vg.grid, vg.block, 0, st>>>((double2*)c->d_y, c->d_perm, uc, c->Nv, R, 0, c->Nv);
      HB_CHECK_LAUNCH();
      ts.end();
    } else {
      // the gather and every depth (the last one writes u): one persistent
      // launch, or a gather and one launch per depth; the timer brackets the
      // step launches (with the gather inside them in the first form)
      flow_launch(c->flow_plan[adjoint], c->tc_plan[adjoint], c->d_tc[adjoint], c->d_nat[adjoint], sc, scale,
                  c->d_mx, c->d_mx_tc, c->d_mxh, uc, c->d_pperm, c->Nv, c->nv_tiles, R, c->d_flags, c->d_epoch,
                  c->d_err,
                  c->opt.barrier_cycles > 0 ? c->opt.barrier_cycles : (1LL << 31), c->wait_selftest,
                  c->opt.autotune, st, [&](int, bool begin) {
                    if (begin) ts.begin(adjoint ? "bf_tc_adjoint" : "bf_tc");
                    else ts.end();
                  });
    }
  }
  ts.finish();
}

// ------------------------------------------------------------- shards ----
// Rank `rank` of `nranks` (a power of two, at most 2^L_v) owns node `rank`
// of level log2(nranks) of the cluster tree: the tree positions [lo, hi).
void shard_rows(const hb_ctx* c, int nranks, int rank, long long* lo, long long* hi) {
  if (nranks < 1 || (nranks & (nranks - 1)) || rank < 0 || rank >= nranks)
    throw arg_error("nranks must be a power of two and 0 <= rank < nranks (got %d, %d)", nranks, rank);
  int k = 0;
  while ((1 << k) < nranks) ++k;
  if (k > c->Lv) throw arg_error("nranks=%d exceeds the %lld leaves of the cluster tree", nranks, 1LL << c->Lv);
  *lo = c->bounds[k][rank];
  *hi = c->bounds[k][rank + 1];
}

namespace {
struct ShardSteps {
  std::vector<int> begin;
  TaskPlan plan;
  Task* d_tasks = nullptr;
};
}  // namespace

// The FP64 step lists of one shard: the tasks whose rows meet [lo, hi).
static ShardSteps& shard_steps(hb_ctx* c, int dir, long long lo, long long hi) {
  static_assert(sizeof(void*) == 8, "");
  auto key = std::make_tuple(dir, lo, hi);
  auto it = c->shard_cache.find(key);
  if (it != c->shard_cache.end()) return *static_cast<ShardSteps*>(it->second);
  ShardSteps* S = new ShardSteps();
  std::vector<Task> keep;
  const std::vector<int>& sb = c->step_begin[dir];
  for (size_t q = 0; q + 1 < sb.size(); ++q) {
    S->begin.push_back((int)keep.size());
    for (int t = sb[q]; t < sb[q + 1]; ++t) {
      const auto& rr = c->task_rows[dir][(size_t)t];
      if (rr.first < hi && rr.second > lo) keep.push_back(c->tasks_h[dir][(size_t)t]);
    }
  }
  S->begin.push_back((int)keep.size());
  try {
    S->plan = task_plan(keep, S->begin, 4);
    S->d_tasks = upload(keep);
    task_exponents(S->plan, S->d_tasks, c->d_f64, 0);
    HB_CUDA(cudaStreamSynchronize(0));   // the caller's stream may not wait for this one
  } catch (...) {
    task_plan_free(S->plan);
    dev_free(S->d_tasks);
    delete S;
    throw;
  }
  c->shard_cache[key] = S;
  return *S;
}

void shard_cache_free(hb_ctx* c) {
  for (auto& kv : c->shard_cache) {
    ShardSteps* S = static_cast<ShardSteps*>(kv.second);
    task_plan_free(S->plan);
    dev_free(S->d_tasks);
    delete S;
  }
  c->shard_cache.clear();
}

// The padded row (mixed path) where the leaf starting at tree position pos
// starts (pos = N_v: the end).
static long long padded_row_of(const hb_ctx* c, long long pos) {
  const std::vector<long long>& b = c->bounds[(size_t)c->Lv];
  const auto it = std::lower_bound(b.begin(), b.end(), pos);
  if (it == b.end() || *it != pos) throw Error{HB_ERR_STATE, "shard boundary is not a leaf boundary"};
  return 8 * c->leaf_tile[(size_t)(it - b.begin())];
}

// One rank's share of the apply.  Forward (u = A s): s is the whole input
// (natural order, every rank's cells); the rank computes every task whose
// rows meet its own and writes u on its cells only.  Adjoint (s = A^H u):
// u holds the rank's cells (the rest is ignored, read as zero); the rank
// computes the tasks whose rows meet its own with the skeleton vectors of
// the others zero, and writes its share of s on every cell; the shares of
// all ranks add up to the adjoint.
void apply_bf_shard(hb_ctx* c, const double2* s, double2* u, int nrhs, int adjoint, int precision, int nranks,
                    int rank, cudaStream_t st) {
  NvtxRange nr(adjoint ? "hb_apply_shard_adjoint" : "hb_apply_shard");
  if (c->h_err && *reinterpret_cast<volatile int*>(c->h_err)) {
    *reinterpret_cast<volatile int*>(c->h_err) = 0;
    throw Error{HB_ERR_TIMEOUT, "a bounded device wait of an earlier apply gave up"};
  }
  long long lo = 0, hi = 0;
  shard_rows(c, nranks, rank, &lo, &hi);
  const int chunk = std::min(nrhs, precision == HB_FP64 ? 16 : 32);
  ensure_scratch(c, chunk, precision == HB_FP64);
  const double scale = c->h * c->h;
  const long long glo = adjoint ? lo : 0, ghi = adjoint ? hi : c->Nv;    // input rows
  const long long slo = adjoint ? 0 : lo, shi = adjoint ? c->Nv : hi;   // output rows
  for (int r0 = 0; r0 < nrhs; r0 += chunk) {
    const int R = std::min(chunk, nrhs - r0);
    const double2* sc = s + (size_t)r0 * c->Nv;
    double2* uc = u + (size_t)r0 * c->Nv;
    const VecGrid vg(c->Nv, R);
    if (precision == HB_FP64) {
      gather_kernel<<<vg.grid, vg.block, 0, st>>>(sc, c->d_perm, (double2*)c->d_x, c->Nv, R, scale, glo, ghi);
      HB_CHECK_LAUNCH();
      if (adjoint) {
        HB_CUDA(cudaMemsetAsync(c->d_y, 0, sizeof(double2) * (size_t)c->Nv * R, st));
        HB_CUDA(cudaMemsetAsync(c->d_xh, 0, sizeof(double2) * (size_t)std::max<long long>(c->xh_rows, 1) * R, st));
      }
      ShardSteps& S = shard_steps(c, adjoint, lo, hi);
      for (size_t q = 0; q + 1 < S.begin.size(); ++q) {
        const int n = S.begin[q + 1] - S.begin[q];
        if (n == 0) continue;
        run_tasks_fp64(S.plan, (int)q, S.d_tasks, c->d_f64, (double2*)c->d_x, (double2*)c->d_y, (double2*)c->d_xh, R, st);
      }
      const VecGrid vs(shi - slo, R);
      scatter_kernel<<<vs.grid, vs.block, 0, st>>>((double2*)c->d_y, c->d_perm, uc, c->Nv, R, slo, shi);
      HB_CHECK_LAUNCH();
    } else {
      flow_launch_shard(c->flow_plan[adjoint], c->d_nat[adjoint], sc, scale, c->d_mx, c->d_mxh, c->xh_tiles, uc,
                        c->d_pperm, c->Nv, c->nv_tiles, R, lo, hi, adjoint ? padded_row_of(c, lo) : 0,
                        adjoint ? padded_row_of(c, hi) : (long long)8 * c->nv_tiles, adjoint != 0, c->d_err,
                        c->opt.barrier_cycles > 0 ? c->opt.barrier_cycles : (1LL << 31), st);
    }
  }
}

}  // namespace hb
