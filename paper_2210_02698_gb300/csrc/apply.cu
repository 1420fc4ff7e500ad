// apply.cu - butterfly / HODBF apply and its adjoint on the device
// (Sec. 4.2.1, Eq. butterfly_mat, Eq. butterfly_factors; Sec. 4.2 HODBF).
//
//   x  = h^2 s, gathered into cluster-tree order            (Eq. m_v2v)
//   steps of small dense products over all butterflies      (build.cu plans)
//   u  = y scattered back to natural order
//
// FP64 path: complex128 factors and vectors, the step tasks' products on the
// FP16 tensor cores by integer digits, as accurate as FP64 FMAs.  Mixed path (HB_MIXED_BF16X3): split-BF16 factors and
// vectors in the MMA-fragment layout of bf_mma.cu, up to 32 right-hand
// sides per pass.
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
// Y = op(F) X of one task on the FP16 tensor cores by integer digits
// (split_fixed.cuh), in the orientation of the mixed apply: the MMA's M is
// right-hand sides, N outputs, K = 2 x 8 inputs with real and imaginary
// parts interleaved; D_r takes A rows (Re X, -Im X), D_i (Im X, Re X).  Up to
// eight right-hand sides (HALF) both go into one MMA, rows 0-7 and 8-15.
//
// A CTA of 8 warps takes up to 64 outputs (8 n-tiles; row_blocks CTAs per task) of
// one task.  It scales X per right-hand side and F per task (tk.fe, found
// when the plan is made), splits X into digit fragments in shared memory,
// KC k-steps at a time, and every warp streams its n-tile's F straight from
// global memory into registers, one k-step ahead, splitting it there (each
// F value is used by one warp only).  With fewer than 8 n-tiles the k-steps
// are dealt over 2, 4 or 8 warps and the integer sums added: the result does
// not depend on the split.  The split is a function of the task alone, so a
// shard's sums equal the whole apply's.
//
// Bound by instruction issue: 42 (21) MMAs and about 150 integer instructions
// a warp per 8 outputs x 8 inputs, as much again to split the task's X where
// its rank is near 16, and the epilogue, against 1024 x 4 FP64 FMAs for 16
// right-hand sides (2048 cycles of an SM's FP64 unit).  Measured (192^2, 16
// right-hand sides): 3.67 -> 1.92 ms against one FP64 FMA loop per output;
// 120 x 88 adjoint with 5: 601 -> 251 us.
constexpr int TASK_THREADS = 256;
constexpr int TASK_WARPS = TASK_THREADS / 32;
constexpr int TASK_KC = 16;              // k-steps of X held at a time
constexpr uint32_t SPLIT_IM_SIGN = 0x80000000u;

// Rows [row0, row1) of a task with plain FP64 FMAs: what a task does whose
// inputs are not all finite (thread -> (row, right-hand side), rows fastest).
__device__ __noinline__ void task_plain(const Task* __restrict__ task, const double2* __restrict__ F, double2* x, double2* y,
                                        double2* xh, int R, int row0, int row1) {
  const Task& tk = *task;
  double2* bufs[3] = {x, y, xh};
  double2* out = bufs[tk.y_buf] + (size_t)tk.y_off * R;
  const int rows = row1 - row0, total = rows * R;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int row = row0 + idx % rows, rr = idx / rows;
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

template <bool HALF>
__global__ void __launch_bounds__(TASK_THREADS, HALF ? 3 : 2)
    task_kernel(const Task* __restrict__ tasks, const double2* __restrict__ F, double2* x, double2* y, double2* xh,
                int R, int row_blocks) {
  constexpr int NR = HALF ? 8 : 16;        // right-hand sides of the MMA rows
  constexpr int NE = HALF ? 4 : 8;         // accumulator elements per lane and digit diagonal
  constexpr int XW = HALF ? 2 : 4;         // X fragment words per lane
  extern __shared__ __align__(16) uint32_t xs[];   // [k-step][digit][lane][XW]
  __shared__ int s_ex[16];
  __shared__ int s_bad;
  const Task* task = tasks + blockIdx.x / row_blocks;
  const Task tk = *task;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int tile0 = 8 * (blockIdx.x % row_blocks);
  const int ntile = min(8, (tk.r_out + 7) / 8 - tile0);
  if (ntile <= 0) return;
  const double2* xin = tk.x_buf == 0 ? x : tk.x_buf == 1 ? y : xh;
  const int rin0 = tk.r_in[0], rin1 = tk.nterm > 1 ? tk.r_in[1] : 0;
  const int ks0 = (rin0 + 7) / 8, ks = ks0 + (rin1 + 7) / 8;

  // the exponent of every right-hand side over the task's inputs
  if (tid < 16) s_ex[tid] = 1;
  if (tid == 0) s_bad = (tk.fe == SPLIT_NONFINITE) ? 1 : 0;
  __syncthreads();
  const int xr = tid & (NR - 1), xk = tid / NR;
  constexpr int XK = TASK_THREADS / NR;
  if (xr < R) {
    int e = 1;
    for (int k = xk; k < rin0; k += XK) e = max(e, block_exponent(xin[(tk.x_off[0] + k) * R + xr]));
    for (int k = xk; k < rin1; k += XK) e = max(e, block_exponent(xin[(tk.x_off[1] + k) * R + xr]));
    atomicMax(&s_ex[xr], e);
    if (e == SPLIT_NONFINITE) s_bad = 1;
  }
  __syncthreads();
  if (s_bad) {
    task_plain(task, F, x, y, xh, R, 8 * tile0, min(tk.r_out, 8 * (tile0 + 8)));
    return;
  }

  // warp -> n-tile and share of the k-steps
  const int kw = ntile > 4 ? 1 : ntile > 2 ? 2 : ntile > 1 ? 4 : 8;
  const int wt = warp % (TASK_WARPS / kw), kp = warp / (TASK_WARPS / kw);
  const bool work = wt < ntile;
  const int row = 8 * (tile0 + wt) + g;
  const bool rok = work && row < tk.r_out;

  // F values (row, k = 2t) and (row, 2t + 1) of k-step q
  auto load_f = [&](int q, double2& f0, double2& f1) {
    f0 = f1 = make_double2(0.0, 0.0);
    if (!rok || q >= ks) return;
    const int term = q >= ks0, rin = term ? rin1 : rin0;
    const int k = 8 * (term ? q - ks0 : q) + 2 * t;
    const double2* f = F + (term ? tk.f_off[1] : tk.f_off[0]);
    if (!tk.conj_t) {
      if (k < rin) f0 = __ldcs(f + (size_t)k * tk.r_out + row);
      if (k + 1 < rin) f1 = __ldcs(f + (size_t)(k + 1) * tk.r_out + row);
    } else {
      const double2* fr = f + (size_t)row * rin + k;
      if (k < rin) f0 = __ldcs(fr);
      if (k + 1 < rin) f1 = __ldcs(fr + 1);
      f0.y = -f0.y;
      f1.y = -f1.y;
    }
  };

  float acc[SPLIT_ACC][NE];
  long long hi[NE], lo[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    hi[e] = lo[e] = 0;
#pragma unroll
    for (int d = 0; d < SPLIT_ACC; ++d) acc[d][e] = 0.f;
  }
  const int myex = s_ex[xr];
  double2 f0, f1;
  load_f(kp, f0, f1);
  for (int c0 = 0; c0 < ks; c0 += TASK_KC) {
    const int c1 = min(ks, c0 + TASK_KC);
    if (c0) __syncthreads();
    // X of k-steps [c0, c1) into digit fragments: word j of lane (g, t) is
    // (right-hand side g + 8 (j & 1), input 2t + (j >> 1)); HALF: (g, 2t + j)
    for (int k = 8 * c0 + xk; k < 8 * c1; k += XK) {
      const int q = k >> 3, kk = k & 7;
      const int term = q >= ks0, kin = term ? k - 8 * ks0 : k;
      double2 v = make_double2(0.0, 0.0);
      if (xr < R && kin < (term ? rin1 : rin0)) v = xin[((term ? tk.x_off[1] : tk.x_off[0]) + kin) * R + xr];
      uint32_t w[SPLIT_DIGITS];
      split_pair(v.x, v.y, myex, w);
      const int j = HALF ? (kk & 1) : 2 * (kk & 1) + (xr >> 3);
      uint32_t* dst = xs + (((q - c0) * SPLIT_DIGITS) * 32 + (xr & 7) * 4 + (kk >> 1)) * XW + j;
#pragma unroll
      for (int s = 0; s < SPLIT_DIGITS; ++s) dst[s * 32 * XW] = w[s];
    }
    __syncthreads();
    if (work) {
      int since = 0;
      for (int q = c0 + (kp - c0 % kw + kw) % kw; q < c1; q += kw) {
        const double2 a0 = f0, a1 = f1;
        load_f(q + kw, f0, f1);
        uint32_t b0[SPLIT_DIGITS], b1[SPLIT_DIGITS];
        split_pair(a0.x, a0.y, tk.fe, b0);
        split_pair(a1.x, a1.y, tk.fe, b1);
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
  // add the shares of the k-steps
  if (kw > 1) {
    longlong2* red = reinterpret_cast<longlong2*>(xs);   // [kp - 1][n-tile][element][lane]
    __syncthreads();
    if (work && kp > 0)
#pragma unroll
      for (int e = 0; e < NE; ++e) red[(((kp - 1) * ntile + wt) * NE + e) * 32 + lane] = make_longlong2(hi[e], lo[e]);
    __syncthreads();
    if (!work || kp > 0) return;
    for (int p = 0; p < kw - 1; ++p)
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const longlong2 v = red[((p * ntile + wt) * NE + e) * 32 + lane];
        hi[e] += v.x;
        lo[e] += v.y;
      }
  }
  if (!work) return;
  double2* out = (tk.y_buf == 0 ? x : tk.y_buf == 1 ? y : xh) + (size_t)tk.y_off * R;
  // element e of D: right-hand side g + 8 (e >> 1), output 2t + (e & 1); HALF:
  // elements 0, 1 are D_r and 2, 3 D_i of right-hand side g
#pragma unroll
  for (int e = 0; e < NE / 2; ++e) {
    const int rr = HALF ? g : g + 8 * (e >> 1);
    const int ro = 8 * (tile0 + wt) + 2 * t + (e & 1);
    if (rr >= R || ro >= tk.r_out) continue;
    const int ex = tk.fe + s_ex[rr] - 2 * SPLIT_EXP_BIAS;
    const int ei = HALF ? e + 2 : e + 4;
    double2 v = make_double2(fixed_to_double(hi[e], lo[e], ex), fixed_to_double(hi[ei], lo[ei], ex));
    double2* o = out + (size_t)ro * R + rr;
    if (tk.accumulate) {
      const double2 prev = *o;
      v.x += prev.x;
      v.y += prev.y;
    }
    *o = v;
  }
}

// tasks[i].fe = the largest exponent of task i's factor blocks (1 before),
// blockIdx.y of gridDim.y shares of them
__global__ void __launch_bounds__(256) task_exponent_kernel(Task* __restrict__ tasks, const double2* __restrict__ F) {
  Task& tk = tasks[blockIdx.x];
  int e = 1;
  for (int t = 0; t < tk.nterm; ++t) {
    const long long cnt = (long long)tk.r_out * tk.r_in[t];
    const double2* f = F + tk.f_off[t];
#pragma unroll 4
    for (long long k = blockIdx.y * 256 + threadIdx.x; k < cnt; k += 256 * gridDim.y) e = max(e, block_exponent(f[k]));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&tk.fe, e);
}

void task_exponents(Task* d_tasks, int n, const double2* F, cudaStream_t st) {
  if (n <= 0) return;
  const unsigned share = (unsigned)std::max(1, std::min(128, 608 / n));
  task_exponent_kernel<<<dim3((unsigned)n, share), 256, 0, st>>>(d_tasks, F);
  HB_CHECK_LAUNCH();
}

StepShape step_shape(const Task* tasks, int n) {
  StepShape s{0, 0};
  for (int i = 0; i < n; ++i) {
    const Task& t = tasks[i];
    s.max_out = std::max(s.max_out, t.r_out);
    s.max_ks = std::max(s.max_ks, (t.r_in[0] + 7) / 8 + (t.nterm > 1 ? (t.r_in[1] + 7) / 8 : 0));
  }
  return s;
}

// One launch of FP64 step tasks, R <= 16 right-hand sides.
void run_tasks_fp64(const Task* d_tasks, int n, const StepShape& sh, const double2* F, double2* x, double2* y,
                    double2* xh, int R, cudaStream_t st) {
  if (n <= 0) return;
  const int rb = std::max(1, (sh.max_out + 63) / 64);
  const unsigned grid = (unsigned)n * (unsigned)rb;
  const size_t frag = (size_t)std::min(TASK_KC, std::max(1, sh.max_ks)) * SPLIT_DIGITS * 32 * 4;
  const size_t red = (size_t)7 * 32 * sizeof(longlong2);   // the k-step shares of one CTA: at most 7 n-tile shares
  if (R <= 8) {
    const size_t smem = std::max(frag * 2, red * 4);
    task_kernel<true><<<grid, TASK_THREADS, smem, st>>>(d_tasks, F, x, y, xh, R, rb);
  } else {
    const size_t smem = std::max(frag * 4, red * 8);
    HB_CUDA(cudaFuncSetAttribute(task_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 56 << 10));
    task_kernel<false><<<grid, TASK_THREADS, smem, st>>>(d_tasks, F, x, y, xh, R, rb);
  }
  HB_CHECK_LAUNCH();
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
  D.shape = step_shape(tasks.data(), D.ntask);
  D.d_tasks = upload(tasks, st);
  task_exponents(D.d_tasks, D.ntask, A, st);
  HB_CUDA(cudaStreamSynchronize(st));
  return D;
}

void dense_op_free(DenseOp& D) {
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
  run_tasks_fp64(D.d_tasks, D.ntask, D.shape, D.A, x, y, nullptr, R, st);
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
    run_tasks_fp64(c->d_tasks[dir] + sb[s], n, c->step_shapes[dir][s], F, (double2*)c->d_x, (double2*)c->d_y,
                   (double2*)c->d_xh, nrhs, st);
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
  std::vector<StepShape> shapes;
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
  for (size_t q = 0; q + 1 < S->begin.size(); ++q)
    S->shapes.push_back(step_shape(keep.data() + S->begin[q], S->begin[q + 1] - S->begin[q]));
  try {
    S->d_tasks = upload(keep);
  } catch (...) {
    delete S;
    throw;
  }
  c->shard_cache[key] = S;
  return *S;
}

void shard_cache_free(hb_ctx* c) {
  for (auto& kv : c->shard_cache) {
    ShardSteps* S = static_cast<ShardSteps*>(kv.second);
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
        run_tasks_fp64(S.d_tasks + S.begin[q], n, S.shapes[q], c->d_f64, (double2*)c->d_x, (double2*)c->d_y,
                       (double2*)c->d_xh, R, st);
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
