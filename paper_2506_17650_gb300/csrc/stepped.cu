// Stepped periods: a resident period's attempts in plain launches.
//
// A stepped period does what a resident one does, row for row and sum for sum in
// the same order, so that the two give the same bits, but its blocks wait for
// nothing: the plan's CTAs are the blocks of two launches per attempt (A^T y and
// x+; A x+, y+ and, in the last block to finish, the step control), which read
// the matrix and the vectors from global memory (L2).  It is what a period runs as when
// the SMs for a resident one are not to be had.  One solve alone takes 15.6 us per
// attempt so on the 60k-nonzero LP (resident 8.5), 30 on the transportation LP (17),
// 57 on the power-law LP of 1M nonzeros (33): chains of loads again, and blocks
// enough for one wave only.  What counts is several at a time, see SmTokens.
#include "resident.hpp"

#include <algorithm>
#include <type_traits>

#include "ops.cuh"
#include "resident_sums.cuh"

namespace lpop {

namespace {

// A block sums its rows with as many warps as it has items (resident_build), so
// that several problems share an SM.  Its rows' terms go into the resident
// kernel's kResThreads slots (row t into slot t mod kResThreads) whatever
// its threads.  Rows cut into segments: the block that has the row forms all of
// them, or, with a row of more than kOwnSegs, all blocks do in a launch before.
constexpr int kOwnSegs = 32;
bool segments_apart(int longest) { return longest > kOwnSegs * kResSeg; }
constexpr int kStepThreads = kResThreads;

// Slots of a block's sums that are ever read: res_sum goes through them 128 at a time.
LPOP_HD int sum_slots(int rows) { return rows >= kResThreads ? kResThreads : (rows + 127) & ~127; }

// Sum of `size` entries from `beg` on, in the order of a resident segment, into a word.
template <class V>
__device__ __forceinline__ void step_segment(const CsrT<V>& M, int beg, int size, const ResGather<V, kBarriersKind>& g,
                                             ulonglong2* word) {
  const int lane = threadIdx.x & 31;
  bool ok = true;
  const V s = res_dot(M.v + beg + lane, M.ci + beg + lane, (size - lane + 31) >> 5, (size + 31) >> 5, 32, g, &ok);
  const double w = lane_sum((double)s);
  if (lane == 0) word->x = (unsigned long long)__double_as_longlong(w);
}

template <class V, bool kPrimal>
__global__ void __launch_bounds__(kStepThreads, 2) stepped_segments_kernel(Dev d, ResPlan pl) {
  pdl_wait();
  const ResCta C = pl.cta[blockIdx.x];
  const int first = kPrimal ? C.p0 : C.d0, end = kPrimal ? C.p1 : C.d1;
  const Vecs<V>& v = vecs<V>(d);
  const CsrT<V> M = kPrimal ? csr_at<V>(d) : csr_a<V>(d);
  const int cur = d.st->cur;
  const ResGather<V, kBarriersKind> g{kPrimal ? v.y[cur] : v.x[cur ^ 1], nullptr, 0u, kPrimal ? d.m : d.n, d.bad_gathers, 0};
#pragma unroll 1
  for (int i = first + (int)(threadIdx.x >> 5); i < end; i += (int)(blockDim.x >> 5)) {
    const ResItem I = pl.items[i];
    if (I.kind != kSegKind) break;  // (segments come first)
    step_segment(M, M.rp[I.row0] + I.len, I.nrows, g, pl.seg + I.vec);
  }
  pdl_trigger();
}

template <class V, bool kPrimal>
__global__ void __launch_bounds__(kStepThreads, 2) stepped_kernel(Dev d, Params prm, ResPlan pl, bool apart) {
  constexpr int kAcc = kPrimal ? 3 : 4;
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ double s_tot[8];
  __shared__ double s_fac[2];
  __shared__ DevState s_st;
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x, warps = threads >> 5;
  pdl_wait();
  const ResCta C = pl.cta[blockIdx.x];
  const ResItem* const it = pl.items + (kPrimal ? C.p0 : C.d0);
  const int items = kPrimal ? C.p1 - C.p0 : C.d1 - C.d0, rows = kPrimal ? C.rp : C.rd;
  const int most_rows = kPrimal ? pl.rp : pl.rd, slots = sum_slots(most_rows);
  double* const s_red = reinterpret_cast<double*>(s_raw);  // kAcc fields of `slots`
  V* const s_sum = reinterpret_cast<V*>(s_red + kAcc * slots);  // by local row
  int* const s_row = reinterpret_cast<int*>(s_sum + most_rows);
  const Vecs<V>& v = vecs<V>(d);
  const CsrT<V> M = kPrimal ? csr_at<V>(d) : csr_a<V>(d);
  std::conditional_t<kPrimal, PrimalOp<V, true>, DualOp<V, true>> op;
  op.sc = read_scalars<V>(d.st, kPrimal);
  const int cur = op.sc.cur;
  if constexpr (kPrimal) op.bind(v, prm, cur);
  else op.bind(v, prm, d.sense, cur);
  const bool collect = op.sc.collect != 0;
  const ResGather<V, kBarriersKind> g{kPrimal ? v.y[cur] : v.x[cur ^ 1], nullptr, 0u, kPrimal ? d.m : d.n, d.bad_gathers, 0};
  bool ok = true;
  // ---- row sums -----------------------------------------------------------------
  int own = items;  // the rows cut into segments come last
  for (int c = 32; c == 32; own -= c) {
    const int i = own - 1 - lane;
    const unsigned int rest = __ballot_sync(0xffffffffu, i < 0 || it[i].kind != kOwnKind);
    c = rest ? __ffs((int)rest) - 1 : 32;
  }
#pragma unroll 1
  for (int i = warp; i < own; i += warps) {
    const ResItem I = it[i];
    if (I.kind == kSegKind) continue;
    if (lane < I.nrows) s_row[I.vec + lane] = I.row0 + lane;
    const int width = I.kind == 0 ? 1 : I.kind, lg = 31 - __clz(width);
    const int l = lane & (width - 1), r = lane >> lg;
    const bool has = r < I.nrows;
    const int e0 = has ? M.rp[I.row0 + r] : 0, len = has ? M.rp[I.row0 + r + 1] - e0 : 0;
    const int count = max(len - l + width - 1, 0) >> lg;
    const int most = __reduce_max_sync(0xffffffffu, count);
    V s = res_dot(M.v + e0 + l, M.ci + e0 + l, count, most, width, g, &ok);
#pragma unroll 1
    for (int o = width / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, width);
    if (l == 0 && has) s_sum[I.vec + r] = s;
  }
  if (own < items) {
    int at = 0;  // segments of the rows before
#pragma unroll 1
    for (int i = own; i < items && !apart; ++i) {
      const ResItem I = it[i];
      const int e0 = M.rp[I.row0], e1 = M.rp[I.row0 + 1];
#pragma unroll 1
      for (int k = (warp + warps - at) % warps; k < I.len; k += warps)
        step_segment(M, e0 + k * kResSeg, min(kResSeg, e1 - e0 - k * kResSeg), g, pl.seg + I.ent + k);
      at = (at + I.len) % warps;
    }
    __syncthreads();
#pragma unroll 1
    for (int i = own + warp; i < items; i += warps) {
      const ResItem I = it[i];
      const double t = sum_words(pl.seg + I.ent, I.len);
      if (lane == 0) {
        s_sum[I.vec] = (V)t;
        s_row[I.vec] = I.row0;
      }
    }
  }
  __syncthreads();
  // ---- x+ or y+ -------------------------------------------------------------------
#pragma unroll 1
  for (int slot = tid; slot < slots; slot += threads) {
#pragma unroll
    for (int q = 0; q < kAcc; ++q) op.acc[q] = V(0);
#pragma unroll 1
    for (int t = slot; t < rows; t += kResThreads) {
      const V s[1] = {s_sum[t]};
      op.prefetch(s_row[t]);
      op.row(s_row[t], s);
    }
#pragma unroll
    for (int q = 0; q < kAcc; ++q) s_red[q * slots + slot] = (double)op.acc[q];
  }
  // ---- this block's record ----------------------------------------------------------
  __syncthreads();
  const int fields = collect ? kAcc : kPrimal ? 1 : 2;  // (the others are 0 unless they are recorded)
  if (warp < fields) {
    const double t = res_sum(s_red + warp * slots, min(kResWarps, (rows + 31) / 32));
    if (lane == 0) s_tot[warp] = t;
  }
  __syncthreads();
  if (tid == 0) {
    const int field[4] = {kPrimal ? 2 : 0, kPrimal ? 5 : 1, kPrimal ? 6 : 3, 4};  // (as in resident_kernel)
    for (int q = 0; q < fields; ++q)
      pl.rec[field[q] * pl.G + blockIdx.x].x = (unsigned long long)__double_as_longlong(s_tot[q]);
    if (!kPrimal) {
      unsigned int t;
      asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(t) : "l"(pl.bar + 4) : "memory");
      s_last = t == gridDim.x - 1;
    }
  }
  if constexpr (kPrimal) {
    pdl_trigger();
  } else {
    __syncthreads();
    if (!s_last) return;
    pdl_trigger();
    // ---- totals and step control ----------------------------------------------------
    double* const sd = reinterpret_cast<double*>(&s_st);
    for (int t = tid; t < (int)(sizeof(DevState) / 8); t += threads) sd[t] = reinterpret_cast<const double*>(d.st)[t];
    for (int f = warp; f < (collect ? 7 : 3); f += warps) {
      const double t = sum_words(pl.rec + f * pl.G, pl.G);
      if (lane == 0) s_tot[f] = t;
    }
    __syncthreads();
    if (tid == 0) {
      step_factors(d.step_tab, s_st.attempts + 1, s_fac, s_fac + 1);
      const double t1[3] = {s_tot[2], collect ? s_tot[5] : 0.0, collect ? s_tot[6] : 0.0};
      const double t2[4] = {s_tot[0], s_tot[1], collect ? s_tot[3] : 0.0, collect ? s_tot[4] : 0.0};
      step_control_state(s_st, prm, s_fac[0], s_fac[1], t1, t2);
      pl.bar[4] = 0u;
    }
    __syncthreads();
    for (int t = tid; t < (int)(sizeof(DevState) / 8); t += threads) reinterpret_cast<double*>(d.st)[t] = sd[t];
  }
}

// (at most 4 x 512 sums, and 5,800 rows of a CTA by 8 bytes or 3,200 by 12)
constexpr int kSteppedSmem = 56 * 1024;

template <class... KArgs, class... Args>
void launch_stepped_part(void (*kernel)(KArgs...), int grid, int warps, int smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(32u * (unsigned)warps, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, args...);  // errors surface through cudaGetLastError
}

template <class V, bool kPrimal>
void launch_stepped_half(const Dev& d, const Params& prm, const ResPlan& pl, const StepPlan& sp, bool crowd,
                         cudaStream_t s) {
  const int side = kPrimal ? 0 : 1, rows = kPrimal ? pl.rp : pl.rd;
  const int warps = crowd ? std::max(4, (sp.warps[side] + 1) / 2) : sp.warps[side];
  const bool apart = segments_apart(sp.longest[side]);
  if (apart) launch_stepped_part(stepped_segments_kernel<V, kPrimal>, pl.G, warps, 0, s, d, pl);
  launch_stepped_part(stepped_kernel<V, kPrimal>, pl.G, warps,
                      (kPrimal ? 3 : 4) * sum_slots(rows) * 8 + rows * (int)(sizeof(V) + 4), s, d, prm, pl, apart);
}

}  // namespace

void launch_stepped(const Dev& d, const Params& prm, const ResPlan& pl, const StepPlan& sp, bool fp32, bool crowd,
                    cudaStream_t s) {
  if (fp32) {
    launch_stepped_half<float, true>(d, prm, pl, sp, crowd, s);
    launch_stepped_half<float, false>(d, prm, pl, sp, crowd, s);
  } else {
    launch_stepped_half<double, true>(d, prm, pl, sp, crowd, s);
    launch_stepped_half<double, false>(d, prm, pl, sp, crowd, s);
  }
}

int stepped_launches(const StepPlan& sp) { return 2 + segments_apart(sp.longest[0]) + segments_apart(sp.longest[1]); }

cudaError_t stepped_smem_limit() {
  for (const void* fn : {(const void*)stepped_kernel<double, true>, (const void*)stepped_kernel<double, false>,
                         (const void*)stepped_kernel<float, true>, (const void*)stepped_kernel<float, false>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSteppedSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace lpop
