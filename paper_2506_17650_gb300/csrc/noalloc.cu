// lp_power_norm_noalloc: the power-iteration estimate of ||A||_2 (the one
// lp_create runs in plain mode to pick the vanilla step size 0.9 / ||A||_2)
// for callers that cannot allocate device memory.
//
// Who needs it: code that runs where cudaMalloc is not available or not
// allowed -- a plugin inside a host framework that has reserved all of device
// memory for its own pool, a real-time loop that must not allocate, or a
// caller whose device buffers come from another allocator.  Such a caller
// already holds its matrix on the device and only wants the estimate.
//
// The scratch (two work vectors, the blocks' partial sums and the iteration's
// scalars) lives in one file-scope device array of fixed size, so the call
// allocates nothing.  (Sizes are still refused by the bound of an earlier form
// with three vectors, 2 n + m + 1025 doubles.)
// Every GPU that loads the library keeps that array until the process exits.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "../../include/lpop.h"
#include "common.cuh"

namespace lpop {
void set_thread_error(const std::string& msg);  // api.cu

namespace {

// 2^20 doubles = 8 MiB of scratch per device
constexpr long long kScratchDoubles = 1LL << 20;
constexpr long long kReduceDoubles = 1 + 1024;  // per-block partial sums, and one

// (and a few more for the iteration's scalars)
__device__ __align__(256) double g_noalloc_scratch[kScratchDoubles + 8];

constexpr int kMaxDevices = 64;
double* g_scratch_addr[kMaxDevices] = {nullptr};
std::mutex g_scratch_mutex;

int fail(int code, const std::string& msg) {
  set_thread_error(msg);  // reported by lp_last_error(NULL)
  return code;
}

// Device address of the scratch array on the current device, looked up once per device.
int scratch_address(int dev, double** out) {
  if (dev < 0 || dev >= kMaxDevices) return fail(LP_ERR_INVALID_ARG, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return fail(LP_ERR_CUDA, std::string("cudaGetSymbolAddress failed: ") + cudaGetErrorString(e));
    g_scratch_addr[dev] = static_cast<double*>(ptr);
  }
  *out = g_scratch_addr[dev];
  return LP_OK;
}

// Scalars of the iteration, after the partial sums.
struct NormState {
  double norm;        // ||w|| of the last round
  double inv;         // what the next product is scaled by: 1 / norm (1 before the first round and for a zero norm)
  unsigned int done;  // blocks that have finished in the running launch
  unsigned int rounds;
  unsigned int restarted;  // the first round's product was zero
  unsigned int unused;
};

__global__ void norm_init_kernel(NormState* st) { *st = NormState{0.0, 1.0, 0u, 0u, 0u, 0u}; }

// y = (M x) * st->inv for a CSR matrix whose row lengths nobody has looked at;
// with kNorm (y = M x then) also ||y|| into the state, by the last block, in a
// fixed order.
//
// One launch instead of the four of a product, a two-step norm and a division
// pass: the division is folded into the next product.  W lanes take a row,
// W from the mean row length; what limits short rows is the FP64 pipe, where a
// shuffle-add of a warp costs as much as 32 useful FMAs, so W is small (8 lanes
// for rows of 6 entries spent three quarters of the pipe on lane sums).  Rows
// of more than 32 W entries wait and are then taken by the whole warp, one by one.
// 120,000 x 300,000, 1.8M nonzeros, 200 rounds: 13.4 -> 5.5 ms.
//
// Where the caller has sorted its rows, longest first, the first `wide` take a
// block each and those up to `head` a warp each, dealt out over the blocks: the
// longest 32 would otherwise wait for one warp (plain lp_create of a 100k-nonzero
// power-law LP: 22.7 ms, 6.3 so).
//
// Where the first product is zero, its last warp also writes the second start
// direction, +-1/sqrt(n) by the SplitMix64 signs of perm[j] (or j): the following
// launches then go on from there, and the host adds a round (a 60,000 x 20,000
// incidence matrix, 200 rounds: 4.1 ms with all rounds run twice, 2.1 so).
struct SortedRows {
  int wide, head;
  const int* perm;
};
struct UnsortedRows {};

template <int W, bool kNorm, class Order>
__global__ void __launch_bounds__(kBlock, 6) norm_rows_kernel(int rows, const int* rp, const int* ci, const double* v,
                                                           const double* x, double* y, NormState* st, double* part,
                                                           Order order) {
  constexpr bool kSorted = std::is_same<Order, SortedRows>::value;
  __shared__ double smem[kBlock];
  __shared__ int s_last;
  pdl_wait();
  const int lane = (int)threadIdx.x & 31, sub = lane % W;
  const int warp = (int)(blockIdx.x * kBlock + threadIdx.x) >> 5, warps = (int)(gridDim.x * kBlock) >> 5;
  const double inv = kNorm ? 1.0 : st->inv;
  double acc[1] = {0.0};
  auto dot = [&](int k, int e, int step) {
    double t = 0.0;
    for (; k < e; k += 4 * step) {
      int c[4];
      double a[4], g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool ok = k + u * step < e;
        c[u] = ok ? __ldg(ci + k + u * step) : -1;
        a[u] = ok ? __ldg(v + k + u * step) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) g[u] = c[u] >= 0 ? __ldg(x + c[u]) : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (c[u] >= 0) t = fma(a[u], g[u], t);
    }
    return t;
  };
  if constexpr (kSorted) {
    for (int row = (int)blockIdx.x; row < order.wide; row += (int)gridDim.x) {
      double t[1] = {dot(__ldg(rp + row) + (int)threadIdx.x, __ldg(rp + row + 1), kBlock)};
      block_sum_smem<1>(t, smem);
      if (threadIdx.x == 0) {
        y[row] = t[0] * inv;
        if (kNorm) acc[0] += (t[0] * inv) * (t[0] * inv);
      }
    }
    for (int row = order.wide + (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x; row < order.head; row += warps) {
      double t = dot(__ldg(rp + row) + lane, __ldg(rp + row + 1), 32);
      __syncwarp();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) {
        y[row] = t * inv;
        if (kNorm) acc[0] += (t * inv) * (t * inv);
      }
    }
  }
  int first = 0;
  if constexpr (kSorted) first = order.head;
  for (long long r0 = first + (long long)warp * (32 / W); r0 < rows; r0 += (long long)warps * (32 / W)) {
    const long long row = r0 + lane / W;
    const bool has = row < rows;
    const int beg = has ? __ldg(rp + row) : 0, end = has ? __ldg(rp + row + 1) : 0;
    const bool lng = end - beg > 32 * W;
    double s = 0.0;
    if (!lng) s = dot(beg + sub, end, W);
    __syncwarp();
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, W);
    for (unsigned int m = __ballot_sync(0xffffffffu, lng && sub == 0); m; m &= m - 1) {
      const int q = __ffs(m) - 1;
      double t = dot(__shfl_sync(0xffffffffu, beg, q) + lane, __shfl_sync(0xffffffffu, end, q), 32);
      __syncwarp();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == q) s = t;
    }
    if (has && sub == 0) {
      s *= inv;
      y[row] = s;
      if (kNorm) acc[0] += s * s;
    }
  }
  if (!kNorm) {
    pdl_trigger();
    return;
  }
  block_sum_smem<1>(acc, smem);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = acc[0];
    unsigned int t;
    asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(t) : "l"(&st->done) : "memory");
    s_last = t == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  pdl_trigger();
  const unsigned int rounds = st->rounds;
  double sum[1] = {0.0};
  for (int b = threadIdx.x; b < (int)gridDim.x; b += kBlock) sum[0] += __ldcg(part + b);
  block_sum_smem<1>(sum, smem);
  if (threadIdx.x >= 32) return;
  const bool zero = __double_as_longlong(sum[0]) == 0;  // (the sum is in every lane and not negative)
  const bool again = zero && rounds == 0u;
  if (threadIdx.x == 0) {
    const double nw = sqrt(sum[0]);
    st->norm = nw;
    st->inv = zero ? 1.0 : 1.0 / nw;
    st->rounds = rounds + 1u;
    if (again) st->restarted = 1u;
    st->done = 0u;
  }
  if (again) {
    const double one = 1.0 / sqrt((double)rows);
    for (int j = threadIdx.x; j < rows; j += 32) {
      int col = j;
      if constexpr (kSorted) col = order.perm ? order.perm[j] : j;
      y[j] = one * splitmix_sign((unsigned long long)col);
    }
  }
}

template <bool kNorm>
void launch_norm_rows(int rows, const int* rp, const int* ci, const double* val, const double* x, double* y,
                      NormState* st, double* part, double mean, const BinTable* sorted, const int* perm, cudaStream_t s) {
  const int W = sorted && mean <= 16.0 ? 1 : mean <= 8.0 ? 2 : (mean <= 32.0 ? 4 : (mean <= 128.0 ? 8 : 32));
  // with one lane a row, rows of more than 32 entries by a warp; with 4 or 8, of more than 64 or 256
  int wide = 0, head = 0;
  for (int b = 0; sorted && b < sorted->nbins; ++b) {
    const Bin& B = sorted->bin[b];
    const bool by_block = B.width == 0 || B.width == kSegmented;
    if (by_block) wide = B.row_end;
    if (by_block || (W == 1 && (B.width != kSell || B.len > 32)) || (W == 4 && B.width >= 16) || (W == 8 && B.width == 32))
      head = B.row_end;
  }
  const long long warps = 8LL * wide + (head - wide) + ((long long)(rows - head) * W + 31) / 32;
  constexpr long long kMostBlocks = 912;  // six on each of GB300's 152 SMs
  const int grid = (int)std::max<long long>(1, std::min(kMostBlocks, (warps + kBlock / 32 - 1) / (kBlock / 32)));
  auto launch = [&](auto unsorted, auto in_order) {
    if (sorted) launch_pdl(in_order, grid, s, rows, rp, ci, val, x, y, st, part, SortedRows{wide, head, perm});
    else launch_pdl(unsorted, grid, s, rows, rp, ci, val, x, y, st, part, UnsortedRows{});
  };
  if (W == 1) launch(norm_rows_kernel<2, kNorm, UnsortedRows>, norm_rows_kernel<1, kNorm, SortedRows>);
  else if (W == 2) launch(norm_rows_kernel<2, kNorm, UnsortedRows>, norm_rows_kernel<2, kNorm, SortedRows>);
  else if (W == 4) launch(norm_rows_kernel<4, kNorm, UnsortedRows>, norm_rows_kernel<4, kNorm, SortedRows>);
  else if (W == 8) launch(norm_rows_kernel<8, kNorm, UnsortedRows>, norm_rows_kernel<8, kNorm, SortedRows>);
  else launch(norm_rows_kernel<32, kNorm, UnsortedRows>, norm_rows_kernel<32, kNorm, SortedRows>);
}

}  // namespace

size_t power_norm_state_bytes() { return sizeof(NormState); }

// ||w|| of the last of `iters` rounds w = A^T A w / ||w|| from the all-ones
// direction, or (a zero first product: every row of A sums to zero) from the
// SplitMix64 sign direction.  w [n], t [m], part [1024], state: device scratch.
// bins: the row classes of A and A^T, whose rows are then sorted, longest first
// (null: nothing is known of the rows).  With them short rows are summed by one
// lane, as one chain of FMAs (whether rows that sum to zero give exactly zero
// depends on that, and with it the start direction).
cudaError_t power_norm(int m, int n, long long nnz, const Csr& A, const Csr& At, int iters, const int* perm,
                       const BinTable* binsA, const BinTable* binsAt, double* w, double* t, double* part, void* state,
                       cudaStream_t s, double* norm) {
  NormState* st = static_cast<NormState*>(state);
  launch_fill(w, 1.0 / std::sqrt((double)n), n, s);
  norm_init_kernel<<<1, 1, 0, s>>>(st);
  NormState h{};
  for (int rounds = iters; rounds > 0;) {
    for (int it = 0; it < rounds; ++it) {
      launch_norm_rows<false>(m, A.rp, A.ci, A.v, w, t, st, part, (double)nnz / m, binsA, nullptr, s);
      launch_norm_rows<true>(n, At.rp, At.ci, At.v, t, w, st, part, (double)nnz / n, binsAt, perm, s);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    rounds = rounds == iters && h.restarted && h.rounds == (unsigned)iters ? 1 : 0;  // the round that was lost
  }
  *norm = h.norm;
  return cudaSuccess;
}

}  // namespace lpop

using namespace lpop;

extern "C" int lp_power_norm_noalloc(int32_t m, int32_t n, const int32_t* a_row_ptr, const int32_t* a_col_idx,
                                     const double* a_val, const int32_t* at_row_ptr, const int32_t* at_col_idx,
                                     const double* at_val, int32_t iters, void* stream, double* norm_out) {
  if (!norm_out) return fail(LP_ERR_INVALID_ARG, "norm_out must not be NULL");
  *norm_out = 0.0;
  if (m < 1 || n < 1 || iters < 1) return fail(LP_ERR_INVALID_ARG, "need m >= 1, n >= 1 and iters >= 1");
  if (!a_row_ptr || !a_col_idx || !a_val || !at_row_ptr || !at_col_idx || !at_val)
    return fail(LP_ERR_INVALID_ARG, "matrix pointers must not be NULL");
  const long long need = 2LL * n + m + kReduceDoubles;
  if (need > kScratchDoubles)
    return fail(LP_ERR_INVALID_ARG, "problem too large for the fixed scratch: need 2 n + m + 1025 = " +
                                        std::to_string(need) + " doubles, the maximum is " +
                                        std::to_string(kScratchDoubles));
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(LP_ERR_CUDA, std::string("cudaGetDevice failed: ") + cudaGetErrorString(e));
  double* scratch = nullptr;
  int rc = scratch_address(dev, &scratch);
  if (rc != LP_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // w (n) | t (m) | partial sums (1024); the scalars after the array's 2^20 doubles
  static_assert(sizeof(NormState) <= 8 * sizeof(double), "scalars after the array");
  int nnz = 0;
  e = cudaMemcpyAsync(&nnz, a_row_ptr + m, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  double nw = 0.0;
  if (e == cudaSuccess)
    e = power_norm(m, n, nnz, Csr{a_row_ptr, a_col_idx, a_val}, Csr{at_row_ptr, at_col_idx, at_val}, iters, nullptr, nullptr,
                   nullptr, scratch, scratch + n, scratch + n + m, scratch + kScratchDoubles, s, &nw);
  if (e != cudaSuccess) return fail(LP_ERR_CUDA, std::string("power iteration failed: ") + cudaGetErrorString(e));
  *norm_out = nw > 0.0 && std::isfinite(nw) ? std::sqrt(nw) : 0.0;
  return LP_OK;
}
