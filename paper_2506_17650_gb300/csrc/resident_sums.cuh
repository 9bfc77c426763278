// Row sums and block sums of the resident kernel (resident.cu), which the stepped
// kernels (stepped.cu) form in the same order.
#pragma once

#include "common.cuh"
#include "resident_plan.hpp"

namespace lpop {

namespace {

// The word of one element of x+ or y+.
template <class V>
struct ResElt;
template <>
struct ResElt<double> {
  using T = ulonglong2;
  static __device__ __forceinline__ void put(T* p, double v, unsigned int seq) {
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p),
                 "l"(__double_as_longlong(v)), "l"((unsigned long long)seq)
                 : "memory");
  }
  // the value, and whether it is of attempt `seq` (or later)
  static __device__ __forceinline__ bool get(const T* p, unsigned int seq, double* v) {
    unsigned long long a, b;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=l"(a), "=l"(b)
                 : "l"(p)
                 : "memory");
    *v = __longlong_as_double((long long)a);
    return (int)((unsigned int)b - seq) >= 0;
  }
};
template <>
struct ResElt<float> {
  using T = unsigned long long;
  static __device__ __forceinline__ void put(T* p, float v, unsigned int seq) {
    const T w = (T)seq << 32 | (T)__float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
  }
  static __device__ __forceinline__ bool get(const T* p, unsigned int seq, float* v) {
    T w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    *v = __uint_as_float((unsigned int)w);
    return (int)((unsigned int)(w >> 32) - seq) >= 0;
  }
};

// What the rows of one side gather: the vector x (one CTA: in shared memory;
// with barriers: the global vector, by plain loads that the L1 may serve), or
// the words of the other CTAs of this launch.
// How a launch's CTAs see one another's x+ and y+.
enum ResKind { kSoloKind = 0, kWordsKind = 1, kBarriersKind = 2 };

template <class V, int kKind>
struct ResGather {
  const V* x;
  const typename ResElt<V>::T* g;
  unsigned int seq;
  int n;
  unsigned int* bad;
  int spins;
  // xv[u] = x[c[u step]] for u < min(4, count); false if a word did not come
  __device__ __forceinline__ bool four(const int* c, int step, int count, V (&xv)[4]) const {
    const int none = -1;
    int j[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      j[u] = u < count ? c[u * step] : none;
      xv[u] = V(0);
#ifdef LPOP_CHECK_BOUNDS
      if (j[u] != none && (unsigned)j[u] >= (unsigned)n) {
        if (bad) atomicAdd(bad, 1u);
        j[u] = none;
      }
#endif
    }
    if constexpr (kKind != kWordsKind) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j[u] != none) xv[u] = x[j[u]];
      return true;
    } else {
      for (int t = 0; t < spins; ++t) {
        bool here = true;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j[u] != none) here = ResElt<V>::get(g + j[u], seq, xv + u) && here;
        if (here) return true;
      }
      return false;
    }
  }
};

// sum over k < count of v[k step] x[c[k step]], four gathers in flight.
// `most` is the warp's largest count: terms past it are skipped by a uniform
// branch.  FP64 sums over several CTAs in two chains (a gather's latency is
// already there, and a chain of 55-65 cycles a term on top of it); one CTA's,
// bound by the FP64 pipe, and FP32 in one.
template <class V, int kKind>
__device__ __forceinline__ V res_dot(const V* v, const int* c, int count, int most, int step,
                                     const ResGather<V, kKind>& g, bool* ok) {
  constexpr int kChains = sizeof(V) == 8 && kKind != kSoloKind ? 2 : 1;
  V a[kChains];
#pragma unroll
  for (int q = 0; q < kChains; ++q) a[q] = V(0);
#pragma unroll 1
  for (int k0 = 0; k0 < most; k0 += 4) {
    V xv[4] = {V(0), V(0), V(0), V(0)};
    if (*ok && !g.four(c, step, count - k0, xv)) *ok = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (k0 + u >= most) break;
      if (k0 + u < count) a[u % kChains] = fma(v[u * step], xv[u], a[u % kChains]);
    }
    v += 4 * step;
    c += 4 * step;
  }
  return kChains == 2 ? a[0] + a[kChains - 1] : a[0];
}

// The kernel's loop over the attempts is straight-line code that each warp
// runs once per attempt, so its instruction fetches are on the critical path
// like every other latency: the pieces below are short loops rather than
// unrolled code (the same sums unrolled took about twice the cycles).

// Sum over the lanes (valid in every lane).
__device__ __forceinline__ double lane_sum(double t) {
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Sum of red[32 k + lane] over the lanes and k < nw (slots past nw are 0).
__device__ __forceinline__ double res_sum(const double* red, int nw) {
  red += threadIdx.x & 31;
  double t = 0.0;
#pragma unroll 1
  for (int k = 0; k < nw; k += 4, red += 128) t += (red[0] + red[32]) + (red[64] + red[96]);
  return lane_sum(t);
}

// Sum over the CTAs (or a row's segments) of words that are known to be there, in
// the order of the resident kernel's (all lanes of the calling warp).
__device__ __forceinline__ double sum_words(const ulonglong2* rec, int G) {
  const int lane = threadIdx.x & 31;
  double v[kResMaxCtas / 32];
#pragma unroll
  for (int q = 0; q < kResMaxCtas / 32; ++q) {
    const int g = lane + 32 * q;
    v[q] = g < G ? __longlong_as_double((long long)__ldcg(&rec[g].x)) : 0.0;
  }
  return lane_sum(((v[0] + v[1]) + (v[2] + v[3])) + v[4]);
}

}  // namespace

}  // namespace lpop
