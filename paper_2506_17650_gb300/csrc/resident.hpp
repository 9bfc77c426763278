// Check periods of small and medium problems in one launch: the whole
// problem is kept in the shared memory of the CTAs that iterate on it.
//
// The two step kernels (kernels_iter.cu) cost 15-25 us per attempt however
// small the problem is: two dependent launches, each with its own chain of
// loads from L2, a last block that sums every record while the rest of the
// GPU waits, and a step control with cold instruction caches.  A problem whose
// matrix copies and vectors fit in the shared memory of the GPU's SMs is
// instead split by rows over G CTAs (one per SM) that hold their rows of
// A and A^T, the rows' vectors and the solver state for a whole check period:
// per attempt only x+ and y+ travel (through L2), between grid-wide barriers,
// and every CTA sums the G records and runs the step control on its own copy
// of the state.  A problem that fits in one SM takes a single CTA and no grid
// barrier.  Where the vectors fit but not both copies of the matrix, one or both
// copies are read from global memory (L2) in each attempt.  resident.cu and
// resident_plan.cpp have the measured times and the choices.
#pragma once

#include "common.cuh"
#include "resident_plan.hpp"

namespace lpop {

// Up to `attempts` step attempts in one launch (cooperative when G > 1).
cudaError_t launch_resident(const Dev& d, const Params& prm, const ResPlan& pl, bool fp32, int attempts,
                            cudaStream_t s);
// One step attempt of the plan in two plain launches, with the same bits (G > 1).
void launch_stepped(const Dev& d, const Params& prm, const ResPlan& pl, bool fp32, cudaStream_t s);
cudaError_t resident_smem_limit(int device, int* bytes);  // dynamic shared memory a CTA may take

// The SMs of a device (shared by every problem and batch on it).
SmTokens& sm_tokens(int device, int sms);

// Between `least` and `most` SMs, held for the lifetime of the object (none for least 0).
struct SmLease {
  SmTokens* tokens;
  int count;
  SmLease(int device, int sms, int least, int most)
      : tokens(least > 0 ? &sm_tokens(device, sms) : nullptr), count(tokens ? tokens->acquire(least, most) : 0) {}
  ~SmLease() {
    if (tokens) tokens->release(count);
  }
  SmLease(const SmLease&) = delete;
  SmLease& operator=(const SmLease&) = delete;
};

}  // namespace lpop
