// Check periods of small and medium problems in one launch: the whole
// problem is kept in the shared memory of the CTAs that iterate on it.
//
// The two step kernels (kernels_iter.cu) cost 15-25 us per attempt however
// small the problem is: two dependent launches, each with its own chain of
// loads from L2, a last block that sums every record while the rest of the
// GPU waits, and a step control with cold instruction caches.  A problem whose
// matrix copies and vectors fit in the shared memory of the GPU's SMs is
// instead split by rows over G CTAs (one per SM) that hold their rows of
// A and A^T, the rows' vectors and the solver state for a whole check period.
// Per attempt only x+ and y+ travel (through L2), as words of a value and the
// number of its attempt or, with rows that many others gather, between grid-wide
// barriers; CTA 0 sums the CTAs' records, runs the step control and sends its
// result to the others.  A problem that fits in one SM takes a single CTA and
// exchanges nothing.  Where the vectors fit but not both copies of the matrix, one
// or both copies are read from global memory (L2) in each attempt.  resident.cu
// and resident_plan.cpp have the measured times and the choices.
//
// The same plan can run stepped (stepped.cu): plain launches with the same bits,
// for periods that cannot have the SMs to themselves.
#pragma once

#include "common.cuh"
#include "resident_plan.hpp"

namespace lpop {

// Up to `attempts` step attempts in one launch (cooperative when G > 1).
cudaError_t launch_resident(const Dev& d, const Params& prm, const ResPlan& pl, bool fp32, int attempts,
                            cudaStream_t s);
// One step attempt of the plan in plain launches, with the same bits (G > 1); crowd: with fewer warps.
void launch_stepped(const Dev& d, const Params& prm, const ResPlan& pl, const StepPlan& sp, bool fp32, bool crowd,
                    cudaStream_t s);
bool single_attempt_stepped(const ResPlan& pl);  // whether a launch of one attempt had better be stepped
int shortest_period(const ResPlan& pl);  // check periods below this take the two step kernels
int stepped_launches(const StepPlan& sp);  // kernels of that
cudaError_t stepped_smem_limit();  // lets the stepped kernels have the shared memory they may need
cudaError_t resident_smem_limit(int device, int* bytes);  // dynamic shared memory a CTA may take

// The SMs of a device (shared by every problem and batch on it).
SmTokens& sm_tokens(int device, int sms);

// Between `least` and `most` SMs, held for the lifetime of the object.
struct SmLease {
  SmTokens& tokens;
  int count;
  SmLease(int device, int sms, int least, int most)
      : tokens(sm_tokens(device, sms)), count(tokens.acquire(least, most)) {}
  ~SmLease() { tokens.release(count); }
  SmLease(const SmLease&) = delete;
  SmLease& operator=(const SmLease&) = delete;
};

// The SMs of a resident period, if it may be one (a plan of one CTA needs none).
struct ResidentLease {
  SmTokens* tokens;
  const int count;
  bool ok = true;
  ResidentLease(int device, int sms, int ctas) : tokens(ctas > 1 ? &sm_tokens(device, sms) : nullptr), count(ctas) {
    if (tokens) ok = tokens->acquire_resident(count);
  }
  ~ResidentLease() {
    if (tokens && ok) tokens->release(count);
  }
  ResidentLease(const ResidentLease&) = delete;
  ResidentLease& operator=(const ResidentLease&) = delete;
};

// What a solve or a batch round in progress takes of the SMs.
struct SmDemand {
  SmTokens& tokens;
  const bool round;
  int count = 0;
  SmDemand(int device, int sms, bool batch_round) : tokens(sm_tokens(device, sms)), round(batch_round) {
    tokens.announce(0, round);
  }
  void set(int want) {
    if (want != count) tokens.announce(want - count, false);
    count = want;
  }
  ~SmDemand() { tokens.withdraw(count, round); }
  SmDemand(const SmDemand&) = delete;
  SmDemand& operator=(const SmDemand&) = delete;
};

}  // namespace lpop
