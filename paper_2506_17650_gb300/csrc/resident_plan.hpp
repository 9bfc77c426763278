// Plan of a resident check period (resident.hpp): how the rows of a problem are
// split over the CTAs and laid out in their shared memory, and the SMs that
// co-resident launches hold.  Pure C++ (no CUDA calls), so that it runs and is
// tested without a GPU.
#pragma once

#include <condition_variable>
#include <mutex>
#include <vector>

#include "layout_types.h"

struct ulonglong2;  // (CUDA vector type)

namespace lpop {

constexpr int kResThreads = 512;
constexpr int kResWarps = kResThreads / 32;
constexpr int kResMaxCtas = 160;   // records and tables are sized for this many
constexpr int kResSeg = 512;       // entries of a segment of a long row (G > 1)
constexpr int kResMaxSegs = 160;   // segments of a row, at most
constexpr int kSegKind = 64;       // kinds of items (1, 2, ... 32: lanes per row)
constexpr int kOwnKind = 65;

// A warp's work: `nrows` consecutive rows from row0 (bin order), local rows
// from `vec`, entries from `ent` in the CTA's entry arrays.  kind 0: a slice
// of 32 rows of at most kSellMaxLen entries, one lane each (entry k of its row
// t at ent + 32 k + t, `len` the longest row; neighbours in bin order have
// similar lengths, so few lanes idle, and a small matrix needs one slice where
// slices of one exact length would take many).  kind 2..32: CSR rows of kind
// lanes each; `len` is then the row's index among the CTA's long rows, which
// are its first local rows.  A row of more than kResSeg entries is cut: its
// segments (kind kSegKind: `nrows` entries of row row0 from entry `len` on) are
// dealt to warps of all CTAs and leave their sums in words `vec`; the CTA that
// has the row adds them up (kind kOwnKind: words ent, ent + 1, ... `len` of
// them).  A segment of a side whose entries stay in global memory has its place
// in the CSR arrays in ent; other items of such a side are all of CSR rows, and
// their ent is unused.
struct ResItem {
  int row0, nrows, len, kind;
  int ent, vec;
};

// A CTA's items [p0, p1) of A^T and [d0, d1) of A, long rows (nlp, nld) and rows.
struct ResCta {
  int p0, p1, d0, d1;
  int nlp, nld, rp, rd;
};

// What the kernel gets (device pointers; sizes are the largest over the CTAs).
struct ResPlan {
  const ResItem* items;
  const ResCta* cta;
  ulonglong2* rec;    // [7 * G] records of an attempt, field by field
  ulonglong2* ctl;    // [8 * (G / 8 + 1)] result of the step control, a line for each eight CTAs
  ulonglong2* seg;    // words of the segments: those of A^T, then those of A
  void* gx;           // words of x+ [n], then of y+ [2][m]
  unsigned int* bar;  // arrivals, number of the last attempt, start decision, arrivals before this launch; [4]: a
                      // stepped launch's finished blocks
  int G;
  int ep, ed, rp, rd, lp, ld, it;  // entries, rows, long rows of A^T / A; items of both
  int far;                         // 1: the entries of A^T, 2: those of A are read from the global CSR arrays
  int segs, segs_d;                // segments of both sides, and of A
  int longest;                     // entries of the longest row of A or A^T
  int smem;                        // dynamic shared memory, bytes
#ifdef LPOP_CHECK_BOUNDS
  // shorter limits of the waits (0: the usual ones), arrivals at the start and numbers of words (or arrivals)
  // within an attempt that nothing reaches, and whether the launch is refused
  struct {
    int start_spins, spins, missing_arrivals, missing_words, refuse;
  } test;
#endif
};

// The same plan's blocks as stepped launches (stepped.cu), for A^T (0) and A (1).  (Not in ResPlan: the compiler
// lays out the resident kernel anew with the size of its arguments, and with four words more an attempt of the
// 200,000-variable transportation LP took 17.0 us instead of 16.5.)
struct StepPlan {
  int longest[2];  // entries of the longest row
  int warps[2];    // warps of a block
};

// Byte offsets of a CTA's arrays in dynamic shared memory.
struct ResLayout {
  int vp, vd;    // values of A^T / A entries
  int xp, xd;    // ten vectors per A^T row, eight per A row
  int red;       // block sums: four fields of kResThreads doubles
  int cp, cd;    // column indices
  int lrp;       // first entry and length of the long rows (A^T rows, then A rows)
  int gp, gd;    // global rows
  int it, sense;
  int lenp, lend;  // lengths of the slices' rows
  int total;
};

LPOP_HD inline int up16(int b) { return (b + 15) & ~15; }

LPOP_HD inline ResLayout res_layout(const ResPlan& p, int esize) {
  ResLayout L;
  int o = 0;
  L.vp = o; o += up16(p.ep * esize);
  L.vd = o; o += up16(p.ed * esize);
  L.xp = o; o += up16(10 * p.rp * esize);
  L.xd = o; o += up16(8 * p.rd * esize);
  L.red = o; o += 4 * kResThreads * 8;
  L.cp = o; o += up16(p.ep * 4);
  L.cd = o; o += up16(p.ed * 4);
  L.lrp = o; o += up16((p.lp + p.ld) * 8);
  L.gp = o; o += up16(p.rp * 4);
  L.gd = o; o += up16(p.rd * 4);
  L.it = o; o += up16(p.it * (int)sizeof(ResItem));
  L.sense = o; o += up16(p.rd);
  L.lenp = o; o += up16(p.rp);
  L.lend = o; o += up16(p.rd);
  L.total = o;
  return L;
}

// Whether a problem of this size may be resident with values of `esize`
// bytes, and the device bytes its plan takes at most.
bool resident_possible(long long m, long long n, long long nnz, int esize);
long long resident_bytes(long long m, long long n, long long nnz, int esize);

struct ResHost {
  std::vector<ResItem> items;
  std::vector<ResCta> cta;
  ResPlan plan{};  // without its device pointers
  StepPlan step{};
};

// The plan of a problem's rows (bin tables of A and A^T) for values of
// `esize` bytes, at most `sms` CTAs and `smem_limit` bytes each.  head_a /
// head_at: row pointers of the rows before the first sliced row.  Returns
// false when the problem does not fit.
bool resident_build(const BinTable& binsA, const BinTable& binsAt, long long m, long long n, long long nnz,
                    const std::vector<int>& head_a, const std::vector<int>& head_at, int esize, int sms,
                    int smem_limit, ResHost& out);
int resident_long_rows(const BinTable& bt);  // rows before the first sliced row

// SMs of a device that co-resident kernels hold.  The CTAs of a resident
// launch wait for one another, so two launches that each got part of the GPU
// would wait for ever: lp_solve takes the SMs of its launch first and gives them
// back when the period has finished; the batched kernel (which would otherwise
// hold every SM for a whole round) takes what is free.
//
// One after the other, resident periods leave most of the GPU idle: their
// attempts are chains of latencies.  Solves from several threads whose plans do
// not fit side by side therefore run stepped, which gives the same bits and fills
// the GPU between them; two of them, and small ones, take turns.  us per attempt
// over all threads, FP64, all in turns / as now (with the two step kernels):
//   threads                       2                 4                 8                 16
//   60k nonzeros, 123 CTAs   8.6 / 8.7 (9.7)   8.6 / 4.3 (5.2)   8.7 / 2.9 (3.1)   9.0 / 2.2 (2.4)
//   linking rows, 152       12.7 /12.7 (14.7) 12.7 / 8.1 (8.4)  12.9 / 5.9 (6.2)  13.2 / 5.3 (6.3)
//   transport, 152          17.3 /17.9 (18.0) 17.3 /15.6 (16.7) 17.3 /16.6 (16.9) 17.6 /14.4 (17.3)
//   power law 1e6, 152      32.3 /32.3 (28.1) 31.9 /29.0 (27.6) 31.6 /26.8 (27.5) 32.0 /22.5 (27.6)
// The stepped blocks have a warp per item, or, with very many solves, one per two.
constexpr int kFewSms = 8;  // plans of at most this fraction of the SMs take turns
constexpr int kCrowd = 8;   // very many: plans of this many times the SMs

class SmTokens {
 public:
  explicit SmTokens(int sms) : sms_(sms), free_(sms) {}
  // Takes between `least` and `most` SMs, waiting for `least` and for earlier callers.
  int acquire(int least, int most);
  // Takes `count` SMs for a resident period, or returns false: it should run stepped.
  bool acquire_resident(int count);
  bool crowded();
  void release(int count);
  // SMs that a solve or a batch round in progress takes, or would take by itself.
  void announce(int count, bool round);
  void withdraw(int count, bool round);

 private:
  int wait_turn(std::unique_lock<std::mutex>& lk, int least, int most);
  std::mutex mu_;
  std::condition_variable cv_;
  const int sms_;
  int free_;
  int wanted_ = 0, rounds_ = 0;
  unsigned long long next_ = 0, serving_ = 0;
};

}  // namespace lpop
