#include "resident_plan.hpp"

#include <algorithm>
#include <utility>

namespace lpop {

namespace {

// FP64-pipe cost of an item, in warp instructions: a slice's FMAs and epilogue, a group of long rows' FMAs,
// shuffle adds and (one lane per row, so shared by 32 rows) epilogue.
double item_cost(const ResItem& I, int longest) {
  if (I.kind == 0) return I.len + 9.0;
  if (I.kind <= 32) return (longest + I.kind - 1) / I.kind + 3.0 + 10.0 * I.nrows / 32.0;
  return I.kind == kSegKind ? (I.nrows + 31) / 32 + 6.0 : 7.0;
}

// `count` items of the same cost and number of entries, `step` rows apart.
struct Run {
  ResItem item;
  int count, step, entries;
  double cost;
};

// One side's items; short rows (those of the sliced bins) by `lanes` lanes each,
// rows of more than kResSeg entries cut into segments if `cut`.
std::vector<Run> side_items(const BinTable& bt, const std::vector<int>& head, int lanes, bool cut) {
  std::vector<Run> out;
  int b = 0, slot = 0;
  for (; b < bt.nbins && bt.bin[b].width != kSell; ++b) {
    const Bin& B = bt.bin[b];
    const int kind = B.width <= 0 ? 32 : (B.width < 4 ? 4 : B.width);  // (whole-block and segmented rows: a warp)
    for (int r = B.row_begin; r < B.row_end;) {
      const int len = head[r + 1] - head[r];
      if (cut && len > kResSeg) {
        const int n = (len + kResSeg - 1) / kResSeg;
        for (int k = 0; k < n; ++k) {
          const int beg = k * kResSeg, size = std::min(kResSeg, len - beg);
          ResItem I{r, size, beg, kSegKind, head[r] + beg, slot + k};
          out.push_back(Run{I, 1, 0, size, item_cost(I, 0)});
        }
        ResItem I{r, 1, n, kOwnKind, slot, 0};
        out.push_back(Run{I, 1, 0, 0, item_cost(I, 0)});
        slot += n;
        ++r;
        continue;
      }
      const int rows = std::min(32 / kind, B.row_end - r);
      ResItem I{r, rows, 0, kind, 0, 0};
      // (rows are longest first within a class)
      out.push_back(Run{I, 1, 0, head[r + rows] - head[r], item_cost(I, len)});
      r += rows;
    }
  }
  const int end = bt.nbins > 0 ? bt.bin[bt.nbins - 1].row_end : 0;
  const int per = 32 / lanes;
  for (int r = b < bt.nbins ? bt.bin[b].row_begin : end; r < end;) {
    while (bt.bin[b].row_end <= r) ++b;  // bins hold one exact length each, longest first
    const int longest = bt.bin[b].len, whole = (bt.bin[b].row_end - r) / per;
    if (whole > 0) {  // the items that end within the bin
      ResItem I{r, per, lanes == 1 ? longest : 0, lanes == 1 ? 0 : lanes, 0, 0};
      out.push_back(Run{I, whole, per, per * longest, item_cost(I, longest)});
      r += whole * per;
      continue;
    }
    const int rows = std::min(per, end - r);
    int entries = 32 * longest;
    if (lanes > 1) {
      entries = 0;
      for (int k = r, q = b; k < r + rows; ++q) {
        const int upto = std::min(r + rows, bt.bin[q].row_end);
        if (upto > k) {
          entries += (upto - k) * bt.bin[q].len;
          k = upto;
        }
      }
    }
    ResItem I{r, rows, lanes == 1 ? longest : 0, lanes == 1 ? 0 : lanes, 0, 0};
    out.push_back(Run{I, 1, 0, entries, item_cost(I, longest)});
    r += rows;
  }
  return out;
}

// Lanes per short row when a CTA has `rows` rows of `length` entries on
// average: more than one while the CTA's warps are not filled and a lane still
// gets about four entries (a row's gathers are then in flight together).
int short_row_lanes(double rows, double length) {
  int w = 1;
  while (w < 8 && rows * 2 * w <= kResThreads - 96 && length > 3.0 * w) w *= 2;
  return w;
}

// Order of a CTA's items: segments first (others wait for them), the rows that wait for them last.
int rank_of(const ResItem& I) { return I.kind == kSegKind ? 0 : I.kind == kOwnKind ? 3 : I.kind > 0 ? 1 : 2; }

// Longest-first assignment of one side's items to G CTAs: each item, most
// costly first, to the CTA with the least work so far (in bin order for G = 1:
// a local row is then the global one).
struct Deal {
  struct Cta {
    int entries = 0, nlong = 0, rows = 0, items = 0;  // (nlong: rows that are not in slices)
  };
  std::vector<Run> runs;
  std::vector<int> owner;  // of the runs' items in turn
  std::vector<Cta> cta;
};

// Among items of one cost the CTAs that took one stand in line in the order in
// which they took it, so the next is the first of that line or of the CTAs that
// have not had one: no heap is needed.  The first solve pays for the plan (a
// power-law LP of 1M entries: three deals of 16,000 to 24,000 items); with the
// items sorted and dealt through a heap it took 7,476 us, now 2,828 (a later
// solve 2,157).
void deal(std::vector<Run> runs, int G, Deal& out) {
  if (G > 1)
    std::stable_sort(runs.begin(), runs.end(), [](const Run& a, const Run& b) { return a.cost > b.cost; });
  out.cta.assign(G, Deal::Cta{});
  out.owner.clear();
  using Load = std::pair<double, int>;
  std::vector<Load> idle(G), line, merged(G);
  for (int g = 0; g < G; ++g) idle[g] = {0.0, g};
  size_t i0 = 0, l0 = 0;
  double cost = runs.empty() ? 0.0 : runs[0].cost;
  for (const Run& r : runs) {
    const bool seg = r.item.kind == kSegKind, own = r.item.kind == kOwnKind;
    if (r.cost != cost) {
      std::merge(idle.begin() + i0, idle.end(), line.begin() + l0, line.end(), merged.begin());
      idle.swap(merged);
      line.clear();
      i0 = l0 = 0;
      cost = r.cost;
    }
    for (int i = 0; i < r.count; ++i) {
      const bool from_line = l0 < line.size() && (i0 == idle.size() || line[l0] < idle[i0]);
      const Load l = from_line ? line[l0++] : idle[i0++];
      line.push_back({l.first + r.cost, l.second});
      out.owner.push_back(l.second);
      Deal::Cta& C = out.cta[l.second];
      C.items += 1;
      C.entries += own ? 0 : r.entries;
      C.rows += seg ? 0 : r.item.nrows;
      C.nlong += seg || r.item.kind == 0 ? 0 : r.item.nrows;
    }
  }
  out.runs = std::move(runs);
}

// The CTAs' items, one CTA after the other, A^T's before A's, with their places in the CTA's arrays.
void lay_out(const Deal (&sides)[2], ResHost& out) {
  ResPlan& pl = out.plan;
  const int G = pl.G;
  for (int side = 0; side < 2; ++side) {
    int segs = 0;
    for (const Run& r : sides[side].runs) segs += r.item.kind == kSegKind;
    (side ? pl.segs_d : pl.segs) = segs;
  }
  const int segs_p = pl.segs;
  pl.segs += pl.segs_d;
  out.cta.assign(G, ResCta{});
  int total = 0;
  for (int g = 0; g < G; ++g) {
    ResCta& C = out.cta[g];
    C.p0 = total;
    C.p1 = C.d0 = total += sides[0].cta[g].items;
    C.d1 = total += sides[1].cta[g].items;
    C.nlp = sides[0].cta[g].nlong;
    C.nld = sides[1].cta[g].nlong;
    C.rp = sides[0].cta[g].rows;
    C.rd = sides[1].cta[g].rows;
  }
  out.items.resize(total);
  struct Next {
    int item, ent, lrow, srow;  // long rows first
  };
  std::vector<Next> next(G);
  for (int side = 0; side < 2; ++side) {
    const Deal& D = sides[side];
    const bool near = !(pl.far >> side & 1);
    for (int g = 0; g < G; ++g) next[g] = Next{side ? out.cta[g].d0 : out.cta[g].p0, 0, 0, D.cta[g].nlong};
    for (int rank = 0; rank < (G > 1 ? 4 : 1); ++rank) {
      const int* owner = D.owner.data();
      for (const Run& r : D.runs) {
        if (G > 1 && rank_of(r.item) != rank) {
          owner += r.count;
          continue;
        }
        for (int i = 0; i < r.count; ++i) {
          Next& nx = next[*owner++];
          ResItem I = r.item;
          I.row0 += i * r.step;
          if (near && I.kind != kOwnKind) {
            I.ent = nx.ent;
            nx.ent += r.entries;
          }
          if (I.kind == kSegKind) {
            I.vec += side ? segs_p : 0;
          } else {
            int& row = I.kind > 0 ? nx.lrow : nx.srow;
            I.vec = G == 1 ? I.row0 : row;
            if (I.kind == kOwnKind) I.ent += side ? segs_p : 0;
            else if (I.kind > 0) I.len = row;
            row += I.nrows;
          }
          out.items[nx.item++] = I;
        }
      }
    }
  }
}

constexpr long long kResMaxEntries = 2 << 20;  // both matrix copies stay in L2 (129 MB) beside the vectors
constexpr long long kResSmem = 220 * 1024;  // what a CTA's rows may take, roughly (the exact limit is checked later)

// Lanes per short row of a side whose entries are read from global memory (four
// lanes read a sector of values at a time; with both sides there, two: the lane
// sums cost more than the sectors), and the entries up to which both may be: 64
// attempts of power-law LPs, FP64, against the two step kernels: 0.8M entries,
// one side, 2,150 -> 1,527 us (two lanes 1,575, eight 1,690); 1.0M, both sides,
// 2,439 -> 2,004 (four lanes 2,197); 1.4M, both sides, 2,608 -> 3,076, so not.
constexpr int kFarLanes = 4, kFarLanesBoth = 2;
// So both may be while a copy's entries take 12 MB: 1,048,576 in FP64, 1,572,864 in
// FP32 (1.5M, step kernels / both sides far: power law 37.0 / 33.1, random 32.5 / 30.1
// us per attempt).
constexpr long long kFarBothBytes = 12LL << 20;
// (FP64, 0.6M to 1.04M entries of five families, 27 LPs: 0.49 to 0.99 of the step kernels' time.)

// Shared memory of a CTA up to which one side may be read from L2 when there are
// more entries than that: above it the next size of the shared memory leaves 28 KB of
// the SM's 256 for the L1, which serves the gathers and what several lanes read
// of a sector.  us per attempt, step kernels / one side far: FP64 1.3M entries (187 KB
// of shared memory) 31.1 / 26.0, 1.4M (205 KB) 31.1 / 34.0, 1.5M (215 KB) 32.0 / 35.6;
// FP32 1.4M (191 KB) 31.9 / 25.5, 1.5M (205 KB) 32.8 / 35.6, linking rows 1.8M (189 KB)
// 36.6 / 29.6, 1.96M (203 KB) 38.5 / 40.9.  (Fewer entries: never slower.)
constexpr long long kFarSmemEntries = 1 << 20;
constexpr int kFarSmem = 193 * 1024;  // of 196 KB, with the kernel's static share and the system's

// Cycles of the FP64 pipe per attempt and CTA that a problem is split down to
// (600 to 2,000 measured the same within 2%: the chain of latencies between the
// phases is then the longer part, see resident.cu).
constexpr double kTargetCycles = 1000.0;

}  // namespace

int resident_long_rows(const BinTable& bt) {
  for (int b = 0; b < bt.nbins; ++b)
    if (bt.bin[b].width == kSell) return bt.bin[b].row_begin;
  return bt.nbins > 0 ? bt.bin[bt.nbins - 1].row_end : 0;
}

bool resident_possible(long long m, long long n, long long nnz, int esize) {  // the vectors at least
  return m > 0 && nnz > 0 && nnz <= kResMaxEntries && 10 * esize * (m + n) <= kResMaxCtas * kResSmem;
}

long long resident_bytes(long long m, long long n, long long nnz, int esize) {
  if (!resident_possible(m, n, nnz, esize)) return 0;
  const long long items = (m + n) / 32 + 2 * (kSellMaxLen + 2) + 2 * (nnz / (kSellMaxLen + 1)) + 2 * kResMaxCtas * kResThreads / 32 + (m + n) / 8 + 64 + 4 * (nnz / kResSeg + 1);
  auto r = [](long long b) { return (b + 255) / 256 * 256; };
  return r(items * (long long)sizeof(ResItem)) + r(kResMaxCtas * (long long)sizeof(ResCta)) + r((7 * kResMaxCtas + kResMaxCtas + 8 + 4 * (nnz / kResSeg + 1)) * 16) + r((n + 2 * m) * 2 * esize) + 256;
}

bool resident_build(const BinTable& binsA, const BinTable& binsAt, long long m, long long n, long long nnz,
                    const std::vector<int>& head_a, const std::vector<int>& head_at, int esize, int sms,
                    int smem_limit, ResHost& out) {
  double cost = 0.0;
  for (const auto& side : {side_items(binsAt, head_at, 1, true), side_items(binsA, head_a, 1, true)})
    for (const Run& r : side) {
      cost += r.count * r.cost;
      if (r.item.kind == kOwnKind && r.item.len > kResMaxSegs) return false;
    }
  Deal sides[2];  // of A^T, of A
  auto longest = [](const BinTable& bt, const std::vector<int>& head) {
    return bt.nbins == 0 ? 0 : bt.bin[0].width == kSell ? bt.bin[0].len : head[1] - head[0];
  };
  const int most = std::min(sms, kResMaxCtas);
  // everything in shared memory, or the entries of A read from L2 each time, or those of A^T, or both
  for (int far : {0, 2, 1, 3}) {
    const long long foot = (far == 3 ? 0 : far ? 1 : 2) * nnz * (esize + 4) + 9LL * esize * (m + n);
    int G = (int)std::min<double>(most, std::max(16.0 * cost / kTargetCycles, (double)foot / (double)kResSmem));
    if (G < 1 || (!far && foot + 48 * 1024 <= (long long)smem_limit)) G = 1;  // (retried with more CTAs if it does not fit after all)
    if (far) G = most;
    if (far == 3 && nnz * (esize + 4) > kFarBothBytes) continue;
    const int limit = far && nnz > kFarSmemEntries ? std::min(smem_limit, kFarSmem) : smem_limit;
    // what the CTAs' arrays hold at least (res_layout): no need to deal the rows out when that does not fit
    const long long least = (far == 3 ? 0 : far ? 1 : 2) * nnz * (esize + 4) + esize * (10 * n + 8 * m) + 5 * n + 6 * m +
                            9 * ((far & 1 ? n : 0) + (far & 2 ? m : 0)) + (long long)most * 4 * kResThreads * 8;
    if (least > (long long)most * limit) continue;
    const int far_lanes = far == 3 ? kFarLanesBoth : kFarLanes;
    for (;; G = std::min(most, G + std::max(1, G / 8))) {
      ResPlan& pl = out.plan;
      pl = ResPlan{};
      pl.G = G;
      out.step.longest[0] = longest(binsAt, head_at);
      out.step.longest[1] = longest(binsA, head_a);
      pl.longest = std::max(out.step.longest[0], out.step.longest[1]);
      pl.far = far;
      deal(side_items(binsAt, head_at,
                      far & 1 ? far_lanes : short_row_lanes((double)n / G, (double)nnz / (double)n), G > 1),
           G, sides[0]);
      deal(side_items(binsA, head_a,
                      far & 2 ? far_lanes : short_row_lanes((double)m / G, (double)nnz / (double)m), G > 1),
           G, sides[1]);
      for (int side = 0; side < 2; ++side) {
        const bool near = !(far >> side & 1);
        int& e = side ? pl.ed : pl.ep;
        int& r = side ? pl.rd : pl.rp;
        int& l = side ? pl.ld : pl.lp;
        for (const Deal::Cta& C : sides[side].cta) {
          e = std::max(e, near ? C.entries : 0);
          r = std::max(r, (C.rows + 1) / 2 * 2);
          l = std::max(l, C.nlong);
        }
        int items = 0;
        for (const Deal::Cta& C : sides[side].cta) items = std::max(items, C.items);
        out.step.warps[side] = std::min(kResWarps, std::max(4, items));
      }
      for (int g = 0; g < G; ++g) pl.it = std::max(pl.it, sides[0].cta[g].items + sides[1].cta[g].items);
      pl.smem = res_layout(pl, esize).total;
      if (pl.smem <= limit) {
        lay_out(sides, out);
        return true;
      }
      if (G == most) break;
    }
  }
  return false;
}

int SmTokens::wait_turn(std::unique_lock<std::mutex>& lk, int least, int most) {
  const unsigned long long me = next_++;
  cv_.wait(lk, [&] { return serving_ == me && free_ >= least; });
  const int got = std::min(free_, most);
  free_ -= got;
  ++serving_;
  cv_.notify_all();
  return got;
}

int SmTokens::acquire(int least, int most) {
  std::unique_lock<std::mutex> lk(mu_);
  return wait_turn(lk, least, most);
}

bool SmTokens::acquire_resident(int count) {
  std::unique_lock<std::mutex> lk(mu_);
  const bool turns = count * kFewSms <= sms_ || wanted_ <= 2 * sms_;
  if (!turns && wanted_ > sms_) return false;
  // (a round lasts for many periods: nobody waits for one)
  if ((next_ != serving_ || free_ < count) && (!turns || rounds_ > 0)) return false;
  wait_turn(lk, count, count);
  return true;
}

bool SmTokens::crowded() {
  std::lock_guard<std::mutex> lk(mu_);
  return wanted_ > kCrowd * sms_;
}

void SmTokens::release(int count) {
  {
    std::lock_guard<std::mutex> lk(mu_);
    free_ += count;
  }
  cv_.notify_all();
}

void SmTokens::announce(int count, bool round) {
  std::lock_guard<std::mutex> lk(mu_);
  wanted_ += count;
  rounds_ += round;
}

void SmTokens::withdraw(int count, bool round) {
  std::lock_guard<std::mutex> lk(mu_);
  wanted_ -= count;
  rounds_ -= round;
}

}  // namespace lpop
