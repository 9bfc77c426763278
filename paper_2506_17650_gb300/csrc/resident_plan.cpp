#include "resident_plan.hpp"

#include <algorithm>
#include <queue>

namespace lpop {

namespace {

// FP64-pipe cost of an item, in warp instructions: a slice's FMAs and epilogue, a group of long rows' FMAs,
// shuffle adds and (one lane per row, so shared by 32 rows) epilogue.
double item_cost(const ResItem& I, int longest) {
  if (I.kind == 0) return I.len + 9.0;
  if (I.kind <= 32) return (longest + I.kind - 1) / I.kind + 3.0 + 10.0 * I.nrows / 32.0;
  return I.kind == kSegKind ? (I.nrows + 31) / 32 + 6.0 : 7.0;
}

struct Costed {
  ResItem item;
  double cost;
  int entries;
};

// One side's items; short rows (those of the sliced bins) by `lanes` lanes each,
// rows of more than kResSeg entries cut into segments if `cut`.
std::vector<Costed> side_items(const BinTable& bt, const std::vector<int>& head, int lanes, bool cut) {
  std::vector<Costed> out;
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
          out.push_back(Costed{I, item_cost(I, 0), size});
        }
        ResItem I{r, 1, n, kOwnKind, slot, 0};
        out.push_back(Costed{I, item_cost(I, 0), 0});
        slot += n;
        ++r;
        continue;
      }
      const int rows = std::min(32 / kind, B.row_end - r);
      ResItem I{r, rows, 0, kind, 0, 0};
      // (rows are longest first within a class)
      out.push_back(Costed{I, item_cost(I, len), head[r + rows] - head[r]});
      r += rows;
    }
  }
  const int end = bt.nbins > 0 ? bt.bin[bt.nbins - 1].row_end : 0;
  const int per = 32 / lanes;
  for (int r = b < bt.nbins ? bt.bin[b].row_begin : end; r < end; r += per) {
    while (bt.bin[b].row_end <= r) ++b;  // bins hold one exact length each, longest first
    const int rows = std::min(per, end - r), longest = bt.bin[b].len;
    if (lanes == 1) {
      ResItem I{r, rows, longest, 0, 0, 0};
      out.push_back(Costed{I, item_cost(I, longest), 32 * longest});
    } else {
      int entries = 0;
      for (int k = r, q = b; k < r + rows; ++k) {
        while (bt.bin[q].row_end <= k) ++q;
        entries += bt.bin[q].len;
      }
      ResItem I{r, rows, 0, lanes, 0, 0};
      out.push_back(Costed{I, item_cost(I, longest), entries});
    }
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

// Longest-first assignment of one side's items to G CTAs; within a CTA each
// kind most costly first.
std::vector<std::vector<Costed>> assign_items(const std::vector<Costed>& items, int G) {
  if (G == 1) return {items};  // in bin order: a local row is the global one
  std::vector<int> order(items.size());
  for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return items[a].cost > items[b].cost; });
  std::vector<std::vector<Costed>> out(G);
  using Load = std::pair<double, int>;
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> q;
  for (int g = 0; g < G; ++g) q.push({0.0, g});
  for (int i : order) {
    Load l = q.top();
    q.pop();
    out[l.second].push_back(items[i]);
    l.first += items[i].cost;
    q.push(l);
  }
  // segments first (others wait for them), the rows that wait last
  auto rank = [](const Costed& c) {
    return c.item.kind == kSegKind ? 0 : c.item.kind == kOwnKind ? 3 : c.item.kind > 0 ? 1 : 2;
  };
  for (auto& c : out)
    std::stable_sort(c.begin(), c.end(), [&](const Costed& a, const Costed& b) { return rank(a) < rank(b); });
  return out;
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
constexpr long long kFarBothMax = 1 << 20;

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
  std::vector<Costed> P = side_items(binsAt, head_at, 1, true), D = side_items(binsA, head_a, 1, true);
  double cost = 0.0;
  for (const auto* side : {&P, &D})
    for (const Costed& c : *side) {
      cost += c.cost;
      if (c.item.kind == kOwnKind && c.item.len > kResMaxSegs) return false;
    }
  int longest = 0;
  for (const auto& side : {std::make_pair(&binsAt, &head_at), std::make_pair(&binsA, &head_a)}) {
    const BinTable& bt = *side.first;
    if (bt.nbins == 0) continue;
    longest = std::max(longest, bt.bin[0].width == kSell ? bt.bin[0].len : (*side.second)[1] - (*side.second)[0]);
  }
  const int most = std::min(sms, kResMaxCtas);
  // everything in shared memory, or the entries of A read from L2 each time, or those of A^T, or both
  for (int far : {0, 2, 1, 3}) {
    const long long foot = (far == 3 ? 0 : far ? 1 : 2) * nnz * (esize + 4) + 9LL * esize * (m + n);
    int G = (int)std::min<double>(most, std::max(16.0 * cost / kTargetCycles, (double)foot / (double)kResSmem));
    if (G < 1 || (!far && foot + 48 * 1024 <= (long long)smem_limit)) G = 1;  // (retried with more CTAs if it does not fit after all)
    if (far) G = most;
    if (foot > (long long)most * smem_limit || (far == 3 && nnz > kFarBothMax)) continue;  // (no need to deal the rows out)
    const int far_lanes = far == 3 ? kFarLanesBoth : kFarLanes;
    for (;; G = std::min(most, G + std::max(1, G / 8))) {
      out.items.clear();
      out.cta.assign(G, ResCta{});
      ResPlan& pl = out.plan;
      pl = ResPlan{};
      pl.G = G;
      pl.longest = longest;
      pl.far = far;
      P = side_items(binsAt, head_at, far & 1 ? far_lanes : short_row_lanes((double)n / G, (double)nnz / (double)n),
                     G > 1);
      D = side_items(binsA, head_a, far & 2 ? far_lanes : short_row_lanes((double)m / G, (double)nnz / (double)m),
                     G > 1);
      int segs_p = 0, segs_d = 0;
      for (const Costed& c : P) segs_p += c.item.kind == kSegKind;
      for (const Costed& c : D) segs_d += c.item.kind == kSegKind;
      pl.segs = segs_p + segs_d;
      pl.segs_d = segs_d;
      const auto pa = assign_items(P, G), da = assign_items(D, G);
      for (int g = 0; g < G; ++g) {
        ResCta& C = out.cta[g];
        for (int side = 0; side < 2; ++side) {
          const bool near = !(far >> side & 1);
          const std::vector<Costed>& mine = side ? da[g] : pa[g];
          int ent = 0, nlong = 0;
          for (const Costed& c : mine)
            if (c.item.kind > 0 && c.item.kind != kSegKind) nlong += c.item.nrows;
          int lrow = 0, srow = nlong;  // long rows first
          (side ? C.d0 : C.p0) = (int)out.items.size();
          for (const Costed& c : mine) {
            ResItem I = c.item;
            if (near && I.kind != kOwnKind) {
              I.ent = ent;
              ent += c.entries;
            }
            if (I.kind == kSegKind) {
              I.vec += side ? segs_p : 0;
            } else {
              int& next = I.kind > 0 ? lrow : srow;
              I.vec = G == 1 ? I.row0 : next;
              if (I.kind == kOwnKind) I.ent += side ? segs_p : 0;
              else if (I.kind > 0) I.len = next;
              next += I.nrows;
            }
            out.items.push_back(I);
          }
          (side ? C.d1 : C.p1) = (int)out.items.size();
          (side ? C.nld : C.nlp) = nlong;
          (side ? C.rd : C.rp) = srow;
          int& e = side ? pl.ed : pl.ep;
          int& r = side ? pl.rd : pl.rp;
          int& l = side ? pl.ld : pl.lp;
          e = std::max(e, ent);
          r = std::max(r, (srow + 1) / 2 * 2);
          l = std::max(l, nlong);
        }
        pl.it = std::max(pl.it, C.p1 - C.p0 + C.d1 - C.d0);
      }
      pl.smem = res_layout(pl, esize).total;
      if (pl.smem <= smem_limit) return true;
      if (G == most) break;
    }
  }
  return false;
}


int SmTokens::acquire(int least, int most) {
  std::unique_lock<std::mutex> lk(mu_);
  const unsigned long long me = next_++;
  cv_.wait(lk, [&] { return serving_ == me && free_ >= least; });
  const int got = std::min(free_, most);
  free_ -= got;
  ++serving_;
  cv_.notify_all();
  return got;
}

void SmTokens::release(int count) {
  {
    std::lock_guard<std::mutex> lk(mu_);
    free_ += count;
  }
  cv_.notify_all();
}

}  // namespace lpop
