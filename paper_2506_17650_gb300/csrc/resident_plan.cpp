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
  return longest / 32.0 + 20.0;
}

struct Costed {
  ResItem item;
  double cost;
  int entries;
};

// One side's items; short rows (those of the sliced bins) by `lanes` lanes each.
std::vector<Costed> side_items(const BinTable& bt, const std::vector<int>& head, int lanes) {
  std::vector<Costed> out;
  int b = 0;
  for (; b < bt.nbins && bt.bin[b].width != kSell; ++b) {
    const Bin& B = bt.bin[b];
    const int kind = B.width == 0 || B.width == kSegmented ? kResThreads : (B.width < 4 ? 4 : B.width);
    const int per = kind == kResThreads ? 1 : 32 / kind;
    for (int r = B.row_begin; r < B.row_end; r += per) {
      ResItem I{r, std::min(per, B.row_end - r), 0, kind, 0, 0};
      // (rows are longest first within a class)
      out.push_back(Costed{I, item_cost(I, head[r + 1] - head[r]), head[r + I.nrows] - head[r]});
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

// Longest-first assignment of one side's items to G CTAs; within a CTA the
// CTA-wide rows first, then the other long rows, then the slices, each most
// costly first.
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
  auto rank = [](const Costed& c) { return c.item.kind == kResThreads ? 0 : (c.item.kind > 0 ? 1 : 2); };
  for (auto& c : out)
    std::stable_sort(c.begin(), c.end(), [&](const Costed& a, const Costed& b) { return rank(a) < rank(b); });
  return out;
}

constexpr long long kResSmem = 220 * 1024;  // what a CTA's rows may take, roughly (the exact limit is checked later)

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

bool resident_possible(long long m, long long n, long long nnz, int esize) {
  return m > 0 && nnz > 0 && 2 * nnz * (esize + 4) + 9 * esize * (m + n) <= kResMaxCtas * kResSmem;
}

long long resident_bytes(long long m, long long n, long long nnz, int esize) {
  if (!resident_possible(m, n, nnz, esize)) return 0;
  const long long items = (m + n) / 32 + 2 * (kSellMaxLen + 2) + 2 * (nnz / (kSellMaxLen + 1)) + 2 * kResMaxCtas * kResThreads / 32 + 16;
  auto r = [](long long b) { return (b + 255) / 256 * 256; };
  return r(items * (long long)sizeof(ResItem)) + r(kResMaxCtas * (long long)sizeof(ResCta)) + r((7 * kResMaxCtas + kResMaxCtas + 8) * 16) + r((n + 2 * m) * 2 * esize) + 256;
}

bool resident_build(const BinTable& binsA, const BinTable& binsAt, long long m, long long n, long long nnz,
                    const std::vector<int>& head_a, const std::vector<int>& head_at, int esize, int sms,
                    int smem_limit, ResHost& out) {
  std::vector<Costed> P = side_items(binsAt, head_at, 1), D = side_items(binsA, head_a, 1);
  double cost = 0.0;
  for (const auto* side : {&P, &D})
    for (const Costed& c : *side) {
      cost += c.cost;
      if (c.item.kind > 0 && c.entries > kResMaxRow) return false;
    }
  int longest = 0;
  for (const auto& side : {std::make_pair(&binsAt, &head_at), std::make_pair(&binsA, &head_a)}) {
    const BinTable& bt = *side.first;
    if (bt.nbins == 0) continue;
    longest = std::max(longest, bt.bin[0].width == kSell ? bt.bin[0].len : (*side.second)[1] - (*side.second)[0]);
  }
  const long long foot = 2 * nnz * (esize + 4) + 9LL * esize * (m + n);
  const int most = std::min(sms, kResMaxCtas);
  int G = (int)std::min<double>(most, std::max(16.0 * cost / kTargetCycles, (double)foot / (double)kResSmem));
  if (G < 1 || foot + 48 * 1024 <= (long long)smem_limit) G = 1;  // (retried with more CTAs if it does not fit after all)
  for (;; G = std::min(most, G + std::max(1, G / 8))) {
    out.items.clear();
    out.cta.assign(G, ResCta{});
    ResPlan& pl = out.plan;
    pl = ResPlan{};
    pl.G = G;
    pl.longest = longest;
    P = side_items(binsAt, head_at, short_row_lanes((double)n / G, (double)nnz / (double)n));
    D = side_items(binsA, head_a, short_row_lanes((double)m / G, (double)nnz / (double)m));
    const auto pa = assign_items(P, G), da = assign_items(D, G);
    bool fits = true;
    for (int g = 0; g < G; ++g) {
      ResCta& C = out.cta[g];
      for (int side = 0; side < 2; ++side) {
        int ent = 0, vec = 0, nlong = 0, nwide = 0;
        (side ? C.d0 : C.p0) = (int)out.items.size();
        for (const Costed& c : side ? da[g] : pa[g]) {
          ResItem I = c.item;
          I.ent = ent;
          I.vec = G == 1 ? I.row0 : vec;
          if (I.kind > 0) {
            I.len = nlong;
            nlong += I.nrows;
            if (I.kind == kResThreads) ++nwide;
          }
          ent += c.entries;
          vec += I.nrows;
          out.items.push_back(I);
        }
        fits = fits && nwide <= kResWide;
        (side ? C.d1 : C.p1) = (int)out.items.size();
        (side ? C.nld : C.nlp) = nlong;
        (side ? C.rd : C.rp) = vec;
        int& e = side ? pl.ed : pl.ep;
        int& r = side ? pl.rd : pl.rp;
        int& l = side ? pl.ld : pl.lp;
        e = std::max(e, ent);
        r = std::max(r, (vec + 1) / 2 * 2);
        l = std::max(l, nlong);
      }
      pl.it = std::max(pl.it, C.p1 - C.p0 + C.d1 - C.d0);
    }
    pl.smem = res_layout(pl, esize).total;
    if (fits && pl.smem <= smem_limit) return true;
    if (G == most) return false;
  }
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
