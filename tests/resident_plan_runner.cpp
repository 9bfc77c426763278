// Reads a CSR matrix and prints the resident plan of its rows (binary, see
// test_resident_plan.py): argv = input file, output file, esize, sms, limit.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "host_layout.hpp"
#include "resident_plan.hpp"

using namespace lpop;

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  FILE* f = std::fopen(argv[1], "rb");
  int64_t h[3];
  if (!f || std::fread(h, 8, 3, f) != 3) return 2;
  std::vector<int64_t> rp(h[0] + 1);
  std::vector<int32_t> ci(h[2]);
  std::vector<double> v(h[2]);
  if (std::fread(rp.data(), 8, rp.size(), f) != rp.size() || std::fread(ci.data(), 4, ci.size(), f) != ci.size() ||
      std::fread(v.data(), 8, v.size(), f) != v.size())
    return 2;
  std::fclose(f);
  HostLayout lay;
  std::string err;
  if (build_layout((int)h[0], (int)h[1], h[2], rp.data(), ci.data(), v.data(), lay, err, 1) != 0) return 3;
  BinTable A = lay.binsA, At = lay.binsAt;
  segment_long_rows(A, lay.A_rp, 4096);
  segment_long_rows(At, lay.At_rp, 4096);
  const std::vector<int> ha(lay.A_rp.begin(), lay.A_rp.begin() + resident_long_rows(A) + 1);
  const std::vector<int> hat(lay.At_rp.begin(), lay.At_rp.begin() + resident_long_rows(At) + 1);
  const int esize = std::atoi(argv[3]), sms = std::atoi(argv[4]), limit = std::atoi(argv[5]);
  ResHost out;
  const bool ok = resident_build(A, At, lay.m, lay.n, lay.nnz, ha, hat, esize, sms, limit, out);
  f = std::fopen(argv[2], "wb");
  const ResLayout L = res_layout(out.plan, esize);
  const int64_t head[] = {ok, (int64_t)out.items.size(), (int64_t)out.cta.size(), out.plan.G, out.plan.ep, out.plan.ed,
                          out.plan.rp, out.plan.rd, out.plan.lp, out.plan.ld, out.plan.it, out.plan.smem, L.total,
                          resident_bytes(lay.m, lay.n, lay.nnz, esize), out.plan.far};
  std::fwrite(head, 8, sizeof(head) / 8, f);
  for (const ResItem& i : out.items) {
    const int64_t r[] = {i.row0, i.nrows, i.len, i.kind, i.ent, i.vec};
    std::fwrite(r, 8, 6, f);
  }
  for (const ResCta& c : out.cta) {
    const int64_t r[] = {c.p0, c.p1, c.d0, c.d1, c.nlp, c.nld, c.rp, c.rd};
    std::fwrite(r, 8, 8, f);
  }
  std::fwrite(lay.A_rp.data(), 4, lay.A_rp.size(), f);
  std::fwrite(lay.At_rp.data(), 4, lay.At_rp.size(), f);
  std::fclose(f);
  return 0;
}
