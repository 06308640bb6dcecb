"""Which rows of one launch of adjoint steps read what other rows of it write, on the CPU: the plan that the library makes for every
such launch (csrc/adj_sweep.h) against a row by row enumeration.  A C-step behind F-steps replaces what the next interval started
from; the launch has to say so, and the tiles that the kernel then waits for have to hold those rows.  And the sizes at which such
a launch is taken at all."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <stdio.h>
#include <set>
#include <vector>
#include "adj_sweep.h"
using namespace mg;
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
static const int H = 4;
struct Level { int B, cf, nki, tail; std::vector<float> U, G, V; };
// kinds as in the multigrid cycle: 1 .. cf - 1 an F-step to that slot, cf a C-step, cf + 1 the step that evaluates v
static AdjSweepArgs launch(Level& q, const std::vector<int>& kinds, int kz) {
  const i64 bh = (i64)q.B * H;
  AdjSweepArgs a{};
  a.B = q.B; a.H = H; a.n = (int)kinds.size();
  a.lin = q.U.data() + (kinds[0] < q.cf ? kinds[0] - 1 : q.cf - 1) * bh; a.lin_ks = q.cf * bh;
  for (int i = 0; i < a.n; ++i) {
    const int kd = kinds[i], nk = q.nki + (kd < q.cf && kd <= q.tail ? 1 : 0);
    AdjSweepStep& t = a.st[i];
    t.out = kd > q.cf ? q.V.data() + bh : q.U.data() + kd * bh; t.out_ks = kd > q.cf ? bh : q.cf * bh;
    t.g = q.G.data() + (kd > q.cf ? q.cf : kd) * bh; t.g_ks = q.cf * bh;
    t.nk = nk < kz ? nk : kz; t.ahead = -1;
  }
  return a;
}
// does a row of one interval write what a row of another one reads, or writes as well?
static bool meets(const AdjSweepArgs& a) {
  const i64 len = (i64)a.B * a.H;
  auto hit = [&](const float* p, const float* q) { return p < q + len && q < p + len; };
  for (int i = 0; i < a.n; ++i)
    for (int k = 0; k < a.st[i].nk; ++k) {
      const float* w = a.st[i].out + k * a.st[i].out_ks;
      for (int k2 = 0; k2 < a.st[0].nk; ++k2) {
        if (k2 == k) continue;
        if (hit(w, a.lin + k2 * a.lin_ks)) return true;
        for (int j = 0; j < a.n; ++j)
          if (k2 < a.st[j].nk && (hit(w, a.st[j].out + k2 * a.st[j].out_ks) || hit(w, a.st[j].g + k2 * a.st[j].g_ks))) return true;
      }
    }
  return false;
}
int main() {
  int ordered = 0, plain = 0, refused = 0;
  for (int B : {1, 8, 24, 33, 100, 128, 200})
    for (int cf : {2, 3, 4, 8})
      for (int nki : {1, 2, 5, 17})
        for (int tail = 0; tail < cf; tail += cf > 4 ? 3 : 1) {
          Level q{B, cf, nki, tail, {}, {}, {}};
          const size_t n = (size_t)(nki * cf + tail + 1) * B * H;
          q.U.resize(n); q.G.resize(n); q.V.resize((size_t)(nki + 1) * B * H);
          for (int kz : {1, 3, 1000}) {
            std::vector<int> f, fc, fv, cfs, fcf;
            for (int s = 1; s < cf; ++s) f.push_back(s);
            fc = fv = cfs = fcf = f;
            fc.push_back(cf); fv.push_back(cf + 1); cfs.insert(cfs.begin(), cf); fcf.push_back(cf); fcf.insert(fcf.end(), f.begin(), f.end());
            for (const auto& kinds : {f, fc, fv, cfs, fcf}) {
              if (kinds.size() > (size_t)kMaxAdjSweepSteps) continue;
              AdjSweepArgs a = launch(q, kinds, kz);
              const bool conflict = meets(a), ok = plan_adj_sweep(&a);
              const int M = a.st[a.n - 1].nk * B;
              if (kinds == f || kinds == fv) {      // nothing meets, nothing is waited for
                CHECK(ok && !conflict);
                for (int i = 0; i < a.n; ++i) CHECK(a.st[i].ahead == 0);
                ++plain;
              } else if (kinds == fc) {
                if (cf == 2 && a.n == 1) continue;
                CHECK(ok);
                for (int i = 0; i + 1 < a.n; ++i) CHECK(a.st[i].ahead == 0);
                if (conflict) CHECK(a.st[a.n - 1].ahead == B);
                if (a.st[a.n - 1].ahead == 0) continue;
                ++ordered;
                for (int nr : {64, 128})
                  for (int r0 = 0; r0 < M + 8; r0 += 4) {
                    int lo, hi;
                    tiles_ahead(r0, M, B, nr, &lo, &hi);
                    std::set<int> need;
                    for (int r = r0; r < r0 + 4 && r < M; ++r)
                      for (int r2 = 0; r2 < a.st[0].nk * B; ++r2) {      // the row that starts from what r replaces
                        const float* w = a.st[a.n - 1].out + (r / B) * a.st[a.n - 1].out_ks + (r % B) * H;
                        if (w == a.lin + (r2 / B) * a.lin_ks + (r2 % B) * H) need.insert(r2 / nr);
                      }
                    for (int t : need) CHECK(lo <= t && t <= hi);
                    CHECK(hi - lo < 32);      // (a lane for each)
                    if (r0 >= M) CHECK(hi < lo);
                  }
              } else if (conflict) {
                CHECK(!ok);      // steps behind a C-step start from what other rows left
                ++refused;
              }
            }
          }
          // results on other rows' sources, or on one another
          if (cf > 2 && nki > 2) {
            AdjSweepArgs a = launch(q, {1, 2}, 1000);
            a.st[1].g = q.U.data() + ((i64)cf + 1) * B * H;
            CHECK(!plan_adj_sweep(&a));
            a = launch(q, {1, 2}, 1000);
            a.st[1].out = a.st[0].out + a.st[0].out_ks;
            CHECK(!plan_adj_sweep(&a));
          }
        }
  CHECK(ordered > 100 && plain > 100 && refused > 100);
  // rounds of row tiles against waves of single steps, on both sides of every jump (33 clusters of four, 74 of two)
  const int rule[][3] = {{1024, 64, 8}, {1024, 65, 0}, {960, 64, 0}, {1024, 511, 0}, {1024, 512, 4}, {1024, 1024, 4}, {1024, 1025, 0}, {1024, 1153, 4},
                         {1024, 2048, 4}, {1024, 2049, 0}, {640, 512, 0}, {640, 896, 0}, {640, 897, 4}, {640, 1537, 0}, {704, 640, 4}, {704, 641, 0},
                         {576, 1024, 0}, {576, 1025, 4}, {576, 1537, 0}, {512, 1535, 0}, {512, 1536, 2}, {512, 4096, 2}, {512, 4097, 0}, {448, 2304, 2},
                         {448, 2305, 0}, {448, 2688, 0}, {448, 2689, 2}, {448, 2816, 2}, {320, 1792, 0}, {320, 1793, 2}, {320, 3072, 2}, {320, 3073, 0}, {256, 2048, 0},
                         {1088, 1024, 0}};
  for (const auto& r : rule) CHECK(adj_sweep_split(r[0], r[1], 33, 74) == r[2]);
  for (int M = 65; M <= 4096; ++M) CHECK(adj_sweep_split(1024, M, 7, 74) == 0 && adj_sweep_split(512, M, 33, 3) == 0);      // (no room for one group)
  printf("ok\n");
  return 0;
}
"""


def test_rows_that_meet_are_ordered_or_refused(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2203_04738_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
