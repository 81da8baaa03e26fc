// A hierarchy cut back to a larger coarsest level is the one built with that
// level.  Usage: amg_truncate_check n fine_max coarse_max (sheet of n^2 nodes);
// prints "ok" and the smoothed levels of the three.
#include <cstdio>
#include <cstdlib>

#include "../paper_2510_27447_gb300/csrc/bd_internal.h"

using namespace bd;

static bool same(const HCsr& a, const HCsr& b) {
  return a.n == b.n && a.m == b.m && a.rp == b.rp && a.ci == b.ci && a.v == b.v;
}

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  const int n = std::atoi(argv[1]);
  std::vector<double> xyz;
  std::vector<int32_t> el;
  for (int j = 0; j < n; ++j)
    for (int i = 0; i < n; ++i) {
      xyz.push_back(0.01 * i);
      xyz.push_back(0.011 * j);
    }
  for (int j = 0; j + 1 < n; ++j)
    for (int i = 0; i + 1 < n; ++i)
      for (int v : {0, 1, n + 1, 0, n + 1, n}) el.push_back(j * n + i + v);
  bd_mesh_t m{};
  m.dim = 2;
  m.n_nodes = int64_t(n) * n;
  m.n_elems = int64_t(el.size()) / 3;
  m.xyz = xyz.data();
  m.elems = el.data();
  const bd_cond_t cond{3.0, 0.31, 2.0, 1.35, 2000.0, 1.0, 20.0};
  HostOps H;
  std::string err;
  if (assemble_host(&m, &cond, &H, &err) != BD_OK) return 1;
  HCsr A;
  A.n = A.m = H.n;
  A.rp.assign(H.rowptr.begin(), H.rowptr.end());
  A.ci = H.col;
  A.v = H.Aie;
  AmgHost a, b;
  AmgParams prm;
  prm.coarse_max = std::atoi(argv[2]);
  if (amg_build(A, prm, &a, &err) != BD_OK) return 1;
  const size_t deep = a.lev.size();
  prm.coarse_max = std::atoi(argv[3]);
  if (amg_build(A, prm, &b, &err) != BD_OK || amg_truncate(prm.coarse_max, &a, &err) != BD_OK) return 1;
  bool ok = a.lev.size() == b.lev.size() && a.nc == b.nc && a.cinv == b.cinv;
  for (size_t l = 0; ok && l < a.lev.size(); ++l)
    ok = same(a.lev[l].A, b.lev[l].A) && same(a.lev[l].P, b.lev[l].P) && same(a.lev[l].R, b.lev[l].R) &&
         a.lev[l].invdiag == b.lev[l].invdiag && a.lev[l].omega == b.lev[l].omega;
  std::printf("%s %zu %zu %zu\n", ok ? "ok" : "differs", deep, a.lev.size(), b.lev.size());
  return 0;
}
