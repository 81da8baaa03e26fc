// Checks the plan of the cluster-resident solves on the CPU: every column,
// slot and offset in range, every halo slot filled by exactly one send, and
// the products of all operators of a hierarchy, formed block by block from the
// images and the sent halos, equal to the plain CSR products.  Usage:
// resident_plan_check nx ny nz coarse_max (nz = 0: triangles); prints "ok".
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <string>
#include <vector>

#include "../paper_2510_27447_gb300/csrc/resident.h"

using namespace bd;

static void require(bool ok, const char* what) {
  if (ok) return;
  std::printf("failed: %s\n", what);
  std::exit(1);
}

using Vec = std::vector<double>;
using Words = std::function<const uint32_t*(int)>;
using Count = std::function<int(int)>;

// block copies of x over a space of q entries per block, halos filled by the sends
static std::vector<Vec> spread(const Vec& x, int C, int q, int slots, const Count& nown, const Count& nsend,
                               const Words& word, const Count& nhalo) {
  std::vector<Vec> v(C, Vec(slots, 0.0));
  for (size_t i = 0; i < x.size(); ++i) v[i / q][i % q] = x[i];
  std::vector<std::vector<int>> hit(C, std::vector<int>(slots, 0));
  for (int c = 0; c < C; ++c)
    for (int k = 0; k < nsend(c); ++k) {
      const uint32_t w = word(c)[k];
      const int from = int(w >> 20), to = int(w >> 16 & 15u), slot = int(w & 0xffffu);
      require(to < C && to != c && slot >= q && slot < slots && from < nown(c), "send in range");
      v[to][slot] = v[c][from];
      ++hit[to][slot];
    }
  for (int c = 0; c < C; ++c) {
    int n = 0;
    for (int h : hit[c]) {
      require(h <= 1, "one send per halo slot");
      n += h;
    }
    require(n == nhalo(c), "expected halo bytes");
  }
  return v;
}

static void same(const Vec& a, const Vec& b) {
  double big = 0.0, off = 0.0;
  for (size_t i = 0; i < a.size(); ++i) {
    big = std::max(big, std::fabs(b[i]));
    off = std::max(off, std::fabs(a[i] - b[i]));
  }
  require(off <= 1e-13 * big + 1e-300, "product");   // a few additions reordered
}

static Vec product(const HCsr& M, const Vec& x) {
  Vec y(M.n, 0.0);
  for (int64_t i = 0; i < M.n; ++i)
    for (int64_t p = M.rp[i]; p < M.rp[i + 1]; ++p) y[i] += M.v[p] * x[M.ci[p]];
  return y;
}

static Vec random_vec(int64_t n) {
  Vec x(n);
  for (double& t : x) t = drand48() - 0.5;
  return x;
}

static void mesh(int nx, int ny, int nz, Vec* xyz, std::vector<int32_t>* el) {
  auto id = [&](int i, int j, int k) { return (k * ny + j) * nx + i; };
  for (int k = 0; k < std::max(nz, 1); ++k)
    for (int j = 0; j < ny; ++j)
      for (int i = 0; i < nx; ++i) {
        xyz->push_back(0.01 * i);
        xyz->push_back(0.011 * j);
        if (nz) xyz->push_back(0.012 * k);
      }
  const int step[6][2][3] = {{{1, 0, 0}, {1, 1, 0}}, {{1, 0, 0}, {1, 0, 1}}, {{0, 1, 0}, {1, 1, 0}},
                             {{0, 1, 0}, {0, 1, 1}}, {{0, 0, 1}, {1, 0, 1}}, {{0, 0, 1}, {0, 1, 1}}};
  if (!nz) {
    for (int j = 0; j + 1 < ny; ++j)
      for (int i = 0; i + 1 < nx; ++i)
        for (int v : {id(i, j, 0), id(i + 1, j, 0), id(i + 1, j + 1, 0), id(i, j, 0), id(i + 1, j + 1, 0), id(i, j + 1, 0)})
          el->push_back(v);
    return;
  }
  for (int k = 0; k + 1 < nz; ++k)
    for (int j = 0; j + 1 < ny; ++j)
      for (int i = 0; i + 1 < nx; ++i)
        for (auto& s : step) {
          el->push_back(id(i, j, k));
          for (auto& t : s) el->push_back(id(i + t[0], j + t[1], k + t[2]));
          el->push_back(id(i + 1, j + 1, k + 1));
        }
}

static void check(const HostOps& H, const HCsr& A, const AmgHost& AH, int C) {
  const int64_t N = H.n, nsl = (N + 31) / 32;
  std::vector<int64_t> sptr(nsl);
  std::vector<int> sw(nsl);
  int64_t len = 0;
  for (int64_t s = 0; s < nsl; ++s) {
    for (int64_t i = 32 * s; i < std::min<int64_t>(N, 32 * s + 32); ++i)
      sw[s] = std::max(sw[s], H.rowptr[i + 1] - H.rowptr[i]);
    sptr[s] = len;
    len += 32 * sw[s];
  }
  Vec val(len, 0.0);
  for (int64_t i = 0; i < N; ++i)
    for (int k = 0; k < H.rowptr[i + 1] - H.rowptr[i]; ++k) val[sptr[i / 32] + i % 32 + 32 * k] = A.v[H.rowptr[i] + k];
  ResPlan P;
  if (!res_plan_build(C, N, H.rowptr.data(), H.col.data(), sptr.data(), sw.data(), AH.lev.empty() ? nullptr : &AH, true,
                      true, &P))
    return;   // too large for this cluster
  const ResShape& S = P.s;
  require(S.block <= kResBlock && S.block >= 128 && S.block % 32 == 0 && S.block * S.rpt >= S.q0, "rows per thread");
  auto own0 = [&](int c) { return int(std::max<int64_t>(0, std::min<int64_t>(N - int64_t(c) * S.q0, S.q0))); };
  auto img0 = [&](int c) { return P.img0.data() + size_t(c) * S.img0; };
  auto spread0 = [&](const Vec& x) {
    return spread(x, C, S.q0, S.slots0, own0, [&](int c) { return P.cta[c].npush; },
                  [&](int c) { return reinterpret_cast<const uint32_t*>(img0(c) + S.off_push); },
                  [&](int c) { return P.cta[c].nhalo; });
  };
  {
    const Vec x = random_vec(N);
    const std::vector<Vec> v = spread0(x);
    Vec y(N, 0.0);
    for (int c = 0; c < C; ++c) {
      const ResCta& t = P.cta[c];
      require(t.nent <= S.nent_max && t.ent0 + t.nent <= len && t.ent0 % 32 == 0, "entry range");
      const uint32_t* sl = reinterpret_cast<const uint32_t*>(img0(c));
      const uint16_t* lc = reinterpret_cast<const uint16_t*>(img0(c) + S.off_lcol);
      for (int r = 0; r < own0(c); ++r) {
        require(r / 32 < t.ns, "slice");
        const int at = int(sl[r / 32] >> 12) * 32 + r % 32;
        for (int k = 0; k < int(sl[r / 32] & 4095u); ++k) {
          require(at + 32 * k < t.nent && lc[at + 32 * k] < S.slots0, "column slot");
          y[int64_t(c) * S.q0 + r] += val[t.ent0 + at + 32 * k] * v[c][lc[at + 32 * k]];
        }
      }
    }
    same(y, product(A, x));
  }
  if (S.nlev == 0) return;
  auto hdr = [&](int c) { return reinterpret_cast<const ResAmgHdr*>(P.imgA64.data() + size_t(c) * S.imgA[1]); };
  auto base = [&](int c) { return P.imgA64.data() + size_t(c) * S.imgA[1]; };
  // operator M with rows in space rs and columns in space cs (nlev: the coarsest)
  auto op = [&](const HCsr& M, int rs, int cs, const std::function<const ResOp&(const ResAmgHdr&)>& pick) {
    const Vec x = random_vec(M.m);
    const int slots = cs == S.nlev ? S.ldc : cs == 0 ? S.slots0 : S.slotsL[cs];
    std::vector<Vec> v;
    if (cs == S.nlev) {
      v.assign(C, Vec(slots, 0.0));
      for (Vec& t : v) std::copy(x.begin(), x.end(), t.begin());
    } else if (cs == 0) {
      v = spread0(x);
    } else {
      v = spread(x, C, S.qL[cs], slots, [&](int c) { return hdr(c)->L[cs].nown; },
                 [&](int c) { return hdr(c)->L[cs].npush; },
                 [&](int c) { return reinterpret_cast<const uint32_t*>(base(c) + hdr(c)->L[cs].off_push); },
                 [&](int c) { return hdr(c)->L[cs].nhalo; });
    }
    Vec y(M.n, 0.0);
    std::vector<int> seen(M.n, 0);
    for (int c = 0; c < C; ++c) {
      const ResOp& o = pick(*hdr(c));
      const int64_t first = rs == S.nlev ? hdr(c)->c0 : int64_t(c) * (rs == 0 ? S.q0 : S.qL[rs]);
      const uint32_t* sl = reinterpret_cast<const uint32_t*>(base(c) + o.off_slice);
      const uint16_t* col = reinterpret_cast<const uint16_t*>(base(c) + o.off_col);
      const double* va = reinterpret_cast<const double*>(base(c) + o.off_val);
      for (int s = 0; s < o.ns; ++s)
        for (int lane = 0; lane < 32; ++lane) {
          const int row = s * (32 / o.g) + lane / o.g;
          double sum = 0.0;
          for (int k = 0; k < int(sl[s] & 4095u); ++k) {
            const int at = int(sl[s] >> 12) * 32 + 32 * k + lane;
            require(o.off_col + 2 * at + 2 <= S.imgA[1] && o.off_val + 8 * at + 8 <= S.imgA[1] && col[at] < slots,
                    "image offset");
            sum += va[at] * v[c][col[at]];
          }
          if (row >= o.nr) continue;
          require(first + row < M.n, "row");
          y[first + row] += sum;
          seen[first + row] += lane % o.g == 0;
        }
    }
    for (int n : seen) require(n == 1, "every row once");
    same(y, product(M, x));
  };
  for (int c = 0; c < C; ++c) {
    const ResAmgHdr& h = *hdr(c);
    require(h.nlev == S.nlev && h.c0 + h.ncown <= S.nc, "coarse range");
    require(h.ncown == 0 || (h.c0 % 4 == 0 && h.c0 + (h.ncown + 3) / 4 * 4 <= S.ldc), "coarse rows in fours");
  }
  for (int l = 0; l < S.nlev; ++l) {
    if (l > 0) op(AH.lev[l].A, l, l, [l](const ResAmgHdr& h) -> const ResOp& { return h.L[l].A; });
    op(AH.lev[l].P, l, l + 1, [l](const ResAmgHdr& h) -> const ResOp& { return h.L[l].P; });
    op(AH.lev[l].R, l + 1, l, [l](const ResAmgHdr& h) -> const ResOp& { return h.L[l].R; });
  }
}

int main(int argc, char** argv) {
  if (argc != 5) return 2;
  Vec xyz;
  std::vector<int32_t> el;
  const int nz = std::atoi(argv[3]);
  mesh(std::atoi(argv[1]), std::atoi(argv[2]), nz, &xyz, &el);
  bd_mesh_t m{};
  m.dim = nz ? 3 : 2;
  m.n_nodes = int64_t(xyz.size()) / m.dim;
  m.n_elems = int64_t(el.size()) / (m.dim + 1);
  m.xyz = xyz.data();
  m.elems = el.data();
  const bd_cond_t cond{3.0, 0.31, 2.0, 1.35, 2000.0, 1.0, 20.0};
  HostOps H;
  std::string err;
  require(assemble_host(&m, &cond, &H, &err) == BD_OK, "assembly");
  HCsr A;
  A.n = A.m = H.n;
  A.rp.assign(H.rowptr.begin(), H.rowptr.end());
  A.ci = H.col;
  A.v = H.Aie;
  AmgHost AH;
  AmgParams prm;
  prm.coarse_max = std::atoi(argv[4]);
  require(amg_build(A, prm, &AH, &err) == BD_OK, "hierarchy");
  for (int C : {16, 8, 4, 2, 1}) check(H, A, AH, C);
  std::printf("ok\n");
  return 0;
}
