// resident_plan.cpp -- host plan of the cluster-resident solves: which block
// of the cluster owns which rows of every level, the halo slots it needs, the
// push lists that fill other blocks' halos, and the shared-memory images.
#include <algorithm>
#include <cstring>

#include "resident.h"

namespace bd {

namespace {

struct Space {                        // one level's vector space, split over the blocks
  int64_t n = 0;
  int q = 0;                          // owned entries per block (the last ones may own fewer)
  std::vector<std::vector<int32_t>> halo;   // per block: sorted remote entries it reads
  int slots = 0;                      // largest owned + halo count
  int owner(int64_t i) const { return int(i / q); }
  int first(int c) const { return int(std::min<int64_t>(n, int64_t(c) * q)); }
  int count(int c) const { return int(std::min<int64_t>(n, int64_t(c + 1) * q)) - first(c); }
  int slot(int c, int64_t i) const {
    if (owner(i) == c) return int(i - first(c));
    const auto& h = halo[c];
    return q + int(std::lower_bound(h.begin(), h.end(), int32_t(i)) - h.begin());
  }
};

void need(Space& sp, int c, int64_t i) {
  if (sp.owner(i) != c) sp.halo[c].push_back(int32_t(i));
}

struct Image {
  std::vector<unsigned char> b;
  size_t put(const void* p, size_t bytes) {
    const size_t at = (b.size() + 15) & ~size_t(15);
    b.resize(at + bytes);
    if (bytes) std::memcpy(b.data() + at, p, bytes);
    return at;
  }
};

// sends of block c: words source slot << 20 | block << 16 | destination slot,
// by destination block, then slot (neighbouring words go to neighbouring slots)
std::vector<uint32_t> push_words(const Space& sp, int c) {
  std::vector<uint32_t> w;
  for (int d = 0; d < int(sp.halo.size()); ++d) {
    if (d == c) continue;
    const auto& h = sp.halo[d];
    for (auto it = std::lower_bound(h.begin(), h.end(), int32_t(sp.first(c)));
         it != h.end() && *it < sp.first(c) + sp.count(c); ++it)
      w.push_back(uint32_t(*it - sp.first(c)) << 20 | uint32_t(d) << 16 | uint32_t(sp.q + (it - h.begin())));
  }
  return w;
}

// rows [first, first + nr) of M with columns through colslot, g lanes a row
template <class T, class F>
ResOp put_op(Image& im, const HCsr& M, int64_t first, int nr, int g, F&& colslot) {
  ResOp o{};
  o.nr = nr;
  o.g = g;
  const int rps = 32 / g;
  o.ns = (nr + rps - 1) / rps;
  std::vector<uint32_t> sl(o.ns);
  std::vector<uint16_t> col;
  std::vector<T> val;
  for (int s = 0; s < o.ns; ++s) {
    int steps = 0;
    for (int r = s * rps; r < std::min(nr, (s + 1) * rps); ++r) {
      const int len = int(M.rp[first + r + 1] - M.rp[first + r]);
      steps = std::max(steps, (len + g - 1) / g);
    }
    const size_t base = col.size();
    sl[s] = uint32_t(base / 32) << 12 | uint32_t(steps);
    col.resize(base + 32 * size_t(steps), 0);
    val.resize(base + 32 * size_t(steps), T(0));
    for (int r = s * rps; r < std::min(nr, (s + 1) * rps); ++r)
      for (int64_t p = M.rp[first + r], k = 0; p < M.rp[first + r + 1]; ++p, ++k) {
        const size_t at = base + 32 * size_t(k / g) + size_t(g * (r - s * rps) + k % g);
        col[at] = uint16_t(colslot(M.ci[p]));
        val[at] = T(M.v[p]);
      }
  }
  o.off_slice = int(im.put(sl.data(), sl.size() * 4));
  o.off_col = int(im.put(col.data(), col.size() * 2));
  o.off_val = int(im.put(val.data(), val.size() * sizeof(T)));
  return o;
}

// lanes per row: spread few rows over the block's threads, at least about
// four entries a lane
int lanes(const HCsr& M, int rows, int block) {
  const double mean = M.n ? double(M.ci.size()) / double(M.n) : 1.0;
  int g = 1;
  while (g < 16 && rows * 2 * g <= block && mean >= 4.0 * g) g *= 2;
  return g;
}

}  // namespace

bool res_plan_build(int C, int64_t N, const int32_t* rowptr, const int32_t* col, const int64_t* sptr, const int* sw,
                    const AmgHost* H, bool f32, bool f64, ResPlan* out) {
  ResShape& s = out->s;
  s = ResShape{};
  s.C = C;
  const int nlev = H ? int(H->lev.size()) : 0;
  if (nlev > kResLevels) return false;
  std::vector<Space> sp(nlev + 1);
  sp[0].n = N;
  sp[0].q = int((((N + C - 1) / C) + 31) / 32) * 32;
  for (int l = 1; l <= nlev; ++l) {
    sp[l].n = l < nlev ? H->lev[l].A.n : H->nc;
    sp[l].q = std::max(1, int((sp[l].n + C - 1) / C));
    if (l == nlev) sp[l].q = (sp[l].q + 3) & ~3;   // the coarse gather sends four values at a time
  }
  for (Space& x : sp) x.halo.resize(C);
  s.q0 = sp[0].q;
  s.rpt = 1;
  while (s.rpt * kResBlock < s.q0) ++s.rpt;
  if (s.rpt > kResMaxRows) return false;
  s.block = std::max(128, ((s.q0 + s.rpt - 1) / s.rpt + 31) / 32 * 32);
  const int64_t nsl = (N + 31) / 32;
  for (int c = 0; c < C; ++c) {
    for (int64_t i = sp[0].first(c); i < sp[0].first(c) + sp[0].count(c); ++i)
      for (int32_t p = rowptr[i]; p < rowptr[i + 1]; ++p) need(sp[0], c, col[p]);
    for (int l = 0; l < nlev; ++l) {
      const AmgHostLevel& L = H->lev[l];
      if (l > 0)
        for (int64_t i = sp[l].first(c); i < sp[l].first(c) + sp[l].count(c); ++i)
          for (int64_t p = L.A.rp[i]; p < L.A.rp[i + 1]; ++p) need(sp[l], c, L.A.ci[p]);
      if (l + 1 < nlev)   // the coarsest space is gathered whole in every block
        for (int64_t i = sp[l].first(c); i < sp[l].first(c) + sp[l].count(c); ++i)
          for (int64_t p = L.P.rp[i]; p < L.P.rp[i + 1]; ++p) need(sp[l + 1], c, L.P.ci[p]);
      for (int64_t i = sp[l + 1].first(c); i < sp[l + 1].first(c) + sp[l + 1].count(c); ++i)
        for (int64_t p = L.R.rp[i]; p < L.R.rp[i + 1]; ++p) need(sp[l], c, L.R.ci[p]);
    }
  }
  for (Space& x : sp)
    for (auto& h : x.halo) {
      std::sort(h.begin(), h.end());
      h.erase(std::unique(h.begin(), h.end()), h.end());
      x.slots = std::max(x.slots, x.q + int(h.size()));
    }
  for (int l = 0; l <= nlev; ++l)
    if (sp[l].slots > 65535 || sp[l].q > 4095) return false;
  s.slots0 = sp[0].slots;
  // level-0 images
  std::vector<Image> im0(C);
  std::vector<std::vector<uint32_t>> sl(C);
  out->cta.assign(C, ResCta{});
  for (int c = 0; c < C; ++c) {
    const int64_t s0 = sp[0].first(c) / 32, s1 = std::min<int64_t>(nsl, (sp[0].first(c) + sp[0].count(c) + 31) / 32);
    ResCta& ct = out->cta[c];
    ct.ns = int(std::max<int64_t>(0, s1 - s0));
    ct.ent0 = ct.ns > 0 ? int(sptr[s0]) : 0;
    ct.nent = ct.ns > 0 ? int(sptr[s1 - 1] + 32 * int64_t(sw[s1 - 1]) - sptr[s0]) : 0;
    ct.nhalo = int(sp[0].halo[c].size());
    s.nent_max = std::max(s.nent_max, ct.nent);
  }
  const int nsmax = s.q0 / 32;
  size_t npush = 0;
  std::vector<std::vector<uint32_t>> pw(C);
  for (int c = 0; c < C; ++c) {
    pw[c] = push_words(sp[0], c);
    out->cta[c].npush = int(pw[c].size());
    npush = std::max(npush, pw[c].size());
  }
  auto up16 = [](size_t v) { return (v + 15) & ~size_t(15); };
  s.off_lcol = int(up16(size_t(nsmax) * 4));
  s.off_push = int(up16(s.off_lcol + size_t(s.nent_max) * 2));
  s.img0 = int(up16(s.off_push + npush * 4));
  out->img0.assign(size_t(C) * s.img0, 0);
  for (int c = 0; c < C; ++c) {
    unsigned char* b = out->img0.data() + size_t(c) * s.img0;
    const int64_t s0 = sp[0].first(c) / 32;
    uint32_t* words = reinterpret_cast<uint32_t*>(b);
    uint16_t* lc = reinterpret_cast<uint16_t*>(b + s.off_lcol);
    for (int k = 0; k < out->cta[c].ns; ++k) {
      const int64_t base = sptr[s0 + k] - out->cta[c].ent0;
      if (sw[s0 + k] > 4095) return false;
      words[k] = uint32_t(base / 32) << 12 | uint32_t(sw[s0 + k]);
      for (int l = 0; l < 32; ++l) {
        const int64_t i = (s0 + k) * 32 + l;
        const int len = i < N ? rowptr[i + 1] - rowptr[i] : 0;
        for (int e = 0; e < sw[s0 + k]; ++e)
          lc[base + 32 * e + l] = e < len ? uint16_t(sp[0].slot(c, col[rowptr[i] + e])) : uint16_t(32 * k + l);
      }
    }
    if (!pw[c].empty()) std::memcpy(b + s.off_push, pw[c].data(), pw[c].size() * 4);
  }
  // hierarchy images
  s.nlev = nlev;
  if (nlev == 0) return true;
  s.nc = int(H->nc);
  s.ldc = int((H->nc + 3) & ~int64_t(3));   // a multiple of what one message carries
  for (int l = 1; l < nlev; ++l) {
    s.slotsL[l] = sp[l].slots;
    s.qL[l] = sp[l].q;
  }
  out->cinv.assign(size_t(s.nc) * s.ldc, 0.0);
  for (int64_t i = 0; i < H->nc; ++i)
    std::copy(H->cinv.begin() + i * H->nc, H->cinv.begin() + (i + 1) * H->nc, out->cinv.begin() + i * s.ldc);
  bool ok = true;
  auto images = [&](auto zero, std::vector<unsigned char>* dst, int* bytes) {
    using T = decltype(zero);
    std::vector<Image> im(C);
    size_t most = 0;
    for (int c = 0; c < C; ++c) {
      ResAmgHdr h{};
      im[c].put(&h, sizeof(h));
      h.nlev = nlev;
      h.nc = int(H->nc);
      h.c0 = sp[nlev].first(c);
      h.ncown = sp[nlev].count(c);
      for (int l = 0; l < nlev; ++l) {
        const AmgHostLevel& L = H->lev[l];
        ResLevel& o = h.L[l];
        o.nown = sp[l].count(c);
        o.nhalo = int(sp[l].halo[c].size());
        o.omega = L.omega;
        o.omega32 = float(L.omega);
        std::vector<T> id(L.invdiag.begin() + sp[l].first(c), L.invdiag.begin() + sp[l].first(c) + sp[l].count(c));
        o.off_invd = int(im[c].put(id.data(), id.size() * sizeof(T)));
        if (l > 0) {
          const std::vector<uint32_t> w = push_words(sp[l], c);
          o.npush = int(w.size());
          o.off_push = int(im[c].put(w.data(), w.size() * 4));
          o.A = put_op<T>(im[c], L.A, sp[l].first(c), sp[l].count(c), lanes(L.A, sp[l].q, s.block),
                          [&](int64_t j) { return sp[l].slot(c, j); });
        }
        o.P = put_op<T>(im[c], L.P, sp[l].first(c), sp[l].count(c), l == 0 ? 1 : lanes(L.P, sp[l].q, s.block),
                        [&](int64_t j) { return l + 1 < nlev ? sp[l + 1].slot(c, j) : int(j); });
        o.R = put_op<T>(im[c], L.R, sp[l + 1].first(c), sp[l + 1].count(c), lanes(L.R, sp[l + 1].q, s.block),
                        [&](int64_t j) { return sp[l].slot(c, j); });
        for (const ResOp* q : {&o.A, &o.P, &o.R})
          for (int k = 0; k < q->ns; ++k)
            if ((reinterpret_cast<uint32_t*>(im[c].b.data() + q->off_slice)[k] & 4095u) == 4095u) ok = false;
      }
      std::memcpy(im[c].b.data(), &h, sizeof(h));
      most = std::max(most, im[c].b.size());
    }
    *bytes = int(up16(most));
    dst->assign(size_t(C) * *bytes, 0);
    for (int c = 0; c < C; ++c) std::memcpy(dst->data() + size_t(c) * *bytes, im[c].b.data(), im[c].b.size());
  };
  if (f32) images(float(0), &out->imgA32, &s.imgA[0]);
  if (f64) images(double(0), &out->imgA64, &s.imgA[1]);
  return ok;
}

}  // namespace bd
