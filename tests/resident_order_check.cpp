// Model of the messages of the cluster-resident solves on the CPU: blocks run
// the phases of a loop in order, messages and blocks are late at random, now and
// then by many iterations' time, and an mbarrier counts whatever arrives.  A
// block that reads another value than the one its phase was to bring, or waits
// for ever, is a fault.  Usage:
// resident_order_check jacobi|pipelined|amg turns|single seeds; prints the
// number of seeds with a fault ("single": every dot product on one mbarrier and
// one buffer, which must show up in the Jacobi loop).
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <queue>
#include <random>
#include <string>
#include <vector>

#include "../paper_2510_27447_gb300/csrc/resident_order.h"

using namespace bd;

namespace {

constexpr int C = 16, kOwners = 11, kIters = 40, kMb = kLev + 8, kBufs = 12;
enum Buf { ZR, X0, BC, XC, NX, NY, TOK, SUM };   // SUM + turn

struct Send { int to, buf; };
// one phase of a block: its mbarrier, what it sends, what it reads afterwards
struct Step {
  int phase;
  std::vector<Send> sends;
  std::vector<Send> reads;                       // .to: the block the value comes from
};

struct Model {
  std::string loop;
  bool single;
  std::mt19937_64 rng;
  struct Mb { int arrivals = 0, tx = 0, done = 0; } mb[C][kMb];
  int buf[C][kBufs][C];                          // tag of the value that src left there
  int expects[C][kMb] = {}, used[C][kMb] = {};
  std::vector<Step> prog[C];
  size_t pc[C] = {};
  bool waiting[C] = {}, fault = false;
  struct Event { double t; int kind, blk, a, b, src, tag; };   // 0 message, 1 run
  struct Later { bool operator()(const Event& x, const Event& y) const { return x.t > y.t; } };
  std::priority_queue<Event, std::vector<Event>, Later> q;

  double delay() {
    const double u = std::uniform_real_distribution<double>(0.5, 1.5)(rng);
    return rng() % 100 == 0 ? 300 * u : u;
  }
  static bool owner(int c) { return c < kOwners; }
  static std::vector<int> near(int c) {
    std::vector<int> n;
    if (owner(c))
      for (int d : {c - 1, c + 1})
        if (d >= 0 && owner(d)) n.push_back(d);
    return n;
  }
  void halo(Step& s, int c, int b) {
    for (int d : near(c)) {
      s.sends.push_back({d, b});
      s.reads.push_back({d, b});
    }
  }
  void all(Step& s, int b, int senders, int c) {
    for (int d = 0; d < C; ++d) {
      if (c < senders) s.sends.push_back({d, b});
      if (d < senders) s.reads.push_back({d, b});
    }
  }
  void program(int c) {
    SumTurns turns;
    auto step = [&](int phase, auto&& fill) {
      Step s{phase, {}, {}};
      fill(s);
      prog[c].push_back(s);
    };
    for (int it = 0; it < kIters; ++it) {
      const int t = single ? 0 : turns.next();
      if (loop == "pipelined") {   // halo and sums in one phase
        step(kRed + t, [&](Step& s) { halo(s, c, t ? ZR : X0); all(s, SUM + t, C, c); });
        continue;
      }
      if (loop == "amg") {
        step(kX0, [&](Step& s) { halo(s, c, X0); });
        step(kRes, [&](Step& s) { halo(s, c, ZR); });
        step(kLev, [&](Step& s) { halo(s, c, NX); });
        step(kLev + 1, [&](Step& s) { halo(s, c, NY); });
        step(kBc, [&](Step& s) { all(s, BC, 3, c); all(s, TOK, C, c); });
        step(kXc, [&](Step& s) { all(s, XC, 3, c); });
        step(kLev + 2, [&](Step& s) { halo(s, c, NX); });
        step(kLev + 3, [&](Step& s) { halo(s, c, NY); });
        step(kX0b, [&](Step& s) { halo(s, c, X0); });
      }
      step(kZ, [&](Step& s) { halo(s, c, ZR); });
      step(kSum0 + t, [&](Step& s) { all(s, SUM + t, C, c); });
    }
  }
  void settle(Mb& m) {
    if (m.arrivals == 1 && m.tx == 0) {
      m.arrivals = 0;
      ++m.done;
    }
  }
  bool passed(int c) {
    const int k = prog[c][pc[c]].phase;
    return (mb[c][k].done & 1) != (used[c][k] & 1);   // as the hardware tests it: by parity
  }
  void begin(int c, double now) {
    const Step& s = prog[c][pc[c]];
    Mb& m = mb[c][s.phase];
    m.arrivals += 1;
    m.tx += int(s.reads.size());
    settle(m);
    for (const Send& x : s.sends) q.push({now + delay(), 0, x.to, s.phase, x.buf, c, int(pc[c])});
    waiting[c] = true;
    wake(c, now);
  }
  void wake(int c, double now) {
    if (!waiting[c] || !passed(c)) return;
    waiting[c] = false;
    q.push({now + delay(), 1, c, 0, 0, 0, 0});       // reads at the end of its work
  }
  bool run(int seed) {
    rng.seed(uint64_t(seed));
    std::memset(buf, -1, sizeof buf);
    for (int c = 0; c < C; ++c) program(c);
    for (int c = 0; c < C; ++c) begin(c, delay());
    while (!q.empty()) {
      const Event e = q.top();
      q.pop();
      if (e.kind == 0) {
        buf[e.blk][e.b][e.src] = e.tag;
        Mb& m = mb[e.blk][e.a];
        m.tx -= 1;
        settle(m);
        wake(e.blk, e.t);
        continue;
      }
      const int c = e.blk;
      const Step& s = prog[c][pc[c]];
      for (const Send& r : s.reads) fault = fault || buf[c][r.buf][r.to] != int(pc[c]);
      ++used[c][s.phase];
      if (++pc[c] < prog[c].size()) begin(c, e.t);
    }
    for (int c = 0; c < C; ++c) fault = fault || pc[c] < prog[c].size();
    return fault;
  }
};

}  // namespace

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  int bad = 0;
  for (int seed = 1; seed <= std::atoi(argv[3]); ++seed) {
    auto m = new Model;
    m->loop = argv[1];
    m->single = !std::strcmp(argv[2], "single");
    bad += m->run(seed);
    delete m;
  }
  std::printf("%d\n", bad);
  return 0;
}
