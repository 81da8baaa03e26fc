// Waits of the cluster-resident solves that run out, on a model of two blocks of
// four warps (threads here): PhaseOrder (resident_order.h) over barriers and
// phases that count messages, and a script of messages that come late or never.
// Every barrier of the model gives up after three seconds: a warp that meets
// that limit would have hung (so would a phase expected twice).  Usage: resident_expiry_check rule script
//   rule    order   PhaseOrder
//           alone   a late warp leaves by itself (the block's first to the cluster
//                   barrier, the others end), which hangs in script "between"
//   script  none, lost, between (the message comes after the first warp's limit
//           and before the other warps'), random<seed>
// Prints "stuck" or "done", and how many warps finished and how many were late.
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <random>
#include <string>
#include <thread>
#include <vector>

#include "../paper_2510_27447_gb300/csrc/resident_order.h"

using namespace bd;
using Clock = std::chrono::steady_clock;
using Ms = std::chrono::milliseconds;

namespace {

constexpr int kBlocks = 2, kWarps = 4, kSteps = 12;
std::atomic<bool> stuck{false};
std::atomic<int> finished{0}, lates{0};

// counts arrivals; ended warps count as arrived
struct Barrier {
  std::mutex m;
  std::condition_variable cv;
  int members, here = 0, gen = 0;
  explicit Barrier(int n) : members(n) {}
  void flip() {
    here = 0;
    ++gen;
    cv.notify_all();
  }
  void arrive() {
    std::unique_lock<std::mutex> l(m);
    const int g = gen;
    if (++here == members) flip();
    else if (!cv.wait_for(l, Ms(3000), [&] { return gen != g; })) stuck = true;
  }
  void leave() {
    std::lock_guard<std::mutex> l(m);
    if (--members == here && members > 0) flip();
  }
};

struct Mb {
  std::mutex m;
  std::condition_variable cv;
  int arrivals = 0, tx = 0, done = 0;
  void add(int a, int t) {
    std::lock_guard<std::mutex> l(m);
    arrivals += a;
    tx += t;
    if (arrivals > 1) stuck = true;   // a phase expected again before it was complete
    if (arrivals == 1 && tx == 0) {
      arrivals = 0;
      ++done;
      cv.notify_all();
    }
  }
};

struct Block {
  Barrier bar{kWarps};
  Mb mb[kLev];
  std::atomic<int> flag[2] = {0, 0};
};
struct Cluster {
  Block blk[kBlocks];
  Barrier all{kBlocks * kWarps};
} *cl;
std::string script;

// ms until the message of step `step` from block `from` arrives; < 0: never
int travel(int from, int step, std::mt19937& g) {
  if (script == "lost") return from == 1 && step == 5 ? -1 : 0;
  if (script == "between") return from == 1 && step == 5 ? 150 : 0;
  if (script.rfind("random", 0) == 0) {
    const int r = int(g() % 40);
    return r == 0 ? -1 : r < 4 ? int(g() % 300) : 0;
  }
  return 0;
}

struct Hw {
  int block, warp;
  int limit() const { return warp == 0 ? 50 : 400; }
  int block_sync(bool late, bool turn) const {
    Block& b = cl->blk[block];
    if (late) b.flag[turn] = 1;
    b.bar.arrive();
    // now and then much later than the others
    if (script.rfind("random", 0) == 0 && std::rand() % 16 == 0) std::this_thread::sleep_for(Ms(120));
    return b.flag[turn];
  }
  struct Ended {};
  void end_unless_first() const {
    if (warp > 0) throw Ended{};
  }
  bool await(int k, unsigned p) const {
    Mb& b = cl->blk[block].mb[k];
    std::unique_lock<std::mutex> l(b.m);
    if (b.cv.wait_for(l, Ms(limit()), [&] { return unsigned(b.done & 1) != p; })) return true;
    ++lates;
    return false;
  }
};

void send(int to, int k, int ms) {
  if (ms < 0) return;
  if (ms == 0) return cl->blk[to].mb[k].add(0, -1);
  std::thread([=] {
    std::this_thread::sleep_for(Ms(ms));
    cl->blk[to].mb[k].add(0, -1);
  }).detach();
}

void solve(int block, int w, bool alone, std::mt19937& g) {
  PhaseOrder<Hw> ph{{block, w}};
  SumTurns turns;
  for (int step = 0; step < kSteps; ++step) {
    const int k = step % 2 ? kSum0 + turns.next() : int(kZ);   // as the Jacobi loop
    const int gone = ph.meet();
    if (w == 0) {
      cl->blk[block].mb[k].add(1, 1);
      send(1 - block, k, travel(block, step, g));
    }
    ph.learn(gone);
    ph.wait(k);
    if (alone && ph.late()) {
      if (w > 0) throw Hw::Ended{};
      return;
    }
    // the loop's test, once an iteration; a late warp may take another way at its decisions
    if (step % 2 && (!ph.ok() || (ph.late() && w % 2))) break;
  }
  if (!alone) ph.sync();
}

void warp(int block, int w, bool alone, unsigned seed) {
  std::mt19937 g(seed);
  try {
    solve(block, w, alone, g);
    cl->all.arrive();
  } catch (Hw::Ended&) {
    cl->blk[block].bar.leave();
    cl->all.leave();
  }
  ++finished;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  script = argv[2];
  cl = new Cluster;
  const unsigned seed = script.rfind("random", 0) == 0 ? unsigned(std::atoi(argv[2] + 6)) : 1u;
  std::vector<std::thread> th;
  for (int b = 0; b < kBlocks; ++b)
    for (int w = 0; w < kWarps; ++w) th.emplace_back(warp, b, w, !std::strcmp(argv[1], "alone"), seed * 100 + b * 10 + w);
  for (auto& t : th) t.join();
  std::printf("%s %d %d\n", stuck ? "stuck" : "done", finished.load(), lates.load());
  std::fflush(stdout);
  std::_Exit(0);   // messages may still be under way
}
