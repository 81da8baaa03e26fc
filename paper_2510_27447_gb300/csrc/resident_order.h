// resident_order.h -- order of the messages of the cluster-resident solves
// (resident.cu): their phases, the buffers that dot products take in turn, and
// how a block leaves when a wait runs out.  Host code includes it too:
// tests/resident_order_check.cpp and resident_expiry_check.cpp run the phases on
// models of a cluster with late blocks, late warps and late messages.
#pragma once

#ifdef __CUDACC__
#define BD_ORDER_FN __host__ __device__ __forceinline__
#else
#define BD_ORDER_FN inline
#endif

namespace bd {

// phases (one mbarrier each); levels l >= 1 have four from kLev on: pre-smoothed
// x, residual, corrected x, result
enum : int { kRed = 0, kRed2, kSum0, kSum1, kXF, kZ, kX0, kRes, kX0b, kBc, kXc, kPin, kLev };

// Dot products take two mbarriers and two buffers in turn.  One that has
// completed at a block shows it that every block has SENT its partial sums,
// not that every block has received and read them: the next one's must not meet
// them.  It does show that every block has read the totals of the one before,
// since a block sends after reading, so the one after the next may use that
// one's buffer.  (Halo exchanges do not help: a block waits there for its
// neighbours only, and one that owns no rows for nobody.)
struct SumTurns {
  int n = 0;
  BD_ORDER_FN int next() { return n++ & 1; }
};

// A warp's view of the phases: the parities of its next waits, and whether the
// solve goes on.  Hw::await(k, parity) waits for phase k of this block with a
// limit and returns false when that has passed.  Hw::block_sync(late, turn) is
// the block's barrier: a late warp sets the block's flag of this turn before it,
// every warp returns that flag as it finds it behind it.
//   A wait that has run out concerns its warp alone (the message may arrive
// before another warp's limit), so nothing but late() follows from it there and
// then.  At the block's next barrier every warp learns of it at once: ok() is the
// same in the whole block, and a block that is not ok passes no further barrier.
// (Two flags, for barriers in turn: with one, a warp whose next wait has run out
// already could set it before a slow one has read what the barrier brought.)  A
// late warp goes on to its next barrier, whichever that is, without waiting for
// peers; every path of a solve has one (the one before its results are stored,
// if no other).  So all warps of a block pass equally many barriers, and every
// wait has an end.
//   The flag is read with the barrier and used after the phase's sends (meet,
// learn).  With a reducing barrier (__syncthreads_or) instead, measured on GB300,
// a step against this form: TP06 129^2 mixed 1.88 / 1.83 ms, LR91 65^2 FP64 1.96 /
// 1.92, a batch of twelve 3.43 / 3.35.
template <class Hw>
struct PhaseOrder : Hw {
  unsigned par = 0;      // parity of each phase's next completion, and three flags
  static constexpr unsigned kLate = 1u << 31, kGone = 1u << 30, kTurn = 1u << 29;

  // a wait of this warp has run out; no warp's had at the block's last barrier
  BD_ORDER_FN bool late() const { return (par & kLate) != 0u; }
  BD_ORDER_FN bool ok() const { return (par & kGone) == 0u; }
  // barrier of a block that is ok; its outcome, for learn()
  BD_ORDER_FN int meet() {
    const int gone = Hw::block_sync(late(), (par & kTurn) != 0u);
    par ^= kTurn;
    return gone;
  }
  BD_ORDER_FN void learn(int gone) {
    if (gone) par |= kGone;
  }
  BD_ORDER_FN bool sync() {
    if (ok()) learn(meet());
    return ok();
  }
  BD_ORDER_FN void wait(int k) {
    const unsigned p = par >> k & 1u;
    par ^= 1u << k;
    if (!(par & (kLate | kGone)) && !Hw::await(k, p)) par |= kLate;
  }
};

}  // namespace bd
