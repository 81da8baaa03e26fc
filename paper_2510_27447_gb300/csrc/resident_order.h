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
// every warp returns that flag as it finds it behind it.  Hw::end_unless_first()
// ends every warp but the block's first (ended warps count as arrived at all
// barriers to come).
//   A wait that has run out concerns its warp alone (the message may arrive
// before another warp's limit), so nothing but late() follows from it there and
// then.  A late warp goes on to its next barrier, whichever that is, without
// waiting for peers; every path of a solve has one (the one before its results
// are stored, if no other).  There every warp of the block learns of it at once:
// all end but the first, which meets no one at the block's further barriers,
// waits for no phase and goes to the kernel's last barrier, so that the block
// is there as long as a peer may send to it (before that barrier it lets a
// millisecond pass, in which what the block has sent arrives: a peer that has given
// up does not wait for it).  No warp is left waiting.
//   (Two flags, for barriers in turn: with one, a warp whose next wait has run
// out already could set it before a slow one has read what the barrier brought.)
//   The flag is read with the barrier and used after the phase's sends (meet,
// learn).  Measured on GB300, ms per step with a reducing barrier
// (__syncthreads_or) whose outcome every phase waits for and tests / with this:
// TP06 129^2 mixed 1.88 / 1.76, LR91 65^2 FP64 1.96 / 1.91, a batch of twelve 3.43 /
// 3.30.
template <class Hw>
struct PhaseOrder : Hw {
  unsigned par = 0;      // parity of each phase's next completion, and three flags
  static constexpr unsigned kLate = 1u << 31, kGone = 1u << 30, kTurn = 1u << 29;

  // a wait of this warp has run out; no warp's had at the block's last barrier
  BD_ORDER_FN bool late() const { return (par & kLate) != 0u; }
  BD_ORDER_FN bool ok() const { return (par & kGone) == 0u; }
  // the block's barrier; its outcome, for learn()
  BD_ORDER_FN int meet() {
    const int gone = Hw::block_sync(late(), (par & kTurn) != 0u);
    par ^= kTurn;
    return gone;
  }
  BD_ORDER_FN void learn(int gone) {
    if (gone) {
      Hw::end_unless_first();
      par |= kGone;
    }
  }
  BD_ORDER_FN bool sync() {
    learn(meet());
    return ok();
  }
  BD_ORDER_FN void wait(int k) {
    const unsigned p = par >> k & 1u;
    par ^= 1u << k;
    if (!(par & (kLate | kGone)) && !Hw::await(k, p)) par |= kLate;
  }
};

}  // namespace bd
