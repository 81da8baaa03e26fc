// resident_order.h -- order of the messages of the cluster-resident solves
// (resident.cu): their phases, and the buffers that dot products take in turn.
// Host code includes it too: tests/resident_order_check.cpp runs the loops'
// phases on a model of a cluster with arbitrarily late blocks and messages.
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

}  // namespace bd
