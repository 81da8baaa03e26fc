// resident.h -- solves whose operators, hierarchy and vectors stay in the
// shared memory of one thread-block cluster (resident.cu), and their plan
// (resident_plan.cpp).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <vector>

#include "bd_internal.h"

namespace bd {

constexpr int kResMaxCluster = 16;    // blocks of a cluster (non-portable size)
constexpr int kResBlock = 512;        // threads per block the kernels are built for (128 registers each)
constexpr int kResMaxRows = 4;        // level-0 rows a thread may own
constexpr int kResLevels = 5;         // smoothed levels the kernels can hold
constexpr int kResSmemMax = 227 * 1024;   // shared memory a block may have
constexpr int kResCoarseMax = 384;    // rows of the dense coarsest level by default (see plan_resident)

// An operator's rows of one block, in the block's shared-memory image
// (offsets in bytes from the image's start).  Rows are dealt 32 / g to a warp
// slice, g lanes a row; entry k of a row belongs to lane k % g, step k / g:
// word base32[s] << 12 | steps, entry (step, lane) at 32 (base32 + step) +
// lane, padding entries value 0 and slot 0.
struct ResOp {
  int nr, ns, g;
  int off_slice, off_col, off_val;
};
struct ResLevel {
  int nown, nhalo;                    // owned and halo entries of the level's space
  int off_invd, off_push, npush;      // 1/diag; sends: source slot << 20 | block << 16 | destination slot
  float omega32;
  ResOp A, P, R;                      // A unused on level 0
  double omega;
};
// header of one block's hierarchy image
struct ResAmgHdr {
  int nlev, nc, c0, ncown;            // smoothed levels; coarse rows, first owned and owned
  ResLevel L[kResLevels];
};

// One block's share of the level-0 structure (host-computed, in device memory)
struct ResCta {
  int ent0, nent;                     // its range of the shared SELL-32 arrays
  int ns, nhalo, npush;               // slices; halo entries; sends
};
// Level-0 image of a block: slice words, local columns (u16, SELL order),
// send words; offsets in bytes from the image's start, the same in every block.
struct ResShape {
  int C = 0;                          // blocks of the cluster
  int q0 = 0;                         // level-0 rows per block (a multiple of 32)
  int block = 0;                      // threads per block
  int rpt = 0;                        // level-0 rows per thread (1 to kResMaxRows)
  int slots0 = 0;                     // level-0 slots (owned + halo), the largest over the blocks
  int nent_max = 0;                   // SELL entries of a block, the largest
  int off_lcol = 0, off_push = 0, img0 = 0;   // level-0 image
  int nlev = 0, nc = 0, ldc = 0;      // hierarchy (nlev = 0: Jacobi)
  int imgA[2] = {0, 0};               // bytes of a hierarchy image, FP32 / FP64
  int slotsL[kResLevels] = {};        // slots of levels >= 1
  int qL[kResLevels] = {};            // owned entries of levels >= 1, the largest
};

// host plan of a handle
struct ResPlan {
  ResShape s;
  std::vector<ResCta> cta;            // C
  std::vector<unsigned char> img0;    // C images of s.img0 bytes
  std::vector<unsigned char> imgA32, imgA64;   // C images each (empty without a hierarchy)
  std::vector<double> cinv;           // dense coarse inverse, nc rows of ldc
};
// Build the plan for clusters of C blocks; false when the problem does not
// suit it (too many rows per thread or halo slots).  rowptr/col: the shared
// CSR pattern of N rows; sptr/sw its SELL-32 layout; H: hierarchy or NULL.
bool res_plan_build(int C, int64_t N, const int32_t* rowptr, const int32_t* col, const int64_t* sptr, const int* sw,
                    const AmgHost* H, bool f32, bool f64, ResPlan* out);

struct ResLaunch {
  int n, N;                           // active rows; rows of the plan (the rest hold zeros)
  int q0, C;
  int off_lcol, off_push, img0, imgA;
  int slots0, nent_max;
  const ResCta* cta;
  const unsigned char* g0;            // level-0 images
  const unsigned char* gA;            // hierarchy images of the inner type (use_amg)
  const void* cinv;
  int nlev, nc, ldc;
  int slotsL[kResLevels], qL[kResLevels];
  const int64_t* sptr;                // shared SELL-32 pattern (right-hand side products)
  const int* swidth;
  const int* col;
  const int* diagpos;
  const double* valA;
  const void* valT;                   // operator values in the inner type
  const double* dextra;
  const double* rl;                   // rhs = rl + c1 V1 va + c2 V2 vb
  const double* val1;
  const double* va;
  double c1;
  const double* val2;
  const double* vb;
  double c2;
  int project, warm, pin, max_outer, inner_cap, use_amg;
  double tol, tol_inner;
  double* x;
  int* status;
  long long* iters_acc;
  long long* solves_acc;
  long long* outer_acc;
  const int* gate;
};

// shared memory of a launch (bytes per block)
size_t res_smem_bytes(const ResShape& s, bool f32, bool amg);
// can clusters of this shape run on the current device? (sets the kernels' attributes)
bool res_prepare(const ResShape& s, bool f32, bool amg);
// nsys (1 or 2) systems of one shape by value, or nsys systems from a device
// table that share C, block and rpt: one cluster each.  smem: shared memory per
// block (0: the shape's; the largest of the table's shapes otherwise)
cudaError_t res_solve(const ResShape& s, bool f32, bool amg, const ResLaunch* host, int nsys, const ResLaunch* tab,
                      size_t smem, cudaStream_t st);

}  // namespace bd
