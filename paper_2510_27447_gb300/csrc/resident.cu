// resident.cu -- conjugate gradients held in the shared memory of one
// thread-block cluster.
//
// On small meshes a solve is a chain of dependent steps: in the grid-wide
// kernels (pcg.cu, amg.cu, mixed.cu) every phase waits for a device-wide
// barrier (1.25 us) and walks slice header -> column -> gathered value through
// L2.  Here the rows of every level are split over the C blocks of ONE cluster
// and a block keeps its share of the operator, of the AMG hierarchy and of all
// vectors in shared memory for the whole solve; the finest level's Krylov
// vectors, and the first eight entries of its rows, live in registers.
//
// Exchange.  A vector is stored as its owned entries followed by the halo
// entries the block's rows read.  After a phase of the iteration has written
// its owned entries, the block sends those its peers need into their halo
// slots (st.async), and every send counts its bytes on an mbarrier of the
// receiving block; each phase has its own mbarrier, which completes when the
// expected bytes are there.  A one-way message thus takes the place of a
// store, its acknowledgement and a cluster barrier (measured, 16 blocks: 425
// against 1,020 clocks).  Dot products travel the same way: partial sums go to
// every block, and all add them in the same order.
//   A buffer is sent to again, and an mbarrier counted on again, only after
// another phase in which every block hears from every other (a dot product, or
// the coarse gather, which carries a token of each block for this) has completed
// at the sender: every block sent in it after reading the buffer.  A phase of
// this kind does not protect its own buffer, so dot products use two buffers
// and two mbarriers in turn (SumTurns), and so do the halos that travel with
// them in the pipelined loop.
//   Waits for peers are bounded (kWaitLimitNs).  On expiry a warp records
// ST_TIMEOUT; the block's next barrier tells all its warps, which then end, except
// the first, which leaves through the cluster barrier at the kernel's end, so
// that no block is gone while a peer may still send to it (PhaseOrder).
//
// The iteration is the one of the grid kernels: Jacobi- or AMG-V(1,1)-
// preconditioned CG; T = double solves in FP64, T = float is the mixed path's
// FP32 inner solve with FP64 right-hand side, outer residual and solution
// update (mixed.cu states the refinement, and the pipelined form of the
// Jacobi iteration that the single FP32 solves take).  Independent systems
// (the two elliptic solves of a later sweep, the members of a batch) are
// further clusters of the same launch.
//
// Apart from the pipelined loop the iteration is CG with one reduction
// (Chronopoulos & Gear, J. Comput. Appl. Math. 25, 1989): w = A z is formed
// before the dot products (r, z), (w, z), (r, r), and p.Ap follows from them.
//
// What bounds it: the chain of phases (1 an iteration pipelined, 2 Jacobi,
// 3 + 4 L AMG) and, in FP64, the FP64 pipe (two lanes a clock on an SM): a
// problem takes the whole 16-block cluster however small it is, FP64 scalars
// are formed by one thread, and sums are added by four warps a block.
//
// Registers: every instance is built for kResBlock threads, 128 registers each, and
// the AMG instances spill (stores: FP32 0.6 to 1.7 KB, FP64 1.0 to 2.4 KB; pipelined
// Jacobi 0.2 to 0.7 KB, FP64 Jacobi below 0.1), to L1; without opaque() it was more.
// Instances built for the 128 to 416 threads that the plans ask for would spill less.
//
// Measured on GB300, ms per step (three nodes, two sweeps), grid kernels / one
// cluster: LR91 33^2 mixed 4.10 / 0.65, LR91 65^2 FP64 6.35 / 1.91, TP06 129^2
// mixed 2.63 / 1.76, LR91 101^2 FP64 adaptive 5.66 / 2.73 and CN-RK2 1.20 / 0.68,
// a batch of twelve 65^2 and 129^2 requests (against streaming chains) 9.23 / 3.30.
// Both sides near the largest sizes that fit: LR91 119^2 mixed 2.12 / 1.20 and FP64
// 5.28 / 2.88, slabs 30x30x8 mixed 2.63 / 1.42 and 25x25x8 FP64 5.58 / 2.79.
#include <cuda_runtime.h>

#include <algorithm>

#include "resident.h"
#include "resident_order.h"
#include "sparse.cuh"

namespace bd {

namespace {

struct ResPair {
  ResLaunch a[2];
};

__host__ __device__ constexpr size_t up16(size_t v) { return (v + 15) & ~size_t(15); }

constexpr int kPhases = kLev + 4 * (kResLevels - 1);
static_assert(kPhases <= 29, "the parities and three flags are the bits of one word");

// dynamic shared memory of a block: identical offsets in every block of the
// cluster (a send addresses a peer's copy by the local offset)
struct ResMem {
  int img0, valA, x0, zr, xf, st, part, lv[kResLevels][3], bc, xc, imgA, total;   // lv: b, x, y
};
// partial sums of two turns: FP32 (16 warps x 16 blocks) x float4, FP64 3 values x (4 warps x 16 blocks)
constexpr int kPartF = 2 * 16 * kResMaxCluster * 4, kPartD = 2 * 3 * 4 * kResMaxCluster;
template <class S>
__host__ __device__ __forceinline__ void res_mem(const S& s, int img0, int imgA, int block, int vb, bool amg,
                                                 ResMem* m) {
  size_t o = 0;
  m->img0 = int(o);
  o = up16(o + img0);
  m->valA = int(o);
  o = up16(o + size_t(s.nent_max) * vb);
  m->zr = int(o);
  o = up16(o + size_t(s.slots0) * vb);
  m->x0 = int(o);
  if (amg || vb == 4) o = up16(o + size_t(s.slots0) * vb);
  m->st = int(o);
  o = up16(o + size_t(3) * block * 8);
  m->part = int(o);
  o = up16(o + size_t(kPartD) * 8 + (vb == 4 ? size_t(kPartF) * 4 : 0));
  m->xf = int(o);
  if (vb == 4) o = up16(o + size_t(s.slots0) * 8);
  m->bc = m->xc = m->imgA = int(o);
  if (amg) {
    for (int l = 1; l < s.nlev; ++l) {
      m->lv[l][0] = int(o);
      o = up16(o + size_t(s.qL[l]) * vb);
      for (int k = 1; k < 3; ++k) {
        m->lv[l][k] = int(o);
        o = up16(o + size_t(s.slotsL[l]) * vb);
      }
    }
    m->bc = int(o);
    o = up16(o + size_t(s.ldc) * vb);
    m->xc = int(o);
    o = up16(o + size_t(s.ldc) * vb);
    m->imgA = int(o);
    o = up16(o + imgA);
  }
  m->total = int(o);
}

// v, unknown to the optimiser: what is derived from it is formed where it is
// used.  The iteration loop has a dozen phases; addresses hoisted out of it
// for all of them were 130 registers more than a thread has.
__device__ __forceinline__ int opaque(int v) {
  asm volatile("" : "+r"(v));
  return v;
}
__device__ __forceinline__ unsigned smem_addr(const void* p) { return unsigned(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ unsigned peer_addr(unsigned a, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// copy bytes (a multiple of 16) into shared memory; waited for by cp_wait()
__device__ __forceinline__ void cp_block(unsigned char* dst, const void* src, int bytes) {
  const unsigned d = smem_addr(dst);
  for (int i = threadIdx.x * 16; i < bytes; i += blockDim.x * 16)
    cp_async16(d + i, static_cast<const unsigned char*>(src) + i);
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr unsigned long long kDrainNs = 1000000ull;

// the block's mbarriers, its barrier and flags, as PhaseOrder uses them
struct PhaseHw {
  unsigned mb;          // shared address of the mbarriers
  int* status;

  __device__ __forceinline__ unsigned addr(int k) const { return mb + 8u * unsigned(k); }
  // (the two flags follow the mbarriers)
  __device__ __forceinline__ int block_sync(bool late, bool turn) const {
    const unsigned flag = addr(kPhases) + (turn ? 4u : 0u);
    if (late) asm volatile("st.volatile.shared.u32 [%0], 1;" ::"r"(flag) : "memory");
    __syncthreads();
    int gone;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(gone) : "r"(flag) : "memory");
    return gone;
  }
  __device__ __forceinline__ void end_unless_first() const {
    if (threadIdx.x >= 32) asm volatile("exit;");
  }
  // the block expects bytes from its peers in phase k (thread 0, after a
  // barrier of the block behind the phase's own work)
  __device__ __forceinline__ void expect(int k, int bytes) const {
    if (threadIdx.x == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr(k)), "r"(bytes) : "memory");
  }
  // false (in all lanes of the warp) once kWaitLimitNs have passed
  __device__ __forceinline__ bool await(int k, unsigned parity) const {
    unsigned long long t0 = 0;
#pragma unroll 1
    for (unsigned n = 1;; ++n) {
      unsigned d;
      asm volatile(
          "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 q, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(d)
          : "r"(addr(k)), "r"(parity)
          : "memory");
      if (__all_sync(0xffffffffu, d != 0u)) return true;
      if ((n & 63u) == 0u) {
        const unsigned long long t = device_ns();
        if (t0 == 0) t0 = t;
        if (__any_sync(0xffffffffu, t - t0 > kWaitLimitNs)) {
          if ((threadIdx.x & 31) == 0) atomicOr(status, ST_TIMEOUT);
          return false;
        }
      }
    }
  }
  // v into a peer's copy of *p, counted on the peer's phase k
  __device__ __forceinline__ void send(const float* p, unsigned rank, float v, int k) const {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                     peer_addr(smem_addr(p), rank)),
                 "r"(__float_as_uint(v)), "r"(peer_addr(addr(k), rank))
                 : "memory");
  }
  __device__ __forceinline__ void send(const double* p, unsigned rank, double v, int k) const {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(
                     peer_addr(smem_addr(p), rank)),
                 "l"(__double_as_longlong(v)), "r"(peer_addr(addr(k), rank))
                 : "memory");
  }
  __device__ __forceinline__ void send4(const float* p, unsigned rank, float4 v, int k) const {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
            peer_addr(smem_addr(p), rank)),
        "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)),
        "r"(peer_addr(addr(k), rank))
        : "memory");
  }
};
using Phases = PhaseOrder<PhaseHw>;

// The owned entries of vec are written: send the peers theirs and wait for
// the block's own halo (bytes: what the block expects in phase k besides)
template <class T>
__device__ __forceinline__ void exchange(Phases& ph, const uint32_t* word, int n, T* vec, int k, int bytes) {
  const int gone = ph.meet();
  ph.expect(k, bytes);
#pragma unroll 1
  for (int e = opaque(threadIdx.x); e < n; e += blockDim.x) {
    const uint32_t w = word[e];
    ph.send(vec + (w & 0xffffu), w >> 16 & 15u, vec[w >> 20], k);
  }
  ph.learn(gone);
  ph.wait(k);
}
// count values of a coarse vector, owned from c0 on (a multiple of 4), to every block
template <class T>
__device__ __forceinline__ void gather_all(Phases& ph, T* vec, int c0, int count, int C, int k, int bytes) {
  const int gone = ph.meet();
  ph.expect(k, bytes);
  const int sh = 31 - __clz(C);          // C is a power of two
  if constexpr (sizeof(T) == 4) {        // the padding entries travel along
#pragma unroll 1
    for (int e = opaque(threadIdx.x); e < ((count + 3) >> 2) << sh; e += blockDim.x) {
      float* p = vec + c0 + 4 * (e >> sh);
      ph.send4(p, unsigned(e & (C - 1)), *reinterpret_cast<const float4*>(p), k);
    }
  } else {
#pragma unroll 1
    for (int e = opaque(threadIdx.x); e < count << sh; e += blockDim.x) {
      T* p = vec + c0 + (e >> sh);
      ph.send(p, unsigned(e & (C - 1)), *p, k);
    }
  }
  ph.learn(gone);
  ph.wait(k);
}

// lane's part of the rows of one slice: sum over steps [k0, steps) of val x[col]
template <class TV, class TX>
__device__ __forceinline__ TX slice_dot(const uint16_t* col, const TV* val, int k0, int steps, const TX* x) {
  TX acc = TX(0);
#pragma unroll 1
  for (int k = k0; k < steps; k += 4) {
    int c[4];
    TV v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < steps) {
        c[j] = col[32 * (k + j)];
        v[j] = val[32 * (k + j)];
      }
    TX g[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < steps) g[j] = x[c[j]];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < steps) acc += TX(v[j]) * g[j];
  }
  return acc;
}

// every row of an operator image: epi(row, sum, lane's index among the row's
// g lanes); all lanes of a row hold the sum
template <class T, class F>
__device__ __forceinline__ void op_rows(const ResOp& o, const unsigned char* img, const T* x, F&& epi) {
  const uint32_t* sl = reinterpret_cast<const uint32_t*>(img + o.off_slice);
  const uint16_t* col = reinterpret_cast<const uint16_t*>(img + o.off_col);
  const T* val = reinterpret_cast<const T*>(img + o.off_val);
  const int tid = opaque(threadIdx.x), lane = tid & 31, nw = blockDim.x >> 5, g = o.g;
#pragma unroll 1
  for (int s = tid >> 5; s < o.ns; s += nw) {
    const uint32_t w = sl[s];
    const int at = int(w >> 12) * 32 + lane;
    T a = slice_dot<T, T>(col + at, val + at, 0, int(w & 4095u), x);
#pragma unroll 1
    for (int d = g >> 1; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    const int row = s * (32 / g) + lane / g;
    if (row < o.nr) epi(row, a, lane & (g - 1));
  }
}

// FP64 sums over the cluster: through shared memory to four warps (whose lanes
// all add distinct values, see sparse.cuh:block_sum), their partials to every
// block; thread 0 adds the totals and runs f(totals), which writes shared
// variables the block reads afterwards.  Returns what the last barrier brought,
// for learn() (the caller's reads of those variables may go ahead of it).
template <int NV, class F>
__device__ __forceinline__ int sum_f64(Phases& ph, int k, int part_slot, double (&v)[NV], double* stage, double* part,
                                        int C, int rank, F&& f) {
  static_assert(NV <= 3, "up to three values");
  constexpr int G = NV == 1 ? 32 : NV == 2 ? 16 : 8;   // lanes that end with one value
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, bd = blockDim.x;
  double* pt = part + part_slot * 3 * 4 * kResMaxCluster;
#pragma unroll
  for (int i = 0; i < NV; ++i) stage[i * bd + threadIdx.x] = v[i];
  const int gone = ph.meet();
  ph.expect(k, C * 4 * NV * 8);
  if (wid < 4) {
#pragma unroll 1
    for (int t = threadIdx.x + 128; t < bd; t += 128)
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] += stage[i * bd + t];
    const double x = warp_sum_spread<NV>(v);
    const int i = lane_value<NV>(lane);
    if (i < NV)
      for (int c = lane & (G - 1); c < C; c += G)
        ph.send(pt + i * 4 * kResMaxCluster + rank * 4 + wid, unsigned(c), x, k);
  }
  ph.learn(gone);
  ph.wait(k);
  if (wid == 0) {
    double p[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const double* q = pt + i * 4 * kResMaxCluster;
      p[i] = lane < 4 * C ? q[lane] : 0.0;
      if (32 + lane < 4 * C) p[i] += q[32 + lane];
    }
    const double x = warp_sum_spread<NV>(p);
#pragma unroll
    for (int i = 0; i < NV; ++i) p[i] = __shfl_sync(0xffffffffu, x, i * G);
    if (lane == 0 && !ph.late()) f(p);
  }
  return ph.meet();
}

// FP32 sums of three values over the cluster: every warp sends its partials
// to every block in one message, every warp adds the totals
__device__ __forceinline__ void sum_f32_send(Phases& ph, int k, int part_slot, const float (&v)[3], float* part, int C,
                                             int rank, int nw) {
  const int lane = threadIdx.x & 31;
  const float x = warp_sum_spread<3>(v);
  const float4 m = make_float4(__shfl_sync(0xffffffffu, x, 0), __shfl_sync(0xffffffffu, x, 8),
                               __shfl_sync(0xffffffffu, x, 16), 0.f);
  if (lane < C)
    ph.send4(part + (part_slot * 16 * kResMaxCluster + rank * nw + (threadIdx.x >> 5)) * 4, unsigned(lane), m, k);
}
__device__ __forceinline__ void sum_f32_get(int part_slot, float (&v)[3], const float* part, int n) {
  const float4* q = reinterpret_cast<const float4*>(part) + part_slot * 16 * kResMaxCluster;
  v[0] = v[1] = v[2] = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < n; i += 32) {
    const float4 a = q[i];
    v[0] += a.x;
    v[1] += a.y;
    v[2] += a.z;
  }
  const float x = warp_sum_spread<3>(v);
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i] = __shfl_sync(0xffffffffu, x, 8 * i);
}

// products of up to three operators on the shared SELL-32 pattern over row i
// (global memory, vectors through L2): four entries of all of them in flight
__device__ __forceinline__ void rhs_row(const int64_t* sptr, const int* sw, const int* col, const double* const (&val)[3],
                                        const double* const (&x)[3], int i, double (&out)[3]) {
  const int64_t base = sptr[i >> 5] + (i & 31);
  const int w = sw[i >> 5];
  out[0] = out[1] = out[2] = 0.0;
#pragma unroll 1
  for (int k0 = 0; k0 < w; k0 += 4) {
    int c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = k0 + k < w ? col[base + 32 * (k0 + k)] : -1;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (!val[q]) continue;
      double v[4], g[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = c[k] >= 0 ? __ldg(val[q] + base + 32 * (k0 + k)) : 0.0;
        g[k] = c[k] >= 0 ? __ldcg(x[q] + c[k]) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (c[k] >= 0) out[q] += v[k] * g[k];
    }
  }
}

template <class T, int RPT, bool AMG>
__global__ void __launch_bounds__(kResBlock, 1) res_kernel(const __grid_constant__ ResPair pr,
                                                          const ResLaunch* __restrict__ tab) {
  constexpr bool F32 = sizeof(T) == 4;
  // the first eight entries of a thread's rows in registers while they fit
  constexpr bool HOLD = F32 ? RPT <= 3 : RPT <= 2;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ __align__(16) ResLaunch a;
  __shared__ ResMem M;    // the level loops index it at run time
  __shared__ __align__(8) unsigned long long s_mb[kPhases + 1];   // and the block's two flags
  __shared__ double s_pin, s_d[6];
  __shared__ int s_code;
  __shared__ float s_tok[kResMaxCluster];
  unsigned C, rank;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int tid = threadIdx.x, lane = tid & 31, bd = blockDim.x, nw = bd >> 5;
  {
    const int sys = blockIdx.x / C;
    const int* src = reinterpret_cast<const int*>(tab ? tab + sys : pr.a + sys);
    int* dst = reinterpret_cast<int*>(&a);
    for (int i = tid; i < int(sizeof(ResLaunch) / 4); i += bd) dst[i] = src[i];
  }
  __syncthreads();
  if (a.gate && *a.gate == 0) return;   // the same in every block of the cluster
  if (tid == 0) res_mem(a, a.img0, a.imgA, bd, int(sizeof(T)), AMG, &M);
  if (tid < kPhases) asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&s_mb[tid])), "r"(1));
  if (tid == kPhases) s_mb[kPhases] = 0ull;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  const ResCta ct = a.cta[rank];
  cp_block(sm + M.img0, a.g0 + size_t(rank) * a.img0, a.img0);
  cp_block(sm + M.valA, static_cast<const T*>(a.valT) + ct.ent0, ct.nent * int(sizeof(T)));
  if constexpr (AMG) cp_block(sm + M.imgA, a.gA + size_t(rank) * a.imgA, a.imgA);
  // zero vectors: padding entries multiply slot 0, which a block that owns no
  // entry of a level never writes
  for (int i = M.zr + 16 * tid; i < M.imgA; i += 16 * bd) *reinterpret_cast<float4*>(sm + i) = make_float4(0.f, 0.f, 0.f, 0.f);

  Phases ph{{smem_addr(s_mb), a.status}};
  const uint32_t* sl0 = reinterpret_cast<const uint32_t*>(sm + M.img0);
  const uint16_t* lcol = reinterpret_cast<const uint16_t*>(sm + M.img0 + a.off_lcol);
  const uint32_t* push0 = reinterpret_cast<const uint32_t*>(sm + M.img0 + a.off_push);
  const T* valA = reinterpret_cast<const T*>(sm + M.valA);
// read from the shared descriptor at each use (see opaque)
#define ZR reinterpret_cast<T*>(sm + M.zr)
#define X0 reinterpret_cast<T*>(sm + M.x0)
#define XF reinterpret_cast<double*>(sm + M.xf)
#define stage reinterpret_cast<double*>(sm + M.st)
#define partd reinterpret_cast<double*>(sm + M.part)
#define partf reinterpret_cast<float*>(sm + M.part + kPartD * 8)
#define img (static_cast<const unsigned char*>(sm) + M.imgA)
#define H (*reinterpret_cast<const ResAmgHdr*>(img))
  const int r0 = int(rank) * a.q0;
  auto clampq = [&](int n) { return n - r0 < 0 ? 0 : (n - r0 < a.q0 ? n - r0 : a.q0); };
  const int nloc = clampq(a.n), nown = clampq(a.N);   // active and owned rows
  const int halo0 = ct.nhalo * int(sizeof(T));
  const int iC = int(C), irank = int(rank);
  const int nparts = iC * nw;   // FP32 partial sums of a phase

  // ---- FP64 right-hand side and first residual (global SELL-32 operators) ----
  double b[RPT], xs[RPT], r64[RPT];
  T invd[RPT], dx[RPT], r[RPT], p[RPT], q[RPT], d[RPT], z[RPT];
  double s2[2] = {0.0, 0.0};
  {
    const double* const pv[3] = {a.val1, a.val2, a.warm ? a.valA : nullptr};
    const double* const px[3] = {a.va, a.vb, a.x};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      b[j] = xs[j] = r64[j] = 0.0;
      invd[j] = dx[j] = r[j] = p[j] = q[j] = d[j] = z[j] = T(0);
      const int row = tid + j * bd;
      if (row < nloc) {
        const int i = r0 + row;
        double sp[3];
        rhs_row(a.sptr, a.swidth, a.col, pv, px, i, sp);
        double bi = a.rl ? a.rl[i] : 0.0;
        if (a.val1) bi += a.c1 * sp[0];
        if (a.val2) bi += a.c2 * sp[1];
        const double de = a.dextra ? a.dextra[i] : 0.0;
        invd[j] = jacobi_scale<T>(a.valA[a.diagpos[i]] + de);
        dx[j] = T(de);
        double ri = bi;
        if (a.warm) {
          xs[j] = a.x[i];
          ri -= de * xs[j] + sp[2];
        }
        b[j] = bi;
        r64[j] = ri;
        s2[0] += a.project ? bi : ri * ri;
        s2[1] += bi * bi;
      }
    }
  }
  cp_wait();
  __syncthreads();
  // row tid + j bd of the block: slice, first entries
  int st[RPT], at[RPT];
  T hv[HOLD ? RPT : 1][8];
  uint32_t hc[HOLD ? RPT : 1][4];
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int row = tid + j * bd;
    const bool own = row < nown;
    const uint32_t w = own ? sl0[row >> 5] : 0u;
    st[j] = int(w & 4095u);
    at[j] = int(w >> 12) * 32 + lane;
    if constexpr (HOLD) {
#pragma unroll
      for (int k = 0; k < 4; ++k) hc[j][k] = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        hv[j][k] = k < st[j] ? valA[at[j] + 32 * k] : T(0);
        if (k < st[j]) hc[j][k >> 1] |= uint32_t(lcol[at[j] + 32 * k]) << (16 * (k & 1));
      }
    }
  }
  // product of row j with a vector in slot order
  auto row_dot = [&](int j, const T* x) {
    if constexpr (HOLD) {
      T g[8], acc = T(0);
      // keep the columns packed: unpacked outside the loops they would spill
#pragma unroll
      for (int k = 0; k < 4; ++k) asm volatile("" : "+r"(hc[j][k]));
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < st[j]) g[k] = x[(hc[j][k >> 1] >> (16 * (k & 1))) & 0xffffu];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < st[j]) acc += hv[j][k] * g[k];
      if (st[j] > 8) acc += slice_dot<T, T>(lcol + at[j], valA + at[j], 8, st[j], x);
      return acc;
    } else {
      return slice_dot<T, T>(lcol + at[j], valA + at[j], 0, st[j], x);
    }
  };
  // own entry of a level-0 vector
  auto put0 = [&](int j, T* vec, T v) {
    if (tid + j * bd < nown) vec[tid + j * bd] = v;
  };
  auto exchange0 = [&](T* vec, int k) { exchange<T>(ph, push0, ct.npush, vec, k, halo0); };
  __syncwarp();
  cluster_barrier();   // every block's mbarriers and buffers are ready for its peers

  // scalars of the block: s_d = mean of b, |b|^2, tol^2 |b|^2, scale, 1 / scale, inner target
  int outer = 0;
  SumTurns turns, turns32;                  // FP64 sums (kSum0, kSum1), FP32 sums (kRed, kRed2)
  auto next_sum = [&] { return kSum0 + turns.next(); };
  // thread 0: what to do with the outer residual (s_code: 0 solve, 1 non-finite, 2 done, 3 out of passes)
  auto decide = [&](double rr64) {
    s_code = 0;
    s_d[3] = s_d[4] = 1.0;
    s_d[5] = s_d[2];
    if constexpr (F32) {
      s_code = !isfinite(rr64)                        ? 1
               : a.max_outer > 1 && rr64 <= s_d[2]    ? 2
               : outer >= a.max_outer                 ? 3
               : !(rr64 > 0.0)                        ? 2
                                                      : 0;
      const double scale = sqrt(rr64);
      double tgt = a.tol_inner * a.tol_inner;
      if (a.max_outer > 1) tgt = fmax(tgt, 0.25 * s_d[2] / rr64);
      else if (a.warm) tgt = fmax(tgt, tgt * s_d[1] / rr64);
      s_d[3] = scale;
      s_d[4] = 1.0 / scale;
      s_d[5] = tgt;
    }
  };
  {
    const int k = next_sum();
    ph.learn(sum_f64<2>(ph, k, k - kSum0, s2, stage, partd, iC, irank, [&](const double (&t)[2]) {
      double bb = t[1];
      s_d[0] = 0.0;
      if (a.project) {
        s_d[0] = t[0] / double(a.n);
        bb -= double(a.n) * s_d[0] * s_d[0];
        if (bb < 0.0) bb = 0.0;
      }
      s_d[1] = bb;
      s_d[2] = a.tol * a.tol * bb;
      if (!a.project) decide(t[0]);
    }));
  }
  if (a.project) {
    const double mean = s_d[0];
    double s1[1] = {0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (tid + j * bd < nloc) {
        b[j] -= mean;
        r64[j] -= mean;
        s1[0] += r64[j] * r64[j];
      }
    const int k = next_sum();
    ph.learn(sum_f64<1>(ph, k, k - kSum0, s1, stage, partd, iC, irank, [&](const double (&t)[1]) { decide(t[0]); }));
  }

  int fail = 0;
  long long inner_total = 0, outer_total = 0;
  for (;; ++outer) {
    ++outer_total;
    if (F32 && outer > 0) {
      // refinement: the FP64 residual of the updated solution
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (tid + j * bd < nown) XF[tid + j * bd] = xs[j];
      exchange<double>(ph, push0, ct.npush, XF, kXF, ct.nhalo * 8);
      double s1[1] = {0.0};
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (tid + j * bd < nloc) {
          const double de = a.dextra ? a.dextra[r0 + tid + j * bd] : 0.0;
          r64[j] = b[j] - (de * xs[j] +
                           slice_dot<double, double>(lcol + at[j], a.valA + ct.ent0 + at[j], 0, st[j], XF));
          s1[0] += r64[j] * r64[j];
        }
      const int k = next_sum();
      ph.learn(sum_f64<1>(ph, k, k - kSum0, s1, stage, partd, iC, irank, [&](const double (&t)[1]) { decide(t[0]); }));
    }
    if (!ph.ok()) break;
    const int code = s_code;
    if (code != 0) {
      if (code == 1) fail = ST_NONFINITE;
      if (code == 3 && a.max_outer > 1) fail = ST_NOT_CONVERGED;
      break;
    }
    const double scale = s_d[3], inv_scale = s_d[4];
    const T target2 = T(s_d[5]);
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      r[j] = F32 ? T(r64[j] * inv_scale) : T(r64[j]);
      d[j] = p[j] = q[j] = T(0);
    }
    int it = 0;
    if (F32 && !AMG && a.max_outer == 1) {
      // ---- pipelined Jacobi-CG (mixed.cu): one phase an iteration --------------
      if constexpr (F32 && !AMG) {
        float u[RPT], w[RPT], zz[RPT], s[RPT], mm[RPT];
        float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          u[j] = invd[j] * r[j];
          put0(j, ZR, u[j]);
        }
        exchange0(ZR, kRes);
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          w[j] = mm[j] = zz[j] = s[j] = 0.f;
          if (tid + j * bd < nloc) {
            w[j] = dx[j] * u[j] + row_dot(j, ZR);
            mm[j] = invd[j] * w[j];
            acc[0] += r[j] * u[j];
            acc[1] += w[j] * u[j];
            acc[2] += r[j] * r[j];
          }
          put0(j, X0, mm[j]);
        }
        const int bytes = nparts * 16 + halo0;
        sum_f32_send(ph, kRed, 0, acc, partf, iC, irank, nw);
        exchange<T>(ph, push0, ct.npush, X0, kRed, bytes);
        float gam_prev = 1.f, alpha_prev = 1.f;
        for (;;) {
          const int odd = it & 1;
          if (!ph.ok()) break;
          float t[3];
          sum_f32_get(odd, t, partf, nparts);
          const float gam = t[0], del = t[1], rr = t[2];
          if (!isfinite(rr) || !isfinite(gam) || !isfinite(del)) {
            fail = ST_NONFINITE;
            break;
          }
          if (!(rr > target2)) break;
          if (it >= a.inner_cap) {
            fail = ST_NOT_CONVERGED;
            break;
          }
          const float beta = it == 0 ? 0.f : gam / gam_prev;
          const float den = it == 0 ? del : del - beta * gam / alpha_prev;
          if (!(den > 0.f)) {
            if (!isfinite(den)) fail = ST_NONFINITE;
            break;   // FP32 breakdown: keep d
          }
          const float alpha = gam / den;
          const T* const mc = odd ? ZR : X0;
          T* const mn = odd ? X0 : ZR;
          const int kn = odd ? kRed : kRed2;
          acc[0] = acc[1] = acc[2] = 0.f;
#pragma unroll
          for (int j = 0; j < RPT; ++j) {
            if (tid + j * bd < nloc) {
              const float ni = dx[j] * mm[j] + row_dot(j, mc);
              // beta = 0 on the first pass: the recurrences start from n, m, w, u
              zz[j] = ni + beta * zz[j];
              q[j] = mm[j] + beta * q[j];
              s[j] = w[j] + beta * s[j];
              p[j] = u[j] + beta * p[j];
              d[j] += alpha * p[j];
              r[j] -= alpha * s[j];
              u[j] -= alpha * q[j];
              w[j] -= alpha * zz[j];
              mm[j] = invd[j] * w[j];
              acc[0] += r[j] * u[j];
              acc[1] += w[j] * u[j];
              acc[2] += r[j] * r[j];
            }
            put0(j, mn, mm[j]);
          }
          sum_f32_send(ph, kn, odd ^ 1, acc, partf, iC, irank, nw);
          exchange<T>(ph, push0, ct.npush, mn, kn, bytes);
          gam_prev = gam;
          alpha_prev = alpha;
          ++it;
        }
      }
    } else {
      // ---- preconditioned CG on A d = r, one reduction an iteration ----------------
      T rho = T(0), alpha = T(0), beta = T(0);   // FP64: rho kept by thread 0
      for (bool first = true;; first = false) {
        // z = M^-1 r
        if constexpr (AMG) {
          T x0[RPT];
          T* const bc = reinterpret_cast<T*>(sm + M.bc);
          T* const xc = reinterpret_cast<T*>(sm + M.xc);
          {
            const T om0 = F32 ? T(H.L[0].omega32) : T(H.L[0].omega);
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
              x0[j] = om0 * invd[j] * r[j];
              put0(j, X0, x0[j]);
            }
          }
          exchange0(X0, kX0);
#pragma unroll
          for (int j = 0; j < RPT; ++j)
            if (tid + j * bd < nloc) put0(j, ZR, r[j] - row_dot(j, X0));
          exchange0(ZR, kRes);
          for (int l = 0; l + 1 < H.nlev; ++l) {
            const T* rl = l == 0 ? ZR : reinterpret_cast<const T*>(sm + M.lv[l][2]);
            const ResLevel& N = H.L[l + 1];
            T* const nb = reinterpret_cast<T*>(sm + M.lv[l + 1][0]);
            T* const nx = reinterpret_cast<T*>(sm + M.lv[l + 1][1]);
            T* const ny = reinterpret_cast<T*>(sm + M.lv[l + 1][2]);
            const T om = F32 ? T(N.omega32) : T(N.omega);
            const T* id = reinterpret_cast<const T*>(img + N.off_invd);
            const uint32_t* pw = reinterpret_cast<const uint32_t*>(img + N.off_push);
            op_rows<T>(H.L[l].R, img, rl, [&](int row, T v, int sub) {
              if (sub != 0) return;
              nb[row] = v;
              nx[row] = om * id[row] * v;
            });
            exchange<T>(ph, pw, N.npush, nx, kLev + 4 * l, N.nhalo * int(sizeof(T)));
            op_rows<T>(N.A, img, nx, [&](int row, T v, int sub) {
              if (sub == 0) ny[row] = nb[row] - v;
            });
            exchange<T>(ph, pw, N.npush, ny, kLev + 4 * l + 1, N.nhalo * int(sizeof(T)));
          }
          {   // restriction onto the coarsest level, gathered whole by every block
            const T* rl = H.nlev == 1 ? ZR : reinterpret_cast<const T*>(sm + M.lv[H.nlev - 1][2]);
            op_rows<T>(H.L[H.nlev - 1].R, img, rl, [&](int row, T v, int sub) {
              if (sub == 0) bc[H.c0 + row] = v;
            });
            if (tid < iC) ph.send(s_tok + irank, unsigned(tid), 0.f, kBc);
            gather_all<T>(ph, bc, H.c0, H.ncown, iC, kBc, (F32 ? a.ldc : H.nc) * int(sizeof(T)) + iC * 4);
          }
          {   // coarsest level: rows of the dense inverse against the gathered right-hand side
            using V = typename std::conditional<F32, float4, double2>::type;
            constexpr int E = 16 / int(sizeof(T));
            int g = 8;
            while (g < 32 && H.ncown * 2 * g <= bd) g *= 2;
            const int nvec = a.nc / E, sub = lane & (g - 1);
            for (int i0 = (tid >> 5) * (32 / g); i0 < H.ncown; i0 += nw * (32 / g)) {
              const int i = i0 + lane / g;
              T s = T(0);
              if (i < H.ncown) {
                const T* row = static_cast<const T*>(a.cinv) + size_t(H.c0 + i) * a.ldc;
#pragma unroll 4
                for (int v = sub; v < nvec; v += g) {
                  const V cv = __ldg(reinterpret_cast<const V*>(row) + v);
                  const T* ce = reinterpret_cast<const T*>(&cv);
#pragma unroll
                  for (int e = 0; e < E; ++e) s += ce[e] * bc[v * E + e];
                }
                if (sub < a.nc - nvec * E) s += row[nvec * E + sub] * bc[nvec * E + sub];
              }
#pragma unroll 1
              for (int o = g >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
              if (i < H.ncown && sub == 0) xc[H.c0 + i] = s;
            }
            gather_all<T>(ph, xc, H.c0, H.ncown, iC, kXc, (F32 ? a.ldc : H.nc) * int(sizeof(T)));
          }
          for (int l = H.nlev - 1; l >= 1; --l) {
            const ResLevel& N = H.L[l];
            T* const nb = reinterpret_cast<T*>(sm + M.lv[l][0]);
            T* const nx = reinterpret_cast<T*>(sm + M.lv[l][1]);
            T* const ny = reinterpret_cast<T*>(sm + M.lv[l][2]);
            const T om = F32 ? T(N.omega32) : T(N.omega);
            const T* id = reinterpret_cast<const T*>(img + N.off_invd);
            const uint32_t* pw = reinterpret_cast<const uint32_t*>(img + N.off_push);
            const T* cy = l + 1 == H.nlev ? xc : reinterpret_cast<const T*>(sm + M.lv[l + 1][2]);
            op_rows<T>(N.P, img, cy, [&](int row, T v, int sub) {
              if (sub == 0) nx[row] += v;
            });
            exchange<T>(ph, pw, N.npush, nx, kLev + 4 * l - 2, N.nhalo * int(sizeof(T)));
            op_rows<T>(N.A, img, nx, [&](int row, T v, int sub) {
              if (sub == 0) ny[row] = nx[row] + om * id[row] * (nb[row] - v);
            });
            exchange<T>(ph, pw, N.npush, ny, kLev + 4 * l - 1, N.nhalo * int(sizeof(T)));
          }
          {
            const ResOp& P = H.L[0].P;
            const uint32_t* sl = reinterpret_cast<const uint32_t*>(img + P.off_slice);
            const uint16_t* pc = reinterpret_cast<const uint16_t*>(img + P.off_col);
            const T* pvl = reinterpret_cast<const T*>(img + P.off_val);
            const T* cy = H.nlev == 1 ? xc : reinterpret_cast<const T*>(sm + M.lv[1][2]);
#pragma unroll
            for (int j = 0; j < RPT; ++j)
              if (tid + j * bd < nloc) {
                const uint32_t w = sl[(tid + j * bd) >> 5];
                const int pa = int(w >> 12) * 32 + lane;
                x0[j] += slice_dot<T, T>(pc + pa, pvl + pa, 0, int(w & 4095u), cy);
                put0(j, X0, x0[j]);
              }
          }
          exchange0(X0, kX0b);
          const T om0 = F32 ? T(H.L[0].omega32) : T(H.L[0].omega);
#pragma unroll
          for (int j = 0; j < RPT; ++j)
            if (tid + j * bd < nloc) {
              z[j] = x0[j] + om0 * invd[j] * (r[j] - row_dot(j, X0));
              put0(j, ZR, z[j]);
            }
        } else {
#pragma unroll
          for (int j = 0; j < RPT; ++j) {
            z[j] = invd[j] * r[j];
            put0(j, ZR, z[j]);
          }
        }
        exchange0(ZR, kZ);
        // w = A z; (r, z), (w, z), (r, r)
        T w[RPT], t3[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          w[j] = T(0);
          if (tid + j * bd < nloc) {
            w[j] = dx[j] * z[j] + row_dot(j, ZR);
            t3[0] += r[j] * z[j];
            t3[1] += w[j] * z[j];
            t3[2] += r[j] * r[j];
          }
        }
        if (!first) ++it;
        if constexpr (F32) {
          const int turn = turns32.next(), k = kRed + turn;
          const int gone = ph.meet();   // the products' vector is read
          ph.expect(k, nparts * 16);
          sum_f32_send(ph, k, turn, t3, partf, iC, irank, nw);
          ph.learn(gone);
          if (!ph.ok()) break;
          ph.wait(k);
          sum_f32_get(turn, t3, partf, nparts);
          const T rz = t3[0], rr = t3[2];
          if (first) {
            if (!(rr > target2)) break;      // includes b = 0
          } else {
            if (!isfinite(rr) || !isfinite(rz)) {
              fail = ST_NONFINITE;
              break;
            }
            if (rr <= target2) break;
            if (it >= a.inner_cap) {
              if (a.max_outer == 1) fail = ST_NOT_CONVERGED;
              break;
            }
            beta = rz / rho;
          }
          const T den = first ? t3[1] : t3[1] - beta * rz / alpha;
          if (!(den > T(0))) {
            if (!isfinite(den)) fail = ST_NONFINITE;
            break;                           // FP32 breakdown: keep d, the outer step decides
          }
          rho = rz;
          alpha = rz / den;
        } else {
          double (&td)[3] = reinterpret_cast<double (&)[3]>(t3);
          // s_code: 0 go on, -1 converged, else the failure
          const int k = next_sum();
          const int gone = sum_f64<3>(ph, k, k - kSum0, td, stage, partd, iC, irank, [&](const double (&t)[3]) {
            s_code = first ? (!(t[2] > s_d[2]) ? -1 : 0)   // includes b = 0
                     : !isfinite(t[2]) || !isfinite(t[0]) ? ST_NONFINITE
                     : t[2] <= s_d[2]                     ? -1
                     : it >= a.inner_cap                  ? ST_NOT_CONVERGED
                                                          : 0;
            if (s_code == 0) {
              const double be = first ? 0.0 : t[0] / rho;
              const double den = first ? t[1] : t[1] - be * t[0] / alpha;
              if (!(den > 0.0)) s_code = isfinite(den) ? ST_INDEFINITE : ST_NONFINITE;
              s_d[4] = be;
              s_d[3] = t[0] / den;
              rho = t[0];
            }
          });
          const int next = s_code;
          beta = s_d[4];
          alpha = s_d[3];
          ph.learn(gone);
          if (!ph.ok()) break;
          if (next != 0) {
            fail = next > 0 ? next : 0;
            break;
          }
        }
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          p[j] = z[j] + beta * p[j];         // beta = 0 on the first pass
          q[j] = w[j] + beta * q[j];
          d[j] += alpha * p[j];
          r[j] -= alpha * q[j];
        }
      }
    }
    inner_total += it;
    if ((fail && F32) || !ph.ok()) break;
#pragma unroll
    for (int j = 0; j < RPT; ++j) xs[j] += F32 ? scale * double(d[j]) : double(d[j]);
    if (!F32 || a.max_outer == 1) break;
  }

  // ---- normalisation of the singular elliptic solution -------------------------
  double shift = 0.0;
  if (a.pin >= 0) {
    const int at_pin = a.pin - r0;
    if (at_pin >= 0 && at_pin < nloc)
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (tid + j * bd == at_pin)
#pragma unroll 1
          for (unsigned c = 0; c < C; ++c) ph.send(&s_pin, c, xs[j], kPin);
    ph.expect(kPin, 8);
    ph.wait(kPin);
    shift = s_pin;
  } else if (a.pin == -1) {
    double s1[1] = {0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (tid + j * bd < nloc) s1[0] += xs[j];
    const int k = next_sum();
    ph.learn(sum_f64<1>(ph, k, k - kSum0, s1, stage, partd, iC, irank,
                        [&](const double (&t)[1]) { s_d[0] = t[0] / double(a.n); }));
    shift = s_d[0];
  }
  if (ph.sync()) {
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (tid + j * bd < nloc) a.x[r0 + tid + j * bd] = xs[j] - shift;
  }
  if (rank == 0 && tid == 0) {
    if (fail) atomicOr(a.status, fail);
    if (a.iters_acc) atomicAdd((unsigned long long*)a.iters_acc, (unsigned long long)inner_total);
    if (a.outer_acc && F32) atomicAdd((unsigned long long*)a.outer_acc, (unsigned long long)outer_total);
    if (a.solves_acc) atomicAdd((unsigned long long*)a.solves_acc, 1ull);
  }
  // after an expiry, messages of this block may still be on their way to blocks
  // that wait for nothing any more; they land in a few microseconds
  if (!ph.ok()) {
    const unsigned long long t0 = device_ns();
    for (int n = 0; n < 100000 && device_ns() - t0 < kDrainNs; ++n) __nanosleep(100);
  }
  __syncwarp();
  cluster_barrier();   // no block leaves while a peer may still send to it
}

#undef ZR
#undef X0
#undef XF
#undef stage
#undef partd
#undef partf
#undef img
#undef H

using ResKernel = void (*)(const ResPair, const ResLaunch*);
template <class T, bool AMG>
ResKernel kernel_rpt(int rpt) {
  return rpt == 1   ? res_kernel<T, 1, AMG>
         : rpt == 2 ? res_kernel<T, 2, AMG>
         : rpt == 3 ? res_kernel<T, 3, AMG>
                    : res_kernel<T, 4, AMG>;
}
ResKernel kernel_of(const ResShape& s, bool f32, bool amg) {
  if (f32) return amg ? kernel_rpt<float, true>(s.rpt) : kernel_rpt<float, false>(s.rpt);
  return amg ? kernel_rpt<double, true>(s.rpt) : kernel_rpt<double, false>(s.rpt);
}

void config_of(const ResShape& s, bool f32, bool amg, int nsys, cudaStream_t st, cudaLaunchConfig_t* cfg,
               cudaLaunchAttribute* at) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3(unsigned(nsys * s.C));
  cfg->blockDim = dim3(unsigned(s.block));
  cfg->dynamicSmemBytes = res_smem_bytes(s, f32, amg);
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = unsigned(s.C);
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

}  // namespace

size_t res_smem_bytes(const ResShape& s, bool f32, bool amg) {
  ResMem m;
  res_mem(s, s.img0, amg ? s.imgA[f32 ? 0 : 1] : 0, s.block, f32 ? 4 : 8, amg, &m);
  return size_t(m.total);
}

bool res_prepare(const ResShape& s, bool f32, bool amg) {
  const ResKernel k = kernel_of(s, f32, amg);
  int dev = 0, most = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, k) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (res_smem_bytes(s, f32, amg) + fa.sharedSizeBytes > size_t(most)) return false;
  int clusters = 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  config_of(s, f32, amg, 1, nullptr, &cfg, &at);
  // the limit is the kernel's, not the launch's: allow what the device has
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most - int(fa.sharedSizeBytes)) != cudaSuccess ||
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return clusters >= 1;
}

cudaError_t res_solve(const ResShape& s, bool f32, bool amg, const ResLaunch* host, int nsys, const ResLaunch* tab,
                      size_t smem, cudaStream_t st) {
  if (nsys < 1 || (!tab && (nsys > 2 || !host))) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at;
  config_of(s, f32, amg, nsys, st, &cfg, &at);
  if (smem > 0) cfg.dynamicSmemBytes = smem;
  ResPair pr{};
  if (!tab)
    for (int k = 0; k < nsys; ++k) pr.a[k] = host[k];
  return cudaLaunchKernelEx(&cfg, kernel_of(s, f32, amg), pr, tab);
}

}  // namespace bd
