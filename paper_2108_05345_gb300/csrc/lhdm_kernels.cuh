// lhdm_kernels.cuh -- what the kernels and the host side of the C ABI
// share: the batch descriptor, the scratch layout and the kernel
// declarations.  Each kernel is compiled in a translation unit of its own
// (lhdm_grid_solve.cu, lhdm_batch_solve.cu, their _tall forms,
// lhdm_backward.cu) so the library builds in parallel.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "lhdm.h"
#include "lhdm_solve.cuh"

namespace lhdm {

// Per-instance descriptor of a batch (device array).
struct BatchItem {
  int m, n, lda, cap, ldr, k_max;
  const double* A;
  const double* b;
  double* x;
  int* passive;
  lhdm_info* info;
  double* R;
  int* rslot;
  int* order;
  double* xP;
  double* r;
  int* nP;
  const double* g;   // adjoint inputs/outputs (set per backward call)
  double* dLdb;
  double* dLdA;
  int ld_dA;
};

// Offsets of one team's scratch inside a double region and an int region.
struct ScratchLayout {
  size_t W, bt, yP, rhs, rres, w, u, anorm, V, vtop, beta, T, R22, Gm, yJ, pr, part, pacc, candw, rotc, rots, apu;
  size_t Dinv, accb;  // pipelined triangular solve (teams of more than one CTA)
  size_t dtotal;
  size_t Vd;  // reflector digits of the tensor-core commit
  size_t pos, J, candi, candn, ipart, ctl, qlist, tflag, Ver, csign;
  size_t itotal;
  int ldw;
  bool pipelined;
};

inline size_t up8(size_t x) { return (x + 31) & ~(size_t)31; }  // 256-byte granules of doubles/ints

inline ScratchLayout make_layout(int max_m, int max_n, int team) {
  ScratchLayout L;
  const int m = std::max(max_m, 1), n = std::max(max_n, 1);
  const int cap = std::max(std::min(max_m, max_n), 1);
  L.ldw = (m + 1) & ~1;
  size_t o = 0;
  auto take = [&](size_t cnt) { size_t r = o; o += up8(std::max<size_t>(cnt, 1)); return r; };
  L.W = take((size_t)L.ldw * n);
  L.bt = take(m);
  L.yP = take(cap);
  L.rhs = take(std::max(m, cap));
  L.rres = take(team > 1 ? cap : 1);
  L.w = take(n);
  L.u = take(n);
  L.anorm = take(n);
  L.V = take((size_t)m * KM);
  L.vtop = take(KM);
  L.beta = take(KM);
  L.T = take(KM * KM);
  L.R22 = take(KM * KM);
  L.Gm = take(KM * KM);
  L.yJ = take(KM);
  L.pr = take(KM);
  L.part = take((size_t)team * PW);
  L.pacc = take(3 * PACC_W);
  L.candw = take((size_t)team * KM);
  L.rotc = take(cap);
  L.rots = take(cap);
  L.apu = take(m);
  // diagonal-block inverses and slab accumulators of the pipelined solve
  const size_t nbk = (size_t)(cap + TB - 1) / TB;
  L.pipelined = team > 1;
  L.Dinv = take(L.pipelined ? nbk * TB * TB : 1);
  L.accb = take(L.pipelined ? nbk * TB : 1);
  L.Vd = take((size_t)(m + 32) * ND * KM / 4);  // whole row groups, ND x KM bf16 per row
  L.dtotal = o;
  o = 0;
  L.pos = take(n);
  L.J = take(KM);
  L.candi = take((size_t)team * KM);
  L.candn = take(team);
  L.ipart = take((size_t)team * 8);
  L.ctl = take(16);
  L.qlist = take(cap);
  L.tflag = take(L.pipelined ? nbk * (1 + TB / SLAB + INV_PARTS) : 1);
  L.Ver = take(m + 64);  // pass 1 of the commit reads whole chunks of up to 64 rows
  L.csign = take(n);
  L.itotal = o;
  return L;
}

inline __host__ __device__ void bind_scratch(Inst& I, const ScratchLayout& L, double* d, int* ip) {
  I.ldw = L.ldw;
  I.W = d + L.W;
  I.bt = d + L.bt;
  I.yP = d + L.yP;
  I.rhs = d + L.rhs;
  I.rres = d + L.rres;
  I.Rinv = nullptr;
  I.w = d + L.w;
  I.u = d + L.u;
  I.anorm = d + L.anorm;
  I.V = d + L.V;
  I.vtop = d + L.vtop;
  I.beta = d + L.beta;
  I.T = d + L.T;
  I.R22 = d + L.R22;
  I.Gm = d + L.Gm;
  I.yJ = d + L.yJ;
  I.pr = d + L.pr;
  I.part = d + L.part;
  I.pacc = reinterpret_cast<long long*>(d + L.pacc);
  I.candw = d + L.candw;
  I.rotc = d + L.rotc;
  I.rots = d + L.rots;
  I.pos = ip + L.pos;
  I.J = ip + L.J;
  I.candi = ip + L.candi;
  I.candn = ip + L.candn;
  I.ipart = ip + L.ipart;
  I.ctl = ip + L.ctl;
  I.qlist = ip + L.qlist;
  I.csign = ip + L.csign;
  I.Dinv = L.pipelined ? d + L.Dinv : nullptr;
  I.accb = L.pipelined ? d + L.accb : nullptr;
  I.tflag = L.pipelined ? ip + L.tflag : nullptr;
  I.Vd = reinterpret_cast<unsigned*>(d + L.Vd);
  I.Ver = ip + L.Ver;
  I.amask = nullptr;
  I.wait_ns = WAIT_NS;
  I.bar_extra = 0;
  I.guard_force = 0;
  I.inject = 0;
}

// CTA barriers and tensor memory of the tensor-core commit (every thread of
// the CTA, once per kernel; the memory is freed by tc_close).
struct TcState {
  unsigned long long* mbs;
  unsigned tmem;
};
constexpr int TC_BARS = 18;
inline __device__ void tc_barriers(unsigned long long* mb) {
  if (threadIdx.x == 0) {
    // V's copies and MMA completions: one arrival; pass-1 slots: C digits
    // worth 8; accumulator reads and a failed commit's MMAs: one per warp
    for (int i = 0; i < TC_BARS; ++i) mbar_init(mb + i, i < 5 ? 1 : i < 10 ? 8 : i < 15 ? 1 : NW);
    fence_mbar_init();
  }
}
inline __device__ TcState tc_open() {
  __shared__ unsigned long long s_mb[TC_BARS];
  __shared__ unsigned s_tmem;
  if (threadIdx.x < 32) tmem_alloc(&s_tmem);
  tc_barriers(s_mb);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return TcState{s_mb, s_tmem};
}
// after a wait ran out (and the commit has drained what was in flight):
// fresh barriers for the CTA's next instance
inline __device__ void tc_reset(const TcState& t) {
  __syncthreads();
  if (threadIdx.x == 0)
    for (int i = 0; i < TC_BARS; ++i) mbar_inval(t.mbs + i);
  tc_barriers(t.mbs);
  __syncthreads();
}
inline __device__ void tc_close(const TcState& t) {
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_free(t.tmem);
}

inline __device__ void bind_item(Inst& I, const BatchItem& it) {
  I.m = it.m;
  I.n = it.n;
  I.lda = it.lda;
  I.cap = it.cap;
  I.ldr = it.ldr;
  I.A = it.A;
  I.b = it.b;
  I.x_out = it.x;
  I.passive_out = it.passive;
  I.info_out = it.info;
  I.R = it.R;
  I.rslot = it.rslot;
  I.order = it.order;
  I.xP = it.xP;
  I.r = it.r;
  I.nP_out = it.nP;
  I.prm.k_max = it.k_max;
}

// One solve on the whole GPU.
template <bool TALL>
__device__ __forceinline__ void solve_on_grid(const Inst& I, unsigned int* bar, int* err, double* dyn) {
  GridTeam tm{(int)blockIdx.x, (int)gridDim.x, bar, err, I.wait_ns, I.bar_extra};
  Engine<GridTeam, TALL> e(tm, I, dyn);
  const TcState tc = tc_open();
  e.mbs = tc.mbs;
  e.tmem = tc.tmem;
  e.run();
  tc_close(tc);
}

// Many instances in one persistent launch: each CTA takes the next instance
// (largest first) from a device queue and solves it alone.
template <bool TALL>
__device__ __forceinline__ void solve_queue(const BatchItem* items, const int* perm, int batch, int* queue,
                                            const ScratchLayout& L, double* dscr, int* iscr, const DevParams& prm,
                                            double* dyn) {
  __shared__ int s_k;
  Inst I;
  bind_scratch(I, L, dscr + (size_t)blockIdx.x * L.dtotal, iscr + (size_t)blockIdx.x * L.itotal);
  I.phase_ns = nullptr;
  I.trace = nullptr;
  I.trace_cap = 0;
  const TcState tc = tc_open();
  unsigned mpar = 0u;  // parities of tc's barriers, from instance to instance
  for (;;) {
    if (threadIdx.x == 0) s_k = atomicAdd(queue, 1);
    __syncthreads();
    const int k = s_k;
    __syncthreads();
    if (k >= batch) break;
    const BatchItem it = items[perm[k]];
    I.prm = prm;
    bind_item(I, it);
    CtaTeam tm{0, 1};
    Engine<CtaTeam, TALL> e(tm, I, dyn);
    e.mbs = tc.mbs;
    e.tmem = tc.tmem;
    e.mpar = mpar;
    e.run();
    mpar = e.mpar;
    if (e.tc_failed) {
      tc_reset(tc);
      mpar = 0u;
    }
    __syncthreads();
  }
  tc_close(tc);
}

}  // namespace lhdm

// One solve on the whole GPU: one CTA per SM, cooperative launch; the second
// for more than TALL_ROWS rows.
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_solve_grid_kernel(lhdm::Inst I, unsigned int* bar, int* err);
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_solve_grid_tall_kernel(lhdm::Inst I, unsigned int* bar, int* err);
// Adjoint of a solve on the whole GPU (cooperative launch).
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_backward_grid_kernel(lhdm::Inst I, unsigned int* bar, int* err,
                                                                         const double* g, double* dLdb,
                                                                         double* dLdA, int ld_dA, double* apu);
// Many instances in one persistent launch, one instance per CTA at a time; the
// second when any has more than TALL_ROWS rows.
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_solve_batch_kernel(const lhdm::BatchItem* items,
                                                                       const int* perm, int batch, int* queue,
                                                                       lhdm::ScratchLayout L, double* dscr,
                                                                       int* iscr, lhdm::DevParams prm);
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_solve_batch_tall_kernel(const lhdm::BatchItem* items,
                                                                            const int* perm, int batch, int* queue,
                                                                            lhdm::ScratchLayout L, double* dscr,
                                                                            int* iscr, lhdm::DevParams prm);
__global__ void __launch_bounds__(lhdm::NT, 1) lhdm_backward_batch_kernel(const lhdm::BatchItem* items,
                                                                          const int* perm, int batch, int* queue,
                                                                          lhdm::ScratchLayout L, double* dscr,
                                                                          int* iscr);
