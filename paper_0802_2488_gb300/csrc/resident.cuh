// Resident schedule of the two passes: one cooperative launch runs whole
// solves of a small or medium lattice.
//
// In the two-pass loop an iteration of such a lattice costs two launches and
// the serial tail of the row pass (arrival of every CTA, sums and state
// machine in the last one), 16 - 35 us against the few us of work its CTAs
// share.  Here G CTAs (a power of two) stay on the GPU for a solve and do its
// rows and columns in turn, by the same device functions as the passes
// (row_unit, col_unit) and therefore with the same bits; between the phases
// they meet at a barrier of the solve's own, a counter in global memory
// (about 1.2 us with all CTAs of the GPU at it).  The state machine runs in every CTA on a copy of the solve in shared
// memory, from the same sums in the same order, so nothing has to be handed
// out; and it runs off the critical path: after the row phase a CTA first
// does its columns of the next iteration on the assumption that there is one
// (when the increment turns out to be finished the warm start overwrites the
// spectrum), arrives at the barrier, and only then sums the row phase's
// records and advances the state while the others arrive.
//
// Hazards: spectrum and stress are read by other CTAs only after the barrier
// that follows their writes, past the L1 or after the acquire of that barrier;
// a stress or strain buffer is rewritten one iteration (two barriers) after
// its last reader; the sums' records alternate between two buffers, and a CTA
// passes the barrier after its sums before any CTA writes that buffer again.
// Measured, one lattice, us an iteration against the two-pass loop: FP32 L = 16
// 9.0 / 17.8, 64 9.8 / 20.3, 128 10.7 / 23.3, 256 16.6 / 25.9, 512 25.5 / 31.3;
// FP64 L = 16 21.2 / 31.9, 64 22.2 / 29.3, 128 25.8 / 33.3 (bound by chains of FP64
// instructions, 64 clocks each).
//
// Every CTA of a launch is resident at once (cooperative launch), and every
// wait is bounded: when it runs out the solve stops with the batch's
// timed_out set.
#pragma once
#include "passes.cuh"

namespace epfft {

template <typename T, int L, int V>
struct ResCfg {
  using C = Cfg<T, L, V>;
  static constexpr int NT = C::NT_ROW;
  // 128 registers a thread for FP32 from 256 threads on (two CTAs per SM)
  static constexpr int MINB = !C::F64 && NT >= 256 ? 2 : 1;
  static constexpr int DATA = C::ROW_DATA > C::COL_DATA ? C::ROW_DATA : C::COL_DATA;
  // tile | row stage table | twist octant | column stage table
  static constexpr int OFF_RT = DATA, OFF_CT = DATA + C::ROW_TW + C::TB::OCT;
  // then the CTA's copy of the solve
  static constexpr size_t OFF_S = ((size_t)(OFF_CT + C::COL_TW) * sizeof(C2<T>) + 15) / 16 * 16;
  static constexpr size_t SMEM = OFF_S + sizeof(Solve);
  static_assert(SMEM <= 222000, "shared memory per CTA");
  static_assert(C::grp(3 * C::W, L, NT) * L <= 16 * NT, "elements per thread and stage");
};

constexpr int RES_POLLS = 1 << 22;  // of a barrier's wait: some seconds

// Counts this CTA in at the solve's barrier (every thread's writes before it).
__device__ __forceinline__ void res_arrive(unsigned* ctr) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
}
// Waits until `target` arrivals; false when the wait ran out.  *ok: shared.
__device__ __forceinline__ bool res_wait(const unsigned* ctr, unsigned target, int* ok) {
  if (threadIdx.x == 0) {
    int n = 0;
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    } while ((int)(v - target) < 0 && ++n < RES_POLLS);
    *ok = (int)(v - target) >= 0;
  }
  __syncthreads();
  return *ok != 0;
}

// The phases' work as functions of their own, so that the compiler keeps no
// address of theirs in registers across the loop (inlined, the loop took 255
// registers and spilled).
template <typename T, int L, int V>
__device__ __noinline__ void res_row(int phase, int cur, int inc, int u, double* pt) {
  using R = ResCfg<T, L, V>;
  extern __shared__ __align__(16) unsigned char smraw[];
  C2<T>* sp = reinterpret_cast<C2<T>*>(smraw);
  const Solve& S = *reinterpret_cast<const Solve*>(smraw + R::OFF_S);
  row_unit<T, L, V, true>(S, S.Eprev, phase, cur, inc, u, sp, nullptr, sp + R::OFF_RT, pt);
}
template <typename T, int L, int V, bool GEN>
__device__ __noinline__ void res_col(int inc, int b, const C2<T>* ktab) {
  using R = ResCfg<T, L, V>;
  extern __shared__ __align__(16) unsigned char smraw[];
  C2<T>* sp = reinterpret_cast<C2<T>*>(smraw);
  const Solve& S = *reinterpret_cast<const Solve*>(smraw + R::OFF_S);
  col_unit<T, L, V, GEN, R::NT, true>(S, inc, b, sp, nullptr, sp + R::OFF_CT, ktab, []() {});
}

// Grid: (G, solves), cooperative.  part2: the second buffer of partial sums
// (L / RR records per solve); bars: one zeroed counter per solve, 32 words
// apart.  bound: as in the loop (BatchCtl::max_body_iters).
template <typename T, int L, int V, bool GEN>
__global__ void __launch_bounds__(ResCfg<T, L, V>::NT, ResCfg<T, L, V>::MINB)
solve_resident(Solve* __restrict__ solves, BatchCtl* bc, double* part2, unsigned* bars, const C2<T>* __restrict__ tw,
               const C2<T>* __restrict__ ktab) {
  using R = ResCfg<T, L, V>;
  using C = typename R::C;
  constexpr int NT = R::NT, NREC = L / C::RR, NCOL = C::M / C::W;
  extern __shared__ __align__(16) unsigned char smraw[];
  C2<T>* sp = reinterpret_cast<C2<T>*>(smraw);
  __shared__ double tot[N_ACC];
  __shared__ int ok;
  Solve& S = *reinterpret_cast<Solve*>(smraw + R::OFF_S);
  Solve* G = solves + blockIdx.y;
  const int tid = threadIdx.x, g = blockIdx.x, ng = gridDim.x;
  unsigned* ctr = bars + 32 * blockIdx.y;
  if (!ECHK(blockDim.x - 1, NT, 90) || !ECHK(ng - 1, NREC, 90)) return;
  static_assert(sizeof(Solve) % 4 == 0, "copied in words");
  for (int i = tid; i < (int)(sizeof(Solve) / 4); i += NT)
    reinterpret_cast<unsigned*>(&S)[i] = reinterpret_cast<const unsigned*>(G)[i];
  copy_table<T, NT>(sp + R::OFF_RT, tw + C::TB::off_row(V), C::ROW_TW);
  copy_table<T, NT>(sp + R::OFF_RT + C::ROW_TW, tw, C::TB::OCT);
  copy_table<T, NT>(sp + R::OFF_CT, tw + C::TB::off_col(V), C::COL_TW);
  cp_async_wait_all();
  __syncthreads();
  double* const part[2] = {S.partials, part2 + (size_t)blockIdx.y * NREC * PART_STRIDE};
  const int64_t bound = bc->max_body_iters;
  unsigned met = 0;  // barriers passed
  int64_t step = 0;
  bool late = false;
  while (S.phase != PH_DONE) {
    if (step >= bound) {
      late = true;
      break;
    }
    const int phase = S.phase, cur = S.cur, inc = S.inc;
    double* const pt = part[step & 1];
    for (int u = g; u < NREC; u += ng) {
      res_row<T, L, V>(phase, cur, inc, u, pt);
      __syncthreads();  // the unit's tile and reductions, before the next unit
    }
    step++;
    if (phase == PH_FINAL) {
      __syncthreads();
      if (tid == 0) S.phase = PH_DONE;
      __syncthreads();
      break;
    }
    res_arrive(ctr);
    if (!res_wait(ctr, ++met * (unsigned)ng, &ok)) {
      late = true;
      break;
    }
    // the columns of the next iteration, if there is one
    for (int b = g; b < NCOL; b += ng) {
      res_col<T, L, V, GEN>(inc, b, ktab);
      __syncthreads();
    }
    res_arrive(ctr);
    // every record of the row phase was complete at the barrier above
    sum_partials<NT, NREC>(pt, tot);
    __syncthreads();
    if (tid == 0) finalize_solve<L>(S, phase, tot, g == 0);
    if (!res_wait(ctr, ++met * (unsigned)ng, &ok)) {
      late = true;
      break;
    }
  }
  if (tid == 0) {
    if (late) atomicOr(&bc->timed_out, 1);
    if (g == 0) {
      // the final state, and the batch's accounting
      G->phase = S.phase;
      G->inc = S.inc;
      G->iter = S.iter;
      G->cur = S.cur;
      G->status = S.status;
      G->total_iters = S.total_iters;
      atomicMax(reinterpret_cast<unsigned long long*>(&bc->body_iters), (unsigned long long)step);
      if (S.phase == PH_DONE) atomicSub(&bc->active, 1);
    }
  }
}

}  // namespace epfft
