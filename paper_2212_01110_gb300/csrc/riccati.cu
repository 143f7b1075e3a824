// Online projection on the tree dynamics S1 (Algorithm 2) with the factors
// of Algorithm 1 (factor.cpp).
//
// Backward pass, for every nonleaf node i from stage N-1 to 0, with
// q^j = -xbar^j at the leaves:
//   d^i = Rt^-1 (ubar^i - sum_c B^cT q^c)
//   q^i = K^iT (d^i - ubar^i) - xbar^i + W^i d^i + sum_c Abar^cT q^c
// (W^i = sum_c Abar^cT P^c B^c gathers the P^c B^c d^i terms of the paper's
// recursion); as read, q^i = E^iT g^i - K^iT ubar^i - xbar^i + sum_c Abar^cT q^c
// with g^i = ubar^i - sum_c B^cT q^c and E = Rt^-1 (K + W^T).  Forward pass from
// x^0 = x:
//   u^i = K^i x^i + d^i,   x^c = A^c x^i + B^c u^i = Abar^c x^i + B^c d^i.
//
// GB300 mapping.  One warp owns one node at a time.  Every factor is read
// exactly once per pass, with lanes over output entries so that each warp
// load instruction reads a contiguous row segment (coalesced) and the
// reduction index runs through registers; the small vectors (q, x, d, ubar)
// live in per-warp shared memory so any lane can broadcast-read any entry.
//   * chain kernels: below the "chain stage" every node has one child
//     (4096 chains of 15 nodes for the 62,805-node tree), so one warp walks
//     a whole chain, carrying q (backward) or x (forward) in shared memory
//     with no grid-wide synchronisation;
//   * stage kernels: above it (branching stages) one launch per stage, one
//     warp per node, children's q / parent's x exchanged through global
//     memory between launches.
// The backward layout [Abar^c | B^c] (nx x (nx+nu), row-major) serves
// h = [Abar^c | B^c]^T q^c; the forward layout is its transpose so that
// x^c = [Abar^c | B^c] (x; d) is again lanes-over-outputs.

#include "batch.cuh"
#include "kernels.cuh"
#include "riccati_body.cuh"
#include "spock_internal.h"

namespace spock {

template <typename S, int SL>
__global__ void __launch_bounds__(128) k_bwd_chain(KP<S> p) {
  bwd_chain_body<S, SL>(p, blockIdx.x, gridDim.x);
}

template <typename S, int SL>
__global__ void __launch_bounds__(128) k_bwd_stage(KP<S> p, int t) {
  bwd_stage_body<S, SL>(p, t, blockIdx.x, gridDim.x);
}

template <typename S, int SL>
__global__ void __launch_bounds__(128) k_fwd_stage(KP<S> p, int t, S* __restrict__ zo) {
  fwd_stage_body<S, SL>(p, t, zo, blockIdx.x, gridDim.x);
}

template <typename S, int SL>
__global__ void __launch_bounds__(128) k_fwd_chain(KP<S> p, S* __restrict__ zo) {
  fwd_chain_body<S, SL>(p, zo, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------------------
// launcher: the whole S1 projection (prep kernel already ran)
// ---------------------------------------------------------------------------
// staged kernels, a block per node sequence (riccati_seq.cu)
template <typename S>
int launch_bwd_seq(const KP<S>& p, int t_hi, int t_lo, int cnt, cudaStream_t st);
template <typename S>
int launch_fwd_seq(const KP<S>& p, int t_lo, int t_hi, int cnt, S* zo, cudaStream_t st);

// A single problem runs the staged sequence kernels; SPOCK_RICCATI_KERNELS =
// direct forces the direct ones of this file (the tests cover both), which
// the single-block solve and batches of very small problems use.
static bool direct_kernels() { return riccati_choice() == RK_DIRECT; }

// Launches both passes; ev (optional, 3 events) is recorded after the
// backward chain kernel, the backward stage kernels and the forward stage
// kernels.  Returns the number of kernels launched.
template <typename S, int SL>
static int riccati_passes_sl(const KP<S>& p, const std::vector<int32_t>& stage_begin, S* zo, cudaStream_t st,
                             cudaEvent_t* ev) {
  const int cs = p.chain_stage;
  int launches = 0;
  const bool chains = p.n_chains > 0 && cs < p.N;
  const int chain_grid = (p.n_chains + kWarpsPerBlock - 1) / kWarpsPerBlock;
  if (chains) {
    k_bwd_chain<S, SL><<<chain_grid, 128, 0, st>>>(p);
    ++launches;
  }
  if (ev) record_event(ev[0], st);
  for (int t = cs - 1; t >= 0; --t, ++launches) {
    const int cnt = stage_begin[t + 1] - stage_begin[t];
    k_bwd_stage<S, SL><<<(cnt + kWarpsPerBlock - 1) / kWarpsPerBlock, 128, 0, st>>>(p, t);
  }
  if (ev) record_event(ev[1], st);
  for (int t = 0; t < cs; ++t, ++launches) {
    const int cnt = stage_begin[t + 1] - stage_begin[t];
    k_fwd_stage<S, SL><<<(cnt + kWarpsPerBlock - 1) / kWarpsPerBlock, 128, 0, st>>>(p, t, zo);
  }
  if (ev) record_event(ev[2], st);
  if (chains) {
    k_fwd_chain<S, SL><<<chain_grid, 128, 0, st>>>(p, zo);
    ++launches;
  }
  return launches;
}

// The same with the sequence kernels: the chains with their leaves (or the
// leaves alone) in one launch, then the branching stages.
template <typename S>
static int riccati_passes_seq(const KP<S>& p, const std::vector<int32_t>& stage_begin, S* zo, cudaStream_t st,
                              cudaEvent_t* ev) {
  const int cs = p.chain_stage, top = cs > 0 ? cs : 1;
  auto cnt = [&](int t) { return (int)(stage_begin[t + 1] - stage_begin[t]); };
  int launches = launch_bwd_seq<S>(p, p.N, cs, cnt(cs), st);
  if (ev) record_event(ev[0], st);
  for (int t = cs - 1; t >= 0; --t) launches += launch_bwd_seq<S>(p, t, t, cnt(t), st);
  if (ev) record_event(ev[1], st);
  for (int t = 1; t < top; ++t) launches += launch_fwd_seq<S>(p, t, t, cnt(t), zo, st);
  if (ev) record_event(ev[2], st);
  return launches + launch_fwd_seq<S>(p, top, p.N, cnt(top), zo, st);
}

template <typename S>
int launch_riccati(const KP<S>& p, const std::vector<int32_t>& stage_begin, S* zo, cudaStream_t st,
                   cudaEvent_t* ev) {
  if (!direct_kernels()) return riccati_passes_seq<S>(p, stage_begin, zo, st, ev);
  const int sl = (p.nx + p.nu + 31) / 32;
  switch (sl) {
    case 1: return riccati_passes_sl<S, 1>(p, stage_begin, zo, st, ev);
    case 2: return riccati_passes_sl<S, 2>(p, stage_begin, zo, st, ev);
    case 3: return riccati_passes_sl<S, 3>(p, stage_begin, zo, st, ev);
    default: return riccati_passes_sl<S, 4>(p, stage_begin, zo, st, ev);
  }
}

// ---------------------------------------------------------------------------
// batched: direct kernels over the block map of the launch (chains of every
// instance, or one stage of every instance: stage[i] from the map)
// ---------------------------------------------------------------------------
template <typename S, int SL>
__global__ void __launch_bounds__(128) k_bwd_chain_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x];
  const KP<S> p = bi[i].kp;
  bwd_chain_body<S, SL>(p, blockIdx.x - m.base[i], m.cnt[i]);
}
template <typename S, int SL>
__global__ void __launch_bounds__(128) k_bwd_stage_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x];
  const KP<S> p = bi[i].kp;
  bwd_stage_body<S, SL>(p, m.stage[i], blockIdx.x - m.base[i], m.cnt[i]);
}
template <typename S, int SL>
__global__ void __launch_bounds__(128) k_fwd_stage_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x];
  const KP<S> p = bi[i].kp;
  fwd_stage_body<S, SL>(p, m.stage[i], bi[i].TVt, blockIdx.x - m.base[i], m.cnt[i]);
}
template <typename S, int SL>
__global__ void __launch_bounds__(128) k_fwd_chain_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x];
  const KP<S> p = bi[i].kp;
  fwd_chain_body<S, SL>(p, bi[i].TVt, blockIdx.x - m.base[i], m.cnt[i]);
}

template <typename S>
void launch_riccati_b(int which, const BInst<S>* bi, const BMap& m, int nblocks, int SL, cudaStream_t st) {
  if (nblocks <= 0) return;
#define SPOCK_RB(L)                                                                    \
  case L:                                                                              \
    if (which == 0) k_bwd_chain_b<S, L><<<nblocks, 128, 0, st>>>(bi, m);              \
    else if (which == 1) k_bwd_stage_b<S, L><<<nblocks, 128, 0, st>>>(bi, m);         \
    else if (which == 2) k_fwd_stage_b<S, L><<<nblocks, 128, 0, st>>>(bi, m);         \
    else k_fwd_chain_b<S, L><<<nblocks, 128, 0, st>>>(bi, m);                         \
    break;
  switch (SL) {
    SPOCK_RB(1) SPOCK_RB(2) SPOCK_RB(3)
    default: SPOCK_RB(4)
  }
#undef SPOCK_RB
}
template void launch_riccati_b<double>(int, const BInst<double>*, const BMap&, int, int, cudaStream_t);
template void launch_riccati_b<float>(int, const BInst<float>*, const BMap&, int, int, cudaStream_t);

template int launch_riccati<double>(const KP<double>&, const std::vector<int32_t>&, double*, cudaStream_t,
                                    cudaEvent_t*);
template int launch_riccati<float>(const KP<float>&, const std::vector<int32_t>&, float*, cudaStream_t,
                                   cudaEvent_t*);

}  // namespace spock
