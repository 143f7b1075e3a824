// Device bodies of the round kernels (rounds.cu), shared with the
// single-block solve kernel (cta.cu): decision, commit with the Anderson
// column and Gram row, Gram solve, next evaluation point.
#pragma once

#include <cmath>
#include <cstdint>

#include "kernels.cuh"
#include "supermann.cuh"

namespace spock {

static __device__ void round_trace(SmState* st, int32_t* trace, int branch, int nb) {
  if (st->record_trace && trace && st->k < st->max_iter) {
    trace[2 * st->k] = branch;
    trace[2 * st->k + 1] = nb;
  }
}

// The next iteration; c2^k is kept as a running product (FP64 pow is some 100
// instructions of 64 cycles each, in one thread that the GPU waits for).
static __device__ __forceinline__ void round_next_k(SmState* st) {
  st->k++;
  st->c2k *= st->c2;
}

// Decisions after an iterate has been accepted (its statistics in stats_cur).
static __device__ void round_after_accept(SmState* st, int32_t* trace) {
  const double* sc = st->stats_cur;
  const double om2 = sc[ST_RZ2] + sc[ST_RE2] - 2.0 * st->alpha * sc[ST_RE_LRZ];
  const double omega = sqrt(fmax(om2, 0.0));
  const double xi = fmax(sc[ST_XIP], sc[ST_XID]);
  if (!st->initialized) {
    st->zeta = omega;
    st->omega_safe = omega;
    st->xi0 = xi;
    if (!(st->tol > 0.0)) st->tol = fmax(st->eps_abs, st->eps_rel * xi);
    st->best_xi = xi;
    st->best_k = 0;
    st->initialized = 1;
  }
  st->omega = omega;
  st->xi = xi;
  if (xi < 0.5 * st->best_xi) {
    st->best_xi = xi;
    st->best_k = st->k;
  }
  st->op_aa = 0;
  st->op_point = PT_NONE;
  int act;
  if (!isfinite(om2) || !isfinite(xi)) act = A_NUMERICAL;
  else if (xi <= st->tol) act = A_DONE;
  else if (st->k >= st->max_iter) act = A_MAXIT;
  else if (st->stall_window > 0 && st->k - st->best_k > st->stall_window && xi <= 30.0 * st->tol) act = A_STALL;
  else act = A_NONE;
  if (act != A_NONE) {
    st->action = act;
    st->done = 1;
    return;
  }
  if (st->have_prev && st->mem > 0) {  // Anderson update with (v, c = r) of this iterate
    st->op_aa = 1;
    st->aa_slot = st->aa_next;
    st->aa_next = (st->aa_next + 1) % st->mem;
    st->aa_cnt = min(st->aa_cnt + 1, st->mem);
  }
  st->have_prev = 1;
  st->op_point = PT_DIR;
  if (omega <= st->c0 * st->zeta) {  // K0: blind step v + d
    st->zeta = omega;
    round_trace(st, trace, 0, 0);
    st->n_k0++;
    round_next_k(st);
    st->pending = P_K0;
    st->action = A_K0;
  } else {
    st->tau = 1.0;
    st->nb = 0;
    st->pending = P_LS;
    st->action = A_LS;
  }
}

static __device__ void round_decide_body(SmState* st, const double* stats_t, int32_t* trace) {
  st->op_accept = 0;
  st->op_aa = 0;
  st->op_point = PT_NONE;
  if (st->done) return;
  st->rounds++;
  const int pend = st->pending;
  bool accept = false;
  if (pend == P_INIT || pend == P_K0 || pend == P_K2) {
    accept = true;
  } else {  // P_LS: line-search trial v~ = v + tau d evaluated
    const double om2 = stats_t[ST_RZ2] + stats_t[ST_RE2] - 2.0 * st->alpha * stats_t[ST_RE_LRZ];
    const double omt = sqrt(fmax(om2, 0.0));
    st->omega_t = omt;
    const double omega = st->omega;
    if (!isfinite(om2)) {
      st->action = A_NUMERICAL;
      st->done = 1;
      return;
    }
    if (omega <= st->omega_safe && omt <= st->c1 * omega) {  // K1
      st->omega_safe = omt + st->c2k;
      round_trace(st, trace, 1, st->nb);
      st->n_k1++;
      round_next_k(st);
      accept = true;
    } else {
      const double rdM = stats_t[ST_RD] - st->alpha * (stats_t[ST_LRZ_DE] + stats_t[ST_RE_LDZ]);
      const double rho = om2 - st->rho_coef * st->tau * rdM;
      st->rho = rho;
      if (rho >= st->sigma * omt * omega && omt > 0.0) {  // K2
        st->coef = st->lam * rho / (omt * omt);
        round_trace(st, trace, 2, st->nb);
        st->n_k2++;
        round_next_k(st);
        st->op_point = PT_K2;
        st->pending = P_K2;
        st->action = A_K2;
      } else {
        st->nb++;
        st->n_back++;
        st->tau *= st->beta;
        if (st->nb >= st->max_back) {  // cap: tau = 0, relaxed step v - lambda r
          round_trace(st, trace, 3, st->nb);
          st->n_cap++;
          round_next_k(st);
          st->op_point = PT_KM;
          st->pending = P_K2;
          st->action = A_CAP;
        } else {
          st->op_point = PT_LS;
          st->pending = P_LS;
          st->action = A_RETRY;
        }
      }
    }
  }
  if (accept) {
    st->op_accept = 1;
    for (int i = 0; i < 8; ++i) st->stats_cur[i] = stats_t[i];
    round_after_accept(st, trace);
  }
  if (!st->done) st->n_T++;  // the T evaluation that follows this round
}


template <typename S>
struct RPack;
template <>
struct RPack<float> {
  using T = float4;
  static constexpr int N = 4;
};
template <>
struct RPack<double> {
  using T = double2;
  static constexpr int N = 2;
};
template <typename S>
__device__ __forceinline__ S& rpk(typename RPack<S>::T& v, int e) {
  return reinterpret_cast<S*>(&v)[e];
}
template <typename S>
__device__ __forceinline__ typename RPack<S>::T rld(const S* p, int64_t q) {
  return reinterpret_cast<const typename RPack<S>::T*>(p)[q];
}
template <typename S>
__device__ __forceinline__ void rst(S* p, int64_t q, const typename RPack<S>::T& v) {
  reinterpret_cast<typename RPack<S>::T*>(p)[q] = v;
}

// Commit an accepted (Vt, TVt) and, with op_aa, write the new Anderson
// column (slot st->aa_slot) and the dot products of the stored columns with
// it and with the new residual (terms in S, FP64 accumulation per pack).
// The Anderson differences are formed from the old (V, TV) as it is read, so
// the previous pair is not kept.
template <typename S, int MEM>
__device__ __forceinline__ void round_commit_body(SmState* st, S* __restrict__ V, S* __restrict__ TV,
                                                  const S* __restrict__ Vt, const S* __restrict__ TVt,
                                                  S* __restrict__ MR, S* __restrict__ D, int64_t n, int64_t ld,
                                                  double* __restrict__ partials, int bid, int nblk) {
  if (!st->op_accept) return;
  const bool aa = st->op_aa != 0;
  const int slot = st->aa_slot, cnt = st->aa_cnt;
  constexpr int NP = RPack<S>::N;
  using PT = typename RPack<S>::T;
  double gr[MEM > 0 ? MEM : 1], rh[MEM > 0 ? MEM : 1];
#pragma unroll
  for (int j = 0; j < MEM; ++j) gr[j] = rh[j] = 0.0;
  const int64_t stride = (int64_t)nblk * blockDim.x;
  const int64_t gt = (int64_t)bid * blockDim.x + threadIdx.x;
  const int64_t npack = n / NP;
  for (int64_t q = gt; q < npack; q += stride) {
    PT nv = rld(Vt, q), nt = rld(TVt, q), ov = rld(V, q), ot = rld(TV, q);
    rst(V, q, nv);
    rst(TV, q, nt);
    if (MEM > 0 && aa) {
      PT rr, dc, dd;
#pragma unroll
      for (int t = 0; t < NP; ++t) {
        rpk<S>(rr, t) = rpk<S>(nv, t) - rpk<S>(nt, t);
        rpk<S>(dc, t) = rpk<S>(rr, t) - (rpk<S>(ov, t) - rpk<S>(ot, t));
        rpk<S>(dd, t) = (rpk<S>(nv, t) - rpk<S>(ov, t)) - rpk<S>(dc, t);
      }
      rst(MR + (int64_t)slot * ld, q, dc);
      rst(D + (int64_t)slot * ld, q, dd);
#pragma unroll
      for (int j = 0; j < MEM; ++j) {
        if (j < cnt) {
          PT col = (j == slot) ? dc : rld(MR + (int64_t)j * ld, q);
          S g = 0, h = 0;
#pragma unroll
          for (int t = 0; t < NP; ++t) {
            g += rpk<S>(col, t) * rpk<S>(dc, t);
            h += rpk<S>(col, t) * rpk<S>(rr, t);
          }
          gr[j] += (double)g;
          rh[j] += (double)h;
        }
      }
    }
  }
  for (int64_t i = npack * NP + gt; i < n; i += stride) {  // tail
    const S nv = Vt[i], nt = TVt[i], ov = V[i], ot = TV[i];
    V[i] = nv;
    TV[i] = nt;
    if (MEM > 0 && aa) {
      const S r = nv - nt, dc = r - (ov - ot);
      MR[(int64_t)slot * ld + i] = dc;
      D[(int64_t)slot * ld + i] = (nv - ov) - dc;
#pragma unroll
      for (int j = 0; j < MEM; ++j) {
        if (j < cnt) {
          const S c = (j == slot) ? dc : MR[(int64_t)j * ld + i];
          gr[j] += (double)(c * dc);
          rh[j] += (double)(c * r);
        }
      }
    }
  }
  if (MEM == 0 || !aa) return;
  // row bid of the partials: [2 kMaxMemory], entries j < MEM of the Gram row and
  // kMaxMemory + j of the right-hand side
  __shared__ double red[8][2 * kMaxMemory];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int g = 0; g < (2 * MEM + 7) / 8; ++g) {
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int e = 8 * g + i;
      v[i] = e < MEM ? gr[e < MEM ? e : 0] : (e < 2 * MEM ? rh[e < 2 * MEM && e >= MEM ? e - MEM : 0] : 0.0);
    }
    const double t = warp_sum8(v, lane);
    const int e = 8 * g + warp_sum8_index(lane);
    if ((lane & 3) == 0 && e < 2 * MEM) red[w][e < MEM ? e : kMaxMemory + e - MEM] = t;
  }
  __syncthreads();
  if (threadIdx.x < 2 * MEM) {
    const int j = threadIdx.x < MEM ? threadIdx.x : kMaxMemory + threadIdx.x - MEM;
    double sum = 0.0;
    if ((j & (kMaxMemory - 1)) < cnt)
      for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) sum += red[ww][j];
    partials[(int64_t)bid * 2 * kMaxMemory + j] = sum;
  }
}

// Gram update and least squares for gamma (FP64), newest columns first;
// numerically singular Gram matrices drop their oldest columns from the solve.
// One block.  A warp sums one value over the rows of the partials (lanes over
// rows); then one warp factors L D L^T, lane a holding row a: one reciprocal
// per pivot and products otherwise (a division or a square root is a chain of
// some 10 FP64 instructions, 67 cycles each).
__device__ __forceinline__ void round_aa_solve_body(SmState* st, const double* __restrict__ partials,
                                                    int nblocks) {
  if (!st->op_aa) return;
  __shared__ double sums[2 * kMaxMemory];
  __shared__ double Mx[kMaxMemory][kMaxMemory + 1];   // row a: l_ab d_b for b < a, then the pivot d_a
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int M = kMaxMemory, slot = st->aa_slot, cnt = st->aa_cnt, mem = st->mem;
  for (int v = threadIdx.x >> 5; v < 2 * cnt; v += nw) {
    const int j = v < cnt ? v : M + v - cnt;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += __ldcg(partials + (int64_t)b * 2 * M + j);
    s = warp_sum(s);
    if (lane == 0) sums[j] = s;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  auto order = [&](int a) {   // a-th newest column
    const int o = slot - a;
    return o < 0 ? o + mem : o;
  };
  if (lane < cnt) {
    st->G[slot * M + lane] = sums[lane];
    st->G[lane * M + slot] = sums[lane];
    st->rhs[lane] = sums[M + lane];
  }
  if (lane < M) st->gamma[lane] = 0.0;
  __syncwarp();
  const int oa = order(lane < cnt ? lane : 0);
  double diag = lane < cnt ? st->G[oa * M + oa] : 0.0;
  if (lane < cnt)
    for (int b = 0; b <= lane; ++b) {
      const int ob = order(b);
      Mx[lane][b] = (oa == slot || ob == slot) ? sums[oa == slot ? ob : oa] : st->G[oa * M + ob];
    }
  if (lane < cnt && oa == slot) diag = sums[slot];
  __syncwarp();
  // factor while the pivots are positive: lane a's l_ab d_b - sum of products
  int good = 0;   // pivots that could be formed
  double inv = 0.0;
  for (int c = 0; c < cnt; ++c) {
    const double piv = Mx[c][c];
    if (!(piv > 0.0)) break;
    const double r = 1.0 / piv;
    if (lane == c) inv = r;
    if (lane > c && lane < cnt) {
      const double l = Mx[lane][c] * r;
      for (int b = c + 1; b <= lane; ++b) Mx[lane][b] = fma(-l, Mx[b][c], Mx[lane][b]);
    }
    __syncwarp();
    good = c + 1;
  }
  // the most columns whose pivots are all above 1e-13 of their largest diagonal
  int use = 0;
  {
    const double d = lane < good ? Mx[lane][lane] : 0.0;
    double mx = diag;   // largest diagonal of the first lane + 1 columns
    double mn = d;
    for (int o = 1; o < 32; o <<= 1) {
      const double up = __shfl_up_sync(kFull, mx, o), un = __shfl_up_sync(kFull, mn, o);
      if (lane >= o) {
        mx = fmax(mx, up);
        mn = fmin(mn, un);
      }
    }
    const bool ok = lane < good && mn > 1e-13 * mx;
    const unsigned okm = __ballot_sync(kFull, ok);
    use = 32 - __clz(okm);
  }
  if (lane == 0) st->aa_dropped = cnt - use;
  if (use == 0) return;
  // L y = rhs, then L^T gamma = D^-1 y
  double y = lane < use ? sums[M + oa] : 0.0;
  for (int c = 0; c < use; ++c) {
    const double yc = __shfl_sync(kFull, y, c) * __shfl_sync(kFull, inv, c);
    if (lane > c && lane < use) y = fma(-Mx[lane][c], yc, y);
  }
  y *= inv;
  for (int c = use - 1; c > 0; --c) {
    const double yc = __shfl_sync(kFull, y, c);
    if (lane < c) y = fma(-Mx[c][lane] * inv, yc, y);
  }
  if (lane < use) st->gamma[oa] = y;
}

// After the commit: the block that finishes last solves for gamma (every
// block of the grid calls it, all threads).
__device__ __forceinline__ void round_commit_last(SmState* st, const double* __restrict__ partials, int nblk) {
  if (!st->op_accept || !st->op_aa) return;
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == (unsigned)nblk - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) st->ticket = 0;
  round_aa_solve_body(st, partials, nblk);
}


// Next evaluation point in Vt (and the direction d for PT_DIR).
template <typename S, int MEM>
__device__ __forceinline__ void round_point_body(const SmState* __restrict__ st, const S* __restrict__ V,
                                                 const S* __restrict__ TV, S* __restrict__ Vt,
                                                 const S* __restrict__ TVt, S* __restrict__ d,
                                                 const S* __restrict__ D, int64_t n, int64_t ld, int bid,
                                                 int nblk) {
  const int op = st->op_point;
  if (op == PT_NONE) return;
  constexpr int NP = RPack<S>::N;
  using PT = typename RPack<S>::T;
  const int cnt = st->aa_cnt;
  S g[MEM > 0 ? MEM : 1];
#pragma unroll
  for (int j = 0; j < MEM; ++j) g[j] = (j < cnt) ? (S)st->gamma[j] : S(0);
  const S tau = (S)st->tau, coef = (S)st->coef, lam = (S)st->lam;
  const int64_t stride = (int64_t)nblk * blockDim.x;
  const int64_t gt = (int64_t)bid * blockDim.x + threadIdx.x;
  const int64_t npack = n / NP;
  for (int64_t q = gt; q < npack; q += stride) {
    PT v = rld(V, q), out;
    if (op == PT_DIR) {
      PT tv = rld(TV, q), dd;
#pragma unroll
      for (int t = 0; t < NP; ++t) rpk<S>(dd, t) = rpk<S>(tv, t) - rpk<S>(v, t);
#pragma unroll
      for (int j = 0; j < MEM; ++j) {
        if (j < cnt) {
          PT c = rld(D + (int64_t)j * ld, q);
#pragma unroll
          for (int t = 0; t < NP; ++t) rpk<S>(dd, t) -= g[j] * rpk<S>(c, t);
        }
      }
      rst(d, q, dd);
#pragma unroll
      for (int t = 0; t < NP; ++t) rpk<S>(out, t) = rpk<S>(v, t) + rpk<S>(dd, t);
    } else if (op == PT_LS) {
      PT dd = rld(d, q);
#pragma unroll
      for (int t = 0; t < NP; ++t) rpk<S>(out, t) = rpk<S>(v, t) + tau * rpk<S>(dd, t);
    } else if (op == PT_K2) {
      PT a = rld(Vt, q), b = rld(TVt, q);
#pragma unroll
      for (int t = 0; t < NP; ++t) rpk<S>(out, t) = rpk<S>(v, t) - coef * (rpk<S>(a, t) - rpk<S>(b, t));
    } else {  // PT_KM
      PT tv = rld(TV, q);
#pragma unroll
      for (int t = 0; t < NP; ++t) rpk<S>(out, t) = rpk<S>(v, t) - lam * (rpk<S>(v, t) - rpk<S>(tv, t));
    }
    rst(Vt, q, out);
  }
  for (int64_t i = npack * NP + gt; i < n; i += stride) {
    const S v = V[i];
    S o;
    if (op == PT_DIR) {
      S di = TV[i] - v;
#pragma unroll
      for (int j = 0; j < MEM; ++j)
        if (j < cnt) di -= g[j] * D[(int64_t)j * ld + i];
      d[i] = di;
      o = v + di;
    } else if (op == PT_LS) {
      o = v + tau * d[i];
    } else if (op == PT_K2) {
      o = v - coef * (Vt[i] - TVt[i]);
    } else {
      o = v - lam * (v - TV[i]);
    }
    Vt[i] = o;
  }
}

}  // namespace spock
