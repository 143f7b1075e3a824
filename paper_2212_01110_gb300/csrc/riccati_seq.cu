// Riccati passes (Algorithm 2), a block per node sequence, every node's
// factors staged in shared memory.
//
// A sequence is a run of nodes that follow one another through single
// children: the chain below the last branching stage with its leaf (one launch
// for all chains), or one node of a branching stage (one launch per stage).
// The backward step of node k
//   h   = sum over the children of h^c           (leaf: q^k = -xbar^k)
//   g   = ubar^k - h_u
//   d^k = Rt^-1 g,   q^k = h_x - xbar^k + E^T g - K^T ubar^k
//   h^k = [Abar^k | B^k]^T q^k                   (not at the root)
// with E = Rt^-1 (K + W^T), formed once with the factors (q^k = h_x - xbar^k +
// K^T (d^k - ubar^k) + W d^k, so that d^k and q^k come from one product; K + W^T is
// zero but for what rounding K left in Rt K, and taking it along keeps the
// projection as exact as K allows: without it states in mixed units lose up to a
// digit and a half), reads the factors of node k only and hands nx + nu numbers on to the parent: in
// registers along a sequence, through p.hb between launches.  A branching
// stage reads a quarter of what a step over the children's [Abar | B] reads at
// four children per node; those of the chains' tops are streamed by the chain
// launch.  The forward step of a node k > 0
//   x^k = [Abar^k | B^k] (x; d)^parent,   u^parent = K^parent x^parent + d^parent
// (u by the first child) is one product as well.
//
// T threads of a block work on one node at a time: thread (row group, column)
// of a product, the row groups' partial sums added through shared memory.  One
// more warp fetches the nodes' blocks by bulk asynchronous copies into a ring
// of D slots (address arithmetic, fence and copies in one of the T threads
// would lengthen every step, and so would a second barrier to wait on: 200
// cycles each, measured).  What latency is left, and the serial sums and
// barriers of a step, is covered by the other blocks of the SM.
//
// FP64 factors and vectors are held and multiplied as doubles.  (A form with
// 57-bit integers relative to a column's largest entry and exact integer sums
// ran the chains below in 670 and 473 us, but entries far below the largest
// lost digits without limit: a dynamics residual of 1e-10 for states whose units
// differ by 1e6, 5e-4 by 1e12, against 2e-15.)
//
// What bounds it and what it measured (GB300, nx = 50, nu = 20).  Chains of the
// 62,805-node tree, FP64: backward 886 us (2.88 GB), forward 576 us (2.2 GB),
// where direct-load kernels took 1,073 and 705 us; FP32: 228 and 174 us, 6.0 TB/s
// (278 and 237 with one warp per chain).  The FP64 chains are bound by
// the FP64 pipes (1.9 multiply-adds per clock and SM: a warp instruction holds
// its sub-partition's pipe for 64 cycles; 85 and 88% busy), the FP32 ones by
// memory.
//
// Bounded waits: a wait that exceeds kWaitLimit polls sets *p.err and the
// thread stops waiting (the fetching warp: stops issuing); the block finishes
// its loop on whatever the buffers hold (every access stays inside them), and
// the fetching warp waits for its copies in flight (bounded) before it returns.
#include <algorithm>
#include <atomic>
#include <vector>

#include "batch.cuh"
#include "kernels.cuh"
#include "launch.cuh"
#include "spock_internal.h"
#include "tma.cuh"

namespace spock {

constexpr int kMaxSeqThreads = 224;   // T; 32 more fetch
constexpr int kMaxSlots = 2;
constexpr int kMaxGroups = 4;         // row groups of an FP64 product

// Shared memory of a block, in bytes: D slots of one node's blocks each,
// prepared vectors, partial sums.
struct SeqLayout {
  uint32_t item, vecA, vecB, part;
  __host__ __device__ uint32_t bytes(int D) const { return D * item + vecA + vecB + part; }
};
__host__ __device__ inline int up4(int n) { return (n + 3) & ~3; }
template <typename S>
__host__ __device__ inline SeqLayout seq_layout_bwd(const KP<S>& p, int T) {
  SeqLayout L;
  L.item = up128((p.gstride + p.nbstride + p.xs + p.us) * (uint32_t)sizeof(S));   // [Abar | B] | [E | K | Rt^-1] | xbar | ubar
  L.vecA = up16(2 * up4(p.nu) * (uint32_t)sizeof(S));                               // (g; -ubar)
  L.vecB = up16(up4(p.nx) * (uint32_t)sizeof(S));                                   // q
  L.part = up16(T * (uint32_t)sizeof(S));
  return L;
}
template <typename S>
__host__ __device__ inline SeqLayout seq_layout_fwd(const KP<S>& p, int T) {
  SeqLayout L;
  L.item = up128((p.gstride + p.ktstride + p.us) * (uint32_t)sizeof(S));   // [Abar | B]^T | K^T of the parent | d of the node
  L.vecA = up16(up4(p.nx + p.nu) * (uint32_t)sizeof(S));                   // (x; d) of the parent and of the node
  L.vecB = L.vecA;
  L.part = up16(T * (uint32_t)sizeof(S));
  return L;
}

// Barrier of the T working threads of a block.
__device__ __forceinline__ void seq_bar(int T) { named_bar(1, T); }

// Columns of a product: those of x (nx) and those of u (nu), a thread each, in
// RG row groups.  FP32: per row group the x columns, then the u columns from a
// warp boundary on (both in one warp when they fit), so that no warp runs the
// sums of both: with 50 and 20 packed into 70 threads, one warp ran 120 rows
// where the others ran 70.  FP64: a warp instruction holds its sub-partition's
// FP64 pipe for 64 cycles whatever its lanes do, so the x columns of all row
// groups come first, then the u columns, without gaps (nx = 50, nu = 20, three
// groups: 210 of 224 lanes; few warps run the longer sums for columns of both).
template <typename S>
__host__ __device__ inline int seq_off(int nx, int nu) { return nx + nu <= 32 ? nx : (nx + 31) & ~31; }
template <typename S>
__host__ __device__ inline int seq_cols(int nx, int nu) {   // threads of one row group
  return sizeof(S) == 8 ? nx + nu : (seq_off<S>(nx, nu) + nu + 31) & ~31;
}
struct SeqCols {
  int RG;       // row groups
  int rg, col;  // this thread's group and its column of x or of u
  int off;      // thread of the first u column of group 0
  int step;     // threads from a column's group to its next group
  bool xcol, live;
};
template <typename S>
__device__ __forceinline__ SeqCols seq_columns(int nx, int nu, int T, int tid) {
  SeqCols c;
  const int CP = seq_cols<S>(nx, nu);
  if (sizeof(S) == 8) {
    c.RG = min(T / CP, kMaxGroups);
    c.off = c.RG * nx;
    c.xcol = tid < c.off;
    c.step = c.xcol ? nx : nu;
    const int t = c.xcol ? tid : tid - c.off;
    c.rg = t / c.step;
    c.col = t - c.rg * c.step;
  } else {
    c.RG = T / CP;
    c.off = seq_off<S>(nx, nu);
    c.step = CP;
    c.rg = tid / CP;
    const int t = tid - c.rg * CP;
    c.xcol = t < nx;
    c.col = c.xcol ? t : t - c.off;
  }
  c.live = c.rg < c.RG && c.col >= 0 && c.col < (c.xcol ? nx : nu);
  return c;
}
// Rows of a row group.
template <typename S>
__device__ __forceinline__ int seq_chunk(int n, int RG) {
  const int c = (n + RG - 1) / RG;
  return sizeof(S) == 8 ? c : up4(c);   // FP32 reads the vector in 16-byte pieces
}

// acc + sum over n rows of M[r] v[r]; `m` the shared-memory address of the
// thread's entry in the first row, rows ldB bytes apart, `v` that of the vector
// (FP32: 16-byte aligned).  FP32: eight rows are loaded before their products,
// without a branch among them.
__device__ __forceinline__ float seq_rows(float acc, uint32_t m, uint32_t ldB, uint32_t v, int n) {
  for (; n >= 8; n -= 8, m += 8 * ldB, v += 32) {
    float a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = lds_f32(m + i * ldB);
    const float4 x = lds_f32x4(v), y = lds_f32x4(v + 16);
    acc = fmaf(a[0], x.x, acc);
    acc = fmaf(a[1], x.y, acc);
    acc = fmaf(a[2], x.z, acc);
    acc = fmaf(a[3], x.w, acc);
    acc = fmaf(a[4], y.x, acc);
    acc = fmaf(a[5], y.y, acc);
    acc = fmaf(a[6], y.z, acc);
    acc = fmaf(a[7], y.w, acc);
  }
  if (n > 0) {
    float a[7], x[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      const int r = i < n ? i : n - 1;
      a[i] = lds_f32(m + r * ldB);
      x[i] = lds_f32(v + 4 * r);
    }
#pragma unroll
    for (int i = 0; i < 7; ++i)
      if (i < n) acc = fmaf(a[i], x[i], acc);
  }
  return acc;
}
__device__ __forceinline__ double seq_rows(double acc, uint32_t m, uint32_t ldB, uint32_t v, int n) {
  const char* mp = (const char*)__cvta_shared_to_generic(m);
  const double* vp = (const double*)__cvta_shared_to_generic(v);
  __builtin_assume(__isShared(mp));
  __builtin_assume(__isShared(vp));
#pragma unroll 4
  for (int r = 0; r < n; ++r, mp += ldB) acc = fma(*(const double*)mp, vp[r], acc);
  return acc;
}

// Sum of the row groups' accumulators in the threads of row group 0 (one
// barrier if there is more than one group; every thread calls it).
template <typename S>
__device__ __forceinline__ S seq_reduce(S acc, const SeqCols& c, bool live, S* part, int T) {
  if (c.RG == 1) return acc;
  if (live && c.rg > 0) part[threadIdx.x] = acc;
  seq_bar(T);
  if (live && c.rg == 0)
    for (int i = 1; i < c.RG; ++i) acc += part[i * c.step + threadIdx.x];
  return acc;
}

// The ring: per slot a barrier for "full" (the copies have arrived) and one for
// "empty" (the T threads are through with it); a thread keeps the parity of its
// next wait per slot.
struct SeqRing {
  uint64_t* full;
  uint64_t* empty;
  uint32_t phase;
  bool dead;     // a wait gave up
  __device__ __forceinline__ void wait(uint64_t* bar, int s, int32_t* err) {
    if (dead) return;
    if (mbar_wait(&bar[s], (phase >> s) & 1u)) {
      phase ^= 1u << s;
    } else {
      dead = true;
      atomicExch(err, 1);
    }
  }
};

// The fetching thread's loop.  fixed(slot, k, above) starts the copies of node
// k's factors and announces the bytes of all its copies, moving(slot, k, above)
// those of what earlier kernels write (above: the node before it in the
// sequence, -1 at the first one).  The factors of the first D nodes are on
// their way while the previous kernel still runs.  On return nothing is in
// flight (bounded).
template <typename F, typename M>
__device__ __forceinline__ void seq_fetch(SeqRing& ring, const int32_t* skip, const int32_t* stage_begin, int t_first,
                                          int t_last, int cnt, int bid, int nblk, int D, int32_t* err, F fixed,
                                          M moving) {
  const int dt = t_first < t_last ? 1 : -1;
  int slot = 0, issued = 0, early = 0;
  for (int ci = bid; ci < cnt && early < D; ci += nblk)
    for (int t = t_first; early < D; t += dt) {
      fixed(early, stage_begin[t] + ci, t == t_first ? -1 : stage_begin[t - dt] + ci);
      ++early;
      if (t == t_last) break;
    }
  pdl_enter();
  bool done = false;   // the solve has finished: only complete what has been announced
  for (int ci = bid; ci < cnt && !ring.dead && !done; ci += nblk) {
    for (int t = t_first;; t += dt) {
      const int k = stage_begin[t] + ci, above = t == t_first ? -1 : stage_begin[t - dt] + ci;
      if (issued == early && skip && *skip) done = true;
      if (issued >= D && !done) ring.wait(ring.empty, slot, err);
      if (ring.dead || done) break;
      fence_proxy_async();
      if (issued >= early) fixed(slot, k, above);
      moving(slot, k, above);
      ++issued;
      if (++slot == D) slot = 0;
      if (t == t_last) break;
    }
  }
  for (int s = 0; s < D; ++s) {
    const int uses = (issued - s + D - 1) / D;
    if (uses > 0) mbar_wait(&ring.full[s], (uint32_t)(uses - 1) & 1u);
  }
}

// Sequences from stage t_hi down to t_lo, of which block bid of nblk takes
// every nblk-th.  LAM: the recursion of the multipliers (grad.cu), lambda^k =
// h_x - xbar^k - K^T h_u -- q with g = 0 and ubar = h_u -- into lam instead of
// d.
template <typename S, bool LAM>
__device__ __forceinline__ void bwd_seq_body(const KP<S>& p, int t_hi, int t_lo, int bid, int nblk, int D,
                                             S* lam = nullptr) {
  constexpr uint32_t B = sizeof(S);
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint64_t bars[2][kMaxSlots];
  const int tid = threadIdx.x, T = blockDim.x - 32;
  const int nx = p.nx, nu = p.nu, ncol = nx + nu;
  const uint32_t gB = p.gstride * B, nbB = p.nbstride * B;   // bytes of a node's blocks
  const SeqLayout Ly = seq_layout_bwd(p, T);
  const int cnt = p.stage_begin[t_lo + 1] - p.stage_begin[t_lo];
  if (bid >= cnt) return;
  SeqRing ring{bars[0], bars[1], 0u, false};
  if (tid == 0) {
    for (int s = 0; s < D; ++s) {
      mbar_init(&ring.full[s], 1);
      mbar_init(&ring.empty[s], 1);
    }
    fence_mbar_init();
  }
  __syncthreads();
  if (tid >= T) {
    if (tid > T) return;
    const uint32_t xB = p.xs * (uint32_t)sizeof(S), uB = p.us * (uint32_t)sizeof(S);
    seq_fetch(
        ring, p.skip, p.stage_begin, t_hi, t_lo, cnt, bid, nblk, D, p.err,
        [&](int slot, int k, int) {
          const bool leaf = k >= p.nl;
          unsigned char* dst = smem + slot * Ly.item;
          uint64_t* bar = &ring.full[slot];
          mbar_expect_tx(bar, xB + (leaf ? 0u : nbB + uB) + (k > 0 ? gB : 0u));
          if (!leaf) bulk_g2s(dst + gB, p.NB + (size_t)k * p.nbstride, nbB, bar);
          if (k > 0) bulk_g2s(dst, p.Gb + (size_t)(k - 1) * p.gstride, gB, bar);
        },
        [&](int slot, int k, int) {
          unsigned char* dst = smem + slot * Ly.item + gB + nbB;
          if (k < p.nl) bulk_g2s(dst + xB, p.ubar + (size_t)k * p.us, uB, &ring.full[slot]);
          bulk_g2s(dst, p.xbar + (size_t)k * p.xs, xB, &ring.full[slot]);
        });
    return;
  }
  pdl_enter();
  if (p.skip && *p.skip) return;
  S* const vA = reinterpret_cast<S*>(smem + D * Ly.item);               // (g; -ubar), 16-byte aligned halves
  S* const vB = reinterpret_cast<S*>(smem + D * Ly.item + Ly.vecA);     // q
  S* const part = reinterpret_cast<S*>(smem + D * Ly.item + Ly.vecA + Ly.vecB);
  const uint32_t aA = smem_u32(vA), aB = smem_u32(vB), a0 = smem_u32(smem);
  // q and h_x in the x columns, d and h_u in the u columns; entry e of h; row
  // group rg takes rows u0 .. or x0 .. of a vector
  const SeqCols cl = seq_columns<S>(nx, nu, T, tid);
  const bool inx = tid < nx, inu = tid >= cl.off && tid < cl.off + nu, own = inx || inu;
  const int a = tid - cl.off, e = inx ? tid : nx + a;
  const int nu4 = up4(nu), cu = seq_chunk<S>(nu, cl.RG), cx = seq_chunk<S>(nx, cl.RG);
  const int u0 = cl.rg * cu, un = max(0, min(cu, nu - u0)), x0 = cl.rg * cx, xn = max(0, min(cx, nx - x0));
  S h = S(0);   // h of the current node: this thread's column
  int slot = 0;
  for (int ci = bid; ci < cnt; ci += nblk) {
    for (int t = t_hi; t >= t_lo; --t) {
      const int k = p.stage_begin[t] + ci;
      const bool leaf = k >= p.nl;
      if (t == t_hi && !leaf && own) {   // sum of the children's h, from the launch below
        const int c0 = p.ch_begin[k], m = p.ch_count[k];
        const S* src = p.hb + (int64_t)(c0 - 1) * p.hst + e;
        h = src[0];
#pragma unroll 4
        for (int c = 1; c < m; ++c) h += src[(int64_t)c * p.hst];
      }
      const unsigned char* it = smem + slot * Ly.item;
      const uint32_t ait = a0 + slot * Ly.item;
      const S* xb = reinterpret_cast<const S*>(it + gB + nbB);
      ring.wait(ring.full, slot, p.err);
      S q = S(0);
      if (leaf) {
        if (inx) q = -xb[tid];
      } else {
        if (inu) {
          const S u = LAM ? h : (xb + p.xs)[a];
          vA[a] = LAM ? S(0) : u - h;   // g
          vA[nu4 + a] = -u;
        }
        const S base = inx ? h - xb[tid] : S(0);
        seq_bar(T);
        S acc = S(0);
        if (cl.live) {   // E (nu x nx) or Rt^-1 (nu x nu) with g, then K (nu x nx) with -ubar
          const uint32_t m = ait + gB;
          acc = seq_rows(acc, m + (cl.xcol ? u0 * nx + cl.col : 2 * nu * nx + u0 * nu + cl.col) * B,
                         (cl.xcol ? nx : nu) * B, aA + u0 * B, un);
          if (cl.xcol) acc = seq_rows(acc, m + ((nu + u0) * nx + cl.col) * B, nx * B, aA + (nu4 + u0) * B, un);
        }
        acc = seq_reduce<S>(acc, cl, cl.live, part, T);
        if (inx) q = base + acc;
        if (LAM) {
          if (inx) lam[(int64_t)k * p.xs + tid] = q;
        } else if (inu) {
          p.d[(int64_t)k * p.us + a] = acc;
        }
      }
      if (k > 0) {
        if (inx) vB[tid] = q;
        seq_bar(T);
        S acc = S(0);
        if (cl.live)   // [Abar | B] (nx x ncol)
          acc = seq_rows(acc, ait + (x0 * ncol + (cl.xcol ? cl.col : nx + cl.col)) * B, ncol * B, aB + x0 * B, xn);
        acc = seq_reduce<S>(acc, cl, cl.live, part, T);
        if (own) {
          h = acc;
          if (t == t_lo) p.hb[(int64_t)(k - 1) * p.hst + e] = h;
        }
        // every thread is through with the slot and the vectors; with several row
        // groups the barrier of the sum has said so (what group 0 reads after it,
        // the others' sums, is written again behind the next node's first barrier)
        if (cl.RG == 1) seq_bar(T);
        if (tid == 0) mbar_arrive(&ring.empty[slot]);
      }
      if (++slot == D) slot = 0;
    }
  }
}

// Sequences from stage t_lo >= 1 down to the leaves' side t_hi.
template <typename S>
__device__ __forceinline__ void fwd_seq_body(const KP<S>& p, int t_lo, int t_hi, S* __restrict__ zo, int bid,
                                             int nblk, int D) {
  constexpr uint32_t B = sizeof(S);
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint64_t bars[2][kMaxSlots];
  const int tid = threadIdx.x, T = blockDim.x - 32;
  const int nx = p.nx, nu = p.nu, ncol = nx + nu;
  const uint32_t gB = p.gstride * B, ktB = p.ktstride * B;   // bytes of a node's blocks
  const SeqLayout Ly = seq_layout_fwd(p, T);
  const int cnt = p.stage_begin[t_lo + 1] - p.stage_begin[t_lo];
  if (bid >= cnt) return;
  SeqRing ring{bars[0], bars[1], 0u, false};
  if (tid == 0) {
    for (int s = 0; s < D; ++s) {
      mbar_init(&ring.full[s], 1);
      mbar_init(&ring.empty[s], 1);
    }
    fence_mbar_init();
  }
  __syncthreads();
  if (tid >= T) {
    if (tid > T) return;
    const uint32_t uB = p.us * (uint32_t)sizeof(S);
    seq_fetch(
        ring, p.skip, p.stage_begin, t_lo, t_hi, cnt, bid, nblk, D, p.err,
        [&](int slot, int k, int above) {
          const int par = above < 0 ? p.parent[k] : above;
          const bool first = above >= 0 || k == 1 || p.parent[k - 1] != par;   // k is its parent's first child
          unsigned char* dst = smem + slot * Ly.item;
          uint64_t* bar = &ring.full[slot];
          mbar_expect_tx(bar, gB + (first ? ktB : 0u) + (k < p.nl ? uB : 0u));
          bulk_g2s(dst, p.Gf + (size_t)(k - 1) * p.gstride, gB, bar);
          if (first) bulk_g2s(dst + gB, p.Kt + (size_t)par * p.ktstride, ktB, bar);
        },
        [&](int slot, int k, int) {
          if (k < p.nl)
            bulk_g2s(smem + slot * Ly.item + gB + ktB, p.d + (size_t)k * p.us, uB, &ring.full[slot]);
        });
    return;
  }
  pdl_enter();
  if (p.skip && *p.skip) return;
  S* W = reinterpret_cast<S*>(smem + D * Ly.item);              // (x; d) of the parent
  S* Y = reinterpret_cast<S*>(smem + D * Ly.item + Ly.vecA);    // (x; d) of the node
  S* const part = reinterpret_cast<S*>(smem + D * Ly.item + Ly.vecA + Ly.vecB);
  const uint32_t a0 = smem_u32(smem);
  // x (ncol rows) and u of the parent (nx rows); the threads of row group 0 also
  // hold the entries of (x; d), entry e
  const SeqCols cl = seq_columns<S>(nx, nu, T, tid);
  const bool inx = tid < nx, inu = tid >= cl.off && tid < cl.off + nu, own = inx || inu;
  const int a = tid - cl.off, e = inx ? tid : nx + a;
  const int cc = seq_chunk<S>(ncol, cl.RG), cx = seq_chunk<S>(nx, cl.RG);
  const int w0 = cl.rg * cc, wn = max(0, min(cc, ncol - w0)), x0 = cl.rg * cx, xn = max(0, min(cx, nx - x0));
  S w = S(0);   // entry tid of the parent's (x; d)
  int slot = 0;
  for (int ci = bid; ci < cnt; ci += nblk) {
    for (int t = t_lo; t <= t_hi; ++t) {
      const int k = p.stage_begin[t] + ci;
      const int par = t == t_lo ? p.parent[k] : p.stage_begin[t - 1] + ci;
      const bool first = t > t_lo || k == 1 || p.parent[k - 1] != par;
      const int64_t zxk = p.zx[k], zup = p.zu[par];
      if (t == t_lo) {   // (x; d) of the parent, from the launch above
        if (own) {
          if (inu) w = p.d[(int64_t)par * p.us + a];
          else if (par > 0) w = zo[p.zx[par] + tid];
          else w = p.x0[tid];
          if (par == 0 && first && inx) zo[p.zx[0] + tid] = w;
          W[e] = w;
        }
        seq_bar(T);
      }
      const unsigned char* it = smem + slot * Ly.item;
      const uint32_t ait = a0 + slot * Ly.item, aW = smem_u32(W);
      ring.wait(ring.full, slot, p.err);
      const bool live = cl.live && (cl.xcol || first);
      S acc = S(0);
      if (live)   // [Abar | B]^T (ncol x nx) or K^T (nx x nu), one loop: a warp may hold columns of both
        acc = seq_rows(acc, ait + (cl.xcol ? (w0 * nx + cl.col) * B : gB + (x0 * nu + cl.col) * B),
                       (cl.xcol ? nx : nu) * B, aW + (cl.xcol ? w0 : x0) * B, cl.xcol ? wn : xn);
      acc = seq_reduce<S>(acc, cl, live, part, T);
      if (own && live) {
        if (inx) {
          zo[zxk + tid] = acc;
          w = acc;
        } else {
          zo[zup + a] = w + acc;
        }
      }
      if (t < t_hi) {   // the node's (x; d) for the next step
        if (inu) w = reinterpret_cast<const S*>(it + gB + ktB)[a];
        if (own) Y[e] = w;
        S* y = W;
        W = Y;
        Y = y;
      }
      seq_bar(T);   // every thread is through with the slot, (x; d) complete
      if (tid == 0) mbar_arrive(&ring.empty[slot]);
      if (++slot == D) slot = 0;
    }
  }
}

template <typename S>
__global__ void __launch_bounds__(kMaxSeqThreads + 32, sizeof(S) == 8 ? 4 : 1) k_bwd_seq(KP<S> p, int t_hi, int t_lo, int D) {
  bwd_seq_body<S, false>(p, t_hi, t_lo, blockIdx.x, gridDim.x, D);
}
template <typename S>
__global__ void __launch_bounds__(kMaxSeqThreads + 32, sizeof(S) == 8 ? 4 : 1) k_lambda_seq(KP<S> p, int t_hi, int t_lo, S* lam, int D) {
  bwd_seq_body<S, true>(p, t_hi, t_lo, blockIdx.x, gridDim.x, D, lam);
}
template <typename S>
__global__ void __launch_bounds__(kMaxSeqThreads + 32, sizeof(S) == 8 ? 4 : 1) k_fwd_seq(KP<S> p, int t_lo, int t_hi, S* __restrict__ zo,
                                                            int D) {
  fwd_seq_body<S>(p, t_lo, t_hi, zo, blockIdx.x, gridDim.x, D);
}

// Batched: block -> (instance, block) from the launch's map; stage < 0: the
// chain region of every instance (forward: below the root at the earliest).
template <typename S>
__global__ void __launch_bounds__(kMaxSeqThreads + 32, sizeof(S) == 8 ? 4 : 1) k_bwd_seq_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x], t = m.stage[i];
  const KP<S> p = bi[i].kp;
  bwd_seq_body<S, false>(p, t < 0 ? p.N : t, t < 0 ? p.chain_stage : t, blockIdx.x - m.base[i], m.cnt[i], 1);
}
template <typename S>
__global__ void __launch_bounds__(kMaxSeqThreads + 32, sizeof(S) == 8 ? 4 : 1) k_fwd_seq_b(const BInst<S>* __restrict__ bi, BMap m) {
  const int i = m.inst[blockIdx.x], t = m.stage[i];
  const KP<S> p = bi[i].kp;
  const int top = p.chain_stage > 0 ? p.chain_stage : 1;
  fwd_seq_body<S>(p, t < 0 ? top : t, t < 0 ? p.N : t, bi[i].TVt, blockIdx.x - m.base[i], m.cnt[i], 1);
}

// ---------------------------------------------------------------------------
// launch shapes
// ---------------------------------------------------------------------------
// An attribute of the current device, read once (any thread may be first).
static int device_attr(cudaDeviceAttr attr, std::atomic<int>& cached) {
  int v = cached.load(std::memory_order_relaxed);
  if (v == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, attr, dev);
    cached.store(v, std::memory_order_relaxed);
  }
  return v;
}
static size_t max_dyn_smem() {
  static std::atomic<int> v{0};
  return (size_t)device_attr(cudaDevAttrMaxSharedMemoryPerBlockOptin, v);
}
static int num_sms() {
  static std::atomic<int> v{0};
  return device_attr(cudaDevAttrMultiProcessorCount, v);
}

// Threads per block (without the fetching warp): a multiple of 32 that covers
// the widest product times its row groups.  FP32 and FP64 below nx = 8: those of
// one group (FP64, 3 to 6 states, 511 nodes: 92 to 94 us an evaluation of T with
// any number; the groups' barriers cost what they save; a warp that holds several
// groups of so few columns works in them all the same).
template <typename S>
static int seq_threads(int nx, int nu, int groups) {
  const int CP = seq_cols<S>(nx, nu);
  if (sizeof(S) == 4) return CP;
  const int rg = nx < 8 ? 1 : std::max(1, std::min(groups, kMaxSeqThreads / CP));
  return (rg * CP + 31) & ~31;
}

struct SeqShape {
  int T, D, grid;
  size_t bytes;
};

// Threads, slots and grid for `cnt` sequences of Lq nodes.
//
// Slots: two where they fit, so that a block fetches a node while it works on
// the one before; half as many blocks are resident where shared memory bounds
// them.  One after another the FP64 chain kernels take as long with one slot as
// with two (62,805 nodes: 853 and 602 us, 884 and 575); in the stream, where a
// launch's first blocks start beside the last of the one before, they do not.
// One evaluation of T, one slot and two, us (nx, nu; nodes; chains):
//   FP64  6, 3    8,533 1,024  112, 108      33, 15    661    64   92,  84
//         24, 12    661    64   76,  69      33, 15 17,749 4,096  533, 371
//         24, 12 17,749 4,096  447, 441      50, 20 17,749 4,096  724, 607
//         64, 32 17,749 4,096 1,049, 985     50, 20 62,805 4,096 2,393, 2,017
//   FP32  24, 12 17,749 4,096  126, 109      50, 20 62,805 4,096  618, 604
// Sequences of one node gain by it only if blocks take several and a copy is
// long: full binary tree of 4,095 nodes, FP64, 3 KB a node (12, 5) 121, 128; 13 KB
// (24, 12) 178, 178; 48 KB (50, 20) 267, 240; a solve on 2,047 nodes, 16.5 KB (20,
// 20) 1,747, 1,778: FP64 from 20 KB.  FP32 (from 16 KB) waits for memory and not for the
// FP64 pipes and needs the blocks: with one block per SM many sequences lose
// (90, 38, 17,749 nodes: 447, 476), with two the single nodes (a solve on a full
// binary tree of 4,095 nodes, 50, 50: 1,396, 1,446; with four, on 21,845 nodes,
// 50, 20, 18 and 24 KB a node: 2,445, 2,369).
//
// FP64 row groups spread a node's multiply-adds over the four FP64 pipes of an
// SM.  Few sequences: up to four (one evaluation of T on 511 nodes, one to four
// groups: nx = 12, nu = 5 103, 92, 92, 92 us; 24, 12 117, 105, 103, 98; 50, 20
// 156, 130, 122, 122).  Many, whose blocks fill the pipes together: two (4,437
// nodes, one to three groups: 24, 12 149, 137, 147; 33, 15 182, 158, 171; 21,845
// nodes: 33, 15 475, 440, 473); three where the nodes' size leaves shared memory
// for five blocks or fewer (4,437 nodes, 50, 20: 273, 248, 225; 21,845 nodes:
// 787, 720, 682; 64, 32: 329, 325, 324).
template <typename S, typename F>
static SeqShape seq_shape(const KP<S>& p, int cnt, int Lq, F layout) {
  SeqShape s;
  const int sms = num_sms();
  const bool many = cnt > 2 * sms;
  auto fit = [](size_t bytes) { return (int)(228 * 1024 / (bytes + 1280)); };   // static part and the 1 KB of the system
  s.T = seq_threads<S>(p.nx, p.nu, many ? 2 : kMaxGroups);
  SeqLayout L = layout(p, s.T);
  if (sizeof(S) == 8 && many && fit(L.bytes(1)) < 6) {
    s.T = seq_threads<S>(p.nx, p.nu, 3);
    L = layout(p, s.T);
  }
  s.D = Lq > 1 || (cnt > sms && L.item >= (sizeof(S) == 8 ? 20 : 16) * 1024) ? kMaxSlots : 1;
  const int least = sizeof(S) == 8 ? 1 : (Lq == 1 ? 4 : (many ? 2 : 1));   // resident blocks
  while (s.D > 1 && (L.bytes(s.D) > max_dyn_smem() - 512 || fit(L.bytes(s.D)) < least)) --s.D;
  s.bytes = L.bytes(s.D);
  const int regs = sizeof(S) == 8 ? 64 : 80;
  const int by_thr = std::min(2048 / (s.T + 32), 65536 / ((s.T + 32) * regs));
  const int blocks = std::max(1, std::min(32, std::min(fit(s.bytes), by_thr)));
  s.grid = std::max(1, std::min(cnt, sms * blocks));
  return s;
}

// Raises a kernel's dynamic shared-memory limit, once per kernel and device, and
// asks for the largest shared-memory carve-out: left to itself the driver chose
// one per launch that held fewer blocks than planned (256 chains of nine nodes,
// nx = 33, nu = 15, FP64, two slots: an evaluation of T took 139 us, 114 with it;
// 64 chains of ten, 24, 12: 88, 69; FP32 within 3% either way).
template <typename F>
static void allow_smem(F* fn, std::atomic<uint64_t>& done) {
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return;
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(max_dyn_smem() - 512));
  cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  done.fetch_or(bit, std::memory_order_release);
}

template <typename S>
int launch_bwd_seq(const KP<S>& p, int t_hi, int t_lo, int cnt, cudaStream_t st) {
  const SeqShape s = seq_shape(p, cnt, t_hi - t_lo + 1, [](const KP<S>& q, int T) { return seq_layout_bwd(q, T); });
  static std::atomic<uint64_t> done{0};
  allow_smem(k_bwd_seq<S>, done);
  launch_pdl(k_bwd_seq<S>, s.grid, s.T + 32, s.bytes, st, p, t_hi, t_lo, s.D);
  return 1;
}
template <typename S>
int launch_lambda_seq(const KP<S>& p, int t_hi, int t_lo, int cnt, S* lam, cudaStream_t st) {
  const SeqShape s = seq_shape(p, cnt, t_hi - t_lo + 1, [](const KP<S>& q, int T) { return seq_layout_bwd(q, T); });
  static std::atomic<uint64_t> done{0};
  allow_smem(k_lambda_seq<S>, done);
  launch_pdl(k_lambda_seq<S>, s.grid, s.T + 32, s.bytes, st, p, t_hi, t_lo, lam, s.D);
  return 1;
}
template <typename S>
int launch_fwd_seq(const KP<S>& p, int t_lo, int t_hi, int cnt, S* zo, cudaStream_t st) {
  const SeqShape s = seq_shape(p, cnt, t_hi - t_lo + 1, [](const KP<S>& q, int T) { return seq_layout_fwd(q, T); });
  static std::atomic<uint64_t> done{0};
  allow_smem(k_fwd_seq<S>, done);
  launch_pdl(k_fwd_seq<S>, s.grid, s.T + 32, s.bytes, st, p, t_lo, t_hi, zo, s.D);
  return 1;
}

// One shape for a batch, whose blocks fill the SMs together: the most threads and
// shared memory over the instances.  Returns false if some instance's layout does not fit.
template <typename S>
bool seq_batch_shape(const std::vector<KP<S>>& kps, SeqBatchShape& sh) {
  sh.T = 32;
  for (const KP<S>& p : kps) sh.T = std::max(sh.T, seq_threads<S>(p.nx, p.nu, 2));
  sh.bytes_bwd = sh.bytes_fwd = 0;
  for (const KP<S>& p : kps) {
    sh.bytes_bwd = std::max(sh.bytes_bwd, seq_layout_bwd(p, sh.T).bytes(1));
    sh.bytes_fwd = std::max(sh.bytes_fwd, seq_layout_fwd(p, sh.T).bytes(1));
  }
  return std::max(sh.bytes_bwd, sh.bytes_fwd) <= max_dyn_smem() - 512;
}

// which = 0 backward chains, 1 backward stage, 2 forward stage, 3 forward chains
template <typename S>
void launch_seq_b(int which, const BInst<S>* bi, const BMap& m, int nblocks, const SeqBatchShape& sh,
                  cudaStream_t st) {
  if (nblocks <= 0) return;
  if (which <= 1) {
    static std::atomic<uint64_t> done{0};
    allow_smem(k_bwd_seq_b<S>, done);
    launch_pdl(k_bwd_seq_b<S>, nblocks, sh.T + 32, sh.bytes_bwd, st, bi, m);
  } else {
    static std::atomic<uint64_t> done{0};
    allow_smem(k_fwd_seq_b<S>, done);
    launch_pdl(k_fwd_seq_b<S>, nblocks, sh.T + 32, sh.bytes_fwd, st, bi, m);
  }
}

#define SPOCK_SEQ_INST(S)                                                                            \
  template int launch_bwd_seq<S>(const KP<S>&, int, int, int, cudaStream_t);                         \
  template int launch_lambda_seq<S>(const KP<S>&, int, int, int, S*, cudaStream_t);                  \
  template int launch_fwd_seq<S>(const KP<S>&, int, int, int, S*, cudaStream_t);                     \
  template bool seq_batch_shape<S>(const std::vector<KP<S>>&, SeqBatchShape&);                       \
  template void launch_seq_b<S>(int, const BInst<S>*, const BMap&, int, const SeqBatchShape&, cudaStream_t);
SPOCK_SEQ_INST(double)
SPOCK_SEQ_INST(float)

}  // namespace spock
