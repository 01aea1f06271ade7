// ns_cluster.cuh -- the cluster tree of section 2.1 on one thread block:
// recursive 2-means splits to a fixed depth, per-node covariance and FP64
// regularised Cholesky, bounding-ellipsoid volumes, bottom-up pruning, leaf
// assignment.
//
// Layout: the points are the live set x [d][n_pad] (unit cube).  Splits work
// on the points whitened by the root node's Cholesky factor, stored in
// y [d][n_pad]; side[j] holds point j's child choices, bit k at level k.
// Nodes are in heap order (root 0, children 2n+1, 2n+2).
//
// Determinism: every sum has a fixed thread -> point assignment and a fixed
// reduction tree (warp shuffles, then warps in order); maxima use atomicMax
// on order-preserving keys, which do not depend on order; the eigen-clips of
// several nodes share warps without sharing sums.  A run is therefore
// reproducible bit for bit.
#pragma once

#include <type_traits>

#include "ns_device.cuh"

namespace nsd {

constexpr int kMaxLeaves = 64;  // depth <= 6
constexpr int kRedW = 64;       // partial sums per warp (slot_sums)
constexpr int kSumRows = 64;    // rows of a warp's buffer in slot_sums, at most kRedW

// Scratch of one tree build; L = 2^depth leaves, n_nodes = 2 L - 1.
struct TreeScratch {
  float* c;           // [L][d]: the two centres of each node of the current level (slot 2q+s)
  float* red;         // [nwarps][kRedW] partial sums (slot_sums)
  unsigned long long* far;  // [L / 2] farthest members of the current level: distance bits, slot
  int* cnt;           // [2 L]: members per node of the level, then per (node, side) slot
  int* misc;          // [8]
  double* leaf_mu;    // [L][d]: merge weights of the current level
  double* node_mu;    // [n_nodes][d]
  double* node_M2;    // [n_nodes][d*d]   (d*d: full symmetric, for the Cholesky; the centre sums before)
  int* node_n;        // [n_nodes]
  unsigned* node_m2;  // [n_nodes] bits of the largest squared Mahalanobis distance
  double* lv;         // [n_nodes] log volumes
  double* veff;       // [n_nodes] effective (pruned) log volumes
  int* spl;           // [n_nodes] accepted splits
};

constexpr int kTreeHot = 5;  // the tables that the splits work on are the layout's first

template <class F>
__host__ __device__ inline void tree_layout(int d, int n_nodes, int nwarps, F&& take) {
  const int L = (n_nodes + 1) / 2;
  take(0, sizeof(float) * L * d);
  take(1, sizeof(float) * nwarps * kRedW);
  take(2, sizeof(unsigned long long) * L);
  take(3, sizeof(int) * L * 2);
  take(4, sizeof(int) * 8);
  take(5, sizeof(double) * L * d);
  take(6, sizeof(double) * n_nodes * d);
  take(7, sizeof(double) * (size_t)n_nodes * d * d);
  take(8, sizeof(int) * n_nodes);
  take(9, sizeof(unsigned) * n_nodes);
  take(10, sizeof(double) * n_nodes);
  take(11, sizeof(double) * n_nodes);
  take(12, sizeof(int) * n_nodes);
}

// Bytes of the first n_tables tables of the layout (by default all).
__host__ __device__ inline size_t tree_bytes(int d, int n_nodes, int nwarps, int n_tables = 13) {
  if (n_nodes <= 1) return 0;
  size_t b = 0;
  tree_layout(d, n_nodes, nwarps, [&](int k, size_t x) {
    if (k < n_tables) b += (x + 15) & ~(size_t)15;
  });
  return b;
}

// The tree's share of a handle's arena (spilled runs), and the size by which a
// run spills: the tables for nwarps warps and room for factorising several
// nodes at once (up to 48 KB).  Fixed: a checkpoint restores only into an
// arena of the same layout.
__host__ __device__ inline size_t tree_arena_bytes(int d, int n_nodes, int nwarps) {
  if (n_nodes <= 1) return 0;
  const size_t per = sizeof(double) * (5 * d * d + d);
  size_t w = 48 * 1024 / per;
  w = w < 1 ? 1 : (w > 8 ? 8 : w);
  return tree_bytes(d, n_nodes, nwarps) + sizeof(float) * kRedW + ((w * per + 15) & ~(size_t)15);
}

// hot: where the tables of the splits live (base itself, or shared memory when
// the others are in global memory).
__device__ inline TreeScratch tree_carve(char* base, char* hot, int d, int n_nodes, int nwarps) {
  char* p[13];
  size_t o = 0;
  tree_layout(d, n_nodes, nwarps, [&](int k, size_t x) {
    p[k] = (k < kTreeHot ? hot : base) + o;
    o += (x + 15) & ~(size_t)15;
  });
  TreeScratch T;
  T.c = reinterpret_cast<float*>(p[0]);
  T.red = reinterpret_cast<float*>(p[1]);
  T.far = reinterpret_cast<unsigned long long*>(p[2]);
  T.cnt = reinterpret_cast<int*>(p[3]);
  T.misc = reinterpret_cast<int*>(p[4]);
  T.leaf_mu = reinterpret_cast<double*>(p[5]);
  T.node_mu = reinterpret_cast<double*>(p[6]);
  T.node_M2 = reinterpret_cast<double*>(p[7]);
  T.node_n = reinterpret_cast<int*>(p[8]);
  T.node_m2 = reinterpret_cast<unsigned*>(p[9]);
  T.lv = reinterpret_cast<double*>(p[10]);
  T.veff = reinterpret_cast<double*>(p[11]);
  T.spl = reinterpret_cast<int*>(p[12]);
  return T;
}

// The node of a point with side bits `bits` at level lev, counted within the
// level: the low lev bits reversed.  (At level 0 the one node, 0.)
__device__ __forceinline__ int level_slot(int bits, int lev) {
  return lev == 0 ? 0 : (int)(__brev((unsigned)bits) >> (32 - lev));
}

// Sums of n_items values over the points of each of n_slots slots: out(item,
// slot, sum) with sum = the FP32 sum of val(item, j, slot) over the points j
// with slot_of(j) == slot (slots outside [0, n_slots): none); val gets
// prep(item) for the item.
//
// The order of every sum is fixed by vb alone: point j belongs to virtual
// thread j % vb, which adds its points in ascending order; the 32 threads of
// a virtual warp are added pairwise (lanes 16 apart, then 8, 4, 2, 1), the
// virtual warps in order.  A real warp takes one virtual warp's points for as
// many items as fit its buffer of `rows` rows (a row per item and slot,
// stride 33 so that neither columns nor rows collide on banks): each lane
// adds its points into its own column, then lanes add up rows.  Per point and
// item that is one load, add and store whatever the number of slots, and a
// pass of the block takes rows / n_slots items at once.  (Comparing each point
// with every slot of a register table and reducing every slot by shuffles
// takes 60 of the 86 k cycles of a Lloyd iteration over 64 slots, 2000
// points, d = 10; this 7 k.)
template <int K>
struct Items {
  static constexpr int value = K;
};
template <class SlotOf, class Prep, class Val, class Out>
__device__ __forceinline__ void slot_sums(int N, int vb, int n_slots, int n_items, int rows, float* pbuf, float* red,
                                          SlotOf slot_of, Prep prep, Val val, Out out) {
  const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = B >> 5, nv = vb >> 5;
  const int teams = nw / nv, team = wid / nv, vw = wid - team * nv;  // a team: a warp per virtual warp
  const int SC = min(n_slots, rows), IP = rows / SC;                 // slots and items of a pass
  const int sc_log = 31 - __clz(SC);
  float* pb = pbuf + (size_t)wid * rows * 33;
  const int passes = ((n_slots + SC - 1) / SC) * ((n_items + IP - 1) / IP), ipasses = (n_items + IP - 1) / IP;
  for (int p0 = 0; p0 < passes; p0 += teams) {
    const int p = p0 + team, s0 = (p / ipasses) * SC, it0 = (p % ipasses) * IP;
    if (team < teams && p < passes) {
      const int ns = min(SC, n_slots - s0), ni = min(IP, n_items - it0), nr = ni * SC;
      for (int r = 0; r < nr; ++r) pb[r * 33 + lane] = 0.f;
      constexpr int U = 4;  // points in flight
      for (int j0 = vw * 32; j0 < N; j0 += U * vb) {
        int g[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int j = j0 + q * vb + lane;
          g[q] = j < N ? slot_of(j) : -1;
          if (g[q] < s0 || g[q] >= s0 + ns) g[q] = -1;
        }
        auto add = [&](int it, auto K) {  // K items' rows at a time: their adds do not wait for one another
          constexpr int kItems = decltype(K)::value;
          decltype(prep(0)) ctx[kItems];
#pragma unroll
          for (int k = 0; k < kItems; ++k) ctx[k] = prep(it0 + it + k);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            if (g[q] < 0) continue;
            float* at = pb + (it * SC + g[q] - s0) * 33 + lane;
            float v[kItems];
#pragma unroll
            for (int k = 0; k < kItems; ++k) v[k] = at[k * SC * 33];
#pragma unroll
            for (int k = 0; k < kItems; ++k) v[k] = __fadd_rn(v[k], val(ctx[k], j0 + q * vb + lane, g[q]));
#pragma unroll
            for (int k = 0; k < kItems; ++k) at[k * SC * 33] = v[k];
          }
        };
        int it = 0;
        for (; it + 4 <= ni; it += 4) add(it, Items<4>());
        for (; it < ni; ++it) add(it, Items<1>());
      }
      __syncwarp();
      for (int r = lane; r < nr; r += 32) {
        const float* row = pb + r * 33;
        float t[16];
#pragma unroll
        for (int l = 0; l < 16; ++l) t[l] = __fadd_rn(row[l], row[l + 16]);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
          for (int l = 0; l < o; ++l) t[l] = __fadd_rn(t[l], t[l + o]);
        red[wid * kRedW + r] = t[0];
      }
    }
    __syncthreads();
    for (int q = tid; q < teams * rows; q += B) {  // n_slots and rows are powers of two
      const int tm = q / rows, r = q - tm * rows, pq = p0 + tm;
      if (pq >= passes) continue;
      const int sp = pq / ipasses, ip = pq - sp * ipasses;
      const int item = ip * IP + (r >> sc_log), slot = sp * SC + (r & (SC - 1));
      if (item < n_items && slot < n_slots) {
        float s = 0.f;
        for (int w = 0; w < nv; ++w) s = __fadd_rn(s, red[(tm * nv + w) * kRedW + r]);
        out(item, slot, s);
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ double logaddexp_d(double a, double b) {
  if (a == -CUDART_INF) return b;
  if (b == -CUDART_INF) return a;
  const double mx = fmax(a, b);
  return mx + log1p(exp(-fabs(a - b)));
}

// The tree for depth D >= 1.  Inputs: x, the root's mean mu0 (float [d])
// and FP32 Cholesky L0 (float [d][d]), and its count in node_n[0] (filled by
// the caller, with its centre, factors and log volume in the outputs).
// Outputs: per node centre (float), chol (float + FP64), logvol, count,
// split, mask; cid[j] = accepted leaf of point j.
struct TreeIO {
  const float* x;
  float* y;
  uint8_t* side;
  int N, n_pad, d, depth, n_min, kmeans_iters;
  float vol_frac;
  uint32_t k0, k1, t;
  float* centres;   // global [n_nodes][d]
  float* chol;      // global [n_nodes][d][d]
  double* chol64;   // global
  float* logvol;    // global
  int* count;       // global
  int* split;       // global
  int* mask;        // global
  int* cid;         // global [N]
  float* s_chol;    // smem [n_nodes][d][d]
  float* s_cent;    // smem [n_nodes][d]
  int* s_mask;      // smem [n_nodes]
  int bracket;      // 1: the FP32 factors (the directions') scaled by each node's bounding radius
  int vb;           // threads whose points and order the FP32 sums follow (slot_sums)
  float* pbuf;      // smem: rows * 33 floats per warp (slot_sums)
  int rows;
  float* stage;     // smem: the points [d][N] and their child bits [N], or null (too many)
  size_t work_bytes;  // bytes at pbuf that the eigen-clips may use (pbuf and stage)
};

// Squared Mahalanobis distance of live point j from mu in the units of the
// FP32 factor L (forward substitution).  DM: a register class >= d.
template <int DM, class Ld>
__device__ __forceinline__ float mahalanobis2(const float* live_x, Ld n_pad, int j, int d, const float* L,
                                              const float* mu) {
  float r[DM];
  float s2 = 0.f;
#pragma unroll
  for (int i = 0; i < DM; ++i) r[i] = i < d ? live_x[i * n_pad + j] - mu[i] : 0.f;
#pragma unroll
  for (int i = 0; i < DM; ++i)
    if (i < d) {
      float s = r[i];
#pragma unroll
      for (int k = 0; k < i; ++k) s = fmaf(-L[i * d + k], r[k], s);
      r[i] = s / L[i * d + i];
      s2 = fmaf(r[i], r[i], s2);
    }
  return s2;
}

// This thread's largest squared Mahalanobis distance, over the live points
// j = tid, tid + blockDim.x, ... < N (live_x [d][n_pad]), as the bits of a
// non-negative float (ordered like the values, for atomicMax).
template <int DM>
__device__ __noinline__ unsigned max_mahalanobis2(const float* __restrict__ live_x, int n_pad, int N, int d,
                                                  const float* L, const float* mu) {
  float best = 0.f;
  for (int j = threadIdx.x; j < N; j += blockDim.x) best = fmaxf(best, mahalanobis2<DM>(live_x, (size_t)n_pad, j, d, L, mu));
  return __float_as_uint(best);
}

// The eigen-clips of the listed nodes (fail[0 .. n_fail)), whose Cholesky
// met a pivot that is not positive: a leaf with no more members than
// dimensions has a singular covariance, so a deep tree has dozens of them.
// The rotations and sums of jacobi_eigen_warp, several nodes side by side in a
// warp: an FP64 instruction costs a warp 64 cycles on this part whether one
// lane or 32 use it, and most of a rotation is the divisions and square
// roots of its angle, so JL lanes per node (as many as keep four warps
// busy) cut the time by 32 / JL where nodes are many.  A node's result does
// not depend on JL, on the slots or on its place in the list (which the
// warps fill in any order).  C(nd, i, k): the covariance; done(f0, nf, work,
// per): the clipped matrices of the nodes fail[f0 .. f0 + nf).  work: FP64
// [slots][2 d d + d].  Every thread of the block.
template <class Cov, class Done>
__device__ __noinline__ void clip_nodes(int d, const int* fail, int n_fail, double* work, int slots, Cov C, Done done) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, dd = d * d, per = 2 * dd + d;
  for (int f0 = 0; f0 < n_fail; f0 += slots) {
    const int nf = min(slots, n_fail - f0);
    __syncthreads();
    for (int e = threadIdx.x; e < nf * dd; e += blockDim.x) {
      const int f = e / dd, q = e - f * dd, i = q / d, k = q - i * d;
      work[f * per + q] = C(fail[f0 + f], i, k);
      work[f * per + dd + q] = i == k ? 1.0 : 0.0;
    }
    __syncthreads();
    int JL = 32;
    while (JL > 2 && JL * nf > 128) JL >>= 1;
    const int npw = 32 / JL, g = lane % JL;
    for (int w0 = wid * npw; w0 < nf; w0 += nw * npw) {  // (uniform in the warp)
      const int f = w0 + lane / JL;
      const bool mine = f < nf;
      double* A = work + (mine ? f : w0) * per;
      double* Q = A + dd;
      bool open = mine;
      for (int sweep = 0; sweep < 100; ++sweep) {
        // the sums of squares above and on the diagonal, the whole warp on one
        // node after another: in the order of jacobi_eigen_warp whatever JL is
        double off = 0.0, dia = 0.0;
        for (int u = 0; u < npw; ++u) {
          if (!__any_sync(kFull, open && lane / JL == u)) continue;
          const double* Au = work + (w0 + u) * per;
          double o = 0.0, e = 0.0;
          for (int i = lane; i < dd; i += 32) {
            const int a = i / d, b = i - a * d;
            const double v = Au[i];
            if (b > a) o += v * v;
            else if (a == b) e += v * v;
          }
#pragma unroll
          for (int h = 16; h > 0; h >>= 1) {
            o += __shfl_xor_sync(kFull, o, h);
            e += __shfl_xor_sync(kFull, e, h);
          }
          if (lane / JL == u) {
            off = o;
            dia = e;
          }
        }
        open = open && off > 1e-30 * dia;
        if (!__any_sync(kFull, open)) break;
        for (int p = 0; p < d; ++p)
          for (int q = p + 1; q < d; ++q) {
            const double apq = A[p * d + q];
            const bool turn = open && apq != 0.0;
            const double th = (A[q * d + q] - A[p * d + p]) / (2.0 * (turn ? apq : 1.0));
            const double tt = (th >= 0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            const double c = 1.0 / sqrt(tt * tt + 1.0), s = tt * c;
            __syncwarp();
            if (turn)
              for (int k = g; k < d; k += JL) {
                const double akp = A[k * d + p], akq = A[k * d + q];
                A[k * d + p] = c * akp - s * akq;
                A[k * d + q] = s * akp + c * akq;
              }
            __syncwarp();
            if (turn)
              for (int k = g; k < d; k += JL) {
                const double apk = A[p * d + k], aqk = A[q * d + k];
                A[p * d + k] = c * apk - s * aqk;
                A[q * d + k] = s * apk + c * aqk;
                const double qkp = Q[k * d + p], qkq = Q[k * d + q];
                Q[k * d + p] = c * qkp - s * qkq;
                Q[k * d + q] = s * qkp + c * qkq;
              }
            __syncwarp();
          }
      }
    }
    __syncthreads();
    // the clipped eigenvalues, then A <- Q diag Q^T (the regularisation is added by `done`)
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
      double* A = work + f * per;
      double lmax = 0.0;
      for (int i = 0; i < d; ++i) lmax = fmax(lmax, A[i * d + i]);
      for (int i = 0; i < d; ++i) A[2 * dd + i] = fmax(A[i * d + i], 1e-10 * lmax);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nf * dd; e += blockDim.x) {
      const int f = e / dd, q = e - f * dd, i = q / d, j = q - i * d;
      double* A = work + f * per;
      const double* Q = A + dd;
      double s = 0.0;
      for (int k = 0; k < d; ++k) s += Q[i * d + k] * A[2 * dd + k] * Q[j * d + k];
      A[q] = s;
    }
    __syncthreads();
    done(f0, nf, work, per);
  }
  __syncthreads();
}

// Index type of a point table [d][ld]: 64 bits in global memory, where d n_pad
// is bounded by the caller's memory alone.
template <bool SMEM>
using PointIndex = std::conditional_t<SMEM, int, size_t>;

template <bool SMEM, class P>
__device__ __forceinline__ P* in_smem(char* sm, P* p) {  // p in shared memory, so that the compiler knows it
  if constexpr (SMEM) return reinterpret_cast<P*>(sm + (smem_addr(p) - smem_addr(sm)));
  else return p;
}

// SMEM: the points are staged (io.stage) and the factors are in shared memory.
// (Global loads hardly ever hit the L1 in these kernels, and each pass over
// the points was bound by their latency.)
template <int DM, bool SMEM>
__device__ __noinline__ void cluster_tree(const TreeIO& io_ref, const TreeScratch& T_ref, BlockScratch& S) {
  extern __shared__ __align__(16) char sm[];
  TreeIO io = io_ref;
  TreeScratch T = T_ref;
  const int tid = threadIdx.x, B = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = B >> 5;
  const int d = io.d, N = io.N, D = io.depth, n_nodes = (1 << (D + 1)) - 1;
  const int n_leaves = 1 << D;
  io.s_chol = in_smem<SMEM>(sm, io.s_chol);
  io.s_cent = in_smem<SMEM>(sm, io.s_cent);
  io.pbuf = in_smem<SMEM>(sm, io.pbuf);
  T.c = in_smem<SMEM>(sm, T.c);
  T.red = in_smem<SMEM>(sm, T.red);
  T.cnt = in_smem<SMEM>(sm, T.cnt);
  T.far = in_smem<SMEM>(sm, T.far);
  float* const y = SMEM ? in_smem<SMEM>(sm, io.stage) : io.y;
  const PointIndex<SMEM> ld = SMEM ? N : io.n_pad;
  uint8_t* const side = SMEM ? reinterpret_cast<uint8_t*>(y + d * N) : io.side;
  const size_t n_pad = io.n_pad;
  // ---- whiten by the root factor: y = L0^{-1} (x - mu0) ------------------
  for (int j = tid; j < N; j += B) {
    float r[DM];
#pragma unroll
    for (int i = 0; i < DM; ++i) r[i] = i < d ? io.x[i * n_pad + j] - io.s_cent[i] : 0.f;
#pragma unroll
    for (int i = 0; i < DM; ++i)
      if (i < d) {
        float s = r[i];
#pragma unroll
        for (int k = 0; k < i; ++k) s = fmaf(-io.s_chol[i * d + k], r[k], s);
        r[i] = s / io.s_chol[i * d + i];
        y[i * ld + j] = r[i];
      }
    side[j] = 0;
  }
  __syncthreads();
  // ---- 2-means splits, level by level -------------------------------------
  for (int lev = 0; lev < D; ++lev) {
    const int first = (1 << lev) - 1, nlev = 1 << lev;
    // members per node of this level
    for (int q = tid; q < 2 * n_leaves; q += B) T.cnt[q] = (lev == 0 && q == 0) ? N : 0;
    for (int q = tid; q < 2 * nlev; q += B) reinterpret_cast<unsigned*>(T.far)[q] = (q & 1) ? 0xFFFFFFFFu : 0u;
    __syncthreads();
    if (lev > 0) {
      for (int j = tid; j < N; j += B) atomicAdd(&T.cnt[level_slot(side[j], lev)], 1);
      __syncthreads();
    }
    // first centre: the Philox-chosen member (ascending slot order), a warp
    // per node
    for (int q = wid; q < nlev; q += nw) {
      const int n_mem = T.cnt[q];
      if (n_mem < 2) continue;
      int p = u_index(draw_at(io.k0, io.k1, io.t, (uint32_t)(first + q), kPurposeKmeans, 0), n_mem);
      int at = p;
      if (lev > 0) {
        for (int jb = 0; jb < N; jb += 32) {
          const bool mine = jb + lane < N && level_slot(side[jb + lane], lev) == q;
          unsigned b = __ballot_sync(kFull, mine);
          const int n = __popc(b);
          if (p < n) {
            for (; p > 0; --p) b &= b - 1;
            at = jb + __ffs(b) - 1;
            break;
          }
          p -= n;
        }
      }
      for (int i = lane; i < d; i += 32) T.c[(2 * q) * d + i] = y[i * ld + at];
    }
    __syncthreads();
    // second centre: the member farthest from the first (ties: lowest slot):
    // the largest distance of each node, then the lowest slot that has it.
    // far[q] as two words: distance bits, slot.  (cid holds the distances.)
    for (int jb = 0; jb < N; jb += B) {
      const int j = jb + tid;
      unsigned bits = 0u;
      int q = -1;
      if (j < N) {
        q = level_slot(side[j], lev);
        if (T.cnt[q] >= 2) {
          float s = 0.f;
#pragma unroll
          for (int i = 0; i < DM; ++i)
            if (i < d) {
              const float u = y[i * ld + j] - T.c[(2 * q) * d + i];
              s = fmaf(u, u, s);
            }
          bits = __float_as_uint(s);
        } else {
          q = -1;
        }
        io.cid[j] = (int)bits;
      }
      if (lev == 0) {
        const unsigned mx = __reduce_max_sync(kFull, bits);
        if (lane == 0 && N >= 2) atomicMax(reinterpret_cast<unsigned*>(T.far), mx);
      } else if (q >= 0) {
        atomicMax(reinterpret_cast<unsigned*>(T.far) + 2 * q, bits);
      }
    }
    __syncthreads();
    for (int j = tid; j < N; j += B) {
      const int q = level_slot(side[j], lev);
      unsigned* f = reinterpret_cast<unsigned*>(T.far) + 2 * q;
      if (T.cnt[q] >= 2 && (unsigned)io.cid[j] == f[0]) atomicMin(f + 1, (unsigned)j);
    }
    __syncthreads();
    for (int e = tid; e < nlev * d; e += B) {
      const int q = e / d, i = e - q * d;
      if (T.cnt[q] >= 2) T.c[(2 * q + 1) * d + i] = y[i * ld + reinterpret_cast<unsigned*>(T.far)[2 * q + 1]];
    }
    __syncthreads();
    // Lloyd iterations: assign, then move the centres; stop at a fixed point
    for (int it = 0; it < io.kmeans_iters; ++it) {
      int changed = 0;
      constexpr int U = 4;  // points in flight
      for (int j0 = tid; j0 < N; j0 += U * B) {
        int bits[U];
        const float* c0[U];
        bool on[U];
        float s0[U], s1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + u * B;
          bits[u] = j < N ? side[j] : 0;
          const int q = level_slot(bits[u], lev);
          on[u] = j < N && T.cnt[q] >= 2;
          c0[u] = T.c + (2 * q) * d;
          s0[u] = s1[u] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < DM; ++i)
          if (i < d) {
            float yi[U];
#pragma unroll
            for (int u = 0; u < U; ++u) yi[u] = on[u] ? y[i * ld + j0 + u * B] : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const float u0 = yi[u] - c0[u][i];
              const float u1 = yi[u] - c0[u][d + i];
              s0[u] = fmaf(u0, u0, s0[u]);
              s1[u] = fmaf(u1, u1, s1[u]);
            }
          }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int sd = (s1[u] < s0[u]) ? 1 : 0;
          if (on[u] && (it == 0 || sd != ((bits[u] >> lev) & 1))) {
            changed = 1;
            side[j0 + u * B] = (uint8_t)((bits[u] & ~(1 << lev)) | (sd << lev));
          }
        }
      }
      const int any = __syncthreads_or(changed);
      if (!any) break;
      // counts (exact in FP32) and centre sums of the (node, side) slots; a slot
      // left empty, or of a node with fewer than two members, keeps its centre
      const int slots = 2 * nlev;
      int* scount = T.cnt + n_leaves;
      auto slot = [&](int j) { return level_slot(side[j], lev + 1); };
      float* sums = reinterpret_cast<float*>(T.node_M2);  // (not in use yet)
      slot_sums(
          N, io.vb, slots, d + 1, io.rows, io.pbuf, T.red, slot,
          [&](int c) { return c == 0 ? nullptr : y + (c - 1) * ld; },
          [&](const float* yc, int j, int) { return yc ? yc[j] : 1.f; },
          [&](int c, int s, float sum) {
            if (c == 0) scount[s] = (int)sum;
            else sums[s * d + c - 1] = sum;
          });
      for (int e = tid; e < slots * d; e += B) {
        const int s = e / d;
        if (T.cnt[s >> 1] >= 2 && scount[s] != 0) T.c[e] = sums[e] / (float)scount[s];
      }
      __syncthreads();
    }
    // nodes with fewer than two members keep every member in the first child
    __syncthreads();
  }
  // ---- node statistics: leaf means, leaf centred products, pairwise merge ---
  const int last_first = n_leaves - 1;
  const int ne = d * (d + 1) / 2;
  // counts per leaf
  for (int q = tid; q < 2 * n_leaves; q += B) T.cnt[q] = 0;
  __syncthreads();
  for (int j = tid; j < N; j += B) atomicAdd(&T.cnt[level_slot(side[j], D)], 1);
  __syncthreads();
  // the points themselves from here on
  const float* const xs = SMEM ? y : io.x;
  if (SMEM) {
    for (int i = wid; i < d; i += nw)
      for (int j = lane; j < N; j += 32) y[i * ld + j] = io.x[i * n_pad + j];
    __syncthreads();
  }
  // leaf means (sums relative to the root mean, FP32 per thread, FP64 after);
  // the FP32 means in T.c (the centres are no longer needed)
  auto leaf_of = [&](int j) { return level_slot(side[j], D); };
  slot_sums(
      N, io.vb, n_leaves, d, io.rows, io.pbuf, T.red, leaf_of, [&](int c) { return c; },
      [&](int c, int j, int) { return xs[c * ld + j] - io.s_cent[c]; },
      [&](int c, int l, float sum) {
        const int n = T.cnt[l];
        const double mu = n > 0 ? (double)sum / n + (double)io.s_cent[c] : 0.0;
        T.node_mu[(last_first + l) * d + c] = mu;
        T.c[l * d + c] = (float)mu;
        T.node_n[last_first + l] = n;
      });
  // leaf centred products
  slot_sums(
      N, io.vb, n_leaves, ne, io.rows, io.pbuf, T.red, leaf_of,
      [&](int e) {
        const int a = packed_row(e);
        return make_int2(a, e - a * (a + 1) / 2);
      },
      [&](int2 ab, int j, int l) {
        const float ua = xs[ab.x * ld + j] - T.c[l * d + ab.x];
        const float ub = xs[ab.y * ld + j] - T.c[l * d + ab.y];
        return __fmul_rn(ua, ub);
      },
      [&](int e, int l, float sum) {
        const int a = packed_row(e);
        const int b = e - a * (a + 1) / 2;
        const int nd = last_first + l;
        T.node_M2[(size_t)nd * d * d + a * d + b] = (double)sum;
        T.node_M2[(size_t)nd * d * d + b * d + a] = (double)sum;
      });
  // internal nodes below the root: merge the children (Chan et al.), level
  // by level; leaf_mu [n1 n2 / n] holds each merged node's weight
  for (int lev = D - 1; lev >= 1; --lev) {
    const int f0 = (1 << lev) - 1, nlev = 1 << lev;
    for (int q = tid; q < nlev; q += B) {
      const int nd = f0 + q, n1 = T.node_n[2 * nd + 1], n2 = T.node_n[2 * nd + 2], n = n1 + n2;
      T.node_n[nd] = n;
      T.leaf_mu[q] = n > 0 ? (double)n1 * n2 / n : 0.0;
    }
    __syncthreads();
    for (int e = tid; e < nlev * d * d; e += B) {
      const int qn = e / (d * d), q = e - qn * d * d, a = q / d, b = q - a * d;
      const int nd = f0 + qn, c1 = 2 * nd + 1, c2 = 2 * nd + 2;
      const int n1 = T.node_n[c1], n2 = T.node_n[c2];
      double v = T.node_M2[c1 * d * d + q] + T.node_M2[c2 * d * d + q];
      if (n1 > 0 && n2 > 0) {
        const double da = T.node_mu[c1 * d + a] - T.node_mu[c2 * d + a];
        const double db = T.node_mu[c1 * d + b] - T.node_mu[c2 * d + b];
        v += da * db * T.leaf_mu[qn];
      }
      T.node_M2[nd * d * d + q] = v;
    }
    for (int e = tid; e < nlev * d; e += B) {
      const int qn = e / d, i = e - qn * d, nd = f0 + qn, c1 = 2 * nd + 1, c2 = 2 * nd + 2;
      const int n1 = T.node_n[c1], n2 = T.node_n[c2], n = n1 + n2;
      T.node_mu[nd * d + i] = n > 0 ? (T.node_mu[c1 * d + i] * n1 + T.node_mu[c2 * d + i] * n2) / n : 0.0;
    }
    __syncthreads();
  }
  // ---- Cholesky of every node below the root: 32 / GL nodes per warp, a lane
  // per row (FP64 instructions are what it costs: one per warp whatever the
  // number of rows in use); nodes whose covariance fails are listed and take
  // the eigen-clip ----------------------------------------------------------
  int* const fail = T.cnt;  // [n_leaves * 2 > n_nodes] (the counts are in node_n now)
  if (tid == 0) T.misc[0] = 0;
  __syncthreads();
  constexpr int GL = chol_lanes(DM), NPW = 32 / GL;
  auto store_row = [&](int nd, int i, const double (&a)[DM]) {
#pragma unroll
    for (int k = 0; k < DM; ++k)
      if (k < d) {
        const double v = k <= i ? a[k] : 0.0;
        const float f = (float)v;
        io.chol64[(size_t)nd * d * d + i * d + k] = v;
        io.chol[(size_t)nd * d * d + i * d + k] = f;
        io.s_chol[nd * d * d + i * d + k] = f;
      }
  };
  {
    const int sub = lane / GL, i = lane % GL;
    for (int nd0 = 1 + wid * NPW; nd0 < n_nodes; nd0 += nw * NPW) {
      const int nd = nd0 + sub;
      const bool act = nd < n_nodes && i < d;
      const int n = nd < n_nodes ? T.node_n[nd] : 0;
      const double inv = n > 0 ? 1.0 / n : 0.0;
      double a[DM];
#pragma unroll
      for (int k = 0; k < DM; ++k)
        a[k] = (act && k <= i && k < d) ? __dmul_rn(T.node_M2[(size_t)nd * d * d + i * d + k], inv) : 0.0;
      const int how = reg_chol_rows<DM>(d, i, a, true);  // per node: 0 fails
      if (act) {
        if (how) store_row(nd, i, a);
        const float c = (float)T.node_mu[nd * d + i];
        io.centres[nd * d + i] = c;
        io.s_cent[nd * d + i] = c;
      }
      if (nd < n_nodes && i == 0) {
        T.lv[nd] = inv;  // (for the clips)
        if (!how) fail[atomicAdd(&T.misc[0], 1)] = nd;
      }
    }
  }
  __syncthreads();
  const int n_fail = T.misc[0];
  if (n_fail > 0) {
    auto cov = [&](int nd, int i, int k) { return __dmul_rn(T.node_M2[(size_t)nd * d * d + i * d + k], T.lv[nd]); };
    // the work slots overlay the slot sums' buffer and the staged points
    const int slots = max(1, (int)(io.work_bytes / (sizeof(double) * (2 * d * d + d))));
    clip_nodes(d, fail, n_fail, reinterpret_cast<double*>(io.pbuf), slots, cov,
               [&](int f0, int nf, double* work, int per) {
                 const int sub = lane / GL, i = lane % GL;
                 for (int b0 = wid * NPW; b0 < nf; b0 += nw * NPW) {
                   const int f = b0 + sub, nd = f < nf ? fail[f0 + f] : 0;
                   const bool act = f < nf && i < d;
                   // C's regularisation, then the clipped matrix with it
                   double tr = act ? cov(nd, i, i) : 0.0;
#pragma unroll
                   for (int o = GL / 2; o > 0; o >>= 1) tr = __dadd_rn(tr, __shfl_xor_sync(kFull, tr, o, GL));
                   const double delta = 1e-10 * tr / d;
                   double a[DM];
#pragma unroll
                   for (int k = 0; k < DM; ++k) {
                     a[k] = (act && k <= i && k < d) ? work[f * per + i * d + k] : 0.0;
                     if (act && k == i) a[k] = __dadd_rn(a[k], delta);
                   }
                   double diag = 0.0;
#pragma unroll
                   for (int k = 0; k < DM; ++k)
                     if (k == i) diag = a[k];
                   const int how = reg_chol_rows<DM>(d, i, a, false);
                   if (!how) {
#pragma unroll
                     for (int k = 0; k < DM; ++k) a[k] = k == i ? sqrt(diag > 0 ? diag : 1e-12) : 0.0;
                   }
                   if (act) store_row(nd, i, a);
                 }
               });
    if (SMEM) {
      for (int i = wid; i < d; i += nw)
        for (int j = lane; j < N; j += 32) y[i * ld + j] = io.x[i * n_pad + j];
    }
  }
  __syncthreads();
  // ---- bounding ellipsoids: largest squared Mahalanobis distance per node ---
  for (int q = tid; q < n_nodes; q += B) T.node_m2[q] = 0u;
  __syncthreads();
  for (int lev = 0; lev <= D; ++lev)
    for (int jb = 0; jb < N; jb += B) {
      const int j = jb + tid;
      unsigned m2 = 0u;
      int nd = 0;
      if (j < N) {
        nd = (1 << lev) - 1 + level_slot(side[j], lev);
        m2 = __float_as_uint(mahalanobis2<DM>(xs, ld, j, d, io.s_chol + nd * d * d, io.s_cent + nd * d));
      }
      if (lev == 0) {
        m2 = __reduce_max_sync(kFull, m2);
        if (lane == 0) atomicMax(&T.node_m2[0], m2);
      } else if (j < N) {
        atomicMax(&T.node_m2[nd], m2);
      }
    }
  __syncthreads();
  // ---- volumes, pruning bottom-up, accepted leaves --------------------------
  for (int nd = tid; nd < n_nodes; nd += B) {
    const int n = T.node_n[nd];
    double l = 0.0;
    for (int i = 0; i < d; ++i) l += log((double)io.s_chol[(size_t)nd * d * d + i * d + i]);
    const double m2 = (double)__uint_as_float(T.node_m2[nd]);
    T.lv[nd] = (n > 0) ? l + 0.5 * d * log(m2) : -CUDART_INF;
  }
  __syncthreads();
  for (int lev = D; lev >= 0; --lev) {
    for (int q = tid; q < (1 << lev); q += B) {
      const int nd = (1 << lev) - 1 + q, c1 = 2 * nd + 1, c2 = 2 * nd + 2;
      if (lev == D) {
        T.spl[nd] = 0;
        T.veff[nd] = T.lv[nd];
      } else {
        const double vc = logaddexp_d(T.veff[c1], T.veff[c2]);
        const int ok =
            T.node_n[c1] > io.n_min && T.node_n[c2] > io.n_min && vc < log(1.0 - (double)io.vol_frac) + T.lv[nd];
        T.spl[nd] = ok;
        T.veff[nd] = ok ? vc : T.lv[nd];
      }
    }
    __syncthreads();
  }
  for (int nd = tid; nd < n_nodes; nd += B) {
    int act = 1;  // every ancestor split
    for (int k = nd; k > 0; k = (k - 1) / 2) act &= T.spl[(k - 1) / 2];
    const int mk = act && !T.spl[nd];
    io.s_mask[nd] = mk;
    io.mask[nd] = mk;
    io.split[nd] = T.spl[nd];
    io.count[nd] = T.node_n[nd];
    io.logvol[nd] = (float)T.lv[nd];
  }
  // ---- second bracket reading: each direction factor times its node's radius
  if (io.bracket == 1) {
    for (int q = tid; q < n_nodes * d * d; q += B) {
      const float rad = sqrtf(__uint_as_float(T.node_m2[q / (d * d)]));
      if (rad > 0.f && isfinite(rad)) {
        io.s_chol[q] *= rad;
        io.chol[q] = io.s_chol[q];
      }
    }
  }
  // ---- each point's accepted leaf --------------------------------------------
  for (int j = tid; j < N; j += B) {
    const int bits = side[j];
    int nd = 0, lev = 0;
    while (lev < D && T.spl[nd]) {
      nd = 2 * nd + 1 + ((bits >> lev) & 1);
      ++lev;
    }
    io.cid[j] = nd;
  }
  __syncthreads();
}

}  // namespace nsd
