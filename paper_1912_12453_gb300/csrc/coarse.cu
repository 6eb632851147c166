// Two-level additive preconditioner for the Krylov solve of Sec. 3.5:
//   z = B^{-1} v + P A_c^{-1} R v
// B: nodal block-Jacobi (vector.cu); P: trilinear interpolation of all fields
// from the nodes of a uniform coarse octree level L_c to the mesh nodes;
// R = P^T; A_c = R J P, the Galerkin projection of the Jacobian.  Nodal
// block-Jacobi alone leaves the smooth pressure modes of the VMS saddle
// point unresolved (they couple across the whole domain); the coarse space
// carries them.
//
// A_c is probed: the image J P e_c of a coarse hat lives within H + h of its
// coarse node c (H, h: coarse and mesh spacing), so the hats of one field
// whose nodes share the residues of their coordinates mod 3 (27 colours in
// 3D, 9 in 2D) are applied together, and each mesh row is credited to the
// nearest coarse node of the probed colour.  Exact when h <= H/2, i.e. every
// leaf at least one level finer than L_c.  All reductions run in a fixed
// order (one block per coarse node); nothing is atomic.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <type_traits>
#include <vector>

#include "chns_internal.h"
#include "coarse.h"
#include "host_util.h"
#include "launch.h"
#include "solver.h"

namespace chns {

namespace {

constexpr int kB = 256;
constexpr unsigned FULL = 0xffffffffu;

inline unsigned grid_n(int64_t n) {
  int64_t b = (n + kB - 1) / kB;
  return (unsigned)std::min<int64_t>(std::max<int64_t>(b, 1), 152 * 8);
}

struct CGeo {
  int dim, nf, nc1;   // nc1 = 2^Lc + 1 coarse nodes per axis
  int64_t n_nodes;
  int64_t ncn_inst;   // coarse nodes per instance
  int64_t nc0;        // coarse unknowns per instance
  int direct;         // the coarse grid is the mesh: unknowns in node order
};

// 16 bytes of T
template <typename T>
struct alignas(16) V16 {
  T a[16 / sizeof(T)];
};

template <typename T>
__device__ __forceinline__ T warp_sum_t(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
  return v;
}

// cell (lowest corner, per axis) and fraction of a position in coarse units
__device__ __forceinline__ void locate(const CGeo &g, const float *pos, int *b, float *t) {
  for (int a = 0; a < g.dim; ++a) {
    int c = (int)floorf(pos[a]);
    c = c < 0 ? 0 : (c > g.nc1 - 2 ? g.nc1 - 2 : c);
    b[a] = c;
    t[a] = pos[a] - float(c);
  }
}

__device__ __forceinline__ int lin(const CGeo &g, const int *c) {
  int idx = 0;
  for (int a = g.dim - 1; a >= 0; --a) idx = idx * g.nc1 + c[a];
  return idx;
}

// probing vectors v0 .. v0 + gridDim.y - 1; number v = k NF + f: field f = sum
// of the coarse hats of colour k; other fields 0
template <typename T, int NF, int DIM>
__global__ void __launch_bounds__(kB) k_probe_coarse(CGeo g, const float *__restrict__ pos, int v0,
                                                     T *__restrict__ w) {
  const int k = (v0 + int(blockIdx.y)) / NF, f = (v0 + int(blockIdx.y)) % NF;
  const int kk[3] = {k % 3, (k / 3) % 3, k / 9};
  w += blockIdx.y * g.n_nodes * NF;
  for (int64_t i = blockIdx.x * int64_t(kB) + threadIdx.x; i < g.n_nodes; i += int64_t(gridDim.x) * kB) {
    int b[3];
    float t[3];
    locate(g, pos + i * g.dim, b, t);
    double s = 0.0;
#pragma unroll
    for (int c = 0; c < (1 << DIM); ++c) {
      double wc = 1.0;
      bool in = true;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        int ca = b[a] + ((c >> a) & 1);
        if (ca % 3 != kk[a]) in = false;
        wc *= ((c >> a) & 1) ? double(t[a]) : 1.0 - double(t[a]);
      }
      if (in) s += wc;
    }
#pragma unroll
    for (int q = 0; q < NF; ++q) w[i * NF + q] = q == f ? T(s) : T(0);
  }
}

// owner coordinates (residue kk mod 3, within two coarse steps of the row
// node cpc) of slot s: bit a set = positive offset along axis a
__device__ __forceinline__ bool slot_owner(const CGeo &g, const int *cpc, const int *kk, int s, int *oc) {
  bool ok = true;
  for (int a = 0; a < g.dim; ++a) {
    oc[a] = -1;
    for (int d = -2; d <= 2; ++d) {
      int o = cpc[a] + d;
      if (o < 0 || o >= g.nc1 || o % 3 != kk[a]) continue;
      if ((d > 0) == (((s >> a) & 1) == 1)) oc[a] = o;
    }
    if (oc[a] < 0) ok = false;
  }
  return ok;
}

constexpr int kPiece = 1024;  // most entries of a restriction list that one block sums
constexpr int kChunk = 64;    // entries whose slots a block finds together

// Block (p, v) takes piece p of the restriction list of coarse row node c' and,
// for probe v (colour k), sums P[i, c'] y[i, q] per owner slot s (the owner of
// mesh node i: the nearest coarse node of colour k): the threads first find the
// slots of kChunk entries together, then thread (s, q) adds up the entries of its
// slot, in T in eight chains of at most eight terms, and the chunks in double:
// 11 roundings of T on the longest way, as many as a tree over the block has.  In
// double two chains of at most 32, since each further chain costs additions on the
// FP64 pipe that binds there, for which entries of other warps' slots are skipped
// too (eight chains: 4.6 ms more of 252 for the build on 29,016 adaptive leaves).
// A block of 256 threads with 48 sums each, reduced over the block, spends its time
// on the reduction: most lists hold 64 to 125 entries.
template <typename T, int NF, int DIM>
__global__ void __launch_bounds__(kChunk) k_gather_coarse(CGeo g, const int32_t *__restrict__ piece_node,
                                                          const int64_t *__restrict__ piece_begin,
                                                          const int32_t *__restrict__ rnode,
                                                          const float *__restrict__ rw, const float *__restrict__ pos,
                                                          int v0, const T *__restrict__ y, double *__restrict__ part) {
  constexpr int NS = 1 << DIM;
  static_assert(NS * NF <= kChunk, "one sum per thread");
  const int cp = piece_node[blockIdx.x], k = (v0 + int(blockIdx.y)) / NF;
  const int kk[3] = {k % 3, (k / 3) % 3, k / 9};
  __shared__ int32_t node[kChunk], slot[kChunk];
  __shared__ T wgt[kChunk];
  y += blockIdx.y * g.n_nodes * NF;
  const int s = threadIdx.x / NF, q = threadIdx.x % NF;
  const int64_t end = piece_begin[blockIdx.x + 1];
  constexpr int G = sizeof(T) == 8 ? 2 : 8;
  const int s0 = (threadIdx.x & ~31) / NF, s1 = (threadIdx.x | 31) / NF;  // slots of the warp
  double acc = 0.0;
  for (int64_t b = piece_begin[blockIdx.x]; b < end; b += kChunk) {
    const int cnt = int(min(int64_t(kChunk), end - b));
    __syncthreads();
    slot[threadIdx.x] = -1;
    if (int(threadIdx.x) < cnt) {
      const int64_t i = rnode[b + threadIdx.x];
      int r = int(cp % g.ncn_inst), sl = 0;
      bool ok = true;
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        const int cpc = r % g.nc1;
        r /= g.nc1;
        const float p = pos[i * DIM + a];
        const int o = kk[a] + 3 * (int)floorf((p - float(kk[a])) / 3.0f + 0.5f);
        if (o < 0 || o >= g.nc1) ok = false;
        if (o > cpc) sl |= 1 << a;
      }
      node[threadIdx.x] = int32_t(i);
      slot[threadIdx.x] = ok ? sl : -1;
      wgt[threadIdx.x] = T(rw[b + threadIdx.x]);
    }
    __syncthreads();
    if (s < NS) {
      T a[G];
#pragma unroll
      for (int g = 0; g < G; ++g) a[g] = T(0);
      for (int e = 0; e < cnt; e += G)
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const int se = slot[e + g];
          const bool mine = sizeof(T) == 8 ? se >= s0 && se <= s1 && se == s : se == s;
          if (mine) a[g] = fma(wgt[e + g], y[int64_t(node[e + g]) * NF + q], a[g]);
        }
#pragma unroll
      for (int h = G / 2; h > 0; h >>= 1)
#pragma unroll
        for (int g = 0; g < h; ++g) a[g] += a[g + h];
      acc += double(a[0]);
    }
  }
  if (s < NS) part[(blockIdx.y * int64_t(gridDim.x) + blockIdx.x) * NS * NF + threadIdx.x] = acc;
}

// A[(c', q), (owner(s), f)] = sum of the pieces, in list order
__global__ void k_gather_sum(CGeo g, int v0, int64_t n_pieces, const int32_t *__restrict__ node_piece,
                             const double *__restrict__ part, double *__restrict__ A, int64_t ldA, int64_t ncn) {
  const int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x;
  const int nf = g.nf, ns = 1 << g.dim, v = v0 + blockIdx.y, k = v / nf, f = v % nf;
  if (t >= ncn * ns * nf) return;
  const int64_t cp = t / (ns * nf);
  const int s = int((t / nf) % ns), q = int(t % nf);
  const int64_t inst = cp / g.ncn_inst, lcp = cp % g.ncn_inst;
  int cpc[3] = {0, 0, 0}, kk[3] = {k % 3, (k / 3) % 3, k / 9}, oc[3];
  {
    int r = int(lcp);
    for (int a = 0; a < g.dim; ++a) { cpc[a] = r % g.nc1; r /= g.nc1; }
  }
  if (!slot_owner(g, cpc, kk, s, oc)) return;
  double sum = 0.0;
  for (int p = node_piece[cp]; p < node_piece[cp + 1]; ++p)
    sum += part[((blockIdx.y * n_pieces + p) * ns + s) * nf + q];
  double *Ai = A + inst * g.nc0 * ldA;
  Ai[(lcp * nf + q) * ldA + int64_t(lin(g, oc)) * nf + f] = sum;
}

// The same for a coarse grid that is the mesh: row (i, q) of A, in the mesh's
// node order, gets y[i, q] in the column of the probed node next to node i
template <typename T, int NF, int DIM>
__global__ void __launch_bounds__(kB) k_collect_direct(CGeo g, const float *__restrict__ pos,
                                                       const int32_t *__restrict__ cinv, int v0,
                                                       const T *__restrict__ y, double *__restrict__ A) {
  const int64_t i = blockIdx.x * int64_t(kB) + threadIdx.x;
  if (i >= g.n_nodes) return;
  const int k = (v0 + int(blockIdx.y)) / NF, f = (v0 + int(blockIdx.y)) % NF;
  const int kk[3] = {k % 3, (k / 3) % 3, k / 9};
  int oc[3];
#pragma unroll
  for (int a = 0; a < DIM; ++a) {
    const int c = int(pos[i * DIM + a]);
    int d = (kk[a] - c % 3 + 3) % 3;  // 0, 1 or 2 = -1
    oc[a] = c + (d == 2 ? -1 : d);
    if (oc[a] < 0 || oc[a] >= g.nc1) return;
  }
  const int64_t inst = i / g.ncn_inst, li = i % g.ncn_inst, lo = cinv[inst * g.ncn_inst + lin(g, oc)] % g.ncn_inst;
  const T *yi = y + (blockIdx.y * g.n_nodes + i) * NF;
  double *Ai = A + inst * g.nc0 * g.nc0 + lo * NF + f;
#pragma unroll
  for (int q = 0; q < NF; ++q) Ai[(li * NF + q) * g.nc0] = double(yi[q]);
}

constexpr int kGroups = 32;   // lists are read by 32 groups of eight lanes

// rc = R v = P^T v: block p sums w v[i, q] over piece p of a coarse node's
// restriction list, lane q of each group of eight the component q: four chains of
// at most eight terms a group, then a tree over the chains and the groups (15
// roundings on the longest way; in double two chains, fewer additions, 22).  part == rc when every list is one piece.  The
// weights are exact (W), so in double R is P^T: a product of the three fractions of
// a node k levels below the coarse grid has up to 3 k bits, more than a float from
// k = 9 on (2D: 13).
// (Sums of all corners of a coarse cell, reduced over 256 threads, took a hundred
// FP64 additions a warp for lists of 49 to 81 nodes.)
template <typename T, int NF, typename W>
__global__ void __launch_bounds__(kGroups * 8) k_restrict_lists(const int64_t *__restrict__ piece_begin,
                                                               const int32_t *__restrict__ rnode,
                                                               const W *__restrict__ rw,
                                                               const T *__restrict__ v, T *__restrict__ part) {
  const int grp = threadIdx.x >> 3, q = threadIdx.x & 7;
  const int64_t b = piece_begin[blockIdx.x];
  const int cnt = int(piece_begin[blockIdx.x + 1] - b);
  int32_t i0 = 0;
  T w0 = T(0);
  if (grp < cnt) {
    i0 = rnode[b + grp];
    w0 = T(rw[b + grp]);
  }
  wait_previous(v, part);
  constexpr int K = sizeof(T) == 8 ? 2 : 4;
  T a[K];
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = T(0);
  if (q < NF && grp < cnt) {
    a[0] = w0 * v[int64_t(i0) * NF + q];
    constexpr int G = 8;  // independent loads, then the products
    for (int e = grp + kGroups; e < cnt; e += G * kGroups) {
      int32_t i[G];
      T w[G], x[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const bool on = e + g * kGroups < cnt;
        i[g] = on ? rnode[b + e + g * kGroups] : -1;
        w[g] = on ? T(rw[b + e + g * kGroups]) : T(0);
      }
#pragma unroll
      for (int g = 0; g < G; ++g) x[g] = i[g] >= 0 ? v[int64_t(i[g]) * NF + q] : T(0);
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (i[g] >= 0) a[g % K] = fma(w[g], x[g], a[g % K]);
    }
  }
#pragma unroll
  for (int h = K / 2; h > 0; h >>= 1)
#pragma unroll
    for (int k = 0; k < h; ++k) a[k] += a[k + h];
  __shared__ T red[kGroups][8];
  red[grp][q] = a[0];
  __syncthreads();
  if (threadIdx.x < 32) {  // a quarter of the groups a lane, then the quarters
    constexpr int G = kGroups / 4;
    T t[G];
#pragma unroll
    for (int g = 0; g < G; ++g) t[g] = red[4 * g + grp][q];
#pragma unroll
    for (int h = G / 2; h > 0; h >>= 1)
#pragma unroll
      for (int g = 0; g < h; ++g) t[g] += t[g + h];
    t[0] += __shfl_xor_sync(FULL, t[0], 8);
    t[0] += __shfl_xor_sync(FULL, t[0], 16);
    if (threadIdx.x < NF) part[int64_t(blockIdx.x) * NF + threadIdx.x] = t[0];
  }
}

// rc = sum of the pieces, every eighth in one chain (double: every second)
template <typename T>
__global__ void k_restrict_pieces(int64_t nc, int nf, const int32_t *__restrict__ node_piece,
                                  const T *__restrict__ part, T *__restrict__ rc) {
  const int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x;
  wait_previous(part, rc);
  if (t >= nc) return;
  const int64_t cp = t / nf;
  constexpr int G = sizeof(T) == 8 ? 2 : 8;
  T s[G];
#pragma unroll
  for (int g = 0; g < G; ++g) s[g] = T(0);
  const int e = node_piece[cp + 1];
#pragma unroll 4
  for (int p = node_piece[cp]; p < e; p += G)
#pragma unroll
    for (int g = 0; g < G; ++g)
      if (p + g < e) s[g] += part[int64_t(p + g) * nf + t % nf];
#pragma unroll
  for (int h = G / 2; h > 0; h >>= 1)
#pragma unroll
    for (int g = 0; g < h; ++g) s[g] += s[g + h];
  rc[t] = s[0];
}

// zc = A_c^{-1} rc, one warp per row, in precision T; row r of instance i at
// Minv + i * inst_stride + (r % nc0) * ld
template <typename T>
__global__ void k_coarse_matvec(const T *__restrict__ Minv, int64_t ld, int64_t inst_stride, int64_t nc,
                                int64_t nc0, const T *__restrict__ rc, T *__restrict__ zc) {
  const int64_t r0 = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int ln = threadIdx.x & 31;
  const int64_t r = r0 < nc ? r0 : nc - 1;
  const int64_t inst = r / nc0, lr = r % nc0;
  const T *row = Minv + inst * inst_stride + lr * ld;
  // the first 24 values of the lane's share of the row (all of it for the
  // bottom levels) before the vector is there
  constexpr int G = 24;
  T a[G];
#pragma unroll
  for (int g = 0; g < G; ++g) a[g] = ln + 32 * g < nc0 ? row[ln + 32 * g] : T(0);
  wait_previous(rc, zc);
  if (r0 != r) return;
  const T *x = rc + inst * nc0;
  T s[4] = {T(0), T(0), T(0), T(0)};  // four chains
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (ln + 32 * g < nc0) s[g & 3] = fma(a[g], x[ln + 32 * g], s[g & 3]);
  int64_t c = ln + 32 * G;
  for (; c + 96 < nc0; c += 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = fma(row[c + 32 * k], x[c + 32 * k], s[k]);
  }
  for (; c < nc0; c += 32) s[0] = fma(row[c], x[c], s[0]);
  const T t = warp_sum_t((s[0] + s[1]) + (s[2] + s[3]));
  if (ln == 0) zc[r] = t;
}

// z = Binv v + P zc  (nodal block-Jacobi plus the prolonged coarse
// correction; zc == nullptr: block-Jacobi only; Binv == nullptr: the coarse
// correction only).  Eight lanes per node, lane q the component q.
template <typename T, int NF, int DIM>
__global__ void __launch_bounds__(kB) k_block_prolong(CGeo g, const float *__restrict__ pos,
                                                      const int32_t *__restrict__ node_inst,
                                                      const T *__restrict__ Binv, const T *__restrict__ v,
                                                      const T *__restrict__ zc, T *__restrict__ z) {
  const int64_t i0 = (blockIdx.x * int64_t(kB) + threadIdx.x) >> 3;
  const int q = threadIdx.x & 7;
  const bool on = i0 < g.n_nodes && q < NF;
  const int64_t i = on ? i0 : 0, at = i * NF + (on ? q : 0);
  T row[NF];
  if (Binv)
#pragma unroll
    for (int c = 0; c < NF; ++c) row[c] = Binv[at * NF + c];
  int64_t idx0 = 0, step[3] = {1, 0, 0};
  T t[DIM];
  if (zc && !g.direct) {
    int b[3];
    float tf[3];
    locate(g, pos + i * DIM, b, tf);
    idx0 = node_inst ? int64_t(node_inst[i]) * g.ncn_inst : 0;
    step[1] = g.nc1;
    step[2] = int64_t(g.nc1) * g.nc1;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      idx0 += b[a] * step[a];
      t[a] = T(tf[a]);
    }
  }
  wait_previous(v, zc, z);
  T s = T(0);
  if (zc && g.direct) {
    s = zc[at];
  } else if (zc) {
    T x[1 << DIM];
#pragma unroll
    for (int c = 0; c < (1 << DIM); ++c) {
      int64_t idx = idx0;
#pragma unroll
      for (int a = 0; a < DIM; ++a) idx += ((c >> a) & 1) ? step[a] : 0;
      x[c] = zc[idx * NF + (on ? q : 0)];
    }
#pragma unroll
    for (int c = 0; c < (1 << DIM); ++c) {
      T wc = T(1);
#pragma unroll
      for (int a = 0; a < DIM; ++a) wc *= ((c >> a) & 1) ? t[a] : T(1) - t[a];
      s = fma(wc, x[c], s);
    }
  }
  if (Binv) {
    const T r = v[at];
#pragma unroll
    for (int c = 0; c < NF; ++c) s = fma(row[c], __shfl_sync(FULL, r, c, 8), s);
  }
  if (on) z[at] = s;
}

// A -> B elementwise with a type change (n values)
template <typename A, typename B>
__global__ void k_copy_cast(const A *__restrict__ x, int64_t n, B *__restrict__ y) {
  for (int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x; t < n; t += int64_t(gridDim.x) * kB) y[t] = B(x[t]);
}

// Gauss-Jordan inversion of each instance's n x n block (row-major) with
// partial pivoting, NB columns at a time.  One pivot step swaps the row of the
// largest |a_rk|, r >= k, into row k, scales it by d = 1/a_kk, puts d on the
// diagonal and eliminates column k from the other rows, whose column k becomes
// -a_rk d.  NB steps change the other columns by one matrix product:
//   A' = [r not in panel] S A + G (S A)[panel rows],
// S the row interchanges of the panel, G (n x NB, stored column by column) what
// the steps leave in the panel's own columns.  So k_gj_panel runs the NB steps on the panel alone, in
// the registers of one block (a row per thread, two barriers a step), and
// k_gj_update applies (S, G) to the whole matrix, from one buffer into the
// other (in place, a row could be overwritten before another one reads it).
// The row each line came from is carried along; the inverse's columns are put
// back by it at the end (A^-1 = G_all S_all).
//
// Bound: the chain of n pivot searches and two barriers each in one block,
// about 0.85 us a column in float (n = 750: 177 instructions a warp and column,
// the schedulers 54 % busy), more in double (the panel's products run on one
// SM's FP64 pipe).  A panel is read in pieces of 32 bytes of a row and G is
// stored column by column: with each thread reading and writing its own row a
// word at a time an access touched 32 lines, and a panel of 32 columns of 750
// rows took 41.6 instead of 31.2 us (8 columns of 405 rows in double: 16.5, 16.0).
// A launch pair per column (pivot, rank-1 elimination of all rows) cost 12 to
// 24 us per column, 9 to 18 ms for n = 405 and 750.
// (abs_key: |x| as an integer of the same order, NaN below everything; the
// search then needs no FP64 comparisons, which run on the narrow FP64 pipe)
__device__ __forceinline__ uint64_t abs_key(float x) {
  const uint32_t b = __float_as_uint(x) & 0x7fffffffu;
  return b > 0x7f800000u ? 0 : b;
}
__device__ __forceinline__ uint64_t abs_key(double x) {
  const uint64_t b = uint64_t(__double_as_longlong(x)) & 0x7fffffffffffffffull;
  return b > 0x7ff0000000000000ull ? 0 : b;
}
// the largest key of the warp and the lowest row that has it, by the warp's
// integer reductions
template <typename T>
__device__ __forceinline__ void warp_arg_max(uint64_t &best, int &arg) {
  bool at = true;
  if (sizeof(T) == 8) {
    const uint32_t h = __reduce_max_sync(FULL, uint32_t(best >> 32));
    at = uint32_t(best >> 32) == h;
    const uint32_t l = __reduce_max_sync(FULL, at ? uint32_t(best) : 0u);
    at = at && uint32_t(best) == l;
    best = (uint64_t(h) << 32) | l;
  } else {
    const uint32_t l = __reduce_max_sync(FULL, uint32_t(best));
    at = uint32_t(best) == l;
    best = l;
  }
  arg = int(__reduce_min_sync(FULL, at ? uint32_t(arg) : 0xffffffffu));
}

template <typename T, int NB, int R>
__global__ void __launch_bounds__(1024) k_gj_panel(const T *__restrict__ Mall, int n, int k0,
                                                   T *__restrict__ Gall, int32_t *__restrict__ permall,
                                                   const int32_t *__restrict__ origin_in,
                                                   int32_t *__restrict__ origin_out, int *__restrict__ bad) {
  const T *M = Mall + int64_t(blockIdx.x) * n * n;
  T *G = Gall + int64_t(blockIdx.x) * n * NB;
  const int nb = min(NB, n - k0);
  const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31, nw = blockDim.x >> 5;
  constexpr int L = 16 / sizeof(T);
  using Row = V16<T>;
  __shared__ uint64_t wv[2][32];
  __shared__ int wr[2][32];
  __shared__ Row prow[2][NB / L], krow[2][NB / L];
  __shared__ T dinv[2];
  __shared__ int psrc[2], ksrc[2];
  // A row's NB values go to one thread by way of shared memory, C columns at a
  // time: a warp reads 32 / C rows at once
  constexpr int C = 32 / sizeof(T);
  __shared__ T tile[32][32][C + 1];
  T a[R][NB];
  int src[R];
  wait_previous(M, G, permall, origin_in, origin_out, bad);
#pragma unroll
  for (int i = 0; i < R; ++i) {
    src[i] = threadIdx.x + i * blockDim.x;
    const int w0 = src[i] - ln;
#pragma unroll
    for (int c = 0; c < NB; c += C) {
      T v[C];
#pragma unroll
      for (int j = 0; j < C; ++j) {
        const int r = w0 + ln / C + j * (32 / C), q = c + ln % C;
        v[j] = r < n && q < nb ? M[int64_t(r) * n + k0 + q] : T(0);
      }
      __syncwarp();
#pragma unroll
      for (int j = 0; j < C; ++j) tile[wid][ln / C + j * (32 / C)][ln % C] = v[j];
      __syncwarp();
#pragma unroll
      for (int j = 0; j < C; ++j) a[i][c + j] = tile[wid][ln][j];
    }
  }
  // the warp's row of the largest |a_rk|, r >= k, the lowest of equals
  uint64_t best = 0;
  int arg = k0;
  auto candidate = [&](int i, int k, T x) {
    const int r = threadIdx.x + i * blockDim.x;
    const uint64_t v = abs_key(x);
    if (r >= k && r < n && (v > best || (v == best && r < arg))) { best = v; arg = r; }
  };
#pragma unroll
  for (int i = 0; i < R; ++i) candidate(i, k0, a[i][0]);
  warp_arg_max<T>(best, arg);
  // The loop stays rolled (unrolled it is 80 KB of code that runs once): the
  // current column is always a[.][0], each step writes its results one place
  // down and the finished column to the end.
#pragma unroll 1
  for (int kk = 0; kk < nb; ++kk) {
    const int k = k0 + kk, sl = kk & 1;
    if (ln == 0) { wv[sl][wid] = best; wr[sl][wid] = arg; }
    __syncthreads();
    best = ln < nw ? wv[sl][ln] : 0;
    arg = ln < nw ? wr[sl][ln] : n;
    warp_arg_max<T>(best, arg);
    const int p = arg;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = threadIdx.x + i * blockDim.x;
      if (r == p) {
#pragma unroll
        for (int c = 0; c < NB; c += L) {
          Row v;
#pragma unroll
          for (int j = 0; j < L; ++j) v.a[j] = a[i][c + j];
          prow[sl][c / L] = v;
        }
        psrc[sl] = src[i];
        const bool ok = fabs(a[i][0]) > T(0);  // false for NaN too
        if (!ok) *bad = 1;
        dinv[sl] = ok ? T(1) / a[i][0] : T(0);
      }
      if (r == k) {
#pragma unroll
        for (int c = 0; c < NB; c += L) {
          Row v;
#pragma unroll
          for (int j = 0; j < L; ++j) v.a[j] = a[i][c + j];
          krow[sl][c / L] = v;
        }
        ksrc[sl] = src[i];
      }
    }
    __syncthreads();
    const T d = dinv[sl];
    T fr[R];
    best = 0;
    arg = k + 1;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = threadIdx.x + i * blockDim.x;
      if (r == p && p != k) {
#pragma unroll
        for (int c = 0; c < NB; c += L) {
          const Row v = krow[sl][c / L];
#pragma unroll
          for (int j = 0; j < L; ++j) a[i][c + j] = v.a[j];
        }
        src[i] = ksrc[sl];
      }
      // row k: prow d; the others: a - (a_k d) prow
      fr[i] = -a[i][0] * d;
      if (r == k) {
        src[i] = psrc[sl];
        fr[i] = d;
#pragma unroll
        for (int c = 1; c < NB; ++c) a[i][c] = T(0);
      }
      // the next column first: its pivot search overlaps the other products
      a[i][0] = fma(fr[i], prow[sl][0].a[1], a[i][1]);
      candidate(i, k + 1, a[i][0]);
    }
    warp_arg_max<T>(best, arg);
#pragma unroll
    for (int c = 0; c < NB; c += L) {
      const Row v = prow[sl][c / L];
#pragma unroll
      for (int j = 0; j < L; ++j)
        if (c + j > 1)
#pragma unroll
          for (int i = 0; i < R; ++i) a[i][c + j - 1] = fma(fr[i], v.a[j], a[i][c + j]);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) a[i][NB - 1] = fr[i];
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = threadIdx.x + i * blockDim.x;
    if (r >= n) continue;
    // a narrow last panel: its nb columns have moved to the end
#pragma unroll
    for (int c = 0; c < NB; ++c)
      if (c >= NB - nb) G[int64_t(c - (NB - nb)) * n + r] = a[i][c];  // column by column
    const int64_t o = int64_t(blockIdx.x) * n;
    permall[o + r] = src[i];
    origin_out[o + r] = origin_in[o + src[i]];
  }
}

// out = [r not in panel] S in + G (S in)[panel rows]; the panel's own columns
// become G.  A block of 256 threads computes a TS x TS tile (TS / 16 squared
// values per thread); blockIdx.z: instance.
template <typename T, int NB, int TS>
__global__ void __launch_bounds__(256) k_gj_update(const T *__restrict__ inall, T *__restrict__ outall, int n, int k0,
                                                   const T *__restrict__ Gall, const int32_t *__restrict__ permall) {
  constexpr int V = TS / 16;
  const T *in = inall + int64_t(blockIdx.z) * n * n;
  T *out = outall + int64_t(blockIdx.z) * n * n;
  const T *G = Gall + int64_t(blockIdx.z) * n * NB;
  const int32_t *perm = permall + int64_t(blockIdx.z) * n;
  const int nb = min(NB, n - k0);
  const int r0 = blockIdx.y * TS, j0 = blockIdx.x * TS;
  __shared__ T g[TS][NB + 1], u[NB][TS];
  wait_previous(in, out, G, perm);
  for (int t = threadIdx.x; t < TS * NB; t += 256) {
    const int r = t % TS, c = t / TS;
    g[r][c] = r0 + r < n && c < nb ? G[int64_t(c) * n + r0 + r] : T(0);
  }
  for (int t = threadIdx.x; t < NB * TS; t += 256) {
    const int c = t / TS, j = t % TS;
    u[c][j] = c < nb && j0 + j < n ? in[int64_t(perm[k0 + c]) * n + j0 + j] : T(0);
  }
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  T acc[V][V];
#pragma unroll
  for (int y = 0; y < V; ++y) {
    const int r = r0 + ty + 16 * y;
    const bool row = r < n && (r < k0 || r >= k0 + nb);
    const int64_t b = row ? int64_t(perm[r]) * n : 0;
#pragma unroll
    for (int x = 0; x < V; ++x) {
      const int j = j0 + tx + 16 * x;
      acc[y][x] = row && j < n ? in[b + j] : T(0);
    }
  }
  __syncthreads();
#pragma unroll 8
  for (int c = 0; c < NB; ++c) {
    T gr[V], uc[V];
#pragma unroll
    for (int y = 0; y < V; ++y) gr[y] = g[ty + 16 * y][c];
#pragma unroll
    for (int x = 0; x < V; ++x) uc[x] = u[c][tx + 16 * x];
#pragma unroll
    for (int y = 0; y < V; ++y)
#pragma unroll
      for (int x = 0; x < V; ++x) acc[y][x] = fma(gr[y], uc[x], acc[y][x]);
  }
#pragma unroll
  for (int y = 0; y < V; ++y) {
    const int r = r0 + ty + 16 * y;
    if (r >= n) continue;
#pragma unroll
    for (int x = 0; x < V; ++x) {
      const int j = j0 + tx + 16 * x;
      if (j >= n) continue;
      out[int64_t(r) * n + j] = j >= k0 && j < k0 + nb ? g[ty + 16 * y][j - k0] : acc[y][x];
    }
  }
}

__global__ void k_gj_init(int32_t *__restrict__ origin, int64_t n, int n_inst) {
  for (int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x; t < n * n_inst; t += int64_t(gridDim.x) * kB)
    origin[t] = int32_t(t % n);
}

// the inverse's columns: column origin[j] is column j of the eliminated matrix
template <typename T, typename D1, typename D2>
__global__ void k_gj_columns(const T *__restrict__ in, int64_t n, int64_t total, const int32_t *__restrict__ origin,
                             D1 *__restrict__ a, D2 *__restrict__ b) {
  for (int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x; t < total; t += int64_t(gridDim.x) * kB) {
    const int64_t row = t / n, inst = row / n;
    const int64_t q = row * n + origin[inst * n + t % n];
    a[q] = D1(in[t]);
    b[q] = D2(in[t]);
  }
}

// The column-by-column form for matrices beyond the panel kernel's rows (n >
// 5120: a coarse level of 4 in 3D, 5 in 2D): two launches per column, in place.
// Pivot step k: the row interchange is recorded in piv and undone as a column
// interchange at the end.
template <typename T>
__global__ void k_gj_pivot(T *__restrict__ Mall, int64_t n, int64_t k, T *__restrict__ colall,
                           int32_t *__restrict__ pivall, int *__restrict__ bad) {
  T *M = Mall + int64_t(blockIdx.x) * n * n;
  T *col = colall + int64_t(blockIdx.x) * n;
  __shared__ T bv[1024];
  __shared__ int64_t bi[1024];
  __shared__ T pv;
  T best = T(-1);
  int64_t arg = k;
  for (int64_t r = k + threadIdx.x; r < n; r += blockDim.x) {
    const T v = fabs(M[r * n + k]);
    if (v > best) { best = v; arg = r; }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = arg;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      if (bv[threadIdx.x + s] > bv[threadIdx.x] ||
          (bv[threadIdx.x + s] == bv[threadIdx.x] && bi[threadIdx.x + s] < bi[threadIdx.x])) {
        bv[threadIdx.x] = bv[threadIdx.x + s];
        bi[threadIdx.x] = bi[threadIdx.x + s];
      }
    }
    __syncthreads();
  }
  const int64_t p = bi[0];
  if (threadIdx.x == 0) {
    pv = M[p * n + k];
    pivall[int64_t(blockIdx.x) * n + k] = int32_t(p);
  }
  __syncthreads();
  if (!(fabs(pv) > T(0))) {
    if (threadIdx.x == 0) *bad = 1;
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x) col[r] = T(0);
    return;
  }
  const T d = T(1) / pv;
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const T a = M[k * n + j], b = M[p * n + j];
    if (p != k) M[p * n + j] = a;
    M[k * n + j] = j == k ? d : b * d;
  }
  __syncthreads();
  for (int64_t r = threadIdx.x; r < n; r += blockDim.x) col[r] = r == k ? T(0) : M[r * n + k];
}

// elimination of column k: thread = one column j (coalesced along rows of
// the row-major block), block y = a range of kRowsGJ rows, z = instance
constexpr int kRowsGJ = 32;
template <typename T>
__global__ void __launch_bounds__(kB) k_gj_elim(T *__restrict__ Mall, int64_t n, int64_t k,
                                                const T *__restrict__ colall) {
  T *M = Mall + int64_t(blockIdx.z) * n * n;
  const T *col = colall + int64_t(blockIdx.z) * n;
  const int64_t j = blockIdx.x * int64_t(kB) + threadIdx.x;
  if (j >= n) return;
  const T d = M[k * n + k];
  const T rk = M[k * n + j];
  const int64_t r0 = int64_t(blockIdx.y) * kRowsGJ, r1 = r0 + kRowsGJ < n ? r0 + kRowsGJ : n;
  for (int64_t r = r0; r < r1; ++r) {
    if (r == k) continue;
    const T fr = col[r];
    T *a = M + r * n + j;
    if (j == k) *a = -fr * d;
    else if (fr != T(0)) *a = fma(-fr, rk, *a);
  }
}

// undo the row interchanges as column interchanges, last first (a thread per row)
template <typename T>
__global__ void k_gj_unswap(T *__restrict__ Mall, int64_t n, const int32_t *__restrict__ pivall, int n_inst) {
  for (int64_t t = blockIdx.x * int64_t(kB) + threadIdx.x; t < n * n_inst; t += int64_t(gridDim.x) * kB) {
    const int64_t inst = t / n, r = t % n;
    T *row = Mall + inst * n * n + r * n;
    const int32_t *piv = pivall + inst * n;
    for (int64_t k = n - 1; k >= 0; --k) {
      const int64_t p = piv[k];
      if (p != k) {
        const T x = row[k];
        row[k] = row[p];
        row[p] = x;
      }
    }
  }
}

constexpr int64_t kPanelRows = 5120;  // rows the panel kernel holds in registers

template <typename T>
void gauss_jordan_columns(T *M, int64_t n, int n_inst, T *col, int32_t *piv, int *bad, cudaStream_t st) {
  const dim3 ge((unsigned)((n + kB - 1) / kB), (unsigned)((n + kRowsGJ - 1) / kRowsGJ), (unsigned)n_inst);
  for (int64_t k = 0; k < n; ++k) {
    k_gj_pivot<T><<<n_inst, 1024, 0, st>>>(M, n, k, col, piv, bad);
    k_gj_elim<T><<<ge, kB, 0, st>>>(M, n, k, col);
  }
  k_gj_unswap<T><<<grid_n(n * n_inst), kB, 0, st>>>(M, n, piv, n_inst);
  note_launches(int(2 * n + 1));
}

// panels of A (buf0), ping-pong with buf1; returns the buffer that holds the
// eliminated matrix; idx: 3 n n_inst indices, the last n n_inst (or the middle
// ones: *origin) say which column of the inverse each column is
template <typename T, int NB, int R>
T *gj_panels(T *buf0, T *buf1, int64_t n, int n_inst, T *G, int32_t *idx, int32_t **origin, int *bad,
             cudaStream_t st) {
  constexpr int TS = sizeof(T) == 8 ? 32 : 64;
  const int threads = int(((n + R - 1) / R + 31) / 32 * 32);
  const unsigned tiles = (unsigned)((n + TS - 1) / TS);
  int32_t *perm = idx, *o0 = idx + n * n_inst, *o1 = idx + 2 * n * n_inst;
  k_gj_init<<<grid_n(n * n_inst), kB, 0, st>>>(o0, n, n_inst);
  for (int64_t k = 0; k < n; k += NB) {
    launch_next(k_gj_panel<T, NB, R>, (unsigned)n_inst, threads, st, buf0, int(n), int(k), G, perm, o0, o1, bad);
    launch_next(k_gj_update<T, NB, TS>, dim3(tiles, tiles, (unsigned)n_inst), 256, st, buf0, buf1, int(n), int(k), G,
                perm);
    std::swap(buf0, buf1);
    std::swap(o0, o1);
    note_launches(2);
  }
  note_launches(1);
  *origin = o0;
  return buf0;
}

// Panel widths: a row's NB values per thread and R rows per thread have to
// stay in the 64 registers of a 1024-thread block; a wider panel means fewer
// passes over the matrix, so the widest that fits.
template <typename T>
T *gauss_jordan_panels(T *buf0, T *buf1, int64_t n, int n_inst, T *G, int32_t *idx, int32_t **origin, int *bad,
                       cudaStream_t st) {
  constexpr bool F = sizeof(T) == 4;
  if (n <= 1024) return gj_panels<T, F ? 32 : 8, 1>(buf0, buf1, n, n_inst, G, idx, origin, bad, st);
  if (n <= 2048) return gj_panels<T, F ? 16 : 8, 2>(buf0, buf1, n, n_inst, G, idx, origin, bad, st);
  return gj_panels<T, F ? 8 : 4, 5>(buf0, buf1, n, n_inst, G, idx, origin, bad, st);
}
constexpr int kPanelMax = 32;  // widest panel
// Working matrices of the inverse are kept for the next build up to this size
// (all instances; one matrix of 2,800 rows in double), beyond it an allocation is a
// small part of the build and they would be the larger part of the coarse space
constexpr size_t kKeepGj = size_t(128) << 20;

}  // namespace

// ---------------------------------------------------------------- host side
Coarse::~Coarse() { release(); }

void Coarse::release() {
  cudaFree(pos);
  cudaFree(rnode);
  cudaFree(rw);
  cudaFree(rw64);
  cudaFree(piece_node);
  cudaFree(piece_begin);
  cudaFree(node_piece);
  pos = nullptr;
  rnode = nullptr;
  rw = nullptr;
  rw64 = nullptr;
  piece_node = node_piece = nullptr;
  piece_begin = nullptr;
  n_pieces = 0;
  M.release();
  Minv32.release();
  piv.release();
  gj.release();
  cpart.release();
  cudaFree(cinv);
  cinv = nullptr;
  direct = false;
  vec.release();
  rpart.release();
  level = -1;
  ready = false;
}

chns_status coarse_setup(chns_mesh *m, int Lc) {
  Coarse &C = m->coarse;
  if (C.level == Lc && C.pos) return CHNS_OK;
  C.release();
  // a uniform mesh may be its own coarse grid (P = I, A_c = J: an exact solve)
  const int lc_max = m->uniform ? m->min_level : m->min_level - 1;
  if (Lc < 1 || Lc > lc_max) {
    set_error("coarse level %d must be in [1, %d] (below the coarsest leaf level, or equal on a uniform mesh)",
              Lc, lc_max);
    return CHNS_ERR_ARG;
  }
  const int dim = m->dim, nf = m->nf, ni = m->n_inst;
  const int nc1 = (1 << Lc) + 1;
  int64_t ncn = 1;
  for (int a = 0; a < dim; ++a) ncn *= nc1;
  std::vector<float> pos(size_t(m->n_nodes) * dim);
  std::vector<int> base(size_t(m->n_nodes) * dim);
  std::vector<int64_t> cbase(m->n_nodes);  // first coarse node of the node's instance
  for (int q = 0; q < ni; ++q) {
    const double scale = std::ldexp(1.0, Lc - m->inst_max_level[q]);
    for (int64_t i = m->inst_node_start[q]; i < m->inst_node_start[q + 1]; ++i) {
      cbase[i] = int64_t(q) * ncn;
      for (int a = 0; a < dim; ++a) {
        double p = double(m->node_xyz[i * dim + a]) * scale;
        pos[i * dim + a] = float(p);
        int b = (int)std::floor(p);
        base[i * dim + a] = std::min(std::max(b, 0), nc1 - 2);
      }
    }
  }
  auto corners = [&](int64_t i, auto &&fn) {
    for (int c = 0; c < (1 << dim); ++c) {
      double w = 1.0;
      int64_t idx = 0;
      for (int a = dim - 1; a >= 0; --a) {
        int ca = base[i * dim + a] + ((c >> a) & 1);
        double t = double(pos[i * dim + a]) - base[i * dim + a];
        w *= ((c >> a) & 1) ? t : 1.0 - t;
        idx = idx * nc1 + ca;
      }
      if (w != 0.0) fn(cbase[i] + idx, w);
    }
  };
  const int64_t ncn_all = ncn * ni;
  std::vector<int64_t> cnt(ncn_all + 1, 0);
  for (int64_t i = 0; i < m->n_nodes; ++i) corners(i, [&](int64_t idx, double) { cnt[idx + 1]++; });
  for (int64_t c = 0; c < ncn_all; ++c) cnt[c + 1] += cnt[c];
  C.direct = m->uniform && Lc == m->min_level;
  if (C.direct) {
    // node i <-> coarse node (the corners of a node on the coarse grid: itself)
    std::vector<int32_t> cinv(ncn_all);
    for (int64_t i = 0; i < m->n_nodes; ++i) corners(i, [&](int64_t idx, double) { cinv[idx] = (int32_t)i; });
    CHNS_CUDA_TRY(cudaMalloc(&C.cinv, sizeof(int32_t) * cinv.size()));
    CHNS_CUDA_TRY(cudaMemcpy(C.cinv, cinv.data(), sizeof(int32_t) * cinv.size(), cudaMemcpyHostToDevice));
  }
  std::vector<int32_t> rnode(cnt[ncn_all]);
  std::vector<float> rw(cnt[ncn_all]);
  std::vector<double> rw64(cnt[ncn_all]);
  bool floats = true;
  std::vector<int64_t> fill(cnt.begin(), cnt.end() - 1);
  for (int64_t i = 0; i < m->n_nodes; ++i)
    corners(i, [&](int64_t idx, double w) {
      rnode[fill[idx]] = (int32_t)i;
      floats = floats && double(float(w)) == w;
      rw64[fill[idx]] = w;
      rw[fill[idx]++] = (float)w;
    });
  if (!floats) TRY_CHNS(upload(&C.rw64, rw64));
  CHNS_CUDA_TRY(cudaMalloc(&C.pos, sizeof(float) * pos.size()));
  CHNS_CUDA_TRY(cudaMemcpy(C.pos, pos.data(), sizeof(float) * pos.size(), cudaMemcpyHostToDevice));
  CHNS_CUDA_TRY(cudaMalloc(&C.rnode, sizeof(int32_t) * std::max<size_t>(rnode.size(), 1)));
  CHNS_CUDA_TRY(cudaMemcpy(C.rnode, rnode.data(), sizeof(int32_t) * rnode.size(), cudaMemcpyHostToDevice));
  CHNS_CUDA_TRY(cudaMalloc(&C.rw, sizeof(float) * std::max<size_t>(rw.size(), 1)));
  CHNS_CUDA_TRY(cudaMemcpy(C.rw, rw.data(), sizeof(float) * rw.size(), cudaMemcpyHostToDevice));
  // the lists cut into pieces of at most kPiece entries (an empty list: one)
  std::vector<int32_t> piece_node, node_piece(ncn_all + 1, 0);
  std::vector<int64_t> piece_begin;
  for (int64_t c = 0; c < ncn_all; ++c) {
    node_piece[c] = (int32_t)piece_node.size();
    int64_t p = cnt[c];
    do {
      piece_node.push_back((int32_t)c);
      piece_begin.push_back(p);
      p += kPiece;
    } while (p < cnt[c + 1]);
  }
  const int64_t np = (int64_t)piece_node.size();
  node_piece[ncn_all] = (int32_t)np;
  piece_begin.push_back(cnt[ncn_all]);
  TRY_CHNS(upload(&C.piece_node, piece_node));
  TRY_CHNS(upload(&C.piece_begin, piece_begin));
  TRY_CHNS(upload(&C.node_piece, node_piece));
  C.n_pieces = np;
  static std::atomic<int64_t> setups{0};
  C.serial = ++setups;
  C.level = Lc;
  C.nc1 = nc1;
  C.n_inst = ni;
  C.ncn_inst = ncn;
  C.nc0 = ncn * nf;
  C.ncn = ncn_all;
  C.nc = ncn_all * nf;
  TRY_CHNS(C.M.ensure(sizeof(double) * C.nc0 * C.nc0 * ni));
  TRY_CHNS(C.piv.ensure(sizeof(int32_t) * 3 * C.nc0 * ni));
  TRY_CHNS(C.Minv32.ensure(sizeof(float) * C.nc0 * C.nc0 * ni));
  TRY_CHNS(C.vec.ensure(sizeof(double) * (3 * C.nc + 8)));
  TRY_CHNS(C.rpart.ensure(sizeof(double) * np * nf));
  return uploads_done(C.node_piece, ncn_all + 1);
}

template <typename T>
chns_status coarse_build(chns_mesh *m, JvFn<T> jv, void *ctx, cudaStream_t st) {
  Coarse &C = m->coarse;
  Workspace &ws = m->ws;
  const int nf = m->nf, dim = m->dim;
  CGeo g{dim, nf, C.nc1, m->n_nodes, C.ncn_inst, C.nc0, C.direct ? 1 : 0};
  double *M = C.M.as<double>();
  const int64_t nc0 = C.nc0, nn = nc0 * nc0 * C.n_inst, n = m->n_nodes * nf;
  CHNS_CUDA_TRY(cudaMemsetAsync(M, 0, sizeof(double) * nn, st));
  // the probes (9 colours in 2D, 27 in 3D, times the fields) go through J.w in
  // batches: 45 or 162 times five launches otherwise, most of them too small to
  // fill the GPU (9 of 18 ms of an FP64 CN step of the 2D droplet, 10 of 22 of a
  // multigrid step of the level-5 3D droplet, with the probes of the nodal blocks)
  const int total = (dim == 2 ? 9 : 27) * nf;
  const size_t piece = C.direct ? 0 : sizeof(double) * size_t(C.n_pieces) * (size_t(1) << dim) * nf;
  const int batch = probe_batch(m, sizeof(T), piece, total);
  TRY_CHNS(ws.wv.ensure(sizeof(T) * n * batch));
  TRY_CHNS(ws.yv.ensure(sizeof(T) * n * batch));
  TRY_CHNS(C.cpart.ensure(piece * batch));
  T *w = ws.wv.as<T>(), *y = ws.yv.as<T>();
  double *part = C.cpart.as<double>();
  for (int v0 = 0; v0 < total; v0 += batch) {
    const unsigned nv = (unsigned)std::min(batch, total - v0);
    const dim3 gp(grid_n(m->n_nodes), nv);
    if (dim == 2) k_probe_coarse<T, 5, 2><<<gp, kB, 0, st>>>(g, C.pos, v0, w);
    else k_probe_coarse<T, 6, 3><<<gp, kB, 0, st>>>(g, C.pos, v0, w);
    note_launches(1);
    TRY_CHNS(jv(ctx, w, y, int(nv)));
    if (C.direct) {
      const dim3 gd((unsigned)((m->n_nodes + kB - 1) / kB), nv);
      if (dim == 2) k_collect_direct<T, 5, 2><<<gd, kB, 0, st>>>(g, C.pos, C.cinv, v0, y, M);
      else k_collect_direct<T, 6, 3><<<gd, kB, 0, st>>>(g, C.pos, C.cinv, v0, y, M);
      note_launches(1);
      continue;
    }
    const dim3 gr((unsigned)C.n_pieces, nv);
    if (dim == 2)
      k_gather_coarse<T, 5, 2><<<gr, kChunk, 0, st>>>(g, C.piece_node, C.piece_begin, C.rnode, C.rw, C.pos, v0, y,
                                                  part);
    else
      k_gather_coarse<T, 6, 3><<<gr, kChunk, 0, st>>>(g, C.piece_node, C.piece_begin, C.rnode, C.rw, C.pos, v0, y,
                                                  part);
    const dim3 gs((unsigned)((C.ncn * (nf << dim) + kB - 1) / kB), nv);
    k_gather_sum<<<gs, kB, 0, st>>>(g, v0, C.n_pieces, C.node_piece, part, M, nc0, C.ncn);
    note_launches(2);
  }
  // A_c^{-1} per instance, in the element precision: the FP32 path inverts
  // in float (A_c is ill-conditioned along a pressure direction only, which
  // float resolves: per-field errors of the applied inverse ~1e-6 at
  // cond(A_c) ~ 1e9), the FP64 path in double.  Both copies are kept: M in
  // double, Minv32 in float.
  int *bad = reinterpret_cast<int *>(C.vec.as<double>() + 3 * C.nc);
  int32_t *piv = C.piv.as<int32_t>();
  float *M32 = C.Minv32.as<float>();
  CHNS_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), st));
  if (nc0 <= kPanelRows) {
    // two matrices to go back and forth between, and the panel's columns
    const int64_t np = nc0 * kPanelMax * C.n_inst;
    TRY_CHNS(C.gj.ensure(sizeof(T) * (2 * nn + np)));
    T *b0 = C.gj.as<T>();
    int32_t *origin = nullptr;
    k_copy_cast<double, T><<<grid_n(nn), kB, 0, st>>>(M, nn, b0);
    const T *r = gauss_jordan_panels<T>(b0, b0 + nn, nc0, C.n_inst, b0 + 2 * nn, piv, &origin, bad, st);
    k_gj_columns<T, double, float><<<grid_n(nn), kB, 0, st>>>(r, nc0, nn, origin, M, M32);
  } else if (sizeof(T) == sizeof(float)) {
    void *colv = C.vec.as<double>() + 2 * C.nc;  // nc0 per instance
    k_copy_cast<double, float><<<grid_n(nn), kB, 0, st>>>(M, nn, M32);
    gauss_jordan_columns<float>(M32, nc0, C.n_inst, static_cast<float *>(colv), piv, bad, st);
    k_copy_cast<float, double><<<grid_n(nn), kB, 0, st>>>(M32, nn, M);
  } else {
    void *colv = C.vec.as<double>() + 2 * C.nc;
    gauss_jordan_columns<double>(M, nc0, C.n_inst, static_cast<double *>(colv), piv, bad, st);
    k_copy_cast<double, float><<<grid_n(nn), kB, 0, st>>>(M, nn, M32);
  }
  note_launches(2);
  int hbad = 0;
  CHNS_CUDA_TRY(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  CHNS_CUDA_TRY(cudaStreamSynchronize(st));
  if (C.gj.bytes > kKeepGj) C.gj.release();  // the stream has drained
  if (hbad) { set_error("singular coarse operator"); return CHNS_ERR_KRYLOV; }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { set_error("coarse build: %s", cudaGetErrorString(e)); return CHNS_ERR_CUDA; }
  C.ready = true;
  return CHNS_OK;
}
template chns_status coarse_build<float>(chns_mesh *, JvFn<float>, void *, cudaStream_t);
template chns_status coarse_build<double>(chns_mesh *, JvFn<double>, void *, cudaStream_t);

// z = B^{-1} v (+ P A_c^{-1} R v when the coarse space is ready and wanted).  On
// a coarse grid that is the mesh, P and R are the identity and the inverse is
// in node order: without a block term the apply is one product.
template <typename T>
void precond_apply(chns_mesh *m, const T *Binv, bool coarse, const T *v, T *z, cudaStream_t st) {
  Coarse &C = m->coarse;
  const bool use = coarse && C.ready;
  CGeo g{m->dim, m->nf, C.nc1, m->n_nodes, C.ncn_inst, C.nc0, C.direct ? 1 : 0};
  const T *zc = nullptr;
  if (use) {
    const T *rc = v;
    T *out = C.direct && !Binv ? z : reinterpret_cast<T *>(C.vec.as<double>() + C.nc);
    if (!C.direct) {
      T *r = reinterpret_cast<T *>(C.vec.as<double>());
      const bool whole = C.n_pieces == C.ncn;
      T *part = whole ? r : reinterpret_cast<T *>(C.rpart.as<double>());
      const unsigned np = (unsigned)C.n_pieces;
      auto restrict_with = [&](auto *rw) {
        using W = std::remove_cv_t<std::remove_reference_t<decltype(*rw)>>;
        if (m->dim == 2)
          launch_next(k_restrict_lists<T, 5, W>, np, kGroups * 8, st, C.piece_begin, C.rnode, rw, v, part);
        else
          launch_next(k_restrict_lists<T, 6, W>, np, kGroups * 8, st, C.piece_begin, C.rnode, rw, v, part);
      };
      if constexpr (sizeof(T) == sizeof(double)) {
        if (C.rw64) restrict_with(C.rw64);
        else restrict_with(C.rw);
      } else {
        restrict_with(C.rw);
      }
      note_launches(1);
      if (!whole) {
        launch_next(k_restrict_pieces<T>, (unsigned)((C.nc + kB - 1) / kB), kB, st, C.nc, m->nf, C.node_piece, part, r);
        note_launches(1);
      }
      rc = r;
    }
    const T *Mi = sizeof(T) == sizeof(float) ? reinterpret_cast<const T *>(C.Minv32.as<float>())
                                             : reinterpret_cast<const T *>(C.M.as<double>());
    const unsigned gm = (unsigned)((C.nc * 32 + kB - 1) / kB);
    launch_next(k_coarse_matvec<T>, gm, kB, st, Mi, C.nc0, C.nc0 * C.nc0, C.nc, C.nc0, rc, out);
    note_launches(1);
    if (out == z) return;
    zc = out;
  }
  const int32_t *ni = (use && m->n_inst > 1) ? m->node_inst : nullptr;
  const unsigned gb = (unsigned)((m->n_nodes * 8 + kB - 1) / kB);
  if (m->dim == 2) launch_next(k_block_prolong<T, 5, 2>, gb, kB, st, g, C.pos, ni, Binv, v, zc, z);
  else launch_next(k_block_prolong<T, 6, 3>, gb, kB, st, g, C.pos, ni, Binv, v, zc, z);
  note_launches(1);
}
template void precond_apply<float>(chns_mesh *, const float *, bool, const float *, float *, cudaStream_t);
template void precond_apply<double>(chns_mesh *, const double *, bool, const double *, double *, cudaStream_t);

}  // namespace chns
