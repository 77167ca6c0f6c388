// Node splitting (Sec. III.B "Node Splitting", Appendix A "Saving Memory"):
// the node read as a matrix (rows over the left legs, columns over the right
// legs, each group in the order given, last leg fastest), decomposed by the
// one-sided Jacobi SVD of Hestenes (1958) in float32, truncated, and written
// out as U sqrt(S) and sqrt(S) V^T (split_node) or U, S, V^T (full SVD).
//
// One-sided Jacobi orthogonalises the columns of a working matrix W (L x r,
// r = min(M, N) columns of length L = max(M, N): the matrix view itself when
// M >= N, else its transpose) by plane rotations of column pairs, accumulating
// the rotations in V (r x r, starting from I). At convergence W = U S and the
// matrix (or its transpose) is W V^T: the singular values are the column norms
// of W.
//
// The method is a chain of rounds, so what bounds it is a round's latency and
// the passes over W and V. Rotating one pair per CTA and round takes r - 1
// rounds a sweep, each a launch that reads and writes all of W and V for one
// rotation per column (5.3 us a round at r = 256). Here the columns are in
// blocks of 16 and a round pairs blocks: a CTA forms the 32 x 32 Gram matrix of
// its two blocks, runs the round's 16 x 16 rotations on it in shared memory
// (16 steps of 16 disjoint pairs; in a sweep's first round all 32 x 31 / 2
// pairs, 31 steps), collecting them in Q, and applies Q to the blocks of W and
// V in one pass: r / 16 - 1 rounds a sweep, the same pairs rotated once each.
// Blocks pair up by the circle method; all sweeps run in one cooperative
// launch, its rounds separated by a device-wide barrier (bounded), and stop
// after a sweep without a rotation. A block is stored row by row (16 floats a
// row): a warp takes one row of the two blocks, lane j column j, the row's
// other entries broadcast from shared memory, for the Gram matrix (lane j: its
// column of it) and for the product with Q alike. The rows are shared out over
// the CTAs of a cluster, which add up their Gram matrices and rotate alike.
// The angles are float32, from approximate roots: an angle that is a little off
// leaves a little for the next round, while the values come from the columns'
// norms (in 64 bits) and c^2 + s^2 = 1 holds to rounding. Error against 64 bits
// of two-site nodes of bond 6 to 160, half and all of the values kept, one pair
// at a time with 64-bit angles -> here: values 1.4e-7 .. 5.4e-7 -> 0.7e-7 ..
// 1.2e-7, the product 3.4e-7 .. 3.8e-6 -> 2.5e-7 .. 2.1e-6, 0.2 to 0.84 of the
// former at every size. Gram sums over warps and CTAs that keep their roundings
// (two-sum) took 10 % longer for the same errors.
// At most two blocks of columns and many rows (svd_tall): the rows are shared
// out over the whole grid, Gram sums go through device memory, and rows are
// stored only as wide as they are (4, 8 or 16 columns). One cluster for such a
// pair took longer than one CTA per two columns: 4e6 x 1 0.69 ms that way, 8.7
// by a cluster, 0.47 now; 4e6 x 2 1.31, 14.5, 0.50; 1e6 x 5 7.1, 9.6, 0.46;
// 2e5 x 32 22.7, 3.5, 0.77.
// Measured (two-site node of bond 128, r = 256, 13 sweeps): 18.7 -> 2.3 ms; a
// round takes ~19,000 cycles: Gram matrix 1,300, its sum over 8 warps and 8
// CTAs 4,800, the 17 rotation steps 9,800 (a dependent chain of ~370 cycles
// each), W and V 2,300, the barrier 2,600. r = 1000: 98 -> 14 ms, 2048: 380 ->
// 77 ms. Rotations that also sort the columns by norm took 1-5 more sweeps.
#include <math.h>
#include <string.h>

#include <vector>

#include "ptx.cuh"
#include "tn_internal.h"

namespace tn {
namespace {

constexpr int SVD_THREADS = 256;
constexpr int SVD_WARPS = SVD_THREADS / 32;
constexpr int SVD_MAX_SWEEPS = 40;
constexpr int SVD_B = 16;      // columns of a block
constexpr int SVD_CH = 256;    // rows staged at once
constexpr int SVD_CLUSTER = 8; // most CTAs that share out a pair's rows
// W is the matrix times a power of two that brings the sum of its squares to
// 2^80 at most; a column whose squared norm is 2^-100 or less there (2^-90 of
// the matrix) is left as it is. So a rotation's quotients stay normal numbers
// whatever the node's scale: squares of 2^-126 and less would count as 0 in
// the approximate roots.
constexpr int SVD_TOP = 40;
constexpr float SVD_NULL = 0x1p-100f;

// The node's matrix view: element (i, j) at A + loff(i) + roff(j).
struct SplitView {
  const float* A;
  int64_t M, N;
  int32_t nl, nr;
  int32_t wide;  // M < N: W holds the transpose
  int32_t pad;
  int32_t ldim[TN_MAX_RANK], rdim[TN_MAX_RANK];
  int64_t lstr[TN_MAX_RANK], rstr[TN_MAX_RANK];
};

__device__ __forceinline__ int64_t leg_offset(int64_t idx, int n, const int32_t* dim, const int64_t* str) {
  int64_t off = 0;
  for (int p = n - 1; p >= 0; --p) {
    int64_t hi;
    if (idx <= 0xFFFFFFFFll) hi = (uint32_t)idx / (uint32_t)dim[p];
    else hi = idx / dim[p];
    off += (idx - hi * dim[p]) * str[p];
    idx = hi;
  }
  return off;
}

// *bits: the bits of the node's largest finite magnitude (0 before); odd[c]:
// bit 0 an infinity, bit 1 a NaN in column c of W (0 before). Such a column
// takes no part: a product with it would spread over its block.
__global__ void svd_largest(SplitView v, unsigned* bits, unsigned* odd) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned m = 0u;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < v.M * v.N; e += stride) {
    const int64_t i = e <= 0xFFFFFFFFll && v.N <= 0xFFFFFFFFll ? (uint32_t)e / (uint32_t)v.N : e / v.N, j = e - i * v.N;
    const float x = v.A[leg_offset(i, v.nl, v.ldim, v.lstr) + leg_offset(j, v.nr, v.rdim, v.rstr)];
    const unsigned b = __float_as_uint(fabsf(x));
    if (b < 0x7F800000u) m = max(m, b);
    else atomicOr(odd + (v.wide ? i : j), b == 0x7F800000u ? 1u : 2u);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(bits, m);
}

// The exponent of the power of two W is scaled by; 0 without a finite entry but
// zeros. half: (log2 of the matrix's entries) / 2, rounded up.
__device__ __forceinline__ int svd_shift(unsigned bits, int half) {
  return bits == 0u ? 0 : SVD_TOP - half - 1 - ilogbf(__uint_as_float(bits));
}

// W in blocks of 2^lw columns (16; a tall node's one block may have fewer),
// [block][row][column] (zeros past column r and for `odd` ones), V = I likewise.
__global__ void svd_gather(SplitView v, const unsigned* bits, const unsigned* odd, int half, int lw, float* __restrict__ W, float* __restrict__ V,
                           int64_t L, int64_t r, int64_t cols) {
  const int shift = svd_shift(*bits, half);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t w = first; w < L * cols; w += stride) {
    // neighbouring threads walk the view's own rows where those are columns of W
    const int64_t blk = (cols >> lw) == 1 ? 0 : w / (L << lw), in = w - ((blk * L) << lw);
    const int64_t row = in >> lw, col = (blk << lw) + (in & ((1 << lw) - 1));
    float x = 0.0f;
    if (col < r && odd[col] == 0u) {
      const int64_t i = v.wide ? col : row, j = v.wide ? row : col;
      x = ldexpf(v.A[leg_offset(i, v.nl, v.ldim, v.lstr) + leg_offset(j, v.nr, v.rdim, v.rstr)], shift);
    }
    W[w] = x;
  }
  for (int64_t e = first; e < r * cols; e += stride) {
    const int64_t blk = e / (r << lw), in = e - ((blk * r) << lw);
    V[e] = in >> lw == (blk << lw) + (in & ((1 << lw) - 1)) ? 1.0f : 0.0f;
  }
}

// Pair `k` of round `t` over rp (even) slots: slot 0 stays, the others
// rotate by one position per round, and position k meets position rp-1-k.
__device__ __forceinline__ int circle_slot(int pos, int t, int rp) {
  return pos == 0 ? 0 : 1 + (pos - 1 + t) % (rp - 1);
}

struct SvdParams {
  float* W;
  float* V;
  int64_t L;
  int32_t r, ns, nb;   // columns; blocks; blocks rounded up to even (the added one is zeros, not stored)
  int32_t cluster;     // CTAs sharing out a pair's rows
  float tol;
  unsigned long long* bar;  // barrier word (zero)
  int* counts;         // rotations per sweep (zero)
  int* sweeps;         // out: sweeps used, negative if the limit was reached
  float* parts;        // tall nodes: the CTAs' Gram sums, two sets in turn
  int* status;
};

struct SvdSmem {
  float X[2][SVD_CH][2 * SVD_B];               // rows of the two blocks
  float part[2 * SVD_B][2 * SVD_B];            // this CTA's part of the Gram matrix, read by its cluster
  float red[SVD_WARPS][2 * SVD_B][2 * SVD_B];  // Gram sums of the warps
  float G[2][2 * SVD_B][2 * SVD_B + 1];
  float Q[2 * SVD_B][2 * SVD_B + 1];
  int32_t abort;
};

// Rows [row0, row0 + rows) of blocks p and q of X (n rows a block) into a
// staging buffer (zeros for a block past the ns stored ones).
__device__ __forceinline__ void svd_stage(float (*x)[2 * SVD_B], const float* __restrict__ X, int64_t n, int p, int q,
                                          int ns, int64_t row0, int rows) {
  const float* xp = X + ((int64_t)p * n + row0) * SVD_B;
  const float* xq = X + ((int64_t)q * n + row0) * SVD_B;
  for (int i = threadIdx.x; i < rows * 8; i += SVD_THREADS) {
    const int row = i >> 3, c = (i & 7) * 4;
    if ((c < SVD_B ? p : q) < ns)
      ptx::cp_async16(ptx::smem_addr(&x[row][c]), (c < SVD_B ? xp + c : xq + c - SVD_B) + row * SVD_B);
    else
      *reinterpret_cast<float4*>(&x[row][c]) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  ptx::cp_async_commit();
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A float of the same shared-memory variable in the cluster's CTA `rank`.
__device__ __forceinline__ float cluster_load(const float* p, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(ptx::smem_addr(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
// Approximate square root, reciprocal and its square root (subnormals as 0).
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The rotations (Hestenes) of one round on the Gram matrix in s.G[0], and
// their product in s.Q: for a pair with a = g_pp, b = g_qq, g = g_pq the
// tangent t is the smaller root, h sign(d) / (|d| + sqrt(d^2 + h^2)) for d = (b
// - a) / sqrt(ab) and h = 2 g / sqrt(ab); c = 1 / sqrt(1 + t^2), s = c t, and
// the columns become (c p - s q, s p + c q). Pairs orthogonal to within tol
// (|g| <= tol sqrt(ab)) are left alone, as are columns of SVD_NULL; counted are
// only those above 16 tol: the sweeps end when none is, and what the last one
// still found below that is rotated away. FULL: all pairs of the 32 columns by
// the circle method, else the pairs across the two blocks. Every warp computes the step's 16 angles
// (lanes 0-15; approximate quotients and roots: they only move the angle, the
// next rounds see what is left); thread (u, v) updates the 2 x 2 block of pairs
// u and v and two rows of Q. Returns whether it rotated anything, and adds to
// the count.
template <bool FULL>
__device__ __forceinline__ bool svd_rotate(SvdSmem& s, float tol, int& count) {
  constexpr int C = 2 * SVD_B;
  const int tid = threadIdx.x, u = tid >> 4, v = tid & 15;
  bool rotated = false;
  for (int t = 0; t < (FULL ? C - 1 : SVD_B); ++t) {
    auto slot = [&](int pos) {  // circle over the 32 columns: slot 0 stays
      int x = pos - 1 + t;
      if (x >= C - 1) x -= C - 1;
      return pos == 0 ? 0 : 1 + x;
    };
    const int pv = FULL ? slot(v) : v, qv = FULL ? slot(C - 1 - v) : SVD_B + ((v + t) & (SVD_B - 1));
    const int pu = FULL ? slot(u) : u, qu = FULL ? slot(C - 1 - u) : SVD_B + ((u + t) & (SVD_B - 1));
    const float(*g)[C + 1] = s.G[t & 1];
    float(*gn)[C + 1] = s.G[(t & 1) ^ 1];
    const float al = g[pv][pv], be = g[qv][qv], ga = g[pv][qv];
    const float b00 = g[pu][pv], b01 = g[pu][qv], b10 = g[qu][pv], b11 = g[qu][qv];
    // scaled by the two norms, so that no square leaves the exponent range
    const float ia = rsqrt_approx(al), ib = rsqrt_approx(be), co = ga * ia * ib;
    const bool go = al > SVD_NULL && be > SVD_NULL && fabsf(co) > tol;
    const float d = (be - al) * ia * ib, h = co + co;
    // the root is at most |d| + |h|, which it gives way to where d^2 overflows
    // (norms far apart: a pair turned by 0 for it would be counted for ever)
    const float root = fminf(sqrt_approx(fmaf(d, d, h * h)), fabsf(d) + fabsf(h));
    const float tt = fminf(fabsf(h) * rcp_approx(fabsf(d) + root), 1.0f);
    const float ts = (d < 0.0f) != (h < 0.0f) ? -tt : tt;
    float c = rsqrt_approx(fmaf(tt, tt, 1.0f)), sn = c * ts;
    // c^2 + s^2 = 1 to the rounding of c and s: a bias here would drift the
    // column norms over a matrix's thousands of rotations
    const float e = -0.5f * fmaf(sn, sn, fmaf(c, c, -1.0f));
    c = go ? fmaf(e, c, c) : 1.0f;
    sn = go ? fmaf(e, sn, sn) : 0.0f;
    rotated |= __any_sync(0xffffffffu, go);
    count += __popc(__ballot_sync(0xffffffffu, go && fabsf(co) > 16.0f * tol) & 0xffffu);
    const float cu = __shfl_sync(0xffffffffu, c, u), su = __shfl_sync(0xffffffffu, sn, u);
    const float x0 = c * b00 - sn * b01, x1 = sn * b00 + c * b01, y0 = c * b10 - sn * b11, y1 = sn * b10 + c * b11;
    gn[pu][pv] = cu * x0 - su * y0;
    gn[qu][pv] = su * x0 + cu * y0;
    gn[pu][qv] = cu * x1 - su * y1;
    gn[qu][qv] = su * x1 + cu * y1;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float* row = s.Q[u + k * SVD_B];
      const float a0 = row[pv], a1 = row[qv];
      row[pv] = c * a0 - sn * a1;
      row[qv] = sn * a0 + c * a1;
    }
    __syncthreads();
  }
  return rotated;
}

// One block pair, by a cluster whose CTAs share out the rows: Gram matrix
// (each its part, then the sum over the cluster), rotations (the same in
// every CTA), Q applied to W and V. Adds the counted rotations (the same in
// every thread).
__device__ void svd_block_pair(const SvdParams& P, SvdSmem& s, int p, int q, bool full, int& count) {
  constexpr int C = 2 * SVD_B;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_rank(), cs = P.cluster;
  const int64_t lp = (P.L + cs - 1) / cs, w0 = min(P.L, lp * rank), wn = min(P.L, w0 + lp) - w0;
  const int vp = (P.r + cs - 1) / cs, v0 = min(P.r, vp * rank), vn = min(P.r, v0 + vp) - v0;
  const int nw = (int)((wn + SVD_CH - 1) / SVD_CH), nv = (vn + SVD_CH - 1) / SVD_CH;
  // item i of the apply pass: rows of W, then of V, in buffer i & 1
  auto rows_of = [&](int i) {
    return i < nw ? (int)min((int64_t)SVD_CH, wn - (int64_t)i * SVD_CH) : min(SVD_CH, vn - (i - nw) * SVD_CH);
  };
  auto stage = [&](int i) {
    if (i >= nw + nv) return;
    if (i < nw) svd_stage(s.X[i & 1], P.W, P.L, p, q, P.ns, w0 + (int64_t)i * SVD_CH, rows_of(i));
    else svd_stage(s.X[i & 1], P.V, P.r, p, q, P.ns, v0 + (int64_t)(i - nw) * SVD_CH, rows_of(i));
  };
  // Gram matrix: lane j sums x_i x_j over the warp's rows for every i
  float2 acc[C / 2];
#pragma unroll
  for (int m = 0; m < C / 2; ++m) acc[m] = make_float2(0.f, 0.f);
  if (nw > 0) stage(0);
  for (int c = 0; c < nw; ++c) {
    ptx::cp_async_wait<0>();
    __syncthreads();
    if (c + 1 < nw) stage(c + 1);
    const float(*x)[C] = s.X[c & 1];
    const int rows = rows_of(c);
#pragma unroll 4
    for (int row = w; row < rows; row += SVD_WARPS) {
      const float mine = x[row][lane];
      const float2 mm = make_float2(mine, mine);
#pragma unroll
      for (int m = 0; m < C / 4; ++m) {
        const float4 f = *reinterpret_cast<const float4*>(&x[row][4 * m]);
        acc[2 * m] = __ffma2_rn(make_float2(f.x, f.y), mm, acc[2 * m]);
        acc[2 * m + 1] = __ffma2_rn(make_float2(f.z, f.w), mm, acc[2 * m + 1]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < C / 2; ++m) {
    s.red[w][2 * m][lane] = acc[m].x;
    s.red[w][2 * m + 1][lane] = acc[m].y;
  }
  __syncthreads();
  // the staging buffers are free unless W fits one: the apply pass's first loads
  if (nw == 1) stage(1);
  else stage(0);
#pragma unroll
  for (int e = 0; e < C * C / SVD_THREADS; ++e) {
    const int i = (tid + e * SVD_THREADS) / C;
    float g[SVD_WARPS];
#pragma unroll
    for (int u = 0; u < SVD_WARPS; ++u) g[u] = s.red[u][i][lane];
#pragma unroll
    for (int o = 1; o < SVD_WARPS; o *= 2)
#pragma unroll
      for (int u = 0; u < SVD_WARPS; u += 2 * o) g[u] += g[u + o];
    s.part[i][lane] = g[0];
    s.Q[i][lane] = i == lane ? 1.0f : 0.0f;
  }
  if (cs > 1) {
    cluster_sync();
    float g[C * C / SVD_THREADS][SVD_CLUSTER];
#pragma unroll
    for (int e = 0; e < C * C / SVD_THREADS; ++e)
#pragma unroll
      for (int k = 0; k < SVD_CLUSTER; ++k)
        g[e][k] = k < cs ? cluster_load(&s.part[(tid + e * SVD_THREADS) / C][lane], k) : 0.0f;
#pragma unroll
    for (int e = 0; e < C * C / SVD_THREADS; ++e) {
#pragma unroll
      for (int k = 1; k < SVD_CLUSTER; ++k) g[e][0] += g[e][k];
      s.G[0][(tid + e * SVD_THREADS) / C][lane] = g[e][0];
    }
  } else {
    __syncthreads();
    for (int e = 0; e < C * C / SVD_THREADS; ++e) {
      const int i = (tid + e * SVD_THREADS) / C;
      s.G[0][i][lane] = s.part[i][lane];
    }
  }
  __syncthreads();
  const bool rotated = full ? svd_rotate<true>(s, P.tol, count) : svd_rotate<false>(s, P.tol, count);
  if (!rotated) {
    ptx::cp_async_wait<0>();
    if (cs > 1) cluster_sync();
    else __syncthreads();
    return;
  }
  // x <- x Q for every row: lane j holds column j of Q
  const bool stored = (lane < SVD_B ? p : q) < P.ns;
  float2 qc[C / 2];
#pragma unroll
  for (int m = 0; m < C / 2; ++m) qc[m] = make_float2(s.Q[2 * m][lane], s.Q[2 * m + 1][lane]);
  for (int i = 0; i < nw + nv; ++i) {
    ptx::cp_async_wait<0>();
    __syncthreads();
    if (i + 1 < nw + nv && !(nw == 1 && i == 0)) stage(i + 1);
    const float(*x)[C] = s.X[i & 1];
    const int rows = rows_of(i);
    const int64_t n = i < nw ? P.L : P.r, row0 = i < nw ? w0 + (int64_t)i * SVD_CH : v0 + (int64_t)(i - nw) * SVD_CH;
    float* out = (i < nw ? P.W : P.V) + ((lane < SVD_B ? (int64_t)p : (int64_t)q) * n + row0) * SVD_B + (lane & (SVD_B - 1));
    for (int r0 = w * 4; r0 < rows; r0 += SVD_WARPS * 4) {
      float2 o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) o[k] = make_float2(0.f, 0.f);
#pragma unroll
      for (int m = 0; m < C / 4; ++m)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 f = *reinterpret_cast<const float4*>(&x[min(r0 + k, rows - 1)][4 * m]);
          o[k] = __ffma2_rn(make_float2(f.x, f.y), qc[2 * m], o[k]);
          o[k] = __ffma2_rn(make_float2(f.z, f.w), qc[2 * m + 1], o[k]);
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (stored && r0 + k < rows) out[(int64_t)(r0 + k) * SVD_B] = o[k].x + o[k].y;
    }
  }
  // the buffers are free for the next pair, the parts read by the cluster
  if (cs > 1) cluster_sync();
  else __syncthreads();
}

__device__ __forceinline__ unsigned svd_load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Device-wide barrier, by one thread of every CTA, arrival `epoch` (from 1).
// Low half of *bar: arrivals; high half: the epoch at which a wait ran out.
// Bounded, and all CTAs get the same answer: only a barrier that is not
// complete can be given up, and one given up stays so when late CTAs arrive.
// So all leave behind the same round, and none reads the shared memory of a CTA
// of its cluster that has left.
__device__ __forceinline__ bool svd_barrier(unsigned long long* bar, unsigned epoch, int* status) {
  __threadfence();
  atomicAdd(bar, 1ull);
  const unsigned target = epoch * gridDim.x;
  const uint64_t start = ptx::globaltimer();
  for (unsigned i = 1;; ++i) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
    if ((unsigned)(v >> 32) == epoch) return false;
    if ((unsigned)v >= target) break;
    if ((i & 63u) == 0u && ptx::globaltimer() - start > ptx::kWaitLimitNs &&
        atomicCAS(bar, v, v | ((unsigned long long)epoch << 32)) == v) {
      ptx::set_status(status, TN_ERR_TIMEOUT);
      return false;
    }
  }
  __threadfence();
  return true;
}

// All sweeps: one cooperative launch.
__global__ void __launch_bounds__(SVD_THREADS) svd_jacobi(const __grid_constant__ SvdParams P) {
  extern __shared__ __align__(16) uint8_t raw[];
  SvdSmem& s = *reinterpret_cast<SvdSmem*>(raw);
  const int tid = threadIdx.x;
  if (tid == 0) s.abort = 0;
  unsigned epoch = 0;
  bool done = false;
  int used = 0;
  while (!done && used < SVD_MAX_SWEEPS) {
    for (int t = 0; t < P.nb - 1; ++t) {
      int rotations = 0;
      for (int k = blockIdx.x / P.cluster; k < P.nb / 2; k += gridDim.x / P.cluster)
        svd_block_pair(P, s, circle_slot(k, t, P.nb), circle_slot(P.nb - 1 - k, t, P.nb), t == 0, rotations);
      // device-wide barrier: every CTA's part of W, V and the count is in place
      __syncthreads();
      if (tid == 0) {
        if (rotations && blockIdx.x % P.cluster == 0) atomicAdd(P.counts + used, rotations);
        if (!svd_barrier(P.bar, ++epoch, P.status)) s.abort = 1;
      }
      __syncthreads();
      if (s.abort) return;
    }
    done = svd_load_acquire(reinterpret_cast<const unsigned*>(P.counts + used)) == 0;
    ++used;
  }
  if (blockIdx.x == 0 && tid == 0) *P.sweeps = done ? used : -used;
}

// s + x, s a sum (x) and what its roundings left (y) (Knuth's two-sum).
__device__ __forceinline__ void add_exact(float2& s, float x) {
  const float t = s.x + x, u = t - s.x;
  s.y += (s.x - (t - u)) + (x - u);
  s.x = t;
}

// All sweeps of a node of at most two blocks (COLS columns stored: one block of
// 4, 8 or 16, or two of 16), its rows shared out over the grid: cooperative
// launch. A warp takes 32 / COLS rows at once. Every CTA adds up all Gram sums
// in the same order and rotates alike, so one barrier a sweep is enough (the
// sums are written to the other set meanwhile) and the count needs no adding.
template <int COLS>
__global__ void __launch_bounds__(SVD_THREADS) svd_tall(const __grid_constant__ SvdParams P) {
  constexpr int C = 2 * SVD_B, BW = COLS < SVD_B ? COLS : SVD_B, Q4 = COLS / 4, SUB = 32 / COLS;
  constexpr int CH = 2 * SVD_CH * SVD_B / COLS;  // rows staged at once
  constexpr int E = COLS * COLS, NP = E < SVD_THREADS ? SVD_THREADS / E : 1;  // threads adding up one entry
  extern __shared__ __align__(16) uint8_t raw[];
  SvdSmem& s = *reinterpret_cast<SvdSmem*>(raw);
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, col = lane % COLS, sub = lane / COLS;
  const int rank = (int)blockIdx.x, cs = (int)gridDim.x;
  const int64_t lp = (P.L + cs - 1) / cs, w0 = min(P.L, lp * rank), wn = min(P.L, w0 + lp) - w0;
  const int nw = (int)((wn + CH - 1) / CH), items = nw + (rank == 0 ? 1 : 0);  // W's chunks; the first CTA: V
  float* X = &s.X[0][0][0];
  auto rows_of = [&](int i) { return i < nw ? (int)min((int64_t)CH, wn - (int64_t)i * CH) : P.r; };
  // element (row, c) of item i's first row on
  auto at = [&](int i, int row, int c) -> float* {
    const int64_t n = i < nw ? P.L : P.r, row0 = i < nw ? w0 + (int64_t)i * CH : 0;
    return (i < nw ? P.W : P.V) + ((c / BW) * n + row0 + row) * BW + c % BW;
  };
  auto stage = [&](int i) {
    float* x = X + (i & 1) * CH * COLS;
    const int words = rows_of(i) * Q4;
    for (int e = tid; e < words; e += SVD_THREADS)
      ptx::cp_async16(ptx::smem_addr(x + e * 4), at(i, e / Q4, e % Q4 * 4));
    ptx::cp_async_commit();
  };
  if (tid == 0) s.abort = 0;
  unsigned epoch = 0;
  bool done = false;
  int used = 0;
  while (!done && used < SVD_MAX_SWEEPS) {
    float2 acc[COLS / 2];
#pragma unroll
    for (int m = 0; m < COLS / 2; ++m) acc[m] = make_float2(0.f, 0.f);
    if (nw > 0) stage(0);
    for (int c = 0; c < nw; ++c) {
      ptx::cp_async_wait<0>();
      __syncthreads();
      if (c + 1 < nw) stage(c + 1);
      const float* x = X + (c & 1) * CH * COLS;
      const int rows = rows_of(c);
#pragma unroll 4
      for (int row = w * SUB + sub; row < rows; row += SVD_WARPS * SUB) {
        const float mine = x[row * COLS + col];
        const float2 mm = make_float2(mine, mine);
#pragma unroll
        for (int m = 0; m < Q4; ++m) {
          const float4 f = *reinterpret_cast<const float4*>(x + row * COLS + 4 * m);
          acc[2 * m] = __ffma2_rn(make_float2(f.x, f.y), mm, acc[2 * m]);
          acc[2 * m + 1] = __ffma2_rn(make_float2(f.z, f.w), mm, acc[2 * m + 1]);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < COLS / 2; ++m) {
#pragma unroll
      for (int o = COLS; o < 32; o <<= 1) {
        acc[m].x += __shfl_xor_sync(0xffffffffu, acc[m].x, o);
        acc[m].y += __shfl_xor_sync(0xffffffffu, acc[m].y, o);
      }
      if (sub == 0) {
        s.red[w][2 * m][col] = acc[m].x;
        s.red[w][2 * m + 1][col] = acc[m].y;
      }
    }
    __syncthreads();
    float* parts = P.parts + (size_t)(used & 1) * cs * E;
    for (int e = tid; e < E; e += SVD_THREADS) {
      float2 g = make_float2(s.red[0][e / COLS][e % COLS], 0.0f);
      for (int u = 1; u < SVD_WARPS; ++u) add_exact(g, s.red[u][e / COLS][e % COLS]);
      __stcg(parts + (size_t)rank * E + e, g.x + g.y);
    }
    for (int e = tid; e < C * C; e += SVD_THREADS) {
      s.Q[e / C][e % C] = e / C == e % C ? 1.0f : 0.0f;
      s.G[0][e / C][e % C] = 0.0f;
    }
    __syncthreads();
    if (tid == 0 && !svd_barrier(P.bar, ++epoch, P.status)) s.abort = 1;
    __syncthreads();
    if (s.abort) return;
    float2* sums = reinterpret_cast<float2*>(X);  // [NP][E]
    for (int e = tid; e < E * NP; e += SVD_THREADS) {
      float2 g = make_float2(0.f, 0.f);
#pragma unroll 8
      for (int k = e / E; k < cs; k += NP) add_exact(g, __ldcg(parts + (size_t)k * E + e % E));
      if (NP == 1) s.G[0][e / COLS][e % COLS] = g.x + g.y;
      else sums[e] = g;
    }
    __syncthreads();
    if (NP > 1 && tid < E) {
      float2 g = sums[tid];
      for (int k = 1; k < NP; ++k) {
        add_exact(g, sums[k * E + tid].x);
        g.y += sums[k * E + tid].y;
      }
      s.G[0][tid / COLS][tid % COLS] = g.x + g.y;
    }
    __syncthreads();
    int count = 0;
    if (svd_rotate<true>(s, P.tol, count)) {
      float2 qc[COLS / 2];
#pragma unroll
      for (int m = 0; m < COLS / 2; ++m) qc[m] = make_float2(s.Q[2 * m][col], s.Q[2 * m + 1][col]);
      if (items > 0) stage(0);
      for (int i = 0; i < items; ++i) {
        ptx::cp_async_wait<0>();
        __syncthreads();
        if (i + 1 < items) stage(i + 1);
        const float* x = X + (i & 1) * CH * COLS;
        const int rows = rows_of(i);
#pragma unroll 4
        for (int row = w * SUB + sub; row < rows; row += SVD_WARPS * SUB) {
          float2 o = make_float2(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < Q4; ++m) {
            const float4 f = *reinterpret_cast<const float4*>(x + row * COLS + 4 * m);
            o = __ffma2_rn(make_float2(f.x, f.y), qc[2 * m], o);
            o = __ffma2_rn(make_float2(f.z, f.w), qc[2 * m + 1], o);
          }
          *at(i, row, col) = o.x + o.y;
        }
      }
      __syncthreads();  // the rows are written and the buffers read
    }
    done = count == 0;
    ++used;
  }
  if (rank == 0 && tid == 0) *P.sweeps = done ? used : -used;
}

// Element (row, col) of a matrix kept in blocks of 2^lw columns, n rows.
__device__ __forceinline__ int64_t blocked(int64_t row, int64_t col, int64_t n, int lw) {
  return ((((col >> lw) * n) + row) << lw) + (col & ((1 << lw) - 1));
}

// Column j's values from its sums of squares: vnorm[j] = |V[:, j]|, wnorm[j] =
// |W[:, j]| and sigma[j] = their quotient, without W's power of two. Both blocks
// took the same products with Q, so what these left of the unit length of V's
// columns is also in W's and cancels. An odd column has the norm its entries have.
struct SvdNorms {
  const unsigned *bits, *odd;
  int half;
  float *sigma, *vnorm, *wnorm;
  __device__ __forceinline__ void put(int64_t j, double a, double b) const {
    const double vn = sqrt(b), wn = odd[j] == 0u ? sqrt(a) : (odd[j] & 2u) ? (double)NAN : (double)INFINITY;
    vnorm[j] = (float)vn;
    wnorm[j] = (float)wn;
    sigma[j] = (float)ldexp(wn / vn, -svd_shift(*bits, half));
  }
};

// Sums of squares of a block's columns over part blockIdx.y of the rows: the
// values of one part, else the parts' sums [part][column][W, V] (svd_values).
__global__ void __launch_bounds__(SVD_THREADS)
svd_norms(const float* __restrict__ W, const float* __restrict__ V, int64_t L, int64_t r, int lw, SvdNorms out,
          double* __restrict__ parts) {
  __shared__ double sa[SVD_THREADS], sb[SVD_THREADS];
  const int tid = threadIdx.x, width = 1 << lw, c = tid & (width - 1), step = SVD_THREADS >> lw;
  const int64_t j = ((int64_t)blockIdx.x << lw) + c;
  const int64_t lp = (L + gridDim.y - 1) / gridDim.y, l1 = min(L, lp * (blockIdx.y + 1));
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (int64_t i = lp * blockIdx.y + (tid >> lw); i < l1; i += step) {
    const double x = W[blocked(i, j, L, lw)];
    a = fma(x, x, a);
  }
  if (blockIdx.y == 0)
    for (int64_t i = tid >> lw; i < r; i += step) {
      const double x = V[blocked(i, j, r, lw)];
      b = fma(x, x, b);
    }
  sa[tid] = a;
  sb[tid] = b;
  __syncthreads();
  for (int o = SVD_THREADS / 2; o >= width; o >>= 1) {
    if (tid < o) {
      sa[tid] += sa[tid + o];
      sb[tid] += sb[tid + o];
    }
    __syncthreads();
  }
  if (tid >= width || j >= r) return;
  if (gridDim.y == 1) {
    out.put(j, sa[tid], sb[tid]);
  } else {
    double* p = parts + 2 * (blockIdx.y * r + j);
    p[0] = sa[tid];
    p[1] = sb[tid];
  }
}
// The values from `n` parts.
__global__ void svd_values(const double* __restrict__ parts, int n, int r, SvdNorms out) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < r; j += gridDim.x * blockDim.x) {
    double a = 0.0, b = 0.0;
#pragma unroll 8
    for (int k = 0; k < n; ++k) {
      a += parts[2 * ((int64_t)k * r + j)];
      b += parts[2 * ((int64_t)k * r + j) + 1];
    }
    out.put(j, a, b);
  }
}

// order[c] = index of the c-th largest singular value (ties by index; a NaN
// sorts last), sorted[c] its value: the rank of j is the number of values
// before it in that strict order, so the ranks are a permutation.
__global__ void svd_sort(const float* __restrict__ sigma, int r, int32_t* __restrict__ order,
                         float* __restrict__ sorted) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= r) return;
  const float sj = isnan(sigma[j]) ? -1.0f : sigma[j];
  int rank = 0;
  for (int i = 0; i < r; ++i) {
    const float si = isnan(sigma[i]) ? -1.0f : sigma[i];
    rank += (si > sj || (si == sj && i < j)) ? 1 : 0;
  }
  order[rank] = j;
  sorted[rank] = sigma[j];
}

// The outputs for the k kept values: columns of V and W over their norms. Left
// (M x k, row-major): W's columns when M >= N, else V's; right (k x N, row-major):
// the other one. absorb: both sides carry sqrt(sigma) (split_node), else
// neither (full SVD). A W column of a zero singular value has no direction:
// its vector is written as zeros (not completed to an orthonormal basis).
__global__ void svd_write(const float* __restrict__ W, const float* __restrict__ V, const int32_t* __restrict__ order,
                          const float* __restrict__ sorted, const float* __restrict__ vnorm,
                          const float* __restrict__ wnorm, int lw, int64_t M, int64_t N, int64_t L, int r, int k, int wide, int absorb, float* __restrict__ U, float* __restrict__ S, float* __restrict__ Vt,
                          float* __restrict__ dropped) {
  const int64_t nl = M * k, nr = (int64_t)k * N, stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t e = t0; e < nl + nr; e += stride) {
    const bool left = e < nl;
    const int64_t f = left ? e : e - nl;
    const int c = left ? (int)(f % k) : (int)(f / N);
    const int64_t i = left ? f / k : f % N;  // row of the left node, column of the right one
    const int j = min(max(order[c], 0), r - 1);
    const float sg = sorted[c];
    const bool from_w = left != (wide != 0);  // left from W iff M >= N
    float x;
    if (from_w) {
      // by the norm itself: a column of rounding noise may be too small for its reciprocal
      x = sg > 0.0f ? W[blocked(i, j, L, lw)] / wnorm[j] * (absorb ? sqrtf(sg) : 1.0f) : 0.0f;
    } else {
      x = V[blocked(i, j, r, lw)] * (absorb ? sqrtf(fmaxf(sg, 0.0f)) / vnorm[j] : 1.0f / vnorm[j]);
    }
    if (left)
      U[f] = x;
    else
      Vt[f] = x;
  }
  for (int64_t c = t0; c < r; c += stride) {
    if (c < k && S) S[c] = sorted[c];
    if (c >= k && dropped) dropped[c - k] = sorted[c];
  }
}

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

struct SplitLayout {
  SplitView v;
  int64_t L, r, ns;  // ns: blocks of 2^lw columns
  int lw, ctas;      // ctas: CTAs of svd_tall, 0: svd_jacobi
  int parts;         // row parts of svd_norms
  size_t w_off, v_off, sig_off, vn_off, wn_off, ord_off, sorted_off, cnt_off, odd_off, parts_off, total;
};

static int plan_split(const tn_tensor* A, const int* left, int nleft, const int* right, int nright,
                      SplitLayout* out) {
  if (!A || A->rank < 0 || A->rank > TN_MAX_RANK || nleft < 0 || nright < 0 || nleft + nright != A->rank)
    return TN_ERR_ARG;
  if ((nleft > 0 && !left) || (nright > 0 && !right)) return TN_ERR_ARG;
  if (A->dtype != TN_F32) return TN_ERR_UNSUPPORTED;
  int seen[TN_MAX_RANK] = {0};
  for (int i = 0; i < nleft + nright; ++i) {
    const int leg = i < nleft ? left[i] : right[i - nleft];
    if (leg < 0 || leg >= A->rank || seen[leg]) return TN_ERR_ARG;
    seen[leg] = 1;
  }
  bool all_zero = true;
  for (int i = 0; i < A->rank; ++i) {
    if (A->shape[i] < 0) return TN_ERR_ARG;
    if (A->stride[i] < 0) return TN_ERR_UNSUPPORTED;
    if (A->stride[i] != 0) all_zero = false;
  }
  int64_t st[TN_MAX_RANK];
  int64_t s = 1;
  for (int i = A->rank - 1; i >= 0; --i) {
    st[i] = all_zero ? s : A->stride[i];
    s *= A->shape[i];
  }
  SplitLayout& o = *out;
  memset(&o, 0, sizeof(o));
  o.v.A = static_cast<const float*>(A->data);
  o.v.nl = nleft;
  o.v.nr = nright;
  o.v.M = o.v.N = 1;
  for (int i = 0; i < nleft; ++i) {
    o.v.ldim[i] = (int32_t)A->shape[left[i]];
    o.v.lstr[i] = st[left[i]];
    o.v.M *= A->shape[left[i]];
  }
  for (int i = 0; i < nright; ++i) {
    o.v.rdim[i] = (int32_t)A->shape[right[i]];
    o.v.rstr[i] = st[right[i]];
    o.v.N *= A->shape[right[i]];
  }
  for (int i = 0; i < A->rank; ++i)
    if (A->shape[i] > 0x7FFFFFFF) return TN_ERR_UNSUPPORTED;
  o.v.wide = o.v.M < o.v.N ? 1 : 0;
  o.L = o.v.wide ? o.v.N : o.v.M;
  o.r = o.v.wide ? o.v.M : o.v.N;
  if (o.r > 0x3FFFFFFF) return TN_ERR_UNSUPPORTED;
  if (o.r > 0 && !o.v.A) return TN_ERR_ARG;
  o.ns = (o.r + SVD_B - 1) / SVD_B;
  // rows shared out over the grid, 1024 or more each, where that makes more
  // CTAs than the widest cluster has
  if (o.ns <= 2 && o.L >= 1024 * (SVD_CLUSTER + 1)) {
    const int64_t most = sm_count();
    o.ctas = (int)(o.L / 1024 < most ? o.L / 1024 : most);
  }
  o.lw = o.ctas && o.r <= 4 ? 2 : o.ctas && o.r <= 8 ? 3 : 4;
  const int64_t cols = o.ns << o.lw, norm_parts = (o.L + 4095) / 4096;
  o.parts = (int)(norm_parts < 256 ? (norm_parts < 1 ? 1 : norm_parts) : 256);
  o.w_off = 0;
  o.v_off = al256(sizeof(float) * (size_t)(o.L * cols));
  o.sig_off = o.v_off + al256(sizeof(float) * (size_t)(o.r * cols));
  o.vn_off = o.sig_off + al256(sizeof(float) * (size_t)o.r);
  o.wn_off = o.vn_off + al256(sizeof(float) * (size_t)o.r);
  o.ord_off = o.wn_off + al256(sizeof(float) * (size_t)o.r);
  o.sorted_off = o.ord_off + al256(sizeof(int32_t) * (size_t)o.r);
  o.cnt_off = o.sorted_off + al256(sizeof(float) * (size_t)(o.r + 1));  // the values, then the sweep count
  o.odd_off = o.cnt_off + 256;  // barrier word, rotations per sweep, the largest magnitude
  o.parts_off = o.odd_off + al256(sizeof(unsigned) * (size_t)o.r);
  // Gram sums of svd_tall's CTAs (two sets), or the norms' parts
  const size_t gram = sizeof(float) * 2 * (size_t)o.ctas * (size_t)(cols * cols);
  const size_t norms = o.parts > 1 ? sizeof(double) * 2 * (size_t)o.parts * (size_t)o.r : 0;
  o.total = o.parts_off + al256(gram > norms ? gram : norms);
  return TN_OK;
}

static unsigned grid_for(int64_t n, int threads) {
  const int64_t b = (n + threads - 1) / threads;
  return (unsigned)(b < 1 ? 1 : (b > 152 * 64 ? 152 * 64 : b));
}

}  // namespace
}  // namespace tn

using namespace tn;

extern "C" {

int64_t tn_split_truncation(const float* sigma_desc, int64_t r, int64_t max_singular_values,
                            double max_truncation_err) {
  if (r <= 0 || !sigma_desc) return 0;
  int64_t k = r;
  if (max_truncation_err >= 0.0) {
    double dropped = 0.0;
    while (k > 0 && dropped + (double)sigma_desc[k - 1] <= max_truncation_err) {
      dropped += (double)sigma_desc[k - 1];
      --k;
    }
  }
  if (max_singular_values > 0 && k > max_singular_values) k = max_singular_values;
  return k < 1 ? 1 : k;
}

size_t tn_split_node_workspace_bytes(const tn_tensor* A, const int* left, int nleft, const int* right, int nright) {
  SplitLayout lay;
  if (plan_split(A, left, nleft, right, nright, &lay) != TN_OK) return 0;
  return lay.total;
}

int tn_split_node(const tn_tensor* A, const int* left, int nleft, const int* right, int nright,
                  int64_t max_singular_values, double max_truncation_err, int absorb, float* U, float* S,
                  float* Vt, float* dropped, int64_t* kept, int32_t* sweeps, void* workspace, size_t ws_bytes,
                  void* stream) {
  SplitLayout lay;
  int rc = plan_split(A, left, nleft, right, nright, &lay);
  if (rc != TN_OK) return rc;
  if (!kept) return TN_ERR_ARG;
  *kept = 0;
  if (sweeps) *sweeps = 0;
  if (lay.r == 0) return TN_OK;
  if (!U || !Vt || (!absorb && !S)) return TN_ERR_ARG;
  if (!workspace || ws_bytes < lay.total || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
    return TN_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint8_t* base = static_cast<uint8_t*>(workspace);
  float* W = reinterpret_cast<float*>(base + lay.w_off);
  float* V = reinterpret_cast<float*>(base + lay.v_off);
  float* sigma = reinterpret_cast<float*>(base + lay.sig_off);
  float* vnorm = reinterpret_cast<float*>(base + lay.vn_off);
  float* wnorm = reinterpret_cast<float*>(base + lay.wn_off);
  int32_t* order = reinterpret_cast<int32_t*>(base + lay.ord_off);
  float* sorted = reinterpret_cast<float*>(base + lay.sorted_off);
  const int64_t L = lay.L, cols = lay.ns << lay.lw;
  const int r = (int)lay.r;
  SvdParams P;
  P.W = W;
  P.V = V;
  P.L = L;
  P.r = r;
  P.ns = (int32_t)lay.ns;
  P.nb = P.ns + (P.ns & 1);
  // counted above 16 tol, a few times the float32 rounding of a length-L dot product
  P.tol = 0.25f * sqrtf((float)L) * 5.9604645e-8f;
  P.bar = reinterpret_cast<unsigned long long*>(base + lay.cnt_off);
  P.counts = reinterpret_cast<int*>(base + lay.cnt_off) + 2;
  P.sweeps = reinterpret_cast<int*>(sorted + r);
  P.status = status_word();
  static_assert(sizeof(int) * (SVD_MAX_SWEEPS + 3) <= 256, "barrier word, rotation counts, largest magnitude");
  unsigned* bits = reinterpret_cast<unsigned*>(P.counts) + SVD_MAX_SWEEPS;
  int half = 0;  // 4^half >= M N
  while (half < 31 && (int64_t(1) << (2 * half)) < L * r) ++half;
  unsigned* odd = reinterpret_cast<unsigned*>(base + lay.odd_off);
  if (cudaMemsetAsync(base + lay.cnt_off, 0, lay.parts_off - lay.cnt_off, s) != cudaSuccess ||
      cudaMemsetAsync(P.sweeps, 0, sizeof(int), s) != cudaSuccess)
    return TN_ERR_CUDA;
  svd_largest<<<grid_for(L * r, 256), 256, 0, s>>>(lay.v, bits, odd);
  svd_gather<<<grid_for(L * cols, 256), 256, 0, s>>>(lay.v, bits, odd, half, lay.lw, W, V, L, lay.r, cols);
  if (cudaGetLastError() != cudaSuccess) return TN_ERR_CUDA;
  P.parts = reinterpret_cast<float*>(base + lay.parts_off);
  void (*kernel)(const SvdParams) = svd_jacobi;
  static std::atomic<uint64_t> attr[5];
  std::atomic<uint64_t>* limit = &attr[0];
  if (lay.ctas) {
    kernel = cols == 4 ? svd_tall<4> : cols == 8 ? svd_tall<8> : cols == 16 ? svd_tall<16> : svd_tall<32>;
    limit = &attr[cols == 4 ? 1 : cols == 8 ? 2 : cols == 16 ? 3 : 4];
  }
  if (!smem_limit_once((const void*)kernel, sizeof(SvdSmem), limit)) return TN_ERR_CUDA;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.blockDim = dim3(SVD_THREADS);
  cfg.dynamicSmemBytes = sizeof(SvdSmem);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (lay.ctas) {
    cfg.gridDim = dim3((unsigned)lay.ctas);
    cfg.numAttrs = 1;
  } else {
    // one CTA per SM; the rows of a pair over as many CTAs (up to 8, at least
    // 32 rows each) as all pairs leave room for
    const int64_t pairs = P.nb / 2, sms = sm_count();
    P.cluster = 1;
    while (P.cluster < SVD_CLUSTER && pairs * P.cluster * 2 <= sms && L >= 64 * P.cluster) P.cluster *= 2;
    for (;; P.cluster /= 2) {
      const int64_t ctas = pairs * P.cluster < sms ? pairs * P.cluster : sms / P.cluster * P.cluster;
      cfg.gridDim = dim3((unsigned)ctas);
      at[1].val.clusterDim.x = (unsigned)P.cluster;
      int fit = 0;
      if (P.cluster == 1 || (cudaOccupancyMaxActiveClusters(&fit, svd_jacobi, &cfg) == cudaSuccess &&
                             (int64_t)fit * P.cluster >= ctas))
        break;
    }
  }
  if (cudaLaunchKernelEx(&cfg, kernel, P) != cudaSuccess) return TN_ERR_CUDA;
  const SvdNorms norms{bits, odd, half, sigma, vnorm, wnorm};
  double* nparts = reinterpret_cast<double*>(base + lay.parts_off);
  svd_norms<<<dim3((unsigned)lay.ns, (unsigned)lay.parts), SVD_THREADS, 0, s>>>(W, V, L, r, lay.lw, norms, nparts);
  if (lay.parts > 1) svd_values<<<grid_for(r, 256), 256, 0, s>>>(nparts, lay.parts, r, norms);
  svd_sort<<<(r + 255) / 256, 256, 0, s>>>(sigma, r, order, sorted);
  if (cudaGetLastError() != cudaSuccess) return TN_ERR_CUDA;
  std::vector<float> host_sorted((size_t)r + 1);
  if (cudaMemcpyAsync(host_sorted.data(), sorted, sizeof(float) * ((size_t)r + 1), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return TN_ERR_CUDA;
  int32_t used = 0;
  memcpy(&used, &host_sorted[(size_t)r], sizeof(used));
  if (used == 0) return TN_ERR_TIMEOUT;  // the barrier's wait expired
  if (sweeps) *sweeps = used;
  const int64_t k = tn_split_truncation(host_sorted.data(), r, max_singular_values, max_truncation_err);
  svd_write<<<grid_for((lay.v.M + lay.v.N) * k + r, 256), 256, 0, s>>>(W, V, order, sorted, vnorm, wnorm, lay.lw, lay.v.M,
                                                                        lay.v.N, L, r, (int)k, lay.v.wide, absorb ? 1 : 0,
                                                                        U, S, Vt, dropped);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) return TN_ERR_CUDA;
  *kept = k;
  return TN_OK;
}

}  // extern "C"
