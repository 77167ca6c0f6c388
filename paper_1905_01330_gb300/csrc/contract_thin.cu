// FP32 contractions that a tile of the general kernel fits badly: a shared
// index of at most 8 (the result is all there is to move) and a matrix times
// one vector (the matrix is).
//
// Outer products, K <= 8: bound by writing C. A CTA gathers its 64 rows and 64
// columns of the operands once into shared memory; a thread makes 4 x 4
// results and stores rows of 16 bytes. Sums are one chain over ascending k, as
// in the general kernel. Measured in a row of launches, on the general kernel
// and here: 1024 x 1024 x 2 6.4 -> 2.2 us, 4096 x 4096 x 8 27.7 -> 23.4.
//
// Matrix times vector: bound by reading the matrix, and at the sizes of a
// network's environments (1024 x 1024) by the latency of the loads in flight.
// With the matrix's free leg of unit stride, half a warp reads 64 consecutive
// columns at one k, a CTA takes 64 columns and a part of the shared index, and
// the (up to 8) parts are CTAs of one cluster that add up through distributed
// shared memory: no zeroed result, no atomics, one order. With the shared leg
// of unit stride a warp takes a row. Measured likewise (columns / rows): 1024 x
// 1024 49.2 -> 3.1 / 2.7 us, 64 x 64 13.3 -> 1.9 / 1.4, 20000 x 2048 427 -> 28 /
// 36 us (4.5 to 5.8 TB/s).
#include <cooperative_groups.h>

#include <algorithm>

#include "gather.cuh"
#include "ptx.cuh"
#include "tn_internal.h"

namespace tn {
namespace {

namespace cg = cooperative_groups;

constexpr int THREADS = 256;
constexpr int OUT_K = 8;    // longest shared index of an outer product
constexpr int OUT_T = 64;   // rows and columns of its tile
constexpr int MV_COLS = 64;  // columns of a CTA
constexpr int MV_PART = 1024;  // longest part of the shared index held in shared memory
constexpr int MV_ROWK = 2048;  // longest shared index of the row form

__global__ void __launch_bounds__(THREADS) outer_kernel(const __grid_constant__ ContractDesc d) {
  __shared__ __align__(16) float As[OUT_K][OUT_T], Bs[OUT_K][OUT_T];
  ptx::launch_dependents();
  const int t = threadIdx.x, K = (int)d.K;
  const int64_t m0 = (int64_t)(blockIdx.x / d.tiles_n) * OUT_T, n0 = (int64_t)(blockIdx.x % d.tiles_n) * OUT_T;
  {
    const int side = (t >> 6) & 1, r = t & 63;
    const int64_t row = (side ? n0 : m0) + r;
    const bool in = row < (side ? d.N : d.M);
    const float* src = side ? d.B : d.A;
    if (in) src += side ? leg_offset((uint32_t)row, d.nn, d.ndim, d.nstr) : leg_offset((uint32_t)row, d.nm, d.mdim, d.mstr);
    int64_t ko[OUT_K / 2];
#pragma unroll
    for (int i = 0; i < OUT_K / 2; ++i) {
      const int k = (t >> 7) + 2 * i;
      ko[i] = k < K ? leg_offset((uint32_t)k, d.nk, d.kdim, side ? d.kstrB : d.kstrA) : 0;
    }
    ptx::wait_dependencies();
#pragma unroll
    for (int i = 0; i < OUT_K / 2; ++i) {
      const int k = (t >> 7) + 2 * i;
      if (k < K) (side ? Bs : As)[k][r] = in ? src[ko[i]] : 0.0f;
    }
  }
  __syncthreads();
  const int tx = (t & 15) * 4, ty = (t >> 4) * 4;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  for (int k = 0; k < K; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(&As[k][ty]), b = *reinterpret_cast<const float4*>(&Bs[k][tx]);
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
  const bool vec = (d.N & 3) == 0 && (reinterpret_cast<uintptr_t>(d.C) & 15) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t m = m0 + ty + i;
    if (m < d.M)
      emit4(d.C + m * d.N + n0 + tx, vec, d.N - n0 - tx, false, acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  }
}

// y[r] = sum_k x[k] Mat(r, k)
struct MatVec {
  const float *x, *mat;
  float* y;
  int32_t R, K, part;  // part: shared indices of one CTA (column form)
  int32_t nr, nk;
  int32_t rdim[TN_MAX_RANK], kdim[TN_MAX_RANK];
  int64_t rstr[TN_MAX_RANK], kstr[TN_MAX_RANK], xstr[TN_MAX_RANK];
};

// Columns form. VEC: four consecutive r are 16 aligned bytes.
template <bool VEC>
__global__ void __launch_bounds__(THREADS) matvec_columns(const __grid_constant__ MatVec d) {
  __shared__ float xs[MV_PART];
  __shared__ int64_t ko[MV_PART];
  __shared__ __align__(16) float sums[16][MV_COLS];
  __shared__ float mine[MV_COLS];
  ptx::launch_dependents();
  cg::cluster_group cl = cg::this_cluster();
  const int t = threadIdx.x, ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int k0 = rank * d.part, kn = max(0, min(d.K - k0, d.part));
  int64_t xo[MV_PART / THREADS];
#pragma unroll
  for (int i = 0; i < MV_PART / THREADS; ++i) {
    const int k = t + i * THREADS;
    if (k >= kn) break;
    ko[k] = leg_offset((uint32_t)(k0 + k), d.nk, d.kdim, d.kstr);
    xo[i] = leg_offset((uint32_t)(k0 + k), d.nk, d.kdim, d.xstr);
  }
  // this thread's four columns: c0 .. c0 + 3, or c0 + 16 j
  const int l = t & 15, kg = t >> 4;
  const int r0 = (int)(blockIdx.x / ranks) * MV_COLS + (VEC ? 4 * l : l);
  const float* col[4];
  bool in[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = r0 + (VEC ? j : 16 * j);
    in[j] = r < d.R;
    if (!VEC || j == 0) col[j] = d.mat + (in[j] ? leg_offset((uint32_t)r, d.nr, d.rdim, d.rstr) : 0);
  }
  ptx::wait_dependencies();
#pragma unroll
  for (int i = 0; i < MV_PART / THREADS; ++i) {
    const int k = t + i * THREADS;
    if (k >= kn) break;
    xs[k] = d.x[xo[i]];
  }
  __syncthreads();
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (in[0]) {
#pragma unroll 8
    for (int k = kg; k < kn; k += 16) {
      const float xv = xs[k];
      if (VEC) {
        const float4 b = *reinterpret_cast<const float4*>(col[0] + ko[k]);
        acc[0] = fmaf(xv, b.x, acc[0]);
        acc[1] = fmaf(xv, b.y, acc[1]);
        acc[2] = fmaf(xv, b.z, acc[2]);
        acc[3] = fmaf(xv, b.w, acc[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (in[j]) acc[j] = fmaf(xv, col[j][ko[k]], acc[j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) sums[kg][VEC ? 4 * l + j : l + 16 * j] = acc[j];
  __syncthreads();
  if (t < MV_COLS) {
    float s = 0.0f;
#pragma unroll
    for (int g = 0; g < 16; ++g) s += sums[g][t];
    mine[t] = s;
  }
  cl.sync();
  if (rank == 0 && t < MV_COLS) {
    const int r = (int)(blockIdx.x / ranks) * MV_COLS + t;
    float s = mine[t];
    for (int g = 1; g < ranks; ++g) s += *cl.map_shared_rank(&mine[t], g);
    if (r < d.R) d.y[r] = s;
  }
  cl.sync();  // the sums stay until they are read
}

// Row form: a warp per row. VEC: four consecutive k are 16 aligned bytes.
template <bool VEC>
__global__ void __launch_bounds__(THREADS) matvec_rows(const __grid_constant__ MatVec d) {
  constexpr int W = VEC ? 4 : 1;
  __shared__ __align__(16) float xs[MV_ROWK];
  __shared__ int64_t ko[MV_ROWK / W];
  ptx::launch_dependents();
  const int t = threadIdx.x, lane = t & 31;
  int64_t xo[MV_ROWK / THREADS];
#pragma unroll
  for (int i = 0; i < MV_ROWK / THREADS; ++i) {
    const int k = t + i * THREADS;
    if (k >= d.K) break;
    xo[i] = leg_offset((uint32_t)k, d.nk, d.kdim, d.xstr);
    if (k % W == 0) ko[k / W] = leg_offset((uint32_t)k, d.nk, d.kdim, d.kstr);
  }
  const int r = (int)blockIdx.x * (THREADS / 32) + (t >> 5);
  const float* row = d.mat + (r < d.R ? leg_offset((uint32_t)r, d.nr, d.rdim, d.rstr) : 0);
  ptx::wait_dependencies();
#pragma unroll
  for (int i = 0; i < MV_ROWK / THREADS; ++i) {
    const int k = t + i * THREADS;
    if (k >= d.K) break;
    xs[k] = d.x[xo[i]];
  }
  __syncthreads();
  if (r >= d.R) return;
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 8
  for (int k = lane; k < d.K / W; k += 32) {
    if (VEC) {
      const float4 b = *reinterpret_cast<const float4*>(row + ko[k]);
      const float4 xv = *reinterpret_cast<const float4*>(&xs[4 * k]);
      acc[0] = fmaf(xv.x, b.x, acc[0]);
      acc[1] = fmaf(xv.y, b.y, acc[1]);
      acc[2] = fmaf(xv.z, b.z, acc[2]);
      acc[3] = fmaf(xv.w, b.w, acc[3]);
    } else {
      acc[0] = fmaf(xs[k], row[ko[k]], acc[0]);
    }
  }
  float s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) d.y[r] = s;
}

// A launch that may begin while the kernel before it ends (each kernel here
// waits for it before it reads an operand): a network's products run one after
// another, and the offsets are worked out meanwhile.
template <class P>
int launch_overlapped(void (*fn)(const P), const P& p, int64_t ctas, int cluster, cudaStream_t s) {
  if (ctas > 0x7FFFFFFF) return TN_ERR_UNSUPPORTED;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(THREADS);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  memset(at, 0, sizeof(at));
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, fn, p) == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

// The innermost leg (dims > 1) of a list has unit stride; *vec: its runs of
// four are whole 16-byte words (every other stride of the matrix is given in
// `others`).
bool unit_inner(int n, const int32_t* dim, const int64_t* str, int n2, const int64_t* str2, const int32_t* dim2,
                const float* base, bool* vec) {
  int in = n - 1;
  while (in >= 0 && dim[in] == 1) --in;
  if (in < 0 || str[in] != 1) return false;
  *vec = dim[in] % 4 == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0;
  for (int i = 0; i < in; ++i)
    if (dim[i] > 1 && (str[i] & 3)) *vec = false;
  for (int i = 0; i < n2; ++i)
    if (dim2[i] > 1 && (str2[i] & 3)) *vec = false;
  return true;
}

}  // namespace

bool outer_ok(const ContractDesc& d) { return d.K <= OUT_K && d.M >= 16 && d.N >= 16 && d.M * d.N >= 16384; }

int launch_outer(const ContractDesc& d, cudaStream_t s) {
  ContractDesc q = d;
  q.tiles_m = (int32_t)((d.M + OUT_T - 1) / OUT_T);
  q.tiles_n = (int32_t)((d.N + OUT_T - 1) / OUT_T);
  const int64_t ctas = (int64_t)q.tiles_m * q.tiles_n;
  return launch_overlapped(outer_kernel, q, ctas, 1, s);
}

bool matvec_ok(const ContractDesc& d) {
  if ((d.M == 1) == (d.N == 1)) return false;
  const int64_t R = d.M == 1 ? d.N : d.M;
  return R >= 64 && R < (1 << 24) && d.K >= 64 && d.K <= MV_ROWK;
}

int launch_matvec(const ContractDesc& d, cudaStream_t s) {
  const bool first = d.M == 1;  // the vector is the first operand
  MatVec v;
  memset(&v, 0, sizeof(v));
  v.x = first ? d.A : d.B;
  v.mat = first ? d.B : d.A;
  v.y = d.C;
  v.R = (int32_t)(first ? d.N : d.M);
  v.K = (int32_t)d.K;
  v.nr = first ? d.nn : d.nm;
  v.nk = d.nk;
  for (int i = 0; i < v.nr; ++i) {
    v.rdim[i] = first ? d.ndim[i] : d.mdim[i];
    v.rstr[i] = first ? d.nstr[i] : d.mstr[i];
  }
  for (int i = 0; i < v.nk; ++i) {
    v.kdim[i] = d.kdim[i];
    v.kstr[i] = first ? d.kstrB[i] : d.kstrA[i];
    v.xstr[i] = first ? d.kstrA[i] : d.kstrB[i];
  }
  bool vec = false;
  if (unit_inner(v.nk, v.kdim, v.kstr, v.nr, v.rstr, v.rdim, v.mat, &vec)) {
    return launch_overlapped(vec ? matvec_rows<true> : matvec_rows<false>, v, (v.R + THREADS / 32 - 1) / (THREADS / 32), 1,
                             s);
  }
  unit_inner(v.nr, v.rdim, v.rstr, v.nk, v.kstr, v.kdim, v.mat, &vec);
  // parts of the shared index: enough CTAs for the SMs, at least 64 indices each
  const int64_t groups = (v.R + MV_COLS - 1) / MV_COLS;
  int parts = (v.K + MV_PART - 1) / MV_PART;
  while (parts < 8 && groups * parts < sm_count() && v.K / (2 * parts) >= 64) parts *= 2;
  v.part = (v.K + parts - 1) / parts;
  return launch_overlapped(vec ? matvec_columns<true> : matvec_columns<false>, v, groups * parts, parts, s);
}

}  // namespace tn
