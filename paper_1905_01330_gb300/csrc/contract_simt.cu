// FP32 pairwise tensordot on the CUDA cores (exact float32 FMA path).
//
// C[m, n] = sum_k A(m, k) B(k, n) over the flattened shared legs
// (Sec. III.B.2 / III.B.4). Operands are gathered in place through their leg
// strides (no transposed copy): per output tile, row offsets of A's free legs
// and column offsets of B's free legs are decoded once, and the offsets of
// each 16-wide slab of shared indices are decoded into a small shared-memory
// table one slab ahead. An operand whose unit-stride leg lets four
// neighbours along the rows or along k be loaded at once (plan_simt) is
// gathered in 16-byte loads, else element by element.
//
// What bounds it: the FMA pipe when the tile fits the contraction. A loop of
// shared-memory reads and FMAs alone reaches 65 TFLOP/s; with the gather, its
// index arithmetic and a barrier per slab in the same warps the kernel stayed
// at 37-38 whatever the register tile. So a CTA has four warps that only
// multiply and four that only gather: the gather warps keep two slabs of
// loads in flight and fill a ring of slabs in shared memory, in the issue
// slots that packed FMAs (two cycles each) leave free; two CTAs share an SM,
// so one's prologue and epilogue run beside the other's products. A
// multiplying warp's 32 threads lie along the columns and share its rows: a
// row operand is one broadcast. Three tile shapes (64, 32 and 32 accumulators
// a thread, packed pairs along the rows) cover square and thin contractions,
// the longer side on the tile's columns whichever operand it belongs to (C's
// element order follows): on 256 random specs (2.3e11 flop) a 128 x 128 tile
// alone spends 1.56 of the work on padding. Every sum runs over ascending k
// in one chain of float32 FMAs per chunk (at most 2048 shared indices); the
// chunks of a unit are added up in shared memory.
// Measured (TFLOP/s before -> now): 4096^3 with rows contiguous 37.9 -> 55.3,
// k contiguous 37.5 -> 40.5, odd sizes 37.5 -> 45; 256 random specs 10.09 ->
// 6.1 ms; 2048 x 1024 x 512 81 -> 60 us.
#include <algorithm>
#include <utility>

#include "gather.cuh"
#include "ptx.cuh"

namespace tn {
namespace {

constexpr int BK = 16;
constexpr int NW = 4;                    // multiplying warps
constexpr int NT = 128;                  // gathering threads (the same number of warps)
constexpr int THREADS = 32 * NW + NT;
constexpr int STAGES = 4;

template <int TM_, int TN_>
struct Tile {
  static constexpr int TM = TM_, TN = TN_, BM = NW * TM, BN = 32 * TN;
  static constexpr int AS = BM + 4, BS = BN + 4;  // row strides: 16-byte aligned, 4 rows 16 banks apart
  static constexpr int STAGE = BK * (AS + BS);    // floats
};
using Tile0 = Tile<16, 4>;  // 64 x 128
using Tile1 = Tile<8, 4>;   // 32 x 128
using Tile2 = Tile<4, 8>;   // 16 x 256
// Ring, and per multiplying warp a region for its part of the result tile:
// the sums of a unit's finished chunks, then the rows on their way to C (4
// floats of padding a row).
template <class T>
constexpr size_t smem_bytes() {
  return sizeof(float) * (STAGES * (size_t)T::STAGE + NW * (size_t)T::TM * (T::BN + 4));
}
constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }
constexpr size_t SMEM_BYTES = cmax(smem_bytes<Tile0>(), cmax(smem_bytes<Tile1>(), smem_bytes<Tile2>()));

struct SimtSmem {
  int32_t row[128];
  int32_t col[256];
  int32_t kA[2][NT];   // offsets of NT shared indices, two tables in turn
  int32_t kB[2][NT];
  uint32_t rec[3][TN_MAX_RANK];  // 2^32 / dimension of the legs of m, n, k
  uint64_t full[STAGES], empty[STAGES];
  ContractDesc d;
  UnitCoord uc;
  int idx;
};

// Quotient by d of n < 2^31, with r = 2^32 / d rounded down: the estimate is
// the quotient or one less.
__device__ __forceinline__ uint32_t div_by(uint32_t n, uint32_t d, uint32_t r) {
  const uint32_t q = __umulhi(n, r);
  return q + (n - q * d >= d ? 1u : 0u);
}

// Offset of composite index idx over legs (dims, strides, reciprocals).
__device__ __forceinline__ int32_t leg_offset_by(uint32_t idx, int n, const int32_t* dims, const uint32_t* rec,
                                                 const int64_t* strides) {
  int64_t off = 0;
  for (int q = n - 1; q >= 0; --q) {
    const uint32_t d = (uint32_t)dims[q], hi = div_by(idx, d, rec[q]);
    off += (int64_t)(idx - hi * d) * strides[q];
    idx = hi;
  }
  return (int32_t)off;
}

// Offsets in A and B of the KT shared indices from k0 (-1 past the range),
// one per gathering thread.
__device__ __forceinline__ void fill_k(SimtSmem& s, int t, int buf, int64_t k0, int64_t k_end) {
  int64_t oa = -1, ob = -1;
  if (k0 + t < k_end) {
    uint32_t idx = (uint32_t)(k0 + t);
    oa = ob = 0;
    for (int q = s.d.nk - 1; q >= 0; --q) {
      const uint32_t d = (uint32_t)s.d.kdim[q], hi = div_by(idx, d, s.rec[2][q]), digit = idx - hi * d;
      oa += (int64_t)digit * s.d.kstrA[q];
      ob += (int64_t)digit * s.d.kstrB[q];
      idx = hi;
    }
  }
  s.kA[buf][t] = (int32_t)oa;
  s.kB[buf][t] = (int32_t)ob;
}

// Loads that give zeros for a negative offset, without a branch (the loads of
// a slab issue back to back).
__device__ __forceinline__ float4 ld4_or0(const float* X, int32_t off) {
  float4 f;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %5, 0;\n\t"
      "mov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
      "@p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=&f"(f.x), "=&f"(f.y), "=&f"(f.z), "=&f"(f.w)
      : "l"(X + off), "r"(off));
  return f;
}
__device__ __forceinline__ float ld1_or0(const float* X, int32_t off) {
  float f;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ge.s32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t"
      "@p ld.global.nc.f32 %0, [%1];\n\t}"
      : "=&f"(f)
      : "l"(X + off), "r"(off));
  return f;
}
// Sum of two offsets, negative if either is (offsets are below 2^31).
__device__ __forceinline__ int32_t off_sum(int32_t a, int32_t b) { return (a | b) < 0 ? -1 : a + b; }

// One operand's slab, R rows x 16 k, global -> registers -> shared [k][r].
// Thread's elements: along rows (4 rows of one k), along k (4 k of one row;
// a half-warp's 16 rows, so the transposing stores are free of conflicts) or
// single ones.
template <int R>
struct Slab {
  static constexpr int NV = R * 4 > NT ? R * 4 / NT : 1;  // 16-byte loads a thread
  static constexpr int NE = R * BK / NT;                  // single elements a thread
  float r[4 * NV];

  __device__ __forceinline__ void load(int t, const float* __restrict__ X, const int32_t* rows, const int32_t* ks,
                                       bool kfast, bool vec) {
    if (vec) {
      int32_t off[NV];
      if (kfast) {
        const int32_t ko = ks[((t >> 5) & 1) * 8 + ((t >> 4) & 1) * 4];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int i = t + NT * v;
          off[v] = (R * 4 >= NT || i < R * 4) ? off_sum(ko, rows[(i >> 6) * 16 + (i & 15)]) : -1;
        }
      } else {
        const int32_t ro = rows[(t % (R / 4)) * 4];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int i = t + NT * v;
          off[v] = (R * 4 >= NT || i < R * 4) ? off_sum(ro, ks[i / (R / 4)]) : -1;
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float4 f = ld4_or0(X, off[v]);
        r[4 * v] = f.x;
        r[4 * v + 1] = f.y;
        r[4 * v + 2] = f.z;
        r[4 * v + 3] = f.w;
      }
    } else if (kfast) {
      const int32_t ko = ks[t & (BK - 1)];
#pragma unroll
      for (int e = 0; e < NE; ++e) r[e] = ld1_or0(X, off_sum(ko, rows[(t >> 4) + NT / BK * e]));
    } else {
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const int i = t + NT * e;
        r[e] = ld1_or0(X, off_sum(rows[i % R], ks[i / R]));
      }
    }
  }

  __device__ __forceinline__ void store(int t, float* x, bool kfast, bool vec) const {
    constexpr int S = R + 4;
    if (vec) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int i = t + NT * v;
        if (R * 4 >= NT || i < R * 4) {
          if (kfast) {
            const int rr = (i >> 6) * 16 + (i & 15), k = ((i >> 5) & 1) * 8 + ((i >> 4) & 1) * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) x[(k + j) * S + rr] = r[4 * v + j];
          } else {
            const int rr = (i % (R / 4)) * 4, k = i / (R / 4);
            *reinterpret_cast<float4*>(x + k * S + rr) = make_float4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
          }
        }
      }
    } else {
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const int i = t + NT * e;
        if (kfast) x[(i & (BK - 1)) * S + (i >> 4)] = r[e];
        else x[(i / R) * S + i % R] = r[e];
      }
    }
  }
};

// Gathering warps: every slab of the unit's `subs` tiles (rows m0 + sub BM)
// into the ring; two slabs of loads in flight per thread.
template <class T>
__device__ __forceinline__ void gather(SimtSmem& s, float* ring, int subs, int* status) {
  const int t = threadIdx.x - 32 * NW;
  const float* __restrict__ A = s.d.A;
  const float* __restrict__ B = s.d.B;
  const bool akf = s.d.a_kfast != 0, bkf = s.d.b_kfast != 0, av = (s.d.vec & 1) != 0, bv = (s.d.vec & 2) != 0;
  const int64_t kb = s.uc.k_begin, ke = s.uc.k_end;
  const int nkt = (int)((ke - kb + BK - 1) / BK), total = nkt * subs;
  Slab<T::BM> ra[2];
  Slab<T::BN> rb[2];
  constexpr int KS = NT / BK;  // slabs per offset table
  fill_k(s, t, 0, kb, ke);
  ptx::named_barrier(1, NT);
  // slab g is loaded in round g and stored in round g + 1
  int kt = 0, sub = 0, tab = 0;  // of slab g: position in the k range, tile, offset table
  bool bad = false;              // a wait expired: no more stores, to the end in step with the other warps
  auto round = [&](int g, Slab<T::BM>& la, Slab<T::BN>& lb, const Slab<T::BM>& pa, const Slab<T::BN>& pb) {
    if (g < total) {
      la.load(t, A, s.row + sub * T::BM, s.kA[tab] + (kt % KS) * BK, akf, av);
      lb.load(t, B, s.col, s.kB[tab] + (kt % KS) * BK, bkf, bv);
    }
    if (g > 0) {
      const int st = (g - 1) % STAGES, use = (g - 1) / STAGES;
      if (use > 0 && !bad) bad = !ptx::mbar_wait(ptx::smem_addr(&s.empty[st]), (use - 1) & 1, status);
      if (!bad) {
        float* x = ring + st * T::STAGE;
        pa.store(t, x, akf, av);
        pb.store(t, x + BK * T::AS, bkf, bv);
      }
      __syncwarp();
      if ((t & 31) == 0) ptx::mbar_arrive(ptx::smem_addr(&s.full[st]));
    }
    if (++kt == nkt) {
      kt = 0;
      ++sub;
    }
    if (kt % KS == 0 && g + 1 < total) {  // the next offsets, into the table two tables back
      tab ^= 1;
      fill_k(s, t, tab, kb + (int64_t)kt * BK, ke);
      bad = ptx::named_barrier_or(1, NT, bad);
    }
  };
  for (int g = 0; g <= total; g += 2) {
    round(g, ra[0], rb[0], ra[1], rb[1]);
    if (g < total) round(g + 1, ra[1], rb[1], ra[0], rb[0]);
  }
}

// Multiplying warps: warp w's rows w TM .. of the tile, thread's columns
// 4 lane .. (+ 128 for the 256-wide tile).
template <class T>
__device__ __forceinline__ void multiply(SimtSmem& s, float* ring, int subs, int* status) {
  constexpr int TM = T::TM, TN = T::TN;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int RS = T::BN + 4;
  float* part = ring + STAGES * T::STAGE + w * TM * RS;
  float4* sums = reinterpret_cast<float4*>(part) + lane;  // [TM TN / 4][32]
  const int64_t chunk = (int64_t)s.d.chunk * 64;
  const int64_t n0 = s.uc.n0;
  int it = 0;  // slabs consumed
  for (int sub = 0; sub < subs; ++sub) {
    const int64_t m0 = s.uc.m0 + (int64_t)sub * T::BM;
    for (int64_t kc = s.uc.k_begin; kc < s.uc.k_end; kc += chunk) {
      const int64_t ke = min(s.uc.k_end, kc + chunk);
      const int nkt = (int)((ke - kc + BK - 1) / BK);
      float2 acc[TM / 2][TN];
#pragma unroll
      for (int i = 0; i < TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = make_float2(0.f, 0.f);
      for (int kt = 0; kt < nkt; ++kt, ++it) {
        const int st = it % STAGES;
        if (!__all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_addr(&s.full[st]), (it / STAGES) & 1, status))) return;
        const float* as = ring + st * T::STAGE + w * TM;
        const float* bs = ring + st * T::STAGE + BK * T::AS + lane * 4;
#pragma unroll
        for (int k = 0; k < BK; ++k) {
          float2 a[TM / 2];
          float b[TN];
#pragma unroll
          for (int g = 0; g < TM / 4; ++g) {
            const float4 f = *reinterpret_cast<const float4*>(as + k * T::AS + g * 4);
            a[2 * g] = make_float2(f.x, f.y);
            a[2 * g + 1] = make_float2(f.z, f.w);
          }
#pragma unroll
          for (int g = 0; g < TN / 4; ++g) {
            const float4 f = *reinterpret_cast<const float4*>(bs + k * T::BS + g * 128);
            b[4 * g] = f.x;
            b[4 * g + 1] = f.y;
            b[4 * g + 2] = f.z;
            b[4 * g + 3] = f.w;
          }
#pragma unroll
          for (int j = 0; j < TN; ++j) {
            const float2 bb = make_float2(b[j], b[j]);
#pragma unroll
            for (int i = 0; i < TM / 2; ++i) acc[i][j] = __ffma2_rn(a[i], bb, acc[i][j]);
          }
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&s.empty[st]));
      }
      if (kc > s.uc.k_begin) {
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
          for (int j = 0; j < TN; j += 2) {
            const float4 f = sums[(i * TN + j) / 2 * 32];
            acc[i][j] = make_float2(f.x + acc[i][j].x, f.y + acc[i][j].y);
            acc[i][j + 1] = make_float2(f.z + acc[i][j + 1].x, f.w + acc[i][j + 1].y);
          }
        __syncwarp();  // the rows below lie over other lanes' sums
      }
      if (ke < s.uc.k_end) {
#pragma unroll
        for (int i = 0; i < TM / 2; ++i)
#pragma unroll
          for (int j = 0; j < TN; j += 2)
            sums[(i * TN + j) / 2 * 32] = make_float4(acc[i][j].x, acc[i][j].y, acc[i][j + 1].x, acc[i][j + 1].y);
        continue;
      }
      // through shared memory, so that the code that reaches C is a short
      // loop (unrolled over the accumulators it took 7,000 cycles a tile, most
      // of them instruction fetches)
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int g = 0; g < TN / 4; ++g) {
          const float2 v0 = acc[i >> 1][4 * g], v1 = acc[i >> 1][4 * g + 1], v2 = acc[i >> 1][4 * g + 2],
                       v3 = acc[i >> 1][4 * g + 3];
          *reinterpret_cast<float4*>(part + i * RS + g * 128 + lane * 4) =
              i & 1 ? make_float4(v0.y, v1.y, v2.y, v3.y) : make_float4(v0.x, v1.x, v2.x, v3.x);
        }
      __syncwarp();
      float* __restrict__ C = s.d.C;
      const int64_t M = s.d.M, N = s.d.N, mw = m0 + w * TM;
      const bool atomic = s.d.splits > 1, aligned = (reinterpret_cast<uintptr_t>(C) & 15) == 0;
      if (!s.d.swapped) {  // C[m][n]: a row's four columns at once
        const bool vec = ((N & 3) == 0) && aligned;
        const int rows = (int)min((int64_t)TM, M - mw);
#pragma unroll 2
        for (int q = 0; q < rows * (T::BN / 128); ++q) {
          const int r = q / (T::BN / 128), c = q % (T::BN / 128) * 128 + lane * 4;
          const float4 f = *reinterpret_cast<const float4*>(part + r * RS + c);
          if (n0 + c < N) emit4(C + (mw + r) * N + n0 + c, vec, N - n0 - c, atomic, f.x, f.y, f.z, f.w);
        }
      } else {  // C[n][m]: a column's four rows at once
        const bool vec = ((M & 3) == 0) && aligned;
        constexpr int QL = TM / 4, CP = 32 / QL;  // lanes along the rows, columns a pass
        const int r = lane % QL * 4;
        const int64_t left = M - mw - r;
#pragma unroll 2
        for (int c = lane / QL; c < T::BN; c += CP) {
          const float* x = part + r * RS + c;
          if (n0 + c < N && left > 0) emit4(C + (n0 + c) * M + mw + r, vec, left, atomic, x[0], x[RS], x[2 * RS], x[3 * RS]);
        }
      }
      __syncwarp();  // the region is free for the next tile
    }
  }
}

template <class T>
__device__ __forceinline__ void run_unit(SimtSmem& s, float* ring, int subs, int* status) {
  if (threadIdx.x < 32 * NW) multiply<T>(s, ring, subs, status);
  else gather<T>(s, ring, subs, status);
}

__global__ void __launch_bounds__(THREADS, 2)
simt_contract_kernel(const __grid_constant__ ContractDesc single, const ContractDesc* group,
                     const int32_t* unit_desc, int* status) {
  extern __shared__ __align__(16) float ring[];
  __shared__ __align__(16) SimtSmem s;
  const int t = threadIdx.x;
  const int64_t unit = fetch_desc(single, group, unit_desc, (int64_t)blockIdx.x, &s.d, &s.idx);
  const int tm = simt_tile_m(s.d.tile), tn = simt_tile_n(s.d.tile);
  if (t == 0) {
    for (int i = 0; i < STAGES; ++i) {
      ptx::mbar_init(ptx::smem_addr(&s.full[i]), NT / 32);
      ptx::mbar_init(ptx::smem_addr(&s.empty[i]), NW);
    }
    ptx::fence_mbar_init();
  }
  // unit = (split, tile row, tile column), below 2^31
  const uint32_t u = (uint32_t)unit, un = u / (uint32_t)s.d.tiles_n, us = un / (uint32_t)s.d.tiles_m;
  const int64_t m0 = (int64_t)(un - us * s.d.tiles_m) * tm, n0 = (int64_t)(u - un * s.d.tiles_n) * tn;
  if (t == 32) {
    s.uc.m0 = m0;
    s.uc.n0 = n0;
    s.uc.k_begin = us * s.d.k_per_split;
    s.uc.k_end = min(s.d.K, s.uc.k_begin + s.d.k_per_split);
  }
  if (t >= 64 && t < 64 + 3 * TN_MAX_RANK) {
    const int l = (t - 64) / TN_MAX_RANK, q = (t - 64) % TN_MAX_RANK;
    const int32_t* dims = l == 0 ? s.d.mdim : (l == 1 ? s.d.ndim : s.d.kdim);
    if (q < (l == 0 ? s.d.nm : (l == 1 ? s.d.nn : s.d.nk)))
      s.rec[l][q] = dims[q] > 1 ? (uint32_t)(0x100000000ull / (uint32_t)dims[q]) : 0xffffffffu;
  }
  __syncthreads();
  for (int i = t; i < tm; i += THREADS)
    s.row[i] = (m0 + i < s.d.M) ? leg_offset_by((uint32_t)(m0 + i), s.d.nm, s.d.mdim, s.rec[0], s.d.mstr) : -1;
  for (int i = t; i < tn; i += THREADS)
    s.col[i] = (n0 + i < s.d.N) ? leg_offset_by((uint32_t)(n0 + i), s.d.nn, s.d.ndim, s.rec[1], s.d.nstr) : -1;
  __syncthreads();
  if (s.d.tile == 1) run_unit<Tile1>(s, ring, 1, status);
  else if (s.d.tile == 2) run_unit<Tile2>(s, ring, 1, status);
  else run_unit<Tile0>(s, ring, s.d.tile == SIMT_TILE_PAIR && s.uc.m0 + Tile0::BM < s.d.M ? 2 : 1, status);
}

// Zeroes the ranges; blockIdx.y shares out a range (a multiple of 4 elements
// each, so only the first part has an unaligned head).
__global__ void zero_kernel(const ZeroRange* ranges) {
  const ZeroRange r = ranges[blockIdx.x];
  const int64_t part = ((r.count + gridDim.y - 1) / gridDim.y + 3) / 4 * 4, first = part * blockIdx.y;
  if (first >= r.count) return;
  float* p = r.ptr + first;
  const int64_t n = min(part, r.count - first);
  int64_t head = 0;
  while (head < n && (reinterpret_cast<uintptr_t>(p + head) & 15) != 0) ++head;
  for (int64_t i = threadIdx.x; i < head; i += blockDim.x) p[i] = 0.0f;
  const int64_t nv = (n - head) / 4;
  float4* q = reinterpret_cast<float4*>(p + head);
  for (int64_t i = threadIdx.x; i < nv; i += blockDim.x) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t i = head + nv * 4 + threadIdx.x; i < n; i += blockDim.x) p[i] = 0.0f;
}

// Whether four neighbours of an operand along its fast direction (the
// innermost free leg, or the innermost shared one) are always one aligned
// 16-byte load: unit stride, an extent that is a multiple of 4, every other
// stride a multiple of 4 elements.
bool vector_gather(const float* X, bool kfast, int nr, const int32_t* rdim, const int64_t* rstr, int nk,
                   const int32_t* kdim, const int64_t* kstr) {
  if (reinterpret_cast<uintptr_t>(X) & 15) return false;
  const int n = kfast ? nk : nr;
  if (n < 1) return false;
  const int32_t* fd = kfast ? kdim : rdim;
  const int64_t* fs = kfast ? kstr : rstr;
  if (fs[n - 1] != 1 || fd[n - 1] % 4 != 0) return false;
  for (int i = 0; i < nr; ++i)
    if (!(!kfast && i == nr - 1) && rdim[i] > 1 && rstr[i] % 4 != 0) return false;
  for (int i = 0; i < nk; ++i)
    if (!(kfast && i == nk - 1) && kdim[i] > 1 && kstr[i] % 4 != 0) return false;
  return true;
}

}  // namespace

void plan_simt(ContractDesc* d, SimtPlan how, int chains) {
  // A unit's chain lengths are those of the k ranges plan_units gave; a lone
  // contraction may run several of them in one unit.
  const int64_t slabs = (d->K + 63) / 64, chunk = d->k_per_split < 2048 ? d->k_per_split / 64 : 32;
  d->chunk = (int16_t)chunk;
  int tile = SIMT_TILE_PAIR, swap = 0;
  int64_t per = std::min<int64_t>(chains, d->splits) * d->k_per_split;
  if (how != SimtPlan::pairs) {
    // cycles of a 16-wide slab (two CTAs an SM), measured at 2048^3 and, for
    // the thin tiles, in proportion to their FMAs and shared-memory reads
    static const double slab[SIMT_TILES] = {1000.0, 620.0, 680.0};
    double best = -1.0;
    for (int s = 0; s < 2; ++s)
      for (int k = 0; k < SIMT_TILES; ++k) {
        const int64_t bm = simt_tile_m(k), bn = simt_tile_n(k), M = s ? d->N : d->M, N = s ? d->M : d->N;
        const int64_t tiles = ((M + bm - 1) / bm) * ((N + bn - 1) / bn);
        if (how == SimtPlan::group) {  // many contractions share the GPU: the padded work decides
          const double c = (double)tiles * slab[k];
          if (best < 0.0 || c < best) {
            best = c;
            tile = k;
            swap = s;
          }
          continue;
        }
        // alone: units per SM (two at a time) times a unit's slabs and its
        // start and end; more than one k range costs a zeroing pass. Chunks of
        // a unit: every count to 8, then steps of a quarter (all counts of a
        // shared index of 1e8 took 2.1 ms on the host), and all of them. In a
        // sweep one or all, so that a result is the sum of the k ranges one by
        // one, in whatever order.
        const int64_t most = d->splits, sms = sm_count();
        for (int64_t c = 1, next; c <= most; c = next) {
          next = c == most ? most + 1 : std::min(most, how == SimtPlan::sweep ? most : c + 1 + (c >= 8 ? c / 4 : 0));
          const int64_t sp = (slabs + c * chunk - 1) / (c * chunk), u = (tiles * sp + sms - 1) / sms;
          double t = (double)((u + 1) / 2) * 8000.0 +
                     (double)u * (double)(4 * std::min(slabs, c * chunk)) * slab[k] + (sp > 1 ? 6000.0 : 0.0);
          // two addends commute, more make a result vary from run to run: not
          // in a sweep of 16 tiles or more, and alone not for nothing (885 x
          // 150 x 2862 held to two: 91 us, 64 with three; before tiles of this
          // kind 66)
          if (sp > 2 && tiles >= 16) {
            if (how == SimtPlan::sweep) continue;
            t *= 1.005;
          }
          if (best < 0.0 || t < best) {
            best = t;
            tile = k;
            swap = s;
            per = c * chunk * 64;
          }
        }
      }
  }
  d->k_per_split = per;
  d->splits = (int32_t)((d->K + per - 1) / per);
  if (swap) {
    std::swap(d->A, d->B);
    std::swap(d->M, d->N);
    std::swap(d->nm, d->nn);
    std::swap(d->a_kfast, d->b_kfast);
    for (int i = 0; i < TN_MAX_RANK; ++i) {
      std::swap(d->mdim[i], d->ndim[i]);
      std::swap(d->mstr[i], d->nstr[i]);
      std::swap(d->kstrA[i], d->kstrB[i]);
    }
  }
  d->swapped = swap;
  d->tile = tile;
  d->tiles_m = (int32_t)((d->M + simt_tile_m(tile) - 1) / simt_tile_m(tile));
  d->tiles_n = (int32_t)((d->N + simt_tile_n(tile) - 1) / simt_tile_n(tile));
  d->vec = (vector_gather(d->A, d->a_kfast != 0, d->nm, d->mdim, d->mstr, d->nk, d->kdim, d->kstrA) ? 1 : 0) |
           (vector_gather(d->B, d->b_kfast != 0, d->nn, d->ndim, d->nstr, d->nk, d->kdim, d->kstrB) ? 2 : 0);
}

int launch_zero(const ZeroRange* ranges, int n, cudaStream_t stream) {
  if (n <= 0) return TN_OK;
  // a range of megabytes over 16 CTAs (one alone took 322 us on 256 specs)
  zero_kernel<<<dim3((unsigned)n, 16), 512, 0, stream>>>(ranges);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

int launch_contract_simt(const ContractDesc& single, const ContractDesc* group, const int32_t* unit_desc,
                         int64_t total_tiles, cudaStream_t stream) {
  if (total_tiles <= 0) return TN_OK;
  if (total_tiles > 0x7FFFFFFF) return TN_ERR_UNSUPPORTED;
  if (group && !unit_desc) return TN_ERR_ARG;
  static std::atomic<uint64_t> attr{0};
  if (!smem_limit_once((const void*)simt_contract_kernel, SMEM_BYTES, &attr)) return TN_ERR_CUDA;
  simt_contract_kernel<<<(unsigned)total_tiles, THREADS, SMEM_BYTES, stream>>>(single, group, unit_desc, status_word());
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

}  // namespace tn
