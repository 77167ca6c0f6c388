// MPS classifier sweeps on the tcgen05 tensor cores: the BF16 and split
// BF16x3 paths of tn_mps_classify / tn_mps_classify_backward (Sec. IV.A).
//
// Forward step of a half-chain for a tile of 128 samples b, with the site's
// core seen as L[k, s, j] (k the incoming bond, j the outgoing one):
//     U[b, (s, j)] = sum_k v_b[k] L[k, s, j]             (M = 128, N = 2 chi, K = chi)
//     u_b[j] = Phi_0(x_b) U[b, (0, j)] + Phi_1(x_b) U[b, (1, j)]
// then u_b is scaled by 2^-e_b, e_b the binary exponent of max_j |u_b[j]|
// (so the largest magnitude lands in [1/2, 1)), and e_b ln 2 is added to the
// sample's log-scale. A power of two keeps the scaling exact: the scaled
// vector and its bf16 rounding are the unscaled ones with a shifted exponent.
//
// Adjoint step (walking back from the label core), with g the adjoint of the
// vector leaving the step and sc_b = 2^e_b the forward's scale:
//     x_b[(s, j)] = Phi_s(x_b) g_b[j] / sc_b
//     g'_b[k] = sum_{(s, j)} x_b[(s, j)] L[k, s, j]        (M = 128, N = chi, K = 2 chi)
//     dL[k, s, j] += sum_b v_b[k] x_b[(s, j)]              (M = 2 chi, N = chi, K = 128)
// with v_b the forward vector entering the step. The gradient product runs in
// the same CTA on the same staged x (the 128-byte-swizzled K-major x tile of
// the first product is the MN-major operand of the second) and the v tile the
// recomputing forward wrote, and is added to the step's float32 gradient with
// coalesced reductions (one 128-byte line per warp instruction).
//
// Split BF16x3 (Henry, Tang and Heinecke, ARITH 2019): every operand is
// hi = bf16(x) plus lo = bf16(x - hi) and each product is hi*hi + lo*hi +
// hi*lo in the float32 accumulator.
//
// One launch covers both half-chains (CTA = (half, tile)). A CTA has NG
// epilogue threads per sample (thread r owns TMEM lane r % 128 and its group's
// columns), one producer warp that streams the packed core slabs (and, in the
// adjoint, the v tiles) into shared-memory rings with 1-D bulk async copies,
// and one warp that issues the MMAs.
//
// What bounds it: a step is a chain, MMAs, accumulator, mixing, splitting,
// shared memory, MMAs, and nothing else of the tile can run meanwhile (a
// second tile's operands do not fit beside the first's). So the MMA warp does
// nothing else (with an epilogue thread as issuer, which the tensor pipe's
// short queue holds until its last MMAs run, that thread's own part of the
// step came after the MMAs: 6,500 cycles a step of which the MMAs are 3,070
// at chi = 128); the exchange of the scales runs while the MMAs do; at chi =
// 128 the forward step's columns are two halves, so that the first half's
// epilogue and the next step's MMAs on it run beside the second half's; and
// the adjoint's epilogue works on g' while the gradient product runs.
// Measured (4096 samples, 784 sites, split BF16x3; before -> now): forward chi
// = 128 1117 -> 783 us, chi = 64 with recomputation 1435 -> 1056 us, adjoint
// chi = 64 1425 -> 957 us; those two then side by side (cls_pair_tc, 14 segments) 2010 -> 1190 us.
// Every mbarrier wait is bounded; a CTA that gives up records
// TN_ERR_TIMEOUT, lets its copies land, frees its TMEM and returns.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "classifier_tc.h"
#include "ptx.cuh"

namespace tn {
namespace {

constexpr int TS = CLS_TILE;         // samples per tile
constexpr int PXS = 16;              // steps of pixels staged at once
constexpr int SLAB_V = TS * 128;     // one 64-column slab of a 128-row tile (bytes)
constexpr int SMEM_BUDGET = 200 * 1024;

constexpr int pow2ceil(int x) {
  int p = 32;
  while (p < x) p *= 2;
  return p;
}

template <int CHI, int SPLIT>
struct Cfg {
  static constexpr int PARTS = SPLIT ? 2 : 1;
  static constexpr int KPAD = CHI < 64 ? 64 : CHI;  // sweep vector, padded to whole slabs
  static constexpr int KSL = KPAD / 64;
  static constexpr int VT = KSL * SLAB_V;           // one part of a vector tile
  static constexpr int VTS = VT * PARTS;
  static constexpr int NG = CHI >= 64 ? 4 : 2;      // epilogue threads per sample
  static constexpr int NEPI = NG * TS;
  static constexpr int NTHREADS = NEPI + 96;        // + producer, MMA and (forward) vector-image store warps
  static constexpr int HC = CHI / NG;               // columns per epilogue thread
  // forward: image rows (j / (CHI / NH), s, j % (CHI / NH)), K = k; NH column
  // halves, each with its own accumulator, blocks (k slab, half) in this order
  static constexpr int NH = CHI == 128 ? 2 : 1;
  static constexpr int FN = 2 * CHI / NH;
  static constexpr int FSLAB = FN * 128;
  static constexpr int FSET = FSLAB * PARTS;
  static constexpr int FRING_RAW = (SMEM_BUDGET - VTS) / FSET;
  static constexpr int FRING = FRING_RAW > 8 ? 8 : FRING_RAW;
  static constexpr int VCOL = 2 * CHI;              // TMEM columns of the vector: part p at VCOL + p KPAD / 2
  static constexpr uint32_t FCOLS = (uint32_t)pow2ceil(VCOL + PARTS * KPAD / 2);
  // adjoint: x tile rows b, columns m = (s, j); image rows k, K = m
  static constexpr int XSL = 2 * CHI / 64;
  static constexpr int XPART = (XSL + (CHI == 32 ? 1 : 0)) * SLAB_V;  // + a zero M half at chi = 32
  static constexpr int XTS = XPART * PARTS;
  static constexpr int ASLAB = CHI * 128;
  static constexpr int ASET = ASLAB * PARTS;
  static constexpr int MH = (2 * CHI + 127) / 128;  // M halves of the gradient product
  static constexpr int ARING_RAW = (SMEM_BUDGET - XTS - 2 * VTS) / ASET;
  static constexpr int ARING = ARING_RAW > 8 ? 8 : ARING_RAW;
  static constexpr int A2OFF = CHI < 64 ? 64 : CHI;  // TMEM column of the gradient accumulator
  // two gradient accumulators when they fit (step q's is drained while step
  // q + 1's products run), else one
  static constexpr int A2BUF = A2OFF + 2 * MH * KPAD + PARTS * CHI <= 512 ? 2 : 1;
  static constexpr int XCOL = A2OFF + A2BUF * MH * KPAD;  // x in TMEM: part p at XCOL + p CHI
  static constexpr uint32_t ACOLS = (uint32_t)pow2ceil(XCOL + PARTS * CHI);
};

struct __align__(8) Bars {
  uint64_t full[8];
  uint64_t empty[8];
  uint64_t vfull[2];
  uint64_t vempty[2];
  uint64_t acc_full[2];  // forward: a half's accumulator is complete; adjoint: g', the gradient
  uint64_t ready[2];     // the next step's operand is written (forward at chi = 128: its k slabs)
  uint64_t drained;      // the second half's accumulator has been read
  uint64_t image;        // forward: the vector's image for the gradients is written
  uint64_t stored;       // and its copy to device memory has been read out
  uint64_t final_bar;
  uint32_t tmem_base;
  int32_t abort;
};

struct StageTail {
  float2 phi[PXS][TS];
  float pmax[2][4][TS];
  Bars bars;
};

// K-major 128-byte swizzle: byte offset of 16-byte chunk g (of 8) of row r
// inside a 64-column slab.
__device__ __forceinline__ uint32_t sw128(int r, int g) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((g ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat162 h) { return *reinterpret_cast<uint32_t*>(&h); }

// hi = bf16(a), lo = bf16(a - hi), two values at a time
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  hi = bf16x2_bits(h);
  lo = bf16x2_bits(__floats2bfloat162_rn(a - hf.x, b - hf.y));
}

// 2^-e and 2^e as floats (e in [-126, 126]).
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// Binary exponent e with m * 2^-e in [1/2, 1) (0 for m == 0), clamped so that
// 2^e and 2^-e are normal floats.
__device__ __forceinline__ int scale_exponent(float m) {
  if (!(m > 0.0f)) return 0;
  const int ex = (__float_as_int(m) >> 23) & 0xff;
  int e = ex == 0 ? -126 : ex - 126;
  return e < -126 ? -126 : (e > 126 ? 126 : e);
}

__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

// 1-D bulk async copy shared -> global (bulk group of this thread).
__device__ __forceinline__ void bulk_copy_s2g(void* dst, uint32_t src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src_smem), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Stages (cos, sin)(pi x / 2) of steps [q0, q0 + PXS) of this tile (zeros
// past the end), between barriers of the epilogue threads: the previous ones
// are read by then, the new ones visible after.
template <int NEPI, class SiteOf>
__device__ __forceinline__ void stage_pixels(float2 (&phi)[PXS][TS], const float* pixels, int n, int B, int b0, int q0,
                                             int nsteps, SiteOf site_of) {
  ptx::named_barrier(1, NEPI);
  for (int e = threadIdx.x; e < PXS * TS; e += NEPI) {
    const int qq = e % PXS, bb = e / PXS;
    float val = 0.0f;
    if (q0 + qq < nsteps && b0 + bb < B) val = __ldg(pixels + (int64_t)(b0 + bb) * n + site_of(q0 + qq));
    phi[qq][bb] = make_float2(cospif(0.5f * val), sinpif(0.5f * val));
  }
  ptx::named_barrier(1, NEPI);
}

// N packed columns of this lane's row of an operand in tensor memory.
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t* r) {
  if constexpr (N == 16) ptx::tmem_st_32x32b_x16(taddr, r);
  else ptx::tmem_st_32x32b_x8(taddr, r);
}

// Waits of an epilogue warp: once one has run out the warp stops waiting (and
// the CTA is winding down) but keeps taking part in the named barriers.
struct EpiWait {
  int32_t* abort;
  int* status;
  bool dead = false;
  __device__ __forceinline__ void operator()(uint64_t* bar, uint32_t parity) {
    if (!dead && !__all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_addr(bar), parity, status))) {
      *(volatile int32_t*)abort = 1;
      dead = true;
    }
    ptx::tc_fence_after();
  }
};
// The warp's arrival after its generic writes / TMEM reads.
__device__ __forceinline__ void warp_arrive(uint64_t* bar) {
  ptx::tc_fence_before();
  __syncwarp();
  if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(ptx::smem_addr(bar));
}

// ------------------------------------------------------------------ packing
__device__ __forceinline__ uint4 swap_chunk(const uint4& a) {
  return make_uint4(__shfl_xor_sync(0xffffffffu, a.x, 1), __shfl_xor_sync(0xffffffffu, a.y, 1),
                    __shfl_xor_sync(0xffffffffu, a.z, 1), __shfl_xor_sync(0xffffffffu, a.w, 1));
}

// Value L[k, s, j] of the core of step t: the left half reads A[k, s, j],
// the right half (swept from the chain's right end) A[j, s, k].
__global__ void __launch_bounds__(256) cls_pack_kernel(const __grid_constant__ ClsPackParams p) {
  const int t = blockIdx.x, h = blockIdx.y;
  if (t >= p.T[h]) return;
  const int site = h == 0 ? t : p.n - 1 - t;
  const int Da = p.bond[site], Dc = p.bond[site + 1];
  const int Din = h == 0 ? Da : Dc, Dout = h == 0 ? Dc : Da;
  const float* __restrict__ A = p.core[site];
  const int chi = p.chi, lc = 31 - __clz(chi), parts = p.split ? 2 : 1;  // chi = 32, 64 or 128
  uint8_t* img = p.images[h] + (size_t)t * p.step_bytes;
  // log2 of the rows and of the K extent of the image kind; a 16-byte chunk is 8 consecutive K of one row
  const int lr = p.adjoint ? lc : lc + 1;
  const int lk = p.adjoint ? lc + 1 : (lc < 6 ? 6 : lc);
  // forward at chi = 128: blocks of one half's 128 rows
  const int halves = !p.adjoint && chi == 128 ? 2 : 1;
  const int slab_bytes = (128 << lr) / halves;
  // The K index runs along the core's unit stride (forward image of the right
  // half, adjoint image of the left): 16 consecutive values as four 16-byte
  // loads where they are aligned.
  const bool kfast = (h == 1) != (p.adjoint != 0);
  const bool vec = kfast && (Dc & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const int lane = threadIdx.x & 31, odd = lane & 1;
  const int pairs = 1 << (lr + lk - 4);  // two chunks of one row each
  for (int c = threadIdx.x; c < pairs; c += 256) {
    const int row = c & ((1 << lr) - 1), k0 = (c >> lr) * 16;
    float v[16];
    // value(K index, row) at base + 16 steps of `stride`, real below `real`
    int fixed_ok, s2, k2;
    if (p.adjoint) {
      s2 = k0 >> lc;  // chi is a multiple of 16: one s
      k2 = k0 & (chi - 1);
      fixed_ok = row < Din;
    } else {
      s2 = row >> lc;
      k2 = k0;
      fixed_ok = (row & (chi - 1)) < Dout;
    }
    const int kreal = (p.adjoint ? Dout : Din) - k2, rowi = p.adjoint ? row : row & (chi - 1);
    // element (k or j along K, the other index along the rows) of A[k, s, j] / A[j, s, k]
    const float* src = kfast ? A + ((int64_t)rowi * 2 + s2) * Dc + k2 : A + ((int64_t)k2 * 2 + s2) * Dc + rowi;
    const int64_t stride = kfast ? 1 : 2 * (int64_t)Dc;
    if (vec && fixed_ok && kreal >= 16) {
#pragma unroll
      for (int e = 0; e < 16; e += 4) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(src + e));
        v[e] = f.x;
        v[e + 1] = f.y;
        v[e + 2] = f.z;
        v[e + 3] = f.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = fixed_ok && e < kreal ? __ldg(src + e * stride) : 0.0f;
    }
    const int ks = k0 >> 6, g = (k0 >> 3) & 7;
    const int half = halves == 2 ? (row >> 6) & 1 : 0;
    const int rb = halves == 2 ? ((row >> 7) << 6) | (row & 63) : row;  // row of its block
    uint8_t* blk = img + (size_t)(ks * halves + half) * parts * slab_bytes;
    uint4 hh[2], ll[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      split_pair(v[8 * i], v[8 * i + 1], hh[i].x, ll[i].x);
      split_pair(v[8 * i + 2], v[8 * i + 3], hh[i].y, ll[i].y);
      split_pair(v[8 * i + 4], v[8 * i + 5], hh[i].z, ll[i].z);
      split_pair(v[8 * i + 6], v[8 * i + 7], hh[i].w, ll[i].w);
    }
    // lanes 2i and 2i + 1 (neighbouring rows) swap a chunk, so that the pair's
    // stores are whole 32-byte sectors
    const uint4 hs = swap_chunk(odd ? hh[0] : hh[1]), ls = swap_chunk(odd ? ll[0] : ll[1]);
    const int r0 = rb & ~1;
    const uint32_t o0 = sw128(r0, g + odd), o1 = sw128(r0 + 1, g + odd);
    *reinterpret_cast<uint4*>(blk + o0) = odd ? hs : hh[0];
    *reinterpret_cast<uint4*>(blk + o1) = odd ? hh[1] : hs;
    if (p.split) {
      *reinterpret_cast<uint4*>(blk + slab_bytes + o0) = odd ? ls : ll[0];
      *reinterpret_cast<uint4*>(blk + slab_bytes + o1) = odd ? ll[1] : ls;
    }
  }
}

// ----------------------------------------------------------------- forward
template <int CHI, int SPLIT>
constexpr size_t fwd_smem_bytes() {
  using C = Cfg<CHI, SPLIT>;
  return 1024 + (size_t)C::VTS + (size_t)C::FRING * C::FSET + sizeof(StageTail);
}

template <int CHI, int SPLIT>
__device__ __forceinline__ void forward_tile(const ClsTcParams& p, const int cta) {
  using C = Cfg<CHI, SPLIT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* vt = base;
  uint8_t* ring = base + C::VTS;
  StageTail& st = *reinterpret_cast<StageTail*>(ring + (size_t)C::FRING * C::FSET);
  Bars& x = st.bars;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int h = cta / p.ntiles, tile = cta % p.ntiles;
  const int B = p.batch, b0 = tile * TS;
  const int t0 = p.t_begin[h];
  const int nsteps = p.t_end[h] - t0;
  const int n = p.n;
  auto site_of = [&](int q) { return p.half_site[h] + p.half_dir[h] * (t0 + q); };
  constexpr int BLOCKS = C::KSL * C::NH;  // core blocks of a step

  if (tid == 0) {
    for (int i = 0; i < C::FRING; ++i) {
      ptx::mbar_init(ptx::smem_addr(&x.full[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.empty[i]), 1);
    }
    for (int i = 0; i < C::NH; ++i) {
      ptx::mbar_init(ptx::smem_addr(&x.acc_full[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.ready[i]), C::NEPI / 32 / C::NH);
    }
    ptx::mbar_init(ptx::smem_addr(&x.drained), C::NEPI / 64);
    ptx::mbar_init(ptx::smem_addr(&x.image), C::NEPI / 32);
    ptx::mbar_init(ptx::smem_addr(&x.stored), 1);
    ptx::mbar_init(ptx::smem_addr(&x.final_bar), 1);
    x.abort = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_addr(&x.tmem_base), C::FCOLS);
    ptx::tmem_relinquish();
  }
  // zero the vector tile (padding columns stay zero)
  for (int i = tid; i < C::VTS / 16; i += C::NTHREADS) reinterpret_cast<uint4*>(vt)[i] = make_uint4(0, 0, 0, 0);
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = x.tmem_base;

  if (warp == C::NEPI / 32) {
    // ---------------- producer: core blocks into the ring
    if ((tid & 31) == 0) {
      const int nblocks = nsteps * BLOCKS;
      const uint8_t* src = p.images[h] + (size_t)t0 * BLOCKS * C::FSET;
      int g = 0;
      for (; g < nblocks; ++g, src += C::FSET) {
        const int slot = g % C::FRING;
        if (g >= C::FRING &&
            !ptx::mbar_wait(ptx::smem_addr(&x.empty[slot]), (uint32_t)(((g / C::FRING) - 1) & 1), p.status)) {
          x.abort = 1;
          break;
        }
        if (*(volatile int32_t*)&x.abort) break;
        const uint32_t bar = ptx::smem_addr(&x.full[slot]);
        ptx::mbar_arrive_expect_tx(bar, C::FSET);
        ptx::bulk_copy_g2s(ptx::smem_addr(ring + (size_t)slot * C::FSET), src, C::FSET, bar);
      }
      // let every copy issued land before the CTA can leave
      for (int gg = g - C::FRING < 0 ? 0 : g - C::FRING; gg < g; ++gg)
        ptx::mbar_wait(ptx::smem_addr(&x.full[gg % C::FRING]), (uint32_t)((gg / C::FRING) & 1), p.status);
    }
    __syncwarp();
  } else if (warp == C::NEPI / 32 + 1) {
    // ---------------- MMAs. At chi = 128 (two halves, two k slabs) in the
    // order (k0, half 0), (k0, half 1), (k1, half 0), (k1, half 1): slab 0 of
    // the vector tile is free again when half 0's accumulator is complete, so
    // half 0 writes its part of the next vector, slab 0, while half 1's last
    // MMAs run, and the next step's first two blocks need nothing else.
    const uint32_t raddr = ptx::smem_addr(ring);
    constexpr int KS = CHI < 64 ? CHI / 16 : 4;  // MMAs along K of a slab (chi = 32: without the padding)
    constexpr uint32_t idesc = ptx::idesc_bf16_f32(128, C::FN);
    int slot = 0;
    uint32_t phase = 0;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      const bool w = __all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_addr(bar), parity, p.status));
      ptx::tc_fence_after();
      return w;
    };
    // A wait takes some 150 cycles when its barrier has completed long ago, and
    // the tensor pipe's queue is short: a block's barriers are waited for
    // before the last MMAs of the block before it are issued.
    bool ok = nsteps > 0 && wait(&x.full[0], 0u);
    for (int q = 0; q < nsteps && ok; ++q) {
      const uint32_t par = (uint32_t)(q & 1);
      ok = wait(&x.ready[0], par);
#pragma unroll
      for (int ks = 0; ks < C::KSL; ++ks) {
#pragma unroll
        for (int nh = 0; nh < C::NH; ++nh) {
          const uint32_t vh = tmem + (uint32_t)(C::VCOL + ks * 32), vl = vh + C::KPAD / 2;
          const uint32_t bh = ptx::desc_lo(raddr + (uint32_t)(slot * C::FSET)), bl = bh + (C::FSLAB >> 4);
          const uint32_t d = tmem + (uint32_t)(nh * C::FN), empty = ptx::smem_addr(&x.empty[slot]);
          auto step = [&](int kk) {
            ptx::mma_bf16_ta(d, vh + kk * 8u, bh + kk * 2u, idesc, (ks | kk) ? 1u : 0u);
            if (SPLIT) {
              ptx::mma_bf16_ta(d, vl + kk * 8u, bh + kk * 2u, idesc, 1u);
              ptx::mma_bf16_ta(d, vh + kk * 8u, bl + kk * 2u, idesc, 1u);
            }
          };
          if (ok && ptx::elect_one()) {
#pragma unroll
            for (int kk = 0; kk < KS - 1; ++kk) step(kk);
          }
          __syncwarp();
          if (++slot == C::FRING) {
            slot = 0;
            phase ^= 1u;
          }
          const bool last = ks == C::KSL - 1 && nh == C::NH - 1;
          if (C::NH == 2 && ks == 0 && nh == 0 && q > 0) ok = ok && wait(&x.drained, par ^ 1u);
          if (C::KSL == 2 && ks == 0 && nh == C::NH - 1) ok = ok && wait(&x.ready[1], par);
          if (!last || q + 1 < nsteps) ok = ok && wait(&x.full[slot], phase);
          if (ok && ptx::elect_one()) {
            step(KS - 1);
            ptx::mma_commit(empty);
            if (ks == C::KSL - 1) ptx::mma_commit(ptx::smem_addr(&x.acc_full[nh]));
          }
          __syncwarp();
        }
      }
    }
    if (!ok && nsteps > 0) x.abort = 1;
    if (ptx::elect_one()) {
      ptx::mma_commit(ptx::smem_addr(&x.final_bar));
      ptx::mbar_wait(ptx::smem_addr(&x.final_bar), 0u, p.status);
    }
    __syncwarp();
  } else if (warp == C::NEPI / 32 + 2) {
    // ---------------- the vectors entering the steps, for the adjoint's gradient product
    if (p.vseg[h] && (tid & 31) == 0) {
      for (int q = 0; q < nsteps; ++q) {
        if (!ptx::mbar_wait(ptx::smem_addr(&x.image), (uint32_t)(q & 1), p.status)) {
          x.abort = 1;
          break;
        }
        bulk_copy_s2g(p.vseg[h] + ((size_t)q * p.ntiles + tile) * C::VTS, ptx::smem_addr(vt), C::VTS);
        bulk_wait_read();
        ptx::mbar_arrive(ptx::smem_addr(&x.stored));
      }
      bulk_wait_all();
    }
    __syncwarp();
  } else {
    // ---------------- epilogue threads
    const int r = tid & (TS - 1), hc = tid >> 7;  // sample row, column group
    const int half = hc * C::NH / C::NG;
    const int b = b0 + r;
    const bool live = b < B;
    const int c0 = hc * C::HC;  // first column of this thread
    float v[C::HC];
#pragma unroll
    for (int k = 0; k < C::HC; ++k) v[k] = live ? p.state_in[h][(int64_t)b * CHI + c0 + k] : 0.0f;
    double lam0 = (live && hc == 0) ? p.lam[h][b] : 0.0;
    int lam_e = 0;
    // scale of the vector in the tile not yet applied (deferred mode)
    int e_prev = 0;
    const bool defer = p.vseg[h] == nullptr;
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    // v, split, as the next step's operand: a lane's row of tensor memory
    auto write_operand = [&]() {
#pragma unroll
      for (int c = 0; c < C::HC; c += 16) {
        uint32_t vh[8], vl[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) split_pair(v[c + 2 * k], v[c + 2 * k + 1], vh[k], vl[k]);
        const uint32_t col = lanes + (uint32_t)(C::VCOL + (c0 + c) / 2);
        ptx::tmem_st_32x32b_x8(col, vh);
        if (SPLIT) ptx::tmem_st_32x32b_x8(col + C::KPAD / 2, vl);
      }
      ptx::tmem_st_wait();
      warp_arrive(&x.ready[half]);
    };
    // and as the image the gradient product reads (128-byte swizzle)
    auto write_image = [&]() {
#pragma unroll
      for (int g8 = 0; g8 < C::HC / 8; ++g8) {
        const int col = c0 + g8 * 8;
        uint8_t* dst = vt + (col >> 6) * SLAB_V + sw128(r, (col >> 3) & 7);
        uint4 hh, ll;
        split_pair(v[8 * g8], v[8 * g8 + 1], hh.x, ll.x);
        split_pair(v[8 * g8 + 2], v[8 * g8 + 3], hh.y, ll.y);
        split_pair(v[8 * g8 + 4], v[8 * g8 + 5], hh.z, ll.z);
        split_pair(v[8 * g8 + 6], v[8 * g8 + 7], hh.w, ll.w);
        *reinterpret_cast<uint4*>(dst) = hh;
        if (SPLIT) *reinterpret_cast<uint4*>(dst + C::VT) = ll;
      }
      ptx::fence_proxy_async_smem();
      warp_arrive(&x.image);
    };
    write_operand();
    if (!defer) write_image();
    // this thread's columns of the accumulators: U[b, (s, j)] at column (half, s, j % (CHI / NH))
    constexpr int JH = CHI / C::NH;
    const uint32_t acc = lanes + (uint32_t)(half * C::FN + c0 % JH);
    EpiWait wait{&x.abort, p.status};
    for (int q = 0; q < nsteps; ++q) {
      const int t = t0 + q;
      if (q % PXS == 0) stage_pixels<C::NEPI>(st.phi, p.pixels, n, B, b0, q, nsteps, site_of);
      // keep the float32 vector entering step t (v holds it times 2^e_prev)
      const float ip = pow2f(-e_prev);
      if (p.store[h] && live && ((t - p.store_base[h]) % p.store_every) == 0) {
        float* dst = p.store[h] + ((int64_t)((t - p.store_base[h]) / p.store_every) * B + b) * CHI + c0;
#pragma unroll
        for (int k = 0; k < C::HC; k += 4)
          *reinterpret_cast<float4*>(dst + k) = make_float4(v[k] * ip, v[k + 1] * ip, v[k + 2] * ip, v[k + 3] * ip);
      }
      // the MMA read v_t 2^e_prev: the step's output times 2^-e_prev is u_t itself (exact)
      const float2 phi = st.phi[q % PXS][r];
      const float g0 = phi.x * ip, g1 = phi.y * ip;
      wait(&x.acc_full[half], (uint32_t)(q & 1));
#pragma unroll
      for (int c = 0; c < C::HC; c += 16) {
        uint32_t u0[16], u1[16];
        ptx::tmem_ld_32x32b_x16(acc + (uint32_t)c, u0);
        ptx::tmem_ld_32x32b_x16(acc + (uint32_t)(JH + c), u1);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) v[c + e] = g0 * __uint_as_float(u0[e]) + g1 * __uint_as_float(u1[e]);
      }
      if (C::NH == 2 && half == 1) warp_arrive(&x.drained);
      // the step's scale 2^e_t from the sample's largest |u_t| over its
      // column groups. Without a vector-image store it is applied one step
      // late (the next MMA reads u_t itself, bf16(u_t) = bf16(v_{t+1}) 2^e_t),
      // so the exchange runs while that MMA does; the recomputation keeps
      // the normalised v_{t+1} in the tile it stores for the gradients.
      auto exchange = [&]() {
        float m = 0.0f;
#pragma unroll
        for (int k = 0; k < C::HC; ++k) m = fmaxf(m, fabsf(v[k]));
        float(*pm)[TS] = st.pmax[q & 1];  // the other one is still being read
        pm[hc][r] = m;
        ptx::named_barrier(2 + (warp & 3), 32 * C::NG);
#pragma unroll
        for (int i = 0; i < C::NG; ++i) m = fmaxf(m, pm[i][r]);
        const int e = scale_exponent(m);
        lam_e += e;
        if (hc == 0 && live) p.sc[h][(int64_t)t * B + b] = pow2f(e);
        return e;
      };
      if (!defer) {
        const float inv = pow2f(-exchange());
#pragma unroll
        for (int k = 0; k < C::HC; ++k) v[k] *= inv;
      }
      write_operand();
      if (defer) {
        e_prev = exchange();
      } else if (q + 1 < nsteps) {
        wait(&x.stored, (uint32_t)(q & 1));
        write_image();
      }
    }
    {
      const float ip = pow2f(-e_prev);
#pragma unroll
      for (int k = 0; k < C::HC; ++k) v[k] *= ip;
    }
    if (live) {
#pragma unroll
      for (int k = 0; k < C::HC; k += 4)
        *reinterpret_cast<float4*>(p.state[h] + (int64_t)b * CHI + c0 + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
      if (hc == 0) p.lam[h][b] = lam0 + (double)lam_e * 0.69314718055994530942;
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, C::FCOLS);
  }
}

// ----------------------------------------------------------------- adjoint
template <int CHI, int SPLIT>
constexpr size_t adj_smem_bytes() {
  using C = Cfg<CHI, SPLIT>;
  return 1024 + (size_t)C::XTS + 2 * (size_t)C::VTS + (size_t)(C::ARING > 0 ? C::ARING : 0) * C::ASET +
         sizeof(StageTail);
}

template <int CHI, int SPLIT>
__device__ __forceinline__ void adjoint_tile(const ClsTcParams& p, const int cta) {
  using C = Cfg<CHI, SPLIT>;
  static_assert(C::ARING >= 2, "adjoint staging does not fit in shared memory");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* xt = base;                      // x tile parts: [x slabs (+ zero slab)] per part
  uint8_t* vring = base + C::XTS;          // 2 v tiles
  uint8_t* cring = vring + 2 * C::VTS;     // adjoint core slabs
  StageTail& st = *reinterpret_cast<StageTail*>(cring + (size_t)C::ARING * C::ASET);
  Bars& x = st.bars;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int h = cta / p.ntiles, tile = cta % p.ntiles;
  const int B = p.batch, b0 = tile * TS;
  const int t0 = p.t_begin[h], t1 = p.t_end[h];
  const int nsteps = t1 - t0;
  const int n = p.n;
  auto step_t = [&](int q) { return t1 - 1 - q; };
  auto site_of = [&](int q) { return p.half_site[h] + p.half_dir[h] * step_t(q); };

  if (tid == 0) {
    for (int i = 0; i < C::ARING; ++i) {
      ptx::mbar_init(ptx::smem_addr(&x.full[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(ptx::smem_addr(&x.vfull[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.vempty[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.acc_full[i]), 1);
    }
    for (int i = 0; i < 2; ++i) ptx::mbar_init(ptx::smem_addr(&x.ready[i]), C::NEPI / 32);
    ptx::mbar_init(ptx::smem_addr(&x.final_bar), 1);
    x.abort = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_addr(&x.tmem_base), C::ACOLS);
    ptx::tmem_relinquish();
  }
  for (int i = tid; i < C::XTS / 16; i += C::NTHREADS) reinterpret_cast<uint4*>(xt)[i] = make_uint4(0, 0, 0, 0);
  ptx::fence_proxy_async_smem();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = x.tmem_base;

  if (warp == C::NEPI / 32) {
    // ---------------- producer: per step the core slabs, then the v tile
    if ((tid & 31) == 0) {
      int g = 0, q = 0;
      bool stop = false;
      for (; q < nsteps && !stop; ++q) {
        const int t = step_t(q);
        for (int ks = 0; ks < C::XSL; ++ks, ++g) {
          const int slot = g % C::ARING;
          if ((g >= C::ARING &&
               !ptx::mbar_wait(ptx::smem_addr(&x.empty[slot]), (uint32_t)(((g / C::ARING) - 1) & 1), p.status)) ||
              *(volatile int32_t*)&x.abort) {
            x.abort = 1;
            stop = true;
            break;
          }
          const uint32_t bar = ptx::smem_addr(&x.full[slot]);
          ptx::mbar_arrive_expect_tx(bar, C::ASET);
          ptx::bulk_copy_g2s(ptx::smem_addr(cring + (size_t)slot * C::ASET),
                             p.images[h] + ((size_t)t * C::XSL + ks) * C::ASET, C::ASET, bar);
        }
        if (stop) break;
        const int vs = q & 1;
        if ((q >= 2 && !ptx::mbar_wait(ptx::smem_addr(&x.vempty[vs]), (uint32_t)(((q >> 1) - 1) & 1), p.status)) ||
            *(volatile int32_t*)&x.abort) {
          x.abort = 1;
          break;
        }
        const uint32_t bar = ptx::smem_addr(&x.vfull[vs]);
        ptx::mbar_arrive_expect_tx(bar, C::VTS);
        ptx::bulk_copy_g2s(ptx::smem_addr(vring + (size_t)vs * C::VTS),
                           p.vseg[h] + ((size_t)(t - t0) * p.ntiles + tile) * C::VTS, C::VTS, bar);
      }
      // let every copy issued land before the CTA can leave
      for (int gg = g - C::ARING < 0 ? 0 : g - C::ARING; gg < g; ++gg)
        ptx::mbar_wait(ptx::smem_addr(&x.full[gg % C::ARING]), (uint32_t)((gg / C::ARING) & 1), p.status);
      // v tiles issued: those of steps 0 .. q-1 (a break leaves q at the step not issued)
      for (int qq = q - 2 < 0 ? 0 : q - 2; qq < q; ++qq)
        ptx::mbar_wait(ptx::smem_addr(&x.vfull[qq & 1]), (uint32_t)((qq >> 1) & 1), p.status);
    }
    __syncwarp();
  } else if (warp == C::NEPI / 32 + 1) {
    // ---------------- MMAs: g' first (the next step waits for it), then the gradient
    const uint32_t xaddr = ptx::smem_addr(xt), vaddr = ptx::smem_addr(vring), caddr = ptx::smem_addr(cring);
    constexpr uint32_t idesc1 = ptx::idesc_bf16_f32(128, CHI);
    constexpr uint32_t idesc2 = ptx::idesc_bf16_f32(128, C::KPAD, 1, 1);
    int slot = 0;
    uint32_t phase = 0;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      const bool w = __all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_addr(bar), parity, p.status));
      ptx::tc_fence_after();
      return w;
    };
    // barriers are waited for ahead of their MMAs, as in the forward
    bool ok = nsteps > 0 && wait(&x.full[0], 0u);
    for (int q = 0; q < nsteps && ok; ++q) {
      const int vs = q & 1;
      ok = wait(&x.ready[0], (uint32_t)(q & 1));
      // g'[b, k] = sum_m x[b, m] L[k, m]
#pragma unroll 1
      for (int ks = 0; ks < C::XSL && ok; ++ks) {
        const uint32_t ah = tmem + (uint32_t)(C::XCOL + ks * 32), al = ah + CHI;
        const uint32_t bh = ptx::desc_lo(caddr + (uint32_t)(slot * C::ASET)), bl = bh + (C::ASLAB >> 4);
        const uint32_t empty = ptx::smem_addr(&x.empty[slot]);
        auto step = [&](int kk) {
          ptx::mma_bf16_ta(tmem, ah + kk * 8u, bh + kk * 2u, idesc1, (ks | kk) ? 1u : 0u);
          if (SPLIT) {
            ptx::mma_bf16_ta(tmem, al + kk * 8u, bh + kk * 2u, idesc1, 1u);
            ptx::mma_bf16_ta(tmem, ah + kk * 8u, bl + kk * 2u, idesc1, 1u);
          }
        };
        if (ptx::elect_one()) {
          step(0);
          step(1);
          step(2);
        }
        __syncwarp();
        if (++slot == C::ARING) {
          slot = 0;
          phase ^= 1u;
        }
        if (ks + 1 < C::XSL) ok = wait(&x.full[slot], phase);
        if (ok && ptx::elect_one()) {
          step(3);
          ptx::mma_commit(empty);
          if (ks == C::XSL - 1) ptx::mma_commit(ptx::smem_addr(&x.acc_full[0]));
        }
        __syncwarp();
      }
      ok = ok && wait(&x.ready[1], (uint32_t)(q & 1)) && wait(&x.vfull[vs], (uint32_t)((q >> 1) & 1));
      // dL[m, k] = sum_b x[b, m] v[b, k]: both operands MN-major (the
      // K-major x tile read transposed; the v tile as the forward wrote it)
      auto grad = [&](int mh, int kk) {
        const uint32_t d = tmem + (uint32_t)(C::A2OFF + ((q & 1) % C::A2BUF) * C::MH * C::KPAD + mh * C::KPAD);
        const uint32_t ah = ptx::desc_lo(xaddr + (uint32_t)(mh * 2 * SLAB_V), SLAB_V), al = ah + (C::XPART >> 4);
        const uint32_t bh = ptx::desc_lo(vaddr + (uint32_t)(vs * C::VTS), SLAB_V), bl = bh + (C::VT >> 4);
        ptx::mma_bf16_lo(d, ah + kk * 128u, bh + kk * 128u, idesc2, kk ? 1u : 0u);
        if (SPLIT) {
          ptx::mma_bf16_lo(d, al + kk * 128u, bh + kk * 128u, idesc2, 1u);
          ptx::mma_bf16_lo(d, ah + kk * 128u, bl + kk * 128u, idesc2, 1u);
        }
      };
      if (ok && ptx::elect_one()) {
#pragma unroll
        for (int mh = 0; mh < C::MH; ++mh)
#pragma unroll
          for (int kk = 0; kk < TS / 16; ++kk)
            if (mh < C::MH - 1 || kk < TS / 16 - 1) grad(mh, kk);
      }
      __syncwarp();
      if (q + 1 < nsteps) ok = ok && wait(&x.full[slot], phase);
      if (ok && ptx::elect_one()) {
        grad(C::MH - 1, TS / 16 - 1);
        ptx::mma_commit(ptx::smem_addr(&x.vempty[vs]));
        ptx::mma_commit(ptx::smem_addr(&x.acc_full[1]));
      }
      __syncwarp();
    }
    if (!ok && nsteps > 0) x.abort = 1;
    if (ptx::elect_one()) {
      ptx::mma_commit(ptx::smem_addr(&x.final_bar));
      ptx::mbar_wait(ptx::smem_addr(&x.final_bar), 0u, p.status);
    }
    __syncwarp();
  } else if (warp < C::NEPI / 32) {
    const int r = tid & (TS - 1), hc = tid >> 7;
    const int b = b0 + r;
    const bool live = b < B;
    const int c0 = hc * C::HC;
    float g[C::HC];
#pragma unroll
    for (int k = 0; k < C::HC; ++k) g[k] = live ? p.state[h][(int64_t)b * CHI + c0 + k] : 0.0f;
    // x of the step q: Phi_s(x at that step's site) g / sc, columns (s, c0 + k)
    constexpr int HX = C::HC / 2;  // packed columns of one s
    uint32_t xh[2][HX], xl[2][HX];
    float f[2], inv;
    auto load_scale = [&](int q) { return live && q < nsteps ? __ldg(p.sc[h] + (int64_t)step_t(q) * B + b) : 1.0f; };
    float scl = load_scale(0);  // of the next x, a step ahead of its use
    auto load_factors = [&](int q) {
      const float2 phi = st.phi[q % PXS][r];
      f[0] = phi.x;
      f[1] = phi.y;
      inv = __frcp_rn(scl);  // scales are powers of two: exact
      scl = load_scale(q + 1);
    };
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    // as g's operand: a lane's row of tensor memory
    auto make_x = [&]() {
#pragma unroll
      for (int s = 0; s < 2; ++s) {
#pragma unroll
        for (int k = 0; k < HX; ++k)
          split_pair(f[s] * g[2 * k] * inv, f[s] * g[2 * k + 1] * inv, xh[s][k], xl[s][k]);
        const uint32_t col = lane_base + (uint32_t)(C::XCOL + (s * CHI + c0) / 2);
        tmem_st<HX>(col, xh[s]);
        if (SPLIT) tmem_st<HX>(col + CHI, xl[s]);
      }
      ptx::tmem_st_wait();
      warp_arrive(&x.ready[0]);
    };
    // as the gradient's, transposed there: the swizzled tile
    auto write_xtile = [&]() {
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int g8 = 0; g8 < C::HC / 8; ++g8) {
          const int col = s * CHI + c0 + g8 * 8;
          uint8_t* dst = xt + (col >> 6) * SLAB_V + sw128(r, (col >> 3) & 7);
          const uint32_t *hp = &xh[s][4 * g8], *lp = &xl[s][4 * g8];
          *reinterpret_cast<uint4*>(dst) = make_uint4(hp[0], hp[1], hp[2], hp[3]);
          if (SPLIT) *reinterpret_cast<uint4*>(dst + C::XPART) = make_uint4(lp[0], lp[1], lp[2], lp[3]);
        }
      ptx::fence_proxy_async_smem();
      warp_arrive(&x.ready[1]);
    };
    if (nsteps > 0) {
      stage_pixels<C::NEPI>(st.phi, p.pixels, n, B, b0, 0, nsteps, site_of);
      load_factors(0);
      make_x();
      write_xtile();
    }
    const int mrow = r;  // gradient row (x column) of this lane in M half 0
    // this tile's share of step t's core gradient, from accumulator `buf`
    auto drain_grad = [&](int t, int buf) {
      float* gbase = p.grad[h] + (size_t)t * CHI * 2 * CHI;
#pragma unroll
      for (int mh = 0; mh < C::MH; ++mh) {
        const int m = mh * 128 + mrow;
#pragma unroll
        for (int c = 0; c < C::KPAD / C::NG; c += 16) {
          const int k0 = hc * (C::KPAD / C::NG) + c;
          if (k0 < CHI) {
            uint32_t u[16];
            ptx::tmem_ld_32x32b_x16(lane_base + (uint32_t)(C::A2OFF + buf * C::MH * C::KPAD + mh * C::KPAD + k0), u);
            ptx::tmem_ld_wait();
            if (m < 2 * CHI) {
#pragma unroll
              for (int e = 0; e < 16; ++e)
                if (k0 + e < CHI) red_add(gbase + (size_t)(k0 + e) * 2 * CHI + m, __uint_as_float(u[e]));
            }
          }
        }
      }
    };

    EpiWait wait{&x.abort, p.status};
    for (int q = 0; q < nsteps; ++q) {
      const int t = step_t(q);
      const bool more = q + 1 < nsteps;
      // pixels of steps q + 1 .. q + PXS (the x of the next step needs them)
      if ((q + 1) % PXS == 0 && more) stage_pixels<C::NEPI>(st.phi, p.pixels, n, B, b0, q + 1, nsteps, site_of);
      if (more) load_factors(q + 1);
      // g' and the next step's operand made of it; then, once the gradient
      // product has read the x tile, the tile
      wait(&x.acc_full[0], (uint32_t)(q & 1));
#pragma unroll
      for (int c = 0; c < C::HC; c += 16) {
        uint32_t u[16];
        ptx::tmem_ld_32x32b_x16(lane_base + (uint32_t)(c0 + c), u);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) g[c + e] = __uint_as_float(u[e]);
      }
      if (more) make_x();
      wait(&x.acc_full[1], (uint32_t)(q & 1));
      if (C::A2BUF == 1 && !wait.dead) drain_grad(t, 0);
      if (more) write_xtile();
      // with two accumulators this step's gradient is drained while the next
      // step's products run (its buffer is rewritten by the products two
      // steps on, which wait for this warp's next tile)
      if (C::A2BUF == 2 && !wait.dead) drain_grad(t, q & 1);
    }
    if (live) {
#pragma unroll
      for (int k = 0; k < C::HC; k += 4)
        *reinterpret_cast<float4*>(p.state[h] + (int64_t)b * CHI + c0 + k) = make_float4(g[k], g[k + 1], g[k + 2], g[k + 3]);
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, C::ACOLS);
  }
}

template <int CHI, int SPLIT>
__global__ void __launch_bounds__(Cfg<CHI, SPLIT>::NTHREADS, 1) cls_fwd_tc(const __grid_constant__ ClsTcParams p) {
  forward_tile<CHI, SPLIT>(p, (int)blockIdx.x);
}

// The adjoint of one segment beside the recomputation of the next one: each
// leaves more than half of the SMs idle at 4096 samples (64 CTAs).
struct ClsPairParams {
  ClsTcParams adj, fwd;
};
template <int CHI, int SPLIT>
__global__ void __launch_bounds__(Cfg<CHI, SPLIT>::NTHREADS, 1) cls_pair_tc(const __grid_constant__ ClsPairParams p) {
  const int n = 2 * p.adj.ntiles;
  if ((int)blockIdx.x < n) adjoint_tile<CHI, SPLIT>(p.adj, (int)blockIdx.x);
  else forward_tile<CHI, SPLIT>(p.fwd, (int)blockIdx.x - n);
}

// dcore[site] from the step's accumulated gradient G[t][k][(s, j)]: the left
// half's core is L itself (A[k, s, j]), the right half's its transpose
// (A[j, s, k]).
__global__ void cls_scatter_kernel(const __grid_constant__ ClsScatterParams p) {
  int t = blockIdx.x, h = 0;
  if (t >= p.T[0]) {
    t -= p.T[0];
    h = 1;
  }
  const int site = h == 0 ? t : p.n - 1 - t;
  const int Da = p.bond[site], Dc = p.bond[site + 1], chi = p.chi;
  const float* __restrict__ G = p.grad[h] + (size_t)t * chi * 2 * chi;
  float* __restrict__ d = p.dcore[site];
  const int total = Da * 2 * Dc;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    const int c = i % Dc, s = (i / Dc) & 1, a = i / (2 * Dc);
    d[i] = h == 0 ? G[(size_t)a * 2 * chi + s * chi + c] : G[(size_t)c * 2 * chi + s * chi + a];
  }
}

template <int CHI, int SPLIT>
int launch_fwd(const ClsTcParams& p, cudaStream_t s) {
  const size_t smem = fwd_smem_bytes<CHI, SPLIT>();
  static std::atomic<uint64_t> attr{0};
  if (!smem_limit_once((const void*)cls_fwd_tc<CHI, SPLIT>, smem, &attr)) return TN_ERR_CUDA;
  cls_fwd_tc<CHI, SPLIT><<<2 * p.ntiles, Cfg<CHI, SPLIT>::NTHREADS, smem, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

template <int CHI, int SPLIT>
int launch_pair(const ClsTcParams& a, const ClsTcParams* f, cudaStream_t s) {
  if constexpr (Cfg<CHI, SPLIT>::ARING < 2) {
    return TN_ERR_UNSUPPORTED;
  } else {
    const size_t smem = std::max(adj_smem_bytes<CHI, SPLIT>(), fwd_smem_bytes<CHI, SPLIT>());
    static std::atomic<uint64_t> attr{0};
    if (!smem_limit_once((const void*)cls_pair_tc<CHI, SPLIT>, smem, &attr)) return TN_ERR_CUDA;
    ClsPairParams p;
    p.adj = a;
    p.fwd = f ? *f : a;
    cls_pair_tc<CHI, SPLIT><<<(f ? 4 : 2) * a.ntiles, Cfg<CHI, SPLIT>::NTHREADS, smem, s>>>(p);
    return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
  }
}

}  // namespace

size_t cls_fwd_image_bytes(int chi, int split) {
  const int kpad = chi < 64 ? 64 : chi;
  return (size_t)(2 * chi) * kpad * 2 * (split ? 2 : 1);
}

size_t cls_adj_image_bytes(int chi, int split) { return (size_t)chi * (2 * chi) * 2 * (split ? 2 : 1); }

size_t cls_vtile_bytes(int chi, int split) {
  const int kpad = chi < 64 ? 64 : chi;
  return (size_t)TS * kpad * 2 * (split ? 2 : 1);
}

int cls_pack(const ClsPackParams& p, cudaStream_t s) {
  const int steps = p.T[0] > p.T[1] ? p.T[0] : p.T[1];
  if (steps <= 0) return TN_OK;
  cls_pack_kernel<<<dim3((unsigned)steps, 2), 256, 0, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

int cls_fwd_tc_launch(int chi, int split, const ClsTcParams& p, cudaStream_t s) {
  if (p.t_end[0] <= p.t_begin[0] && p.t_end[1] <= p.t_begin[1]) return TN_OK;
  if (chi == 32) return split ? launch_fwd<32, 1>(p, s) : launch_fwd<32, 0>(p, s);
  if (chi == 64) return split ? launch_fwd<64, 1>(p, s) : launch_fwd<64, 0>(p, s);
  if (chi == 128) return split ? launch_fwd<128, 1>(p, s) : launch_fwd<128, 0>(p, s);
  return TN_ERR_UNSUPPORTED;
}

bool cls_adj_tc_supported(int chi, int split) {
  if (chi == 32) return split ? Cfg<32, 1>::ARING >= 2 : Cfg<32, 0>::ARING >= 2;
  if (chi == 64) return split ? Cfg<64, 1>::ARING >= 2 : Cfg<64, 0>::ARING >= 2;
  if (chi == 128) return split ? Cfg<128, 1>::ARING >= 2 : Cfg<128, 0>::ARING >= 2;
  return false;
}

int cls_adj_tc_launch(int chi, int split, const ClsTcParams& a, const ClsTcParams* f, cudaStream_t s) {
  if (f && f->t_end[0] <= f->t_begin[0] && f->t_end[1] <= f->t_begin[1]) f = nullptr;
  if (a.t_end[0] <= a.t_begin[0] && a.t_end[1] <= a.t_begin[1]) return f ? cls_fwd_tc_launch(chi, split, *f, s) : TN_OK;
  if (chi == 32) return split ? launch_pair<32, 1>(a, f, s) : launch_pair<32, 0>(a, f, s);
  if (chi == 64) return split ? launch_pair<64, 1>(a, f, s) : launch_pair<64, 0>(a, f, s);
  if (chi == 128) return split ? launch_pair<128, 1>(a, f, s) : launch_pair<128, 0>(a, f, s);
  return TN_ERR_UNSUPPORTED;
}

int cls_scatter_grad(const ClsScatterParams& p, cudaStream_t s) {
  const int blocks = p.T[0] + p.T[1];
  if (blocks <= 0) return TN_OK;
  cls_scatter_kernel<<<(unsigned)blocks, 256, 0, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

}  // namespace tn
