// MPS classifier sweeps in float32 on the CUDA cores: the FP32 path of
// tn_mps_classify / tn_mps_classify_backward (Sec. IV.A).
//
// One step of a half-chain, for a tile of samples b and the site's core seen
// as the image I[k, s, j] (k the index summed over, j the outgoing one):
//     out_b[j] = sum_s Phi_s(x_b) sum_k in_b[k] I[k, s, j].
// Forward: in = v, and out is divided by its largest magnitude (the log of
// which joins the sample's float64 log-scale). Adjoint: I is the transposed
// core, in = h = g / scale with g the adjoint entering the step and scale the
// forward's; h is kept, for the core gradients
//     dL[k, s, j] = sum_b v_b[k] Phi_s(x_b) h_b[j].
//
// What bounds it: the FMA pipe, once the operands are fed and the steps'
// serial part is short. A thread holds RS samples x 4 outgoing indices x both
// s (64 accumulators at RS = 8, as packed pairs), so a k step is RS / 4 + 2
// 16-byte shared-memory reads for 4 RS packed FMAs; a warp covers 4 x 8
// threads (samples x outgoing), which halves the shared-memory passes of its
// reads against 2 x 16. Every sum keeps one chain over k: splitting k over two
// groups of threads gained 1 % (4.28 against 4.34 us a step at chi = 64, batch
// 4096) and moved the float64 log-scales. The images stream through a ring of shared-memory
// slabs (1-D bulk copies by a producer warp, across steps), so no step waits
// for its core; further warps compute the next step's features and the
// log-scales beside the products. The vector lives in two shared-memory
// buffers [k][sample], 16-byte chunks XOR-swizzled by k / 4 so that
// publishing four rows at once and reading one row are both free of bank
// conflicts. A step at chi = 64 takes ~7,300 cycles for 64 samples, 5,070 of
// them the products (the FMA pipe's own 4,096), the rest the wait for the slab
// (~250), the maximum, the division and the publishing.
// Measured (784 sites, batch 4096, chi = 64): forward 10.9 -> 1.5 ms, training
// step 53.2 -> 6.3 ms.
#include <math.h>

#include "classifier_f32.h"
#include "divide.cuh"
#include "ptx.cuh"

namespace tn {
namespace {

// Image of step t of half h: out[k][s][j] = core element of (in k, s, out j).
__global__ void __launch_bounds__(256) cls_f32_pack_kernel(const __grid_constant__ ClsF32PackParams p) {
  const int t = blockIdx.x, h = blockIdx.y;
  if (t >= p.T[h]) return;
  const int site = h == 0 ? t : p.n - 1 - t;
  const int Da = p.bond[site], Dc = p.bond[site + 1], chi = p.chi;
  const bool natural = (h == 0) == (p.adjoint == 0);  // in = a, out = c; else in = c, out = a
  const float* __restrict__ A = p.core[site];
  float* __restrict__ o = p.images[h] + (size_t)t * 2 * chi * chi;
  if (natural) {
    for (int i = threadIdx.x; i < 2 * chi * chi; i += 256) {
      const int j = i % chi, ks = i / chi;  // ks = 2 k + s
      o[i] = (ks < 2 * Da && j < Dc) ? __ldg(A + (int64_t)ks * Dc + j) : 0.0f;
    }
    return;
  }
  // transposed through a 32 x 32 tile per s
  __shared__ float tile[32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int s = 0; s < 2; ++s)
    for (int a0 = 0; a0 < chi; a0 += 32)
      for (int c0 = 0; c0 < chi; c0 += 32) {
        for (int r = y; r < 32; r += 8) {
          const int a = a0 + r, c = c0 + x;
          tile[r][x] = (a < Da && c < Dc) ? __ldg(A + ((int64_t)a * 2 + s) * Dc + c) : 0.0f;
        }
        __syncthreads();
        for (int r = y; r < 32; r += 8) o[((size_t)(c0 + r) * 2 + s) * chi + a0 + x] = tile[x][r];
        __syncthreads();
      }
}

template <int CHI, int RS>
struct SweepCfg {
  static constexpr int OG = CHI / 4;                  // threads along the outgoing index
  static constexpr int SG = CHI == 32 ? 16 : 8;       // threads along the samples
  static constexpr int NC = OG * SG;                  // compute threads
  static constexpr int OW = OG / 8;                   // warps along the outgoing index
  static constexpr int TB = RS * SG;                  // samples per CTA
  static constexpr int NS = TB < 32 ? 32 : TB;        // sampler threads
  static constexpr int NT = NC + 32 + NS;
  static constexpr int MASK = TB / 4 - 1 < 7 ? TB / 4 - 1 : 7;
  static constexpr int KS = CHI == 128 ? 32 : CHI;    // k rows of a slab (8, 32 and 32 KB)
  static constexpr int SLAB = KS * 2 * CHI;           // floats of a slab
  static constexpr int RING = CHI == 32 ? 4 : (CHI == 64 ? 3 : 4);
  static constexpr size_t SMEM = sizeof(float) * ((size_t)RING * SLAB + 2 * CHI * TB);
};

struct SweepBars {
  uint64_t full[8], empty[8];
};

template <int CHI, int RS, int ADJ>
__global__ void __launch_bounds__(SweepCfg<CHI, RS>::NT)
cls_f32_sweep_kernel(const __grid_constant__ ClsF32Params p) {
  using C = SweepCfg<CHI, RS>;
  constexpr int NC = C::NC, TB = C::TB;
  extern __shared__ __align__(128) float smem[];
  float* ring = smem;
  float* S = smem + C::RING * C::SLAB;  // two buffers [CHI][TB]
  __shared__ __align__(16) float phi[2][2][TB];
  __shared__ float scl[2][TB];
  __shared__ float smax[C::OW][TB];
  __shared__ __align__(8) SweepBars bars;
  const int half = blockIdx.y, tid = threadIdx.x;
  const int t0 = p.t_begin[half], t1 = p.t_end[half], nsteps = t1 - t0;
  if (nsteps <= 0) return;
  const int b0 = blockIdx.x * TB, B = p.batch, n = p.n, kmax = p.kmax;
  const int nslab = (kmax + C::KS - 1) / C::KS;
  if (tid == 0) {
    for (int i = 0; i < C::RING; ++i) {
      ptx::mbar_init(ptx::smem_addr(&bars.full[i]), 1);
      ptx::mbar_init(ptx::smem_addr(&bars.empty[i]), NC / 32);
    }
    ptx::fence_mbar_init();
  }
  __syncthreads();

  if (tid >= NC && tid < NC + 32) {  // producer warp: one lane streams the images
    if (tid != NC) return;
    const int total = nsteps * nslab;
    bool ok = true;
    int issued = 0;
    for (; issued < total; ++issued) {
      const int st = issued % C::RING, use = issued / C::RING;
      if (use > 0 && !(ok = ptx::mbar_wait(ptx::smem_addr(&bars.empty[st]), (use - 1) & 1, p.status))) break;
      const int q = issued / nslab, sl = issued - q * nslab;
      const int t = ADJ ? t1 - 1 - q : t0 + q;
      const int rows = min(C::KS, kmax - sl * C::KS);
      const uint32_t bytes = (uint32_t)(rows * 2 * CHI * sizeof(float)), full = ptx::smem_addr(&bars.full[st]);
      ptx::mbar_arrive_expect_tx(full, bytes);
      ptx::bulk_copy_g2s(ptx::smem_addr(ring + st * C::SLAB),
                         p.images[half] + (size_t)t * 2 * CHI * CHI + (size_t)sl * C::SLAB, bytes, full);
    }
    if (!ok)  // let the copies in flight land before the CTA may end
      for (int i = issued > C::RING ? issued - C::RING : 0; i < issued; ++i)
        ptx::mbar_wait(ptx::smem_addr(&bars.full[i % C::RING]), (i / C::RING) & 1, p.status);
    return;
  }

  constexpr int NB = NC + C::NS;  // threads of the step barriers
  auto site_of = [&](int t) { return half == 0 ? t : n - 1 - t; };
  auto step_t = [&](int q) { return ADJ ? t1 - 1 - q : t0 + q; };

  if (tid >= NC) {  // samplers: one thread per sample
    const int i = tid - NC - 32, sb = b0 + i;
    const bool in = i < TB, live = in && sb < B;
    auto pixel = [&](int q) { return live && q < nsteps ? __ldg(p.pixels + (int64_t)sb * n + site_of(step_t(q))) : 0.0f; };
    auto scale_of = [&](int q) { return live && q < nsteps ? p.sc[half][(int64_t)step_t(q) * B + sb] : 1.0f; };
    auto put_features = [&](int q, float x) {  // of step q into buffer q & 1
      if (!in || q >= nsteps) return;
      const float c = cospif(0.5f * x), s = sinpif(0.5f * x);
      phi[q & 1][0][i] = c;
      phi[q & 1][1][i] = s;
      if (ADJ && live) p.phi[half][(int64_t)(step_t(q) - t0) * ((B + 1) & ~1) + sb] = make_float2(c, s);
    };
    double lam = !ADJ && live ? p.lam[half][sb] : 0.0;
    if (ADJ && in) {  // scl[q & 1]: the scale the vector entering step q is divided by
      scl[0][i] = scale_of(0);
      scl[1][i] = scale_of(1);
    }
    float nsc = ADJ ? scale_of(2) : 1.0f;
    put_features(0, pixel(0));
    float x = pixel(1);
    ptx::named_barrier(1, NB);
    ptx::named_barrier(1, NB);
    auto add_scale = [&](int q) {  // the scale of the vector that left step q
      if (ADJ || !live) return;
      const float sc = scl[q & 1][i];
      lam += (double)logf(sc);
      p.sc[half][(int64_t)step_t(q) * B + sb] = sc;
    };
    for (int q = 0; q < nsteps; ++q) {
      const float x1 = x;
      x = pixel(q + 2);
      if (ADJ && in) {  // the vector of step q is behind the last barrier: its slot takes step q + 2's scale
        scl[q & 1][i] = nsc;
        nsc = scale_of(q + 3);
      }
      put_features(q + 1, x1);
      if (q > 0) add_scale(q - 1);
      if (ptx::named_barrier_or(1, NB, false)) return;
    }
    add_scale(nsteps - 1);
    if (!ADJ && live) p.lam[half][sb] = lam;
    return;
  }

  // thread: samples f0 .. f0 + RS - 1 of the tile, outgoing indices 4 og .. + 3
  const int og = (tid >> 5) % C::OW * 8 + (tid & 7), f0 = ((tid >> 5) / C::OW * 4 + ((tid >> 3) & 3)) * RS;
  // out[i][j]: sample b0 + f0 + i, outgoing index 4 og + j
  float out[RS][4];
#pragma unroll
  for (int i = 0; i < RS; ++i) {
    const int b = b0 + f0 + i;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b < B) v = *reinterpret_cast<const float4*>(p.state[half] + (int64_t)b * CHI + og * 4);
    out[i][0] = v.x;
    out[i][1] = v.y;
    out[i][2] = v.z;
    out[i][3] = v.w;
  }
  ptx::named_barrier(1, NB);

  float* kept = nullptr;  // where the next kept vector goes, in `until` steps
  int until = 0;
  if (!ADJ && p.store[half]) {
    const int since = t0 - p.store_base[half], slot = (since + p.store_every - 1) / p.store_every;
    kept = p.store[half] + (int64_t)slot * B * CHI;
    until = slot * p.store_every - since;
  }
  // out as the vector entering step q (of t): divided by the step's scale in
  // the adjoint, kept when asked, and written to S's buffer q & 1
  auto publish = [&](int q) {
    const int t = step_t(q);
    if (ADJ) {
      float sc[RS];
#pragma unroll
      for (int i = 0; i < RS; ++i) sc[i] = scl[q & 1][f0 + i];
      divide_rows<false>(out, sc);
    }
    float* keep = nullptr;
    if (ADJ) {
      keep = p.h[half] + (int64_t)(t - t0) * B * CHI;
    } else if (kept) {
      if (until == 0) {
        keep = kept;
        kept += (int64_t)B * CHI;
        until = p.store_every;
      }
      --until;
    }
    if (keep) {
#pragma unroll
      for (int i = 0; i < RS; ++i) {
        const int b = b0 + f0 + i;
        if (b < B)
          *reinterpret_cast<float4*>(keep + (int64_t)b * CHI + og * 4) =
              make_float4(out[i][0], out[i][1], out[i][2], out[i][3]);
      }
    }
    float* d = S + (q & 1) * CHI * TB;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* row = d + (og * 4 + j) * TB;
      const int at = (((f0 >> 2) ^ (og & C::MASK)) << 2) + (f0 & 3);
      if constexpr (RS == 2) {
        *reinterpret_cast<float2*>(row + at) = make_float2(out[0][j], out[1][j]);
      } else {
#pragma unroll
        for (int u = 0; u < RS / 4; ++u)
          *reinterpret_cast<float4*>(row + ((((f0 >> 2) + u) ^ (og & C::MASK)) << 2)) =
              make_float4(out[u * 4][j], out[u * 4 + 1][j], out[u * 4 + 2][j], out[u * 4 + 3][j]);
      }
    }
  };
  publish(0);
  ptx::named_barrier(1, NB);

  int it = 0;  // slabs consumed
  for (int q = 0; q < nsteps; ++q) {
    float2 acc0[RS][2], acc1[RS][2];
#pragma unroll
    for (int i = 0; i < RS; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc0[i][j] = acc1[i][j] = make_float2(0.f, 0.f);
    const float* Sq = S + (q & 1) * CHI * TB;
    bool ok = true;
    for (int sl = 0; sl < nslab; ++sl, ++it) {
      const int st = it % C::RING;
      ok = ok && ptx::mbar_wait(ptx::smem_addr(&bars.full[st]), (it / C::RING) & 1, p.status);
      const int k0 = sl * C::KS, rows = min(C::KS, kmax - k0);
      const float* L = ring + st * C::SLAB + og * 4;
#pragma unroll 1
      for (int kq = 0; kq < rows; kq += 4) {
        const int x = ((k0 + kq) >> 2) & C::MASK;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const float* row = Sq + (k0 + kq + kk) * TB;
          float v[RS];
          if constexpr (RS == 2) {
            const float2 a = *reinterpret_cast<const float2*>(row + (((f0 >> 2) ^ x) << 2) + (f0 & 3));
            v[0] = a.x;
            v[1] = a.y;
          } else {
#pragma unroll
            for (int u = 0; u < RS / 4; ++u) {
              const float4 a = *reinterpret_cast<const float4*>(row + ((((f0 >> 2) + u) ^ x) << 2));
              v[u * 4] = a.x;
              v[u * 4 + 1] = a.y;
              v[u * 4 + 2] = a.z;
              v[u * 4 + 3] = a.w;
            }
          }
          const float4 l0 = *reinterpret_cast<const float4*>(L + (kq + kk) * 2 * CHI);
          const float4 l1 = *reinterpret_cast<const float4*>(L + (kq + kk) * 2 * CHI + CHI);
          const float2 a0[2] = {make_float2(l0.x, l0.y), make_float2(l0.z, l0.w)};
          const float2 a1[2] = {make_float2(l1.x, l1.y), make_float2(l1.z, l1.w)};
#pragma unroll
          for (int i = 0; i < RS; ++i) {
            const float2 vv = make_float2(v[i], v[i]);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              acc0[i][j] = __ffma2_rn(vv, a0[j], acc0[i][j]);
              acc1[i][j] = __ffma2_rn(vv, a1[j], acc1[i][j]);
            }
          }
        }
      }
      __syncwarp();
      if ((tid & 31) == 0) ptx::mbar_arrive(ptx::smem_addr(&bars.empty[st]));
    }
#pragma unroll
    for (int i = 0; i < RS; i += 2) {
      const float2 p0 = *reinterpret_cast<const float2*>(&phi[q & 1][0][f0 + i]);
      const float2 p1 = *reinterpret_cast<const float2*>(&phi[q & 1][1][f0 + i]);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        out[i][2 * j] = p0.x * acc0[i][j].x + p1.x * acc1[i][j].x;
        out[i][2 * j + 1] = p0.x * acc0[i][j].y + p1.x * acc1[i][j].y;
        out[i + 1][2 * j] = p0.y * acc0[i + 1][j].x + p1.y * acc1[i + 1][j].x;
        out[i + 1][2 * j + 1] = p0.y * acc0[i + 1][j].y + p1.y * acc1[i + 1][j].y;
      }
    }
    if (!ADJ) {
      // the sample's largest magnitude: over the thread's four, the warp's
      // eight threads of the sample, then the warps along the outgoing index
      float m[RS];
#pragma unroll
      for (int i = 0; i < RS; ++i) {
        m[i] = fmaxf(fmaxf(fabsf(out[i][0]), fabsf(out[i][1])), fmaxf(fabsf(out[i][2]), fabsf(out[i][3])));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) m[i] = fmaxf(m[i], __shfl_xor_sync(0xffffffffu, m[i], o));
      }
      if constexpr (C::OW > 1) {
        if ((tid & 7) == 0) {
#pragma unroll
          for (int i = 0; i < RS; ++i) smax[og >> 3][f0 + i] = m[i];
        }
        ptx::named_barrier(2, NC);
#pragma unroll
        for (int i = 0; i < RS; ++i) {
          m[i] = smax[0][f0 + i];
#pragma unroll
          for (int u = 1; u < C::OW; ++u) m[i] = fmaxf(m[i], smax[u][f0 + i]);
        }
      }
#pragma unroll
      for (int i = 0; i < RS; ++i) {
        if (!(m[i] > 0.0f)) m[i] = 1.0f;
        if (og == 0) scl[q & 1][f0 + i] = m[i];
      }
      divide_rows<true>(out, m);
    }
    if (q + 1 < nsteps) publish(q + 1);
    // the next vector, features and scales are in place for every warp; a
    // warp whose copy never came takes all of them out together
    if (ptx::named_barrier_or(1, NB, !ok)) return;
  }
#pragma unroll
  for (int i = 0; i < RS; ++i) {
    const int b = b0 + f0 + i;
    if (b < B)
      *reinterpret_cast<float4*>(p.state[half] + (int64_t)b * CHI + og * 4) =
          make_float4(out[i][0], out[i][1], out[i][2], out[i][3]);
  }
}

template <int CHI, int RS, int ADJ>
int launch_sweep(const ClsF32Params& p, cudaStream_t s) {
  using C = SweepCfg<CHI, RS>;
  static std::atomic<uint64_t> attr{0};
  if (!smem_limit_once((const void*)cls_f32_sweep_kernel<CHI, RS, ADJ>, C::SMEM, &attr)) return TN_ERR_CUDA;
  const dim3 grid((unsigned)((p.batch + C::TB - 1) / C::TB), 2);
  cls_f32_sweep_kernel<CHI, RS, ADJ><<<grid, C::NT, C::SMEM, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

template <int CHI, int ADJ>
int launch_sweep_chi(const ClsF32Params& p, cudaStream_t s) {
  // a step takes about as long as its tile has samples, so the tile is the
  // smallest with which both halves still fit the SMs in one wave
  constexpr int SG = SweepCfg<CHI, 2>::SG;
  auto ctas = [&](int rs) { return 2 * ((p.batch + rs * SG - 1) / (rs * SG)); };
  const int sms = sm_count();
  if (ctas(2) <= sms) return launch_sweep<CHI, 2, ADJ>(p, s);
  if (ctas(4) <= sms) return launch_sweep<CHI, 4, ADJ>(p, s);
  return launch_sweep<CHI, 8, ADJ>(p, s);
}

// Core gradients of a segment. CTA (k range of the batch, step, half and j
// range): a CHI x (2 s x JW j) tile of dL summed over `chunk` samples, then
// added to the step's gradient with 16-byte reductions. A thread holds KT k x
// 4 j x both s; the products Phi_s h are formed in registers (8 multiplies
// for 8 KT FMAs), so only v and h are read, GB samples at a time through two
// stages of 1-D bulk copies (v, h and the feature pairs of consecutive
// samples are contiguous).
template <int CHI>
struct GradCfg {
  static constexpr int JW = CHI < 64 ? CHI : 64;      // j per CTA
  static constexpr int KT = CHI == 32 ? 4 : 8;        // k per thread
  static constexpr int JG = JW / 4, KG = CHI / KT;
  static constexpr int NT = JG * KG;
  static constexpr int GB = 32;                       // samples per stage
  static constexpr int STAGE = GB * (2 * CHI + 2);    // floats: v, h (whole rows), phi
  static constexpr int STAGES = 3;
  static constexpr size_t SMEM = sizeof(float) * (size_t)STAGES * STAGE;
};

template <int CHI>
__global__ void __launch_bounds__(GradCfg<CHI>::NT) cls_f32_grad_kernel(const __grid_constant__ ClsF32GradParams p) {
  using C = GradCfg<CHI>;
  constexpr int JG = C::JG, KT = C::KT, GB = C::GB;
  extern __shared__ __align__(128) float smem[];
  __shared__ __align__(8) uint64_t full[C::STAGES];
  const int half = blockIdx.z & 1, jr = (blockIdx.z >> 1) * C::JW, tid = threadIdx.x;
  const int st = blockIdx.y, nst = p.t_end[half] - p.t_begin[half];
  if (st >= nst) return;
  const int B = p.batch, lo = blockIdx.x * p.chunk, hi = min(B, lo + p.chunk);
  if (lo >= hi) return;
  const int nblk = (hi - lo + GB - 1) / GB;
  const float* vb = p.v[half] + (int64_t)st * B * CHI;
  const float* hb = p.h[half] + (int64_t)st * B * CHI;
  const float2* fb = p.phi[half] + (int64_t)st * ((B + 1) & ~1);
  if (tid == 0) {
    for (int i = 0; i < C::STAGES; ++i) ptx::mbar_init(ptx::smem_addr(&full[i]), 1);
    ptx::fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int g) {  // one thread: block g of samples into stage g % STAGES
    const int s = g % C::STAGES, c0 = lo + g * GB, nb = min(GB, hi - c0);
    const uint32_t bar = ptx::smem_addr(&full[s]), dst = ptx::smem_addr(smem + s * C::STAGE);
    const uint32_t rows = (uint32_t)(nb * CHI * sizeof(float)), fbytes = (uint32_t)(((nb + 1) & ~1) * sizeof(float2));
    ptx::mbar_arrive_expect_tx(bar, 2 * rows + fbytes);
    ptx::bulk_copy_g2s(dst, vb + (int64_t)c0 * CHI, rows, bar);
    ptx::bulk_copy_g2s(dst + GB * CHI * 4, hb + (int64_t)c0 * CHI, rows, bar);
    ptx::bulk_copy_g2s(dst + 2 * GB * CHI * 4, fb + c0, fbytes, bar);
  };
  if (tid == 0)
    for (int g = 0; g < C::STAGES - 1 && g < nblk; ++g) issue(g);
  const int jg = tid % JG, kg = tid / JG;
  float acc0[KT][4], acc1[KT][4];
#pragma unroll
  for (int i = 0; i < KT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc0[i][j] = acc1[i][j] = 0.0f;
  for (int g = 0; g < nblk; ++g) {
    const int s = g % C::STAGES;
    const bool ok = ptx::mbar_wait(ptx::smem_addr(&full[s]), (g / C::STAGES) & 1, p.status);
    // every thread is done with block g - 1, whose stage takes block g + 2
    if (ptx::named_barrier_or(1, C::NT, !ok)) {
      if (tid == 0)  // let the copies in flight land before the CTA ends
        for (int u = g; u < min(nblk, g + C::STAGES - 1); ++u)
          ptx::mbar_wait(ptx::smem_addr(&full[u % C::STAGES]), (u / C::STAGES) & 1, p.status);
      return;
    }
    if (tid == 0 && g + C::STAGES - 1 < nblk) issue(g + C::STAGES - 1);
    const float* vs = smem + s * C::STAGE + kg * KT;
    const float* hs = smem + s * C::STAGE + GB * CHI + jr + jg * 4;
    const float2* fs = reinterpret_cast<const float2*>(smem + s * C::STAGE + 2 * GB * CHI);
    const int nb = min(GB, hi - lo - g * GB);
#pragma unroll 4
    for (int b = 0; b < nb; ++b) {
      const float2 f = fs[b];
      const float4 h4 = *reinterpret_cast<const float4*>(hs + b * CHI);
      const float x0[4] = {f.x * h4.x, f.x * h4.y, f.x * h4.z, f.x * h4.w};
      const float x1[4] = {f.y * h4.x, f.y * h4.y, f.y * h4.z, f.y * h4.w};
      float v[KT];
#pragma unroll
      for (int u = 0; u < KT / 4; ++u) {
        const float4 a = *reinterpret_cast<const float4*>(vs + b * CHI + u * 4);
        v[u * 4] = a.x;
        v[u * 4 + 1] = a.y;
        v[u * 4 + 2] = a.z;
        v[u * 4 + 3] = a.w;
      }
#pragma unroll
      for (int i = 0; i < KT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc0[i][j] = fmaf(v[i], x0[j], acc0[i][j]);
          acc1[i][j] = fmaf(v[i], x1[j], acc1[i][j]);
        }
    }
  }
  float* G = p.grad[half] + (size_t)(p.t_begin[half] + st) * CHI * 2 * CHI + jr + jg * 4;
#pragma unroll
  for (int i = 0; i < KT; ++i) {
    float* g = G + (size_t)(kg * KT + i) * 2 * CHI;
    atomicAdd(reinterpret_cast<float4*>(g), make_float4(acc0[i][0], acc0[i][1], acc0[i][2], acc0[i][3]));
    atomicAdd(reinterpret_cast<float4*>(g + CHI), make_float4(acc1[i][0], acc1[i][1], acc1[i][2], acc1[i][3]));
  }
}

template <int CHI>
int launch_grad(const ClsF32GradParams& p0, cudaStream_t s) {
  using C = GradCfg<CHI>;
  static std::atomic<uint64_t> attr{0};
  if (!smem_limit_once((const void*)cls_f32_grad_kernel<CHI>, C::SMEM, &attr)) return TN_ERR_CUDA;
  ClsF32GradParams p = p0;
  const int n0 = p.t_end[0] - p.t_begin[0], n1 = p.t_end[1] - p.t_begin[1], ny = n0 > n1 ? n0 : n1;
  if (ny <= 0) return TN_OK;
  // four CTAs share an SM: the batch is cut so that all tiles run as one such
  // wave (few cuts: each adds its whole tile to the gradient), a segment with
  // more tiles in four parts, so that the last wave is short
  const int jparts = CHI / C::JW, tiles = (n0 + n1) * jparts;
  const int room = 4 * sm_count();
  int want = tiles <= room ? room / tiles : 4;
  const int most = (p.batch + 127) / 128;
  if (want > most) want = most;
  p.chunk = ((p.batch + want - 1) / want + C::GB - 1) / C::GB * C::GB;
  const dim3 grid((unsigned)((p.batch + p.chunk - 1) / p.chunk), (unsigned)ny, 2 * (unsigned)jparts);
  cls_f32_grad_kernel<CHI><<<grid, C::NT, C::SMEM, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

}  // namespace

int cls_f32_pack(const ClsF32PackParams& p, cudaStream_t s) {
  const int steps = p.T[0] > p.T[1] ? p.T[0] : p.T[1];
  if (steps <= 0) return TN_OK;
  cls_f32_pack_kernel<<<dim3((unsigned)steps, 2), 256, 0, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

int cls_f32_sweep(int chi, int adjoint, const ClsF32Params& p, cudaStream_t s) {
  if (p.t_end[0] <= p.t_begin[0] && p.t_end[1] <= p.t_begin[1]) return TN_OK;
  if (chi == 32) return adjoint ? launch_sweep_chi<32, 1>(p, s) : launch_sweep_chi<32, 0>(p, s);
  if (chi == 64) return adjoint ? launch_sweep_chi<64, 1>(p, s) : launch_sweep_chi<64, 0>(p, s);
  return adjoint ? launch_sweep_chi<128, 1>(p, s) : launch_sweep_chi<128, 0>(p, s);
}

int cls_f32_grad(int chi, const ClsF32GradParams& p, cudaStream_t s) {
  if (chi == 32) return launch_grad<32>(p, s);
  if (chi == 64) return launch_grad<64>(p, s);
  return launch_grad<128>(p, s);
}

}  // namespace tn
