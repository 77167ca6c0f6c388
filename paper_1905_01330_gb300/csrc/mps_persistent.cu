// Persistent energy sweep: <psi|H|psi> and <psi|psi> of one MPS (Sec. II,
// Fig. 3a) in ONE cooperative launch for the whole chain. Every CTA stays
// resident from the first site to the last; the environment, its packed bf16
// image and the per-site intermediates stay in device memory that the 129 MB
// L2 holds at these bonds, and the sites' phases are separated by device-wide
// barriers instead of kernel launches:
//   (0) once: every site's core in the two operand layouts of (i) and (iii);
//   (B) tcgen05 GEMM  T1[(w, a'), (s, b)] = sum_a L[(w, a'), a] A[a, (s, b)],
//       and step (ii) of its tile straight into (iii)'s packed operand;
//   (D) tcgen05 GEMM  L'[(w', b), b'] = sum_{(a', s')} T2 A[(a', s'), b'],
//       packed as the next site's operand, with its largest magnitude.
// What bounds it: latency. A site of bond 256 is 0.7 us of tensor-core work,
// so its time is the chain of copies, MMAs, epilogue and barrier of the two
// phases. Hence:
//   - a tile of (i) holds every channel w of a group of a' (its rows are (w,
//     a' of the group)) and every s of its b (its columns are (16 b, s)), so
//     step (ii), which mixes (w, s), is local to the tile: T1 never leaves the
//     SM, and a phase, its barrier and 2 x 2 MB of traffic a site are gone;
//   - a tile has 128 rows and as few columns as a cost model of one phase
//     says (tile_cols): at bond 256 both phases make 64 units of work where
//     128 x 128 tiles made 32 and 16;
//   - copies and MMAs are issued by two warps: one thread issuing both took
//     2,000 cycles a slab of a narrow tile, of which the MMAs are 500;
//   - stores to the packed operands fill whole 32-byte sectors. Threads that
//     store 16 bytes of a row each took as long as the rest of the phase
//     (seen as 4,000 to 9,000 cycles of waiting in the barrier behind them).
// A site of bond 256 is now about 26,000 cycles (53,000 before): two barriers
// of 2,500 each, 9,000 of copies and MMAs, 3,500 of step (ii), 1,500 of packing,
// the rest the latencies at the head of a phase. Measured, N = 100, before ->
// now: BF16X3 bond 16 1.41 -> 0.78 ms, 64 1.74 -> 0.94, 256 2.81 -> 1.39, 512
// 3.95 -> 2.41; BF16 bond 256 2.30 -> 1.12 ms.
// A GEMM phase: CTA c takes units c, c + grid, ...; one thread streams the
// packed blocks of each 64-wide shared slab into a ring of shared-memory
// stages (1-D bulk copies), one issues the MMAs, eight warps drain the TMEM
// accumulator (double-buffered across units), four per half of its columns.
// BF16X3 issues hi*hi, hi*lo, lo*hi per step and promotes the accumulator
// into registers every 512 shared indices, as the grouped GEMM.
// Every wait (mbarriers and the device-wide barrier) is bounded; on expiry
// the status word records TN_ERR_TIMEOUT and every CTA winds down.
#include <string.h>

#include <algorithm>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

#include "mpo_step.cuh"
#include "packed.h"
#include "ptx.cuh"
#include "tn_internal.h"

namespace tn {
namespace {

constexpr int PS_THREADS = 384;  // 12 warps: warp 0 copies, warp 1 MMAs, warps 2, 3 zero fill, warps 4..11 drain TMEM
constexpr int PS_EPI0 = 4;       // first draining warp
constexpr int PS_EPI = 8;        // draining warps: two per TMEM lane quadrant, half of the columns each
constexpr int PS_GROUP = 128;    // threads of one half
constexpr int PS_KC = 8;         // BF16X3: slabs between promotions (512 shared indices)
constexpr int PS_BLOCK = 16384;  // one block of a first operand: 128 rows x 64 shared indices of bf16
constexpr int PS_MAX_SITES = 512;
constexpr int PS_MAX_STAGES = 8;
constexpr uint32_t PS_TMEM_COLS = 256;  // two accumulators of up to 128 columns
constexpr int PS_RING = 192 * 1024;     // the ring of stages
constexpr int PS_STAGED = 16 * 1024;    // T1 of a group's round: 128 rows (w, a') x d s x 8 or 16 b

// A site, with its two phases' tiles worked out on the host: one warp's
// divisions at the head of a phase are on the path of the whole sweep.
struct PsTiles {
  uint32_t off;    // the packed core at Cp + 1024 off
  uint32_t magic;  // u / tq = umulhi(u, magic) (0: tq = 1)
  uint16_t tp, tq; // row and column tiles
  int16_t cols;    // columns of a tile
  int16_t slabs;   // 64-wide slabs of the shared index
};
struct PsSite {
  const float* A;  // core (Da, d, Db), row-major
  uint32_t unit0;  // its first pack unit
  int32_t woff;    // its extended MPO at Wx + woff
  int16_t Da, Db;
  int8_t wa, wb;
  PsTiles t[2];    // (i), (iii)
};

struct PsParams {
  int32_t n, d;
  int32_t stages, stage_bytes;
  const float* Wx;       // extended MPO of every site
  float* L[2];           // the first environment and the last one
  uint8_t* Lp;           // packed L: rows (a' / G, w, a' % G), shared a (MN-major blocks)
  uint8_t* T2p;          // packed T2 for (iii): rows (w', b), shared a' d + s' (MN-major blocks)
  uint8_t* Cp;           // every site's packed cores (K-major blocks)
  int64_t Lp_lo, T2p_lo, Cp_lo;  // byte distance from a hi block to its lo block (BF16X3)
  uint32_t units;        // pack units of all the cores
  unsigned* bits;        // per site: bits of the largest |L| entering it
  double* lg;            // float64 log-scale
  unsigned* bar;         // device-wide barrier counter (zero at launch)
  double* result;        // {energy, log-scale, norm, log-scale}
  int* status;
  PsSite site[PS_MAX_SITES];
};

struct __align__(8) PsAux {
  uint64_t full[PS_MAX_STAGES];   // stage s holds its blocks
  uint64_t empty[PS_MAX_STAGES];  // the MMAs that read stage s are complete
  uint64_t acc_full[2];   // accumulator b holds a finished chunk
  uint64_t acc_empty[2];  // the draining warps have read accumulator b
  uint64_t final_bar;     // every MMA of the launch is complete
  uint32_t tmem_base;
  volatile int32_t abort;
  uint4 unit[2][2][4];      // batch, per half and parity of the unit: its chain's words,
  unsigned unit_max[2][4];  // the bits of the largest |L| entering, and the chain's number
  float4 Ws[2][8][4];     // per half: the site's W' as [(w, s)][(w', s') by reader], zero past the MPO
};

__device__ __forceinline__ uint32_t ld_acquire_gpu(const unsigned* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Device-wide barrier of the cooperative grid (all threads of every CTA):
// arrival `epoch` completes when the counter at `bar` reaches (epoch + 1) *
// gridDim.x. Writes before it are visible after it to every CTA's generic
// loads and to the bulk copies (async proxy) that read packed blocks.
// Bounded: after limit_ns of waiting the status word records TN_ERR_TIMEOUT,
// *abort is set and false is returned everywhere in this CTA (the CTAs that
// did arrive time out too and wind down).
__device__ bool grid_barrier(unsigned* bar, uint32_t& epoch, int* status, uint64_t limit_ns, volatile int32_t* abort) {
  fence_proxy_async_global();
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t target = (epoch + 1) * gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    if (ld_acquire_gpu(bar) < target) {
      const uint64_t t0 = ptx::globaltimer();
      for (uint32_t i = 1;; ++i) {
        if (ld_acquire_gpu(bar) >= target) break;
        if ((i & 63u) == 0u && ptx::globaltimer() - t0 > limit_ns) {
          ptx::set_status(status, TN_ERR_TIMEOUT);
          *abort = 1;
          break;
        }
      }
    }
    fence_proxy_async_global();
  }
  ++epoch;
  __syncthreads();
  return *abort == 0;
}

__device__ __forceinline__ bool grid_sync(const PsParams& p, uint32_t& epoch, PsAux& x) {
  return grid_barrier(p.bar, epoch, p.status, ptx::kWaitLimitNs, &x.abort);
}

// Failure-path check of the device-wide barrier: CTA 1 of a two-CTA
// cooperative launch leaves without arriving, so CTA 0's wait runs out.
__global__ void grid_barrier_timeout_kernel(unsigned* bar, int* status, uint64_t limit_ns) {
  __shared__ volatile int32_t abort;
  if (threadIdx.x == 0) abort = 0;
  __syncthreads();
  if (blockIdx.x != 0) return;
  uint32_t epoch = 0;
  grid_barrier(bar, epoch, status, limit_ns, &abort);
}

__device__ __forceinline__ uint32_t ps_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ int32_t ceil_div(int32_t a, int32_t b) { return (a + b - 1) / b; }

// Rows of (i)'s first operand a channel has in one 128-row tile: 2^shift, 128
// / wa rounded down to a power of two (wa <= 8: at least 16).
__host__ __device__ __forceinline__ int32_t group_shift(int32_t wa) { return wa <= 2 ? 6 : wa <= 4 ? 5 : 4; }
// b rounded up to whole cells of 16.
__host__ __device__ __forceinline__ int32_t pad16(int32_t x) { return (x + 15) & ~15; }

// hi (and lo) of 8 values as 16-byte chunks.
__device__ __forceinline__ void split8(const float* v, uint4& h, uint4& l) {
  h.x = ps_bf16x2(v[0], v[1]);
  h.y = ps_bf16x2(v[2], v[3]);
  h.z = ps_bf16x2(v[4], v[5]);
  h.w = ps_bf16x2(v[6], v[7]);
  const __nv_bfloat162* hb = reinterpret_cast<const __nv_bfloat162*>(&h);
  l.x = ps_bf16x2(v[0] - __low2float(hb[0]), v[1] - __high2float(hb[0]));
  l.y = ps_bf16x2(v[2] - __low2float(hb[1]), v[3] - __high2float(hb[1]));
  l.z = ps_bf16x2(v[4] - __low2float(hb[2]), v[5] - __high2float(hb[2]));
  l.w = ps_bf16x2(v[6] - __low2float(hb[3]), v[7] - __high2float(hb[3]));
}

// A site's core as the second operand of (i) or (iii): K-major blocks of
// `cols` rows x 64 shared indices (128-byte swizzle), one per tile of the
// result's columns and slab, zeros past the core. Row rho of (i) is (b / 16,
// s, b % 16), so a tile holds every s of its b; of (iii) it is b'.
struct PsPack {
  const float* src;
  uint8_t* hi;
  int64_t lo;  // byte distance to the lo plane, 0: none
  int32_t cols, slabs, K, Db, ns;  // ns: d for (i), 1 for (iii)
  int32_t run;  // (iii) with shared index (s', a'): Da, and the core rows run by d; else 0
  int32_t d;
};

__device__ __forceinline__ uint4 pick(bool c, const uint4& a, const uint4& b) {
  return make_uint4(c ? a.x : b.x, c ? a.y : b.y, c ? a.z : b.z, c ? a.w : b.w);
}
__device__ __forceinline__ uint4 swap_pair(const uint4& a) {
  return make_uint4(__shfl_xor_sync(0xffffffffu, a.x, 1), __shfl_xor_sync(0xffffffffu, a.y, 1),
                    __shfl_xor_sync(0xffffffffu, a.z, 1), __shfl_xor_sync(0xffffffffu, a.w, 1));
}

// One pack unit (a warp): 32 rows (b: the source's unit-stride index) of one
// slab; units numbered (tile, slab, rows / 32). Lanes 2i and 2i + 1 swap
// chunks, so that a pair's store is one 32-byte sector.
__device__ __forceinline__ void pack_unit(const PsPack& q, uint32_t u) {
  const int lane = threadIdx.x & 31, odd = lane & 1;
  const uint32_t parts = (uint32_t)q.cols >> 5, rest = u / parts;
  const int32_t t = (int32_t)(rest / (uint32_t)q.slabs), sl = (int32_t)(rest - (uint32_t)t * q.slabs);
  const int32_t rr = (int32_t)(u - rest * parts) * 32 + lane, rho = t * q.cols + rr;
  const int32_t cell = (rho >> 4) / q.ns, sk = (rho >> 4) - cell * q.ns, b = cell * 16 + (rho & 15);
  const int64_t ks = (int64_t)q.ns * q.Db;
  const int32_t k0 = sl * 64, kn = b < q.Db ? q.K - k0 : 0;
  const float* src = q.src + k0 * ks + (int64_t)sk * q.Db + b;
  uint8_t* blk = q.hi + ((size_t)t * q.slabs + sl) * (size_t)(q.cols * 128) + (size_t)(rr >> 3) * 1024;
  const int r0 = rr & 6;  // row of the pair's even lane, in its group of 8
  // the whole unit's loads before anything waits on one: beside a GEMM phase
  // each takes thousands of cycles
  float all[64];
  if (q.run == 0) {
#pragma unroll
    for (int j = 0; j < 64; ++j) all[j] = j < kn ? __ldg(src + j * ks) : 0.0f;
  } else {
    // k = s' Da + a': row a' d + s'
    int s1 = k0 / q.run, a1 = k0 - s1 * q.run;
#pragma unroll
    for (int j = 0; j < 64; ++j) {
      all[j] = j < kn ? __ldg(q.src + ((int64_t)a1 * q.d + s1) * q.Db + b) : 0.0f;
      if (++a1 == q.run) {
        a1 = 0;
        ++s1;
      }
    }
  }
#pragma unroll
  for (int g = 0; g < 8; g += 2) {
    const float* v = all + 8 * g;
    uint4 h[2], l[2];
    split8(v, h[0], l[0]);
    split8(v + 8, h[1], l[1]);
    const uint4 hs = swap_pair(pick(odd, h[0], h[1])), ls = swap_pair(pick(odd, l[0], l[1]));
    const int o0 = r0 * 128 + (((g + odd) ^ r0) << 4), o1 = (r0 + 1) * 128 + (((g + odd) ^ (r0 + 1)) << 4);
    *reinterpret_cast<uint4*>(blk + o0) = pick(odd, hs, h[0]);
    *reinterpret_cast<uint4*>(blk + o1) = pick(odd, h[1], hs);
    if (q.lo) {
      *reinterpret_cast<uint4*>(blk + q.lo + o0) = pick(odd, ls, l[0]);
      *reinterpret_cast<uint4*>(blk + q.lo + o1) = pick(odd, l[1], ls);
    }
  }
}

// Pack units of one of a site's cores.
__host__ __device__ __forceinline__ uint32_t pack_units(const PsTiles& t) {
  return (uint32_t)t.tq * (uint32_t)t.slabs * ((uint32_t)t.cols >> 5);
}

// One 16-byte chunk (8 rows at one shared index) of the first environment
// L[w, a, a'] as (i)'s first operand, zeros past it; chunks numbered (tile,
// slab, row group, k), k fastest.
__device__ __forceinline__ void pack_mn_chunk(const float* L, int32_t Da, int32_t wa, int32_t lg, int32_t slabs,
                                              uint8_t* hi, int64_t lo, int64_t e) {
  const int32_t kk = (int32_t)(e & 63);
  int64_t rest = e >> 6;
  const int32_t mg = (int32_t)(rest & 15);
  rest >>= 4;
  const int32_t sl = (int32_t)(rest % slabs), t = (int32_t)(rest / slabs);
  const int32_t k = sl * 64 + kk;
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int32_t r = mg * 8 + j, w = r >> lg, a2 = (t << lg) + r - (w << lg);
    v[j] = w < wa && a2 < Da && k < Da ? L[((int64_t)w * Da + k) * Da + a2] : 0.0f;
  }
  uint4 h, l;
  split8(v, h, l);
  const size_t off = ((size_t)t * slabs + sl) * PS_BLOCK + mn_block_chunk(mg, kk);
  *reinterpret_cast<uint4*>(hi + off) = h;
  if (lo) *reinterpret_cast<uint4*>(hi + lo + off) = l;
}

// Zeros at the shared indices [K, 64 slabs) of an MN-major operand (whole
// rows of its blocks): thread `tid` of `nthreads`.
__device__ __forceinline__ void zero_shared_tail(uint8_t* hi, int64_t lo, int32_t tiles, int32_t slabs, int32_t K,
                                                 int32_t tid, int32_t nthreads) {
  const int32_t npad = slabs * 64 - K, total = tiles * 16 * npad;
  for (int32_t e = tid; e < total; e += nthreads) {
    const int32_t mg = e & 15, rest = e >> 4;
    const int32_t t = rest / npad, kk = K + rest - t * npad;
    const size_t off = ((size_t)t * slabs + (kk >> 6)) * PS_BLOCK + mn_block_chunk(mg, kk & 63);
    *reinterpret_cast<uint4*>(hi + off) = make_uint4(0u, 0u, 0u, 0u);
    if (lo) *reinterpret_cast<uint4*>(hi + lo + off) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// One GEMM phase: C[r, c] = sum_k P[r, k] Q[c, k] over whole packed blocks (P
// MN-major, Q K-major), output tiles of 128 x cols.
struct PsGemm {
  const uint8_t* P;
  const uint8_t* Q;
  int64_t P_lo, Q_lo;  // byte distance from a hi block to its lo block (BF16X3)
  int32_t units, tq, slabs, cols;
  uint32_t magic;
};

// What the roles of a phase need of a unit.
struct UnitOps {  // the copies
  const uint8_t *P, *Q;
  int64_t P_lo, Q_lo;
  int32_t slabs, cols;
};
struct UnitShape {
  int32_t slabs, cols, tpi, tqi;
  bool cross;  // BF16X3: lo*hi before hi*lo
};

// The units of one chain's phase: CTA c takes c, c + grid, ...
struct OneUnits {
  const PsGemm& g;
  int u;
  __device__ __forceinline__ explicit OneUnits(const PsGemm& gg) : g(gg), u((int)blockIdx.x) {}
  __device__ __forceinline__ bool valid() const { return u < g.units; }
  __device__ __forceinline__ void advance() { u += (int)gridDim.x; }
  __device__ __forceinline__ UnitShape shape() const {
    UnitShape s;
    s.slabs = g.slabs;
    s.cols = g.cols;
    s.tpi = g.magic ? (int)__umulhi((uint32_t)u, g.magic) : u;
    s.tqi = u - s.tpi * g.tq;
    s.cross = false;
    return s;
  }
  __device__ __forceinline__ UnitOps ops() const {
    const UnitShape s = shape();
    return UnitOps{g.P + (size_t)s.tpi * g.slabs * PS_BLOCK, g.Q + (size_t)s.tqi * g.slabs * (size_t)(g.cols * 128),
                   g.P_lo, g.Q_lo, g.slabs, g.cols};
  }
  __device__ __forceinline__ void stage(int) const {}
};

// Pipeline positions kept across the phases of the launch: slabs through the
// stage ring (the copying thread's and the MMA issuer's own counts) and
// accumulator chunks (issuer and draining warps).
struct PsRing {
  int32_t stages, stage_bytes;
  int* status;
};
struct PsPipe {
  uint32_t slab, stage, phase, gc;  // phase: rounds of the ring, stage: slab % stages
};

// Copies of a GEMM phase (one thread): every slab of its units into the ring,
// as soon as its stage is free. A stage holds P hi, (P lo,) Q hi, (Q lo).
template <int SPLIT, class Units>
__device__ __forceinline__ bool gemm_copy(Units it, const PsRing& rg, uint32_t stage0, PsAux& x, PsPipe& pp) {
  const uint32_t S = (uint32_t)rg.stages, stage_bytes = (uint32_t)rg.stage_bytes, qoff = (SPLIT ? 2 : 1) * PS_BLOCK;
  uint32_t st = pp.stage, round = pp.phase;
  for (; it.valid(); it.advance()) {
    const UnitOps g = it.ops();
    const uint8_t *pb = g.P, *qb = g.Q;
    const uint32_t qbytes = (uint32_t)g.cols * 128u;
    for (int ks = 0; ks < g.slabs; ++ks, pb += PS_BLOCK, qb += qbytes) {
      // the stage's previous contents: read by MMAs that must be complete
      if (round && !ptx::mbar_wait(ptx::smem_addr(&x.empty[st]), (round - 1u) & 1u, rg.status)) return false;
      const uint32_t full = ptx::smem_addr(&x.full[st]), dst = stage0 + st * stage_bytes;
      ptx::mbar_arrive_expect_tx(full, (SPLIT ? 2u : 1u) * (PS_BLOCK + qbytes));
      ptx::bulk_copy_g2s(dst, pb, PS_BLOCK, full);
      ptx::bulk_copy_g2s(dst + qoff, qb, qbytes, full);
      if (SPLIT) {
        ptx::bulk_copy_g2s(dst + PS_BLOCK, pb + g.P_lo, PS_BLOCK, full);
        ptx::bulk_copy_g2s(dst + qoff + qbytes, qb + g.Q_lo, qbytes, full);
      }
      ++pp.slab;
      if (++st == S) {
        st = 0;
        ++round;
      }
    }
  }
  pp.stage = st;
  pp.phase = round;
  return true;
}

// MMAs of a GEMM phase, by a warp of its own (copies and MMAs issued by one
// thread took it 2,000 cycles a slab, the MMAs themselves 500): the warp runs
// the loop together and one lane issues, so that the descriptors stay in
// uniform registers.
template <int SPLIT, class Units>
__device__ __forceinline__ bool gemm_issue(Units it, const PsRing& rg, uint32_t stage0, PsAux& x, uint32_t tmem,
                                           PsPipe& pp) {
  const uint32_t S = (uint32_t)rg.stages, stage_bytes = (uint32_t)rg.stage_bytes, qoff = (SPLIT ? 2 : 1) * PS_BLOCK;
  int* status = rg.status;
  uint32_t st = pp.stage, phase = pp.phase;
  auto wait_full = [&]() {
    const bool w = ptx::mbar_wait(ptx::smem_addr(&x.full[st]), phase, status);
    if (!__all_sync(0xffffffffu, w)) return false;
    ptx::tc_fence_after();
    return true;
  };
  for (; it.valid(); it.advance()) {
    const UnitShape g = it.shape();
    const uint32_t idesc = ptx::idesc_bf16_f32(128, g.cols, 1, 0), qbytes = (uint32_t)g.cols * 128u;
    const int nks = g.slabs, chunk = SPLIT ? PS_KC : nks;
    for (int k0 = 0; k0 < nks; k0 += chunk) {
      // the accumulator this chunk overwrites has been drained
      const uint32_t b = pp.gc & 1u, dt = tmem + b * 128u;
      const bool w = ptx::mbar_wait(ptx::smem_addr(&x.acc_empty[b]), ((pp.gc >> 1) & 1u) ^ 1u, status);
      if (!__all_sync(0xffffffffu, w)) return false;
      const int k1 = min(k0 + chunk, nks);
      if (!wait_full()) return false;
      for (int ks = k0; ks < k1; ++ks) {
        const uint32_t sa = stage0 + st * stage_bytes, empty = ptx::smem_addr(&x.empty[st]);
        const uint32_t ph = ptx::desc_lo(sa, 8192), pl = ph + (PS_BLOCK >> 4);
        const uint32_t qh = ptx::desc_lo(sa + qoff), ql = qh + (qbytes >> 4);
        auto step = [&](int kk) {
          ptx::mma_bf16_lo(dt, ph + kk * 128u, qh + kk * 2u, idesc, (ks != k0 || kk != 0) ? 1u : 0u);
          if (SPLIT) {
            const uint32_t c0 = g.cross ? pl : ph, d0 = g.cross ? qh : ql;
            const uint32_t c1 = g.cross ? ph : pl, d1 = g.cross ? ql : qh;
            ptx::mma_bf16_lo(dt, c0 + kk * 128u, d0 + kk * 2u, idesc, 1u);
            ptx::mma_bf16_lo(dt, c1 + kk * 128u, d1 + kk * 2u, idesc, 1u);
          }
        };
        if (ptx::elect_one()) {
          step(0);
          step(1);
        }
        __syncwarp();
        if (++st == S) {
          st = 0;
          phase ^= 1u;
        }
        // the tensor pipe's queue is short: the next slab is waited for (200
        // cycles when it is there) behind half of this one's MMAs
        const bool more = ks + 1 < k1;
        if (more && !wait_full()) return false;
        if (ptx::elect_one()) {
          step(2);
          step(3);
          ptx::mma_commit(empty);
          if (!more) ptx::mma_commit(ptx::smem_addr(&x.acc_full[b]));
        }
        __syncwarp();
      }
      ++pp.gc;
    }
  }
  pp.stage = st;
  pp.phase = phase;
  return true;
}

// Draining warps of a GEMM phase: warp (PS_EPI0 + 4 half + quad) reads TMEM
// lanes quad * 32 .. + 31 (one result row per thread) of its half of the
// columns (ng = cols / 32 groups of 16); BF16X3 adds each chunk's partial
// sums into float32 registers. fin(row tile, column tile, values) finishes a
// unit; it is entered by a whole half together, and a wait that ran out in one
// of its warps ends all four.
template <int SPLIT, class Units, class Fin>
__device__ __forceinline__ bool gemm_drain(Units it, PsAux& x, uint32_t tmem, PsPipe& pp, int* status, Fin fin) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quad = warp & 3, half = (warp - PS_EPI0) >> 2;
  for (int i = 0; it.valid(); it.advance(), ++i) {
    const UnitShape g = it.shape();
    const int ng = g.cols >> 5;
    const int nks = g.slabs, nchunks = SPLIT ? (nks + PS_KC - 1) / PS_KC : 1;
    it.stage(i & 1);
    float acc[64];
#pragma unroll
    for (int j = 0; j < 64; ++j) acc[j] = 0.0f;
    for (int c = 0; c < nchunks; ++c) {
      const uint32_t b = pp.gc & 1u;
      const bool w = ptx::mbar_wait(ptx::smem_addr(&x.acc_full[b]), (pp.gc >> 1) & 1u, status);
      if (ptx::named_barrier_or(1 + half, PS_GROUP, !w)) return false;
      ptx::tc_fence_after();
      const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + b * 128u + (uint32_t)(half * ng * 16);
#pragma unroll
      for (int gi = 0; gi < 4; ++gi) {
        if (gi < ng) {
          uint32_t r[16];
          ptx::tmem_ld_32x32b_x16(ta + 16u * gi, r);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (SPLIT) acc[16 * gi + j] += __uint_as_float(r[j]);
            else acc[16 * gi + j] = __uint_as_float(r[j]);
          }
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&x.acc_empty[b]));
      ++pp.gc;
    }
    fin(g.tpi, g.tqi, i & 1, acc);
  }
  return true;
}

// What the draining warps make of a tile of (i): step (ii), T2[w', s', a', b]
// = 2^-e sum_{w, s} W'[w, w', s, s'] T1[w, a', s, b], into (iii)'s packed
// operand. A half goes through its columns in rounds of bw = 16 b (d <= 2) or
// 8 b: T1 of the round to shared memory, row (w, s, a') of bw floats; then a
// thread takes 8 b of one a' and every ms-th output channel, four at a time.
// Neighbouring lanes take the two halves of 16 b: whole 32-byte sectors.
struct PsStepII {
  uint8_t* hi;   // packed T2
  int64_t lo;    // byte distance to the lo plane, 0: none
  float inv;     // 2^-e
  int32_t Da, Db, DbP, wa, wb, d, slabs, lg;
  int32_t ps, pa;  // shared index of (iii): s' ps + a' pa
  uint32_t rd;   // m / d = m * rd >> 16 (m < 8)
};

template <int HR>  // rounds of 8 HR columns
__device__ __forceinline__ void step_ii_rounds(const PsStepII& q, const float4 (*Ws)[4], uint8_t* staged, int half,
                                               int cells, int tpi, int tqi, const float* acc) {
  const int tid = (threadIdx.x - PS_EPI0 * 32) & (PS_GROUP - 1);
  const int lg = q.lg, d = q.d, wad = q.wa * d, wbd = q.wb * d;
  const int rw = tid >> lg, ra = tid - (rw << lg);  // this thread's T1 row (w, a')
  constexpr int CH = 2 * HR;                  // 16-byte chunks of a staged row
  auto slot = [&](int k, int a, int c) -> uint8_t* {
    const int sw = HR == 2 ? (a >> 1) & 3 : (a >> 2) & 1;
    return staged + (((k << lg) + a) * CH + (c ^ sw)) * 16;
  };
  const int ib = HR == 2 ? tid & 1 : 0, rest = tid / HR, mh = rest >> lg, ia = rest - (mh << lg);
  const int ms = (PS_GROUP / HR) >> lg, kst = CH * 16 << lg;
  const int a = (tpi << lg) + ia;
  for (int c = 0; c < cells; ++c) {
    const int b0 = (((tqi * 2 + half) * cells) + c) * 16;
    if (b0 >= q.Db) break;
#pragma unroll
    for (int hb = 0; hb < 2; hb += HR) {
      // the group's readers of the previous round are done
      ptx::named_barrier(1 + half, PS_GROUP);
#pragma unroll
      for (int gi = 0; gi < 4; ++gi) {
        const int sk = gi - c * d;
        if (sk >= 0 && sk < d && rw < q.wa) {
#pragma unroll
          for (int ch = 0; ch < CH; ++ch) {
            const float* v = acc + 16 * gi + 8 * hb + 4 * ch;
            *reinterpret_cast<float4*>(slot(rw * d + sk, ra, ch)) = make_float4(v[0], v[1], v[2], v[3]);
          }
        }
      }
      ptx::named_barrier(1 + half, PS_GROUP);
      if (a < q.Da) {
        for (int m0 = mh; m0 < wbd; m0 += 4 * ms) {
          float2 o[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) o[i][j] = make_float2(0.0f, 0.0f);
          const uint8_t *row0 = slot(0, ia, 2 * ib), *row1 = slot(0, ia, 2 * ib + 1);
#pragma unroll 4
          for (int k = 0; k < wad; ++k) {
            const float4 t0 = *reinterpret_cast<const float4*>(row0 + k * kst);
            const float4 t1 = *reinterpret_cast<const float4*>(row1 + k * kst);
            const float2 t[4] = {{t0.x, t0.y}, {t0.z, t0.w}, {t1.x, t1.y}, {t1.z, t1.w}};
            const float4 w4 = Ws[k][ms == 1 ? m0 >> 2 : mh];
            const float wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) o[i][j] = __ffma2_rn(make_float2(wv[i], wv[i]), t[j], o[i][j]);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int m = m0 + i * ms;
            if (m >= wbd) break;
            float v[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              v[2 * j] = o[i][j].x * q.inv;
              v[2 * j + 1] = o[i][j].y * q.inv;
            }
            const int w2 = (int)((uint32_t)m * q.rd >> 16), s2 = m - w2 * d;
            const int32_t r0 = w2 * q.DbP + b0 + (hb + ib) * 8, kx = a * q.pa + s2 * q.ps;
            const size_t off = ((size_t)(r0 >> 7) * q.slabs + (kx >> 6)) * PS_BLOCK +
                               mn_block_chunk((r0 & 127) >> 3, kx & 63);
            uint4 h, l;
            split8(v, h, l);
            *reinterpret_cast<uint4*>(q.hi + off) = h;
            if (q.lo) *reinterpret_cast<uint4*>(q.hi + q.lo + off) = l;
          }
        }
      }
    }
  }
}

// What the draining warps make of a tile of (iii): rows (w', b) of L', columns
// b', packed as the next site's first operand of (i) (row (w', b') at shared
// index b) with the largest magnitude. Lanes 2i and 2i + 1 hold rows b and b +
// 1 and swap chunks, so that each store of the pair is one 32-byte sector.
struct PsNext {
  uint8_t* hi;
  int64_t lo;
  int32_t Db, DbP, wb, lg, slabs, cols;
};

__device__ __forceinline__ void pack_next(const PsNext& q, int half, int tpi, int tqi, const float* acc, float& mx) {
  const int lane = threadIdx.x & 31, quad = (threadIdx.x >> 5) & 3, ng = q.cols >> 5;
  const int row = tpi * 128 + quad * 32 + lane, odd = lane & 1;
  const int wq = row / q.DbP, b = row - wq * q.DbP, b0 = b & ~1;
  const bool live = wq < q.wb, valid = live && b < q.Db;  // DbP is even: the pair has one w'
#pragma unroll
  for (int gi = 0; gi < 4; ++gi) {
    const int cb = tqi * q.cols + (half * ng + gi) * 16;
    if (gi < ng && cb < q.Db) {
      const float* v = acc + 16 * gi;
      uint4 h[2], l[2];
      split8(v, h[0], l[0]);
      split8(v + 8, h[1], l[1]);
      if (valid) {
#pragma unroll
        for (int j = 0; j < 16; ++j) mx = fmaxf(mx, fabsf(v[j]));
      }
      const int t = cb >> q.lg, mg = ((wq << q.lg) + cb - (t << q.lg)) >> 3;
      uint8_t* blk = q.hi + (size_t)t * q.slabs * PS_BLOCK;
      const size_t o0 = (size_t)(b0 >> 6) * PS_BLOCK + mn_block_chunk(mg + odd, b0 & 63);
      const size_t o1 = (size_t)(b0 >> 6) * PS_BLOCK + mn_block_chunk(mg + odd, (b0 + 1) & 63);
      // chunk `odd` of rows b0 (o0) and b0 + 1 (o1)
      const uint4 hs = swap_pair(pick(odd, h[0], h[1])), ls = swap_pair(pick(odd, l[0], l[1]));
      if (live && b0 < q.Db) {
        *reinterpret_cast<uint4*>(blk + o0) = pick(odd, hs, h[0]);
        if (q.lo) *reinterpret_cast<uint4*>(blk + q.lo + o0) = pick(odd, ls, l[0]);
      }
      if (live && b0 + 1 < q.Db) {
        *reinterpret_cast<uint4*>(blk + o1) = pick(odd, h[1], hs);
        if (q.lo) *reinterpret_cast<uint4*>(blk + q.lo + o1) = pick(odd, l[1], ls);
      }
    }
  }
}

// Copies still in flight land, every MMA completes, then TMEM is freed.
__device__ __forceinline__ void wind_down(PsAux& x, const PsPipe& pp, const PsRing& rg, uint32_t tmem) {
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    const uint32_t S = (uint32_t)rg.stages;
    for (uint32_t q = pp.slab < S ? 0u : pp.slab - S; q < pp.slab; ++q)
      ptx::mbar_wait(ptx::smem_addr(&x.full[q % S]), (q / S) & 1u, rg.status);
  }
  __syncwarp();
  if (warp == 1) {
    if (ptx::elect_one()) ptx::mma_commit(ptx::smem_addr(&x.final_bar));  // the lane that issued the MMAs
    __syncwarp();
    ptx::mbar_wait(ptx::smem_addr(&x.final_bar), 0u, rg.status);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, PS_TMEM_COLS);
  }
}

// Each half's copy of W' (its readers wait at the half's barriers), by the
// order step_ii_rounds reads it: the four channels m of a thread's pass (m =
// mh, mh + ms, ...) as one 16-byte word.
__device__ __forceinline__ void load_site_mpo(const float* W, int wa, int wb, int d, PsAux& x, int half) {
  const int tid = threadIdx.x - PS_EPI0 * 32, lms = (d <= 2 ? 6 : 7) - group_shift(wa);
  if ((tid & (PS_GROUP - 1)) >= 64) return;
  const int k = (tid >> 3) & 7, m = tid & 7;
  float v = 0.0f;
  if (k < wa * d && m < wb * d) {
    const int w = k / d, sk = k - w * d, w2 = m / d, s2 = m - w2 * d;
    v = __ldg(W + ((w * wb + w2) * d + sk) * d + s2);
  }
  float* row = reinterpret_cast<float*>(x.Ws[half][k]);
  row[lms == 0 ? m : (m & ((1 << lms) - 1)) * 4 + (m >> lms)] = v;
  if (lms == 2) row[(m & 3) * 4 + 2 + (m >> 2)] = 0.0f;
}

// The whole sweep. Grid: one CTA per SM (cooperative launch).
template <int SPLIT>
__global__ void __launch_bounds__(PS_THREADS, 1) expect_persistent_kernel(const __grid_constant__ PsParams p) {
  extern __shared__ uint8_t ps_smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ps_smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* staged = smem + PS_RING;
  PsAux& x = *reinterpret_cast<PsAux*>(staged + 2 * PS_STAGED);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int st = 0; st < p.stages; ++st) {
      ptx::mbar_init(ptx::smem_addr(&x.full[st]), 1);   // the producer's transaction arrival
      ptx::mbar_init(ptx::smem_addr(&x.empty[st]), 1);  // the MMA issuer's commit
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_addr(&x.acc_full[b]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.acc_empty[b]), PS_EPI);
    }
    ptx::mbar_init(ptx::smem_addr(&x.final_bar), 1);
    x.abort = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_addr(&x.tmem_base), PS_TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = x.tmem_base, stage0 = ptx::smem_addr(smem);
  const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, gstride = (int64_t)gridDim.x * blockDim.x;
  const int32_t d = p.d, half = (warp - PS_EPI0) >> 2;
  const int64_t Lp_lo = SPLIT ? p.Lp_lo : 0, T2p_lo = SPLIT ? p.T2p_lo : 0;
  PsPipe pp{0u, 0u, 0u, 0u};
  const PsRing rg{p.stages, p.stage_bytes, p.status};
  uint32_t epoch = 0;
  // (0) every site's core in the two operand layouts, and the first
  // environment (1 in each channel) as the first site's operand
  for (uint32_t e = blockIdx.x * (PS_THREADS / 32) + warp; e < p.units; e += gridDim.x * (PS_THREADS / 32)) {
    int lo = 0, hi = p.n - 1;  // the site whose units hold e
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (p.site[mid].unit0 <= e) lo = mid;
      else hi = mid - 1;
    }
    const PsSite& st = p.site[lo];
    uint32_t k = e - st.unit0;
    const uint32_t c1 = pack_units(st.t[0]);
    const int third = k >= c1;
    if (third) k -= c1;
    const PsTiles& tt = st.t[third];
    pack_unit(PsPack{st.A, p.Cp + (size_t)tt.off * 1024, p.Cp_lo, tt.cols, tt.slabs, third ? d * st.Da : st.Da, st.Db,
                     third ? 1 : d, 0, d},
              k);
  }
  {
    const PsSite& s0 = p.site[0];
    const int32_t lg = group_shift(s0.wa), tiles = s0.t[0].tp, slabs = s0.t[0].slabs;
    for (int64_t e = gtid; e < (int64_t)tiles * slabs * 16 * 64; e += gstride)
      pack_mn_chunk(p.L[0], s0.Da, s0.wa, lg, slabs, p.Lp, Lp_lo, e);
  }
  bool ok = grid_sync(p, epoch, x);
  for (int i = 0; i < p.n && ok; ++i) {
    const PsSite& st = p.site[i];
    const int32_t Da = st.Da, Db = st.Db, wa = st.wa, wb = st.wb, DbP = pad16(Db);
    const int32_t slabs3 = st.t[1].slabs;
    // (B) T1 and, from its tiles, T2 = 2^-e W' T1
    PsGemm g;
    auto tiles = [&](const PsTiles& t) {
      g.Q = p.Cp + (size_t)t.off * 1024;
      g.units = (int32_t)t.tp * t.tq;
      g.tq = t.tq;
      g.slabs = t.slabs;
      g.cols = t.cols;
      g.magic = t.magic;
    };
    tiles(st.t[0]);
    g.P = p.Lp;
    g.P_lo = p.Lp_lo;
    g.Q_lo = p.Cp_lo;
    if (threadIdx.x == 0) {
      if (!gemm_copy<SPLIT>(OneUnits(g), rg, stage0, x, pp)) x.abort = 1;
    } else if (warp == 1) {
      if (!gemm_issue<SPLIT>(OneUnits(g), rg, stage0, x, tmem, pp)) x.abort = 1;
    } else if (warp >= PS_EPI0) {
      const int tid = threadIdx.x - PS_EPI0 * 32;
      load_site_mpo(p.Wx + st.woff, wa, wb, d, x, half);
      const int lg = group_shift(wa);
      int e = 0;
      if (i > 0) e = pow2_exponent(__uint_as_float(__ldcg(p.bits + i)));
      if (i > 0 && blockIdx.x == 0 && tid == 0) *p.lg += (double)e * 0.69314718055994530942;
      PsStepII q;
      q.hi = p.T2p;
      q.lo = T2p_lo;
      q.inv = __int_as_float((127 - e) << 23);
      q.Da = Da;
      q.Db = Db;
      q.DbP = DbP;
      q.wa = wa;
      q.wb = wb;
      q.d = d;
      q.slabs = slabs3;
      q.lg = lg;
      q.ps = 1;
      q.pa = d;
      q.rd = (uint32_t)(65536 + d - 1) / (uint32_t)d;
      const int cells = (int)((uint32_t)(g.cols >> 5) * q.rd >> 16);
      uint8_t* mine = staged + half * PS_STAGED;
      const bool done = gemm_drain<SPLIT>(OneUnits(g), x, tmem, pp, p.status, [&](int tpi, int tqi, int, const float* acc) {
        if (d <= 2) step_ii_rounds<2>(q, x.Ws[half], mine, half, cells, tpi, tqi, acc);
        else step_ii_rounds<1>(q, x.Ws[half], mine, half, cells, tpi, tqi, acc);
      });
      if (!done) x.abort = 1;
    } else if (warp >= 2) {
      zero_shared_tail(p.T2p, T2p_lo, st.t[1].tp, slabs3, d * Da, blockIdx.x * 64 + threadIdx.x - 64, gridDim.x * 64);
    }
    if (!(ok = grid_sync(p, epoch, x))) break;
    // (D) L'[(w', b), b'] = sum_{(a', s')} T2[(w', b), (a', s')] A[(a', s'), b']
    tiles(st.t[1]);
    g.P = p.T2p;
    g.P_lo = p.T2p_lo;
    const bool last = i + 1 == p.n;
    const int32_t slabsn = ceil_div(Db, 64);
    if (threadIdx.x == 0) {
      if (!gemm_copy<SPLIT>(OneUnits(g), rg, stage0, x, pp)) x.abort = 1;
    } else if (warp == 1) {
      if (!gemm_issue<SPLIT>(OneUnits(g), rg, stage0, x, tmem, pp)) x.abort = 1;
    } else if (warp >= PS_EPI0) {
      float mx = 0.0f;
      PsNext q;
      q.hi = p.Lp;
      q.lo = Lp_lo;
      q.Db = Db;
      q.DbP = DbP;
      q.wb = wb;
      q.lg = group_shift(wb);
      q.slabs = slabsn;
      q.cols = g.cols;
      const bool done = gemm_drain<SPLIT>(OneUnits(g), x, tmem, pp, p.status, [&](int tpi, int tqi, int, const float* acc) {
        if (!last) {
          pack_next(q, half, tpi, tqi, acc, mx);
        } else if (tqi == 0 && half == 0) {
          // Db = 1: the last environment, one value per channel
          const int row = tpi * 128 + (warp & 3) * 32 + lane, wq = row / DbP;
          if (wq < wb && row == wq * DbP) p.L[1][wq] = acc[0];
        }
      });
      if (!done) x.abort = 1;
      if (!last) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0 && mx > 0.0f) atomicMax(p.bits + i + 1, __float_as_uint(mx));
      }
    } else if (warp >= 2 && !last) {
      zero_shared_tail(p.Lp, Lp_lo, ceil_div(Db, 1 << group_shift(wb)), slabsn, Db, blockIdx.x * 64 + threadIdx.x - 64, gridDim.x * 64);
    }
    if (!(ok = grid_sync(p, epoch, x))) break;
  }
  if (ok && blockIdx.x == 0 && threadIdx.x == 0) {
    const float* L = p.L[1];
    p.result[0] = (double)__ldcg(L);
    p.result[1] = __ldcg(p.lg);
    p.result[2] = (double)__ldcg(L + 1);
    p.result[3] = __ldcg(p.lg);
  }
  wind_down(x, pp, rg, tmem);
}

// ------------------------------------------------------------ many chains
// The same sweep for a batch of chains with one MPO: every phase works on the
// units of all of them, in lists the host made (largest first, each to the CTA
// with the least so far), so the device-wide barriers, the copies' latency
// and the ragged tiles of a site are shared. Warps 2 and 3 pack the next
// site's cores meanwhile, into the other of two regions. Sums run in the order
// of the grouped contractions: (iii)'s shared index is (s', a'), and where
// those would have the core as the first operand of (i) the cross terms of
// BF16x3 swap places.
struct PbChain {   // a chain at a site
  const float* A;  // core (Da, d, Db), row-major
  uint32_t unit0;  // its first pack unit of the site
  int16_t Da, Db;
  PsTiles t[2];    // (i), (iii); off: in the site's region
  uint32_t lp, lp_lo, t2, t2_lo;  // packed L and T2 (hi planes and distances to lo), in 1024 bytes
};
static_assert(sizeof(PbChain) == 64, "loaded as four 16-byte words");

struct PbUnit {
  uint16_t chain;
  uint8_t tpi, tqi, slabs, cols16, cross, pad;
};
static_assert(sizeof(PbUnit) == 8, "");

struct PbParams {
  int32_t n, d, count;
  int32_t stages, stage_bytes;
  const float* Wx;
  uint8_t* base;          // of the packed regions
  uint8_t* Cp[2];         // packed cores of a site (even, odd)
  int64_t Cp_lo;
  const PbChain* chains;  // [site][chain]
  const PbUnit* units;
  const int32_t* first;   // [site][phase][CTA]: its first unit; one more: the end
  float* const* last;     // per chain: its last environment (one value per channel)
  unsigned* bits;         // [site - 1][chain]: largest |L| entering the site
  double* lg;
  unsigned* bar;
  int* status;
  int32_t woff[PS_MAX_SITES];
  uint32_t pack[PS_MAX_SITES];  // pack units of the site
  int8_t w[PS_MAX_SITES + 1];   // extended MPO bonds
};

// This CTA's units of a phase.
struct ListUnits {
  const PbUnit* u;
  const PbUnit* end;
  const PbChain* chains;
  const PbParams& p;
  int phase, site;
  uint4 (*slot)[4];      // draining half: the chain's words, for fin
  unsigned* slot_max;
  uint2 cur;
  __device__ __forceinline__ ListUnits(const PbParams& pp, int st, int ph, uint4 (*sl)[4] = nullptr,
                                       unsigned* mx = nullptr)
      : p(pp), phase(ph), site(st), slot(sl), slot_max(mx) {
    const int32_t* f = pp.first + ((size_t)st * 2 + ph) * (gridDim.x + 1) + blockIdx.x;
    u = pp.units + __ldg(f);
    end = pp.units + __ldg(f + 1);
    chains = pp.chains + (size_t)st * pp.count;
    load();
  }
  __device__ __forceinline__ void load() {
    cur = u < end ? __ldg(reinterpret_cast<const uint2*>(u)) : make_uint2(0u, 0u);
  }
  __device__ __forceinline__ bool valid() const { return u < end; }
  __device__ __forceinline__ void advance() {
    ++u;
    load();
  }
  __device__ __forceinline__ UnitShape shape() const {
    return UnitShape{(int32_t)(cur.y & 0xFF), (int32_t)((cur.y >> 8) & 0xFF) * 16, (int32_t)((cur.x >> 16) & 0xFF),
                     (int32_t)(cur.x >> 24), ((cur.y >> 16) & 1) != 0};
  }
  __device__ __forceinline__ UnitOps ops() const {
    const UnitShape s = shape();
    const uint4* c = reinterpret_cast<const uint4*>(chains + (cur.x & 0xFFFF));
    const uint4 r = __ldg(c + 3);                       // lp, lp_lo, t2, t2_lo
    const uint32_t off = __ldg(&chains[cur.x & 0xFFFF].t[phase].off);
    const size_t P = (size_t)(phase ? r.z : r.x) * 1024;
    return UnitOps{p.base + P + (size_t)s.tpi * s.slabs * PS_BLOCK,
                   p.Cp[site & 1] + (size_t)off * 1024 + (size_t)s.tqi * s.slabs * (size_t)(s.cols * 128),
                   (int64_t)(phase ? r.w : r.y) * 1024, p.Cp_lo, s.slabs, s.cols};
  }
  // the chain's words into the half's slot (the half's barrier before fin makes them visible)
  __device__ __forceinline__ void stage(int which) const {
    const int t = threadIdx.x & (PS_GROUP - 1), k = (int)(cur.x & 0xFFFF);
    if (t < 4) slot[which][t] = __ldg(reinterpret_cast<const uint4*>(chains + k) + t);
    if (t == 4) slot_max[2 * which] = site > 0 ? __ldcg(p.bits + (size_t)(site - 1) * p.count + k) : 0u;
    if (t == 5) slot_max[2 * which + 1] = (unsigned)k;
  }
};

// Pack units [e0, e1) of a site's cores, by `nwarps` warps.
__device__ __forceinline__ void pack_site(const PbParams& p, int site, uint32_t e0, uint32_t e1, uint32_t wid,
                                          uint32_t nwarps) {
  const PbChain* chains = p.chains + (size_t)site * p.count;
  int lo = -1, lane = threadIdx.x & 31;  // the chain whose units hold e: e only grows
  for (uint32_t e = e0 + wid; e < e1; e += nwarps) {
    for (;;) {  // 32 chains a look: those whose first unit is not past e
      const int at = lo + 1 + lane;
      const unsigned m = __ballot_sync(0xffffffffu, at < p.count && __ldg(&chains[at].unit0) <= e);
      lo += __popc(m);
      if (m != 0xffffffffu) break;
    }
    const PbChain& c = chains[lo];
    uint32_t k = e - c.unit0;
    const uint32_t c1 = pack_units(c.t[0]);
    const int third = k >= c1;
    if (third) k -= c1;
    const PsTiles& tt = c.t[third];
    pack_unit(PsPack{c.A, p.Cp[site & 1] + (size_t)tt.off * 1024, p.Cp_lo, tt.cols, tt.slabs,
                     third ? p.d * c.Da : c.Da, c.Db, third ? 1 : p.d, third ? c.Da : 0, p.d},
              k);
  }
}

template <int SPLIT>
__global__ void __launch_bounds__(PS_THREADS, 1) expect_batch_kernel(const __grid_constant__ PbParams p) {
  extern __shared__ uint8_t ps_smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ps_smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* staged = smem + PS_RING;
  PsAux& x = *reinterpret_cast<PsAux*>(staged + 2 * PS_STAGED);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int st = 0; st < p.stages; ++st) {
      ptx::mbar_init(ptx::smem_addr(&x.full[st]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.empty[st]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_addr(&x.acc_full[b]), 1);
      ptx::mbar_init(ptx::smem_addr(&x.acc_empty[b]), PS_EPI);
    }
    ptx::mbar_init(ptx::smem_addr(&x.final_bar), 1);
    x.abort = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_addr(&x.tmem_base), PS_TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = x.tmem_base, stage0 = ptx::smem_addr(smem);
  const int32_t d = p.d, half = (warp - PS_EPI0) >> 2;
  PsPipe pp{0u, 0u, 0u, 0u};
  const PsRing rg{p.stages, p.stage_bytes, p.status};
  uint32_t epoch = 0;
  // (0) the first site's cores, and the first environments: 1 in each channel
  pack_site(p, 0, 0u, p.pack[0], blockIdx.x * (PS_THREADS / 32) + warp, gridDim.x * (PS_THREADS / 32));
  for (int c = blockIdx.x; c < p.count; c += gridDim.x) {
    const PbChain& ch = p.chains[c];
    uint8_t* hi = p.base + (size_t)ch.lp * 1024;
    const int lg = group_shift(p.w[0]);
    for (int e = threadIdx.x; e < 1024; e += PS_THREADS) {  // one block: row (w, 0) at shared index 0
      const int kk = e & 63, mg = e >> 6, w = (mg * 8) >> lg;
      const bool one = kk == 0 && w < p.w[0] && (w << lg) == mg * 8;
      *reinterpret_cast<uint4*>(hi + mn_block_chunk(mg, kk)) = make_uint4(one ? 0x3F80u : 0u, 0u, 0u, 0u);
      if (SPLIT) *reinterpret_cast<uint4*>(hi + (size_t)ch.lp_lo * 1024 + mn_block_chunk(mg, kk)) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  bool ok = grid_barrier(p.bar, epoch, p.status, ptx::kWaitLimitNs, &x.abort);
  const uint32_t bw = blockIdx.x * 2 + warp - 2, nbw = gridDim.x * 2;  // the packing warps
  for (int i = 0; i < p.n && ok; ++i) {
    const int32_t wa = p.w[i], wb = p.w[i + 1];
    const bool last = i + 1 == p.n;
    // (B) T1 and, from its tiles, T2 = 2^-e W' T1
    if (threadIdx.x == 0) {
      if (!gemm_copy<SPLIT>(ListUnits(p, i, 0), rg, stage0, x, pp)) x.abort = 1;
    } else if (warp == 1) {
      if (!gemm_issue<SPLIT>(ListUnits(p, i, 0), rg, stage0, x, tmem, pp)) x.abort = 1;
    } else if (warp >= PS_EPI0) {
      load_site_mpo(p.Wx + p.woff[i], wa, wb, d, x, half);
      uint8_t* mine = staged + half * PS_STAGED;
      const uint32_t rd = (uint32_t)(65536 + d - 1) / (uint32_t)d;
      const bool done = gemm_drain<SPLIT>(
          ListUnits(p, i, 0, x.unit[half], x.unit_max[half]), x, tmem, pp, p.status,
          [&](int tpi, int tqi, int which, const float* acc) {
            const PbChain& ch = *reinterpret_cast<const PbChain*>(x.unit[half][which]);
            const int e = i > 0 ? pow2_exponent(__uint_as_float(x.unit_max[half][2 * which])) : 0;
            // one unit of the chain adds the site's exponent to its log-scale
            if (i > 0 && tpi == 0 && tqi == 0 && threadIdx.x == PS_EPI0 * 32) {
              double* l = p.lg + x.unit_max[half][2 * which + 1];
              __stcg(l, __ldcg(l) + (double)e * 0.69314718055994530942);
            }
            PsStepII q;
            q.hi = p.base + (size_t)ch.t2 * 1024;
            q.lo = SPLIT ? (int64_t)ch.t2_lo * 1024 : 0;
            q.inv = __int_as_float((127 - e) << 23);
            q.Da = ch.Da;
            q.Db = ch.Db;
            q.DbP = pad16(ch.Db);
            q.wa = wa;
            q.wb = wb;
            q.d = d;
            q.slabs = ch.t[1].slabs;
            q.lg = group_shift(wa);
            q.ps = ch.Da;
            q.pa = 1;
            q.rd = rd;
            const int cells = (int)((uint32_t)(ch.t[0].cols >> 5) * rd >> 16);
            if (d <= 2) step_ii_rounds<2>(q, x.Ws[half], mine, half, cells, tpi, tqi, acc);
            else step_ii_rounds<1>(q, x.Ws[half], mine, half, cells, tpi, tqi, acc);
          });
      if (!done) x.abort = 1;
    } else if (warp >= 2) {
      for (int c = blockIdx.x; c < p.count; c += gridDim.x) {
        const PbChain& ch = p.chains[(size_t)i * p.count + c];
        zero_shared_tail(p.base + (size_t)ch.t2 * 1024, SPLIT ? (int64_t)ch.t2_lo * 1024 : 0, ch.t[1].tp,
                         ch.t[1].slabs, d * ch.Da, threadIdx.x - 64, 64);
      }
      if (!last) pack_site(p, i + 1, 0u, p.pack[i + 1] / 2, bw, nbw);
    }
    if (!(ok = grid_barrier(p.bar, epoch, p.status, ptx::kWaitLimitNs, &x.abort))) break;
    // (D) L' from T2 and the core
    if (threadIdx.x == 0) {
      if (!gemm_copy<SPLIT>(ListUnits(p, i, 1), rg, stage0, x, pp)) x.abort = 1;
    } else if (warp == 1) {
      if (!gemm_issue<SPLIT>(ListUnits(p, i, 1), rg, stage0, x, tmem, pp)) x.abort = 1;
    } else if (warp >= PS_EPI0) {
      const bool done = gemm_drain<SPLIT>(
          ListUnits(p, i, 1, x.unit[half], x.unit_max[half]), x, tmem, pp, p.status,
          [&](int tpi, int tqi, int which, const float* acc) {
            const PbChain& ch = *reinterpret_cast<const PbChain*>(x.unit[half][which]);
            const unsigned k = x.unit_max[half][2 * which + 1];
            PsNext q;
            q.hi = p.base + (size_t)ch.lp * 1024;
            q.lo = SPLIT ? (int64_t)ch.lp_lo * 1024 : 0;
            q.Db = ch.Db;
            q.DbP = pad16(ch.Db);
            q.wb = wb;
            q.lg = group_shift(wb);
            q.slabs = ceil_div(ch.Db, 64);
            q.cols = ch.t[1].cols;
            if (!last) {
              float mx = 0.0f;
              pack_next(q, half, tpi, tqi, acc, mx);
#pragma unroll
              for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
              if (lane == 0 && mx > 0.0f) atomicMax(p.bits + (size_t)i * p.count + k, __float_as_uint(mx));
            } else if (tqi == 0 && half == 0) {
              // Db = 1: the last environment, one value per channel
              const int row = tpi * 128 + (warp & 3) * 32 + lane, wq = row / q.DbP;
              if (wq < wb && row == wq * q.DbP) p.last[k][wq] = acc[0];
            }
          });
      if (!done) x.abort = 1;
    } else if (warp >= 2 && !last) {
      for (int c = blockIdx.x; c < p.count; c += gridDim.x) {
        const PbChain& ch = p.chains[(size_t)i * p.count + c];
        zero_shared_tail(p.base + (size_t)ch.lp * 1024, SPLIT ? (int64_t)ch.lp_lo * 1024 : 0,
                         ceil_div(ch.Db, 1 << group_shift(wb)), ceil_div(ch.Db, 64), ch.Db, threadIdx.x - 64, 64);
      }
      pack_site(p, i + 1, p.pack[i + 1] / 2, p.pack[i + 1], bw, nbw);
    }
    if (!(ok = grid_barrier(p.bar, epoch, p.status, ptx::kWaitLimitNs, &x.abort))) break;
  }
  wind_down(x, pp, rg, tmem);
}

}  // namespace

// Bytes of one plane (hi or lo) of an operand in blocks of `rows` rows.
size_t ps_bytes(int64_t tiles, int64_t K, int64_t rows) { return (size_t)tiles * (size_t)((K + 63) / 64) * (size_t)rows * 128; }

int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return 152;
  return sms;
}

int64_t ceil64(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Columns of a GEMM phase's tiles (step, 2 step, .. up to 128; step: the
// columns that must stay together in both halves, 32 d for (i), 32 for
// (iii)): the count that makes the phase shortest by a model of it, rounds of
// units over the SMs, each the copies of its slabs (32 KB of P and 256 bytes
// a column for BF16X3, at about 64 bytes a cycle; its MMAs, 40 to 64 cycles
// each whatever the width, take about as long) and its epilogue (about 20
// cycles a column). At bond 256 it takes 64 and 32 columns, 64 units in each
// phase; at 512 128 and 64.
int tile_cols(int64_t tp, int64_t total, int64_t K, int step, int64_t sms) {
  const int64_t slabs = ceil64(K, 64);
  int best = step;
  int64_t best_cost = INT64_MAX;
  for (int c = step; c <= 128; c *= 2) {
    const int64_t units = tp * ceil64(total, c);
    const int64_t cost = ceil64(units, sms) * (slabs * (512 + 4 * c) + 20 * c + 1000);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

// Tiles of a site's phases: first operands' row tiles and the columns.
struct SiteTiles {
  int64_t t1, t3;
  int n1, n3;
};
SiteTiles site_tiles(int64_t Da, int64_t Db, int64_t wa, int64_t wb, int64_t d, int64_t sms) {
  SiteTiles t;
  const int64_t DbP = pad16((int32_t)Db);
  t.t1 = ceil64(Da, int64_t(1) << group_shift((int32_t)wa));
  t.t3 = ceil64(wb * DbP, 128);
  t.n1 = tile_cols(t.t1, d * DbP, Da, (int)(32 * d), sms);
  t.n3 = tile_cols(t.t3, DbP, d * Da, 32, sms);
  return t;
}

ExpectRegions expect_persistent_regions(const tn_mps* psi, const tn_mpo* H) {
  ExpectRegions r{0, 0, 0};
  const int64_t sms = device_sms();
  const int64_t d = psi->d;
  for (int i = 0; i < psi->n; ++i) {
    const int64_t Da = psi->bond[i], Db = psi->bond[i + 1];
    const SiteTiles t = site_tiles(Da, Db, H->bond[i] + 1, H->bond[i + 1] + 1, d, sms);
    r.env = std::max(r.env, ps_bytes(t.t1, Da, 128));
    r.t2 = std::max(r.t2, ps_bytes(t.t3, d * Da, 128));
    const int64_t DbP = pad16((int32_t)Db);
    r.cores += ps_bytes(ceil64(d * DbP, t.n1), Da, t.n1) + ps_bytes(ceil64(DbP, t.n3), d * Da, t.n3);
  }
  r.env = align256(r.env);
  r.t2 = align256(r.t2);
  r.cores = align256(r.cores);
  return r;
}

// Raises a sweep kernel's shared-memory limit, once per device.
bool smem_limit_sweep(const void* fn, size_t smem) {
  static std::atomic<uint64_t> attr[4];
  const void* all[4] = {(const void*)expect_persistent_kernel<0>, (const void*)expect_persistent_kernel<1>,
                        (const void*)expect_batch_kernel<0>, (const void*)expect_batch_kernel<1>};
  for (int i = 0; i < 4; ++i)
    if (all[i] == fn) return smem_limit_once(fn, smem, &attr[i]);
  return false;
}

// One CTA per SM, all resident.
template <class P>
int launch_sweep(void (*fn)(const P), const P& p, cudaStream_t s) {
  const size_t smem = 1024 + (size_t)PS_RING + 2 * PS_STAGED + sizeof(PsAux);
  if (!smem_limit_sweep((const void*)fn, smem)) return TN_ERR_CUDA;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)fn, PS_THREADS, smem) != cudaSuccess ||
      per_sm < 1)
    return TN_ERR_UNSUPPORTED;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)device_sms());
  cfg.blockDim = dim3(PS_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, p) == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

bool expect_persistent_ok(const tn_mps* psi, const tn_mpo* H, int prec) {
  if (prec != TN_PREC_BF16 && prec != TN_PREC_BF16X3) return false;
  if (psi->n > PS_MAX_SITES) return false;
  for (int i = 0; i <= H->n; ++i)
    if ((H->bond[i] + 1) * psi->d > 8) return false;
  return true;
}

int expect_persistent(const tn_mps* psi, const tn_mpo* H, int prec, const ExpectBuffers& w, double* result,
                      cudaStream_t s) {
  if (!expect_persistent_ok(psi, H, prec)) return TN_ERR_UNSUPPORTED;
  const bool split = prec == TN_PREC_BF16X3;
  PsParams p;
  memset(&p, 0, sizeof(p));
  p.n = psi->n;
  p.d = (int32_t)psi->d;
  p.Wx = w.Wx;
  p.L[0] = w.L0;
  p.L[1] = w.L1;
  // packed regions (hi plane, then lo): L in scratch, T2 in scratch3, every
  // site's cores in cores
  const ExpectRegions need = expect_persistent_regions(psi, H);
  if (w.scratch_bytes < 2 * need.env || w.scratch3_bytes < 2 * need.t2 || w.cores_bytes < 2 * need.cores)
    return TN_ERR_WORKSPACE;
  const int64_t d = psi->d;
  p.Lp = w.scratch;
  p.Lp_lo = split ? (int64_t)need.env : 0;
  p.T2p = w.scratch3;
  p.T2p_lo = split ? (int64_t)need.t2 : 0;
  p.Cp = w.cores;
  p.Cp_lo = split ? (int64_t)need.cores : 0;
  p.bits = w.bits;
  p.lg = w.lg;
  p.bar = w.bar;
  p.result = result;
  p.status = status_word();
  // the cores' places, pack units and tiles, site by site
  size_t off = 0;
  uint32_t units = 0;
  int widest = 0;
  const int sms = device_sms();
  for (int i = 0; i < psi->n; ++i) {
    PsSite& st = p.site[i];
    const int64_t Da = psi->bond[i], Db = psi->bond[i + 1], DbP = pad16((int32_t)Db);
    st.A = psi->cores[i];
    st.Da = (int16_t)Da;
    st.Db = (int16_t)Db;
    st.wa = (int8_t)(H->bond[i] + 1);
    st.wb = (int8_t)(H->bond[i + 1] + 1);
    st.woff = (int32_t)w.woff[(size_t)i];
    st.unit0 = units;
    const SiteTiles t = site_tiles(Da, Db, st.wa, st.wb, d, sms);
    for (int j = 0; j < 2; ++j) {
      PsTiles& q = st.t[j];
      const int cols = j ? t.n3 : t.n1;
      const int64_t K = j ? d * Da : Da, tq = ceil64(j ? DbP : d * DbP, cols);
      q.off = (uint32_t)(off / 1024);
      q.tp = (uint16_t)(j ? t.t3 : t.t1);
      q.tq = (uint16_t)tq;
      q.magic = tq == 1 ? 0u : (uint32_t)(((uint64_t(1) << 32) + (uint64_t)tq - 1) / (uint64_t)tq);
      q.cols = (int16_t)cols;
      q.slabs = (int16_t)ceil64(K, 64);
      off += ps_bytes(tq, K, cols);
      units += pack_units(q);
      widest = std::max(widest, cols);
    }
  }
  p.units = units;
  p.stage_bytes = (split ? 2 : 1) * (PS_BLOCK + widest * 128);
  p.stages = std::min(PS_RING / p.stage_bytes, PS_MAX_STAGES);
  // the device-wide barrier counts arrivals from zero
  if (cudaMemsetAsync(w.bar, 0, sizeof(unsigned), s) != cudaSuccess) return TN_ERR_CUDA;
  return split ? launch_sweep(expect_persistent_kernel<1>, p, s) : launch_sweep(expect_persistent_kernel<0>, p, s);
}

// ------------------------------------------------------------ many chains
namespace {

// Cycles of a unit: its copies and MMAs as in tile_cols; the epilogue of (i),
// step (ii), about as long as 8 slabs of a 128-column tile, overlaps the next
// unit's.
double unit_cost(int slabs, int cols, int phase) {
  const double gemm = slabs * (512.0 + 4.0 * cols);
  return phase == 0 ? std::max(gemm, 90.0 * cols) + 1000.0 : gemm + 20.0 * cols + 1000.0;
}

// Columns of a tile when many chains share the SMs: the least padded work.
int batch_cols(int64_t total, int64_t K, int step, int phase) {
  int best = step;
  double best_cost = 1e30;
  for (int c = step; c <= 128; c *= 2) {
    const double cost = (double)ceil64(total, c) * unit_cost((int)ceil64(K, 64), c, phase);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

}  // namespace

struct BatchSweep::Tables {
  std::vector<PbChain> chains;
  std::vector<PbUnit> units;
  std::vector<int32_t> first;
  std::vector<float*> last;
  PbParams p;
};

BatchSweep::BatchSweep() : t(new Tables()) {}
BatchSweep::~BatchSweep() { delete t; }

bool batch_sweep_ok(const tn_mps* psis, int count, const tn_mpo* H, int prec) {
  if (count > PB_MAX_CHAINS) return false;
  for (int k = 0; k < count; ++k) {
    if (!expect_persistent_ok(&psis[k], H, prec)) return false;
    for (int i = 0; i <= psis[k].n; ++i)
      if (psis[k].bond[i] > PERSISTENT_MAX_BOND) return false;
  }
  return true;
}

int BatchSweep::build(const tn_mps* psis, int cnt, const tn_mpo* H, int prec) {
  count = cnt;
  split = prec == TN_PREC_BF16X3;
  const int n = psis[0].n, planes = split ? 2 : 1;
  const int64_t d = psis[0].d;
  const int grid = device_sms();
  PbParams& p = t->p;
  memset(&p, 0, sizeof(p));
  p.n = n;
  p.d = (int32_t)d;
  p.count = count;
  for (int i = 0; i <= n; ++i) p.w[i] = (int8_t)(H->bond[i] + 1);
  // per chain: one packed environment and one packed T2, sized for its sites
  size_t off = 0;
  std::vector<size_t> lp((size_t)count), t2((size_t)count), lpb((size_t)count), t2b((size_t)count);
  for (int k = 0; k < count; ++k) {
    for (int i = 0; i < n; ++i) {
      const int64_t Da = psis[k].bond[i], Db = psis[k].bond[i + 1];
      lpb[k] = std::max(lpb[k], ps_bytes(ceil64(Da, int64_t(1) << group_shift(p.w[i])), Da, 128));
      t2b[k] = std::max(t2b[k], ps_bytes(ceil64(p.w[i + 1] * (int64_t)pad16((int32_t)Db), 128), d * Da, 128));
    }
    lp[k] = off;
    off += lpb[k] * planes;
    t2[k] = off;
    off += t2b[k] * planes;
  }
  if (off / 1024 > 0xFFFFFFFFull) return TN_ERR_UNSUPPORTED;
  off_cores = off;
  t->chains.resize((size_t)n * count);
  t->first.assign((size_t)n * 2 * (grid + 1), 0);
  t->last.resize((size_t)count);
  size_t cores = 0;
  int widest = 0;
  struct Cost {
    double c;
    PbUnit u;
  };
  std::vector<Cost> list;
  for (int i = 0; i < n; ++i) {
    size_t co = 0;
    uint32_t pu = 0;
    for (int k = 0; k < count; ++k) {
      PbChain& c = t->chains[(size_t)i * count + k];
      memset(&c, 0, sizeof(c));
      const int64_t Da = psis[k].bond[i], Db = psis[k].bond[i + 1], DbP = pad16((int32_t)Db);
      c.A = psis[k].cores[i];
      c.Da = (int16_t)Da;
      c.Db = (int16_t)Db;
      c.unit0 = pu;
      c.lp = (uint32_t)(lp[k] / 1024);
      c.lp_lo = split ? (uint32_t)(lpb[k] / 1024) : 0u;
      c.t2 = (uint32_t)(t2[k] / 1024);
      c.t2_lo = split ? (uint32_t)(t2b[k] / 1024) : 0u;
      for (int j = 0; j < 2; ++j) {
        PsTiles& q = c.t[j];
        const int64_t total = j ? DbP : d * DbP, K = j ? d * Da : Da;
        const int cols = batch_cols(total, K, j ? 32 : (int)(32 * d), j);
        q.off = (uint32_t)(co / 1024);
        q.tp = (uint16_t)(j ? ceil64(p.w[i + 1] * DbP, 128) : ceil64(Da, int64_t(1) << group_shift(p.w[i])));
        q.tq = (uint16_t)ceil64(total, cols);
        q.cols = (int16_t)cols;
        q.slabs = (int16_t)ceil64(K, 64);
        co += ps_bytes(q.tq, K, cols);
        pu += pack_units(q);
        widest = std::max(widest, cols);
      }
    }
    if (co / 1024 > 0xFFFFFFFFull) return TN_ERR_UNSUPPORTED;
    cores = std::max(cores, co);
    p.pack[i] = pu;
    // a site like the one before it, as most of a chain's are, has its units
    bool same = i > 0 && p.w[i] == p.w[i - 1] && p.w[i + 1] == p.w[i];
    for (int k = 0; k < count && same; ++k)
      same = psis[k].bond[i] == psis[k].bond[i - 1] && psis[k].bond[i + 1] == psis[k].bond[i];
    if (same) {
      const auto before = t->first.begin() + (ptrdiff_t)(i - 1) * 2 * (grid + 1);
      std::copy(before, before + 2 * (grid + 1), before + 2 * (grid + 1));
      continue;
    }
    for (int j = 0; j < 2; ++j) {
      list.clear();
      for (int k = 0; k < count; ++k) {
        const PbChain& c = t->chains[(size_t)i * count + k];
        const PsTiles& q = c.t[j];
        // the grouped contraction's first operand: the core when the
        // environment has fewer than 128 rows and fewer than the core
        const int64_t M = (int64_t)p.w[i] * c.Da, N = d * c.Db;
        PbUnit u;
        memset(&u, 0, sizeof(u));
        u.chain = (uint16_t)k;
        u.slabs = (uint8_t)q.slabs;
        u.cols16 = (uint8_t)(q.cols / 16);
        u.cross = j == 0 && N > M && M < 128;
        for (int a = 0; a < q.tp; ++a)
          for (int b = 0; b < q.tq; ++b) {
            u.tpi = (uint8_t)a;
            u.tqi = (uint8_t)b;
            list.push_back(Cost{unit_cost(q.slabs, q.cols, j), u});
          }
      }
      std::stable_sort(list.begin(), list.end(), [](const Cost& a, const Cost& b) { return a.c > b.c; });
      // each to the CTA with the least so far; a CTA's units lie together
      std::vector<std::vector<PbUnit>> mine((size_t)grid);
      std::priority_queue<std::pair<double, int>, std::vector<std::pair<double, int>>, std::greater<>> load;
      for (int c = 0; c < grid; ++c) load.push({0.0, c});
      for (const Cost& e : list) {
        const auto least = load.top();
        load.pop();
        mine[(size_t)least.second].push_back(e.u);
        load.push({least.first + e.c, least.second});
      }
      int32_t* first = t->first.data() + ((size_t)i * 2 + j) * (grid + 1);
      for (int c = 0; c < grid; ++c) {
        first[c] = (int32_t)t->units.size();
        t->units.insert(t->units.end(), mine[(size_t)c].begin(), mine[(size_t)c].end());
      }
      first[grid] = (int32_t)t->units.size();
    }
  }
  p.stage_bytes = planes * (PS_BLOCK + widest * 128);
  p.stages = std::min(PS_RING / p.stage_bytes, PS_MAX_STAGES);
  cores = align256(cores);
  p.Cp_lo = split ? (int64_t)cores : 0;
  site_bytes = cores * planes;
  off = off_cores + 2 * site_bytes;
  off_chains = off;
  off += align256(sizeof(PbChain) * t->chains.size());
  off_units = off;
  off += align256(sizeof(PbUnit) * std::max<size_t>(t->units.size(), 1));
  off_first = off;
  off += align256(sizeof(int32_t) * t->first.size());
  off_last = off;
  off += align256(sizeof(float*) * (size_t)count);
  off_bar = off;
  off += 256;
  bytes = off;
  return TN_OK;
}

int BatchSweep::upload(uint8_t* region, float* const* last, const float* Wx, const int64_t* woff, unsigned* bits,
                       double* lg, cudaStream_t s) {
  PbParams& p = t->p;
  p.base = region;
  p.Cp[0] = region + off_cores;
  p.Cp[1] = region + off_cores + site_bytes;
  p.chains = reinterpret_cast<const PbChain*>(region + off_chains);
  p.units = reinterpret_cast<const PbUnit*>(region + off_units);
  p.first = reinterpret_cast<const int32_t*>(region + off_first);
  p.last = reinterpret_cast<float* const*>(region + off_last);
  p.bar = reinterpret_cast<unsigned*>(region + off_bar);
  p.Wx = Wx;
  p.bits = bits;
  p.lg = lg;
  p.status = status_word();
  for (int i = 0; i < p.n; ++i) p.woff[i] = (int32_t)woff[i];
  for (int k = 0; k < count; ++k) t->last[(size_t)k] = last[k];
  auto up = [&](size_t at, const void* src, size_t b) {
    return b == 0 || cudaMemcpyAsync(region + at, src, b, cudaMemcpyHostToDevice, s) == cudaSuccess;
  };
  return up(off_chains, t->chains.data(), sizeof(PbChain) * t->chains.size()) &&
                 up(off_units, t->units.data(), sizeof(PbUnit) * t->units.size()) &&
                 up(off_first, t->first.data(), sizeof(int32_t) * t->first.size()) &&
                 up(off_last, t->last.data(), sizeof(float*) * t->last.size())
             ? TN_OK
             : TN_ERR_CUDA;
}

int BatchSweep::run(cudaStream_t s) const {
  if (cudaMemsetAsync(t->p.bar, 0, sizeof(unsigned), s) != cudaSuccess) return TN_ERR_CUDA;
  return split ? launch_sweep(expect_batch_kernel<1>, t->p, s) : launch_sweep(expect_batch_kernel<0>, t->p, s);
}

}  // namespace tn

extern "C" int tn_check_grid_barrier_timeout(uint64_t limit_ns, void* counter, void* stream) {
  if (!counter || (reinterpret_cast<uintptr_t>(counter) & 3)) return TN_ERR_ARG;
  const uint64_t lo = 10000000ull, hi = 2000000000ull;
  uint64_t lim = limit_ns < lo ? lo : (limit_ns > hi ? hi : limit_ns);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(counter, 0, sizeof(unsigned), s) != cudaSuccess) return TN_ERR_CUDA;
  unsigned* bar = static_cast<unsigned*>(counter);
  int* status = tn::status_word();
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(2);
  cfg.blockDim = dim3(32);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, tn::grid_barrier_timeout_kernel, bar, status, lim) == cudaSuccess ? TN_OK
                                                                                                   : TN_ERR_CUDA;
}
