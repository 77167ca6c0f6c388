// MPS image classifier (Sec. IV.A): forward scores and the adjoint backward.
//
// Forward: the local feature map Phi(p) = (cos(pi p/2), sin(pi p/2)) of each
// pixel is contracted into the chain from both ends towards the label core.
// One step of a half-chain, for a tile of samples b and the site's core seen
// as L[k, s, j] (k the incoming bond, j the outgoing one):
//     v'_b[j] = sum_s Phi_s(x_b) sum_k v_b[k] L[k, s, j],
// then v'_b is divided by its largest magnitude and log(scale_b) is added to
// the sample's float64 log-scale. The two half-chain vectors meet at the
// label core: ftilde_b[l] = sum_{a,s,c} vL_b[a] C[a, s, l, c] Phi_s vR_b[c].
//
// Backward (adjoint): the same step with the transposed core and the recorded
// scale, g_b[k] = sum_s Phi_s sum_j L[k, s, j] g'_b[j] / scale_b, walks from
// the label core outwards; the core gradients are sums over the batch,
// dL[k, s, j] = sum_b v_b[k] Phi_s(x_b) g'_b[j] / scale_b, summed over the
// batch per checkpoint segment. Sweep vectors are kept every `ckpt_every`
// steps and the steps in between are recomputed segment by segment
// (checkpointing). The sweeps themselves: classifier_f32.cu (FP32) and
// classifier_tc.cu (BF16, BF16x3).
#include <math.h>

#include <algorithm>

#include "classifier_f32.h"
#include "classifier_tc.h"
#include "packed.h"
#include "tn_internal.h"

namespace tn {
namespace {

constexpr int CLS_MAXN = 1024;  // sites passed by value to the sweep kernel
constexpr int CLS_MAXCHI = 128;

// ------------------------------------------------------------- label core
// The label core C[a, s, l, c] meets the two half-chain vectors vL, vR:
//   ftilde_b[l] = sum_{a,s} vL_b[a] Phi_s(x_b) G_b[a, s, l],  G_b[a, s, l] = sum_c C[a, s, l, c] vR_b[c],
// with G one float32 contraction over c for the whole batch. Its adjoint,
// for d_b = dLoss/dftilde_b and H_b[a, s, l] = vL_b[a] Phi_s(x_b) d_b[l]:
//   gL_b[a] = sum_{s,l} d_b[l] Phi_s(x_b) G_b[a, s, l],
//   gR_b[c] = sum_{a,s,l} H_b[a, s, l] C[a, s, l, c]   (a contraction over (a, s, l)),
//   dC[a, s, l, c] = sum_b H_b[a, s, l] vR_b[c]         (a contraction over b).
constexpr int LABEL_MAXL = 16;

struct LabelParams {
  int32_t n, batch, ls, L, chi, DL, DR;
  const float* pixels;  // [batch, n]
  const float* vL;      // [batch, chi]
  const double* lamL;
  const double* lamR;
  const float* G;       // [batch, DL, 2, L]
  float* ftilde;        // [batch, L]
  double* log_scale;    // [batch]
  const float* dft;     // adjoint: [batch, L]
  float* gL;            // adjoint: [batch, chi] (zero past DL)
  float* H;             // adjoint: [batch, DL, 2, L]
};

// One warp per sample: ftilde_b[l] = sum_{a,s} vL_b[a] Phi_s G_b[a, s, l].
__global__ void __launch_bounds__(256) cls_label_reduce(const __grid_constant__ LabelParams p) {
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= p.batch) return;
  const float x = __ldg(p.pixels + (int64_t)b * p.n + p.ls);
  const float ph[2] = {cospif(0.5f * x), sinpif(0.5f * x)};
  const float* vL = p.vL + (int64_t)b * p.chi;
  const float* G = p.G + (int64_t)b * p.DL * 2 * p.L;
  float acc[LABEL_MAXL];
#pragma unroll
  for (int l = 0; l < LABEL_MAXL; ++l) acc[l] = 0.0f;
  for (int as = lane; as < p.DL * 2; as += 32) {
    const float w = vL[as >> 1] * ph[as & 1];
#pragma unroll
    for (int l = 0; l < LABEL_MAXL; ++l)
      if (l < p.L) acc[l] = fmaf(w, G[(int64_t)as * p.L + l], acc[l]);
  }
#pragma unroll
  for (int l = 0; l < LABEL_MAXL; ++l)
    for (int o = 16; o > 0; o >>= 1) acc[l] += __shfl_xor_sync(0xffffffffu, acc[l], o);
  if (lane < p.L) {
    float v = acc[0];
#pragma unroll
    for (int l = 1; l < LABEL_MAXL; ++l)
      if (lane == l) v = acc[l];
    p.ftilde[(int64_t)b * p.L + lane] = v;
  }
  if (lane == 0) p.log_scale[b] = p.lamL[b] + p.lamR[b];
}

// One warp per sample: gL_b and H_b.
__global__ void __launch_bounds__(256) cls_label_adjoint(const __grid_constant__ LabelParams p) {
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= p.batch) return;
  const float x = __ldg(p.pixels + (int64_t)b * p.n + p.ls);
  const float ph[2] = {cospif(0.5f * x), sinpif(0.5f * x)};
  const float* vL = p.vL + (int64_t)b * p.chi;
  const float* G = p.G + (int64_t)b * p.DL * 2 * p.L;
  float* H = p.H + (int64_t)b * p.DL * 2 * p.L;
  const float* d = p.dft + (int64_t)b * p.L;
  for (int a = lane; a < p.chi; a += 32) {
    float acc = 0.0f;
    if (a < p.DL)
      for (int s = 0; s < 2; ++s)
        for (int l = 0; l < p.L; ++l) {
          const int64_t i = ((int64_t)a * 2 + s) * p.L + l;
          acc = fmaf(d[l] * ph[s], G[i], acc);
          H[i] = vL[a] * ph[s] * d[l];
        }
    p.gL[(int64_t)b * p.chi + a] = acc;
  }
}

// dst[b, c] = src[b, c] for c < D, 0 for D <= c < chi.
__global__ void cls_pad_rows(const float* __restrict__ src, int D, float* __restrict__ dst, int batch, int chi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)batch * chi) return;
  const int64_t b = i / chi;
  const int c = (int)(i % chi);
  dst[i] = c < D ? src[b * D + c] : 0.0f;
}

// Loss head: one CTA of 1024 threads, samples strided over the threads; the
// softmax of the normalised scores (|z| <= 1) in float32, the norm and the
// batch sum in float64, reduced in a fixed order (deterministic).
constexpr int LOSS_THREADS = 1024;
__global__ void __launch_bounds__(LOSS_THREADS)
cls_loss_kernel(const float* __restrict__ ft, const int64_t* __restrict__ y, int batch, int L, double* loss,
                float* dft) {
  __shared__ double red[LOSS_THREADS];
  double acc = 0.0;
  for (int b = threadIdx.x; b < batch; b += LOSS_THREADS) {
    const float* f = ft + (int64_t)b * L;
    double nrm = 0.0;
    for (int l = 0; l < L; ++l) nrm += (double)f[l] * f[l];
    nrm = sqrt(nrm);
    const float inv = nrm > 0.0 ? (float)(1.0 / nrm) : 0.0f;
    float z[LABEL_MAXL], pz[LABEL_MAXL], zmax = -3.0e38f;
    for (int l = 0; l < L; ++l) {
      z[l] = f[l] * inv;
      zmax = fmaxf(zmax, z[l]);
    }
    float se = 0.0f;
    for (int l = 0; l < L; ++l) {
      pz[l] = expf(z[l] - zmax);
      se += pz[l];
    }
    const int64_t yb = y[b];
    acc += (double)(zmax + logf(se) - z[yb]);
    if (dft) {
      float zg = 0.0f;
      const float ise = 1.0f / se;
      for (int l = 0; l < L; ++l) {
        pz[l] = pz[l] * ise - (l == yb ? 1.0f : 0.0f);
        zg += z[l] * pz[l];
      }
      const float sc = inv / (float)batch;
      for (int l = 0; l < L; ++l) dft[(int64_t)b * L + l] = (pz[l] - z[l] * zg) * sc;
    }
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = LOSS_THREADS / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0] / batch;
}

// First vector of each half-chain: e_0 (bond 1 at the chain's ends), log-scale 0.
__global__ void cls_init_state(float* state, double* lam, int batch, int chi) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < (int64_t)batch * chi) state[i] = (i % chi) == 0 ? 1.0f : 0.0f;
  if (i < batch) lam[i] = 0.0;
}

// ----------------------------------------------------------------- layout
// Workspace of one classifier. The forward leaves the half-chain vectors,
// their log-scales, the per-step scales and the kept vectors here for the
// backward.
struct ClsLayout {
  int n, ls, L, batch, chi, ck, ntiles;
  int T[2];        // steps per half
  int nck[2];      // kept vectors per half
  int seg_len;     // steps per backward segment
  float* state[2];
  double* lam[2];
  float* ckpt[2];
  float* sc[2];
  float* g[2];
  float* replay[2];     // running vector of a segment's recomputation [batch][chi]
  double* replay_lam[2];
  // float32 path
  float* seg[2];   // recomputed vectors of one segment [seg_len][batch][chi]
  float* H[2];     // the adjoint's g / scale of one segment, likewise
  float2* phi[2];  // its feature pairs [seg_len][cls_f32_phi_row]
  // tensor-core path (the images are the float32 path's too)
  uint8_t* fimg[2];  // forward core images per half
  uint8_t* aimg[2];  // adjoint core images per half
  uint8_t* vseg[2][2];  // bf16 vector tiles of a segment per half; two: one being written, one read
  float* grad[2];    // [t][chi][2 chi] accumulated core gradients per half
  // label core
  float* labG;     // [batch][DL][2][L]
  float* labH;     // [batch][DL][2][L]
  float* gR;       // [batch][DR]
  uint8_t* scratch;  // packed operands of G = vR C (BF16X3), or none
  size_t scratch_bytes;
  size_t bytes;
};

int chi_of(const tn_mps* W) {
  int64_t c = 1;
  for (int i = 0; i <= W->n; ++i) c = std::max(c, W->bond[i]);
  if (c <= 32) return 32;
  if (c <= 64) return 64;
  return 128;
}

ClsLayout cls_layout(uint8_t* base, const tn_mps* W, int ls, int L, int batch, int ck) {
  ClsLayout w;
  memset(&w, 0, sizeof(w));
  w.n = W->n;
  w.ls = ls;
  w.L = L;
  w.batch = batch;
  w.chi = chi_of(W);
  w.ck = ck;
  w.ntiles = (batch + CLS_TILE - 1) / CLS_TILE;
  w.T[0] = ls;
  w.T[1] = W->n - 1 - ls;
  const int cke = ck > 0 ? ck : 1;
  for (int h = 0; h < 2; ++h) w.nck[h] = ck > 0 ? (w.T[h] + cke - 1) / cke : 0;
  const int Tmax = std::max(w.T[0], w.T[1]);
  w.seg_len = ck <= 1 ? std::max(Tmax, 1) : ck;
  size_t off = 0;
  auto take = [&](size_t b) { uint8_t* p = base ? base + off : nullptr; off += align256(b); return p; };
  const int chi = w.chi;
  const size_t vec = sizeof(float) * (size_t)batch * chi;
  const bool bwd = ck > 0;
  for (int h = 0; h < 2; ++h) {
    w.state[h] = reinterpret_cast<float*>(take(vec));
    w.lam[h] = reinterpret_cast<double*>(take(sizeof(double) * (size_t)batch));
    w.ckpt[h] = reinterpret_cast<float*>(take(vec * (size_t)w.nck[h]));
    w.sc[h] = reinterpret_cast<float*>(take(sizeof(float) * (size_t)batch * std::max(w.T[h], 1)));
    w.g[h] = reinterpret_cast<float*>(take(bwd ? vec : 0));
    w.replay[h] = reinterpret_cast<float*>(take(bwd ? vec : 0));
    w.replay_lam[h] = reinterpret_cast<double*>(take(bwd ? sizeof(double) * (size_t)batch : 0));
  }
  // float32 backward: recomputed vectors, adjoint vectors and features of
  // both halves' segments
  for (int h = 0; h < 2; ++h) {
    const size_t steps = (size_t)std::min(w.seg_len, std::max(w.T[h], 1));
    w.seg[h] = reinterpret_cast<float*>(take(bwd && ck > 1 ? vec * steps : 0));
    w.H[h] = reinterpret_cast<float*>(take(bwd ? vec * steps : 0));
    w.phi[h] = reinterpret_cast<float2*>(take(bwd ? sizeof(float2) * cls_f32_phi_row(batch) * steps : 0));
  }
  // core images (sized for the split BF16x3 ones, as large as the float32
  // ones or larger) and the tensor-core path's vector tiles
  for (int h = 0; h < 2; ++h) {
    w.fimg[h] = take(cls_fwd_image_bytes(chi, 1) * (size_t)w.T[h]);
    w.aimg[h] = take(bwd ? cls_adj_image_bytes(chi, 1) * (size_t)w.T[h] : 0);
    const size_t steps = (size_t)std::min(w.seg_len, std::max(w.T[h], 1));
    for (int i = 0; i < 2; ++i)
      w.vseg[h][i] = i == 0 || w.T[h] > w.seg_len ? take(bwd ? cls_vtile_bytes(chi, 1) * (size_t)w.ntiles * steps : 0)
                                                  : w.vseg[h][0];
    w.grad[h] = reinterpret_cast<float*>(take(bwd ? sizeof(float) * (size_t)w.T[h] * chi * 2 * chi : 0));
  }
  const int64_t DL = W->bond[ls], DR = W->bond[ls + 1];
  const size_t lab = sizeof(float) * (size_t)batch * (size_t)(DL * 2 * L);
  w.labG = reinterpret_cast<float*>(take(lab));
  w.labH = reinterpret_cast<float*>(take(bwd ? lab : 0));
  w.gR = reinterpret_cast<float*>(take(bwd ? sizeof(float) * (size_t)batch * DR : 0));
  // G = vR C on packed operands (in place its gather bounds it: 4096 samples, chi =
  // 128: 66 us, packed and multiplied by the grouped kernel 36). Only where that
  // gives the same bits: a batch of 128 or more is the first operand there too,
  // and K <= 128 is one accumulation. The backward's two (K up to a batch) would
  // add in other pieces, which a BF16 adjoint's roundings blow up.
  w.scratch_bytes = batch >= 128 ? packed_scratch_bound(batch, DL * 2 * L, DR, TN_PREC_BF16X3) : 0;
  w.scratch = take(w.scratch_bytes);
  w.bytes = off;
  return w;
}

int check_classifier(const tn_mps* W, int ls, int L, const float* pixels, int batch) {
  if (!W || !W->bond || !W->cores || !pixels || batch < 0) return TN_ERR_ARG;
  if (W->n < 2 || W->n > CLS_MAXN || ls < 0 || ls >= W->n || L < 1 || L > LABEL_MAXL) return TN_ERR_ARG;
  if (W->d != 2) return TN_ERR_UNSUPPORTED;
  if (W->bond[0] != 1 || W->bond[W->n] != 1) return TN_ERR_SHAPE;
  for (int i = 0; i < W->n; ++i) {
    if (!W->cores[i] || W->bond[i + 1] < 1) return TN_ERR_ARG;
    if (W->bond[i + 1] > CLS_MAXCHI) return TN_ERR_UNSUPPORTED;
  }
  return TN_OK;
}

// Both halves' cores packed into the float32 images of one kind.
int pack_images_f32(const tn_mps* W, const ClsLayout& w, int adjoint, cudaStream_t s) {
  ClsF32PackParams pp;
  memset(&pp, 0, sizeof(pp));
  pp.n = W->n;
  pp.chi = w.chi;
  pp.adjoint = adjoint;
  for (int i = 0; i <= W->n; ++i) pp.bond[i] = (int32_t)W->bond[i];
  for (int i = 0; i < W->n; ++i) pp.core[i] = W->cores[i];
  for (int h = 0; h < 2; ++h) {
    pp.T[h] = w.T[h];
    pp.images[h] = reinterpret_cast<float*>(adjoint ? w.aimg[h] : w.fimg[h]);
  }
  return cls_f32_pack(pp, s);
}

ClsF32Params f32_params(const tn_mps* W, const ClsLayout& w, const float* pixels, int adjoint) {
  ClsF32Params p;
  memset(&p, 0, sizeof(p));
  p.n = W->n;
  p.batch = w.batch;
  int64_t kmax = 1;
  for (int i = 0; i <= W->n; ++i) kmax = std::max(kmax, W->bond[i]);
  p.kmax = (int32_t)((kmax + 3) / 4 * 4);
  p.store_every = 1;
  p.pixels = pixels;
  for (int h = 0; h < 2; ++h) {
    p.t_end[h] = w.T[h];
    p.images[h] = reinterpret_cast<const float*>(adjoint ? w.aimg[h] : w.fimg[h]);
    p.sc[h] = w.sc[h];
  }
  p.status = status_word();
  return p;
}

// Both halves' cores packed into the tensor-core images of one kind.
int pack_images(const tn_mps* W, const ClsLayout& w, int split, int adjoint, cudaStream_t s) {
  ClsPackParams pp;
  memset(&pp, 0, sizeof(pp));
  pp.n = W->n;
  pp.chi = w.chi;
  pp.split = split;
  pp.adjoint = adjoint;
  pp.T[0] = w.T[0];
  pp.T[1] = w.T[1];
  for (int i = 0; i <= W->n; ++i) pp.bond[i] = (int32_t)W->bond[i];
  for (int i = 0; i < W->n; ++i) pp.core[i] = W->cores[i];
  for (int h = 0; h < 2; ++h) pp.images[h] = adjoint ? w.aimg[h] : w.fimg[h];
  pp.step_bytes = adjoint ? cls_adj_image_bytes(w.chi, split) : cls_fwd_image_bytes(w.chi, split);
  return cls_pack(pp, s);
}

ClsTcParams tc_params(const tn_mps* W, const ClsLayout& w, const float* pixels) {
  ClsTcParams q;
  memset(&q, 0, sizeof(q));
  q.n = W->n;
  q.batch = w.batch;
  q.ntiles = w.ntiles;
  q.store_every = 1;
  q.half_site[0] = 0;
  q.half_dir[0] = 1;
  q.half_site[1] = W->n - 1;
  q.half_dir[1] = -1;
  q.pixels = pixels;
  for (int h = 0; h < 2; ++h) {
    q.sc[h] = w.sc[h];
    q.t_end[h] = w.T[h];
  }
  q.status = status_word();
  return q;
}

tn_tensor strided(float* p, int rank, const int64_t* shape, const int64_t* stride) {
  tn_tensor t;
  memset(&t, 0, sizeof(t));
  t.data = p;
  t.rank = rank;
  t.dtype = TN_F32;
  for (int i = 0; i < rank; ++i) {
    t.shape[i] = shape[i];
    t.stride[i] = stride[i];
  }
  return t;
}

LabelParams label_params(const tn_mps* W, const ClsLayout& w, const float* pixels) {
  LabelParams lp;
  memset(&lp, 0, sizeof(lp));
  lp.n = W->n;
  lp.batch = w.batch;
  lp.ls = w.ls;
  lp.L = w.L;
  lp.chi = w.chi;
  lp.DL = (int)W->bond[w.ls];
  lp.DR = (int)W->bond[w.ls + 1];
  lp.pixels = pixels;
  lp.vL = w.state[0];
  lp.lamL = w.lam[0];
  lp.lamR = w.lam[1];
  lp.G = w.labG;
  return lp;
}

// The label core's contractions: float32 for an FP32 classifier; the split
// BF16X3 tensor-core contraction for BF16 / BF16X3 (relative error ~2^-16 of
// |A||B| per element, below either mode's own sweep error, at a fraction of
// the float32 kernel's time).
int label_prec(int prec) { return prec == TN_PREC_FP32 ? TN_PREC_FP32 : TN_PREC_BF16X3; }

// The accumulated per-step gradients of both halves into the cores' shapes.
int scatter_gradients(const tn_mps* W, const ClsLayout& w, float* const* dcores, cudaStream_t s) {
  ClsScatterParams sp;
  memset(&sp, 0, sizeof(sp));
  sp.n = W->n;
  sp.chi = w.chi;
  sp.T[0] = w.T[0];
  sp.T[1] = w.T[1];
  for (int i = 0; i <= W->n; ++i) sp.bond[i] = (int32_t)W->bond[i];
  for (int i = 0; i < W->n; ++i) sp.dcore[i] = dcores[i];
  sp.grad[0] = w.grad[0];
  sp.grad[1] = w.grad[1];
  return cls_scatter_grad(sp, s);
}

// G[b, a, s, l] = sum_c vR[b, c] C[a, s, l, c].
int label_G(const tn_mps* W, const ClsLayout& w, int prec, cudaStream_t s) {
  const int64_t DL = W->bond[w.ls], DR = W->bond[w.ls + 1], B = w.batch, L = w.L;
  const int64_t shv[2] = {B, DR}, stv[2] = {w.chi, 1};
  const int64_t shc[4] = {DL, 2, L, DR}, stc[4] = {0, 0, 0, 0};
  const int64_t shg[4] = {B, DL, 2, L}, stg[4] = {0, 0, 0, 0};
  tn_tensor tv = strided(w.state[1], 2, shv, stv);
  tn_tensor tc = strided(const_cast<float*>(W->cores[w.ls]), 4, shc, stc);
  tn_tensor tg = strided(w.labG, 4, shg, stg);
  const int lv[1] = {1}, lc[1] = {3};
  return contract_internal(&tv, lv, &tc, lc, 1, &tg, label_prec(prec), s, w.scratch_bytes ? w.scratch : nullptr, w.scratch_bytes);
}

}  // namespace
}  // namespace tn

using namespace tn;

extern "C" {

int tn_mps_classify_loss(const float* ftilde, const int64_t* labels, int batch, int n_labels, double* loss,
                         float* dftilde, void* stream) {
  if (!ftilde || !labels || !loss || batch < 1 || n_labels < 1 || n_labels > LABEL_MAXL) return TN_ERR_ARG;
  cls_loss_kernel<<<1, LOSS_THREADS, 0, static_cast<cudaStream_t>(stream)>>>(ftilde, labels, batch, n_labels, loss,
                                                                             dftilde);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

size_t tn_mps_classify_workspace_bytes(const tn_mps* W, int label_site, int n_labels, int batch, int ckpt_every) {
  if (!W || !W->bond || W->n < 2 || label_site < 0 || label_site >= W->n || batch < 0 || ckpt_every < 0) return 0;
  return cls_layout(nullptr, W, label_site, n_labels, batch, ckpt_every).bytes;
}

int tn_mps_classify(const tn_mps* W, int label_site, int n_labels, const float* pixels, int batch, int prec,
                    int ckpt_every, float* ftilde, double* log_scale, void* workspace, size_t ws_bytes,
                    void* stream) {
  int rc = check_classifier(W, label_site, n_labels, pixels, batch);
  if (rc != TN_OK) return rc;
  if (!ftilde || !log_scale || ckpt_every < 0) return TN_ERR_ARG;
  if (prec != TN_PREC_FP32 && prec != TN_PREC_BF16 && prec != TN_PREC_BF16X3) return TN_ERR_ARG;
  if (batch == 0) return TN_OK;
  ClsLayout w = cls_layout(static_cast<uint8_t*>(workspace), W, label_site, n_labels, batch, ckpt_every);
  if (!workspace || ws_bytes < w.bytes || (reinterpret_cast<uintptr_t>(workspace) & 255)) return TN_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t nvec = (int64_t)batch * w.chi;
  for (int h = 0; h < 2; ++h) {
    cls_init_state<<<(unsigned)((nvec + 255) / 256), 256, 0, s>>>(w.state[h], w.lam[h], batch, w.chi);
    if (cudaGetLastError() != cudaSuccess) return TN_ERR_CUDA;
  }
  if (prec == TN_PREC_FP32) {
    if ((rc = pack_images_f32(W, w, 0, s)) != TN_OK) return rc;
    ClsF32Params p = f32_params(W, w, pixels, 0);
    for (int h = 0; h < 2; ++h) {
      p.state[h] = w.state[h];
      p.lam[h] = w.lam[h];
      if (ckpt_every > 0) p.store[h] = w.ckpt[h];
    }
    p.store_every = ckpt_every > 0 ? ckpt_every : 1;
    if ((rc = cls_f32_sweep(w.chi, 0, p, s)) != TN_OK) return rc;
  } else {
    // both half-chains in one tcgen05 launch
    const int split = prec == TN_PREC_BF16X3;
    if ((rc = pack_images(W, w, split, 0, s)) != TN_OK) return rc;
    ClsTcParams q = tc_params(W, w, pixels);
    for (int h = 0; h < 2; ++h) {
      q.state_in[h] = q.state[h] = w.state[h];
      q.lam[h] = w.lam[h];
      q.images[h] = w.fimg[h];
      if (ckpt_every > 0) q.store[h] = w.ckpt[h];
    }
    q.store_every = ckpt_every > 0 ? ckpt_every : 1;
    if ((rc = cls_fwd_tc_launch(w.chi, split, q, s)) != TN_OK) return rc;
  }
  if ((rc = label_G(W, w, prec, s)) != TN_OK) return rc;
  LabelParams lp = label_params(W, w, pixels);
  lp.ftilde = ftilde;
  lp.log_scale = log_scale;
  cls_label_reduce<<<(unsigned)((batch + 7) / 8), 256, 0, s>>>(lp);
  return cudaGetLastError() == cudaSuccess ? TN_OK : TN_ERR_CUDA;
}

int tn_mps_classify_backward(const tn_mps* W, int label_site, int n_labels, const float* pixels, int batch,
                             int prec, int ckpt_every, const float* dftilde, float* const* dcores,
                             void* workspace, size_t ws_bytes, void* stream) {
  int rc = check_classifier(W, label_site, n_labels, pixels, batch);
  if (rc != TN_OK) return rc;
  if (!dftilde || !dcores || ckpt_every < 1) return TN_ERR_ARG;
  for (int i = 0; i < W->n; ++i)
    if (!dcores[i]) return TN_ERR_ARG;
  if (prec != TN_PREC_FP32 && prec != TN_PREC_BF16 && prec != TN_PREC_BF16X3) return TN_ERR_ARG;
  ClsLayout w = cls_layout(static_cast<uint8_t*>(workspace), W, label_site, n_labels, batch, ckpt_every);
  if (!workspace || ws_bytes < w.bytes || (reinterpret_cast<uintptr_t>(workspace) & 255)) return TN_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int chi = w.chi, n = W->n, ls = label_site, L = n_labels;
  const int split = prec == TN_PREC_BF16X3;
  if (prec != TN_PREC_FP32 && !cls_adj_tc_supported(chi, split)) return TN_ERR_UNSUPPORTED;
  if (prec == TN_PREC_FP32 && batch > 0 && stream_capturing(s)) return TN_ERR_UNSUPPORTED;  // by the entry point's contract; nothing below needs it
  if (batch == 0) {
    for (int i = 0; i < n; ++i) {
      const int64_t e = W->bond[i] * 2 * W->bond[i + 1] * (i == ls ? L : 1);
      if (cudaMemsetAsync(dcores[i], 0, sizeof(float) * (size_t)e, s) != cudaSuccess) return TN_ERR_CUDA;
    }
    return TN_OK;
  }

  // label core: the adjoints entering both half-chains, and dC
  {
    if ((rc = label_G(W, w, prec, s)) != TN_OK) return rc;
    LabelParams lp = label_params(W, w, pixels);
    lp.dft = dftilde;
    lp.gL = w.g[0];
    lp.H = w.labH;
    cls_label_adjoint<<<(unsigned)((batch + 7) / 8), 256, 0, s>>>(lp);
    if (cudaGetLastError() != cudaSuccess) return TN_ERR_CUDA;
    const int64_t B = batch, DL = lp.DL, DR = lp.DR;
    const int64_t shh[4] = {B, DL, 2, L}, sth[4] = {0, 0, 0, 0};
    const int64_t shc[4] = {DL, 2, L, DR}, stc[4] = {0, 0, 0, 0};
    const int64_t shr[2] = {B, DR}, str[2] = {0, 0};
    const int64_t shv[2] = {B, DR}, stv[2] = {chi, 1};
    tn_tensor th = strided(w.labH, 4, shh, sth);
    tn_tensor tc = strided(const_cast<float*>(W->cores[ls]), 4, shc, stc);
    tn_tensor tr = strided(w.gR, 2, shr, str);
    const int lh[3] = {1, 2, 3}, lc[3] = {0, 1, 2};
    if ((rc = contract_internal(&th, lh, &tc, lc, 3, &tr, label_prec(prec), s)) != TN_OK) return rc;
    const int64_t nvec = B * chi;
    cls_pad_rows<<<(unsigned)((nvec + 255) / 256), 256, 0, s>>>(w.gR, (int)DR, w.g[1], batch, chi);
    if (cudaGetLastError() != cudaSuccess) return TN_ERR_CUDA;
    tn_tensor tv = strided(w.state[1], 2, shv, stv);
    tn_tensor td = strided(dcores[ls], 4, shc, stc);
    const int l0[1] = {0};
    if ((rc = contract_internal(&th, l0, &tv, l0, 1, &td, label_prec(prec), s)) != TN_OK) return rc;
  }

  const int seg = ckpt_every <= 1 ? std::max(std::max(w.T[0], w.T[1]), 1) : ckpt_every;
  int nseg[2];
  for (int h = 0; h < 2; ++h) nseg[h] = (w.T[h] + seg - 1) / seg;
  const int rounds = std::max(nseg[0], nseg[1]);
  // segment of half h handled in round k (segments run from the label core outwards)
  auto seg_range = [&](int h, int k, int* t0, int* t1) {
    const int sg = nseg[h] - 1 - k;
    if (sg < 0) {
      *t0 = *t1 = 0;
      return false;
    }
    *t0 = sg * seg;
    *t1 = std::min(w.T[h], *t0 + seg);
    return true;
  };
  const size_t vbytes = sizeof(float) * (size_t)batch * chi;

  if (prec != TN_PREC_FP32) {
    // tcgen05: per round, one launch runs both halves' adjoint segments,
    // accumulating every step's core gradient, and recomputes the next
    // segments from their kept vectors (their bf16 vector tiles kept for the
    // gradient products)
    if ((rc = pack_images(W, w, split, 0, s)) != TN_OK) return rc;
    if ((rc = pack_images(W, w, split, 1, s)) != TN_OK) return rc;
    for (int h = 0; h < 2; ++h)
      if (w.T[h] > 0 &&
          cudaMemsetAsync(w.grad[h], 0, sizeof(float) * (size_t)w.T[h] * chi * 2 * chi, s) != cudaSuccess)
        return TN_ERR_CUDA;
    auto recompute = [&](int k) {
      ClsTcParams f = tc_params(W, w, pixels);
      for (int h = 0; h < 2; ++h) {
        const bool any = seg_range(h, k, &f.t_begin[h], &f.t_end[h]);
        f.state_in[h] = any ? w.ckpt[h] + (int64_t)(f.t_begin[h] / ckpt_every) * batch * chi : w.replay[h];
        f.state[h] = w.replay[h];
        f.lam[h] = w.replay_lam[h];
        f.vseg[h] = w.vseg[h][k & 1];
        f.images[h] = w.fimg[h];
      }
      return f;
    };
    if (rounds > 0 && (rc = cls_fwd_tc_launch(chi, split, recompute(0), s)) != TN_OK) return rc;
    for (int k = 0; k < rounds; ++k) {
      ClsTcParams a = tc_params(W, w, pixels);
      for (int h = 0; h < 2; ++h) {
        seg_range(h, k, &a.t_begin[h], &a.t_end[h]);
        a.state[h] = w.g[h];
        a.vseg[h] = w.vseg[h][k & 1];
        a.images[h] = w.aimg[h];
        a.grad[h] = w.grad[h];
      }
      ClsTcParams f;
      if (k + 1 < rounds) f = recompute(k + 1);
      if ((rc = cls_adj_tc_launch(chi, split, a, k + 1 < rounds ? &f : nullptr, s)) != TN_OK) return rc;
    }
    return scatter_gradients(W, w, dcores, s);
  }

  // float32: per round one launch recomputes both halves' segments from
  // their kept vectors (the replay rewrites the same per-step scales), one
  // runs both adjoint segments keeping g / scale and the features of every
  // step, and one sums the segment's core gradients over the batch
  if ((rc = pack_images_f32(W, w, 0, s)) != TN_OK) return rc;
  if ((rc = pack_images_f32(W, w, 1, s)) != TN_OK) return rc;
  for (int h = 0; h < 2; ++h)
    if (w.T[h] > 0 &&
        cudaMemsetAsync(w.grad[h], 0, sizeof(float) * (size_t)w.T[h] * chi * 2 * chi, s) != cudaSuccess)
      return TN_ERR_CUDA;
  for (int k = 0; k < rounds; ++k) {
    ClsF32Params f = f32_params(W, w, pixels, 0);
    ClsF32Params a = f32_params(W, w, pixels, 1);
    ClsF32GradParams g;
    memset(&g, 0, sizeof(g));
    g.batch = batch;
    g.status = f.status;
    for (int h = 0; h < 2; ++h) {
      int t0, t1;
      seg_range(h, k, &t0, &t1);
      f.t_begin[h] = a.t_begin[h] = g.t_begin[h] = t0;
      f.t_end[h] = a.t_end[h] = g.t_end[h] = t1;
      if (ckpt_every > 1) {
        if (t1 > t0 && cudaMemcpyAsync(w.replay[h], w.ckpt[h] + (int64_t)(t0 / ckpt_every) * batch * chi, vbytes,
                                       cudaMemcpyDeviceToDevice, s) != cudaSuccess)
          return TN_ERR_CUDA;
        f.state[h] = w.replay[h];
        f.lam[h] = w.replay_lam[h];
        f.store[h] = w.seg[h];
        f.store_base[h] = t0;
      }
      a.state[h] = w.g[h];
      a.h[h] = w.H[h];
      a.phi[h] = w.phi[h];
      g.v[h] = ckpt_every > 1 ? w.seg[h] : w.ckpt[h] + (int64_t)t0 * batch * chi;
      g.h[h] = w.H[h];
      g.phi[h] = w.phi[h];
      g.grad[h] = w.grad[h];
    }
    if (ckpt_every > 1 && (rc = cls_f32_sweep(chi, 0, f, s)) != TN_OK) return rc;
    if ((rc = cls_f32_sweep(chi, 1, a, s)) != TN_OK) return rc;
    if ((rc = cls_f32_grad(chi, g, s)) != TN_OK) return rc;
  }
  return scatter_gradients(W, w, dcores, s);
}

}  // extern "C"
