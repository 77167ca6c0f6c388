// Internal interface of the float32 classifier sweeps (classifier_f32.cu).
#pragma once

#include "tn_internal.h"

namespace tn {

constexpr int CLS_F32_MAXN = 1024;

// Bytes of one step's float32 core image [in][s][out], both bonds padded to chi.
inline size_t cls_f32_image_bytes(int chi) { return sizeof(float) * 2 * (size_t)chi * chi; }
// Row length of the kept feature pairs: the batch rounded up to an even count
// (each row a multiple of 16 bytes).
inline size_t cls_f32_phi_row(int batch) { return ((size_t)batch + 1) & ~size_t(1); }

// Packs the cores of both half-chains into images of one kind (adjoint = 0:
// forward, 1: adjoint), steps 0 .. T[h]-1 of half h (half 0: sites 0 ..
// ls-1; half 1: sites n-1 .. ls+1).
struct ClsF32PackParams {
  int32_t n, chi, adjoint;
  int32_t T[2];
  int32_t bond[CLS_F32_MAXN + 1];
  const float* core[CLS_F32_MAXN];
  float* images[2];
};
int cls_f32_pack(const ClsF32PackParams& p, cudaStream_t s);

// One launch sweeps both half-chains over the steps [t_begin[h], t_end[h])
// (forward in increasing, adjoint in decreasing order).
struct ClsF32Params {
  int32_t n, batch, kmax;     // kmax: largest inner bond, rounded up to a multiple of 4
  int32_t store_every;
  int32_t t_begin[2], t_end[2];
  int32_t store_base[2];
  const float* images[2];
  const float* pixels;        // [batch, n]
  float* state[2];            // [batch, chi] in/out (forward: v, adjoint: g)
  double* lam[2];             // forward: [batch] log-scale, in/out
  float* store[2];            // forward: vectors entering kept steps, [slot][batch][chi] (or null)
  float* sc[2];               // [t][batch] per-step scales (forward writes, adjoint reads)
  float* h[2];                // adjoint: g / scale per step, [t - t_begin][batch][chi]
  float2* phi[2];             // adjoint: the feature pair per step, [t - t_begin][cls_f32_phi_row]
  int* status;
};
int cls_f32_sweep(int chi, int adjoint, const ClsF32Params& p, cudaStream_t s);

// grad[h][t][k][s chi + j] += sum_b v_b[k] phi_s(b) h_b[j] for the steps
// [t_begin[h], t_end[h]): v[h], h[h] as [t - t_begin][batch][chi].
struct ClsF32GradParams {
  int32_t batch, chunk;       // chunk: samples per CTA (a multiple of the staging depth)
  int32_t t_begin[2], t_end[2];
  const float* v[2];
  const float* h[2];
  const float2* phi[2];
  float* grad[2];
  int* status;
};
int cls_f32_grad(int chi, const ClsF32GradParams& p, cudaStream_t s);

}  // namespace tn
