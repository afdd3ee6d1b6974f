// Fractional scan offsets (f2 of Eq. 2 by the Fourier shift theorem) and the gradient with
// respect to them.
//
// With offsets delta[l][j] (rows, columns; pixels) the object patch of position j at
// wavelength l is the F x F window at the integer position resampled at r + delta:
//   p_delta = F2^-1[ ramp * F2 p ],   ramp(k) = exp(2 pi i (f(k_y) d_y + f(k_x) d_x)),
// with f(k) = k/F for k < F/2 and (k - F)/F otherwise, the window taken as one period.
// The ramp is a product of one factor per axis, so the shift is a shift of every column followed by one of
// every row, each DFT, ramp, inverse DFT within one thread group: a pass per axis instead of the three
// (rows, columns with the ramp, rows) of a 2D transform and back, and no spectrum kept for the adjoint.
// Per position batch, before the forward row pass:
//   k_shift_cols      (columns of the window, gathered from O) -> u
//   k_shift_rows      (rows of u) -> the batch's patch buffer, read by the row passes
// and after the adjoint row pass, on the mode-summed object-gradient patch g (the gradient
// with respect to p_delta) in its scratch slot:
//   k_shift_rows_adj  (rows: conjugate ramp) -> g'; with G, U the row spectra of g and u,
//                     dL/d delta_x = -(2 pi / F) sum f_x Im(conj(G) ramp_x U)   (Parseval's theorem)
//   k_shift_cols_adj  (columns: conjugate ramp) -> back into the slot: the adjoint-shifted patch gradient
//                     that the object-gradient kernel adds into grad O; with G', U the column spectra of
//                     g' and u, dL/d delta_y = -(2 pi / F) sum f_y Im(conj(G') U): u is
//                     already shifted along its columns
// A block's vectors share one ramp, evaluated once per block.  All transforms are the unscaled two-stage
// register FFTs of fft_regs.cuh.
// 400 positions of 256^2 x 4 modes x 3 wavelengths with every position optimised: 4.64 -> 4.46 ms per step
// (112 -> 80 bytes of HBM traffic per window element, one ramp value per block and frequency instead of one
// per element).
#pragma once
#include "kernels.cuh"

namespace ptycho {

// Frequency of DFT index k in cycles per pixel (numpy's fftfreq order).
template <int F>
__device__ __forceinline__ float dft_freq(int k) {
  return (float)(k < F / 2 ? k : k - F) * (1.0f / (float)F);
}

struct ShiftArgs {
  const float* delta;            // [L][J][2] fractional offsets (device)
  float2* u;                     // [B][L][F][F] windows shifted along their columns
  float2* patch;                 // [B][L][F][F] shifted windows
  float2* g1;                    // [B][L][F][F] patch gradients after the row adjoint
  float2* slot;                  // patch gradients in the scratch: slot l*M of position b
  long long slot_b, slot_l;      // its element strides between positions and wavelengths
  int slot_pair;                 // a slot of the pair passes: positions 2p and 2p+1 share rows of 2 F
                                 // values (2p first)
  double* dpart;                 // [nbatch][L][F/W][2] position-gradient partials (y, x), or null
};

// Offset of row r of the patch of (position b, wavelength l) in the scratch, and between its rows.
__device__ __forceinline__ long long slot_row(const ShiftArgs& sa, int b, int l, int r, int F) {
  return sa.slot_pair ? 2 * ((b >> 1) * sa.slot_b + l * sa.slot_l + (long long)r * F) + (b & 1) * F
                      : b * sa.slot_b + l * sa.slot_l + (long long)r * F;
}

// exp(2 pi i f(k) d) for every k, by the whole block.
template <int F>
__device__ __forceinline__ void stage_ramp(float d, float2* ramp) {
  for (int k = threadIdx.x; k < F; k += blockDim.x) {
    float sn, cs;
    sincospif(2.0f * dft_freq<F>(k) * d, &sn, &cs);
    ramp[k] = make_float2(cs, sn);
  }
  __syncthreads();
}

// Sum over the block of double-float terms (256 threads), times ``scale``, in FP64; valid in thread 0.
__device__ __forceinline__ double shift_block_sum(float hi, float lo, float (*red)[8], double scale) {
  df_warp_sum(hi, lo);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = hi;
    red[1][threadIdx.x >> 5] = lo;
  }
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) s += (double)red[0][w] + (double)red[1][w];
  return s * scale;
}

template <int F> __host__ __device__ constexpr int shift_cols_smem() { return ColCfg<F>::smem_xch + F * 8; }
template <int F> __host__ __device__ constexpr int shift_rows_smem() { return RowCfg<F>::smem + F * 8; }

// grid (F/W, L, nb)
template <int F>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_shift_cols(const float2* __restrict__ O, KArgs a, ShiftArgs sa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ float2 smem[];
  float2* ramp = smem + W * Xch<F>::region_cols;
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col = blockIdx.x * W + c, l = blockIdx.y, b = blockIdx.z;
  const int j = batch_pos(a, a.batch_off + b);
  if (j < 0) return;                                  // uniform over the block
  const float2* src = O + a.obj_off[l] + (long long)a.pos[(l * a.J + j) * 2] * a.obj_w[l] + a.pos[(l * a.J + j) * 2 + 1] + col;
  float2 v[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) v[n2] = __ldg(src + (long long)(t + N1 * n2) * a.obj_w[l]);
  stage_ramp<F>(__ldg(sa.delta + (l * a.J + j) * 2), ramp);
  fft_fwd_I2O<F>(v, t, smem + c * Xch<F>::region_cols, a.tw, BlockSync{});
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) v[sl] = cmul(v[sl], ramp[idxO<F>(t, sl)]);
  fft_inv_O2I<F>(v, t, smem + c * Xch<F>::region_cols, a.tw, BlockSync{});
  float2* dst = sa.u + ((long long)b * a.L + l) * F * F + col;
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) dst[(t + N1 * n2) * F] = cscale(v[n2], 1.0f / (float)F);
}

// grid (F/RPB, L, nb)
template <int F>
__global__ void __launch_bounds__(RowCfg<F>::threads)
k_shift_rows(KArgs a, ShiftArgs sa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = RowCfg<F>::T;
  extern __shared__ float2 smem[];
  float2* ramp = smem + RowCfg<F>::RPB * Xch<F>::region_rows;
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int r = blockIdx.x * RowCfg<F>::RPB + vec, l = blockIdx.y, b = blockIdx.z;
  const int j = batch_pos(a, a.batch_off + b);
  if (j < 0) return;                                  // uniform over the block
  const long long off = (((long long)b * a.L + l) * F + r) * F + t;
  float2* xc = smem + vec * Xch<F>::region_rows;
  float2 v[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) v[n2] = sa.u[off + N1 * n2];
  stage_ramp<F>(__ldg(sa.delta + (l * a.J + j) * 2 + 1), ramp);
  fft_fwd_I2O<F>(v, t, xc, a.tw, WarpSync{});
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) v[sl] = cmul(v[sl], ramp[idxO<F>(t, sl)]);
  fft_inv_O2I<F>(v, t, xc, a.tw, WarpSync{});
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) sa.patch[off + N1 * n2] = cscale(v[n2], 1.0f / (float)F);
}

// grid (F/RPB, L, nb)
template <int F>
__global__ void __launch_bounds__(RowCfg<F>::threads)
k_shift_rows_adj(KArgs a, ShiftArgs sa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = RowCfg<F>::T;
  static_assert(RowCfg<F>::RPB == ColCfg<F>::W && RowCfg<F>::threads == 256 && ColCfg<F>::threads == 256,
                "both adjoint passes leave F/W partials per window, from blocks of eight warps");
  extern __shared__ float2 smem[];
  __shared__ float red[2][8];
  float2* ramp = smem + RowCfg<F>::RPB * Xch<F>::region_rows;
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int r = blockIdx.x * RowCfg<F>::RPB + vec, l = blockIdx.y, b = blockIdx.z;
  const int j = batch_pos(a, a.batch_off + b);
  double* dx = sa.dpart ? sa.dpart + (((long long)(a.batch_off + b) * a.L + l) * gridDim.x + blockIdx.x) * 2 + 1 : nullptr;
  if (j < 0) {                                        // uniform over the block
    if (dx && threadIdx.x == 0) *dx = 0.0;
    return;
  }
  const long long off = (((long long)b * a.L + l) * F + r) * F + t;
  const float2* src = sa.slot + slot_row(sa, b, l, r, F) + t;
  float2* xc = smem + vec * Xch<F>::region_rows;
  float2 g[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) g[n2] = src[N1 * n2];
  stage_ramp<F>(__ldg(sa.delta + (l * a.J + j) * 2 + 1), ramp);
  fft_fwd_I2O<F>(g, t, xc, a.tw, WarpSync{});
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) g[sl] = cmulc(g[sl], ramp[idxO<F>(t, sl)]);   // conj(ramp) G: conj of it times U is conj(G) ramp U
  if (sa.dpart) {
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = sa.u[off + N1 * n2];
    fft_fwd_I2O<F>(v, t, xc, a.tw, WarpSync{});
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl)
      df_add(hi, lo, -6.283185307179586f * dft_freq<F>(idxO<F>(t, sl)) * fmaf(g[sl].x, v[sl].y, -g[sl].y * v[sl].x));
    const double s = shift_block_sum(hi, lo, red, 1.0 / (double)F);
    if (threadIdx.x == 0) *dx = s;
  }
  fft_inv_O2I<F>(g, t, xc, a.tw, WarpSync{});
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) sa.g1[off + N1 * n2] = cscale(g[n2], 1.0f / (float)F);
}

// grid (F/W, L, nb)
template <int F>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_shift_cols_adj(KArgs a, ShiftArgs sa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ float2 smem[];
  __shared__ float red[2][8];
  float2* ramp = smem + W * Xch<F>::region_cols;
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col = blockIdx.x * W + c, l = blockIdx.y, b = blockIdx.z;
  const int j = batch_pos(a, a.batch_off + b);
  double* dy = sa.dpart ? sa.dpart + (((long long)(a.batch_off + b) * a.L + l) * gridDim.x + blockIdx.x) * 2 : nullptr;
  if (j < 0) {                                        // uniform over the block
    if (dy && threadIdx.x == 0) *dy = 0.0;
    return;
  }
  const long long off = ((long long)b * a.L + l) * F * F + col;
  float2* xc = smem + c * Xch<F>::region_cols;
  float2 g[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) g[n2] = sa.g1[off + (t + N1 * n2) * F];
  stage_ramp<F>(__ldg(sa.delta + (l * a.J + j) * 2), ramp);
  fft_fwd_I2O<F>(g, t, xc, a.tw, BlockSync{});
  if (sa.dpart) {
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = sa.u[off + (t + N1 * n2) * F];
    fft_fwd_I2O<F>(v, t, xc, a.tw, BlockSync{});
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl)
      df_add(hi, lo, -6.283185307179586f * dft_freq<F>(idxO<F>(t, sl)) * fmaf(g[sl].x, v[sl].y, -g[sl].y * v[sl].x));
    const double s = shift_block_sum(hi, lo, red, 1.0 / (double)F);
    if (threadIdx.x == 0) *dy = s;
  }
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) g[sl] = cmulc(g[sl], ramp[idxO<F>(t, sl)]);
  fft_inv_O2I<F>(g, t, xc, a.tw, BlockSync{});
  float2* dst = sa.slot + slot_row(sa, b, l, 0, F) + col;
  const int stride = sa.slot_pair ? 2 * F : F;
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) dst[(long long)(t + N1 * n2) * stride] = cscale(g[n2], 1.0f / (float)F);
}

// Position gradient: g_delta[l][j][a] = sum, in call-entry order, of the partials of every
// entry i with bidx[i] = j; 0 for positions outside the call.   grid (ceil(L*J/8))
__global__ void k_delta_grad(const int32_t* __restrict__ bidx, int nbatch, int L, int J, const double* __restrict__ dpart,
                             int nstrips, float* __restrict__ g_delta);

}  // namespace ptycho
