// Kernels of the batched multi-wavelength, multi-mode ptychography forward model and its
// adjoint (Eq. 1 written as f5(f4(f3(f1(sigma_j), f2(s_j)))) of Eq. 2).
//
// Work is organised per *position batch* (B scan positions) and per *mode chunk* (a run of
// the L*M (wavelength, probe-mode) pairs, index mode = l*M + m).  For a batch the 2D DFT of
// every exit wave goes through a scratch buffer S[B][C][F][F] (complex64) sized to stay in
// the GPU's L2 cache:
//
//   k_row_fwd   psi = sigma_j P_lm * O_l(r - s_j) for one row of every mode of a wavelength
//               (the object row is read once); 1D FFT along the row -> S
//   k_col_fwd   1D FFT along columns of S -> Psi (scaled by 1/F); accumulate |Psi|^2 over
//               the modes of a group into Ipart; optionally keep Psi in S for the adjoint
//   k_loss      I = sum of groups (+ background) on the model grid; tilted-plane remap to the
//               camera grid; mask; loss terms (FP64 block partials) and D = mask dL/dI
//   k_remap_adj G = R^T D on the model grid (only with the remap; otherwise G = D)
//   k_col_adj   Psi (kept, or recomputed from S); (2/F) G Psi; inverse column DFT -> S
//   k_row_adj   inverse 1D FFT along rows -> chi = dL/dpsi; grad P_lm += conj(sigma p) chi
//               summed over the batch in registers; S <- conj(sigma P_lm) chi
//   k_obj_grad  grad O_l tile += sum over the batch's overlapping patches and the chunk's
//               modes of S (each object tile is owned by one thread block: deterministic)
//   k_loss_reduce  fixed-order FP64 sum of the per-block loss partials
//   k_sigma_grad, k_bg_accum, k_sum_sets  gradients of the power coefficients and of the
//               background (optional outputs of the adjoint)
//   k_adam      Adam on the real and imaginary parts of O and P
#pragma once
#include "fft_regs.cuh"
#include "tma.cuh"

namespace ptycho {

constexpr int kMaxL = 16;
constexpr int kLossThreads = 256;
constexpr int kLossPx = 4;       // camera pixels per thread in the loss kernel (a multiple of 4)
template <int F> __host__ __device__ constexpr int loss_blocks() { return F * F / (kLossThreads * kLossPx); }
constexpr int kLossPosMax = 8;   // positions per block of the loss kernel, at most
// Positions per block: as many as leave four blocks per SM.
inline int loss_positions(int F, int nb, int sms) {
  int np = kLossPosMax;
  while (np > 1 && (long long)(F * F / (kLossThreads * kLossPx)) * ((nb + np - 1) / np) < 4ll * sms) np /= 2;
  return np;
}
constexpr int kTile = 32;        // object-gradient tile side
constexpr int kMaxB = 512;       // positions per batch (upper bound)

struct KArgs {
  int L, M, F, J;
  const int32_t* pos;            // [L][J][2] (row, col) of the patch corner, device
  long long obj_off[kMaxL];      // complex offset of O_l in the packed object buffer
  int obj_h[kMaxL], obj_w[kMaxL];
  const int32_t* bidx;           // positions of this call, in processing order
  int nbatch;                    // number of entries in bidx
  int batch_off;                 // first entry of the current position batch
  int nb;                        // positions in the current batch (<= B <= kMaxB)
  const float* sigma;            // [J] power coefficients or null
  const float2* tw;              // W_F^(t*k2) table
  int C;                         // stride (modes) of the scratch buffer
  int chunk_base, chunk_len;     // global modes [chunk_base, chunk_base + chunk_len)
  int MG;                        // modes per column-kernel group
  int G;                         // groups per chunk (Ipart has G slices per position)
  int deal;                      // positions dealt to a split of the fused row passes at a time (1 or 2)
  int* status;                   // device status word (bit 0: a position index was out of range)
  int box[kMaxL][4];             // per wavelength: rows [box0, box2) x cols [box1, box3) covered by
                                 // the batch's patches (the whole object when not known on the host)
  const float2* patch;           // [B][L][F][F] object patches shifted by fractional offsets, or null
                                 // (the row passes then gather the patch from O at the integer position)
};

// Programmatic dependent launch: the pipeline launches each kernel so that it may start
// while the previous kernel of its stream finishes.  pdl_wait() blocks until that kernel
// has completed and its writes are visible (a no-op for an ordinary launch); every pipeline
// kernel calls it before touching global memory.  pdl_trigger() lets the next kernel start
// launching its blocks.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// Whether launch_pdl asks for programmatic stream serialisation (per host thread; each
// compute call sets it from its plan's flags).
inline bool& pdl_enabled() {
  static thread_local bool on = true;
  return on;
}

// Launch with programmatic stream serialisation (see pdl_wait above).
template <typename... KP, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KP>(args)...);
}

// Position index of batch entry i, or -1 (and the status bit set) if out of range.
__device__ __forceinline__ int batch_pos(const KArgs& a, int i) {
  const int j = a.bidx[i];
  if (j < 0 || j >= a.J) {
    atomicOr(a.status, 1);
    return -1;
  }
  return j;
}

// Scan positions (row, col) of the current batch for wavelength l and their power
// coefficients, staged in shared memory (block-strided); invalid entries become (-1, -1).
// Ends with a block barrier.
__device__ __forceinline__ void stage_batch(const KArgs& a, int l, int2* spos, float* ssig) {
  for (int b = threadIdx.x; b < a.nb; b += blockDim.x) {
    const int j = batch_pos(a, a.batch_off + b);
    if (j < 0) {
      spos[b] = make_int2(-1, -1);
      ssig[b] = 0.f;
    } else {
      spos[b] = make_int2(a.pos[(l * a.J + j) * 2], a.pos[(l * a.J + j) * 2 + 1]);
      ssig[b] = a.sigma ? __ldg(a.sigma + j) : 1.0f;
    }
  }
  __syncthreads();
}

template <int F> struct RowCfg {
  static constexpr int T = FftShape<F>::N1;
  static constexpr int RPB = 256 / T;            // rows per block
  static constexpr int threads = RPB * T;
  static constexpr int smem = RPB * Xch<F>::region_rows * (int)sizeof(float2);
};
template <int F> struct ColCfg {
  static constexpr int T = FftShape<F>::N1;
  static constexpr int W = 256 / T;              // columns per block
  static constexpr int threads = W * T;
  static constexpr int smem_xch = W * Xch<F>::region_cols * (int)sizeof(float2);
};

__device__ __forceinline__ float sigma_of(const KArgs& a, int j) { return a.sigma ? __ldg(a.sigma + j) : 1.0f; }

// ---------------------------------------------------------------------------------------
// forward row pass: exit waves (f1, f2, f3) of every mode of wavelength l in the chunk and
// the row DFT (first half of f4).   block index (row block, l, position b)
// ---------------------------------------------------------------------------------------
template <int F>
__device__ __forceinline__ void row_fwd_body(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S, const KArgs& a, const uint3 bid) {
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = RowCfg<F>::T;
  extern __shared__ float2 smem[];
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int r = bid.x * RowCfg<F>::RPB + vec;
  const int l = bid.y, b = bid.z;
  const int mlo = max(a.chunk_base, l * a.M), mhi = min(a.chunk_base + a.chunk_len, (l + 1) * a.M);
  if (mlo >= mhi) return;                             // uniform over the block
  const int j = batch_pos(a, a.batch_off + b);
  if (j < 0) return;                                  // uniform over the block
  const int y = a.pos[(l * a.J + j) * 2], x = a.pos[(l * a.J + j) * 2 + 1];
  const float s = sigma_of(a, j);
  const float2* Orow = a.patch ? a.patch + (((long long)b * a.L + l) * F + r) * F
                               : O + a.obj_off[l] + (long long)(y + r) * a.obj_w[l] + x;
  float2 p[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) p[n2] = cscale(__ldg(Orow + t + N1 * n2), s);
  for (int mode = mlo; mode < mhi; ++mode) {
    const float2* Prow = P + ((long long)mode * F + r) * F;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = cmul(__ldg(Prow + t + N1 * n2), p[n2]);
    fft_fwd_I2O<F>(v, t, smem + vec * Xch<F>::region_rows, a.tw, WarpSync{});
    float2* out = S + (((long long)b * a.C + (mode - a.chunk_base)) * F + r) * F;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) out[idxO<F>(t, sl)] = v[sl];
  }
}

// grid (nb, F/RPB, L): the positions of a batch vary fastest, so that the blocks running at the
// same time share probe rows in L2 (the probes of all modes can exceed the L2: 120 MB at 512^2
// with 6 wavelengths x 10 modes)
template <int F>
__global__ void __launch_bounds__(RowCfg<F>::threads)
k_row_fwd(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S, KArgs a) {
  pdl_wait();
  pdl_trigger();
  row_fwd_body<F>(O, P, S, a, make_uint3(blockIdx.y, blockIdx.z, blockIdx.x));
}

// ---------------------------------------------------------------------------------------
// forward column pass: column DFT (second half of f4), |Psi|^2 summed over a mode group
// grid (F/W, G, nb)
// ---------------------------------------------------------------------------------------
template <int F, bool STORE>
__device__ __forceinline__ void col_fwd_body(float2* __restrict__ S, float* __restrict__ Ipart, const KArgs& a, int first_chunk, const uint3 bid) {
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ float2 smem[];
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col = bid.x * W + c;
  const int g = bid.y, b = bid.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  float acc[N2];
#pragma unroll
  for (int i = 0; i < N2; ++i) acc[i] = 0.f;
  const float inv = 1.0f / (float)F;
  for (int cm = m0; cm < m1; ++cm) {
    float2* base = S + ((long long)b * a.C + cm) * F * F + col;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = base[(long long)(t + N1 * n2) * F];
    fft_fwd_I2O<F>(v, t, smem + c * Xch<F>::region_cols, a.tw, BlockSync{});
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) {
      add_abs2(acc[sl], v[sl]);
      if (STORE) base[(long long)idxO<F>(t, sl) * F] = cscale(v[sl], inv);
    }
  }
  float* dst = Ipart + ((long long)b * a.G + g) * F * F;
  const int cc = (col + F / 2) & (F - 1);
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) {
    const int rc = (idxO<F>(t, sl) + F / 2) & (F - 1);
    float val = acc[sl] * (inv * inv);
    if (!first_chunk) val += dst[rc * F + cc];
    dst[rc * F + cc] = val;
  }
}

template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_col_fwd(float2* __restrict__ S, float* __restrict__ Ipart, KArgs a, int first_chunk) {
  pdl_wait();
  pdl_trigger();
  col_fwd_body<F, STORE>(S, Ipart, a, first_chunk, blockIdx);
}

// ---------------------------------------------------------------------------------------
// TMA-staged column passes.  The W x F column block of one mode (W*F*8 bytes) arrives in
// shared memory through cp.async.bulk.tensor (2D tensor map over S viewed as
// [B*C*F rows][F columns] of 8-byte elements); the next mode's block is requested as soon as
// every thread has read the current one into registers, so the copy overlaps the FFT.
// ---------------------------------------------------------------------------------------
template <int F> struct ColTma {
  static constexpr int W = ColCfg<F>::W;
  static constexpr int box_rows = F < 256 ? F : 256;
  static constexpr int stage_bytes = F * W * (int)sizeof(float2);
  // + 128: the stage is placed on a 128-byte boundary inside the dynamic shared memory (whose
  // start moves with the kernel's static shared variables)
  static constexpr int smem_fwd = stage_bytes + ColCfg<F>::smem_xch + 16 + 128;
  static constexpr int smem_adj = smem_fwd + F * W * (int)sizeof(float);
};

// The first 128-byte-aligned address (in the shared window) at or after p: the destination of
// a bulk tensor copy must be 128-byte aligned.
__device__ __forceinline__ float2* align_tma_stage(unsigned char* p) {
  const uint32_t pad = (128u - (smem_addr(p) & 127u)) & 127u;
  return reinterpret_cast<float2*>(p + pad);
}

template <int F>
__device__ __forceinline__ void col_tma_issue(float2* stage, const CUtensorMap* map, int col0, int row0, uint64_t* bar) {
  fence_proxy_async_smem();                    // earlier generic reads of the stage come first
  mbar_arrive_expect_tx(bar, ColTma<F>::stage_bytes);
#pragma unroll
  for (int h = 0; h < F / ColTma<F>::box_rows; ++h)
    tma_load_2d(stage + h * ColTma<F>::box_rows * ColTma<F>::W, map, col0, row0 + h * ColTma<F>::box_rows, bar);
}

// grid (F/W, G, nb); same results as k_col_fwd
template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_col_fwd_tma(const __grid_constant__ CUtensorMap map, float2* __restrict__ S, float* __restrict__ Ipart, KArgs a,
              int first_chunk) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* smem = align_tma_stage(smem_raw);
  float2* stage = smem;
  float2* xch = smem + F * W;
  uint64_t* bar = reinterpret_cast<uint64_t*>(xch + W * Xch<F>::region_cols);
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int g = blockIdx.y, b = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && m0 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + m0) * F, bar);
  float acc[N2];
#pragma unroll
  for (int i = 0; i < N2; ++i) acc[i] = 0.f;
  const float inv = 1.0f / (float)F;
  uint32_t phase = 0;
  bool ok = true;
  for (int cm = m0; cm < m1; ++cm) {
    ok = __syncthreads_and(mbar_wait_bounded(bar, phase, a.status));
    if (!ok) break;
    phase ^= 1;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = stage[(t + N1 * n2) * W + c];
    __syncthreads();                           // the stage is free for the next mode
    if (threadIdx.x == 0 && cm + 1 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + cm + 1) * F, bar);
    fft_fwd_I2O<F>(v, t, xch + c * Xch<F>::region_cols, a.tw, BlockSync{});
    float2* base = S + ((long long)b * a.C + cm) * F * F + col;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) {
      add_abs2(acc[sl], v[sl]);
      if (STORE) base[(long long)idxO<F>(t, sl) * F] = cscale(v[sl], inv);
    }
  }
  if (!ok) {                                   // give a lost copy a bounded chance to land, then stop
    if (threadIdx.x == 0) mbar_wait_bounded(bar, phase, a.status);
    return;
  }
  float* dst = Ipart + ((long long)b * a.G + g) * F * F;
  const int cc = (col + F / 2) & (F - 1);
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) {
    const int rc = (idxO<F>(t, sl) + F / 2) & (F - 1);
    float val = acc[sl] * (inv * inv);
    if (!first_chunk) val += dst[rc * F + cc];
    dst[rc * F + cc] = val;
  }
}

// ---------------------------------------------------------------------------------------
// Staged column passes (one mode chunk holding every mode, one group: G = 1).  A block
// takes W columns of one position and runs over all its modes; the W x F column block of
// the next mode is copied into shared memory (cp.async, double-buffered) while the current
// one is transformed, so a block always has one mode's data in flight.
// grid (F/W, nb), block W*T
// ---------------------------------------------------------------------------------------
template <int F, int WN = 0> struct ColSCfg {
  static constexpr int T = FftShape<F>::N1;
  static constexpr int W = WN > 0 ? WN : (F >= 256 ? 8 : 128 / T);   // columns per block
  static constexpr int threads = W * T;
  static constexpr int stage = F * W;                // float2 per stage
  // exchange-region stride: a warp holds columns c < W and 32/W threads t of each; with the
  // stride = 32/W (mod 16) the offsets c*R + t fall on every 8-byte bank pair exactly twice
  // (two wavefronts, the minimum for 32 x 8 bytes); W >= 32 only needs an odd stride
  static constexpr int R = W >= 32 ? (Xch<F>::base | 1)
                                   : Xch<F>::base + (((32 / W) - Xch<F>::base) % 16 + 16) % 16;
  static constexpr int smem_fwd = (2 * stage + W * R) * (int)sizeof(float2);
  static constexpr int smem_adj = smem_fwd + F * W * (int)sizeof(float);
};

// Issue the copies of mode slot cm's W x F column block (from column col0) into dst.
template <int F, int WN>
__device__ __forceinline__ void col_prefetch(const float2* __restrict__ Sb, int cm, int col0, float2* dst) {
  constexpr int W = ColSCfg<F, WN>::W, CH = F * W / 2;  // 16-byte chunks
  const float2* src = Sb + (long long)cm * F * F + col0;
  for (int e = threadIdx.x; e < CH; e += ColSCfg<F, WN>::threads) {
    const int row = e / (W / 2), cc = (e % (W / 2)) * 2;
    cp_async16(dst + row * W + cc, src + (long long)row * F + cc);
  }
  cp_async_commit();
}

template <int F, bool STORE, int WN>
__global__ void __launch_bounds__(ColSCfg<F, WN>::threads)
k_col_fwd_s(float2* __restrict__ S, float* __restrict__ Ipart, KArgs a) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColSCfg<F, WN>::W, ST = ColSCfg<F, WN>::stage;
  extern __shared__ __align__(16) float2 smem[];
  float2* stage = smem;                               // [2][F][W]
  float2* xch = smem + 2 * ST;
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int b = blockIdx.y;
  const int nm = a.chunk_len;
  float2* Sb = S + (long long)b * a.C * F * F;
  float acc[N2];
#pragma unroll
  for (int i = 0; i < N2; ++i) acc[i] = 0.f;
  const float inv = 1.0f / (float)F;
  if (nm > 0) col_prefetch<F, WN>(Sb, 0, col0, stage);
  for (int cm = 0; cm < nm; ++cm) {
    const float2* cur = stage + (cm & 1) * ST;
    if (cm + 1 < nm) {
      col_prefetch<F, WN>(Sb, cm + 1, col0, stage + ((cm + 1) & 1) * ST);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = cur[(t + N1 * n2) * W + c];
    fft_fwd_I2O<F>(v, t, xch + c * ColSCfg<F, WN>::R, a.tw, BlockSync{});   // its first barrier frees cur
    float2* base = Sb + (long long)cm * F * F + col;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) {
      add_abs2(acc[sl], v[sl]);
      if (STORE) base[(long long)idxO<F>(t, sl) * F] = cscale(v[sl], inv);
    }
  }
  float* dst = Ipart + (long long)b * F * F;
  const int cc = (col + F / 2) & (F - 1);
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) {
    const int rc = (idxO<F>(t, sl) + F / 2) & (F - 1);
    dst[rc * F + cc] = acc[sl] * (inv * inv);
  }
}

// ---------------------------------------------------------------------------------------
// measurement (f5) and loss: camera-grid prediction, masked loss partials, D = mask dL/dI.
// grid (F*F/256, nb)
// ---------------------------------------------------------------------------------------
struct LossArgs {
  const float* Ipart;            // [B][G][F][F] model grid (centred)
  const float* bg;               // [F][F] model grid or null
  const int32_t* tap_base;       // [F*F] top-left model tap of each camera pixel, -1 invalid
  const float2* tap_w;           // [F*F] (wy, wx)
  const float* Imeas;            // [J][F][F] camera grid
  const uint8_t* mask;           // null, [F][F] or [J][F][F]
  int mask_per_frame;
  float eps;
  int loss_kind;                 // 0 amplitude, 1 Poisson, 2 mixed Poisson-Gaussian
  float read_var;                // s2 of the mixed loss
  float* D;                      // [B][F][F] mask * dL/dI (camera grid), null if not needed
  double* loss_part;             // [nbatch][loss_blocks] or null
  double* sig_part;              // [nbatch][loss_blocks] sums of D * (remapped sum |Psi|^2), or null
  float* I_pred;                 // [J][F][F] or null
  int remap;
  int Gsum;                      // intensity slices (mode groups) to add
  int npos;                      // positions per block (1 to kLossPosMax)
  const float2* tap_dz;          // [F*F] d(row, col index of the taps)/dz (remap only)
  double* z_part;                // [nbatch][loss_blocks] sums of D * d(R I)/dz, or null
};

// Model intensity at pixel u: the G intensity slices added in slice order (small G unrolled; the
// rounding is that of the loop, which starts from 0 + slice 0).
__device__ __forceinline__ float model_I(const float* Ip, int G, int FF, int u) {
  const float* p = Ip + u;
  switch (G) {
    case 1: return p[0];
    case 2: return p[0] + p[FF];
    case 3: return (p[0] + p[FF]) + p[2 * FF];
    case 4: return ((p[0] + p[FF]) + p[2 * FF]) + p[3 * FF];
    default: {
      float s = 0.f;
      for (int g = 0; g < G; ++g, p += FF) s += *p;
      return s;
    }
  }
}

// Poisson deviance per pixel, I_hat * (r - 1 - log r) with r = Ie / I_hat, without the
// cancellation of the direct form near r = 1 (series of u - log(1+u), u = r - 1).
__device__ __forceinline__ float poisson_term(float Ie, float Ih) {
  if (Ih <= 0.f) return Ie;
  const float u = (Ie - Ih) / Ih;
  float f;
  if (fabsf(u) < 0.25f) {
    // u - log(1+u) = sum_{n>=2} (-1)^n u^n / n
    float p = 0.f;
#pragma unroll
    for (int n = 12; n >= 2; --n) p = fmaf(p, u, ((n & 1) ? -1.0f : 1.0f) / (float)n);
    f = p * u * u;
  } else {
    f = u - log1pf(u);
  }
  return Ih * f;
}

// Bilinear value of the four taps i00, i01 (row), i10, i11 (row + 1) with weights w = (row, column).
__device__ __forceinline__ float bilinear(float2 w, float i00, float i01, float i10, float i11) {
  return (1.f - w.x) * ((1.f - w.y) * i00 + w.y * i01) + w.x * ((1.f - w.y) * i10 + w.y * i11);
}

// Compensated FP32 sums ("double-float": value = hi + lo).  Knuth's TwoSum gives the exact
// rounding error of an addition, so the pair carries about twice the FP32 mantissa without
// FP64 arithmetic (slow on this part).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void df_add(float& hi, float& lo, float x) {
  float s, e;
  two_sum(hi, x, s, e);
  hi = s;
  lo += e;
}
__device__ __forceinline__ void df_add_df(float& hi, float& lo, float bhi, float blo) {
  float s, e;
  two_sum(hi, bhi, s, e);
  e += lo + blo;
  hi = s + e;                                    // renormalise (Fast2Sum, |s| >= |e|)
  lo = e - (hi - s);
}
// Warp-tree sum of a double-float (fixed pairing: the result does not depend on timing).
__device__ __forceinline__ void df_warp_sum(float& hi, float& lo) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_down_sync(0xffffffffu, hi, o), bl = __shfl_down_sync(0xffffffffu, lo, o);
    df_add_df(hi, lo, bh, bl);
  }
}

// Each thread takes kLossPx camera pixels of la.npos positions; pixel k of lane i of warp w is
// 128 w + 32 k + i of the block's, so that every load, the four tap gathers among them, covers one run of
// neighbouring pixels.  The taps, their weights and the remapped background of a thread's pixels serve
// all its positions.  What bounds the pass is instructions (ncu, Poisson with background: 177-205 thread
// instructions per pixel at two per cycle and SM, DRAM 12 % busy), hence the compile-time REMAP and ONE
// (one intensity slice) and one reduction per position by one warp.
// The loss terms of a block are summed as double-floats: per thread, then, for each position, by one warp
// over the threads of each of the block's eight warps; their sums in FP64 (a double-float holds 48 bits), in a
// fixed order, into one partial per (call entry, block).  The sigma- and z-gradient terms per thread, by a warp
// tree and in FP64 over the eight warps.
// grid (F*F/(kLossThreads*kLossPx), ceil(nb / la.npos))
struct LossShared {
  float2 sum[kLossPosMax][kLossThreads];              // loss terms (hi, lo) of each thread
  float red[kLossPosMax][4][kLossThreads / 32];       // sigma and z terms of each warp
};

template <int F, bool REMAP, bool ONE>
__device__ __forceinline__ void loss_positions_body(const KArgs& a, const LossArgs& la, const uint3 bid, LossShared& sm) {
  constexpr int FF = F * F, NB = loss_blocks<F>(), NW = kLossThreads / 32;
  const int b0 = bid.y * la.npos, nb = min(la.npos, a.nb - b0);
  const int q0 = bid.x * kLossThreads * kLossPx + (threadIdx.x >> 5) * 32 * kLossPx + (threadIdx.x & 31);
  const int G = ONE ? 1 : la.Gsum;
  const bool need = la.D || la.loss_part;
  int tb[kLossPx];
  float2 tw[kLossPx];
  float Ib[kLossPx];                                  // background at the camera pixels
#pragma unroll
  for (int k = 0; k < kLossPx; ++k) {
    const int q = q0 + 32 * k;
    tb[k] = q;
    tw[k] = make_float2(0.f, 0.f);
    Ib[k] = 0.f;
    if (REMAP) {
      tb[k] = __ldg(la.tap_base + q);
      tw[k] = __ldg(la.tap_w + q);
      if (la.bg && tb[k] >= 0)
        Ib[k] = bilinear(tw[k], __ldg(la.bg + tb[k]), __ldg(la.bg + tb[k] + 1), __ldg(la.bg + tb[k] + F),
                         __ldg(la.bg + tb[k] + F + 1));
    } else if (la.bg) {
      Ib[k] = __ldg(la.bg + q);
    }
  }
  const float* Ip = la.Ipart + (long long)b0 * a.G * FF;
  for (int n = 0; n < nb; ++n, Ip += (long long)a.G * FF) {
    const int j = batch_pos(a, a.batch_off + b0 + n); // uniform over the block
    float th = 0.f, tl = 0.f, sh = 0.f, sl = 0.f;     // double-float sums of the loss and sigma terms
    float zh = 0.f, zl = 0.f;                         // and of the z terms
    const long long frame = (long long)max(j, 0) * FF + q0;
    float Is[kLossPx], Im[kLossPx], d[kLossPx];
    bool use[kLossPx];
#pragma unroll
    for (int k = 0; k < kLossPx; ++k) {               // all loads first
      Is[k] = Im[k] = d[k] = 0.f;
      use[k] = j >= 0 && (!REMAP || tb[k] >= 0);      // outside the remap's grid: 0, and not in the loss
      if (use[k]) {
        if (REMAP)
          Is[k] = bilinear(tw[k], model_I(Ip, G, FF, tb[k]), model_I(Ip, G, FF, tb[k] + 1),
                           model_I(Ip, G, FF, tb[k] + F), model_I(Ip, G, FF, tb[k] + F + 1));
        else
          Is[k] = model_I(Ip, G, FF, tb[k]);
      }
      if (need) Im[k] = __ldg(la.Imeas + frame + 32 * k);
    }
    if (la.I_pred && j >= 0) {
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) la.I_pred[frame + 32 * k] = Is[k] + Ib[k];
    }
    if (!need) continue;
    if (la.mask) {
      const uint8_t* m = la.mask + (la.mask_per_frame ? frame : (long long)q0);
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) use[k] = use[k] && m[32 * k] != 0;
    }
    if (la.loss_kind == 0) {
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) {
        if (!use[k]) continue;
        const float se = sqrtf(Is[k] + Ib[k] + la.eps), diff = se - sqrtf(Im[k]);
        df_add(th, tl, diff * diff);
        d[k] = __fdividef(diff, se);                  // 2 ulp: ample for a gradient
      }
    } else {
      const bool shifted = la.loss_kind == 2;         // shifted Poisson
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) {
        if (!use[k]) continue;
        float Ie = Is[k] + Ib[k] + la.eps, Ih = Im[k];
        if (shifted) {
          Ie += la.read_var;
          Ih = fmaxf(Ih + la.read_var, 0.f);
        }
        df_add(th, tl, poisson_term(Ie, Ih));
        d[k] = __fdividef(Ie - Ih, Ie);
      }
    }
    if (la.D) {
      float* Dq = la.D + (long long)(b0 + n) * FF + q0;
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) Dq[32 * k] = d[k];
    }
    if (la.loss_part) sm.sum[n][threadIdx.x] = make_float2(th, tl);
    if (la.sig_part) {
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) df_add(sh, sl, d[k] * Is[k]);
      df_warp_sum(sh, sl);
    }
    if (REMAP && la.z_part) {                         // slopes of the interpolant of field + background
#pragma unroll
      for (int k = 0; k < kLossPx; ++k) {
        if (d[k] == 0.f) continue;
        const int u = tb[k];
        const float2 w = tw[k];
        float i00 = model_I(Ip, G, FF, u), i01 = model_I(Ip, G, FF, u + 1);
        float i10 = model_I(Ip, G, FF, u + F), i11 = model_I(Ip, G, FF, u + F + 1);
        if (la.bg) {
          i00 += __ldg(la.bg + u); i01 += __ldg(la.bg + u + 1);
          i10 += __ldg(la.bg + u + F); i11 += __ldg(la.bg + u + F + 1);
        }
        const float srow = ((1.f - w.y) * i10 + w.y * i11) - ((1.f - w.y) * i00 + w.y * i01);
        const float scol = (1.f - w.x) * (i01 - i00) + w.x * (i11 - i10);
        const float2 rz = __ldg(la.tap_dz + q0 + 32 * k);
        df_add(zh, zl, d[k] * fmaf(srow, rz.x, scol * rz.y));
      }
      df_warp_sum(zh, zl);
    }
    if ((la.sig_part || la.z_part) && (threadIdx.x & 31) == 0) {
      const int wi = threadIdx.x >> 5;
      sm.red[n][0][wi] = sh;
      sm.red[n][1][wi] = sl;
      sm.red[n][2][wi] = zh;
      sm.red[n][3][wi] = zl;
    }
  }
  if (!la.loss_part && !la.sig_part && !la.z_part) return;
  __syncthreads();
  const long long part = (long long)(a.batch_off + b0) * NB + bid.x;
  if (la.loss_part) {
    static_assert(kLossPosMax <= NW, "one warp per position");
    const int n = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (n < nb) {
      // lane i: threads 8 i ... 8 i + 7 (from a different one on each, for the banks), so that four lanes
      // hold a warp's
      float2 v = sm.sum[n][8 * lane + (lane & 7)];
#pragma unroll
      for (int i = 1; i < 8; ++i) {
        const float2 u = sm.sum[n][8 * lane + ((lane + i) & 7)];
        df_add_df(v.x, v.y, u.x, u.y);
      }
#pragma unroll
      for (int o = 1; o < 4; o *= 2) {
        const float uh = __shfl_xor_sync(0xffffffffu, v.x, o), ul = __shfl_xor_sync(0xffffffffu, v.y, o);
        df_add_df(v.x, v.y, uh, ul);
      }
      double s = (double)v.x + (double)v.y;
#pragma unroll
      for (int o = 4; o < 32; o *= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) la.loss_part[part + (long long)n * NB] = s;
    }
  }
  if (la.sig_part || la.z_part) {
    const int n = threadIdx.x >> 1, kind = threadIdx.x & 1;
    double* out = kind == 0 ? la.sig_part : la.z_part;
    if (n < nb && out) {
      double sum = 0.0;
      for (int wi = 0; wi < NW; ++wi) sum += (double)sm.red[n][2 * kind][wi] + (double)sm.red[n][2 * kind + 1][wi];
      out[part + (long long)n * NB] = sum;
    }
  }
}

template <int F>
__device__ __forceinline__ void loss_body(const KArgs& a, const LossArgs& la, const uint3 bid) {
  __shared__ LossShared sm;
  if (la.remap) {
    if (la.Gsum == 1) loss_positions_body<F, true, true>(a, la, bid, sm);
    else loss_positions_body<F, true, false>(a, la, bid, sm);
  } else {
    if (la.Gsum == 1) loss_positions_body<F, false, true>(a, la, bid, sm);
    else loss_positions_body<F, false, false>(a, la, bid, sm);
  }
}

template <int F>
__global__ void __launch_bounds__(kLossThreads, 4)
k_loss(KArgs a, LossArgs la) {
  pdl_wait();
  pdl_trigger();
  loss_body<F>(a, la, blockIdx);
}

// ---------------------------------------------------------------------------------------
// R^T of the tilted-plane remap: G[b][u] = sum over the camera pixels q that sample model
// pixel u of w_uq D[b][q] (CSR rows in increasing q: a fixed order).
// ---------------------------------------------------------------------------------------
struct AdjArgs {
  const float* D;                // [B][F][F] camera grid
  const int32_t* rt_ptr;         // [F*F+1] CSR of R^T over centred model pixels (remap only)
  const int32_t* rt_idx;         // camera pixel of each entry
  const float* rt_w;             // weight of each entry
  float* Gt;                     // [B][F][F] R^T D on the model grid (remap only)
  int remap;
};

// One thread per model pixel u and kRtPos positions of the batch: the CSR entries of u are
// read once and the positions' D loads are independent.   grid (F*F/256, ceil(nb/kRtPos))
constexpr int kRtPos = 8;
template <int F>
__device__ __forceinline__ void remap_adj_body(const KArgs& a, const AdjArgs& aa, const uint3 bid) {
  constexpr int FF = F * F;
  const int u = bid.x * 256 + threadIdx.x;
  const int b0 = bid.y * kRtPos;
  const int nbk = min(kRtPos, a.nb - b0);
  const int e0 = __ldg(aa.rt_ptr + u), e1 = __ldg(aa.rt_ptr + u + 1);
  const float* Db = aa.D + (long long)b0 * FF;
  float gv[kRtPos];
#pragma unroll
  for (int k = 0; k < kRtPos; ++k) gv[k] = 0.f;
  for (int e = e0; e < e1; ++e) {
    const float w = __ldg(aa.rt_w + e);
    const int q = __ldg(aa.rt_idx + e);
#pragma unroll
    for (int k = 0; k < kRtPos; ++k)
      if (k < nbk) gv[k] = fmaf(w, Db[(long long)k * FF + q], gv[k]);
  }
#pragma unroll
  for (int k = 0; k < kRtPos; ++k)
    if (k < nbk) aa.Gt[(long long)(b0 + k) * FF + u] = gv[k];
}

template <int F>
__global__ void __launch_bounds__(256)
k_remap_adj(KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  remap_adj_body<F>(a, aa, blockIdx);
}

// Background gradient, Eq. 1 (N is added before the remap): acc[u] += sum over the batch of
// G[b][u] (R^T D, or D without the remap), in batch order.   grid (F*F/256)
template <int F>
__global__ void __launch_bounds__(256)
k_bg_accum(const float* __restrict__ G, int nb, float* __restrict__ acc) {
  pdl_wait();
  pdl_trigger();
  constexpr int FF = F * F;
  const int u = blockIdx.x * 256 + threadIdx.x;
  float s = acc[u];
  for (int b = 0; b < nb; ++b) s += G[(long long)b * FF + u];
  acc[u] = s;
}

// ---------------------------------------------------------------------------------------
// adjoint column pass: (2/F) G Psi, inverse column DFT.   grid (F/W, G, nb)
// ---------------------------------------------------------------------------------------
template <int F, bool STORE>
__device__ __forceinline__ void col_adj_body(float2* __restrict__ S, const KArgs& a, const AdjArgs& aa, const uint3 bid) {
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ float2 smem[];
  float* gt = reinterpret_cast<float*>(smem + W * Xch<F>::region_cols);   // [F][W]
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = bid.x * W;
  const int g = bid.y, b = bid.z;
  const float* Gb = (aa.remap ? aa.Gt : aa.D) + (long long)b * F * F;
  const float scale = 2.0f / (float)F;
  for (int e = threadIdx.x; e < F * W; e += blockDim.x) {
    const int k = e / W, ce = e % W;
    const int u = ((k + F / 2) & (F - 1)) * F + ((col0 + ce + F / 2) & (F - 1));
    gt[k * W + ce] = Gb[u] * (STORE ? scale : scale / (float)F);   // recomputed Psi: the 1/F folded in
  }
  __syncthreads();
  const int col = col0 + c;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  for (int cm = m0; cm < m1; ++cm) {
    float2* base = S + ((long long)b * a.C + cm) * F * F + col;
    float2 v[N2];
    if (STORE) {
#pragma unroll
      for (int sl = 0; sl < N2; ++sl) v[sl] = base[(long long)idxO<F>(t, sl) * F];
    } else {
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) v[n2] = base[(long long)(t + N1 * n2) * F];
      fft_fwd_I2O<F>(v, t, smem + c * Xch<F>::region_cols, a.tw, BlockSync{});
    }
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) v[sl] = cscale(v[sl], gt[idxO<F>(t, sl) * W + c]);
    fft_inv_O2I<F>(v, t, smem + c * Xch<F>::region_cols, a.tw, BlockSync{});
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) base[(long long)(t + N1 * n2) * F] = v[n2];
  }
}

template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_col_adj(float2* __restrict__ S, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  col_adj_body<F, STORE>(S, a, aa, blockIdx);
}

// The plain-load column passes compiled for two blocks per SM: at 512^2 (32 values per thread)
// they fit 128 registers without spills and measured 10 % faster than the TMA-staged passes (one
// block per SM) with one field per position; from two fields on the TMA-staged passes are faster.
// (Below 512^2 the compiler's own choice is kept: a two-block bound measured 5 % slower at 256^2.)
template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads, 2)
k_col_fwd_2b(float2* __restrict__ S, float* __restrict__ Ipart, KArgs a, int first_chunk) {
  pdl_wait();
  pdl_trigger();
  col_fwd_body<F, STORE>(S, Ipart, a, first_chunk, blockIdx);
}

template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads, 2)
k_col_adj_2b(float2* __restrict__ S, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  col_adj_body<F, STORE>(S, a, aa, blockIdx);
}

// Staged adjoint column pass (see k_col_fwd_s).   grid (F/W, nb), block W*T
template <int F, bool STORE, int WN>
__global__ void __launch_bounds__(ColSCfg<F, WN>::threads)
k_col_adj_s(float2* __restrict__ S, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColSCfg<F, WN>::W, ST = ColSCfg<F, WN>::stage;
  extern __shared__ __align__(16) float2 smem[];
  float2* stage = smem;                               // [2][F][W]
  float2* xch = smem + 2 * ST;
  float* gt = reinterpret_cast<float*>(xch + W * ColSCfg<F, WN>::R);   // [F][W]
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int b = blockIdx.y;
  const int nm = a.chunk_len;
  float2* Sb = S + (long long)b * a.C * F * F;
  if (nm > 0) col_prefetch<F, WN>(Sb, 0, col0, stage);
  const float* Gb = (aa.remap ? aa.Gt : aa.D) + (long long)b * F * F;
  const float scale = 2.0f / (float)F;
  for (int e = threadIdx.x; e < F * W; e += ColSCfg<F, WN>::threads) {
    const int k = e / W, ce = e % W;
    const int u = ((k + F / 2) & (F - 1)) * F + ((col0 + ce + F / 2) & (F - 1));
    gt[k * W + ce] = Gb[u] * scale;
  }
  const float inv = 1.0f / (float)F;
  for (int cm = 0; cm < nm; ++cm) {
    const float2* cur = stage + (cm & 1) * ST;
    if (cm + 1 < nm) {
      col_prefetch<F, WN>(Sb, cm + 1, col0, stage + ((cm + 1) & 1) * ST);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    float2 v[N2];
    if (STORE) {
#pragma unroll
      for (int sl = 0; sl < N2; ++sl) v[sl] = cur[idxO<F>(t, sl) * W + c];
    } else {
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) v[n2] = cur[(t + N1 * n2) * W + c];
      fft_fwd_I2O<F>(v, t, xch + c * ColSCfg<F, WN>::R, a.tw, BlockSync{});
#pragma unroll
      for (int sl = 0; sl < N2; ++sl) v[sl] = cscale(v[sl], inv);
    }
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) v[sl] = cscale(v[sl], gt[idxO<F>(t, sl) * W + c]);
    fft_inv_O2I<F>(v, t, xch + c * ColSCfg<F, WN>::R, a.tw, BlockSync{});   // its first barrier frees cur
    float2* base = Sb + (long long)cm * F * F + col;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) base[(long long)(t + N1 * n2) * F] = v[n2];
  }
}

// grid (F/W, G, nb); same results as k_col_adj
template <int F, bool STORE>
__global__ void __launch_bounds__(ColCfg<F>::threads)
k_col_adj_tma(const __grid_constant__ CUtensorMap map, float2* __restrict__ S, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* smem = align_tma_stage(smem_raw);
  float2* stage = smem;
  float2* xch = smem + F * W;
  uint64_t* bar = reinterpret_cast<uint64_t*>(xch + W * Xch<F>::region_cols);
  float* gt = reinterpret_cast<float*>(bar + 2);                    // [F][W]
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int g = blockIdx.y, b = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && m0 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + m0) * F, bar);
  const float* Gb = (aa.remap ? aa.Gt : aa.D) + (long long)b * F * F;
  const float scale = 2.0f / (float)F;
  for (int e = threadIdx.x; e < F * W; e += blockDim.x) {
    const int k = e / W, ce = e % W;
    const int u = ((k + F / 2) & (F - 1)) * F + ((col0 + ce + F / 2) & (F - 1));
    gt[k * W + ce] = Gb[u] * scale;
  }
  __syncthreads();
  const float inv = 1.0f / (float)F;
  uint32_t phase = 0;
  bool ok = true;
  for (int cm = m0; cm < m1; ++cm) {
    ok = __syncthreads_and(mbar_wait_bounded(bar, phase, a.status));
    if (!ok) break;
    phase ^= 1;
    float2 v[N2];
    if (STORE) {
#pragma unroll
      for (int sl = 0; sl < N2; ++sl) v[sl] = stage[idxO<F>(t, sl) * W + c];
    } else {
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) v[n2] = stage[(t + N1 * n2) * W + c];
    }
    __syncthreads();                           // the stage is free for the next mode
    if (threadIdx.x == 0 && cm + 1 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + cm + 1) * F, bar);
    if (!STORE) {
      fft_fwd_I2O<F>(v, t, xch + c * Xch<F>::region_cols, a.tw, BlockSync{});
#pragma unroll
      for (int sl = 0; sl < N2; ++sl) v[sl] = cscale(v[sl], inv);
    }
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) v[sl] = cscale(v[sl], gt[idxO<F>(t, sl) * W + c]);
    fft_inv_O2I<F>(v, t, xch + c * Xch<F>::region_cols, a.tw, BlockSync{});
    float2* base = S + ((long long)b * a.C + cm) * F * F + col;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) base[(long long)(t + N1 * n2) * F] = v[n2];
  }
  if (!ok && threadIdx.x == 0) mbar_wait_bounded(bar, phase, a.status);
}

// TMA-staged column passes with the half-size exchange (fft_*_half; F = 512) and, in the adjoint,
// the dL/dI factors read through L1/L2 instead of being staged: 99 KB of shared memory per block
// instead of 134 / 166 KB, so two 8-warp blocks fit on an SM.  Same arithmetic as
// k_col_fwd_tma / k_col_adj_tma without STORE.   grid (F/W, G, nb)
template <int F> struct ColTma2 {
  static constexpr int W = ColCfg<F>::W;
  static constexpr int smem = ColTma<F>::stage_bytes + W * XchHalf<F>::region_cols * (int)sizeof(float2) + 16 + 128;
};

template <int F>
__global__ void __launch_bounds__(ColCfg<F>::threads, 2)
k_col_fwd_tma2(const __grid_constant__ CUtensorMap map, float* __restrict__ Ipart, KArgs a, int first_chunk) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W, R = XchHalf<F>::region_cols;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* stage = align_tma_stage(smem_raw);
  float2* xch = stage + F * W;
  uint64_t* bar = reinterpret_cast<uint64_t*>(xch + W * R);
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int g = blockIdx.y, b = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && m0 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + m0) * F, bar);
  float acc[N2];
#pragma unroll
  for (int i = 0; i < N2; ++i) acc[i] = 0.f;
  uint32_t phase = 0;
  bool ok = true;
  for (int cm = m0; cm < m1; ++cm) {
    ok = __syncthreads_and(mbar_wait_bounded(bar, phase, a.status));
    if (!ok) break;
    phase ^= 1;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = stage[(t + N1 * n2) * W + c];
    __syncthreads();                           // the stage is free for the next mode
    if (threadIdx.x == 0 && cm + 1 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + cm + 1) * F, bar);
    fft_fwd_I2O_half<F>(v, t, xch + c * R, a.tw, BlockSync{});
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) add_abs2(acc[sl], v[sl]);
  }
  if (!ok) {                                   // give a lost copy a bounded chance to land, then stop
    if (threadIdx.x == 0) mbar_wait_bounded(bar, phase, a.status);
    return;
  }
  const float inv = 1.0f / (float)F;
  float* dst = Ipart + ((long long)b * a.G + g) * F * F;
  const int cc = (col + F / 2) & (F - 1);
#pragma unroll
  for (int sl = 0; sl < N2; ++sl) {
    const int rc = (idxO<F>(t, sl) + F / 2) & (F - 1);
    float val = acc[sl] * (inv * inv);
    if (!first_chunk) val += dst[rc * F + cc];
    dst[rc * F + cc] = val;
  }
}

template <int F>
__global__ void __launch_bounds__(ColCfg<F>::threads, 2)
k_col_adj_tma2(const __grid_constant__ CUtensorMap map, float2* __restrict__ S, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, W = ColCfg<F>::W, R = XchHalf<F>::region_cols;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* stage = align_tma_stage(smem_raw);
  float2* xch = stage + F * W;
  uint64_t* bar = reinterpret_cast<uint64_t*>(xch + W * R);
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int col0 = blockIdx.x * W, col = col0 + c;
  const int g = blockIdx.y, b = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && m0 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + m0) * F, bar);
  // this thread's column of the dL/dI factors (DC-centred storage), read per mode through L1/L2
  const float* Gc = (aa.remap ? aa.Gt : aa.D) + (long long)b * F * F + ((col + F / 2) & (F - 1));
  const float scale = 2.0f / (float)F;
  const float inv = 1.0f / (float)F;
  uint32_t phase = 0;
  bool ok = true;
  for (int cm = m0; cm < m1; ++cm) {
    ok = __syncthreads_and(mbar_wait_bounded(bar, phase, a.status));
    if (!ok) break;
    phase ^= 1;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = stage[(t + N1 * n2) * W + c];
    __syncthreads();                           // the stage is free for the next mode
    if (threadIdx.x == 0 && cm + 1 < m1) col_tma_issue<F>(stage, &map, col0, ((long long)b * a.C + cm + 1) * F, bar);
    fft_fwd_I2O_half<F>(v, t, xch + c * R, a.tw, BlockSync{});
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) {
      const float gk = __ldg(Gc + (long long)((idxO<F>(t, sl) + F / 2) & (F - 1)) * F) * scale;
      v[sl] = cscale(cscale(v[sl], inv), gk);
    }
    fft_inv_O2I_half<F>(v, t, xch + c * R, a.tw, BlockSync{});
    float2* base = S + ((long long)b * a.C + cm) * F * F + col;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) base[(long long)(t + N1 * n2) * F] = v[n2];
  }
  if (!ok && threadIdx.x == 0) mbar_wait_bounded(bar, phase, a.status);
}

// ---------------------------------------------------------------------------------------
// adjoint row pass: chi = dL/dpsi; probe gradient summed over the batch; object-gradient
// contributions conj(sigma P) chi left in S (or, with ATOMIC, added to grad O with FP32
// atomics).  The batch is split over kAdjSlots groups of
// warps (slot s takes positions s, s + kAdjSlots, ...); their probe-gradient sums are added
// in slot order through shared memory, so the result does not depend on timing.
// grid (F/RPB, chunk_len)
// ---------------------------------------------------------------------------------------
constexpr int kAdjSlots = 4;
template <int F> struct RowAdjCfg {
  static constexpr int T = FftShape<F>::N1;
  static constexpr int RPB = 256 / (T * kAdjSlots);   // rows per block
  static constexpr int threads = RPB * T * kAdjSlots;
  static constexpr int vecs = RPB * kAdjSlots;
  static constexpr int smem_xch = vecs * Xch<F>::region_rows * (int)sizeof(float2);
  static constexpr int smem_red = (kAdjSlots - 1) * RPB * F * (int)sizeof(float2);
  static constexpr int smem = smem_xch > smem_red ? smem_xch : smem_red;
};

template <int F, bool ATOMIC>
__device__ __forceinline__ void row_adj_body(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S,
          float2* __restrict__ gP, float2* __restrict__ gO, const KArgs& a, const uint3 bid) {
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = RowAdjCfg<F>::T, RPB = RowAdjCfg<F>::RPB;
  extern __shared__ float2 smem[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int slot = vec / RPB, rr = vec % RPB;
  const int r = bid.x * RPB + rr;
  const int cm = bid.y;
  const int mode = a.chunk_base + cm;
  const int l = mode / a.M;
  stage_batch(a, l, spos, ssig);
  const float2* Prow = P + ((long long)mode * F + r) * F;
  const float2* Ol = O + a.obj_off[l];
  const int Wl = a.obj_w[l];
  float2 acc[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) acc[n2] = make_float2(0.f, 0.f);
  for (int b = slot; b < a.nb; b += kAdjSlots) {
    const int2 yx = spos[b];
    if (yx.x < 0) continue;                           // uniform over the slot's warps
    const float s = ssig[b];
    float2* row = S + (((long long)b * a.C + cm) * F + r) * F;
    const float2* Orow = Ol + (long long)(yx.x + r) * Wl + yx.y;
    float2 v[N2], p[N2];
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) v[sl] = row[idxO<F>(t, sl)];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) p[n2] = __ldg(Orow + t + N1 * n2);
    fft_inv_O2I<F>(v, t, smem + vec * Xch<F>::region_rows, a.tw, WarpSync{});
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      const float2 gp = cconjmul(p[n2], v[n2]);     // conj(p) chi
      acc[n2].x = fmaf(s, gp.x, acc[n2].x);
      acc[n2].y = fmaf(s, gp.y, acc[n2].y);
      const float2 go = cscale(cconjmul(__ldg(Prow + t + N1 * n2), v[n2]), s);   // conj(sigma P) chi
      if (ATOMIC)
        atomicAdd(gO + a.obj_off[l] + (long long)(yx.x + r) * Wl + yx.y + t + N1 * n2, go);
      else
        row[t + N1 * n2] = go;
    }
  }
  // slots 1.. hand their sums to slot 0 through shared memory (the exchange area is free now)
  __syncthreads();
  float2* red = smem;                                 // [kAdjSlots-1][RPB][F]
  if (slot > 0) {
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) red[((slot - 1) * RPB + rr) * F + t + N1 * n2] = acc[n2];
  }
  __syncthreads();
  if (slot == 0) {
    float2* g = gP + ((long long)mode * F + r) * F;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      const int c = t + N1 * n2;
      float2 sum = acc[n2];
      for (int s2 = 1; s2 < kAdjSlots; ++s2) sum = cadd(sum, red[((s2 - 1) * RPB + rr) * F + c]);
      g[c] = cadd(g[c], sum);
    }
  }
}

template <int F, bool ATOMIC>
__global__ void __launch_bounds__(RowAdjCfg<F>::threads, (F <= 256 ? 2 : 1))
k_row_adj(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S,
          float2* __restrict__ gP, float2* __restrict__ gO, KArgs a) {
  pdl_wait();
  pdl_trigger();
  row_adj_body<F, ATOMIC>(O, P, S, gP, gO, a, blockIdx);
}

// ---------------------------------------------------------------------------------------
// object gradient: one block per 32x32 tile of grad O_l inside the batch's bounding box; it
// adds, in a fixed order, every overlapping patch contribution of the chunk's modes.
// grid (tiles of the largest box, L)
// ---------------------------------------------------------------------------------------
template <int F>
__device__ __forceinline__ void obj_grad_body(const float2* __restrict__ S, float2* __restrict__ gO, const KArgs& a, const uint3 bid) {
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int l = bid.y;
  const int mlo = max(a.chunk_base, l * a.M), mhi = min(a.chunk_base + a.chunk_len, (l + 1) * a.M);
  if (mlo >= mhi) return;                             // uniform over the block
  const int by0 = a.box[l][0], bx0 = a.box[l][1];
  const int ntx = (a.box[l][3] - bx0 + kTile - 1) / kTile;
  const int nty = (a.box[l][2] - by0 + kTile - 1) / kTile;
  if ((int)bid.x >= ntx * nty) return;          // uniform over the block
  stage_batch(a, l, spos, ssig);
  const int oy0 = by0 + ((int)bid.x / ntx) * kTile, ox0 = bx0 + ((int)bid.x % ntx) * kTile;
  const int H = a.obj_h[l], Wd = a.obj_w[l];
  const int tx = threadIdx.x % kTile, ty0 = threadIdx.x / kTile;   // 8 row slots
  const int ox = ox0 + tx;
  float2 acc[kTile / 8];
#pragma unroll
  for (int k = 0; k < kTile / 8; ++k) acc[k] = make_float2(0.f, 0.f);
  for (int b = 0; b < a.nb; ++b) {
    const int y = spos[b].x, x = spos[b].y;
    if (y < 0 || y >= oy0 + kTile || y + F <= oy0 || x >= ox0 + kTile || x + F <= ox0) continue;
    const bool in_x = ox >= x && ox < x + F;
    const float2* src = S + ((long long)b * a.C + (mlo - a.chunk_base)) * F * F + (ox - x);
    for (int m0 = mlo; m0 < mhi; m0 += 4, src += 4ll * F * F) {
      float2 v[4][kTile / 8];
#pragma unroll
      for (int mm = 0; mm < 4; ++mm)
#pragma unroll
        for (int k = 0; k < kTile / 8; ++k) {
          const int oy = oy0 + ty0 + 8 * k;
          const bool ok = m0 + mm < mhi && in_x && oy >= y && oy < y + F;
          v[mm][k] = ok ? src[(long long)mm * F * F + (long long)(oy - y) * F] : make_float2(0.f, 0.f);
        }
#pragma unroll
      for (int mm = 0; mm < 4; ++mm)
#pragma unroll
        for (int k = 0; k < kTile / 8; ++k) acc[k] = cadd(acc[k], v[mm][k]);
    }
  }
  float2* g = gO + a.obj_off[l];
#pragma unroll
  for (int k = 0; k < kTile / 8; ++k) {
    const int oy = oy0 + ty0 + 8 * k;
    if (oy < H && ox < Wd) {
      float2* p = g + (long long)oy * Wd + ox;
      *p = cadd(*p, acc[k]);
    }
  }
}

template <int F>
__global__ void __launch_bounds__(256)
k_obj_grad(const float2* __restrict__ S, float2* __restrict__ gO, KArgs a) {
  pdl_wait();
  pdl_trigger();
  obj_grad_body<F>(S, gO, a, blockIdx);
}

// ---------------------------------------------------------------------------------------
// adjoint row pass over all modes of one wavelength (one mode chunk holds every mode).
// Vector v = rr*M + m of a block takes row r = blockIdx.x*rpb + rr of probe mode (l, m).
// Per scan position of the block's split: chi = dL/dpsi by the inverse row DFT; the probe
// gradient of (l, m, r) is summed in registers over the split's positions; the object-gradient
// row sum_m conj(sigma P_lm) chi is formed in shared memory (modes added in order) and written
// to the slot of mode (l, 0), which is then the only slot the object-gradient kernel reads.
// The probe row sits in shared memory for the whole batch and the object row is read once per
// position.  Probe-gradient sums go to buffer gPs + split*gp_stride (read-modify-write).
// grid (F/rpb, L, nsplit), block T*M*rpb <= 256, dynamic smem row_adj_l_smem<F>(M, rpb)
// ---------------------------------------------------------------------------------------
constexpr int kRowAdjLSmemMax = 200 * 1024;       // dynamic shared memory cap of k_row_adj_l / k_row_fwd_l
template <int F>
__host__ __device__ constexpr int row_adj_l_smem(int M, int rpb, bool probe_l2 = false) {
  return ((probe_l2 ? 0 : M * rpb * F) + 2 * M * rpb * Xch<F>::region_rows + 2 * rpb * F) * (int)sizeof(float2);
}
// Variant of k_row_adj_l whose probe rows are read through L1/L2 instead of being held in
// shared memory: at F = 512 with 10 modes that frees 40 KB per block, and the block (at most
// kRowAdjL2Threads threads) is compiled for two blocks per SM instead of one.
constexpr int kRowAdjL2Threads = 160;

// acc += conj(o) v, in the operations of the pair passes (pair.cuh).
__device__ __forceinline__ void acc_conjmul(float2& acc, float2 o, float2 v) {
  acc.x = fmaf(o.x, v.x, fmaf(o.y, v.y, acc.x));
  acc.y = fmaf(o.x, v.y, fmaf(-o.y, v.x, acc.y));
}

// Positions are dealt to the splits in groups of a.deal: one by one, so that every split gets its share of
// a short batch, or two by two, the order of the pair passes (which the shared launches of a plan with those
// follow).  Next position of this split after b whose index is valid, or -1 (uniform over the block);
// before_split(a, split, nsplit) comes before the first.
__device__ __forceinline__ int before_split(const KArgs& a, int split, int nsplit) {
  return a.deal * (split - nsplit + 1) - 1;
}
__device__ __forceinline__ int next_pos(const KArgs& a, const int2* spos, int b, int nsplit) {
  do b += (b & (a.deal - 1)) == a.deal - 1 ? 1 + a.deal * (nsplit - 1) : 1;
  while (b < a.nb && spos[b].x < 0);
  return b < a.nb ? b : -1;
}

// The same dealt one by one, for the forward rows, which add nothing up: the general form took k_row_fwd_l<512> from
// 168 to 179 registers and its 12-mode blocks from two per SM to one (131 -> 173 us for 16 positions).
__device__ __forceinline__ int next_of_split(const int2* spos, int b, int nb, int nsplit) {
  for (int bb = b + nsplit; bb < nb; bb += nsplit)
    if (spos[bb].x >= 0) return bb;
  return -1;
}

// Copies of the rpb object rows of position (y, x) (8-byte pieces: x may be odd).
template <int F>
__device__ __forceinline__ void prefetch_orows(const float2* __restrict__ Ol, int Wl, int2 yx, int row0, int rpb,
                                               float2* dst) {
  for (int e = threadIdx.x; e < rpb * F; e += blockDim.x) {
    const int rr = e / F, c = e % F;
    cp_async8(dst + e, Ol + (long long)(yx.x + row0 + rr) * Wl + yx.y + c);
  }
}

template <int F, bool PL2>
__device__ __forceinline__ void row_adj_l_body(const float2* __restrict__ O, const float2* __restrict__ P,
                                               float2* __restrict__ S, float2* __restrict__ gPs, long long gp_stride,
                                               const KArgs& a, int rpb, int nsplit, const uint3 bid) {
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = N1, RR = Xch<F>::region_rows;
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int M = a.M, V = M * rpb;
  float2* Psm = smem;                                 // [V][F]    probe rows (not with PL2)
  float2* Sst = Psm + (PL2 ? 0 : V * F);              // [2][V][RR] scratch rows; the current buffer
                                                      //   is also the FFT exchange and the mode-sum area
  float2* Ost = Sst + 2 * V * RR;                     // [2][rpb][F] object rows
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int rr = vec / M, m = vec % M;
  const int row0 = bid.x * rpb, r = row0 + rr;
  const int l = bid.y, split = bid.z;
  const int cm = l * M + m - a.chunk_base;
  const int slot0 = l * M - a.chunk_base;             // slot of the mode sum
  stage_batch(a, l, spos, ssig);
  const float2* Prow = P + ((long long)(l * M + m) * F + r) * F;
  if constexpr (!PL2) {
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) Psm[vec * F + t + N1 * n2] = __ldg(Prow + t + N1 * n2);
  }
  const float2* Ol = O + a.obj_off[l];
  const int Wl = a.obj_w[l];
  // position b's scratch row of this vector (2 KB contiguous, 16-byte pieces by its T threads)
  // and the block's object rows, into buffer buf
  auto prefetch = [&](int b, int buf) {
    const float2* row = S + (((long long)b * a.C + cm) * F + r) * F;
    float2* dst = Sst + (buf * V + vec) * RR;
#pragma unroll
    for (int k = 0; k < F / (2 * T); ++k) cp_async16(dst + 2 * (t + T * k), row + 2 * (t + T * k));
    if (a.patch)
      prefetch_orows<F>(a.patch + ((long long)b * a.L + l) * F * F, F, make_int2(0, 0), row0, rpb, Ost + buf * rpb * F);
    else
      prefetch_orows<F>(Ol, Wl, spos[b], row0, rpb, Ost + buf * rpb * F);
    cp_async_commit();
  };
  float2 acc[N2];
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) acc[n2] = make_float2(0.f, 0.f);
  int b = next_pos(a, spos, before_split(a, split, nsplit), nsplit);
  if (b >= 0) prefetch(b, 0);
  for (int buf = 0; b >= 0; buf ^= 1) {
    cp_async_wait<0>();
    __syncthreads();                                  // position b has landed; buffer buf^1 is free
    const int bn = next_pos(a, spos, b, nsplit);
    if (bn >= 0) prefetch(bn, buf ^ 1);
    const float s = ssig[b];
    float2* reg = Sst + (buf * V + vec) * RR;         // this vector's row, then its exchange/mode-sum area
    const float2* orow = Ost + (buf * rpb + rr) * F;
    float2 v[N2];
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) v[sl] = reg[idxO<F>(t, sl)];
    __syncwarp();                                     // the row is in registers before the exchange reuses it
    fft_inv_O2I<F>(v, t, reg, a.tw, WarpSync{});
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
      const int c = t + N1 * n2;
      const float2 sv = cscale(v[n2], s);                               // sigma chi
      acc_conjmul(acc[n2], orow[c], sv);                                // conj(p) sigma chi
      const float2 pv = PL2 ? __ldg(Prow + c) : Psm[vec * F + c];
      reg[c] = cconjmul(pv, sv);                                        // conj(P) sigma chi
    }
    __syncthreads();
    float2* dst = S + (((long long)b * a.C + slot0) * F + row0) * F;      // the block's rpb rows, contiguous
    for (int e = threadIdx.x; e < rpb * F; e += blockDim.x) {           // modes added in order
      const int rr2 = e / F, c = e % F;
      const float2* red = Sst + (buf * V + rr2 * M) * RR + c;
      float2 sum = red[0];
      switch (M) {                                    // small mode counts unrolled, same order
        case 1: break;
        case 2: sum = cadd(sum, red[RR]); break;
        case 3: sum = cadd(cadd(sum, red[RR]), red[2 * RR]); break;
        case 4: sum = cadd(cadd(cadd(sum, red[RR]), red[2 * RR]), red[3 * RR]); break;
        default:
          for (int mm = 1; mm < M; ++mm) sum = cadd(sum, red[mm * RR]);
      }
      dst[e] = sum;
    }
    b = bn;
  }
  float2* g = gPs + (long long)split * gp_stride + ((long long)(l * M + m) * F + r) * F;
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) {
    const int c = t + N1 * n2;
    g[c] = cadd(g[c], acc[n2]);
  }
}

template <int F, bool PL2>
__global__ void __launch_bounds__(PL2 ? kRowAdjL2Threads : 256, (F <= 256 || PL2 ? 2 : 1))
k_row_adj_l(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S,
            float2* __restrict__ gPs, long long gp_stride, KArgs a, int rpb, int nsplit) {
  pdl_wait();
  pdl_trigger();
  row_adj_l_body<F, PL2>(O, P, S, gPs, gp_stride, a, rpb, nsplit, blockIdx);
}

// Same pass at F = 512 with one warp per row (fft512_inv_warp: 16 values per lane instead of 32
// per thread of a 16-thread vector), probe rows through L1/L2: the row and its probe-gradient
// sums take half the registers, so twice as many warps fit on an SM.  Vector v (warp v) takes
// row blockIdx.x*rpb + v/M of mode v%M; element n of the row is value n/32 of lane n%32.
// grid (512/rpb, L, nsplit), block 32*M*rpb <= kRowAdjWThreads, dynamic smem row_adj_w_smem(M, rpb)
constexpr int kRowAdjWThreads = 320;
constexpr int kRowAdjWRegion = kFft512WarpXch;      // per-vector row / exchange / mode-sum area (>= 512)
__host__ __device__ constexpr int row_adj_w_smem(int M, int rpb) {
  return (2 * M * rpb * kRowAdjWRegion + 2 * rpb * 512) * (int)sizeof(float2);
}

template <int F>
__device__ __forceinline__ void row_adj_w_body(const float2* __restrict__ O, const float2* __restrict__ P,
                                               float2* __restrict__ S, float2* __restrict__ gPs, long long gp_stride,
                                               const KArgs& a, int rpb, int nsplit, const uint3 bid) {
  static_assert(F == 512, "one warp per row is the 512-point layout");
  constexpr int RR = kRowAdjWRegion;
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int M = a.M, V = M * rpb;
  float2* Sst = smem;                                 // [2][V][RR] scratch rows / exchange / mode sums
  float2* Ost = Sst + 2 * V * RR;                     // [2][rpb][F] object rows
  const int vec = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int rr = vec / M, m = vec % M;
  const int row0 = bid.x * rpb, r = row0 + rr;
  const int l = bid.y, split = bid.z;
  const int cm = l * M + m - a.chunk_base;
  const int slot0 = l * M - a.chunk_base;
  stage_batch(a, l, spos, ssig);
  const float2* Prow = P + ((long long)(l * M + m) * F + r) * F;
  const float2* Ol = O + a.obj_off[l];
  const int Wl = a.obj_w[l];
  auto prefetch = [&](int b, int buf) {
    const float2* row = S + (((long long)b * a.C + cm) * F + r) * F;
    float2* dst = Sst + (buf * V + vec) * RR;
#pragma unroll
    for (int k = 0; k < F / 64; ++k) cp_async16(dst + 2 * (t + 32 * k), row + 2 * (t + 32 * k));
    if (a.patch)
      prefetch_orows<F>(a.patch + ((long long)b * a.L + l) * F * F, F, make_int2(0, 0), row0, rpb, Ost + buf * rpb * F);
    else
      prefetch_orows<F>(Ol, Wl, spos[b], row0, rpb, Ost + buf * rpb * F);
    cp_async_commit();
  };
  float2 acc[16];
#pragma unroll
  for (int n2 = 0; n2 < 16; ++n2) acc[n2] = make_float2(0.f, 0.f);
  int b = next_pos(a, spos, before_split(a, split, nsplit), nsplit);
  if (b >= 0) prefetch(b, 0);
  for (int buf = 0; b >= 0; buf ^= 1) {
    cp_async_wait<0>();
    __syncthreads();                                  // position b has landed; buffer buf^1 is free
    const int bn = next_pos(a, spos, b, nsplit);
    if (bn >= 0) prefetch(bn, buf ^ 1);
    const float s = ssig[b];
    float2* reg = Sst + (buf * V + vec) * RR;
    const float2* orow = Ost + (buf * rpb + rr) * F;
    float2 v[16];
    fft512_inv_warp(reg, v, t, reg, a.tw);
#pragma unroll
    for (int n2 = 0; n2 < 16; ++n2) {
      const int c = t + 32 * n2;
      const float2 sv = cscale(v[n2], s);                               // sigma chi
      acc_conjmul(acc[n2], orow[c], sv);                                // conj(p) sigma chi
      reg[c] = cconjmul(__ldg(Prow + c), sv);                           // conj(P) sigma chi
    }
    __syncthreads();
    float2* dst = S + (((long long)b * a.C + slot0) * F + row0) * F;
    for (int e = threadIdx.x; e < rpb * F; e += blockDim.x) {           // modes added in order
      const int rr2 = e / F, c = e % F;
      const float2* red = Sst + (buf * V + rr2 * M) * RR + c;
      float2 sum = red[0];
      for (int mm = 1; mm < M; ++mm) sum = cadd(sum, red[mm * RR]);
      dst[e] = sum;
    }
    b = bn;
  }
  float2* g = gPs + (long long)split * gp_stride + ((long long)(l * M + m) * F + r) * F;
#pragma unroll
  for (int n2 = 0; n2 < 16; ++n2) {
    const int c = t + 32 * n2;
    g[c] = cadd(g[c], acc[n2]);
  }
}

template <int F>
__global__ void __launch_bounds__(kRowAdjWThreads, 2)
k_row_adj_w(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S,
            float2* __restrict__ gPs, long long gp_stride, KArgs a, int rpb, int nsplit) {
  pdl_wait();
  pdl_trigger();
  row_adj_w_body<F>(O, P, S, gPs, gp_stride, a, rpb, nsplit, blockIdx);
}

// ---------------------------------------------------------------------------------------
// forward row pass over all modes of one wavelength (one mode chunk holds every mode).
// Vector v = rr*M + m takes row r = blockIdx.x*rpb + rr of probe mode (l, m); its probe row
// stays in registers while the block runs over the positions of its split; the object rows
// of the next position are copied into shared memory (cp.async) during the current one.
// grid (F/rpb, L, nsplit), block T*M*rpb <= 256, dynamic smem row_fwd_l_smem<F>(M, rpb)
// ---------------------------------------------------------------------------------------
template <int F>
__host__ __device__ constexpr int row_fwd_l_smem(int M, int rpb) {
  return (M * rpb * Xch<F>::region_rows + 2 * rpb * F) * (int)sizeof(float2);
}

template <int F>
__global__ void __launch_bounds__(256, (F <= 256 ? 2 : 1))
k_row_fwd_l(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S, KArgs a, int rpb,
            int nsplit) {
  pdl_wait();
  pdl_trigger();
  constexpr int N1 = FftShape<F>::N1, N2 = FftShape<F>::N2, T = N1, RR = Xch<F>::region_rows;
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int M = a.M, V = M * rpb;
  float2* xch = smem;                                 // [V][RR]
  float2* Ost = xch + V * RR;                         // [2][rpb][F]
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int rr = vec / M, m = vec % M;
  const int row0 = blockIdx.x * rpb, r = row0 + rr;
  const int l = blockIdx.y, split = blockIdx.z;
  const int cm = l * M + m - a.chunk_base;
  stage_batch(a, l, spos, ssig);
  float2 pr[N2];
  {
    const float2* Prow = P + ((long long)(l * M + m) * F + r) * F;
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) pr[n2] = __ldg(Prow + t + N1 * n2);
  }
  const float2* Ol = O + a.obj_off[l];
  const int Wl = a.obj_w[l];
  int b = next_of_split(spos, split - nsplit, a.nb, nsplit);
  if (b >= 0) {
    prefetch_orows<F>(Ol, Wl, spos[b], row0, rpb, Ost);
    cp_async_commit();
  }
  for (int buf = 0; b >= 0; buf ^= 1) {
    cp_async_wait<0>();
    __syncthreads();                                  // position b's rows have landed; buf^1 is free
    const int bn = next_of_split(spos, b, a.nb, nsplit);
    if (bn >= 0) {
      prefetch_orows<F>(Ol, Wl, spos[bn], row0, rpb, Ost + (buf ^ 1) * rpb * F);
      cp_async_commit();
    }
    const float s = ssig[b];
    const float2* orow = Ost + (buf * rpb + rr) * F;
    float2 v[N2];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) v[n2] = cmul(pr[n2], cscale(orow[t + N1 * n2], s));
    fft_fwd_I2O<F>(v, t, xch + vec * RR, a.tw, WarpSync{});
    float2* out = S + (((long long)b * a.C + cm) * F + r) * F;
#pragma unroll
    for (int sl = 0; sl < N2; ++sl) out[idxO<F>(t, sl)] = v[sl];
    b = bn;
  }
}

// Same pass at F = 512 with one warp per row (fft512_fwd_warp): the probe row takes 16 values per
// lane in registers instead of 32, so two blocks of up to 10 warps fit on an SM.
// grid (512/rpb, L, nsplit), block 32*M*rpb <= kRowAdjWThreads, dynamic smem row_fwd_w_smem(M, rpb)
__host__ __device__ constexpr int row_fwd_w_smem(int M, int rpb) {
  return (M * rpb * kFft512WarpXchF + 2 * rpb * 512) * (int)sizeof(float2);
}

template <int F>
__global__ void __launch_bounds__(kRowAdjWThreads, 2)
k_row_fwd_w(const float2* __restrict__ O, const float2* __restrict__ P, float2* __restrict__ S, KArgs a, int rpb,
            int nsplit) {
  static_assert(F == 512, "one warp per row is the 512-point layout");
  pdl_wait();
  pdl_trigger();
  constexpr int RR = kFft512WarpXchF;
  extern __shared__ __align__(16) float2 smem[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  const int M = a.M, V = M * rpb;
  float2* xch = smem;                                 // [V][RR]
  float2* Ost = xch + V * RR;                         // [2][rpb][F]
  const int vec = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int rr = vec / M, m = vec % M;
  const int row0 = blockIdx.x * rpb, r = row0 + rr;
  const int l = blockIdx.y, split = blockIdx.z;
  const int cm = l * M + m - a.chunk_base;
  stage_batch(a, l, spos, ssig);
  float2 pr[16];
  {
    const float2* Prow = P + ((long long)(l * M + m) * F + r) * F;
#pragma unroll
    for (int n2 = 0; n2 < 16; ++n2) pr[n2] = __ldg(Prow + t + 32 * n2);
  }
  const float2* Ol = O + a.obj_off[l];
  const int Wl = a.obj_w[l];
  const int oc = (t & 15) + 256 * (t >> 4);           // output column of x[0] (then + 16 j)
  int b = next_of_split(spos, split - nsplit, a.nb, nsplit);
  if (b >= 0) {
    prefetch_orows<F>(Ol, Wl, spos[b], row0, rpb, Ost);
    cp_async_commit();
  }
  for (int buf = 0; b >= 0; buf ^= 1) {
    cp_async_wait<0>();
    __syncthreads();                                  // position b's rows have landed; buf^1 is free
    const int bn = next_of_split(spos, b, a.nb, nsplit);
    if (bn >= 0) {
      prefetch_orows<F>(Ol, Wl, spos[bn], row0, rpb, Ost + (buf ^ 1) * rpb * F);
      cp_async_commit();
    }
    const float s = ssig[b];
    const float2* orow = Ost + (buf * rpb + rr) * F;
    float2 v[16];
#pragma unroll
    for (int n2 = 0; n2 < 16; ++n2) v[n2] = cmul(pr[n2], cscale(orow[t + 32 * n2], s));
    fft512_fwd_warp(v, t, xch + vec * RR, a.tw);
    float2* out = S + (((long long)b * a.C + cm) * F + r) * F + oc;
#pragma unroll
    for (int j = 0; j < 16; ++j) out[16 * j] = v[j];
    b = bn;
  }
}

// Fixed-order sum of the per-split probe-gradient buffers: out[i] = sum_s part[s][i].
__global__ void k_sum_splits(const float2* __restrict__ part, int nsplit, long long n, float2* __restrict__ out);

// ---------------------------------------------------------------------------------------
// object gradient from one mode-summed slot per (position, wavelength) (after k_row_adj_l):
// one block per tile (32 columns, 8 KR rows) of grad O_l inside the batch's bounding box.  The positions
// whose patches overlap the tile are listed first (ascending), then added in groups with
// their loads issued together: 16 / KR patches of KR rows per thread.  KR = 4 unless that leaves SMs
// idle (k_obj_grad_l's launch).   grid (tiles of the largest box, L)
// ---------------------------------------------------------------------------------------
template <int F, bool PAIR = false, int KR = 4>
__device__ __forceinline__ void obj_grad_l_body(const float2* __restrict__ S, float2* __restrict__ gO, const KArgs& a,
                                                const uint3 bid) {
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  __shared__ int list[kMaxB];
  __shared__ int nlist;
  const int l = bid.y;
  const int by0 = a.box[l][0], bx0 = a.box[l][1];
  const int ntx = (a.box[l][3] - bx0 + kTile - 1) / kTile;
  constexpr int TH = 8 * KR;                          // tile height
  const int nty = (a.box[l][2] - by0 + TH - 1) / TH;
  if ((int)bid.x >= ntx * nty) return;          // uniform over the block
  stage_batch(a, l, spos, ssig);
  const int oy0 = by0 + ((int)bid.x / ntx) * TH, ox0 = bx0 + ((int)bid.x % ntx) * kTile;
  if (threadIdx.x < 32) {                             // ordered compaction by warp 0
    int n = 0;
    for (int b0 = 0; b0 < a.nb; b0 += 32) {
      const int b = b0 + (int)threadIdx.x;
      bool hit = false;
      if (b < a.nb) {
        const int y = spos[b].x, x = spos[b].y;
        hit = !(y < 0 || y >= oy0 + TH || y + F <= oy0 || x >= ox0 + kTile || x + F <= ox0);
      }
      const unsigned mask = __ballot_sync(0xffffffffu, hit);
      if (hit) list[n + __popc(mask & ((1u << threadIdx.x) - 1u))] = b;
      n += __popc(mask);
    }
    if (threadIdx.x == 0) nlist = n;
  }
  __syncthreads();
  const int n = nlist;
  const int H = a.obj_h[l], Wd = a.obj_w[l];
  const int tx = threadIdx.x % kTile, ty0 = threadIdx.x / kTile;   // 8 row slots
  const int ox = ox0 + tx;
  const int slot0 = l * a.M - a.chunk_base;
  float2 acc[KR];
#pragma unroll
  for (int k = 0; k < KR; ++k) acc[k] = make_float2(0.f, 0.f);
  constexpr int PG = 16 / KR;                         // patches per group of loads
  for (int i0 = 0; i0 < n; i0 += PG) {
    float2 v[PG][KR];
#pragma unroll
    for (int pp = 0; pp < PG; ++pp) {
      const int b = i0 + pp < n ? list[i0 + pp] : -1;
      const int y = b >= 0 ? spos[b].x : 0, x = b >= 0 ? spos[b].y : 0;
      const bool in_x = b >= 0 && ox >= x && ox < x + F;
      const int bs = b >= 0 ? b : 0;
      const float2* src = PAIR ? S + ((long long)(bs >> 1) * a.C + slot0) * 2 * F * F + (bs & 1) * F + (ox - x)
                               : S + ((long long)bs * a.C + slot0) * F * F + (ox - x);
#pragma unroll
      for (int k = 0; k < KR; ++k) {
        const int oy = oy0 + ty0 + 8 * k;
        const bool ok = in_x && oy >= y && oy < y + F;
        v[pp][k] = ok ? src[(long long)(oy - y) * (PAIR ? 2 * F : F)] : make_float2(0.f, 0.f);
      }
    }
#pragma unroll
    for (int pp = 0; pp < PG; ++pp)
#pragma unroll
      for (int k = 0; k < KR; ++k) acc[k] = cadd(acc[k], v[pp][k]);
  }
  float2* g = gO + a.obj_off[l];
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const int oy = oy0 + ty0 + 8 * k;
    if (oy < H && ox < Wd) {
      float2* p = g + (long long)oy * Wd + ox;
      *p = cadd(*p, acc[k]);
    }
  }
}

// PAIR: the slots of the pair passes (rows of 2 F float2: lane 0's row, then lane 1's).
template <int F, bool PAIR, int KR>
__global__ void __launch_bounds__(256)
k_obj_grad_l(const float2* __restrict__ S, float2* __restrict__ gO, KArgs a) {
  pdl_wait();
  pdl_trigger();
  obj_grad_l_body<F, PAIR, KR>(S, gO, a, blockIdx);
}

// ---------------------------------------------------------------------------------------
// fixed-order sums
// ---------------------------------------------------------------------------------------
constexpr int kReduceThreads = 256, kReduceBlocks = 8;
__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
// Sum over i = first, first + stride, ... < n of part[i], over a block of kReduceThreads threads; valid in
// thread 0.
__device__ __forceinline__ double block_sum_partials(const double* __restrict__ part, long long n, int first, int stride,
                                                     double* red) {
  constexpr int U = 4;
  double s[U];
#pragma unroll
  for (int u = 0; u < U; ++u) s[u] = 0.0;
  long long i = first;
  for (; i + (U - 1) * stride < n; i += U * stride)
#pragma unroll
    for (int u = 0; u < U; ++u) s[u] += part[i + u * stride];
  for (; i < n; i += stride) s[0] += part[i];
  const double v = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kReduceThreads / 32; ++w) t += red[w];
  return t;
}
// f(i) by a whole warp for every call entry i with bidx[i] = j, in order.
template <class Fn>
__device__ __forceinline__ void for_entries_of(const int32_t* __restrict__ bidx, int nbatch, int j, int lane, Fn&& f) {
  for (int i0 = 0; i0 < nbatch; i0 += 32) {
    unsigned hit = __ballot_sync(0xffffffffu, i0 + lane < nbatch && __ldg(bidx + i0 + lane) == j);
    for (; hit; hit &= hit - 1) f(i0 + __ffs(hit) - 1);
  }
}

// ---------------------------------------------------------------------------------------
// loss reduction and Adam (defined in ptycho_capi.cu)
// ---------------------------------------------------------------------------------------
__global__ void k_loss_reduce(const double* __restrict__ part, long long n, double* out);   // grid kReduceBlocks
__global__ void k_sigma_grad(const int32_t* __restrict__ bidx, int nbatch, int J, const double* __restrict__ part,
                             int nblk, const float* __restrict__ sigma, float* __restrict__ g);
__global__ void k_sum_sets(const float* __restrict__ acc, int nsets, long long n, float* __restrict__ out);
__global__ void k_tick(int* t);
// Real parameters of one array with their gradient, moments and learning rate.
struct AdamArray {
  float* theta;
  const float* grad;
  float* m;
  float* v;
  long long n;
  float lr;
};
__global__ void k_adam_dev(AdamArray p, AdamArray q, float b1, float b2, float eps, const int* __restrict__ t_dev);
__global__ void k_adam(AdamArray p, AdamArray q, float b1, float b2, float eps, float c1, float c2);

}  // namespace ptycho
