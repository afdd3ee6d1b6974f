// The DFT passes over pairs of scan positions: the default pipeline of every plan that keeps all
// fields of a position in the scratch.
//
// Positions 2p and 2p + 1 of a batch (same wavelength, same probe mode) ride in the two lanes of the
// packed FP32 instructions (cpair), so one instruction, one twiddle, one probe value and one address
// serve two fields.  The scratch holds a pair as interleaved float4 elements
//
//   S4[((p*C + mode)*F + r)*F + c] = (re of 2p, re of 2p+1, im of 2p, im of 2p+1),
//
// so every load is a whole operand and no lane ever needs moving.  An odd last position has an empty
// second lane (zeros; nothing of it is written outside the scratch).  The arithmetic of each lane is
// that of the one-field kernels in kernels.cuh, operation by operation: patterns and losses are the same bits
// given the same batches and mode groups (the probe gradient's positions are dealt to its splits in pairs here).
//
// Why: ncu counted 31-46 thread instructions per field element and 1D DFT in the one-field passes
// (256^2 and 512^2), 90 ms of pure issue time in the 136 ms of the 512^2 x 6 wavelengths x 10 modes
// step, beside 88 ms of HBM time; packed passes need about half.
//
// Layout of the work.  A 1D DFT of F points is done by T = F/16 threads with 16 element pairs each
// (F <= 256: two-stage, 16 x T; F = 512: a warp, with the 32-point stage split over lanes l and
// l ^ 16).  The exchange between the stages reuses the shared memory that the vector arrived in, with
// an XOR of the low index bits in place of padding, so a pass needs no exchange buffer of its own.
// Column passes take tiles of CW columns of one pair and mode by TMA (128- or 64-byte rows, hardware
// swizzle: both the column reads and the exchange are free of bank conflicts), two tiles per block,
// the next mode's in flight; the adjoint writes its tile back by TMA.
#pragma once
#include "kernels.cuh"

namespace ptycho {

template <int F> struct PairCfg {
  static constexpr int T = F / 16;                   // threads per vector
  static constexpr int N = F == 512 ? 16 : T;        // exchange cells per k2
  static constexpr int VPW = 32 / T;                 // vectors per warp
  static constexpr int CW = F == 512 ? 4 : 8;        // columns per tile
  static constexpr int cthreads = CW * T;
  static constexpr int row_bytes = CW * 16;          // one row of a tile
  static constexpr int tile_bytes = F * row_bytes;
  // a row vector in shared memory: F float4; at F = 64 two vectors share an 8-lane access phase, and
  // an odd multiple of 64 bytes between them keeps the phase on all banks
  static constexpr int vec = F + (F == 64 ? 4 : 0);  // float4 elements
  // a probe row: F float2, padded likewise for its 16-lane access phases
  static constexpr int pvec = F + (T < 16 ? T : 0);  // float2 elements
  static constexpr int rows_fwd = 4 * VPW;           // rows per block of the forward row pass
  static constexpr int smem_row_fwd = rows_fwd * (vec * 16 + pvec * 8) + F * 8;
  static constexpr int smem_col = 2 * tile_bytes + (F == 512 ? F * 8 : 0) + 1024;   // tiles, twiddles, alignment
};

// A vector in shared memory.  Element p of a row vector lies at 16 p; of column c of a tile at row p,
// with the hardware swizzle: the 16-byte chunk index of a 128-byte line XOR the line index mod 8
// (128-byte rows) or mod 4 (64-byte rows, two to a line).  Exchange cell (k2, n1) of the transpose
// between the two stages is element k2*N + (n1 ^ (k2 & m)), m = min(7, N - 1): free of bank conflicts
// along both indices, and only the vector's own elements are touched.  All of that is linear over
// XOR, so an access is one XOR of a thread constant with a compile-time one:
//   along(k): cell (k, n1) for this thread's n1 and a constant k;  across(n): cell (k2, n) for this
//   thread's k2 and a constant n.
template <int F, bool COL> struct Place {
  static constexpr int N = PairCfg<F>::N, m = N >= 8 ? 7 : N - 1;
  char* base;
  int e0, x, y;                                      // element t; cell (0, n1); cell (k2, 0)
  static __device__ __forceinline__ constexpr int swz(int p) {   // element p of column 0 (or of the row), bytes
    if (!COL) return 16 * p;
    if (F == 512) return p * 64 + (((p >> 1) & 3) << 4);
    return p * 128 + ((p & 7) << 4);
  }
  // n1, k2: this thread's indices; c: its column
  __device__ __forceinline__ Place(char* b, int c, int t, int n1, int k2) : base(b) {
    const int cc = COL ? c << 4 : 0;
    e0 = swz(t) ^ cc;
    x = swz(n1) ^ cc;
    y = swz(k2 * N + (k2 & m)) ^ cc;
  }
  __device__ __forceinline__ float4* ptr(int off) const { return reinterpret_cast<float4*>(base + off); }
  // elements t + T i (T a multiple of 8, or 4 with its own swizzle step) and any element p
  __device__ __forceinline__ float4* elem(int i) const {
    constexpr int T = PairCfg<F>::T;
    return ptr((e0 ^ (COL && T == 4 ? (i & 1) << 6 : 0)) + T * i * (COL ? PairCfg<F>::row_bytes : 16));
  }
  __device__ __forceinline__ float4* along(int k) const {
    // element k*N + (n1 ^ (k & m)); at N = 4 bit 2 of the element index is bit 0 of k
    return ptr((x ^ swz(k & m) ^ (COL && N == 4 ? (k & 1) << 6 : 0)) + k * N * (COL ? PairCfg<F>::row_bytes : 16));
  }
  __device__ __forceinline__ float4* across(int n, int q = 0) const {   // cell (k2 + T q, n)
    return ptr((y ^ swz(n)) + q * PairCfg<F>::T * N * (COL ? PairCfg<F>::row_bytes : 16));
  }
};

__device__ __forceinline__ cpair ld_pair(const float4* p) {
  const float4 v = *p;
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void st_pair(float4* p, cpair v) { *p = make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }

// The bounded wait of a whole warp, with one outcome for its lanes: a lane whose wait ran out must not leave
// alone, the others' warp-wide exchanges and shuffles count on it.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t phase, int* status) {
  return __all_sync(0xffffffffu, mbar_wait_bounded(bar, phase, status));
}

// A give-up's last look at a copy that may still be under way (fetch i of those that go round two buffers, one
// phase each time): a bounded chance to land before the block's shared memory goes to another one.
__device__ __forceinline__ void drain_fetch(uint64_t* bar, int i, int* status) {
  mbar_wait_bounded(&bar[i & 1], (i >> 1) & 1, status);
}

// Element index of slot i of thread t in spectrum order (layout O of fft_regs.cuh; at F = 512
// t + 32 i).  Natural order is t + T i.
template <int F> __device__ __forceinline__ int pidxO(int t, int i) {
  if constexpr (F == 512) return t + 32 * i;
  else return idxO<F>(t, i);
}

// E + T on lanes q = 0, E - T on lanes q = 1, of the pair of lanes l, l ^ 16 (E: even half, T: twiddled
// odd half).
__device__ __forceinline__ cpair half_butterfly(cpair x, int q) {
  cpair o;
  o.re.x = __shfl_xor_sync(0xffffffffu, x.re.x, 16);
  o.re.y = __shfl_xor_sync(0xffffffffu, x.re.y, 16);
  o.im.x = __shfl_xor_sync(0xffffffffu, x.im.x, 16);
  o.im.y = __shfl_xor_sync(0xffffffffu, x.im.y, 16);
  const float s = q ? -1.0f : 1.0f;                  // +-x is exact: o + s x rounds like the sum or difference
  return {__ffma2_rn(x.re, splat(s), o.re), __ffma2_rn(x.im, splat(s), o.im)};
}

// Where a transform takes its twiddles from: the table in shared memory, or this thread's fifteen factors
// in registers (the column passes at F <= 256, where 168 registers hold them: 32 of the 288 shared-memory
// wavefronts of a warp's column transform, 64 of 576 in the adjoint).
template <int F> struct TwTable {
  const float2* tw;
  int t;
  __device__ __forceinline__ float2 operator()(int k2) const { return tw[k2 * PairCfg<F>::N + t]; }
};
template <int F> struct TwRegs {
  float2 w[16];
  __device__ __forceinline__ TwRegs(const float2* __restrict__ tw, int t) {
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) w[k2] = __ldg(tw + k2 * PairCfg<F>::N + t);
  }
  __device__ __forceinline__ float2 operator()(int k2) const { return w[k2]; }
};

// The twiddle table W_F^(t*k2) (tw[k2*N1 + t]) in shared memory.  Through L1 the passes' own traffic evicts
// it (ncu: 17 % of the column passes' and 80 % of the row passes' L1 accesses missed), and one miss in the
// fifteen loads of a transform costs a trip to L2.  Ends without a barrier.
template <int F>
__device__ __forceinline__ const float2* stage_twiddles(const float2* __restrict__ tw, float2* dst, int thread, int threads) {
  for (int i = thread; i < F / 2; i += threads)
    reinterpret_cast<float4*>(dst)[i] = __ldg(reinterpret_cast<const float4*>(tw) + i);
  return dst;
}

// This thread's exchange indices: n1 and k2 (F = 512: the thread of column n1 = t & 15 holds half of
// its k2; row k2 = t).
template <int F> __device__ __forceinline__ int pair_n1(int t) { return F == 512 ? t & 15 : t; }

// Forward 1D DFT of one vector of pairs; x[i] = element t + T i in, pidxO(t, i) out.  ``pl``: the
// vector's shared memory (its elements must be in registers already); a vector belongs to one warp.
template <int F, bool COL, class Tw>
__device__ __forceinline__ void pair_fwd(cpair (&x)[16], int t, const Place<F, COL>& pl, const Tw& tw) {
  if constexpr (F == 512) {
    // thread (n1 = t & 15, q): n2 = 2 s + q, the 32-point stage over n2 split by the parity q
    const int q = t >> 4;                             // n1 = t & 15
    Dft<16, 1, false>::run(x);
    if (q) {
      static_for<1, 16>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        x[j] = twiddle_const<32, false, j>(x[j]);
      });
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = half_butterfly(x[j], q);
    // W512^(n1 k2), k2 = j + 16 q = 4 a + b, as W^(n1 b) * W^(4 n1 a) (apply_twiddles<512>)
    float2 wb[4], wa[4];
    wb[0] = make_float2(1.f, 0.f);
#pragma unroll
    for (int b = 1; b < 4; ++b) wb[b] = tw(b);
#pragma unroll
    for (int a = 0; a < 4; ++a) wa[a] = tw(4 * a + 16 * q);
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = cmul(x[j], (j & 3) ? cmul(wa[j >> 2], wb[j & 3]) : wa[j >> 2]);
    __syncwarp();
    const int off = q * 256 * (COL ? PairCfg<F>::row_bytes : 16);      // cells of k2 = 16 q
#pragma unroll
    for (int j = 0; j < 16; ++j) st_pair(pl.along(j) + off / 16, x[j]);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = ld_pair(pl.across(i));
    Dft<16, 1, false>::run(x);
  } else {
    constexpr int N1 = FftShape<F>::N1;
    Dft<16, 1, false>::run(x);
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) x[k2] = cmul(x[k2], tw(k2));
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) st_pair(pl.along(k2), x[k2]);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 16 / N1; ++q)
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) x[q * N1 + n1] = ld_pair(pl.across(n1, q));
#pragma unroll
    for (int q = 0; q < 16 / N1; ++q) Dft<N1, 1, false>::run(x + q * N1);
  }
}

// Inverse (adjoint, unscaled), the forward's factors in reverse order: spectrum order in, natural order
// (F = 512: (t & 15) + 16 i + 256 (t >> 4)) out.
template <int F, bool COL, class Tw>
__device__ __forceinline__ void pair_inv(cpair (&x)[16], int t, const Place<F, COL>& pl, const Tw& tw) {
  if constexpr (F == 512) {
    const int q = t >> 4;                             // n1 = t & 15
    Dft<16, 1, true>::run(x);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) st_pair(pl.across(i), x[i]);
    __syncwarp();
    // k2 = 2 s + q = 4 (s >> 1) + 2 (s & 1) + q; cell (2 s + q, n1): along() shifted by q
    const float2 wb0 = q ? tw(1) : make_float2(1.f, 0.f), wb1 = tw(2 + q);
    Place<F, COL> pq = pl;
    pq.x ^= Place<F, COL>::swz(q);
    const int off = q * 16 * (COL ? PairCfg<F>::row_bytes : 16);
#pragma unroll
    for (int s = 0; s < 16; ++s) {
      x[s] = ld_pair(pq.along(2 * s) + off / 16);
      const float2 wb = (s & 1) ? wb1 : wb0;
      x[s] = cmulc(x[s], s < 2 ? wb : cmul(tw(4 * (s >> 1)), wb));
    }
    Dft<16, 1, true>::run(x);
    if (q) {
      static_for<1, 16>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        x[j] = twiddle_const<32, true, j>(x[j]);
      });
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = half_butterfly(x[j], q);
  } else {
    constexpr int N1 = FftShape<F>::N1;
#pragma unroll
    for (int q = 0; q < 16 / N1; ++q) Dft<N1, 1, true>::run(x + q * N1);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 16 / N1; ++q)
#pragma unroll
      for (int n1 = 0; n1 < N1; ++n1) st_pair(pl.across(n1, q), x[q * N1 + n1]);
    __syncwarp();
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) x[k2] = ld_pair(pl.along(k2));
#pragma unroll
    for (int k2 = 1; k2 < 16; ++k2) x[k2] = cmulc(x[k2], tw(k2));
    Dft<16, 1, true>::run(x);
  }
}

// Inverse of a row vector at F = 512 with the stages in the order of fft512_inv_warp (the 32-point stage
// first); element t + 32 i in and out.  x holds the spectrum on entry.
template <class Tw>
__device__ __forceinline__ void pair512_inv_rows(cpair (&x)[16], int t, const Place<512, false>& pl, const Tw& tw) {
  const int q = t >> 4;                               // c = t & 15
  Dft<16, 1, true>::run(x);
  if (q) {
    static_for<1, 16>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      x[j] = twiddle_const<32, true, j>(x[j]);
    });
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) x[j] = half_butterfly(x[j], q);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    if (j > 0 || q) x[j] = cmulc(x[j], tw(j + 16 * q));
    st_pair(pl.along(j) + q * 256, x[j]);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = ld_pair(pl.across(k));
  Dft<16, 1, true>::run(x);
}

// Position and power of lane e of pair p (invalid: y = -1, power 0).
struct PairPos {
  int2 yx[2];
  float s[2];
};
__device__ __forceinline__ PairPos pair_pos(const KArgs& a, int p, int l) {
  PairPos o;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int b = 2 * p + e;
    const int j = b < a.nb ? batch_pos(a, a.batch_off + b) : -1;
    o.yx[e] = make_int2(-1, -1);
    o.s[e] = 0.f;
    if (j >= 0) {
      o.yx[e] = make_int2(a.pos[(l * a.J + j) * 2], a.pos[(l * a.J + j) * 2 + 1]);
      o.s[e] = sigma_of(a, j);
    }
  }
  return o;
}

// ---------------------------------------------------------------------------------------
// forward row pass: exit waves of both lanes and the row DFT, every mode of wavelength l.  Each warp
// (32/T rows) works alone over the pairs chunk, chunk + nchunk, ...: the object rows of both lanes stay
// in registers over the modes, the probe row of the next mode (a bulk copy; BULK = false, for probes
// that are not 16-byte aligned: 8-byte cp.async) arrives during the current transform.
// grid (nchunk, F/rows_fwd, L), block 128: the chunks vary fastest, so that concurrent blocks share probe
// rows in L2; a block takes about kRowFwdPairs pairs, so that the rows in use stay far below its size.
// ---------------------------------------------------------------------------------------
constexpr int kRowFwdPairs = 4;
// Calls of a pair plan that take the one-field passes: subsets of up to this many positions, whose pairs are too few
// blocks for the chip (a single position leaves half of every pass empty as well).  us a step, pair / one-field:
// 256^2 x 30 fields 3 positions 198 / 161, 6 218 / 214, 8 257 / 270; 256^2 x 10 5 117 / 100, 9 148 / 131, 12 156 / 159;
// 256^2 x 8 3 84 / 76, 7 114 / 104, 11 134 / 135; 128^2 x 30 3 98 / 89, 9 123 / 110, 12 138 / 131; 64^2 x 30 4 82 / 79,
// 12 83 / 87; 512^2 x 8 4 225 / 240.
constexpr int pair_subset(int F) { return F == 512 ? 1 : F == 128 ? 16 : 10; }

template <int F, bool BULK>
__global__ void __launch_bounds__(128, 3)
k_row_fwd_p(const float2* __restrict__ O, const float2* __restrict__ P, float4* __restrict__ S, KArgs a) {
  pdl_wait();
  pdl_trigger();
  using Cfg = PairCfg<F>;
  constexpr int T = Cfg::T, VPW = Cfg::VPW;
  extern __shared__ __align__(1024) unsigned char smem_pair[];
  __shared__ uint64_t bar[4];
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  uint64_t* pbar = &bar[threadIdx.x >> 5];
  const int r = blockIdx.y * Cfg::rows_fwd + vec, l = blockIdx.z, M = a.M;
  const int np = (a.nb + 1) / 2, step = gridDim.x;
  float4* xch = reinterpret_cast<float4*>(smem_pair) + vec * Cfg::vec;
  float2* Pst = reinterpret_cast<float2*>(smem_pair + Cfg::rows_fwd * Cfg::vec * 16) + vec * Cfg::pvec;
  const float2* Prow = P + ((long long)l * M * F + r) * F;
  auto fetch_probe = [&](int m) {
    if constexpr (BULK) {
      if ((threadIdx.x & 31) == 0) mbar_arrive_expect_tx(pbar, VPW * F * 8);
      __syncwarp();
      if (t == 0) bulk_load(Pst, Prow + (long long)m * F * F, F * 8, pbar);
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) cp_async8(Pst + t + T * i, Prow + (long long)m * F * F + t + T * i);
      mbar_arrive_cp_async(pbar);
    }
  };
  if ((threadIdx.x & 31) == 0) {
    mbar_init(pbar, BULK ? 1 : 32);
    fence_mbar_init();
  }
  __syncwarp();
  int p = blockIdx.x;                                 // < np
  fetch_probe(0);
  PairPos pp = pair_pos(a, p, l);
  const TwTable<F> tw{stage_twiddles<F>(a.tw, reinterpret_cast<float2*>(smem_pair + Cfg::rows_fwd * (Cfg::vec * 16 + Cfg::pvec * 8)),
                                        threadIdx.x, 128), pair_n1<F>(t)};
  __syncthreads();
  const Place<F, false> pl(reinterpret_cast<char*>(xch), 0, t, pair_n1<F>(t), t);
  uint32_t phase = 0;
  for (; p < np; p += step) {
    cpair ob[16];                                     // sigma times the object rows, 0 in an empty lane
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const bool valid = pp.yx[e].x >= 0;             // uniform over the block
      const float2* Orow = (a.patch ? a.patch + (((long long)(2 * p + e) * a.L + l) * F + r) * F
                                    : O + a.obj_off[l] + (long long)(pp.yx[e].x + r) * a.obj_w[l] + pp.yx[e].y) + t;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float2 v = valid ? cscale(__ldg(Orow + T * i), pp.s[e]) : make_float2(0.f, 0.f);
        (e ? ob[i].re.y : ob[i].re.x) = v.x;
        (e ? ob[i].im.y : ob[i].im.x) = v.y;
      }
    }
    const bool more = p + step < np;
    if (more) pp = pair_pos(a, p + step, l);
    float4* out = S + (((long long)p * a.C + l * M) * F + r) * F;
    for (int m = 0; m < M; ++m, out += F * F) {
      if (!mbar_wait_warp(pbar, phase, a.status)) {
        mbar_wait_bounded(pbar, phase, a.status);     // the only copy under way
        return;
      }
      phase ^= 1;
      cpair x[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] = cmul(Pst[t + T * i], ob[i]);
      __syncwarp();                                   // the buffer has been read
      if (m + 1 < M || more) {
        fence_proxy_async_smem();
        fetch_probe(m + 1 < M ? m + 1 : 0);
      }
      pair_fwd<F>(x, t, pl, tw);
#pragma unroll
      for (int i = 0; i < 16; ++i) st_pair(out + pidxO<F>(t, i), x[i]);
    }
  }
}

// ---------------------------------------------------------------------------------------
// column passes
// ---------------------------------------------------------------------------------------
template <int F>
__device__ __forceinline__ void pair_tile_issue(char* tile, const CUtensorMap* map, int col0, int row0, uint64_t* bar) {
  constexpr int H = F < 256 ? F : 256;               // rows per box
  mbar_arrive_expect_tx(bar, PairCfg<F>::tile_bytes);
#pragma unroll
  for (int h = 0; h < F / H; ++h)
    tma_load_2d(tile + h * H * PairCfg<F>::row_bytes, map, 4 * col0, row0 + h * H, bar);
}
template <int F>
__device__ __forceinline__ void pair_tile_store(const char* tile, const CUtensorMap* map, int col0, int row0) {
  constexpr int H = F < 256 ? F : 256;
#pragma unroll
  for (int h = 0; h < F / H; ++h) tma_store_2d(map, 4 * col0, row0 + h * H, tile + h * H * PairCfg<F>::row_bytes);
  bulk_commit();
}

// Column of the tile and thread of the column.  At F = 64 (4 threads a column) an 8-lane access phase
// covers two columns: c and c + 4, whose swizzled chunks never meet.
template <int F>
__device__ __forceinline__ void pair_col_thread(int& c, int& t) {
  constexpr int T = PairCfg<F>::T;
  const int ci = threadIdx.x / T;
  t = threadIdx.x % T;
  c = T == 4 ? (ci & 1) * 4 + (ci >> 1) : ci;
}

template <int F>
__device__ __forceinline__ auto pair_col_twiddles(const float2* __restrict__ tw, char* smem, int t) {
  if constexpr (F == 512)
    return TwTable<F>{stage_twiddles<F>(tw, reinterpret_cast<float2*>(smem), threadIdx.x, PairCfg<F>::cthreads), t & 15};
  else
    return TwRegs<F>(tw, t);
}

// forward: column DFT, |Psi|^2 of both lanes summed over a mode group.  grid (F/CW, G, pairs)
template <int F>
__global__ void __launch_bounds__(PairCfg<F>::cthreads, 384 / PairCfg<F>::cthreads)
k_col_fwd_p(const __grid_constant__ CUtensorMap map, float* __restrict__ Ipart, KArgs a) {
  pdl_wait();
  pdl_trigger();
  constexpr int CW = PairCfg<F>::CW, TB = PairCfg<F>::tile_bytes;
  extern __shared__ __align__(1024) unsigned char smem_pair[];
  __shared__ uint64_t bar[2];
  char* tile = reinterpret_cast<char*>(smem_pair) + ((1024u - (smem_addr(smem_pair) & 1023u)) & 1023u);
  int c, t;
  pair_col_thread<F>(c, t);
  const auto tw = pair_col_twiddles<F>(a.tw, tile + 2 * TB, t);
  const int col0 = blockIdx.x * CW, g = blockIdx.y, p = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG);
  const int row0 = (p * a.C + m0) * F;                // first row of mode m0 in the map
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
    if (m0 < m1) pair_tile_issue<F>(tile, &map, col0, row0, &bar[0]);
  }
  __syncthreads();
  float2 acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = make_float2(0.f, 0.f);
  bool ok = true;
  int k = 0;
  for (; k < m1 - m0; ++k) {
    const int buf = k & 1;
    ok = __syncthreads_and(mbar_wait_bounded(&bar[buf], (k >> 1) & 1, a.status));   // the other tile is free too
    if (!ok) break;
    if (threadIdx.x == 0 && k + 1 < m1 - m0) {
      fence_proxy_async_smem();
      pair_tile_issue<F>(tile + (buf ^ 1) * TB, &map, col0, row0 + (k + 1) * F, &bar[buf ^ 1]);
    }
    const Place<F, true> pl(tile + buf * TB, c, t, pair_n1<F>(t), t);
    cpair x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = ld_pair(pl.elem(i));
    pair_fwd<F>(x, t, pl, tw);
#pragma unroll
    for (int i = 0; i < 16; ++i) add_abs2(acc[i], x[i]);
  }
  if (!ok) {                                          // give a lost copy a bounded chance to land, then stop
    if (threadIdx.x == 0) mbar_wait_bounded(&bar[k & 1], (k >> 1) & 1, a.status);
    return;
  }
  // the sums go out through shared memory, so that a warp writes whole row pieces
  __syncthreads();
  float* st = reinterpret_cast<float*>(tile);         // [2][F][CW]
  const float inv = 1.0f / (float)F;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int r = pidxO<F>(t, i);
    st[r * CW + c] = acc[i].x * (inv * inv);
    st[(F + r) * CW + c] = acc[i].y * (inv * inv);
  }
  __syncthreads();
  const int cc0 = (col0 + F / 2) & (F - 1);
  const int lanes = min(2, a.nb - 2 * p);
  for (int e = threadIdx.x; e < lanes * F * (CW / 4); e += PairCfg<F>::cthreads) {
    const int h = e % (CW / 4), r = (e / (CW / 4)) % F, lane = e / (CW / 4) / F;
    float* dst = Ipart + ((long long)(2 * p + lane) * a.G + g) * F * F;
    *reinterpret_cast<float4*>(dst + ((r + F / 2) & (F - 1)) * F + cc0 + 4 * h) =
        *reinterpret_cast<const float4*>(st + (lane * F + r) * CW + 4 * h);
  }
}

// adjoint: column DFT again, (2/F) G Psi, inverse column DFT, in place.  grid (F/CW, G, pairs)
template <int F>
__global__ void __launch_bounds__(PairCfg<F>::cthreads, 384 / PairCfg<F>::cthreads)
k_col_adj_p(const __grid_constant__ CUtensorMap map, KArgs a, AdjArgs aa) {
  pdl_wait();
  pdl_trigger();
  constexpr int CW = PairCfg<F>::CW, TB = PairCfg<F>::tile_bytes;
  extern __shared__ __align__(1024) unsigned char smem_pair[];
  __shared__ uint64_t bar[2];
  char* tile = reinterpret_cast<char*>(smem_pair) + ((1024u - (smem_addr(smem_pair) & 1023u)) & 1023u);
  int c, t;
  pair_col_thread<F>(c, t);
  const auto tw = pair_col_twiddles<F>(a.tw, tile + 2 * TB, t);
  const int col0 = blockIdx.x * CW, g = blockIdx.y, p = blockIdx.z;
  const int m0 = g * a.MG, m1 = min(a.chunk_len, m0 + a.MG), nm = m1 - m0;
  const int row0 = (p * a.C + m0) * F;
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
    if (nm > 0) pair_tile_issue<F>(tile, &map, col0, row0, &bar[0]);
  }
  // the dL/dI factors of this tile's columns through the second tile (not in use yet), then in
  // registers for every mode of the group
  float* st = reinterpret_cast<float*>(tile + TB);    // [2][F][CW]
  {
    const float* G = aa.remap ? aa.Gt : aa.D;
    const int cc0 = (col0 + F / 2) & (F - 1);
    // 2/F of the adjoint, 1/F of the recomputed Psi, and sigma, a factor of both gradients
    float scale[2] = {0.f, 0.f};
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 2 * p + e < a.nb ? batch_pos(a, a.batch_off + 2 * p + e) : -1;
      if (j >= 0) scale[e] = 2.0f / (float)F / (float)F * sigma_of(a, j);
    }
    for (int e = threadIdx.x; e < 2 * F * (CW / 4); e += PairCfg<F>::cthreads) {
      const int h = e % (CW / 4), r = (e / (CW / 4)) % F, lane = e / (CW / 4) / F;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (2 * p + lane < a.nb)
        v = *reinterpret_cast<const float4*>(G + (long long)(2 * p + lane) * F * F + ((r + F / 2) & (F - 1)) * F + cc0 + 4 * h);
      *reinterpret_cast<float4*>(st + (lane * F + r) * CW + 4 * h) =
          lane ? make_float4(v.x * scale[1], v.y * scale[1], v.z * scale[1], v.w * scale[1])
               : make_float4(v.x * scale[0], v.y * scale[0], v.z * scale[0], v.w * scale[0]);
    }
  }
  __syncthreads();
  float2 gk[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int r = pidxO<F>(t, i);
    gk[i] = make_float2(st[r * CW + c], st[(F + r) * CW + c]);
  }
  __syncthreads();
  if (threadIdx.x == 0 && nm > 1) {
    fence_proxy_async_smem();
    pair_tile_issue<F>(tile + TB, &map, col0, row0 + F, &bar[1]);
  }
  bool ok = true;
  int k = 0;
  for (; k < nm; ++k) {
    const int buf = k & 1;
    ok = __syncthreads_and(mbar_wait_bounded(&bar[buf], (k >> 1) & 1, a.status));
    if (!ok) break;
    const Place<F, true> pl(tile + buf * TB, c, t, pair_n1<F>(t), t);
    cpair x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = ld_pair(pl.elem(i));
    pair_fwd<F>(x, t, pl, tw);
    if (threadIdx.x == 0 && k > 0 && k + 1 < nm) {    // the other tile has been stored: fetch the next mode
      bulk_wait_read();
      pair_tile_issue<F>(tile + (buf ^ 1) * TB, &map, col0, row0 + (k + 1) * F, &bar[buf ^ 1]);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = cscale(x[i], gk[i]);
    pair_inv<F>(x, t, pl, tw);
    __syncwarp();
    if constexpr (F == 512) {                         // elements (t & 15) + 16 i + 256 (t >> 4)
      float4* o = pl.ptr(pl.x) + (t >> 4) * 256 * PairCfg<F>::row_bytes / 16;
#pragma unroll
      for (int i = 0; i < 16; ++i) st_pair(o + i * 16 * PairCfg<F>::row_bytes / 16, x[i]);
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) st_pair(pl.elem(i), x[i]);
    }
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) pair_tile_store<F>(tile + buf * TB, &map, col0, row0 + k * F);
  }
  if (threadIdx.x == 0) {
    if (!ok) mbar_wait_bounded(&bar[k & 1], (k >> 1) & 1, a.status);
    if (!ok && k == 0 && nm > 1) mbar_wait_bounded(&bar[1], 0, a.status);
    bulk_wait_read();                                 // the tiles may go once they have been read
  }
}

// ---------------------------------------------------------------------------------------
// adjoint row pass over all modes of one wavelength (two modes or more).  Vector v = rr*M + m takes row
// blockIdx.x*rpb + rr of mode m.  Per pair of the block's split: inverse row DFT of both lanes, the
// probe gradient summed in registers (lane 0's position first), the object-gradient rows
// conj(sigma P_m) chi left in the vector's shared memory (F values of lane 0, then F of lane 1).
// NPW further warps feed the block: they add the modes' rows (modes in order) and write the sum over
// row r of the pair's mode-0 field, then fetch the next pair but one into the freed buffer (scratch
// rows by bulk copies, object rows by 8-byte cp.async: x may be odd).  The compute warps wait for
// nothing but their buffer, so that their load, transform and store phases drift apart; with block
// barriers in their place all warps were in the same phase and used one pipe at a time (512^2 x 10
// modes: 3.32 ms per 3600 evaluations).
// grid (F/rpb, L, nsplit), block T*M*rpb + 32*NPW (T*M*rpb a multiple of 32), dynamic smem
// row_adj_p_smem<F>(M, rpb)
// ---------------------------------------------------------------------------------------
constexpr int kRowAdjPairThreads = 320;               // compute threads per block, at most
template <int F>
__host__ __device__ constexpr int row_adj_p_smem(int M, int rpb) {
  return 2 * M * rpb * PairCfg<F>::vec * 16 + 2 * rpb * F * 16 + F * 8;
}
// Feeding warps of a block of ct compute threads.  At most 384 threads of 168 registers: 12 warps per SM,
// in as many blocks as that makes.
constexpr int row_adj_p_feeders(int ct) { return ct <= 160 ? 1 : 2; }

// Whether every one of the block's NPW feeding warps agrees (their threads only, all of them); what any of
// them read from shared memory before, it has read.  A wait that ran out for one thread must end the loop
// of all: the others would stand at a barrier that nobody else comes to.
template <int NPW>
__device__ __forceinline__ bool feeders_agree(bool ok) {
  __syncwarp();
  ok = __all_sync(0xffffffffu, ok);
  if constexpr (NPW > 1) {
    uint32_t all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(all)
        : "r"((uint32_t)ok), "n"(32 * NPW)
        : "memory");
    ok = all != 0;
  }
  return ok;
}

// Next pair of this split after p with a valid position, or -1 (uniform over the block).
__device__ __forceinline__ int next_pair(const int2* spos, int p, int nb, int nsplit) {
  for (int q = p + nsplit; 2 * q < nb; q += nsplit)
    if (spos[2 * q].x >= 0 || (2 * q + 1 < nb && spos[2 * q + 1].x >= 0)) return q;
  return -1;
}

// Both gradients of one row element of a thread (x: sigma chi): acc += conj(p) sigma chi of each valid
// lane in lane order; returns conj(P) sigma chi.
__device__ __forceinline__ cpair pair_grads(const cpair& x, float4 o, float2 pr, bool v0, bool v1, float2& acc) {
  if (v0) acc_conjmul(acc, make_float2(o.x, o.y), make_float2(x.re.x, x.im.x));
  if (v1) acc_conjmul(acc, make_float2(o.z, o.w), make_float2(x.re.y, x.im.y));
  return cconjmul(pr, x);
}

template <int F, int NPW>
__global__ void __launch_bounds__(384, 1)
k_row_adj_p(const float2* __restrict__ O, const float2* __restrict__ P, float4* __restrict__ S,
            float2* __restrict__ gPs, long long gp_stride, KArgs a, int rpb, int nsplit) {
  pdl_wait();
  pdl_trigger();
  constexpr int T = PairCfg<F>::T, VEC = PairCfg<F>::vec, NPT = 32 * NPW;
  extern __shared__ __align__(1024) unsigned char smem_pair[];
  __shared__ int2 spos[kMaxB];
  __shared__ float ssig[kMaxB];
  __shared__ uint64_t full[2], done[2];
  const int M = a.M, V = M * rpb, CT = V * T;
  float4* Sst = reinterpret_cast<float4*>(smem_pair); // [2][V][VEC]
  float4* Ost = Sst + 2 * V * VEC;                    // [2][rpb][F]: (lane 0, lane 1)
  const float2* tw = stage_twiddles<F>(a.tw, reinterpret_cast<float2*>(Ost + 2 * rpb * F), threadIdx.x, blockDim.x);
  const int row0 = blockIdx.x * rpb, l = blockIdx.y, split = blockIdx.z;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full[i], 1 + NPT);
      mbar_init(&done[i], CT / 32);
    }
    fence_mbar_init();
  }
  stage_batch(a, l, spos, ssig);                      // ends with a block barrier
  int p = next_pair(spos, split - nsplit, a.nb, nsplit);
  if (threadIdx.x >= CT) {                            // feeding warps
    const int pt = threadIdx.x - CT;
    const float2* Ol = O + a.obj_off[l];
    auto fetch = [&](int q, int buf) {
      if (pt == 0) mbar_arrive_expect_tx(&full[buf], V * F * 16);
      for (int v = pt; v < V; v += NPT)
        bulk_load(Sst + (buf * V + v) * VEC, S + (((long long)q * a.C + l * M + v % M) * F + row0 + v / M) * F, F * 16,
                  &full[buf]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int b = 2 * q + e;
        if (b >= a.nb || spos[b].x < 0) continue;
        const int w = a.patch ? F : a.obj_w[l];
        const float2* src = (a.patch ? a.patch + (((long long)b * a.L + l) * F + row0) * F
                                     : Ol + (long long)(spos[b].x + row0) * w + spos[b].y) + pt;
        float2* dst = reinterpret_cast<float2*>(Ost + buf * rpb * F + pt) + e;
        for (int rr = 0; rr < rpb; ++rr, src += w, dst += 2 * F)
#pragma unroll
          for (int i = 0; i < F / NPT; ++i) cp_async8(dst + 2 * NPT * i, src + NPT * i);
      }
      mbar_arrive_cp_async(&full[buf]);
    };
    int pn = p >= 0 ? next_pair(spos, p, a.nb, nsplit) : -1;
    if (p >= 0) fetch(p, 0);
    if (pn >= 0) fetch(pn, 1);
    for (int k = 0; p >= 0; ++k) {
      const int buf = k & 1;
      const bool ok = mbar_wait_bounded(&done[buf], (k >> 1) & 1, a.status);
      float4* dst = S + (((long long)p * a.C + l * M) * F + row0) * F;  // the block's rows, contiguous
      for (int rr = 0; rr < (ok ? rpb : 0); ++rr) {
        const float4* red = Sst + (buf * V + rr * M) * VEC + pt;
#pragma unroll 4
        for (int i = 0; i < F / NPT; ++i) {
          float4 sum = red[NPT * i];
          for (int mm = 1; mm < M; ++mm) {            // modes added in order, two values at a time
            const float4 v = red[mm * VEC + NPT * i];
            const float2 lo = __fadd2_rn(make_float2(sum.x, sum.y), make_float2(v.x, v.y));
            const float2 hi = __fadd2_rn(make_float2(sum.z, sum.w), make_float2(v.z, v.w));
            sum = make_float4(lo.x, lo.y, hi.x, hi.y);
          }
          dst[rr * F + pt + NPT * i] = sum;
        }
      }
      const int p2 = pn >= 0 ? next_pair(spos, pn, a.nb, nsplit) : -1;
      if (!feeders_agree<NPW>(ok)) {                  // (else every feeder has read the buffer)
        drain_fetch(full, k, a.status);
        if (pn >= 0) drain_fetch(full, k + 1, a.status);
        break;
      }
      if (p2 >= 0) {
        fence_proxy_async_smem();
        fetch(p2, buf);
      }
      p = pn;
      pn = p2;
    }
    return;
  }
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int rr = vec / M, m = vec % M;
  const long long row = ((long long)(l * M + m) * F + row0 + rr) * F + t;
  float2 pr[16], acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    pr[i] = __ldg(P + row + T * i);
    acc[i] = make_float2(0.f, 0.f);
  }
  for (int k = 0; p >= 0; ++k, p = next_pair(spos, p, a.nb, nsplit)) {
    const int buf = k & 1;
    // (the feeding warps, which find done[buf] incomplete then, see to the copies under way)
    if (!mbar_wait_warp(&full[buf], (k >> 1) & 1, a.status)) return;
    const bool v0 = spos[2 * p].x >= 0, v1 = 2 * p + 1 < a.nb && spos[2 * p + 1].x >= 0;
    float4* reg = Sst + (buf * V + vec) * VEC;
    const Place<F, false> pl(reinterpret_cast<char*>(reg), 0, t, pair_n1<F>(t), t);
    cpair x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = ld_pair(reg + pidxO<F>(t, i));
    const TwTable<F> tt{tw, pair_n1<F>(t)};
    if constexpr (F == 512) pair512_inv_rows(x, t, pl, tt);
    else pair_inv<F>(x, t, pl, tt);
    __syncwarp();                                     // the exchange cells are free: object-gradient rows
    const float4* orow = Ost + (buf * rpb + rr) * F + t;
    float2* go = reinterpret_cast<float2*>(reg) + t;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const cpair g = pair_grads(x[i], orow[T * i], pr[i], v0, v1, acc[i]);
      go[T * i] = make_float2(g.re.x, g.im.x);
      go[F + T * i] = make_float2(g.re.y, g.im.y);
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&done[buf]);
  }
  float2* g = gPs + (long long)split * gp_stride + row;
#pragma unroll
  for (int i = 0; i < 16; ++i) g[T * i] = cadd(g[T * i], acc[i]);
}

// Object rows of both lanes of a pair, element t + T i of this thread, as (lane 0, lane 1) float2 pairs.
template <int F>
__device__ __forceinline__ void fetch_pair_rows(const float2* __restrict__ O, const KArgs& a, const PairPos& pp, int p,
                                                int l, int r, int t, float4* dst) {
  constexpr int T = PairCfg<F>::T;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    if (pp.yx[e].x < 0) continue;                     // uniform over the warp
    const float2* src = (a.patch ? a.patch + (((long long)(2 * p + e) * a.L + l) * F + r) * F
                                 : O + a.obj_off[l] + (long long)(pp.yx[e].x + r) * a.obj_w[l] + pp.yx[e].y) + t;
    float2* d = reinterpret_cast<float2*>(dst + t) + e;
#pragma unroll
    for (int i = 0; i < 16; ++i) cp_async8(d + 2 * T * i, src + T * i);
  }
}

// The same pass with one mode: no sum over modes, so a warp (32/T rows) works alone.  Its scratch rows
// arrive two pairs ahead by bulk copies; the object rows of the next pair (L2-resident) as soon as the
// current ones have been used.   grid (F/VPW, L, nsplit), block 32, dynamic smem row_adj_p1_smem<F>()
template <int F>
__host__ __device__ constexpr int row_adj_p1_smem() {
  return PairCfg<F>::VPW * (2 * PairCfg<F>::vec + F) * 16 + F * 8;
}

template <int F>
__global__ void __launch_bounds__(32, 12)
k_row_adj_p1(const float2* __restrict__ O, const float2* __restrict__ P, float4* __restrict__ S,
             float2* __restrict__ gPs, long long gp_stride, KArgs a, int nsplit) {
  pdl_wait();
  pdl_trigger();
  constexpr int T = PairCfg<F>::T, VEC = PairCfg<F>::vec, VPW = PairCfg<F>::VPW;
  extern __shared__ __align__(1024) unsigned char smem_pair[];
  __shared__ uint64_t full[2], obar;
  float4* Sst = reinterpret_cast<float4*>(smem_pair); // [2][VPW][VEC]
  float4* Ost = Sst + 2 * VPW * VEC;                  // [VPW][F]
  const float2* tw = stage_twiddles<F>(a.tw, reinterpret_cast<float2*>(Ost + VPW * F), threadIdx.x, 32);
  const int vec = threadIdx.x / T, t = threadIdx.x % T;
  const int r = blockIdx.x * VPW + vec, l = blockIdx.y, split = blockIdx.z;
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&obar, 32);
    fence_mbar_init();
  }
  __syncwarp();
  const int np = (a.nb + 1) / 2;
  auto fetch = [&](int q, int buf) {
    if (threadIdx.x == 0) mbar_arrive_expect_tx(&full[buf], VPW * F * 16);
    __syncwarp();
    if (t == 0) bulk_load(Sst + (buf * VPW + vec) * VEC, S + (((long long)q * a.C + l) * F + r) * F, F * 16, &full[buf]);
  };
  auto fetch_obj = [&](const PairPos& pp, int q) {
    fetch_pair_rows<F>(O, a, pp, q, l, r, t, Ost + vec * F);
    mbar_arrive_cp_async(&obar);
  };
  int p = split;
  if (p < np) fetch(p, 0);
  if (p + nsplit < np) fetch(p + nsplit, 1);
  PairPos pp = pair_pos(a, min(p, np - 1), l);
  if (p < np) fetch_obj(pp, p);
  const long long row = ((long long)l * F + r) * F + t;
  float2 pr[16], acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    pr[i] = __ldg(P + row + T * i);
    acc[i] = make_float2(0.f, 0.f);
  }
  // what a give-up at pair k leaves under way: scratch rows from fetch i on, the object rows of pair k
  auto drain = [&](int i, int k) {
    for (int q = i; q < i + 2 && split + q * nsplit < np; ++q) drain_fetch(full, q, a.status);
    mbar_wait_bounded(&obar, k & 1, a.status);
  };
  for (int k = 0; p < np; ++k, p += nsplit) {
    const int buf = k & 1;
    const PairPos pn = pair_pos(a, min(p + nsplit, np - 1), l);
    if (!mbar_wait_warp(&full[buf], (k >> 1) & 1, a.status)) {
      drain(k, k);
      return;
    }
    float4* reg = Sst + (buf * VPW + vec) * VEC;
    const Place<F, false> pl(reinterpret_cast<char*>(reg), 0, t, pair_n1<F>(t), t);
    cpair x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = ld_pair(reg + pidxO<F>(t, i));
    const TwTable<F> tt{tw, pair_n1<F>(t)};
    if constexpr (F == 512) pair512_inv_rows(x, t, pl, tt);
    else pair_inv<F>(x, t, pl, tt);
    __syncwarp();                                     // the exchange cells have been read
    if (p + 2 * nsplit < np) {
      fence_proxy_async_smem();
      fetch(p + 2 * nsplit, buf);
    }
    if (!mbar_wait_warp(&obar, k & 1, a.status)) {
      drain(k + 1, k);
      return;
    }
    const bool v0 = pp.yx[0].x >= 0, v1 = pp.yx[1].x >= 0;
    float2* go = reinterpret_cast<float2*>(S + (((long long)p * a.C + l) * F + r) * F) + t;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const cpair g = pair_grads(x[i], Ost[vec * F + t + T * i], pr[i], v0, v1, acc[i]);
      go[T * i] = make_float2(g.re.x, g.im.x);
      go[F + T * i] = make_float2(g.re.y, g.im.y);
    }
    __syncwarp();                                     // the object rows have been used
    pp = pn;
    if (p + nsplit < np) fetch_obj(pp, p + nsplit);
  }
  float2* g = gPs + (long long)split * gp_stride + row;
#pragma unroll
  for (int i = 0; i < 16; ++i) g[T * i] = cadd(g[T * i], acc[i]);
}

}  // namespace ptycho
