// Spectral step in FP32 on the CUDA cores: plans created with precision 1, and
// every power-of-two band count but 64.
//
// The same updates as the tensor-core kernels (Alg. 2 eqs. vt, v, upt and the
// derivative forms of Algs. 3/4), with the orthonormal DCT-II of each pixel
// spectrum (W_lambda, Sec. 4.2.1) computed by a fast transform instead of a
// dense L x L product.  Makhoul's reordering (IEEE Trans. ASSP 28(1), 1980)
// turns a length-L DCT-II into one length-L complex DFT:
//   w_m = x_{2m}, w_{L-1-m} = x_{2m+1} (m < L/2),   W = DFT(w),
//   X'_k = sum_n x_n cos(pi k (2n + 1) / 2L) = Re(e^{-i pi k / 2L} W_k),
// and, for real w, X'_{L-k} = -Im(e^{-i pi k / 2L} W_k); backwards
//   W_k = e^{i pi k / 2L} (X'_k - i X'_{L-k})  (X'_L = 0),  w = DFT^-1(W) / L.
// The orthonormal coefficients are X_0 = X'_0 / sqrt(L), X_k = X'_k sqrt(2/L).
// Two pixels share one complex sequence (real and imaginary parts): after
// the forward DFT they are separated with Z_{L-k} = conj of the real parts'
// spectra, and before the inverse their Hermitian spectra are merged, so
// one DFT of length L serves two pixel spectra each way.  The DFTs are the
// shared-memory Stockham transforms of the gradient passes.  The work is
// O(L log L) per pixel, so the step is bound by its HBM traffic at every L
// (512 x 512 x 256, one chain: 0.28 ms, 4.8 TB/s; the dense 3xTF32 product on
// mma.sync took 1.74 ms).  Where tiles are few, 64-thread CTAs take a quarter of the
// pixels (64 x 64 x 32, three chains: 24.8 -> 17.6 us).  The old
// duals of a chain are requested before the chain's forward DFT (512 x 512 x
// 32, three chains: 165 -> 134 us), and chain 2's gamma v'_gamma + v is formed
// after the inverse DFTs, which are linear, so no dual stays in a register.
//
// A CTA owns a tile of PT = 2 NB pixels of one cube.  Phases: load z = 2 x~ -
// x of every band of the tile (float2 pairs of pixels, coalesced along the
// pixels) into the reordered positions; forward DFTs; per (pixel pair, band
// pair {k, L-k}) task: separate, scale, dual update against the old duals in
// HBM (chain 0 records the mask of sat, the derivative chains apply it),
// store the new duals and write the merged inverse input in place; inverse
// DFTs; store t = gamma alpha C^T v (chain 2: alpha C^T (gamma v'_gamma + v)).
#include <cuda_runtime.h>

#include <cmath>

#include "fft32.cuh"
#include "chain.cuh"
#include "kernels.h"

namespace muffin {

namespace {

// FT threads per CTA: 256, or 64 where the tiles of 256-thread CTAs are too
// few for the SMs
template <int L, int FT>
struct FShape {
  static constexpr int VPT = fft_vpt(L);
  static constexpr int NB0 = FT * VPT / L;            // sequences the DFT threads cover
  static constexpr int NB = NB0 > 128 ? 128 : NB0;    // pixel pairs per tile
  static constexpr int PT = 2 * NB;                   // pixels per tile
  // padded sequence length, odd so that 16 consecutive pairs hit distinct banks
  static constexpr int PITCH = ((L - 1) + (L - 1) / 16 + 1) | 1;
  static constexpr int NTASK = NB * (L / 2);
  static constexpr int TPT = (NTASK + FT - 1) / FT;   // tasks per thread
  static constexpr int KS = FT / NB;                  // band pairs between a thread's tasks
  static_assert(NB * L / VPT <= FT, "the DFT threads fit in the CTA");
  static_assert(FT % NB == 0, "a thread keeps one pixel pair");
  static_assert(TPT * 4 <= 32, "mask bits of a thread's tasks fit in 32 bits");
};

struct F32Args {
  int L, B;
  size_t npix;
  const float2 *tab;    // [tw_len] DFT stage twiddles, [L] (cos, sin)(pi k / 2L)
  int tw_len;
  const float *alpha;   // [B][npix]
  const DevScalars *sc; // [B]
  const float *xt, *x;  // iteration inputs [C][B][L][npix]
  float *v, *t;         // duals (in/out) and back-projection (out)
  const float *in;      // operator input [B][L][npix]
  float *out;           // operator output
  int inverse;          // operator: 0 C in, 1 C^T in
};

__device__ __forceinline__ float2 ld2(const float *p) {
  return *reinterpret_cast<const float2 *>(p);
}
__device__ __forceinline__ void st2(float *p, float2 v) {
  *reinterpret_cast<float2 *>(p) = v;
}

// position of band l in the reordered sequence
template <int L>
__device__ __forceinline__ int mpos(int l) {
  return (l & 1) ? L - 1 - (l >> 1) : (l >> 1);
}

template <int L, int CH, int MODE, int FT>
__global__ void __launch_bounds__(FT, FT == 64 ? 6 : 2) k_dct_f32(F32Args a) {
  chain_enter();
  using S = FShape<L, FT>;
  constexpr int NB = S::NB, PT = S::PT, PITCH = S::PITCH;
  extern __shared__ float2 fsm[];
  float2 *tw = fsm;                 // DFT stage twiddles
  float2 *mk = tw + a.tw_len;       // (cos, sin)(pi k / 2L)
  float2 *dat = mk + L;             // [CH][NB][PITCH]
  const int tid = threadIdx.x;
  const size_t N = a.npix;
  const size_t CS = (size_t)a.B * L * N;   // chain stride
  const size_t n0 = (size_t)blockIdx.x * PT;
  const int cube = blockIdx.y;
  const size_t cb = (size_t)cube * L * N;
  const bool fwd_op = MODE == WAVE_TRANSFORM && !a.inverse;
  const bool inv_op = MODE == WAVE_TRANSFORM && a.inverse;
  const float gamma = MODE == WAVE_ITERATE ? (float)a.sc[cube].gamma : 0.f;
  const float sigma = MODE == WAVE_ITERATE ? (float)a.sc[cube].sigma : 0.f;
  const float *__restrict__ alpha = a.alpha + (size_t)cube * N;
  const float r1 = rsqrtf((float)L), r2 = sqrtf(2.f / (float)L);   // s_0, s_k
  const float q1 = rsqrtf((float)L), q2 = rsqrtf(2.f * (float)L);  // inverse input scales
  const float rt2 = 1.41421356237309505f, ch4 = 0.70710678118654752f;

  for (int i = tid; i < a.tw_len + L; i += FT) fsm[i] = a.tab[i];

  // ---- z of every band of the tile, reordered
  if (!inv_op) {
    // loads of several rounds in flight before their first use
    constexpr int UNR = CH == 3 ? 3 : 8;
#pragma unroll UNR
    for (int it = tid; it < L * NB; it += FT) {
      const int s = it % NB, l = it / NB;
      const size_t pix = n0 + 2 * s;
      float2 z[CH];
#pragma unroll
      for (int c = 0; c < CH; ++c) z[c] = make_float2(0.f, 0.f);
      if (pix < N) {
        const size_t j = cb + (size_t)l * N + pix;
        if (MODE == WAVE_TRANSFORM) {
          z[0] = ld2(a.in + j);
        } else {
#pragma unroll
          for (int c = 0; c < CH; ++c) {
            const float2 xt = ld2(a.xt + c * CS + j), x = ld2(a.x + c * CS + j);
            z[c] = make_float2(2.f * xt.x - x.x, 2.f * xt.y - x.y);
          }
          if (CH == 3)   // Algorithm 4 input: gamma z'_gamma + z
            z[2] = make_float2(fmaf(gamma, z[2].x, z[0].x), fmaf(gamma, z[2].y, z[0].y));
        }
      }
      const int o = s * PITCH + fpad(mpos<L>(l));
#pragma unroll
      for (int c = 0; c < CH; ++c) dat[c * NB * PITCH + o] = z[c];
    }
  }
  // a thread's tasks share its pixel pair; the old duals of a chain are
  // requested before the chain's forward DFT, which covers their latency
  const int ps = tid % NB, kk0 = tid / NB;
  const size_t pix = n0 + 2 * ps;
  const bool valid = pix < N;
  constexpr int TPT = MODE == WAVE_ITERATE ? S::TPT : 1;
  float2 pv1[TPT], pv2[TPT], al = make_float2(0.f, 0.f);
  // (a pixel block of the sharded form starts anywhere: no vector load)
  if (MODE == WAVE_ITERATE && valid) al = make_float2(alpha[pix], alpha[pix + 1]);
  auto duals = [&](int c) {
#pragma unroll
    for (int r = 0; r < TPT; ++r) {
      const int kk = kk0 + r * S::KS;
      pv1[r] = pv2[r] = make_float2(0.f, 0.f);
      if (tid + r * FT < S::NTASK && valid) {
        const float *vp = a.v + c * CS + cb + pix;
        pv1[r] = ld2(vp + (size_t)kk * N);
        pv2[r] = ld2(vp + (size_t)(kk ? L - kk : L / 2) * N);
      }
    }
  };

  // ---- per (pixel pair, band pair) tasks
  uint32_t mask = 0;
#pragma unroll 1
  for (int c = 0; c < CH; ++c) {
    float2 *d = dat + c * NB * PITCH;
    if (MODE == WAVE_ITERATE) duals(c);
    if (c == 0) __syncthreads();   // tables and the tile
    if (!inv_op) fft_inplace<L, false>(d, NB, PITCH, tw);
#pragma unroll
    for (int r = 0; r < S::TPT; ++r) {
      if (tid + r * FT >= S::NTASK) break;
      const int s = ps, kk = kk0 + r * S::KS;
      const int k1 = kk, k2 = kk ? L - kk : L / 2;
      const float2 w = mk[kk];
      // orthonormal coefficients X[k1], X[k2] of pixels A (.x) and B (.y)
      float2 X1 = make_float2(0.f, 0.f), X2 = X1;
      if (!inv_op) {
        const float2 Z1 = d[s * PITCH + fpad(k1)], Z2 = d[s * PITCH + fpad(k2)];
        if (kk == 0) {
          X1 = make_float2(Z1.x * r1, Z1.y * r1);
          X2 = make_float2(Z2.x * (ch4 * r2), Z2.y * (ch4 * r2));
        } else {
          // halves of the separated spectra V_A[k1], V_B[k1]
          const float ax = Z1.x + Z2.x, ay = Z1.y - Z2.y;
          const float bx = Z1.y + Z2.y, by = Z2.x - Z1.x;
          const float h = 0.5f * r2;
          X1 = make_float2(h * fmaf(w.x, ax, w.y * ay), h * fmaf(w.x, bx, w.y * by));
          X2 = make_float2(h * fmaf(w.y, ax, -w.x * ay), h * fmaf(w.y, bx, -w.x * by));
        }
      }
      float2 Y1, Y2;   // orthonormal inverse input at k1, k2
      if (fwd_op) {
        if (valid) {
          st2(a.out + cb + (size_t)k1 * N + pix, X1);
          st2(a.out + cb + (size_t)k2 * N + pix, X2);
        }
        continue;
      } else if (inv_op) {
        Y1 = valid ? ld2(a.in + cb + (size_t)k1 * N + pix) : make_float2(0.f, 0.f);
        Y2 = valid ? ld2(a.in + cb + (size_t)k2 * N + pix) : make_float2(0.f, 0.f);
      } else {
        const float sa = (c == 2) ? sigma : sigma * gamma;
        float *v1p = a.v + c * CS + cb + (size_t)k1 * N + pix;
        float *v2p = a.v + c * CS + cb + (size_t)k2 * N + pix;
        const float2 o1 = pv1[r], o2 = pv2[r];
        float vt[4] = {fmaf(sa * al.x, X1.x, o1.x), fmaf(sa * al.y, X1.y, o1.y),
                       fmaf(sa * al.x, X2.x, o2.x), fmaf(sa * al.y, X2.y, o2.y)};
        float vn[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t bit = 1u << (r * 4 + e);
          if (c == 0) {
            vn[e] = satf(vt[e]);
            if (fabsf(vt[e]) <= 1.f) mask |= bit;
          } else {
            vn[e] = (mask & bit) ? vt[e] : 0.f;
          }
        }
        if (valid) {
          st2(v1p, make_float2(vn[0], vn[1]));
          st2(v2p, make_float2(vn[2], vn[3]));
        }
        Y1 = make_float2(vn[0], vn[1]);
        Y2 = make_float2(vn[2], vn[3]);
      }
      // merged inverse input W[k1], W[k2] (1/L folded into the scales)
      float2 W1, W2;
      if (kk == 0) {
        W1 = make_float2(Y1.x * q1, Y1.y * q1);
        W2 = make_float2(Y2.x * (rt2 * q2), Y2.y * (rt2 * q2));
      } else {
        const float pa = Y1.x * q2, pb = Y2.x * q2;   // pixel A: X''[k1], X''[k2]
        const float qa = Y1.y * q2, qb = Y2.y * q2;   // pixel B
        const float2 WA = make_float2(fmaf(w.x, pa, w.y * pb), fmaf(w.y, pa, -w.x * pb));
        const float2 WB = make_float2(fmaf(w.x, qa, w.y * qb), fmaf(w.y, qa, -w.x * qb));
        W1 = make_float2(WA.x - WB.y, WA.y + WB.x);
        W2 = make_float2(WA.x + WB.y, WB.x - WA.y);
      }
      d[s * PITCH + fpad(k1)] = W1;
      d[s * PITCH + fpad(k2)] = W2;
    }
  }
  if (fwd_op) return;
  __syncthreads();
#pragma unroll 1
  for (int c = 0; c < CH; ++c) fft_inplace<L, true>(dat + c * NB * PITCH, NB, PITCH, tw);

  // ---- back in band order: t (iteration) or C^T in (operator)
#pragma unroll 4
  for (int it = tid; it < L * NB; it += FT) {
    const int l = it / NB;
    if (!valid) continue;
    const int o = ps * PITCH + fpad(mpos<L>(l));
    const size_t j = cb + (size_t)l * N + pix;
    if (MODE == WAVE_TRANSFORM) {
      st2(a.out + j, dat[o]);
    } else {
      const float2 w0 = dat[o];
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        float2 val = c == 0 ? w0 : dat[c * NB * PITCH + o];
        if (c == 2)    // C^T (gamma v'_gamma + v)
          val = make_float2(fmaf(gamma, val.x, w0.x), fmaf(gamma, val.y, w0.y));
        const float s2 = (c == 2) ? 1.f : gamma;
        st2(a.t + c * CS + j, make_float2(s2 * al.x * val.x, s2 * al.y * val.y));
      }
    }
  }
}

template <int L, int CH, int MODE, int FT>
cudaError_t launch_f32_t(const F32Args &a, cudaStream_t st, Prof *prof) {
  using S = FShape<L, FT>;
  const size_t sm = (size_t)(a.tw_len + L + CH * S::NB * S::PITCH) * sizeof(float2);
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_dct_f32<L, CH, MODE, FT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         200 * 1024);
    attr = true;
  }
  const double vox = (double)a.npix * L * a.B;
  ProfScope ps(prof, MODE == WAVE_ITERATE ? "spectral_dual" : "spectral_op",
               MODE == WAVE_ITERATE ? CH * vox * 20.0 : vox * 8.0,
               (MODE == WAVE_ITERATE ? 2.0 : 1.0) * CH * vox * (2.5 * std::log2((double)L) + 6.0),
               st);
  const unsigned gx = (unsigned)((a.npix + S::PT - 1) / S::PT);
  launch_chain(k_dct_f32<L, CH, MODE, FT>, dim3(gx, a.B), FT, sm, st, a);
  return cudaGetLastError();
}

template <int L, int CH, int MODE>
cudaError_t launch_f32(const F32Args &a, cudaStream_t st, Prof *prof) {
  const size_t tiles = (a.npix + FShape<L, 256>::PT - 1) / FShape<L, 256>::PT * a.B;
  // 64-thread CTAs (quarter-size tiles) where the 256-thread ones are too few.  Up to
  // 128 bands below one an SM they fill the chip better (64 x 64 x 32, three chains:
  // 24.8 -> 18 us; from there on the wide tiles' longer rows win, 256 x 256 x 32: 43.7
  // against 35.1).  Short spectra have too little work a thread for it (8 bands, one
  // chain: 8.2 against 7.0 us; 64 x 64 x 16, three: 15.4 against 12.6), and long ones
  // tables that every CTA loads (32 x 32 x 1024, 128 wide tiles: 34.7 against 14.2
  // us; 64 x 64 x 256: 12.8 against 11.4), so the line lies lower there.
  constexpr size_t few = CH == 3 ? (L <= 16 ? 0 : L <= 128 ? 150 : 76)
                                 : (L < 16 || L == 1024 ? 0 : L <= 128 ? 150 : L == 256 ? 76 : 38);
  return tiles < few ? launch_f32_t<L, CH, MODE, 64>(a, st, prof)
                     : launch_f32_t<L, CH, MODE, 256>(a, st, prof);
}

template <int CH, int MODE>
cudaError_t dispatch_f32(const F32Args &a, cudaStream_t st, Prof *prof) {
  switch (a.L) {
    case 2: return launch_f32<2, CH, MODE>(a, st, prof);
    case 4: return launch_f32<4, CH, MODE>(a, st, prof);
    case 8: return launch_f32<8, CH, MODE>(a, st, prof);
    case 16: return launch_f32<16, CH, MODE>(a, st, prof);
    case 32: return launch_f32<32, CH, MODE>(a, st, prof);
    case 64: return launch_f32<64, CH, MODE>(a, st, prof);
    case 128: return launch_f32<128, CH, MODE>(a, st, prof);
    case 256: return launch_f32<256, CH, MODE>(a, st, prof);
    case 512: return launch_f32<512, CH, MODE>(a, st, prof);
    case 1024: return launch_f32<1024, CH, MODE>(a, st, prof);
    default: return cudaErrorInvalidValue;
  }
}

F32Args base_args(const DctArgs &d) {
  F32Args a{};
  a.L = d.L; a.B = d.B > 0 ? d.B : 1;
  a.npix = d.npix ? d.npix : (size_t)d.n * d.n;
  a.tab = d.ftab; a.tw_len = d.ftw_len;
  a.alpha = d.alpha; a.sc = d.sc;
  return a;
}

}  // namespace

int dct_f32_table_len(int L) { return fft_table_len(L) + L; }

void dct_f32_tables(int L, float2 *tab) {
  const int tl = fft_table_len(L);
  fft_tables(L, tab);
  const double pi = 3.14159265358979323846;
  for (int k = 0; k < L; ++k) {
    const double th = pi * k / (2.0 * L);
    tab[tl + k] = make_float2((float)std::cos(th), (float)std::sin(th));
  }
}

cudaError_t dct_dual_f32(const DctArgs &d, const Group &gr, cudaStream_t st) {
  F32Args a = base_args(d);
  a.xt = gr.xt; a.x = gr.x; a.v = gr.v; a.t = gr.t;
  if (gr.C == 3) return dispatch_f32<3, WAVE_ITERATE>(a, st, d.prof);
  return dispatch_f32<1, WAVE_ITERATE>(a, st, d.prof);
}

cudaError_t dct_op_f32(const DctArgs &d, const float *in, float *out, int inverse,
                       cudaStream_t st) {
  F32Args a = base_args(d);
  a.in = in; a.out = out; a.inverse = inverse;
  return dispatch_f32<1, WAVE_TRANSFORM>(a, st, d.prof);
}

}  // namespace muffin
