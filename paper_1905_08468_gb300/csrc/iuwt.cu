// Isotropic undecimated wavelet transform (starlet), the alternative spatial
// dictionary W_s of Sec. 2.1, fused with the MUFFIN updates that consume it
// (Algorithm 2 and the derivative forms of Algorithms 3/4), like the
// Daubechies kernels in wavelet.cu:
//
//   analysis + dual update:  c_0 = 2x~ - x (chain mix of Algorithm 3),
//     c_{j+1} = S_j c_j, plane j gets w = c_j - c_{j+1}, plane J gets c_J;
//     p = u + sigma mu_l plane, u = sat(p) (eqs. stpp, stpu);
//   synthesis + primal prox: W^T u in Horner form
//     P_0 + S_0[(P_1 - P_0) + S_1[(P_2 - P_1) + ... + S_{J-1}(P_J - P_{J-1})]]
//     then m = x - tau (grad + mu_l s + t), x~ = (m)_+ (eqs. stpm, stpx).
//
// S_j is the separable B3 spline [1 4 6 4 1]/16 dilated by D = 2^j with periodic
// boundaries.  One launch per scale and set of chains, specialised on D: a lane
// owns one column of a 32 x 128 tile (8 x 128 where there are few) and its 2 D halo
// rows in registers (loaded coalesced along the rows), smooths it along y there and
// puts the smoothed rows into shared memory; after one barrier it smooths along x (five conflict-free
// reads a pixel) and does the scale's dual update (analysis) or Horner step
// (synthesis) on its own column, whose unsmoothed values it still holds.  U is
// requested eight rows ahead.  The running image of the next scale goes to a
// ping-pong scratch.  J <= 4 (halo <= 16).
//
// What bounds it: DRAM and the latency of a CTA's loads.  A tile with halo of all
// chains in shared memory (two passes over it, 2 CTAs an SM) ran at 0.24-0.36 of
// the copy bandwidth.  512 x 512 x 32, three chains, before and now: analysis 318
// -> 122 us (first two scales, mean; 4.1 TB/s) and 195 -> 95, synthesis 328 and 201
// -> 104 and 83 (4.8 TB/s), prox 257 -> 247 (its four arrays a row; requested two
// rows ahead, and into L2 by the whole CTA first: 295 without).
//
// One chain a CTA: the primal's launch leaves its masks (Pi(p) per coefficient,
// U(m) per pixel: a word a lane, tile and plane) for the derivatives'.
#include <cuda_runtime.h>

#include <stdint.h>

#include "chain.cuh"
#include "kernels.h"

namespace muffin {

namespace {

constexpr int IX = 128, INT = 160;            // output tile's columns, threads (a column each)
constexpr int VP = INT;                       // floats of a smoothed row
constexpr int RB = 8;                         // rows whose U is in flight
static_assert(IX + 4 * 8 <= INT, "a column of the tile and its widest halo a thread");
static_assert(IX == 128, "iuwt_mask_words");

// B3 spline tap m of [1 4 6 4 1] / 16
__device__ __forceinline__ constexpr float b3(int m) {
  return (m == 2 ? 6.f : (m == 1 || m == 3) ? 4.f : 1.f) * (1.f / 16.f);
}

struct IuwtArgs {
  int n, L, Lc, P, J, j;         // P = J + 1 planes per band, j = this scale
  int positivity;
  const float *xt, *x, *g, *t;   // iteration images [C][L][n][n]
  float *xt_out;                 // synthesis j = 0: x-tilde
  const float *in;               // operator input (analysis: x; synthesis: u)
  float *out;                    // synthesis operator output
  float *u;                      // [C][L][P][n][n] duals (analysis writes)
  const float *ur;               // duals read by the synthesis
  float *buf[2];                 // ping-pong running images [C][L][n][n]
  const float *beta;
  const DevScalars *sc;
  uint32_t *masks;               // [L][tiles][min(n, IX)][2]
};

// y smoothing of the lane's column into shared memory, then (after the barrier)
// x smoothing of row r at the lane's own pixel
template <int D, int IY>
__device__ __forceinline__ void smooth_y(const float (&c)[IY + 4 * D], float *v) {
#pragma unroll
  for (int r = 0; r < IY; ++r) {
    float s = 0.f;
#pragma unroll
    for (int m = 0; m < 5; ++m) s = fmaf(b3(m), c[r + m * D], s);
    v[r * VP] = s;
  }
}
template <int D>
__device__ __forceinline__ float smooth_x(const float *v, int r) {
  float s = 0.f;
#pragma unroll
  for (int m = 0; m < 5; ++m) s = fmaf(b3(m), v[r * VP + (m - 2) * D], s);
  return s;
}

struct Place {
  unsigned xx, y0;               // the lane's column (wrapped) and the tile's first row
  int lane;                      // column of the tile (halo: < 0 or >= IX)
  bool own;                      // a pixel column of the image
};
template <int D, int IY>
__device__ __forceinline__ Place place(int n) {
  Place q;
  const int ntx = (n + IX - 1) / IX;
  const int x0 = (blockIdx.x % ntx) * IX;
  q.y0 = (blockIdx.x / ntx) * IY;
  q.lane = (int)threadIdx.x - 2 * D;
  q.xx = (unsigned)(x0 + q.lane) & (n - 1);
  q.own = q.lane >= 0 && q.lane < IX && x0 + q.lane < n;
  return q;
}

// the tile's rows of an image into L2: a 128-byte line a thread and round
template <int IY>
__device__ __forceinline__ void prefetch_tile(const float *img, unsigned n, unsigned y0) {
  const int ntx = (n + IX - 1) / IX;
  const unsigned x0 = (blockIdx.x % ntx) * IX;
  for (unsigned i = threadIdx.x; i < IY * (IX / 32); i += INT) {
    const unsigned x = x0 + 32 * (i % (IX / 32)), y = y0 + i / (IX / 32);
    if (x < n && y < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(img + (size_t)y * n + x));
  }
}

// chain c = 0 (DERIV = false; masks recorded where a.masks is set), or
// 1 + blockIdx.z
template <int MODE, int D, bool LAST, bool DERIV, int IY>
__global__ void __launch_bounds__(INT, 3) k_iuwt_ana(IuwtArgs a) {
  chain_enter();
  __shared__ float vs[IY * VP];
  const unsigned n = a.n, nm = n - 1;
  const int l = blockIdx.y, c = DERIV ? 1 + blockIdx.z : 0, tid = threadIdx.x;
  const Place w = place<D, IY>(n);
  const size_t NN = (size_t)n * n, CS = (size_t)a.L * NN;
  float mu = 0.f, q = 1.f;
  if (MODE == WAVE_ITERATE) {
    const DevScalars &S = a.sc[l / a.Lc];
    mu = (float)S.mu;
    q = (float)(S.sigma * (double)a.beta[l]);
    if (c != 1) q *= mu;
  }
  float col[IY + 4 * D];
  if (tid < IX + 4 * D) {
    const size_t i0 = c * CS + l * NN + w.xx;
    const float *src = D == 1 ? nullptr : a.buf[a.j & 1] + i0;
    const float *xt = a.xt + i0, *x = (MODE == WAVE_TRANSFORM && D == 1 ? a.in : a.x) + i0;
#pragma unroll
    for (int i = 0; i < IY + 4 * D; ++i) {
      const unsigned o = ((w.y0 + i - 2 * D) & nm) * n;
      if (D > 1) col[i] = src[o];
      else col[i] = MODE == WAVE_TRANSFORM ? x[o] : 2.f * xt[o] - x[o];
    }
    if (D == 1 && DERIV && c == 1) {                 // Algorithm 3 input: z0 + mu z1
      xt -= CS;
      x -= CS;
#pragma unroll
      for (int i = 0; i < IY + 4 * D; ++i) {
        const unsigned o = ((w.y0 + i - 2 * D) & nm) * n;
        col[i] = fmaf(mu, col[i], 2.f * xt[o] - x[o]);
      }
    }
    smooth_y<D, IY>(col, vs + tid);
  }
  constexpr int NP = LAST ? 2 : 1;
  float *uj = a.u + ((size_t)(c * a.L + l) * a.P + a.j) * NN + (size_t)w.y0 * n + w.xx;
  float u[2][NP][RB];
  auto request = [&](int r0, float (&d)[NP][RB]) {   // planes j (and J = j + 1) of 8 rows
    if (MODE == WAVE_ITERATE && w.own)
#pragma unroll
      for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int r = 0; r < RB; ++r)
          d[p][r] = w.y0 + r0 + r < n ? uj[p * NN + (size_t)(r0 + r) * n] : 0.f;
  };
  request(0, u[0]);
  uint32_t *mk = a.masks && w.own
                     ? a.masks + (((size_t)l * gridDim.x + blockIdx.x) * (n < IX ? n : IX) + w.lane) * 2
                     : nullptr;
  uint32_t keep[2] = {0u, 0u};
  if (DERIV && w.own) {
    keep[0] = mk[0];
    if (LAST) keep[1] = mk[1];
  }
  __syncthreads();
  if (!w.own) return;
  float *nxt = LAST ? nullptr : a.buf[(a.j + 1) & 1] + c * CS + l * NN + (size_t)w.y0 * n + w.xx;
#pragma unroll
  for (int r0 = 0; r0 < IY; r0 += RB) {
    const int cur = (r0 / RB) & 1;
    if (r0 + RB < IY) request(r0 + RB, u[cur ^ 1]);
#pragma unroll
    for (int k = 0; k < RB; ++k) {
      const int r = r0 + k;
      const float cn = smooth_x<D>(vs + tid, r);
      if (w.y0 + r >= n) continue;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        float val = p == 0 ? col[r + 2 * D] - cn : cn;
        if (MODE == WAVE_ITERATE) {
          const float t = fmaf(q, val, u[cur][p][k]);
          if (DERIV) {
            val = (keep[p] >> r) & 1u ? t : 0.f;
          } else {
            val = satf(t);
            if (fabsf(t) <= 1.0f) keep[p] |= 1u << r;
          }
        }
        uj[p * NN + (size_t)r * n] = val;
      }
      if (!LAST) nxt[(size_t)r * n] = cn;
    }
  }
  if (MODE == WAVE_ITERATE && !DERIV && mk) {
    mk[0] = keep[0];
    if (LAST) mk[1] = keep[1];
  }
}

// TOP: the coarsest step (source P_J - P_{J-1}); otherwise the running image of
// scale j + 1.  Scales j > 0 take chains blockIdx.z; j = 0 (D = 1) ends in the
// prox, chain 0 or chains 1 + blockIdx.z.
template <int MODE, int D, bool TOP, bool DERIV, int IY>
__global__ void __launch_bounds__(INT, 3) k_iuwt_syn(IuwtArgs a) {
  chain_enter();
  __shared__ float vs[IY * VP];
  const unsigned n = a.n, nm = n - 1;
  const int l = blockIdx.y, c = (DERIV ? 1 : 0) + blockIdx.z, tid = threadIdx.x;
  const Place w = place<D, IY>(n);
  const size_t NN = (size_t)n * n, CS = (size_t)a.L * NN, US = CS * a.P;
  // chain 1's W^T u + mu W^T u'_mu (Algorithm 3) by linearity, from mixed inputs
  const bool mix = D == 1 && DERIV && c == 1;
  const float mu = MODE == WAVE_ITERATE && D == 1 ? (float)a.sc[l / a.Lc].mu : 0.f;
  const float *ub = (MODE == WAVE_TRANSFORM ? a.in : a.ur) + c * US + (size_t)l * a.P * NN;
  if (D == 1 && MODE == WAVE_ITERATE) {
    const size_t o = c * CS + l * NN;
    prefetch_tile<IY>(ub, n, w.y0);
    prefetch_tile<IY>(a.x + o, n, w.y0);
    prefetch_tile<IY>(a.g + o, n, w.y0);
    prefetch_tile<IY>(a.t + o, n, w.y0);
  }
  float col[IY + 4 * D];
  if (tid < IX + 4 * D) {
    const float *s1 = TOP ? ub + (size_t)a.J * NN + w.xx
                          : a.buf[(a.j + 1) & 1] + c * CS + l * NN + w.xx;
    const float *s2 = ub + (size_t)(a.J - 1) * NN + w.xx;
#pragma unroll
    for (int i = 0; i < IY + 4 * D; ++i) {
      const unsigned o = ((w.y0 + i - 2 * D) & nm) * n;
      col[i] = TOP ? s1[o] - s2[o] : s1[o];
    }
    if (mix) {
      s1 -= TOP ? US : CS;
      s2 -= US;
#pragma unroll
      for (int i = 0; i < IY + 4 * D; ++i) {
        const unsigned o = ((w.y0 + i - 2 * D) & nm) * n;
        col[i] = fmaf(mu, col[i], TOP ? s1[o] - s2[o] : s1[o]);
      }
    }
    smooth_y<D, IY>(col, vs + tid);
  }
  __syncthreads();
  if (!w.own) return;
  const size_t i0 = (size_t)w.y0 * n + w.xx;
  if constexpr (D > 1) {
    const float *uj = ub + (size_t)a.j * NN + i0;
    float *dst = a.buf[a.j & 1] + c * CS + l * NN + i0;
    float d[2][RB];
    auto request = [&](int r0, float (&v)[RB]) {
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const size_t o = (size_t)(r0 + r) * n;
        v[r] = 0.f;
        if (w.y0 + r0 + r < n) v[r] = uj[o] - (uj - NN)[o];
      }
    };
    request(0, d[0]);
#pragma unroll
    for (int r0 = 0; r0 < IY; r0 += RB) {
      const int cur = (r0 / RB) & 1;
      if (r0 + RB < IY) request(r0 + RB, d[cur ^ 1]);
#pragma unroll
      for (int k = 0; k < RB; ++k) {
        const float s = smooth_x<D>(vs + tid, r0 + k);
        if (w.y0 + r0 + k < n) dst[(size_t)(r0 + k) * n] = s + d[cur][k];
      }
    }
  } else {
    uint32_t *mk = a.masks ? a.masks + (((size_t)l * gridDim.x + blockIdx.x) * (n < IX ? n : IX) + w.lane) * 2
                           : nullptr;
    uint32_t keep = DERIV ? mk[0] : 0u;
    const float tau = MODE == WAVE_ITERATE ? (float)a.sc[l / a.Lc].tau : 0.f;
    const float bl = MODE == WAVE_ITERATE ? a.beta[l] : 0.f;
    const float sc = c == 1 ? bl : bl * mu;          // mu_l, beta_l, mu_l
    const size_t i1 = c * CS + l * NN + i0;
    // four arrays a row: 2 x 2 rows in flight, or all of a low tile's
    constexpr int RQ = IY == 8 ? 8 : 2;
    float in[2][4][RQ];
    auto request = [&](int r0, float (&v)[4][RQ]) {
#pragma unroll
      for (int r = 0; r < RQ; ++r) {
        if (w.y0 + r0 + r >= n) continue;
        const size_t o = (size_t)(r0 + r) * n;
        v[0][r] = ub[i0 + o];
        if (mix) v[0][r] = fmaf(mu, v[0][r], (ub - US)[i0 + o]);
        if (MODE == WAVE_ITERATE) {
          v[1][r] = a.x[i1 + o];
          v[2][r] = a.g[i1 + o];
          v[3][r] = a.t[i1 + o];
        }
      }
    };
    request(0, in[0]);
#pragma unroll
    for (int r0 = 0; r0 < IY; r0 += RQ) {
      const int cur = (r0 / RQ) & 1;
      if (r0 + RQ < IY) request(r0 + RQ, in[cur ^ 1]);
#pragma unroll
      for (int k = 0; k < RQ; ++k) {
        const int r = r0 + k;
        const float s = smooth_x<D>(vs + tid, r);
        if (w.y0 + r >= n) continue;
        const float acc = in[cur][0][k] + s;
        const size_t o = i1 + (size_t)r * n;
        if (MODE == WAVE_TRANSFORM) {
          a.out[o] = acc;
          continue;
        }
        const float m = in[cur][1][k] - tau * (in[cur][2][k] + sc * acc + in[cur][3][k]);
        bool ok;
        if (DERIV) {
          ok = (keep >> r) & 1u;
        } else {
          ok = !a.positivity || m > 0.f;
          if (ok) keep |= 1u << r;
        }
        a.xt_out[o] = ok ? m : 0.f;
      }
    }
    if (MODE == WAVE_ITERATE && !DERIV && mk) mk[0] = keep;
  }
}

inline int itiles(int n, int rows) { return ((n + IX - 1) / IX) * ((n + rows - 1) / rows); }

// Tiles of 8 rows while those of 32 fill less than a wave (3 CTAs on 152 SMs, one
// chain).  A lane walks its rows one after the other, two at a time in the prox, and
// with few CTAs nothing covers that walk: below a wave four times the CTAs with a
// quarter of it, all rows in flight at once, are faster at every size, number of
// scales and number of chains (an iteration of a plain solve, one scale: 32 x 32 x 8 30.9
// -> 18.5 us, 64 x 64 x 32 34.5 -> 21.8, 256 x 256 x 24 51 -> 46; four scales, 128 x 128 x
// 100, 400 tiles: 137 -> 133; three chains 256 x 256 x 16, 489 -> 430).  The lead shrinks
// towards a wave, where the CTAs cover each other and the halo of a low tile (32 rows
// at the widest beside its 8) is what is left of the difference.
inline bool low_tiles(const IuwtArgs &a) { return (long long)itiles(a.n, 32) * a.L < 3 * 152; }

template <int CH, int MODE, int D, int IY>
void launch_ana_y(const IuwtArgs &a, cudaStream_t st) {
  const dim3 g(itiles(a.n, IY), a.L), g2(itiles(a.n, IY), a.L, 2);
  if (a.j == a.J - 1) {
    launch_chain(k_iuwt_ana<MODE, D, true, false, IY>, g, INT, 0, st, a);
    if constexpr (CH == 3) launch_chain(k_iuwt_ana<MODE, D, true, true, IY>, g2, INT, 0, st, a);
  } else {
    launch_chain(k_iuwt_ana<MODE, D, false, false, IY>, g, INT, 0, st, a);
    if constexpr (CH == 3) launch_chain(k_iuwt_ana<MODE, D, false, true, IY>, g2, INT, 0, st, a);
  }
}

template <int CH, int MODE, int D, int IY>
void launch_syn_y(const IuwtArgs &a, cudaStream_t st) {
  const bool top = a.j == a.J - 1;
  const int nt = itiles(a.n, IY);
  const dim3 g(nt, a.L, D > 1 ? CH : 1), g2(nt, a.L, 2);
  if (top) launch_chain(k_iuwt_syn<MODE, D, true, false, IY>, g, INT, 0, st, a);
  else launch_chain(k_iuwt_syn<MODE, D, false, false, IY>, g, INT, 0, st, a);
  if constexpr (CH == 3 && D == 1) {
    if (top) launch_chain(k_iuwt_syn<MODE, D, true, true, IY>, g2, INT, 0, st, a);
    else launch_chain(k_iuwt_syn<MODE, D, false, true, IY>, g2, INT, 0, st, a);
  }
}

template <int CH, int MODE, int D>
void launch_ana_d(const IuwtArgs &a, cudaStream_t st) {
  if (low_tiles(a)) launch_ana_y<CH, MODE, D, 8>(a, st);
  else launch_ana_y<CH, MODE, D, 32>(a, st);
}

template <int CH, int MODE, int D>
void launch_syn_d(const IuwtArgs &a, cudaStream_t st) {
  if (low_tiles(a)) launch_syn_y<CH, MODE, D, 8>(a, st);
  else launch_syn_y<CH, MODE, D, 32>(a, st);
}

template <int CH, int MODE>
cudaError_t ana_all(const WaveArgs &w, IuwtArgs a, cudaStream_t st) {
  const double vox = (double)CH * w.L * w.n * w.n;
  if (CH == 1) a.masks = nullptr;
  for (int j = 0; j < w.J; ++j) {
    a.j = j;
    const double bytes = vox * ((j == 0 && MODE == WAVE_ITERATE ? 8.0 : 4.0) +
                                (MODE == WAVE_ITERATE ? 8.0 : 4.0) * (j == w.J - 1 ? 2 : 1) +
                                (j == w.J - 1 ? 0.0 : 4.0));
    ProfScope ps(w.prof, "iuwt_ana_dual", bytes, vox * 22.0, st);
    switch (j) {
      case 0: launch_ana_d<CH, MODE, 1>(a, st); break;
      case 1: launch_ana_d<CH, MODE, 2>(a, st); break;
      case 2: launch_ana_d<CH, MODE, 4>(a, st); break;
      default: launch_ana_d<CH, MODE, 8>(a, st); break;
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int CH, int MODE>
cudaError_t syn_all(const WaveArgs &w, IuwtArgs a, cudaStream_t st) {
  const double vox = (double)CH * w.L * w.n * w.n;
  if (CH == 1) a.masks = nullptr;
  for (int j = w.J - 1; j >= 0; --j) {
    a.j = j;
    const double bytes = vox * ((j == w.J - 1 ? 8.0 : 4.0) + 8.0 * (j > 0) + 4.0 * (j == 0) +
                                (j > 0 ? 4.0 : (MODE == WAVE_ITERATE ? 16.0 : 4.0)));
    ProfScope ps(w.prof, j == 0 ? "iuwt_syn_prox" : "iuwt_syn", bytes, vox * 22.0, st);
    switch (j) {
      case 0: launch_syn_d<CH, MODE, 1>(a, st); break;
      case 1: launch_syn_d<CH, MODE, 2>(a, st); break;
      case 2: launch_syn_d<CH, MODE, 4>(a, st); break;
      default: launch_syn_d<CH, MODE, 8>(a, st); break;
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

IuwtArgs base_args(const WaveArgs &w, int C) {
  IuwtArgs a{};
  a.n = w.n; a.L = w.L; a.Lc = w.Lc > 0 ? w.Lc : w.L; a.P = w.J + 1; a.J = w.J;
  a.beta = w.beta; a.sc = w.sc; a.masks = w.masks;
  const size_t cl = (size_t)C * w.L * w.n * w.n;
  a.buf[0] = w.scratch;
  a.buf[1] = w.scratch + cl;
  return a;
}

}  // namespace

cudaError_t iuwt_analysis_dual(const WaveArgs &w, const Group &gr, cudaStream_t st) {
  IuwtArgs a = base_args(w, gr.C);
  a.xt = gr.xt; a.x = gr.x; a.u = gr.u;
  if (gr.C == 3) return ana_all<3, WAVE_ITERATE>(w, a, st);
  return ana_all<1, WAVE_ITERATE>(w, a, st);
}

cudaError_t iuwt_synthesis_prox(const WaveArgs &w, const Group &gr, int positivity,
                                cudaStream_t st) {
  IuwtArgs a = base_args(w, gr.C);
  a.x = gr.x; a.g = gr.g; a.t = gr.t; a.ur = gr.u; a.xt_out = gr.xt;
  a.positivity = positivity;
  if (gr.C == 3) return syn_all<3, WAVE_ITERATE>(w, a, st);
  return syn_all<1, WAVE_ITERATE>(w, a, st);
}

cudaError_t iuwt_analysis_op(const WaveArgs &w, const float *x, float *u, cudaStream_t st) {
  IuwtArgs a = base_args(w, 1);
  a.in = x; a.u = u;
  return ana_all<1, WAVE_TRANSFORM>(w, a, st);
}

cudaError_t iuwt_synthesis_op(const WaveArgs &w, const float *u, float *x, cudaStream_t st) {
  IuwtArgs a = base_args(w, 1);
  a.in = u; a.out = x;
  return syn_all<1, WAVE_TRANSFORM>(w, a, st);
}

}  // namespace muffin
