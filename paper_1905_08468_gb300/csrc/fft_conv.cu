// Least-squares gradient H_l^T (H_l x_l - y_l) of Algorithm 2 (eq. grad2)
// and H_l^T H_l x'_l of Algorithms 3/4, by 2D FFT (Eq. model read as a
// circular convolution).  Since H_l^T H_l = F^-1 diag(|h_hat_l|^2) F and
// b_l = H_l^T y_l is fixed per call, the hot path computes
//     g = F^-1 ( |h_hat|^2 . F x ) - b
// in three FP32 passes over the cube:
//   1. rows:    pairs of real rows packed as one complex row, FFT, split into
//               the two half spectra (n/2+1 bins), stored kx-major ("columns
//               contiguous") so that pass 2 reads whole columns;
//   2. columns: forward FFT of each column, multiply by |h_hat|^2 / n^2,
//               inverse FFT, in place;
//   3. rows:    rebuild the Hermitian row spectra of two rows at a time,
//               inverse FFT, subtract b, store.
// Images of 32 and 64 pixels a side go through the three in one kernel.
// The 2D transforms at the bottom, in FP64 or on pairs of FP32 values, are used
// only when a plan or call is set up (PSF spectra, H^T y, H^T delta).
#include <cuda_runtime.h>

#include "fft.cuh"
#include "fft32.cuh"
#include "chain.cuh"
#include "kernels.h"

namespace muffin {

namespace {

constexpr int kThreads = 256;

// sequences per CTA so that every thread owns fft_vpt(n) values per stage
__host__ __device__ constexpr int seqs_per_cta(int n) { return kThreads * fft_vpt(n) / n; }
// complex (row-pair) sequences per CTA of the row passes: 2 * nq real rows
__host__ __device__ constexpr int row_pairs(int n) { return seqs_per_cta(n) < n / 2 ? seqs_per_cta(n) : n / 2; }

// Shared-memory distance of the row passes' sequences: the split into (and the
// rebuild from) half spectra walks the pairs of a bin first, so the pairs of 16
// consecutive threads have to start in different banks (n + n / 16 is a multiple
// of 16 from 256 on, and 4-, 8- and 16-way conflicts bound the passes: 96 images
// of 256 x 256, forward 28.2 -> 17.3 us, inverse 26.9 -> 17.6; 192 images of 1024 x
// 1024, 391 -> 357 and 473 -> 454).
__host__ __device__ constexpr int row_pitch(int n) {
  return n + (n >> 4) + (row_pairs(n) >= 16 ? 1 : 16 / row_pairs(n));
}

// stage the twiddle tables (tlen entries) into shared memory
__device__ __forceinline__ void load_tw(float2 *dst, const float2 *__restrict__ src, int tlen) {
  for (int i = threadIdx.x; i < tlen; i += blockDim.x) dst[i] = src[i];
}

template <int NN, int RMAX>
__global__ void __launch_bounds__(kThreads)
k_rows_fwd(const float *__restrict__ x, float2 *__restrict__ S,
           const float2 *__restrict__ tw, int tlen, int img0) {
  // sizes are compile-time so that the index splits below are shifts
  constexpr int n = NN, nq = row_pairs(NN), nh = (NN >> 1) + 1;
  constexpr int pitch = row_pitch(NN);
  extern __shared__ float2 sm2[];
  const int img = blockIdx.y;           // image of the chunk (its spectrum in S)
  const int gimg = img0 + img;          // image of the cube
  const int y0 = blockIdx.x * 2 * nq;
  float2 *d = sm2, *tws = sm2 + nq * pitch;
  load_tw(tws, tw, tlen);
  chain_enter();
  // the first stage straight from the rows: element j + r q of pair s in the
  // stage's register order (coalesced: consecutive threads, consecutive j)
  constexpr int VPT = fft_vpt(NN), R = n < RMAX ? n : RMAX, q = n / R;
  constexpr int nthr = nq * n / VPT;
  float2 v[VPT];
  if (threadIdx.x < nthr) {
#pragma unroll
    for (int g = 0; g < VPT / R; ++g) {
      const int w = threadIdx.x + g * nthr;
      const float *xi = x + (size_t)gimg * n * n + (size_t)(y0 + 2 * (w / q)) * n + w % q;
#pragma unroll
      for (int r = 0; r < R; ++r) v[g * R + r] = make_float2(xi[r * q], xi[n + r * q]);
    }
  }
  fft_first<NN, R, VPT, false>(v, d, pitch, nthr);
  fft_stages<NN, R, false, RMAX>(d, pitch, nthr, tws);
  float4 *Si = reinterpret_cast<float4 *>(S + (size_t)img * nh * n);
  for (int i = threadIdx.x; i < nh * nq; i += blockDim.x) {
    const int k = i / nq, q = i - k * nq;
    const float2 Z = d[q * pitch + fpad(k)], Zc = d[q * pitch + fpad((n - k) & (n - 1))];
    // row 2q: (Z + conj Zc)/2 ; row 2q+1: (Z - conj Zc)/(2i)
    float4 o;
    o.x = 0.5f * (Z.x + Zc.x);
    o.y = 0.5f * (Z.y - Zc.y);
    o.z = 0.5f * (Z.y + Zc.y);
    o.w = 0.5f * (Zc.x - Z.x);
    Si[((size_t)k * n + y0 + 2 * q) >> 1] = o;
  }
}

template <int NN, int RMAX>
__global__ void __launch_bounds__(kThreads)
k_cols(float2 *__restrict__ S, const float *__restrict__ kspec, int L,
       const float2 *__restrict__ tw, int tlen, int img0) {
  constexpr int n = NN, nh = (NN >> 1) + 1, CB = seqs_per_cta(NN);
  constexpr int pitch = n + (n >> 4);
  extern __shared__ float2 sm2[];
  const int img = blockIdx.y, band = (img0 + img) % L;
  const int k0 = blockIdx.x * CB;
  const int ncol = min(CB, nh - k0);
  float2 *d = sm2, *tws = sm2 + CB * pitch;
  load_tw(tws, tw, tlen);
  chain_enter();
  // element u of the thread is i = tid + 256 u of the CTA's [CB][n] block:
  // column c0 + 256 u / n, row tid % n + (256 u) % n (see k_rows_fwd)
  const int tid = threadIdx.x;
  const int c0 = tid / n, sb = c0 * pitch + fpad(tid % n);
  float2 *Si = S + ((size_t)img * nh + k0) * n + tid;
  const float *Ki = kspec + ((size_t)band * nh + k0) * n + tid;
  // every thread owns at most KPT multiplier entries: prefetch them now
  constexpr int KPT = NN < 16 ? NN : 16;
  float kr[KPT];
#pragma unroll
  for (int u = 0; u < KPT; ++u)
    kr[u] = c0 + (kThreads * u) / n < ncol ? __ldg(Ki + kThreads * u) : 0.f;
  {
    float2 v[KPT];
#pragma unroll
    for (int u = 0; u < KPT; ++u)
      if (c0 + (kThreads * u) / n < ncol) v[u] = Si[kThreads * u];
#pragma unroll
    for (int u = 0; u < KPT; ++u)
      if (c0 + (kThreads * u) / n < ncol)
        d[sb + ((kThreads * u) / n) * pitch + fpad((kThreads * u) % n)] = v[u];
  }
  __syncthreads();
  fft_inplace<NN, false, RMAX>(d, ncol, pitch, tws);
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    if (c0 + (kThreads * u) / n < ncol) {
      float2 &z = d[sb + ((kThreads * u) / n) * pitch + fpad((kThreads * u) % n)];
      z.x *= kr[u];
      z.y *= kr[u];
    }
  }
  __syncthreads();
  fft_inplace<NN, true, RMAX>(d, ncol, pitch, tws);
#pragma unroll
  for (int u = 0; u < KPT; ++u)
    if (c0 + (kThreads * u) / n < ncol)
      Si[kThreads * u] = d[sb + ((kThreads * u) / n) * pitch + fpad((kThreads * u) % n)];
}

// The column pass from 128 rows on.  What bounds the Stockham form above is the
// shared-memory pipe (76 percent busy at 31 percent of the DRAM rate): an element
// crosses it 16 times and the CTA meets at 16 barriers.  Here (in-place plan of
// fft32.cuh) it crosses 8 times and meets at 4, columns come from and go to
// global memory in registers, and the multipliers, stored in the order of the
// positions, are read as the last stage holds them.  192 images of 1024 x 1024:
// 560 -> 413 us (4.9 TB/s); 32 images of 256 x 256: 16.3 -> 10.8 us.
template <int NN>
__global__ void __launch_bounds__(kThreads, 3)
k_cols_dif(float2 *__restrict__ S, const float *__restrict__ kspec, int L,
           const float2 *__restrict__ tw, int img0) {
  constexpr int n = NN, nh = (NN >> 1) + 1, CB = seqs_per_cta(NN), pitch = n + (n >> 4);
  constexpr int T = n / 16, M = n / 16, RL = cols_last_radix(n), GL = 16 / RL;
  constexpr bool three = n > 256;
  constexpr int tlen = cols_table_len(n);
  extern __shared__ float2 sm2[];
  float2 *tw1 = sm2 + CB * pitch, *tw2 = tw1 + 15 * T;
  load_tw(tw1, tw, tlen);
  chain_enter();
  const int img = blockIdx.y, band = (img0 + img) % L;
  const int k0 = blockIdx.x * CB, c = threadIdx.x / T, t = threadIdx.x % T;
  const bool act = c < CB && k0 + c < nh;
  float2 *d = sm2 + c * pitch;
  float2 *Si = S + ((size_t)img * nh + k0 + c) * n + t;
  float2 v[16];
  float kr[16];
  if (act) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = Si[r * T];
    const float *Ki = kspec + ((size_t)band * nh + k0 + c) * n;
#pragma unroll
    for (int g = 0; g < GL; ++g)
#pragma unroll
      for (int e = 0; e < RL; e += (RL < 4 ? 2 : 4)) {
        if constexpr (RL < 4) {
          const float2 k2 = __ldg(reinterpret_cast<const float2 *>(Ki + (t + g * T) * RL + e));
          kr[g * RL + e] = k2.x; kr[g * RL + e + 1] = k2.y;
        } else {
          const float4 k4 = __ldg(reinterpret_cast<const float4 *>(Ki + (t + g * T) * RL + e));
          kr[g * RL + e] = k4.x; kr[g * RL + e + 1] = k4.y;
          kr[g * RL + e + 2] = k4.z; kr[g * RL + e + 3] = k4.w;
        }
      }
  }
  __syncthreads();                       // the tables
  const int t2 = t % (three ? M / 16 : 1), k1 = t / (three ? M / 16 : 1);
  if (act) {
    dft16<false>(v);
    d[fpad(t)] = v[0];
#pragma unroll
    for (int r = 1; r < 16; ++r) d[fpad(r * M + t)] = cmul(v[out_slot<16>(r)], tw1[(r - 1) * T + t]);
  }
  __syncthreads();
  if constexpr (three) {
    if (act) {
      float2 *e = d + fpad(k1 * M);      // M is a multiple of 16
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = e[fpad(t2 + r * (M / 16))];
      dft16<false>(v);
      e[t2] = v[0];
#pragma unroll
      for (int r = 1; r < 16; ++r)
        e[fpad(r * (M / 16) + t2)] = cmul(v[out_slot<16>(r)], tw2[(r - 1) * (M / 16) + t2]);
    }
    __syncthreads();
  }
  if (act) {
#pragma unroll
    for (int g = 0; g < GL; ++g) {
      float2 w[RL], u[RL];
#pragma unroll
      for (int e = 0; e < RL; ++e) w[e] = d[fpad((t + g * T) * RL + e)];
      dftR<RL, false>(w);
#pragma unroll
      for (int e = 0; e < RL; ++e) {
        const float2 z = w[out_slot<RL>(e)];
        u[e] = make_float2(z.x * kr[g * RL + e], z.y * kr[g * RL + e]);
      }
      dftR<RL, true>(u);
#pragma unroll
      for (int e = 0; e < RL; ++e) d[fpad((t + g * T) * RL + e)] = u[out_slot<RL>(e)];
    }
  }
  __syncthreads();
  if constexpr (three) {
    if (act) {
      float2 *e = d + fpad(k1 * M);
      v[0] = e[t2];
#pragma unroll
      for (int r = 1; r < 16; ++r)
        v[r] = cmulc(e[fpad(r * (M / 16) + t2)], tw2[(r - 1) * (M / 16) + t2]);
      dft16<true>(v);
#pragma unroll
      for (int r = 0; r < 16; ++r) e[fpad(t2 + r * (M / 16))] = v[out_slot<16>(r)];
    }
    __syncthreads();
  }
  if (act) {
    v[0] = d[fpad(t)];
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = cmulc(d[fpad(r * M + t)], tw1[(r - 1) * T + t]);
    dft16<true>(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) Si[r * T] = v[out_slot<16>(r)];
  }
}

template <int NN, int RMAX>
__global__ void __launch_bounds__(kThreads)
k_rows_inv(const float2 *__restrict__ S, float *__restrict__ g_out,
           const float *__restrict__ bdata, int L,
           const float2 *__restrict__ tw, int tlen, int img0) {
  constexpr int n = NN, nq = row_pairs(NN), nh = (NN >> 1) + 1, half = NN >> 1;
  constexpr int pitch = row_pitch(NN);
  extern __shared__ float2 sm2[];
  const int img = blockIdx.y, gimg = img0 + img, band = gimg % L;
  const int y0 = blockIdx.x * 2 * nq;
  float2 *d = sm2, *tws = sm2 + nq * pitch;
  load_tw(tws, tw, tlen);
  chain_enter();
  const float4 *Si = reinterpret_cast<const float4 *>(S + (size_t)img * nh * n);
  for (int i = threadIdx.x; i < nh * nq; i += blockDim.x) {
    const int k = i / nq, q = i - k * nq;
    float4 v = Si[((size_t)k * n + y0 + 2 * q) >> 1];   // Xa = (x,y), Xb = (z,w)
    if (k == 0 || k == half) { v.y = 0.f; v.w = 0.f; }
    d[q * pitch + fpad(k)] = make_float2(v.x - v.w, v.y + v.z);    // Xa + i Xb
    if (k > 0 && k < half)
      d[q * pitch + fpad(n - k)] = make_float2(v.x + v.w, v.z - v.y);  // conj Xa + i conj Xb
  }
  __syncthreads();
  const bool sub = (bdata != nullptr) && (gimg < L);
  constexpr int VPT = fft_vpt(NN), NS = fft_last_ns(n, RMAX), R = n / NS;
  constexpr int nthr = nq * n / VPT;
  if constexpr (NS >= 32) {
    // the last stage's registers go straight to the rows (element j + r NS of pair
    // s: whole lines a warp)
    const float2 *twl = fft_middle<NN, 1, true, RMAX>(d, pitch, nthr, tws);
    float2 v[VPT];
    fft_last<NN, NS, R, VPT, true>(v, d, pitch, nthr, twl);
    if (threadIdx.x >= nthr) return;
#pragma unroll
    for (int g = 0; g < VPT / R; ++g) {
      const int w = threadIdx.x + g * nthr;
      const size_t o0 = (size_t)(y0 + 2 * (w / NS)) * n + w % NS;
      float *gi = g_out + (size_t)gimg * n * n + o0;
      const float *bi = sub ? bdata + (size_t)band * n * n + o0 : nullptr;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 z = v[g * R + out_slot<R>(r)];
        float v0 = z.x, v1 = z.y;
        if (sub) {
          v0 -= __ldg(bi + r * NS);
          v1 -= __ldg(bi + n + r * NS);
        }
        gi[r * NS] = v0;
        gi[n + r * NS] = v1;
      }
    }
  } else {
    fft_inplace<NN, true, RMAX>(d, nq, pitch, tws);
    // element u of the thread: row pair tid / n + 256 u / n, column tid % n + ...
    const int tid = threadIdx.x;
    const size_t o0 = (size_t)(y0 + 2 * (tid / n)) * n + tid % n;
    float *gi = g_out + (size_t)gimg * n * n + o0;
    const float *bi = sub ? bdata + (size_t)band * n * n + o0 : nullptr;
    const int sb = (tid / n) * pitch + fpad(tid % n);
#pragma unroll
    for (int u = 0; u < VPT; ++u) {
      if (tid + u * kThreads >= nq * n) continue;
      const int q = (kThreads * u) / n, c = (kThreads * u) % n;
      const float2 z = d[sb + q * pitch + fpad(c)];
      float v0 = z.x, v1 = z.y;
      if (sub) {
        v0 -= __ldg(bi + 2 * q * n + c);
        v1 -= __ldg(bi + (2 * q + 1) * n + c);
      }
      gi[2 * q * n + c] = v0;
      gi[(2 * q + 1) * n + c] = v1;
    }
  }
}

// ---------------------------------------------------------------- small images
// The whole gradient of an image of 32 or 64 pixels a side in one CTA: the half
// spectra stay in shared memory between the passes, so an image is read and
// written once and three launches become one.  A sequence belongs to N / 16 lanes
// of a warp (16 values each, the in-place plan of fft32.cuh in two stages), so the
// CTA meets only between the passes.  What bounds it: latency, at one image a CTA.
// An iteration of a plain solve with one basis and one level, 1, 8 and 32 images:
// 64 pixels 19.4 -> 17.6, 21.2 -> 19.7 and 22.7 -> 20.6 us; 32 pixels 19.4 -> 17.3,
// 20.6 -> 19.5 and 23.6 -> 20.6; 768 images (three chains) 198 -> 190 and 97 -> 87.
// At 128 pixels (141 KB, one CTA an SM) the three passes are faster: 22.6 against
// 26.8 us with one image, 26.2 against 31.3 with 32, 529 against 549 with 768.
template <int N>
struct SmallGrad {
  static constexpr int T = N / 16, RL = N / 16, GL = 16 / RL, nh = N / 2 + 1;
  static constexpr int PITCH = N + N / 16 + 1;     // odd: 16 sequences, 16 bank pairs
  static constexpr int NT = (nh * T + 31) / 32 * 32;
  static constexpr size_t SMEM =
      ((size_t)(N / 2 + nh) * PITCH + 15 * T) * sizeof(float2);
};

template <int N>
__global__ void __launch_bounds__(SmallGrad<N>::NT)
k_grad_small(const float *__restrict__ x, float *__restrict__ g_out, const float *__restrict__ bdata,
             const float *__restrict__ kspec, int L, const float2 *__restrict__ twc) {
  using G = SmallGrad<N>;
  constexpr int T = G::T, nh = G::nh, half = N / 2;
  extern __shared__ float2 sm2[];
  float2 *rows = sm2, *cols = rows + half * G::PITCH, *tw = cols + nh * G::PITCH;
  const int tid = threadIdx.x, s = tid / T, t = tid % T;
  load_tw(tw, twc, 15 * T);
  chain_enter();
  const int img = blockIdx.x, band = img % L;
  const size_t base = (size_t)img * N * N;
  float2 v[16];
  const bool row = s < half, col = s < nh;
  float2 *dr = rows + (row ? s : 0) * G::PITCH, *dc = cols + (col ? s : 0) * G::PITCH;
  const float *xr = x + base + (size_t)(2 * s) * N + t;
  if (row)
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = make_float2(xr[r * T], xr[N + r * T]);
  float kr[16];                                      // the column's multipliers
  if (col) {
    const float *K = kspec + ((size_t)band * nh + s) * N;
#pragma unroll
    for (int g = 0; g < G::GL; ++g)
#pragma unroll
      for (int e = 0; e < G::RL; ++e) kr[g * G::RL + e] = __ldg(K + (t + g * T) * G::RL + e);
  }
  __syncthreads();                                   // the table
  // every lane meets the warp barriers, with a sequence or without
  if (row) {
    dft16<false>(v);
    dr[fpad(t)] = v[0];
#pragma unroll
    for (int r = 1; r < 16; ++r) dr[fpad(r * T + t)] = cmul(v[out_slot<16>(r)], tw[(r - 1) * T + t]);
  }
  __syncwarp();
  if (row) {
#pragma unroll
    for (int g = 0; g < G::GL; ++g) {
      float2 u[G::RL];
#pragma unroll
      for (int e = 0; e < G::RL; ++e) u[e] = dr[fpad((t + g * T) * G::RL + e)];
      dftR<G::RL, false>(u);
#pragma unroll
      for (int e = 0; e < G::RL; ++e) dr[fpad((t + g * T) * G::RL + e)] = u[out_slot<G::RL>(e)];
    }
  }
  __syncthreads();
  // half spectra of the two rows of a pair (see k_rows_fwd)
  for (int i = tid; i < nh * half; i += G::NT) {
    const int k = i / half, q = i % half;
    const float2 *d = rows + q * G::PITCH;
    const float2 Z = d[fpad(cols_pos(k, N))], Zc = d[fpad(cols_pos((N - k) & (N - 1), N))];
    float2 *o = cols + k * G::PITCH;
    o[fpad(2 * q)] = make_float2(0.5f * (Z.x + Zc.x), 0.5f * (Z.y - Zc.y));
    o[fpad(2 * q + 1)] = make_float2(0.5f * (Z.y + Zc.y), 0.5f * (Zc.x - Z.x));
  }
  __syncthreads();
  // columns: forward, multiply, inverse, in place
  {
    if (col)
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = dc[fpad(t + r * T)];
    __syncwarp();
    if (col) {
      dft16<false>(v);
      dc[fpad(t)] = v[0];
#pragma unroll
      for (int r = 1; r < 16; ++r) dc[fpad(r * T + t)] = cmul(v[out_slot<16>(r)], tw[(r - 1) * T + t]);
    }
    __syncwarp();
    if (col) {
#pragma unroll
      for (int g = 0; g < G::GL; ++g) {
        float2 u[G::RL], z[G::RL];
#pragma unroll
        for (int e = 0; e < G::RL; ++e) u[e] = dc[fpad((t + g * T) * G::RL + e)];
        dftR<G::RL, false>(u);
#pragma unroll
        for (int e = 0; e < G::RL; ++e) {
          const float2 y = u[out_slot<G::RL>(e)];
          z[e] = make_float2(y.x * kr[g * G::RL + e], y.y * kr[g * G::RL + e]);
        }
        dftR<G::RL, true>(z);
#pragma unroll
        for (int e = 0; e < G::RL; ++e) dc[fpad((t + g * T) * G::RL + e)] = z[out_slot<G::RL>(e)];
      }
    }
    __syncwarp();
    if (col) {
      v[0] = dc[fpad(t)];
#pragma unroll
      for (int r = 1; r < 16; ++r) v[r] = cmulc(dc[fpad(r * T + t)], tw[(r - 1) * T + t]);
      dft16<true>(v);
    }
    __syncwarp();
    if (col)
#pragma unroll
      for (int r = 0; r < 16; ++r) dc[fpad(t + r * T)] = v[out_slot<16>(r)];
  }
  __syncthreads();
  // Hermitian row spectra of the pairs (see k_rows_inv)
  for (int i = tid; i < nh * half; i += G::NT) {
    const int k = i / half, q = i % half;
    float2 A = cols[k * G::PITCH + fpad(2 * q)], B = cols[k * G::PITCH + fpad(2 * q + 1)];
    if (k == 0 || k == half) { A.y = 0.f; B.y = 0.f; }
    float2 *d = rows + q * G::PITCH;
    d[fpad(cols_pos(k, N))] = make_float2(A.x - B.y, A.y + B.x);                       // A + i B
    if (k > 0 && k < half)
      d[fpad(cols_pos(N - k, N))] = make_float2(A.x + B.y, B.x - A.y);   // conj A + i conj B
  }
  __syncthreads();
  if (row) {
#pragma unroll
    for (int g = 0; g < G::GL; ++g) {
      float2 u[G::RL];
#pragma unroll
      for (int e = 0; e < G::RL; ++e) u[e] = dr[fpad((t + g * T) * G::RL + e)];
      dftR<G::RL, true>(u);
#pragma unroll
      for (int e = 0; e < G::RL; ++e) dr[fpad((t + g * T) * G::RL + e)] = u[out_slot<G::RL>(e)];
    }
  }
  __syncwarp();
  if (!row) return;
  v[0] = dr[fpad(t)];
#pragma unroll
  for (int r = 1; r < 16; ++r) v[r] = cmulc(dr[fpad(r * T + t)], tw[(r - 1) * T + t]);
  dft16<true>(v);
  float *gr = g_out + base + (size_t)(2 * s) * N + t;
  const float *br = bdata && img < L ? bdata + base + (size_t)(2 * s) * N + t : nullptr;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    float2 z = v[out_slot<16>(r)];
    if (br) {
      z.x -= __ldg(br + r * T);
      z.y -= __ldg(br + N + r * T);
    }
    gr[r * T] = z.x;
    gr[N + r * T] = z.y;
  }
}

// ---------------------------------------------------------------- FP64 set-up
// C: double2, or cdd (pairs of FP32 values, see fft.cuh)
template <typename C>
__global__ void k_fft_rows(C *data, int n, bool inverse, const C *__restrict__ tw) {
  extern __shared__ double2 sm4[];
  C *a = reinterpret_cast<C *>(sm4), *b = a + n;
  C *row = data + ((size_t)blockIdx.y * n + blockIdx.x) * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = row[i];
  __syncthreads();
  const C *r = inverse ? fft_batch<C, true>(a, b, n, 1, tw)
                       : fft_batch<C, false>(a, b, n, 1, tw);
  for (int i = threadIdx.x; i < n; i += blockDim.x) row[i] = r[i];
}

__global__ void k_transpose64(const double2 *__restrict__ in,
                              double2 *__restrict__ out, int n) {
  __shared__ double2 tile[32][33];
  const size_t base = (size_t)blockIdx.z * n * n;
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int y = by + j, x = bx + threadIdx.x;
    if (y < n && x < n) tile[j][threadIdx.x] = in[base + (size_t)y * n + x];
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int y = bx + j, x = by + threadIdx.x;
    if (y < n && x < n) out[base + (size_t)y * n + x] = tile[threadIdx.x][j];
  }
}

// ---- real images, two bands of a cube in one complex image
//
// The FP64 pipe bounds these transforms (2 operations a clock and SM against
// 128 in FP32), so bands 2j and 2j + 1 of a cube are the real and imaginary
// parts of one image (an odd last band rides alone): half the butterflies and
// half the traffic of one complex image a band.  Where the result is rounded to
// FP32 (H^T y, H^T delta), the transforms run on pairs of FP32 values (48 bits,
// fft.cuh) instead: 1024 x 1024 x 64, a pass over the rows 2.0 -> 0.58 ms; the
// spectra themselves (beta, |h_hat|^2) and the objective's residual stay in FP64.
// The rounding to FP32 is then the error: against extended precision, dirty and
// white cubes and bands 10^6 apart, 16 to 1024 pixels a side, the relative error is that
// of FP64 transforms in all ten digits (1024 x 1024: 2.505987765e-8 and
// 2.535576586e-8), the largest one too, and at most 5 of 2 M pixels, all near zero,
// round the other way (0.557 units in the last place instead of 0.5).
//
// An image is scaled by a power of two (exact) to a largest magnitude in
// [1, 2), and a band's spectrum h by one to [1, 2) or [2, 4), so that a faint
// band keeps its own precision beside a bright one; a band with NaN/Inf enters
// as zero and comes out as NaN (a PSF with Inf and no NaN as an infinite spectrum,
// which no step size admits), and leaves its neighbour alone.  Spectra stay
// transposed ([kx][ky]): one transpose each way.

// 2^-e of an image from its statistics: 1 for a zero image, NaN if any value is
// not finite
__device__ __forceinline__ double image_scale(const ImageStat &t) {
  const float m = __uint_as_float(t.max_bits);
  return t.nonfinite ? nan("") : (m > 0.f ? ldexp(1.0, -ilogbf(m)) : 1.0);
}

// the inverse of a scale, a power of two between 2^-127 and 2^149 (or NaN): from its
// exponent, as a division a thread weighs on the FP64 pipe
__device__ __forceinline__ double inverse_scale(double s) {
  return s == s ? __hiloint2double((2046 - (__double2hiint(s) >> 20)) << 20, 0) : s;
}

struct Pairs {
  int n, L, per_cube;           // side, bands per cube, pairs per cube
  const ImageStat *stat;        // [images]
  const double *hmax;           // [images] largest |h|^2 (not finite: h is not)
  __device__ double scale(int img) const { return image_scale(stat[img]); }
  __device__ double hscale(int img) const { return spectrum_scale(hmax[img]); }
  // Inf entries and no NaN: the spectrum is infinite (beside a NaN it is NaN)
  __device__ bool infinite(int img) const {
    return stat[img].infinite && stat[img].infinite == stat[img].nonfinite;
  }
  __device__ int first(int p) const { return p / per_cube * L + 2 * (p % per_cube); }
  __device__ bool second(int p) const { return 2 * (p % per_cube) + 1 < L; }
};

__device__ __forceinline__ void set_parts(double2 &z, double x, double y) { z = make_double2(x, y); }
__device__ __forceinline__ void set_parts(cdd &z, double x, double y) {
  z.x.h = (float)x; z.x.l = (float)(x - (double)z.x.h);
  z.y.h = (float)y; z.y.l = (float)(y - (double)z.y.h);
}
// FP32 values times a power of two (FP32: in two factors, for its whole range)
__device__ __forceinline__ float times_pow2(float x, double s) {
  const int e = ilogb(s);
  return x * ldexpf(1.f, e / 2) * ldexpf(1.f, e - e / 2);
}
__device__ __forceinline__ void set_input(double2 &z, float x, double sx, float y, double sy) {
  z = make_double2(sx * (double)x, sy * (double)y);
}
__device__ __forceinline__ void set_input(cdd &z, float x, double sx, float y, double sy) {
  z = cdd{{sx != 0.0 ? times_pow2(x, sx) : 0.f, 0.f}, {sy != 0.0 ? times_pow2(y, sy) : 0.f, 0.f}};
}
__device__ __forceinline__ float to_float(double v, double c) { return (float)(c * v); }
__device__ __forceinline__ float to_float(dd v, double c) {   // c a power of two or NaN
  return c == c ? times_pow2(v.h, c) : __int_as_float(0x7fc00000);
}

// forward transform along x of the packed rows: grid (n, pairs)
template <typename C>
__global__ void k_rows_real(const float *__restrict__ x, C *__restrict__ out, Pairs P,
                            const C *__restrict__ tw) {
  extern __shared__ double2 sm4[];
  const int n = P.n, p = blockIdx.y, ia = P.first(p);
  const bool two = P.second(p);
  C *a = reinterpret_cast<C *>(sm4), *b = a + n;
  const float *xa = x + ((size_t)ia * n + blockIdx.x) * n, *xb = xa + (size_t)n * n;
  const double sa = P.scale(ia), sb = two ? P.scale(ia + 1) : 0.0;
  const bool oka = sa == sa, okb = two && sb == sb;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    set_input(a[i], oka ? xa[i] : 0.f, oka ? sa : 0.0, okb ? xb[i] : 0.f, okb ? sb : 0.0);
  __syncthreads();
  const C *r = fft_batch<C, false>(a, b, n, 1, tw);
  C *row = out + ((size_t)p * n + blockIdx.x) * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) row[i] = r[i];
}

// inverse transform along x of the packed rows and the two real images
// out = (float)(c / scales * part): grid (n, pairs)
template <typename C>
__global__ void k_rows_out(const C *__restrict__ w, float *__restrict__ out, Pairs P,
                           double c, const C *__restrict__ tw) {
  extern __shared__ double2 sm4[];
  const int n = P.n, p = blockIdx.y, ia = P.first(p);
  C *a = reinterpret_cast<C *>(sm4), *b = a + n;
  const C *row = w + ((size_t)p * n + blockIdx.x) * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) a[i] = row[i];
  __syncthreads();
  const C *r = fft_batch<C, true>(a, b, n, 1, tw);
  float *oa = out + ((size_t)ia * n + blockIdx.x) * n, *ob = oa + (size_t)n * n;
  const bool two = P.second(p);
  const double ca = c / (P.scale(ia) * P.hscale(ia));
  const double cb = two ? c / (P.scale(ia + 1) * P.hscale(ia + 1)) : 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    oa[i] = to_float(r[i].x, ca);
    if (two) ob[i] = to_float(r[i].y, cb);
  }
}

__device__ __forceinline__ double half_of(double v) { return 0.5 * v; }
__device__ __forceinline__ dd half_of(dd v) { return dd{0.5f * v.h, 0.5f * v.l}; }

// the spectra A, B of the packed images at k, from Z[k] and Z[-k]
template <typename C>
__device__ __forceinline__ void pair_split(const C &z, const C &m, C &A, C &B) {
  A.x = half_of(z.x + m.x); A.y = half_of(z.y - m.y);
  B.x = half_of(z.y + m.y); B.y = half_of(m.x - z.x);
}

// spectra of every band from the packed ones: grid (n, pairs), row kx
__global__ void k_pair_unpack(const double2 *__restrict__ z, double2 *__restrict__ hh, Pairs P) {
  const int n = P.n, p = blockIdx.y, ia = P.first(p), kx = blockIdx.x;
  const size_t N = (size_t)n * n, row = (size_t)kx * n;
  const double2 *zr = z + p * N + row, *zm = z + p * N + (size_t)((n - kx) & (n - 1)) * n;
  const bool two = P.second(p);
  const double ra = inverse_scale(P.scale(ia)), rb = two ? inverse_scale(P.scale(ia + 1)) : 0.0;
  const bool infa = P.infinite(ia), infb = two && P.infinite(ia + 1);
  const double2 inf = make_double2(HUGE_VAL, 0.0);
  double2 *ha = hh + ia * N + row, *hb = ha + N;
  if (!two) {                                      // an odd last band: nothing to split
    for (int ky = threadIdx.x; ky < n; ky += blockDim.x)
      ha[ky] = infa ? inf : make_double2(ra * zr[ky].x, ra * zr[ky].y);
    return;
  }
  for (int ky = threadIdx.x; ky < n; ky += blockDim.x) {
    double2 A, B;
    pair_split(zr[ky], zm[(n - ky) & (n - 1)], A, B);
    ha[ky] = infa ? inf : make_double2(ra * A.x, ra * A.y);
    hb[ky] = infb ? inf : make_double2(rb * B.x, rb * B.y);
  }
}

// packed spectra times every band's own scaled h (CJ: its conjugate), in place:
// grid (n / 2 + 1, pairs), rows kx and -kx; a thread takes k and -k (the images
// are real, so -k holds the conjugates)
template <typename C, bool CJ>
__global__ void k_pair_mul(C *__restrict__ z, const double2 *__restrict__ hh, Pairs P) {
  const int n = P.n, p = blockIdx.y, ia = P.first(p), kx = blockIdx.x, mx = (n - kx) & (n - 1);
  const size_t N = (size_t)n * n, row = (size_t)kx * n;
  C *zr = z + p * N + row, *zm = z + p * N + (size_t)mx * n;
  const double2 *ha = hh + ia * N + row, *hb = ha + N;
  const bool two = P.second(p);
  const double sa = P.hscale(ia), sb = two ? P.hscale(ia + 1) : 0.0;
  const bool oka = sa == sa, okb = two && sb == sb;
  for (int ky = threadIdx.x; ky < n; ky += blockDim.x) {
    const int my = (n - ky) & (n - 1);
    if (mx == kx && my < ky) continue;
    C A, B, h;
    pair_split(zr[ky], zm[my], A, B);
    set_parts(h, oka ? sa * ha[ky].x : 0.0, oka ? sa * ha[ky].y : 0.0);
    A = CJ ? cmulc(A, h) : cmul(A, h);
    set_parts(h, okb ? sb * hb[ky].x : 0.0, okb ? sb * hb[ky].y : 0.0);
    B = CJ ? cmulc(B, h) : cmul(B, h);
    C w, v;
    w.x = A.x + B.y; w.y = B.x - A.y;              // conj A + i conj B
    v.x = A.x - B.y; v.y = A.y + B.x;              // A + i B (k == -k: the same real parts)
    zm[my] = w;
    zr[ky] = v;
  }
}

__global__ void k_c64_real_to_f32(const double2 *__restrict__ in,
                                  float *__restrict__ out, double scale,
                                  size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = (float)(in[i].x * scale);
}

// grid (n / 2 + 1, L); rows in the order of the column pass's positions;
// max_bits[l]: the largest |hh|^2 of the band (bits of a
// double >= 0, which order as integers, and above them NaN; the other half of a
// spectrum holds the conjugates)
__global__ void k_make_kspec(const double2 *__restrict__ hh, float *__restrict__ kspec,
                             double scale, int n, unsigned long long *max_bits) {
  const int l = blockIdx.y, kx = blockIdx.x;
  const double2 *h = hh + ((size_t)l * n + kx) * n;
  float *k = kspec + ((size_t)l * ((n >> 1) + 1) + kx) * n;
  unsigned long long m = 0;
  for (int ky = threadIdx.x; ky < n; ky += blockDim.x) {
    const double v = h[ky].x * h[ky].x + h[ky].y * h[ky].y;
    m = max(m, (unsigned long long)__double_as_longlong(fabs(v)));
    k[n < 32 ? ky : cols_pos(ky, n)] = (float)(v * scale);
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, m, o);
    m = m > t ? m : t;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(max_bits + l, m);
}

template <typename F>
void allow_smem(F *k) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

inline int grid_for(size_t count) {
  size_t g = (count + 255) / 256;
  return (int)(g > 152 * 32 ? 152 * 32 : (g ? g : 1));
}


template <int NN, int RMAX>
cudaError_t gradient_n(const float *x, float *g, const float *b, float2 *S,
                       const float *kspec, const float2 *tw, const float2 *twc, int L, int C,
                       cudaStream_t st, Prof *prof, int chunk) {
  constexpr int n = NN;
  const int ntot = C * L;
  const int nh = (n >> 1) + 1;
  const double img = (double)n * n, spec = (double)nh * n * 8.0;
  const double fft = 5.0 * n * ilog2(n);   // flops of one length-n complex FFT
  // the whole call: x read, g written, b read, |h_hat|^2 read once per
  // band, and in three passes the spectra of every image written and read twice
  ProfScope all(prof, "grad_total",
                ntot * (img * 8.0 + (n < 32 || n > 64 ? 4.0 * spec : 0.0)) + (b ? (double)L * img * 4.0 : 0.0) +
                    (double)L * nh * n * 4.0,
                ntot * (double)(n + 2 * nh) * fft, st);
  if constexpr (NN == 32 || NN == 64) {
    using G = SmallGrad<NN>;
    static_assert(G::SMEM <= 48 * 1024, "no opt-in needed");
    launch_chain(k_grad_small<NN>, dim3(ntot), G::NT, G::SMEM, st, x, g, b, kspec, L, twc);
  } else {
    const int RB = 2 * row_pairs(n);                  // real rows per CTA (even)
    const int CB = seqs_per_cta(n);                   // columns per CTA
    const int pitch = n + (n >> 4);
    const int tlen = fft_table_len(n, RMAX);
    const size_t smr = ((size_t)(RB / 2) * row_pitch(n) + tlen) * sizeof(float2);
    const size_t smc = ((size_t)CB * pitch + (n >= 128 ? cols_table_len(n) : tlen)) * sizeof(float2);
    static bool attr = false;
    if (!attr) {
      cudaFuncSetAttribute(k_rows_fwd<NN, RMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      cudaFuncSetAttribute(k_rows_inv<NN, RMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      if constexpr (NN >= 128)
        cudaFuncSetAttribute(k_cols_dif<NN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      else
        cudaFuncSetAttribute(k_cols<NN, RMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
      attr = true;
    }
    const int step = chunk > 0 && chunk < ntot ? chunk : ntot;
    for (int i0 = 0; i0 < ntot; i0 += step) {
      const int nimg = step < ntot - i0 ? step : ntot - i0;
      const int nb = b ? (i0 < L ? (L - i0 < nimg ? L - i0 : nimg) : 0) : 0;   // images with b
      {
        ProfScope ps(prof, "grad_rows_fwd", nimg * (img * 4.0 + spec),
                     nimg * (n / 2.0) * fft, st);
        launch_chain(k_rows_fwd<NN, RMAX>, dim3(n / RB, nimg), kThreads, smr, st, x, S, tw, tlen, i0);
      }
      {
        ProfScope ps(prof, "grad_cols", nimg * 2.0 * spec + (double)nimg * nh * n * 4.0,
                     nimg * (double)nh * 2.0 * fft, st);
        const dim3 grid((nh + CB - 1) / CB, nimg);
        if constexpr (NN >= 128) launch_chain(k_cols_dif<NN>, grid, kThreads, smc, st, S, kspec, L, twc, i0);
        else launch_chain(k_cols<NN, RMAX>, grid, kThreads, smc, st, S, kspec, L, tw, tlen, i0);
      }
      {
        ProfScope ps(prof, "grad_rows_inv", nimg * (spec + img * 4.0) + nb * img * 4.0,
                     nimg * (n / 2.0) * fft, st);
        launch_chain(k_rows_inv<NN, RMAX>, dim3(n / RB, nimg), kThreads, smr, st, S, g, b, L, tw, tlen, i0);
      }
    }
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gradient(const float *x, float *g, const float *b,
                            float2 *S, const float *kspec, const float2 *tw, const float2 *twc,
                            int n, int L, int C, cudaStream_t st, Prof *prof, int chunk,
                            int radix) {
  const bool r8 = radix == 8;              // the alternative plan exists from n = 128
#define MUFFIN_GRAD(NN)                                                                    \
  return r8 ? gradient_n<NN, 8>(x, g, b, S, kspec, tw, twc, L, C, st, prof, chunk)              \
            : gradient_n<NN, 16>(x, g, b, S, kspec, tw, twc, L, C, st, prof, chunk)
#define MUFFIN_GRAD16(NN) return gradient_n<NN, 16>(x, g, b, S, kspec, tw, twc, L, C, st, prof, chunk)
  switch (n) {
    case 2: MUFFIN_GRAD16(2);
    case 4: MUFFIN_GRAD16(4);
    case 8: MUFFIN_GRAD16(8);
    case 16: MUFFIN_GRAD16(16);
    case 32: MUFFIN_GRAD16(32);
    case 64: MUFFIN_GRAD16(64);
    case 128: MUFFIN_GRAD(128);
    case 256: MUFFIN_GRAD(256);
    case 512: MUFFIN_GRAD(512);
    case 1024: MUFFIN_GRAD(1024);
    case 2048: MUFFIN_GRAD(2048);
#undef MUFFIN_GRAD
#undef MUFFIN_GRAD16
    default: return cudaErrorInvalidValue;
  }
}

int fft32_table_len(int n, int radix) { return fft_table_len(n, radix); }
void fft32_tables(int n, float2 *tab, int radix) { fft_tables(n, tab, radix); }
int fft32_cols_table_len(int n) { return cols_table_len(n); }
void fft32_cols_tables(int n, float2 *tab) { cols_tables(n, tab); }

cudaError_t fft2d_c64(double2 *data, double2 *tmp, int n, int nimg,
                      bool inverse, const double2 *tw64, cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    allow_smem(k_fft_rows<double2>);
    attr = true;
  }
  const size_t sm = (size_t)2 * n * sizeof(double2);
  const int thr = n < 256 ? (n < 32 ? 32 : n) : 256;
  dim3 tg((n + 31) / 32, (n + 31) / 32, nimg), tb(32, 8);
  k_fft_rows<double2><<<dim3(n, nimg), thr, sm, st>>>(data, n, inverse, tw64);
  k_transpose64<<<tg, tb, 0, st>>>(data, tmp, n);
  k_fft_rows<double2><<<dim3(n, nimg), thr, sm, st>>>(tmp, n, inverse, tw64);
  k_transpose64<<<tg, tb, 0, st>>>(tmp, data, n);
  return cudaGetLastError();
}

namespace {
int row_threads(int n) { return n < 256 ? (n < 32 ? 32 : n) : 256; }

// z (pairs) = spectra of the packed images, [kx][ky]
template <typename C>
cudaError_t pair_forward(const float *x, const Pairs &P, int np, C *z, C *tmp, const C *tw,
                         cudaStream_t st) {
  const int n = P.n;
  const size_t sm = (size_t)2 * n * sizeof(C);
  allow_smem(k_rows_real<C>);
  allow_smem(k_fft_rows<C>);
  k_rows_real<C><<<dim3(n, np), row_threads(n), sm, st>>>(x, tmp, P, tw);
  k_transpose64<<<dim3((n + 31) / 32, (n + 31) / 32, np), dim3(32, 8), 0, st>>>(
      reinterpret_cast<double2 *>(tmp), reinterpret_cast<double2 *>(z), n);
  k_fft_rows<C><<<dim3(n, np), row_threads(n), sm, st>>>(z, n, false, tw);
  return cudaGetLastError();
}

template <typename C, bool CJ>
cudaError_t pair_convolve(const float *x, const Pairs &P, int np, const double2 *hh, C *z, C *tmp,
                          double c, float *out, const C *tw, cudaStream_t st) {
  cudaError_t e = pair_forward<C>(x, P, np, z, tmp, tw, st);
  if (e != cudaSuccess) return e;
  const int n = P.n;
  const size_t sm = (size_t)2 * n * sizeof(C);
  const dim3 rows(n, np);
  k_pair_mul<C, CJ><<<dim3((n >> 1) + 1, np), row_threads(n), 0, st>>>(z, hh, P);
  k_fft_rows<C><<<rows, row_threads(n), sm, st>>>(z, n, true, tw);
  k_transpose64<<<dim3((n + 31) / 32, (n + 31) / 32, np), dim3(32, 8), 0, st>>>(
      reinterpret_cast<double2 *>(z), reinterpret_cast<double2 *>(tmp), n);
  if (out) {
    allow_smem(k_rows_out<C>);
    k_rows_out<C><<<rows, row_threads(n), sm, st>>>(tmp, out, P, c, tw);
  } else {
    k_fft_rows<C><<<rows, row_threads(n), sm, st>>>(tmp, n, true, tw);
  }
  return cudaGetLastError();
}
}  // namespace

cudaError_t spectra_real(const float *x, const ImageStat *stat, int n, int L, int nimg,
                         double2 *hh, double2 *z, double2 *tmp, const double2 *tw64,
                         cudaStream_t st) {
  const Pairs P{n, L, (L + 1) / 2, stat, nullptr};
  const int np = nimg / L * P.per_cube;
  cudaError_t e = pair_forward<double2>(x, P, np, z, tmp, tw64, st);
  if (e != cudaSuccess) return e;
  k_pair_unpack<<<dim3(n, np), row_threads(n), 0, st>>>(z, hh, P);
  return cudaGetLastError();
}

cudaError_t adjoint_real(const float *x, const ImageStat *stat, const double2 *hh,
                         const double *hmax, int n, int L, int nimg, double2 *z, double2 *tmp,
                         float *out, const float4 *twdd, cudaStream_t st) {
  const Pairs P{n, L, (L + 1) / 2, stat, hmax};
  return pair_convolve<cdd, true>(x, P, nimg / L * P.per_cube, hh, reinterpret_cast<cdd *>(z),
                                  reinterpret_cast<cdd *>(tmp), 1.0 / ((double)n * n), out,
                                  reinterpret_cast<const cdd *>(twdd), st);
}

cudaError_t convolve_real(const float *x, const ImageStat *stat, const double2 *hh,
                          const double *hmax, int n, int L, int nimg, double2 *z, double2 *tmp,
                          const double2 *tw64, cudaStream_t st) {
  const Pairs P{n, L, (L + 1) / 2, stat, hmax};
  return pair_convolve<double2, false>(x, P, nimg / L * P.per_cube, hh, z, tmp, 0.0, nullptr,
                                       tw64, st);
}

cudaError_t c64_real_to_f32(const double2 *in, float *out, double scale,
                            size_t count, cudaStream_t st) {
  k_c64_real_to_f32<<<grid_for(count), 256, 0, st>>>(in, out, scale, count);
  return cudaGetLastError();
}

cudaError_t make_kspec(const double2 *hh, float *kspec, double scale, int n,
                       int L, double *hmax, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(hmax, 0, (size_t)L * sizeof(double), st);
  if (e != cudaSuccess) return e;
  k_make_kspec<<<dim3((n >> 1) + 1, L), row_threads(n), 0, st>>>(
      hh, kspec, scale, n, reinterpret_cast<unsigned long long *>(hmax));
  return cudaGetLastError();
}

}  // namespace muffin
