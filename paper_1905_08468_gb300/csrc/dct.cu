// Spectral step of Algorithm 2 (eqs. vt, v, upt), run for every pixel n:
//     v~ = v + sigma gamma_n C (2 x~^n - x^n);   v = sat(v~);   t = gamma_n C^T v
// with C the orthonormal L x L DCT-II (Sec. 4.2.1), for the band counts that
// have no faster form of their own: the FP32 fast DCT (dct_f32.cu) serves the
// powers of two, tcgen05 (dct_tc.cu) 64 bands.
//
// ADA-PT groups (C = 3 chains) reuse the primal's mask Pi(v~) and add the
// inhomogeneous terms of Algorithm 4:
//     v~'_gamma = v'_gamma + sigma alpha_n C (2x~ - x + gamma (2x~' - x'))
//     t'_gamma  = alpha_n C^T (gamma v'_gamma + v)
// while Algorithm 3's spectral step is the homogeneous one.
//
// Rows of C are even or odd about the middle band (C[k][L-1-l] =
// (-1)^k C[k][l]), so with s_l = z_l + z_{L-1-l}, d_l = z_l - z_{L-1-l} the
// product splits into two half-size ones (even k from s, odd k from d), and
// C^T v into e_l + o_l and e_l - o_l: L FP32 FMAs per voxel for both
// directions together, run as packed pairs of pixels (fma.rn.f32x2).
//
// What bounds it: shared-memory and FMA issue, about L / 2 packed FMAs a
// voxel; the 20 bytes a voxel of HBM traffic hide behind them from L ~ 60 on.
// FP32 on the CUDA cores, not 3xTF32 mma.sync, because the legacy tensor path
// needs three full L x L products: 256 x 256 x 37, one chain, 33.3 -> 24.9 us;
// 512 x 512 x 100, 557 -> 261 us, three chains 4671 -> 1047 us; error of C z
// against 64 bits 2.5e-7 -> 9e-8 at 37 bands, 1.2e-6 -> 1.5e-7 at 100.
//
// Layout: every cube is band-major [L][N]; a CTA takes PT consecutive pixels
// of every band (16-byte loads along the pixels).  The coefficients are read
// through L1 (the two halves' tables of every direction, broadcast to the
// warp), so shared memory holds only the folded input and the new duals.
#include <cuda_runtime.h>

#include <algorithm>

#include "chain.cuh"
#include "kernels.h"

namespace muffin {

namespace {

constexpr int DT = 256;           // threads at most
constexpr int RK = 4;             // rows of a task of C z (4 pixels wide)

struct FoldArgs {
  int L, M, Mp, inverse;      // M = ceil(L / 2) rows of the even half, Mp = M rounded up to 4
  int B, tiles_per_cube, ntiles;
  size_t npix;                // pixels per band (n * n, or a pixel block)
  const float *fwd;           // [2][Mp][Mp]: parity, l, k'  (C[2 k' + parity][l])
  const float *bwd;           // [2][Mp][Mp]: parity, k', l
  const float *alpha;
  const DevScalars *sc;
  const float *xt, *x;        // iterate inputs [C][L][N]
  float *v, *t;               // iterate state [C][L][N]
  const float *in;            // operator input [L][N]
  float *out;                 // operator output [L][N]
};

__device__ __forceinline__ float4 ld4(const float *p) {
  return *reinterpret_cast<const float4 *>(p);
}
__device__ __forceinline__ void st4(float *p, float4 v) {
  *reinterpret_cast<float4 *>(p) = v;
}

// acc[r] (4 pixels) += sum_j A[j * Mp + r] * B[j * PT], j < len, r < R; U steps' loads
// in flight
template <int PT, int R, int U>
__device__ __forceinline__ void half_product(const float *__restrict__ A, int Mp, const float *B,
                                             int len, float2 (&acc)[R][2]) {
#pragma unroll U
  for (int j = 0; j < len; ++j) {
    float cr[R];
    if constexpr (R == 4) {
      const float4 c = __ldg(reinterpret_cast<const float4 *>(A + (size_t)j * Mp));
      cr[0] = c.x; cr[1] = c.y; cr[2] = c.z; cr[3] = c.w;
    } else {
      const float2 c = __ldg(reinterpret_cast<const float2 *>(A + (size_t)j * Mp));
      cr[0] = c.x; cr[1] = c.y;
    }
    const float4 z = ld4(B + j * PT);
    const float2 za = make_float2(z.x, z.y), zb = make_float2(z.z, z.w);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2 cc = make_float2(cr[r], cr[r]);
      acc[r][0] = __ffma2_rn(cc, za, acc[r][0]);
      acc[r][1] = __ffma2_rn(cc, zb, acc[r][1]);
    }
  }
}

// RB: rows of a task of C^T v; U: depth of the products' loads
template <int CH, int MODE, int PT, int RB, int U>
__global__ void __launch_bounds__(DT, 3) k_dct_fold(FoldArgs a) {
  chain_enter();
  constexpr int PG = PT / 4;                      // pixel groups
  const int NG = blockDim.x / PG;                 // row groups in flight
  extern __shared__ float sm[];
  const int L = a.L, M = a.M, Mo = a.L / 2, Mp = a.Mp, G = Mp / RK;
  const int half = M * PT;                        // one parity of one chain
  float *zs = sm;                                 // [CH][2][M][PT] folded input
  float *vs = MODE == WAVE_ITERATE ? zs + CH * 2 * half : zs;   // [CH][2][M][PT] new duals
  const size_t N = a.npix;
  const size_t CS = (size_t)a.B * L * N;          // chain stride
  const int pg = threadIdx.x % PG, rg = threadIdx.x / PG;
  const bool fwd = MODE == WAVE_ITERATE || !a.inverse;
  const bool bwd = MODE == WAVE_ITERATE || a.inverse;
  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int cube = tile / a.tiles_per_cube;
    const size_t pix = (size_t)(tile - cube * a.tiles_per_cube) * PT + 4 * pg;
    const bool ok = pix < N;                      // N is a multiple of 4
    const size_t cb = (size_t)cube * L * N + pix; // the thread's pixels in band 0
    float gamma = 0.f, sigma = 0.f, al[4] = {0.f, 0.f, 0.f, 0.f};
    if (MODE == WAVE_ITERATE) {
      gamma = (float)a.sc[cube].gamma;
      sigma = (float)a.sc[cube].sigma;
      // a pixel block of the sharded form starts anywhere: no vector load
      if (ok)
#pragma unroll
        for (int e = 0; e < 4; ++e) al[e] = a.alpha[(size_t)cube * N + pix + e];
    }
    __syncthreads();                              // the previous tile's readers are done
    // ---- input, folded about the middle band (operator C^T: split by parity)
#pragma unroll 2
    for (int j = rg; j < M; j += NG) {
      const int j2 = L - 1 - j;
      float4 p[CH], q[CH];
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        p[c] = q[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!ok) continue;
        if (MODE == WAVE_TRANSFORM) {
          const int r1 = fwd ? j : 2 * j, r2 = fwd ? j2 : 2 * j + 1;
          p[c] = ld4(a.in + cb + (size_t)r1 * N);
          if (fwd || r2 < L) q[c] = ld4(a.in + cb + (size_t)r2 * N);
        } else {
          const size_t o1 = c * CS + cb + (size_t)j * N, o2 = c * CS + cb + (size_t)j2 * N;
          const float4 t1 = ld4(a.xt + o1), x1 = ld4(a.x + o1);
          const float4 t2 = ld4(a.xt + o2), x2 = ld4(a.x + o2);
          p[c] = make_float4(2.f * t1.x - x1.x, 2.f * t1.y - x1.y, 2.f * t1.z - x1.z, 2.f * t1.w - x1.w);
          q[c] = make_float4(2.f * t2.x - x2.x, 2.f * t2.y - x2.y, 2.f * t2.z - x2.z, 2.f * t2.w - x2.w);
        }
      }
      if (CH == 3) {                              // Algorithm 4 input
        p[2] = make_float4(fmaf(gamma, p[2].x, p[0].x), fmaf(gamma, p[2].y, p[0].y),
                           fmaf(gamma, p[2].z, p[0].z), fmaf(gamma, p[2].w, p[0].w));
        q[2] = make_float4(fmaf(gamma, q[2].x, q[0].x), fmaf(gamma, q[2].y, q[0].y),
                           fmaf(gamma, q[2].z, q[0].z), fmaf(gamma, q[2].w, q[0].w));
      }
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        float4 s = p[c], d = q[c];
        if (fwd) {
          if (j < Mo) {
            s = make_float4(p[c].x + q[c].x, p[c].y + q[c].y, p[c].z + q[c].z, p[c].w + q[c].w);
            d = make_float4(p[c].x - q[c].x, p[c].y - q[c].y, p[c].z - q[c].z, p[c].w - q[c].w);
          } else {
            d = make_float4(0.f, 0.f, 0.f, 0.f);  // the middle band of an odd count
          }
        }
        float *z = zs + c * 2 * half + j * PT + 4 * pg;
        st4(z, s);
        st4(z + half, d);
      }
    }
    __syncthreads();
    // ---- C z and the dual update; task = (parity, four rows, four pixels)
    if (fwd)
      for (int f = rg; f < 2 * G; f += NG) {
        const int par = f >= G ? 1 : 0, r0 = (f - par * G) * RK;
        const int len = par ? Mo : M;             // rows of this half, and its inputs
        uint32_t keep = 0;
#pragma unroll 1
        for (int c = 0; c < CH; ++c) {
          const size_t vo = c * CS + cb + (size_t)(2 * r0 + par) * N;
          float4 old[RK];
          if (MODE == WAVE_ITERATE)
#pragma unroll
            for (int r = 0; r < RK; ++r)
              old[r] = ok && r0 + r < len ? ld4(a.v + vo + (size_t)(2 * r) * N)
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
          float2 acc[RK][2];
#pragma unroll
          for (int r = 0; r < RK; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
          half_product<PT, RK, U>(a.fwd + (size_t)par * Mp * Mp + r0, Mp,
                           zs + (2 * c + par) * half + 4 * pg, len, acc);
          const float sg = c == 2 ? sigma : sigma * gamma;
#pragma unroll
          for (int r = 0; r < RK; ++r) {
            if (r0 + r >= len) continue;
            float w[4] = {acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y};
            if (MODE == WAVE_TRANSFORM) {
              if (ok) st4(a.out + vo + (size_t)(2 * r) * N, make_float4(w[0], w[1], w[2], w[3]));
              continue;
            }
            const float o[4] = {old[r].x, old[r].y, old[r].z, old[r].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float vt = fmaf(sg * al[e], w[e], o[e]);
              const uint32_t bit = 1u << (4 * r + e);
              if (c == 0) {
                w[e] = satf(vt);
                if (fabsf(vt) <= 1.f) keep |= bit;
              } else {
                w[e] = (keep & bit) ? vt : 0.f;
              }
            }
            if (ok) st4(a.v + vo + (size_t)(2 * r) * N, make_float4(w[0], w[1], w[2], w[3]));
            float *d = vs + par * half + (r0 + r) * PT + 4 * pg;   // chain 0's duals
            if (CH == 3 && c == 2) {              // gamma v'_gamma + v
              const float4 v0 = ld4(d);
              w[0] = fmaf(gamma, w[0], v0.x); w[1] = fmaf(gamma, w[1], v0.y);
              w[2] = fmaf(gamma, w[2], v0.z); w[3] = fmaf(gamma, w[3], v0.w);
            }
            st4(d + c * 2 * half, make_float4(w[0], w[1], w[2], w[3]));
          }
        }
      }
    if (!bwd) continue;
    __syncthreads();
    // ---- back-projection C^T v; task = (chain, rows l and L - 1 - l, four pixels)
    const int GB = Mp / RB;
    for (int f = rg; f < CH * GB; f += NG) {
      const int c = CH == 1 ? 0 : f / GB, r0 = (f - c * GB) * RB;
      const float *vc = vs + 2 * c * half + 4 * pg;
      float2 ev[RB][2], od[RB][2];
#pragma unroll
      for (int r = 0; r < RB; ++r) ev[r][0] = ev[r][1] = od[r][0] = od[r][1] = make_float2(0.f, 0.f);
      half_product<PT, RB, U>(a.bwd + r0, Mp, vc, M, ev);
      half_product<PT, RB, U>(a.bwd + (size_t)Mp * Mp + r0, Mp, vc + half, Mo, od);
      if (!ok) continue;
      const float g = c == 2 ? 1.f : gamma;
      float s2[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) s2[e] = MODE == WAVE_TRANSFORM ? 1.f : g * al[e];
      float *dst = (MODE == WAVE_TRANSFORM ? a.out : a.t + c * CS) + cb;
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int l = r0 + r;
        if (l >= M) continue;
        st4(dst + (size_t)l * N,
            make_float4(s2[0] * (ev[r][0].x + od[r][0].x), s2[1] * (ev[r][0].y + od[r][0].y),
                        s2[2] * (ev[r][1].x + od[r][1].x), s2[3] * (ev[r][1].y + od[r][1].y)));
        if (l < Mo)
          st4(dst + (size_t)(L - 1 - l) * N,
              make_float4(s2[0] * (ev[r][0].x - od[r][0].x), s2[1] * (ev[r][0].y - od[r][0].y),
                          s2[2] * (ev[r][1].x - od[r][1].x), s2[3] * (ev[r][1].y - od[r][1].y)));
      }
    }
  }
}

template <int CH, int MODE, int PT, int RB, int U = 4>
cudaError_t launch_fold_r(FoldArgs &a, int ctas_per_sm, size_t sm, cudaStream_t st, Prof *prof) {
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_dct_fold<CH, MODE, PT, RB, U>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         208 * 1024);
    attr = true;
  }
  a.tiles_per_cube = (int)((a.npix + PT - 1) / PT);
  a.ntiles = a.tiles_per_cube * a.B;
  // threads: whole row groups of C z in as few rounds as 256 threads allow,
  // all of them busy in every round (37 bands: 160 threads, one round); narrow tiles,
  // which are few, take as many as load the tile in a round and as C^T v of all
  // chains has (64 x 64 x 20, three chains: 17.1 -> 12.7 us)
  int groups = 2 * (a.Mp / RK);
  if (PT == 16) groups = std::max(groups, std::max(std::min(a.M, 32), RB == 2 ? CH * (a.Mp / RB) : 0));
  const int rounds = (groups * (PT / 4) + DT - 1) / DT;
  const int threads = ((groups + rounds - 1) / rounds * (PT / 4) + 31) / 32 * 32;
  int grid = a.ntiles;
  if (ctas_per_sm > 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = (int)std::min<long long>(grid, (long long)ctas_per_sm * sms);
  }
  const double vox = (double)a.npix * a.L * a.B;
  ProfScope ps(prof, MODE == WAVE_ITERATE ? "spectral_dual" : "spectral_op",
               MODE == WAVE_ITERATE ? CH * vox * 20.0 : vox * 8.0,
               (MODE == WAVE_ITERATE ? 2.0 : 1.0) * CH * a.L * vox, st);
  launch_chain(k_dct_fold<CH, MODE, PT, RB, U>, grid, threads, sm, st, a);
  return cudaGetLastError();
}

// Two rows a task of C^T v keep more threads busy below 40 bands (512 x 512 x
// 23: 37 against 48 us); from there on four rows halve the shared-memory reads
// per product (512 x 512 x 100: 261 against 311 us).
template <int CH, int MODE, int PT>
cudaError_t launch_fold(FoldArgs &a, int ctas_per_sm, size_t sm, cudaStream_t st, Prof *prof) {
  return a.L < 40 ? launch_fold_r<CH, MODE, PT, 2>(a, ctas_per_sm, sm, st, prof)
                  : launch_fold_r<CH, MODE, PT, 4>(a, ctas_per_sm, sm, st, prof);
}

// Tiles of 16 pixels.  Few of them are bound by the latency of a thread's tasks, so an
// iteration's step takes the short ones (two rows) up to 200 bands (64 x 64 x 56, one
// chain 13.8 -> 12.4 us), with three chains up to 64 (64 x 64 x 48: 24.8 -> 16.3).  From
// 200 bands on the tables (4 Mp^2 floats, 160 KB) stay in no L1, and the loads of eight
// steps in flight cover L2's latency (128 x 128 x 250 with the line below: 160 -> 120
// us; from 300 on with four rows a task, 64 x 64 x 1000: 1000 -> 919).
template <int CH, int MODE>
cudaError_t launch_narrow(FoldArgs &a, int ctas_per_sm, size_t sm, cudaStream_t st, Prof *prof) {
  if constexpr (MODE == WAVE_ITERATE) {
    if (a.L < (CH == 1 ? 200 : 64)) return launch_fold_r<CH, MODE, 16, 2>(a, ctas_per_sm, sm, st, prof);
    if constexpr (CH == 1) {
      if (a.L < 260) return launch_fold_r<CH, MODE, 16, 2, 8>(a, ctas_per_sm, sm, st, prof);
      if (a.L >= 300) return launch_fold_r<CH, MODE, 16, 4, 8>(a, ctas_per_sm, sm, st, prof);
    }
  }
  return launch_fold<CH, MODE, 16>(a, ctas_per_sm, sm, st, prof);
}

template <int CH, int MODE>
cudaError_t dispatch_fold(FoldArgs &a, int ctas_per_sm, cudaStream_t st, Prof *prof) {
  // The widest pixel tile with room for three CTAs an SM (wider rows for the
  // loads and more products per coefficient read), narrower while the image
  // has too few tiles for two CTAs an SM.  One chain of 200 bands and more, whose
  // tables leave no L1 beside wide tiles, goes on with narrow ones until the wide
  // ones' second wave is a third full (608 of them: 128 x 128 x 250, 512 tiles of 32
  // pixels, 160 -> 120 us; 256 x 256 x 200, 2048: wide 256, narrow 275).
  const auto sm = [&](int pt) {
    return (size_t)(MODE == WAVE_ITERATE ? 4 : 2) * CH * a.M * pt * sizeof(float);
  };
  const bool cold = CH == 1 && a.L >= 200 && (MODE == WAVE_ITERATE || a.L < 260 || a.L >= 300);
  const size_t least = cold ? 608 : 304;
  const auto fits = [&](int pt) {
    return sm(pt) <= 72 * 1024 && (a.npix + pt - 1) / pt * a.B >= least;
  };
  if (fits(64)) return launch_fold<CH, MODE, 64>(a, ctas_per_sm, sm(64), st, prof);
  if (fits(32)) return launch_fold<CH, MODE, 32>(a, ctas_per_sm, sm(32), st, prof);
  return launch_narrow<CH, MODE>(a, ctas_per_sm, sm(16), st, prof);
}

FoldArgs base_args(const DctArgs &d) {
  FoldArgs a{};
  a.L = d.L; a.M = (d.L + 1) / 2; a.Mp = (a.M + 3) / 4 * 4;
  a.B = d.B > 0 ? d.B : 1;
  a.npix = d.npix ? d.npix : (size_t)d.n * d.n;
  a.fwd = d.fold; a.bwd = d.fold + (size_t)2 * a.Mp * a.Mp;
  a.alpha = d.alpha; a.sc = d.sc;
  return a;
}

}  // namespace

int dct_fold_table_len(int L) {
  const int mp = ((L + 1) / 2 + 3) / 4 * 4;
  return 4 * mp * mp;
}

void dct_fold_tables(int L, const double *C, float *tab) {
  const int m = (L + 1) / 2, mp = (m + 3) / 4 * 4;
  float *fwd = tab, *bwd = tab + (size_t)2 * mp * mp;
  std::fill(tab, tab + dct_fold_table_len(L), 0.f);
  for (int k = 0; k < L; ++k)
    for (int l = 0; l < ((k & 1) ? L / 2 : m); ++l) {
      const float c = (float)C[(size_t)k * L + l];
      const size_t par = (size_t)(k & 1) * mp * mp;
      fwd[par + (size_t)l * mp + k / 2] = c;
      bwd[par + (size_t)(k / 2) * mp + l] = c;
    }
}

cudaError_t dct_dual(const DctArgs &d, const Group &gr, cudaStream_t st) {
  if (d.f32) return dct_dual_f32(d, gr, st);
  if (d.tc && d.L == 64 && d.Lp == 64) return dct_dual_tc(d, gr, d.err, st);
  FoldArgs a = base_args(d);
  a.xt = gr.xt; a.x = gr.x; a.v = gr.v; a.t = gr.t;
  if (gr.C == 3) return dispatch_fold<3, WAVE_ITERATE>(a, d.ctas_per_sm, st, d.prof);
  return dispatch_fold<1, WAVE_ITERATE>(a, d.ctas_per_sm, st, d.prof);
}

cudaError_t dct_op(const DctArgs &d, const float *in, float *out, int inverse,
                   cudaStream_t st) {
  if (d.f32) return dct_op_f32(d, in, out, inverse, st);
  FoldArgs a = base_args(d);
  a.in = in; a.out = out; a.inverse = inverse;
  return dispatch_fold<1, WAVE_TRANSFORM>(a, 0, st, d.prof);
}

}  // namespace muffin
