// One level of the wavelet analysis + spatial dual update (eqs. stpp, stpu and
// the derivative forms; the transforms and layouts of wavelet.cu) with the
// columns of a tile in registers, for levels with h >= 16 coefficients a side.
//
// What bounds a level that keeps its tile and both filter passes in shared
// memory (k_ana) is the shared-memory pipe: 66-70 percent busy at 54-61
// percent of the DRAM rate.  So the y filters run first and straight from
// registers: a lane owns one column of the rows its tile needs, loaded once a
// chain (coalesced along the rows), and only their results cross shared
// memory, once, to the x filters.  Per (chain, basis) step:
//   1. the U values of the lane's item are requested, the next step's U tile
//      is prefetched into L2;
//   2. y pass of the lane's column -> low and high rows in shared memory (two
//      buffers, one barrier a step);
//   3. x pass of Q neighbouring coefficients of a row (low rows: LL, DX; high
//      rows: DY, HH), the dual update, 16-byte stores.
// Rows are kept as 16-byte chunks dealt into Q / 2 groups, which makes the y
// pass's 4-byte stores and the x pass's 16-byte loads (lanes Q / 2 chunks
// apart) free of bank conflicts.  Both passes run packed pairs (fma.rn.f32x2)
// over the even and odd taps.
//
// One chain a CTA: the primal's launch records the masks Pi(p) (a word an item
// and basis), the derivatives' launch reads them.  All three chains in one CTA
// took 3.0 - 3.6 ms where the two launches take 2.49 (1024 x 1024 x 64, level
// 1): the chains' column loads do not overlap other work inside a CTA.
// Strips of different bases a warp, which need no barrier at all, thrash the
// instruction cache (hit rate 63 percent; 3.63 ms).
//
// Measured against k_ana, level 1: 1024 x 1024 x 256, one chain 5.87 -> 2.97
// ms (5.8 TB/s of design bytes, 0.85 of the copy bandwidth); 256 x 256 x 32, one
// chain 57.6 -> 33.7 us; three chains 1024 x 1024 x 64 2.91 -> 2.49 ms.
#include <cuda_runtime.h>

#include "chain.cuh"
#include "kernels.h"
#include "wavelet.h"

namespace muffin {

// (h_2j, h_2j+1) and (g_2j, g_2j+1) of db1..db8 (taps beyond 2p are zero)
__constant__ float2 c_cols_h[8][8];
__constant__ float2 c_cols_g[8][8];

namespace {

constexpr int CX = 64;                  // tile columns
constexpr int PMAX = 8;
constexpr int NT = 160;                 // threads: one a column of the tile and its halo
constexpr int VP = 160;                 // floats of a row in shared memory
static_assert(2 * CX + 2 * PMAX - 2 <= NT, "a column a thread");

// Tiles of CY rows.  16 rows read the fewest halo rows and the widest items;
// 8 rows make twice the CTAs, for levels that fill few waves.
template <int CY>
struct Tile {
  static constexpr int RP = CY + PMAX - 1;    // row pairs of a column
  static constexpr int Q = CY / 2;            // coefficients of an item
  static constexpr int ITEMS = CX / Q * CY;   // items of a tile: 128
  static constexpr int NG = Q / 2;            // chunk groups (an item's pixels: NG chunks)
  static constexpr int GRP = 40 / NG;         // chunks of a group
  static constexpr int VB = 2 * CY * VP;      // floats of a buffer: low rows, high rows
  static_assert(ITEMS <= NT && 4 * GRP * NG == VP, "an item a thread, whole rows");
  static_assert(CX == 64 && CY >= 8 && ITEMS == 128, "ana_mask_words");
};

enum Source { SRC_ITERATE, SRC_OPERATOR, SRC_LL };

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// The tap pairs of basis P, read where they are used: as plain constants the
// compiler hoists those of every basis out of the loop over the bases, and
// spills them (2 KB a thread).
template <int P, int J = 0>
__device__ __forceinline__ void taps(float2 (&hp)[P], float2 (&gp)[P]) {
  asm volatile("ld.const.v2.f32 {%0, %1}, [_ZN6muffin8c_cols_hE+%2];"
               : "=f"(hp[J].x), "=f"(hp[J].y) : "n"(((P - 1) * 8 + J) * 8));
  asm volatile("ld.const.v2.f32 {%0, %1}, [_ZN6muffin8c_cols_gE+%2];"
               : "=f"(gp[J].x), "=f"(gp[J].y) : "n"(((P - 1) * 8 + J) * 8));
  if constexpr (J + 1 < P) taps<P, J + 1>(hp, gp);
}

// y pass: v[r] = sum_j (h_2j, h_2j+1) . (z_2(r+j), z_2(r+j)+1), low and high
template <int P, int CY>
__device__ __forceinline__ void ypass(const float2 (&z)[Tile<CY>::RP], float *v) {
  float2 hp[P], gp[P];
  taps<P>(hp, gp);
#pragma unroll
  for (int r = 0; r < CY; ++r) {
    float2 lo = make_float2(0.f, 0.f), hi = lo;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      lo = fma2(hp[j], z[r + j], lo);
      hi = fma2(gp[j], z[r + j], hi);
    }
    v[r * VP] = lo.x + lo.y;
    v[(CY + r) * VP] = hi.x + hi.y;
  }
}

// x pass of one row: low and high outputs of Q coefficients
template <int P, int CY>
__device__ __forceinline__ void xpass(const float *v, float (&lo)[Tile<CY>::Q],
                                      float (&hi)[Tile<CY>::Q]) {
  using T = Tile<CY>;
  constexpr int NP = T::Q + P - 1, NC = (NP + 1) / 2;   // pixel pairs, 16-byte chunks
  float2 hp[P], gp[P], w[2 * NC];
#pragma unroll
  for (int m = 0; m < NC; ++m) {
    const float4 q = *reinterpret_cast<const float4 *>(v + (m % T::NG * T::GRP + m / T::NG) * 4);
    w[2 * m] = make_float2(q.x, q.y);
    w[2 * m + 1] = make_float2(q.z, q.w);
  }
  taps<P>(hp, gp);
#pragma unroll
  for (int k = 0; k < T::Q; ++k) {
    float2 l = make_float2(0.f, 0.f), h = l;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      l = fma2(hp[j], w[k + j], l);
      h = fma2(gp[j], w[k + j], h);
    }
    lo[k] = l.x + l.y;
    hi[k] = h.x + h.y;
  }
}

template <int Q>
__device__ __forceinline__ void load_item(float (&w)[Q], const float *p) {
#pragma unroll
  for (int k = 0; k < Q; k += 4) {
    const float4 v = *reinterpret_cast<const float4 *>(p + k);
    w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
  }
}
template <int Q>
__device__ __forceinline__ void store_item(float *p, const float (&w)[Q]) {
#pragma unroll
  for (int k = 0; k < Q; k += 4)
    *reinterpret_cast<float4 *>(p + k) = make_float4(w[k], w[k + 1], w[k + 2], w[k + 3]);
}

#define MUFFIN_BASES(CALL) \
  switch (b) { \
    case 0: CALL(1); break; case 1: CALL(2); break; case 2: CALL(3); break; \
    case 3: CALL(4); break; case 4: CALL(5); break; case 5: CALL(6); break; \
    case 6: CALL(7); break; default: CALL(8); break; \
  }

// Chain 0 (DERIV = false; records the masks when a.masks is set) or the chains
// 1 + blockIdx.z of the derivatives.  SRC_LL: one basis a CTA (blockIdx.y =
// band * K + basis) of the previous level's approximations; otherwise level 1,
// all bases, or (SPLIT) one of `groups` shares of them.  CTAs an SM: as many as keep the column in registers unspilled
// (the derivatives' code needs more of them).
template <int CY, int SRC, bool LAST, bool DERIV, bool SPLIT>
__global__ void __launch_bounds__(NT, DERIV ? (CY == 16 ? 2 : 3) : (CY == 16 ? 3 : 4))
k_ana_cols(AnaArgs a, bool iterate, int groups) {
  chain_enter();
  using T = Tile<CY>;
  constexpr int Q = T::Q;
  extern __shared__ float vbuf[];                   // [2][low, high][CY][VP]
  const bool ITER = SRC == SRC_ITERATE || (SRC == SRC_LL && iterate);
  const int tid = threadIdx.x;
  const unsigned n = a.n, M = SRC == SRC_LL ? a.M : n, h = M >> 1, Mm = M - 1, hn = h * n;
  const unsigned ntx = (h + CX - 1) / CX;
  const unsigned kx0 = (blockIdx.x % ntx) * CX, ky0 = (blockIdx.x / ntx) * CY;
  // bases b0, b0 + step, ... below b1
  const int K = a.K, shares = SRC == SRC_LL ? K : SPLIT ? groups : 1, l = blockIdx.y / shares;
  const int step = SRC == SRC_LL ? 1 : shares;
  const int b0 = blockIdx.y % shares, b1 = SRC == SRC_LL ? b0 + 1 : K;
  const int c = DERIV ? 1 + blockIdx.z : 0;
  const size_t NN = (size_t)n * n, CS = (size_t)a.L * NN;
  float mu = 0.f, q = 1.f;
  if (ITER) {
    const DevScalars &S = a.sc[l / a.Lc];
    mu = (float)S.mu;
    q = (float)(S.sigma * (double)a.beta[l]);       // sigma beta_l (d/dmu) ...
    if (c != 1) q *= mu;                            // ... or sigma mu_l
  }
  // the thread's item: row iy, coefficients kx .. kx + Q - 1 (h a multiple of Q)
  const int iy = tid / (CX / Q), iq = tid % (CX / Q);
  const unsigned kx = kx0 + Q * iq, ky = ky0 + iy;
  const bool act = tid < T::ITEMS && kx < h && ky < h;
  const unsigned uo = ky * n + kx, lo_off = ky * h + kx;
  const float *vrow = vbuf + iy * VP + 4 * iq;
  // the thread's column of the tile
  const unsigned xx = (2 * kx0 + tid) & Mm;
  float *vcol = vbuf + ((tid >> 2) % T::NG * T::GRP + (tid >> 2) / T::NG) * 4 + (tid & 3);
  const bool own = tid < 2 * CX + 2 * b1 - 2;       // b1: the longest filter's basis
  const int rows = CY + b1 - 1;                     // row pairs the filters reach
  float2 z[T::RP];
  if (own) {
    const float *xt = SRC == SRC_ITERATE ? a.xt + c * CS + l * NN + xx : nullptr;
    const float *x = SRC == SRC_ITERATE   ? a.x + c * CS + l * NN + xx
                     : SRC == SRC_OPERATOR ? a.in + l * NN + xx
                                           : a.in + ((size_t)(c * a.L + l) * K + b0) * M * M + xx;
#pragma unroll
    for (int i = 0; i < T::RP; ++i) {
      // a fence now and then bounds how many loads the compiler keeps in flight
      if (i % 8 == 7) asm volatile("" ::: "memory");
      float v[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const unsigned o = ((2 * ky0 + 2 * i + e) & Mm) * M;
        if (SRC == SRC_LL) {
          v[e] = 0.f;
          if (i < CY || i < rows) v[e] = x[o];
        } else {
          v[e] = SRC == SRC_ITERATE ? 2.f * xt[o] - x[o] : x[o];
        }
      }
      z[i] = make_float2(v[0], v[1]);
    }
    if (SRC == SRC_ITERATE && DERIV && c == 1) {    // Algorithm 3 input: z0 + mu z1
      xt -= CS;
      x -= CS;
#pragma unroll
      for (int i = 0; i < T::RP; ++i) {
        if (i % 8 == 7) asm volatile("" ::: "memory");
        float v[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const unsigned o = ((2 * ky0 + 2 * i + e) & Mm) * M;
          v[e] = 2.f * xt[o] - x[o];
        }
        z[i] = make_float2(fmaf(mu, z[i].x, v[0]), fmaf(mu, z[i].y, v[1]));
      }
    }
  }
  uint32_t *mk = a.masks ? a.masks + ((size_t)l * K * gridDim.x + blockIdx.x) * T::ITEMS + tid
                         : nullptr;
  int buf = 0;
#pragma unroll 1
  for (int b = b0; b < b1; b += step) {
    const size_t img = (size_t)(c * a.L + l) * K + b;
    float *ub = a.u + img * NN;
    uint32_t keep = 0;
    float u[LAST ? 4 : 3][Q];                       // DX, HH, DY (and LL)
    if (ITER && act) {
      load_item(u[0], ub + uo + h);
      load_item(u[1], ub + uo + hn + h);
      load_item(u[2], ub + uo + hn);
      if (LAST) load_item(u[LAST ? 3 : 0], ub + uo);
      if (DERIV) keep = mk[(size_t)b * gridDim.x * T::ITEMS];
    }
    if (SRC == SRC_ITERATE && tid < 6 * CY && b + step < b1) {
      // the next step's U tile into L2, a 128-byte line a thread
      const int sb = (tid % 6) >> 1;
      const unsigned px = kx0 + 32 * (tid & 1), py = ky0 + tid / 6;
      if (px < h && py < h) {
        const float *p = ub + step * NN + (py * n + px) + (sb == 0 ? h : sb == 1 ? hn : hn + h);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
      }
    }
    if (own) {
#define MUFFIN_Y(P) ypass<P, CY>(z, vcol + buf)
      MUFFIN_BASES(MUFFIN_Y)
    }
    __syncthreads();   // the other buffer's readers passed the previous barrier
    if (act) {
#pragma unroll 1
      for (int e = 0; e < 2; ++e) {                 // low rows: DX, LL; high rows: HH, DY
        float cl[Q], ch[Q];
        const float *v = vrow + buf + e * CY * VP;
#define MUFFIN_X(P) xpass<P, CY>(v, cl, ch)
        MUFFIN_BASES(MUFFIN_X)
        auto update = [&](float (&w)[Q], const float (&uv)[Q], int sh) {
          if (!ITER) return;
#pragma unroll
          for (int k = 0; k < Q; ++k) {
            const float p = fmaf(q, w[k], uv[k]);
            if (DERIV) {
              w[k] = (keep >> (k + sh)) & 1u ? p : 0.f;
            } else {
              w[k] = satf(p);
              if (fabsf(p) <= 1.0f) keep |= 1u << (k + sh);
            }
          }
        };
        if (e == 0) {
          update(ch, u[0], 0);
          store_item(ub + uo + h, ch);
          if (LAST) {
            update(cl, u[LAST ? 3 : 0], 3 * Q);
            store_item(ub + uo, cl);
          } else {
            store_item(a.ll_out + img * ((size_t)h * h) + lo_off, cl);
          }
        } else {
          update(ch, u[1], Q);
          store_item(ub + uo + hn + h, ch);
          update(cl, u[2], 2 * Q);
          store_item(ub + uo + hn, cl);
        }
      }
      if (ITER && !DERIV && mk) mk[(size_t)b * gridDim.x * T::ITEMS] = keep;
    }
    buf ^= T::VB;
  }
}

template <int CY, int SRC, bool LAST>
cudaError_t launch(const AnaArgs &a, int chains, bool iterate, cudaStream_t st) {
  using T = Tile<CY>;
  constexpr size_t sm = (size_t)(SRC == SRC_LL ? 1 : 2) * T::VB * sizeof(float);
  static_assert(sm <= 48 * 1024, "no opt-in for more shared memory");
  const int h = a.M >> 1, nt = ((h + CX - 1) / CX) * ((h + CY - 1) / CY);
  // level 1 with few tiles: the bases dealt to CTAs of their own while all fit
  // one wave of the 8-row tiles (64 x 64 x 8: 14.2 -> 8.5 us)
  int groups = 1;
  if (CY == 8 && SRC != SRC_LL)
    while (2 * groups <= a.K && (long long)nt * a.L * 2 * groups <= 608) groups *= 2;
  const int ny = a.L * (SRC == SRC_LL ? a.K : groups);
  AnaArgs g = a;
  if (chains == 1) g.masks = nullptr;
  const dim3 g1(nt, ny), g2(nt, ny, 2);
  if constexpr (CY == 8 && SRC != SRC_LL) {
    if (groups > 1) {
      launch_chain(k_ana_cols<CY, SRC, LAST, false, true>, g1, NT, sm, st, g, iterate, groups);
      if constexpr (SRC != SRC_OPERATOR)
        if (chains == 3) launch_chain(k_ana_cols<CY, SRC, LAST, true, true>, g2, NT, sm, st, g, iterate, groups);
      return cudaGetLastError();
    }
  }
  launch_chain(k_ana_cols<CY, SRC, LAST, false, false>, g1, NT, sm, st, g, iterate, 1);
  if constexpr (SRC != SRC_OPERATOR)
    if (chains == 3) launch_chain(k_ana_cols<CY, SRC, LAST, true, false>, g2, NT, sm, st, g, iterate, 1);
  return cudaGetLastError();
}

template <int SRC>
cudaError_t dispatch(const AnaArgs &a, int chains, bool iterate, bool rows8, cudaStream_t st) {
  if (rows8)
    return a.last ? launch<8, SRC, true>(a, chains, iterate, st)
                  : launch<8, SRC, false>(a, chains, iterate, st);
  return a.last ? launch<16, SRC, true>(a, chains, iterate, st)
                : launch<16, SRC, false>(a, chains, iterate, st);
}

}  // namespace

cudaError_t upload_cols_filters(const float2 hp[8][8], const float2 gp[8][8]) {
  cudaError_t e = cudaMemcpyToSymbol(c_cols_h, hp, sizeof(c_cols_h));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_cols_g, gp, sizeof(c_cols_g));
  return e;
}

cudaError_t ana_cols(const AnaArgs &a, int chains, bool iterate, bool level1, int flip,
                     cudaStream_t st) {
  // 16-row tiles run 3 CTAs an SM (456 in all): below four waves the last,
  // partly empty one costs more than the 8-row tiles' extra halo (256 x 256 x 32:
  // 33.7 us with 8 rows, 35.8 with 16; 1024 x 1024 x 256: 3.14 and 2.97 ms).
  const long long h = a.M >> 1, ctas = ((h + CX - 1) / CX) * ((h + 15) / 16) * a.L * (level1 ? 1 : a.K);
  const bool rows8 = (ctas < 4 * 456) != (flip != 0);
  if (!level1) return dispatch<SRC_LL>(a, chains, iterate, rows8, st);
  return iterate ? dispatch<SRC_ITERATE>(a, chains, true, rows8, st)
                 : dispatch<SRC_OPERATOR>(a, 1, false, rows8, st);
}

}  // namespace muffin
