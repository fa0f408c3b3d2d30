// ray.cu - parallel-beam ray transform (the forward operator of the
// learned primal-dual reconstruction of Sec. 4.4) and its exact transpose.
//
//   k_ray_forward  a CTA takes 256 bins of up to two neighbouring angles and up
//                  to four images: Joseph's method, one linear-interpolation
//                  sample per pixel row (or column), the rows it samples
//                  staged in shared memory with the images interleaved.
//   k_ray_adjoint  one or two pixels and up to four images per thread: for each angle,
//                  the bins whose rays sample this pixel's row (column) near
//                  it, with the forward's own weights.
//
// Sampling of angle a: the ray of bin d meets row (column) t of the image at
// the fractional pixel coordinate u = A_a d + B_a t + C_a along that row
// (column); the image is interpolated between pixels floor(u) and
// floor(u) + 1 with weights 1 - frac(u) and frac(u), and the samples are
// summed with weight w_a = h / |cos phi| (h / |sin phi|).  Both kernels
// evaluate u with the same float32 expression, so the adjoint applies
// exactly the forward's weights.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/shearlet_ray.h"
#include "internal.h"

namespace {

struct AngleParam {
  float A, B, C, w;   // u = A d + B t + C; sample weight w
  int by_rows;        // 1: sample t is a pixel row (|cos phi| >= |sin phi|)
  float inv_a;        // 1 / A
  int bins;           // adjoint: bins from floor(d - 1/|A| - ADJ_MARGIN) on that hold
                      // every bin with |u - k| < 1 around the fractional bin d
  int pad;
};
static_assert(sizeof(AngleParam) == 32, "read as two float4");

__device__ __forceinline__ AngleParam load_angle(const AngleParam* p) {
  const float4 lo = __ldg(reinterpret_cast<const float4*>(p));
  const float4 hi = __ldg(reinterpret_cast<const float4*>(p) + 1);
  AngleParam q;
  q.A = lo.x; q.B = lo.y; q.C = lo.z; q.w = lo.w;
  q.by_rows = __float_as_int(hi.x); q.inv_a = hi.y; q.bins = __float_as_int(hi.z); q.pad = 0;
  return q;
}

__device__ __forceinline__ float sample_u(const AngleParam& q, float d, float t) {
  return fmaf(q.A, d, fmaf(q.B, t, q.C));
}

// Integer nearest to x (ties to even) for |x| < 2^22, as float and int, by
// adding and subtracting 1.5 * 2^23 (two float additions; floorf and the
// conversion run at a quarter of their rate).  With x = u - 1/2 it is floor(u),
// or u - 1 for some integer u, where the weights 0 and 1 then name the same
// pixel.
__device__ __forceinline__ float round_near(float x, int* i) {
  const float m = x + 12582912.f;
  *i = __float_as_int(m) - 0x4B400000;
  return m - 12582912.f;
}

template <int NB> struct Vec;
template <> struct Vec<1> { float v[1]; };
template <> struct __align__(8) Vec<2> { float v[2]; };
template <> struct __align__(16) Vec<4> { float v[4]; };

// ---------------------------------------------------------------- forward
// What bounds it: the wait for the staged pixels and two barriers per staging, at two to
// four CTAs per SM (8 images of 512 x 512, 60 angles: issue 57 %, shared memory 39 % of
// its rate).  Reading the image through L1 instead, one ray per thread, cost a gather
// of up to 32 lines per load at the angles sampled by columns; staging T rows (or,
// transposed, T columns) of the pixels that the CTA's rays cross makes both kinds of
// angle the same, interleaving NB images shares the position and the weights between
// them, and two neighbouring angles share one staging.  Measured at 8 images of
// 512 x 512, 180 angles, 725 bins: 1402 us with one thread per ray, 338 us so (one
// image: 239 and 121 us).
//
// With one or two images per CTA it waits for the staged pixels instead: a thread takes
// its share of a staging in batches of up to FWD_WORDS loads, and launches of fewer CTAs
// than SMs take one angle per CTA.  600 x 600, 60 angles, 849 bins, one and two images:
// 145 and 170 us with one thread per ray, 213 and 216 us without either, 112 and 143 us
// so; one image of 700 x 700, 180 angles, 128 bins: 190, 443 and 170 us.  (Four images:
// batches of four pixels 338 -> 315 us at the size above, but 39 -> 46 us at 130 images
// of 96 x 96; not taken.)
constexpr int FWD_BINS = 256;      // bins (threads) per CTA
constexpr int FWD_ANGLES = 2;      // most angles per CTA
constexpr int FWD_ROWS = 8;        // most samples t staged at a time
constexpr size_t FWD_SMEM = 56 * 1024;   // four CTAs per SM
constexpr int FWD_WORDS = 16;      // most words a thread loads before it stores them

struct AngleGroup { int a0, na; };   // neighbouring angles of one kind

template <int NB>
__global__ void __launch_bounds__(FWD_BINS) k_ray_forward(const float* __restrict__ img,
                                                          float* __restrict__ sino,
                                                          const AngleParam* __restrict__ prm,
                                                          const AngleGroup* __restrict__ groups,
                                                          int n, int A, int D, int B, int T, int pitch) {
  extern __shared__ __align__(16) unsigned char smem[];
  Vec<NB>* S = reinterpret_cast<Vec<NB>*>(smem);     // [T][pitch]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const AngleGroup grp = groups ? groups[blockIdx.y] : AngleGroup{(int)blockIdx.y, 1};
  const int d_lo = blockIdx.x * FWD_BINS, d_hi = min(D - 1, d_lo + FWD_BINS - 1);
  const int d = d_lo + tid, b0 = blockIdx.z * NB;
  const float df = (float)min(d, d_hi);
  AngleParam q[FWD_ANGLES];
#pragma unroll
  for (int k = 0; k < FWD_ANGLES; ++k) q[k] = load_angle(prm + grp.a0 + min(k, grp.na - 1));
  const bool by_rows = q[0].by_rows != 0;
  const float* f[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) f[b] = img + (size_t)min(b0 + b, B - 1) * n * n;
  float acc[FWD_ANGLES][NB];
#pragma unroll
  for (int k = 0; k < FWD_ANGLES; ++k)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[k][b] = 0.f;

  for (int t0 = 0; t0 < n; t0 += T) {
    const int tn = min(T, n - t0);
    // pixels that the block's samples can touch: u is monotone in d and in t
    float lo = 1e30f, hi = -1e30f;
#pragma unroll
    for (int k = 0; k < FWD_ANGLES; ++k) {
      const float da = (float)(q[k].A >= 0.f ? d_lo : d_hi), db = (float)(q[k].A >= 0.f ? d_hi : d_lo);
      const float ta = (float)(q[k].B >= 0.f ? t0 : t0 + tn - 1), tb = (float)(q[k].B >= 0.f ? t0 + tn - 1 : t0);
      lo = fminf(lo, sample_u(q[k], da, ta));
      hi = fmaxf(hi, sample_u(q[k], db, tb));
    }
    if (hi < -1.f || lo > (float)n) continue;        // every sample outside (the whole CTA agrees)
    // two zero pixels on either side stand for everything outside the image
    const int k_lo = max(-2, (int)floorf(fmaxf(lo, -4.f)) - 1);
    const int k_hi = min(n + 1, (int)floorf(fminf(hi, (float)(n + 4))) + 1);
    const int width = min(k_hi - k_lo + 1, pitch);
    __syncthreads();                                 // the earlier rows have been read
    // sample row tt, pixels x0, x0 + 32, ..: pixel k of sample t is at k sk + t st.  U loads
    // per image in flight, halved while the rest of the row needs no more than that.
    auto stage = [&](int tt, int x0, int sk, int st) {
      auto batch = [&](int x, auto uc) {
        constexpr int U = decltype(uc)::value;
        const int at = (k_lo + x) * sk + (t0 + tt) * st;
        Vec<NB> v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = k_lo + x + 32 * u;
          const bool in = k >= 0 && k < n && x + 32 * u < width;
#pragma unroll
          for (int b = 0; b < NB; ++b) v[u].v[b] = in ? __ldg(f[b] + (at + 32 * u * sk)) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (x + 32 * u < width) S[tt * pitch + x + 32 * u] = v[u];
      };
      constexpr int U = FWD_WORDS / NB;
      for (int x = 0; x < width; x += 32 * U) {
        const int rest = (width - x + 31) / 32;
        if (rest > U / 2) batch(x0 + x, std::integral_constant<int, U>{});
        else if (rest > U / 4) batch(x0 + x, std::integral_constant<int, U / 2>{});
        else batch(x0 + x, std::integral_constant<int, (U > 4 ? U / 4 : 1)>{});
      }
    };
    if constexpr (NB < 4) {
      if (by_rows) {
        for (int tt = warp; tt < tn; tt += FWD_BINS / 32) stage(tt, lane, 1, n);
      } else {                                       // FWD_ROWS consecutive columns of a pixel row
        const int tt = lane & (FWD_ROWS - 1);
        if (tt < tn) stage(tt, warp * (32 / FWD_ROWS) + lane / FWD_ROWS, n, 1);
      }
    } else if (by_rows) {
      for (int tt = warp; tt < tn; tt += FWD_BINS / 32)
        for (int x = lane; x < width; x += 32) {
          const int k = k_lo + x;
          Vec<NB> v;
#pragma unroll
          for (int b = 0; b < NB; ++b)
            v.v[b] = k >= 0 && k < n ? __ldg(f[b] + (size_t)(t0 + tt) * n + k) : 0.f;
          S[tt * pitch + x] = v;
        }
    } else {
      const int tt = lane & (FWD_ROWS - 1);          // FWD_ROWS consecutive columns of a pixel row
      for (int x = warp * (32 / FWD_ROWS) + lane / FWD_ROWS; x < width; x += FWD_BINS / FWD_ROWS) {
        const int k = k_lo + x;
        Vec<NB> v;
#pragma unroll
        for (int b = 0; b < NB; ++b)
          v.v[b] = k >= 0 && k < n && tt < tn ? __ldg(f[b] + (size_t)k * n + t0 + tt) : 0.f;
        if (tt < tn) S[tt * pitch + x] = v;
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < FWD_ANGLES; ++k) {
      if (k >= grp.na) break;
      const float ua = sample_u(q[k], df, (float)t0), ub = sample_u(q[k], df, (float)(t0 + tn - 1));
      if (!__any_sync(0xffffffffu, fmaxf(ua, ub) >= -1.f && fminf(ua, ub) <= (float)n)) continue;
#pragma unroll 4
      for (int tt = 0; tt < tn; ++tt) {
        const float u = sample_u(q[k], df, (float)(t0 + tt));
        int i;
        const float w1 = u - round_near(u - 0.5f, &i), w0 = 1.f - w1;
        const Vec<NB>* s = S + tt * pitch + min(max(i - k_lo, 0), width - 2);
        const Vec<NB> v0 = s[0], v1 = s[1];
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[k][b] = fmaf(w0, v0.v[b], fmaf(w1, v1.v[b], acc[k][b]));
      }
    }
  }
  if (d > d_hi) return;
#pragma unroll
  for (int k = 0; k < FWD_ANGLES; ++k)
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (k < grp.na && b0 + b < B)
        sino[((size_t)(b0 + b) * A + grp.a0 + k) * D + d] = acc[k][b] * q[k].w;
}

// ---------------------------------------------------------------- adjoint
// Pixel (t, k) of angle a receives every bin d with |u(d, t) - k| < 1, with the
// forward's own weight, rounding included (hat_weight), so that the two are exact
// transposes.  The bins start at the one below the fractional bin of u = k - 1;
// ADJ_MARGIN covers the rounding of that bin (below 0.01 over the accepted sizes).
// What bounds it: the bins' reads through L1, shared by nothing but the four images'
// position, weights and address.  Measured as above: 1770 us with one thread per pixel
// and image (a floor and a compare per candidate bin), 527 us so; 32 images of 128 x 128
// at 30 angles: 95 and 35 us (forward 107 and 41 us).
constexpr float ADJ_MARGIN = 0.05f;
constexpr int ADJ_PIX = 2;         // pixels per thread, 8 rows apart; one where that leaves
                                   // SMs without two CTAs (16^2, 8 angles, 2000
                                   // bins: 184 -> 117 us, 158 us with one thread per pixel;
                                   // 256^2, 180 angles, one image: 121 -> 92 us)

// What the forward's sample at u gives pixel k (zero or less: nothing): 1 - (u - k) above
// it, u - (k - 1) below.  Both are 1 - |u - k| to the last bit, as u - k is exact or the
// sum rounds once, except at k = 1: for 0 < u < 1/2 u - 1 is not a float32 and would
// round twice.  EDGE: CTAs that may hold k = 1, those of the first row and column of
// the image (8 x 700^2, 90 angles: 234 us without it, 237 us so, 256 us in all CTAs; 8 x
// 512^2, 180 angles, which is one wave: 277, 296 and 301 us).
template <bool EDGE>
__device__ __forceinline__ float hat_weight(float u, float k) {
  return EDGE ? fminf(u - (k - 1.f), 1.f - (u - k)) : __saturatef(1.f - fabsf(u - k));
}

template <int NB, int PIX>
__global__ void __launch_bounds__(256) k_ray_adjoint(const float* __restrict__ sino,
                                                     float* __restrict__ img,
                                                     const AngleParam* __restrict__ prm, int n,
                                                     int A, int D, int B) {
  const int j = blockIdx.x * 32 + (threadIdx.x & 31);
  const int i0 = blockIdx.y * (8 * PIX) + (threadIdx.x >> 5), b0 = blockIdx.z * NB;
  const float* p[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) p[b] = sino + (size_t)min(b0 + b, B - 1) * A * D;
  float acc[PIX][NB];
#pragma unroll
  for (int x = 0; x < PIX; ++x)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[x][b] = 0.f;
  auto angles = [&](auto edge) {
    for (int a = 0; a < A; ++a) {
      const AngleParam q = load_angle(prm + a);
      const float first = fabsf(q.inv_a) + (ADJ_MARGIN + 0.5f);
      const int row = a * D;
#pragma unroll
      for (int x = 0; x < PIX; ++x) {
        const int i = i0 + 8 * x;
        const float t = (float)(q.by_rows ? i : j), k = (float)(q.by_rows ? j : i);
        const float base = fmaf(q.B, t, q.C);
        int lo;
        const float flo = round_near(fminf(fmaxf((k - base) * q.inv_a - first, -1e6f), 1e6f), &lo);
        float sa[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) sa[b] = 0.f;
        auto bin = [&](int m) {
          const float w = hat_weight<decltype(edge)::value>(fmaf(q.A, flo + (float)m, base), k);
          if (w > 0.f) {               // a bin outside the hat is not read into the sum
#pragma unroll
            for (int b = 0; b < NB; ++b) sa[b] = fmaf(w, __ldg(p[b] + (row + lo + m)), sa[b]);
          }
        };
        if (lo >= 0 && lo + q.bins <= D) {
          bin(0);
          bin(1);
          if (q.bins > 2) bin(2);
          for (int m = 3; m < q.bins; ++m) bin(m);
        } else {
          for (int m = max(0, -lo); m < q.bins && lo + m < D; ++m) bin(m);
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[x][b] = fmaf(sa[b], q.w, acc[x][b]);
      }
    }
  };
  if (blockIdx.x > 0 && blockIdx.y > 0) angles(std::false_type{});
  else angles(std::true_type{});
#pragma unroll
  for (int x = 0; x < PIX; ++x)
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (j < n && i0 + 8 * x < n && b0 + b < B)
        img[((size_t)(b0 + b) * n + i0 + 8 * x) * n + j] = acc[x][b];
}

// The same with the bins that a tile of 32 x 32 pixels can receive staged in shared
// memory, images interleaved: one NB-wide read per bin in place of NB gathers
// through L1 (measured as above 527 -> 277 us, 296 us with the exact weights; bound by
// issue, 79 %).  Chunks of `ac` angles, W bins each, from bin s_lo on.
constexpr int ADJ_TILE_PIX = 4;    // pixels per thread, 8 rows apart
constexpr int ADJ_CHUNK = 16;      // most angles staged at a time
constexpr size_t ADJ_SMEM = 48 * 1024;
constexpr double ADJ_TILE_BINS = 160;   // widest staging of one angle

template <int NB>
__global__ void __launch_bounds__(256) k_ray_adjoint_tile(const float* __restrict__ sino,
                                                          float* __restrict__ img,
                                                          const AngleParam* __restrict__ prm, int n,
                                                          int A, int D, int B, int W, int ac) {
  extern __shared__ __align__(16) unsigned char smem[];
  Vec<NB>* S = reinterpret_cast<Vec<NB>*>(smem);     // [ac][W]
  __shared__ int s_lo[ADJ_CHUNK];
  const int tid = threadIdx.x;
  const int j0 = blockIdx.x * 32, r0 = blockIdx.y * (8 * ADJ_TILE_PIX), b0 = blockIdx.z * NB;
  const int j = j0 + (tid & 31), i0 = r0 + (tid >> 5);
  const float* p[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) p[b] = sino + (size_t)min(b0 + b, B - 1) * A * D;
  float acc[ADJ_TILE_PIX][NB];
#pragma unroll
  for (int x = 0; x < ADJ_TILE_PIX; ++x)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[x][b] = 0.f;
  for (int a0 = 0; a0 < A; a0 += ac) {
    const int na = min(ac, A - a0);
    __syncthreads();                                 // the earlier bins have been read
    if (tid < na) {
      // smallest fractional bin over the tile's corners (it is affine in t and k)
      const AngleParam q = load_angle(prm + a0 + tid);
      const int t0 = q.by_rows ? r0 : j0, k0 = q.by_rows ? j0 : r0;
      float lo = 1e30f;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float t = (float)(t0 + (c & 1) * 31), k = (float)(k0 + (c >> 1) * 31);
        lo = fminf(lo, (k - fmaf(q.B, t, q.C)) * q.inv_a);
      }
      s_lo[tid] = (int)floorf(fminf(fmaxf(lo - fabsf(q.inv_a) - ADJ_MARGIN, -1e6f), 1e6f)) - 1;
    }
    __syncthreads();
    for (int idx = tid; idx < na * W; idx += 256) {
      const int a = idx / W, d = s_lo[a] + idx - a * W;
      Vec<NB> v;
#pragma unroll
      for (int b = 0; b < NB; ++b)
        v.v[b] = d >= 0 && d < D ? __ldg(p[b] + (size_t)(a0 + a) * D + d) : 0.f;
      S[idx] = v;
    }
    __syncthreads();
    auto angles = [&](auto edge) {
      for (int a = 0; a < na; ++a) {
        const AngleParam q = load_angle(prm + a0 + a);
        const float first = fabsf(q.inv_a) + (ADJ_MARGIN + 0.5f);
        const int lo0 = s_lo[a];
        const Vec<NB>* s = S + a * W;
#pragma unroll
        for (int x = 0; x < ADJ_TILE_PIX; ++x) {
          const int i = i0 + 8 * x;
          const float t = (float)(q.by_rows ? i : j), k = (float)(q.by_rows ? j : i);
          const float base = fmaf(q.B, t, q.C);
          int lo;
          const float flo = round_near(fminf(fmaxf((k - base) * q.inv_a - first, -1e6f), 1e6f), &lo);
          const Vec<NB>* r = s + min(max(lo - lo0, 0), W - q.bins);
          float sa[NB];
#pragma unroll
          for (int b = 0; b < NB; ++b) sa[b] = 0.f;
          auto bin = [&](int m) {
            const float w = hat_weight<decltype(edge)::value>(fmaf(q.A, flo + (float)m, base), k);
            const Vec<NB> v = r[m];
            if (w > 0.f) {               // a bin outside the hat does not enter the sum
#pragma unroll
              for (int b = 0; b < NB; ++b) sa[b] = fmaf(w, v.v[b], sa[b]);
            }
          };
          bin(0);
          bin(1);
          if (q.bins > 2) bin(2);
          for (int m = 3; m < q.bins; ++m) bin(m);
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[x][b] = fmaf(sa[b], q.w, acc[x][b]);
        }
      }
    };
    if (j0 > 0 && r0 > 0) angles(std::false_type{});
    else angles(std::true_type{});
  }
#pragma unroll
  for (int x = 0; x < ADJ_TILE_PIX; ++x)
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (j < n && i0 + 8 * x < n && b0 + b < B)
        img[((size_t)(b0 + b) * n + i0 + 8 * x) * n + j] = acc[x][b];
}

bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

}  // namespace

struct shl_ray {
  int device = 0, n = 0, A = 0, D = 0;
  AngleParam* dPrm = nullptr;
  AngleGroup* dGrp = nullptr;
  int ngrp = 0;
  double a_max = 0, b_max = 0;      // largest |A| and |B| over the angles
  double pair_max = 0;              // largest |u - u'| between the angles of a group
  double inv_max = 0, tile_max = 0; // largest 1/|A| and (1 + |B|)/|A|
  int sms = 1;
};

namespace {

// Images per CTA: the position and the weights of a sample are shared by the
// images, so as many as there are (up to four) unless the launch would then
// leave SMs without two CTAs.
int images_per_cta(int sms, long long ctas_per_image, int batch) {
  for (int nb = 4; nb > 1; nb /= 2)
    if (batch >= nb && ctas_per_image * ((batch + nb - 1) / nb) >= 2LL * sms) return nb;
  return 1;
}

template <int NB>
cudaError_t forward_nb(const shl_ray* op, const float* img, int batch, float* sino, cudaStream_t st) {
  // staged pixels per sample row: what FWD_BINS bins and T rows can reach, at
  // most the whole row with its zero pixels; odd, so that the transposed stores
  // of the column-sampled angles meet no bank twice
  int T = FWD_ROWS, pitch = 0;
  for (;; T /= 2) {
    const double reach = (FWD_BINS - 1.0) * op->a_max + (T - 1.0) * op->b_max + op->pair_max + 8.0;
    pitch = (reach < op->n + 4.0 ? (int)reach : op->n + 4) | 1;
    if ((size_t)T * pitch * sizeof(Vec<NB>) <= FWD_SMEM || T == 1) break;
  }
  const size_t smem = (size_t)T * pitch * sizeof(Vec<NB>);
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024)
    e = cudaFuncSetAttribute(k_ray_forward<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e) return e;
  dim3 grid((op->D + FWD_BINS - 1) / FWD_BINS, op->ngrp, (batch + NB - 1) / NB);
  const bool single_angles = (long long)grid.x * grid.y * grid.z < op->sms;
  if (single_angles) grid.y = op->A;
  k_ray_forward<NB><<<grid, FWD_BINS, smem, st>>>(img, sino, op->dPrm, single_angles ? nullptr : op->dGrp,
                                                  op->n, op->A, op->D, batch, T, pitch);
  return cudaGetLastError();
}

template <int NB>
cudaError_t adjoint_nb(const shl_ray* op, const float* sino, int batch, float* img, cudaStream_t st) {
  // bins a tile can receive from one angle (31 pixels along each axis, the hat's
  // width, the margins and the rounding of the first bin)
  const double reach = 31.0 * op->tile_max + 2.0 * op->inv_max + 6.0;
  const long long tiles = (op->n + 31LL) / 32 * ((op->n + 31) / 32) * ((batch + NB - 1) / NB);
  if (reach <= ADJ_TILE_BINS && tiles >= 2LL * op->sms) {
    const int W = (int)reach + 1;
    const int ac = (int)std::min<size_t>(ADJ_CHUNK, ADJ_SMEM / (W * sizeof(Vec<NB>)));
    const dim3 grid((op->n + 31) / 32, (op->n + 31) / 32, (batch + NB - 1) / NB);
    k_ray_adjoint_tile<NB><<<grid, 256, (size_t)ac * W * sizeof(Vec<NB>), st>>>(
        sino, img, op->dPrm, op->n, op->A, op->D, batch, W, ac);
    return cudaGetLastError();
  }
  dim3 grid((op->n + 31) / 32, (op->n + 8 * ADJ_PIX - 1) / (8 * ADJ_PIX), (batch + NB - 1) / NB);
  if (NB == 1 && (long long)grid.x * grid.y * grid.z < 2LL * op->sms) {   // NB > 1: never so few
    grid.y = (op->n + 7) / 8;
    k_ray_adjoint<1, 1><<<grid, 256, 0, st>>>(sino, img, op->dPrm, op->n, op->A, op->D, batch);
  } else {
    k_ray_adjoint<NB, ADJ_PIX><<<grid, 256, 0, st>>>(sino, img, op->dPrm, op->n, op->A, op->D, batch);
  }
  return cudaGetLastError();
}

}  // namespace

extern "C" {

shl_status shl_ray_create(int n, int n_angles, int n_det, int device, shl_ray** out) {
  if (!out) return shl::set_error(SHL_EINVAL, "out is NULL");
  *out = nullptr;
  if (n < 2 || n > 4096 || n_angles < 1 || n_angles > 4096 || n_det < 1 || n_det > 16384)
    return shl::set_error(SHL_EINVAL, "need 2 <= n <= 4096, 1 <= n_angles <= 4096, 1 <= n_det <= 16384");
  if (device < 0) return shl::set_error(SHL_EINVAL, "device must be >= 0");
  const double PI = 3.14159265358979323846264338327950288, S = std::sqrt(2.0);
  const double h = 2.0 / n, ds = 2.0 * S / n_det;
  std::vector<AngleParam> prm(n_angles);
  for (int a = 0; a < n_angles; ++a) {
    const double phi = PI * a / n_angles, c = std::cos(phi), s = std::sin(phi);
    AngleParam& q = prm[a];
    q = AngleParam{};
    q.by_rows = std::fabs(c) >= std::fabs(s);
    // row mode:    u = (s_d - y_t sin) / (h cos) + 1/h - 1/2
    // column mode: u = (s_d - x_t cos) / (h sin) + 1/h - 1/2
    // with s_d = -S + (d + 1/2) ds and x_t = y_t = -1 + (t + 1/2) h
    const double den = q.by_rows ? h * c : h * s, other = q.by_rows ? s : c;
    q.A = (float)(ds / den);
    q.B = (float)(-h * other / den);
    q.C = (float)((-S + 0.5 * ds + other * (1.0 - 0.5 * h)) / den + 1.0 / h - 0.5);
    q.w = (float)(h / std::fabs(q.by_rows ? c : s));
    q.inv_a = (float)(den / ds);
    q.bins = (int)std::floor(2.0 * std::fabs(den / ds) + 2.0 * ADJ_MARGIN) + 2;
  }
  // the forward's groups: two neighbouring angles share a staging when the pixels
  // they sample stay within PAIR_PIXELS of each other (u is affine in d and t, so
  // the corners bound the difference)
  constexpr double PAIR_PIXELS = 64.0;
  std::vector<AngleGroup> grp;
  double a_max = 0, b_max = 0, pair_max = 0, inv_max = 0, tile_max = 0;
  for (const AngleParam& q : prm) {
    inv_max = std::max(inv_max, (double)std::fabs(q.inv_a));
    tile_max = std::max(tile_max, (1.0 + std::fabs(q.B)) * std::fabs(q.inv_a));
    a_max = std::max(a_max, (double)std::fabs(q.A));
    b_max = std::max(b_max, (double)std::fabs(q.B));
  }
  for (int a = 0; a < n_angles;) {
    double gap = 1e30;
    if (a + 1 < n_angles && prm[a].by_rows == prm[a + 1].by_rows) {
      gap = 0;
      for (int c = 0; c < 4; ++c) {
        const double d = c & 1 ? n_det - 1.0 : 0.0, t = c & 2 ? n - 1.0 : 0.0;
        gap = std::max(gap, std::fabs(((double)prm[a].A - prm[a + 1].A) * d +
                                      ((double)prm[a].B - prm[a + 1].B) * t +
                                      ((double)prm[a].C - prm[a + 1].C)));
      }
    }
    const int na = gap <= PAIR_PIXELS ? FWD_ANGLES : 1;
    if (na > 1) pair_max = std::max(pair_max, gap);
    grp.push_back({a, na});
    a += na;
  }
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != device) cudaSetDevice(device);
  shl_ray* op = new shl_ray;
  op->device = device; op->n = n; op->A = n_angles; op->D = n_det;
  op->ngrp = (int)grp.size();
  op->a_max = a_max; op->b_max = b_max; op->pair_max = pair_max;
  op->inv_max = inv_max; op->tile_max = tile_max;
  cudaDeviceGetAttribute(&op->sms, cudaDevAttrMultiProcessorCount, device);
  cudaError_t e = cudaMalloc(&op->dPrm, sizeof(AngleParam) * n_angles);
  if (!e) e = cudaMalloc(&op->dGrp, sizeof(AngleGroup) * grp.size());
  if (!e) e = cudaMemcpy(op->dPrm, prm.data(), sizeof(AngleParam) * n_angles, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(op->dGrp, grp.data(), sizeof(AngleGroup) * grp.size(), cudaMemcpyHostToDevice);
  if (prev >= 0 && prev != device) cudaSetDevice(prev);
  if (e) {
    if (op->dPrm) cudaFree(op->dPrm);
    if (op->dGrp) cudaFree(op->dGrp);
    delete op;
    cudaGetLastError();
    return shl::set_error(e == cudaErrorMemoryAllocation ? SHL_ENOMEM : SHL_ECUDA,
                          cudaGetErrorString(e));
  }
  *out = op;
  return SHL_OK;
}

shl_status shl_ray_destroy(shl_ray* op) {
  if (!op) return SHL_OK;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != op->device) cudaSetDevice(op->device);
  cudaFree(op->dPrm);
  cudaFree(op->dGrp);
  if (prev >= 0 && prev != op->device) cudaSetDevice(prev);
  delete op;
  return SHL_OK;
}

shl_status shl_ray_query(const shl_ray* op, int* n, int* n_angles, int* n_det) {
  if (!op) return shl::set_error(SHL_EINVAL, "operator is NULL");
  if (n) *n = op->n;
  if (n_angles) *n_angles = op->A;
  if (n_det) *n_det = op->D;
  return SHL_OK;
}

shl_status shl_ray_forward(const shl_ray* op, const float* img, int batch, float* sino,
                           void* stream) {
  if (!op) return shl::set_error(SHL_EINVAL, "operator is NULL");
  if (batch < 0) return shl::set_error(SHL_EINVAL, "batch must be >= 0");
  if (batch == 0) return SHL_OK;
  if (!img || !sino || !aligned4(img) || !aligned4(sino))
    return shl::set_error(SHL_EINVAL, "img and sino must be 4-byte aligned device pointers");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != op->device) cudaSetDevice(op->device);
  cudaError_t e = cudaSuccess;
  for (int b0 = 0; b0 < batch && !e; b0 += 65535) {
    const int nb = std::min(65535, batch - b0);
    const float* x = img + (size_t)b0 * op->n * op->n;
    float* y = sino + (size_t)b0 * op->A * op->D;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (images_per_cta(op->sms, (op->D + FWD_BINS - 1LL) / FWD_BINS * op->ngrp, nb)) {
      case 4: e = forward_nb<4>(op, x, nb, y, st); break;
      case 2: e = forward_nb<2>(op, x, nb, y, st); break;
      default: e = forward_nb<1>(op, x, nb, y, st); break;
    }
  }
  if (prev >= 0 && prev != op->device) cudaSetDevice(prev);
  return e ? shl::set_error(SHL_ECUDA, cudaGetErrorString(e)) : SHL_OK;
}

shl_status shl_ray_adjoint(const shl_ray* op, const float* sino, int batch, float* img,
                           void* stream) {
  if (!op) return shl::set_error(SHL_EINVAL, "operator is NULL");
  if (batch < 0) return shl::set_error(SHL_EINVAL, "batch must be >= 0");
  if (batch == 0) return SHL_OK;
  if (!img || !sino || !aligned4(img) || !aligned4(sino))
    return shl::set_error(SHL_EINVAL, "img and sino must be 4-byte aligned device pointers");
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != op->device) cudaSetDevice(op->device);
  cudaError_t e = cudaSuccess;
  for (int b0 = 0; b0 < batch && !e; b0 += 65535) {
    const int nb = std::min(65535, batch - b0);
    const float* y = sino + (size_t)b0 * op->A * op->D;
    float* x = img + (size_t)b0 * op->n * op->n;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    switch (images_per_cta(op->sms, (op->n + 31LL) / 32 * ((op->n + 8 * ADJ_PIX - 1) / (8 * ADJ_PIX)), nb)) {
      case 4: e = adjoint_nb<4>(op, y, nb, x, st); break;
      case 2: e = adjoint_nb<2>(op, y, nb, x, st); break;
      default: e = adjoint_nb<1>(op, y, nb, x, st); break;
    }
  }
  if (prev >= 0 && prev != op->device) cudaSetDevice(prev);
  return e ? shl::set_error(SHL_ECUDA, cudaGetErrorString(e)) : SHL_OK;
}

}  // extern "C"
