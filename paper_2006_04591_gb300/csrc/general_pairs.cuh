// general_pairs.cuh - row and column passes of the general path (general.cu) for
// lines of P = A B elements, A, B <= 32: Stockham's autosort FFT in two stages,
//   out[q Ns + k] = sum_{m<R} in[k + m P/R] w^(m (k + q Ns)), w = exp(-2 pi i / P).
// One thread holds one butterfly in registers.  The first stage takes its inputs
// straight from global memory and the last gives its outputs straight back; in
// between a line goes through shared memory once, behind one barrier.
//
// What bounded these passes with radices up to 8 and every stage in shared
// memory (general.cu, still used for the lengths without a pair) were the four or
// five exchanges with a barrier each and the strided gathers of their twiddles
// through L1.  Both radices are compile-time constants: one kernel with a switch
// over the radices spilled and ran at half the speed.  Measured before and after
// (K = 49, float32, decomposition and reconstruction): 16 x 480 x 640 5375 -> 1806 us
// (column pass of the reconstruction 1864 -> 395, of the decomposition 1124 -> 417,
// row passes 1166 -> 452 and 1127 -> 517), 16 x 500^2 4345 -> 1503 us, 4 x 509^2
// (Bluestein, P = 1024) 3992 -> 1262 us; with packed additions and the group sums below
// 1620, 1420 and 1152 us.  With K = 17, 16 x 222 x 301 (Bluestein, P = 512 and 1024)
// 1575 -> 599 us.
// At 480 x 640 the passes now run at 35-55 % of the DRAM rate of the planes and
// coefficients that they move; what is left is latency at 18 to 24 warps per SM.
//
// Lengths up to 512 with a prime factor above 19 (find_pair) go through Bluestein's
// chirp-z identity
// n k = (n^2 + k^2 - (k - n)^2)/2 with a pair P >= 2L - 1:
//   X[k] = c[k] sum_n (x[n] c[n]) conj(c[k - n]),  c[n] = exp(-i pi n^2 / L),
// a circular convolution of length P evaluated with two length-P FFTs against
// the precomputed DFT_P of the chirp kernel.  The second FFT runs the radices in
// reverse order, so its first stage needs exactly the elements a thread holds
// after the last stage of the first (j + q P/R both times): the kernel multiply
// sits between two register DFTs without an exchange.  The fused shrink pass
// joins its inverse and its forward DFT the same way.
//
// The inverse DFT is conj(DFT(conj x)) (exact in floating point).  The forward
// row pass runs the radices in the order of the shrink pass's second transform,
// so that the fused and the separate passes give equal bits.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "dft_small.cuh"
#include "general.h"

namespace shl {
namespace gen {
namespace {

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 conj_mul(float2 a, float2 b) {   // conj(a) * b
  return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// After a first stage of radix R output q of butterfly j is kept at j pitch(R) + q:
// an odd pitch, so that the lanes of a warp meet no bank twice.  The second stage's
// input m of butterfly k then sits at k + m pitch(R).
constexpr int pitch_of(int R) { return R | 1; }

// Shared memory of one line through the orders (A, B) and (B, A).
template <int A, int B>
struct PairT {
  static constexpr int P = A * B;
  static constexpr int TL = A > B ? A : B;                       // threads per line
  static constexpr int LINE = B * pitch_of(A) > A * pitch_of(B) ? B * pitch_of(A) : A * pitch_of(B);
  static constexpr int ROW_LINES = TL <= 8 ? 32 : 256 / TL;      // lines of a row CTA
  static constexpr int ROW_THREADS = (ROW_LINES * TL + 31) / 32 * 32;
  static constexpr int COLS = 8;                                 // columns of a column CTA
  static constexpr int COL_THREADS = COLS * TL;
  // CTAs per SM that the register allocation aims at (about 640 threads, 100
  // registers each; the reconstruction, which also keeps its sums, 512)
  static constexpr int ROW_CTAS = 640 / ROW_THREADS;
  static constexpr int COL_CTAS = 640 / COL_THREADS > 8 ? 8 : 640 / COL_THREADS;
  static_assert(COL_THREADS >= 16, "a thread for each subband group");
  static constexpr int REC_CTAS = 512 / COL_THREADS > 8 ? 8 : 512 / COL_THREADS;
};

template <int R, int STEP>
__device__ __forceinline__ void put_first(const float2 (&v)[R], float2* line, int j) {
#pragma unroll
  for (int q = 0; q < R; ++q) line[(j * pitch_of(R) + q) * STEP] = v[q];
}
// Second stage of order (R0, R), butterfly k < R0: inputs and twiddles
// tw[(m - 1) R0 + k] = w^(m k).
template <int R0, int R, int STEP>
__device__ __forceinline__ void get_second(float2 (&v)[R], const float2* line, const float2* tw, int k) {
#pragma unroll
  for (int m = 0; m < R; ++m) v[m] = line[(k + m * pitch_of(R0)) * STEP];
#pragma unroll
  for (int m = 1; m < R; ++m) v[m] = cmul(v[m], __ldg(tw + (m - 1) * R0 + k));
}

// Bluestein: elements j + m S of the input times the chirp, zero from L on; of the
// result, chirp * conj; between the transforms conj(v * kernel).
template <int R>
__device__ __forceinline__ void chirp_in(float2 (&v)[R], const PairPlan& p, int j, int S) {
#pragma unroll
  for (int m = 0; m < R; ++m) {
    const int e = j + m * S;
    const float2 w = __ldg(p.chirp + min(e, p.L - 1));
    v[m] = e < p.L ? mul2(v[m], w) : make_float2(0.f, 0.f);
  }
}
template <int R>
__device__ __forceinline__ void chirp_out(float2 (&v)[R], const PairPlan& p, int j, int S) {
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = mul2(__ldg(p.chirp + min(j + q * S, p.L - 1)), conjf2(v[q]));
}
template <int R>
__device__ __forceinline__ void kern_turn(float2 (&v)[R], const PairPlan& p, int j, int S) {
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = conjf2(mul2(v[q], __ldg(p.kern + j + q * S)));
}

// ------------------------------------------------------------------ rows
// Two real rows share one complex line DFT: rows 2m and 2m+1 of a plane go
// into the real and imaginary parts (the last row of an odd-height plane is
// paired with zeros).  Forward: z = x_a + i x_b, Z = DFT(z), X_a[k] =
// (Z[k] + conj Z[-k])/2, X_b[k] = (Z[k] - conj Z[-k])/(2i).  Inverse (real
// part wanted): IDFT(T_a + i T_b) = x_a + i x_b for Hermitian T_a, T_b.  The
// pairing depends only on (plane, row), never on how planes are chunked.
//
// Loads past L (Bluestein) read element L - 1, a missing second row reads the
// first: every load is unconditional, and all of a butterfly's are in flight.
struct RowLine {
  size_t ra;                 // global index of the line's first row
  bool two;                  // it has a second row
  float tau;                 // threshold of its plane
};

template <int R>
__device__ __forceinline__ void load_real_rows(float2 (&v)[R], const PairRowArgs& a, const RowLine& ln,
                                               int j, int S) {
  const int L = a.p.L;
  const size_t r0 = ln.ra * L;
  const int rb = ln.two ? L : 0;
  if (a.mode == RIN_F32) {
    const float* x = static_cast<const float*>(a.in) + r0;
#pragma unroll
    for (int m = 0; m < R; ++m) {
      const int e = min(j + m * S, L - 1);
      v[m] = make_float2(__ldcs(x + e), __ldcs(x + rb + e));
    }
  } else if (a.mode == RIN_BF16) {
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(a.in) + r0;
#pragma unroll
    for (int m = 0; m < R; ++m) {
      const int e = min(j + m * S, L - 1);
      v[m] = make_float2(__bfloat162float(x[e]), __bfloat162float(x[rb + e]));
    }
  } else {
    const float *x = static_cast<const float*>(a.in) + r0, *f = a.fest + r0;
    const uint8_t* mk = a.mask + r0;
#pragma unroll
    for (int m = 0; m < R; ++m) {
      const int e = min(j + m * S, L - 1);
      const float xa = x[e], fa = f[e], xb = x[rb + e], fb = f[rb + e];
      v[m] = make_float2(mk[e] ? xa : fa, mk[rb + e] ? xb : fb);
    }
  }
  if (a.thresh) {                                      // ties kept
#pragma unroll
    for (int m = 0; m < R; ++m) {
      if (fabsf(v[m].x) < ln.tau) v[m].x = 0.f;
      if (fabsf(v[m].y) < ln.tau) v[m].y = 0.f;
    }
  }
  if (!ln.two) {
#pragma unroll
    for (int m = 0; m < R; ++m) v[m].y = 0.f;
  }
}

// Hermitian rows from their stored half: T[e] for e < Mh, conj T[M - e] above; the
// DC and (even M) Nyquist bins keep their real parts only.  v = conj(T_a + i T_b).
template <int R>
__device__ __forceinline__ void load_half_rows(float2 (&v)[R], const PairRowArgs& a, const RowLine& ln,
                                               int j, int S) {
  const int M = a.p.L, Mh = M / 2 + 1;
  const float2* za = a.z + ln.ra * Mh;
  const float2* zb = za + (ln.two ? Mh : 0);
  float2 t[R];
#pragma unroll
  for (int m = 0; m < R; ++m) {
    const int e = min(j + m * S, M - 1), eh = e >= Mh ? M - e : e;
    v[m] = za[eh];
    t[m] = zb[eh];
  }
#pragma unroll
  for (int m = 0; m < R; ++m) {
    const int e = j + m * S;
    float ay = v[m].y, bx = t[m].x, by = t[m].y;
    if (e >= Mh) { ay = -ay; by = -by; }
    if (e == 0 || 2 * e == M) { ay = 0.f; by = 0.f; }
    if (!ln.two) { bx = 0.f; by = 0.f; }
    v[m] = make_float2(v[m].x - by, -(ay + bx));
  }
}

template <int R>
__device__ __forceinline__ void store_real_rows(const float2 (&v)[R], const PairRowArgs& a,
                                                const RowLine& ln, int j, int S) {
  const int L = a.p.L;
  if (a.mode) {
    __nv_bfloat16* x = static_cast<__nv_bfloat16*>(a.out) + ln.ra * L;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int e = j + q * S;
      if (e < L) {
        x[e] = __float2bfloat16_rn(v[q].x * a.scale);
        if (ln.two) x[L + e] = __float2bfloat16_rn(-v[q].y * a.scale);
      }
    }
  } else {
    float* x = static_cast<float*>(a.out) + ln.ra * L;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int e = j + q * S;
      if (e < L) {
        __stcs(x + e, v[q].x * a.scale);
        if (ln.two) __stcs(x + L + e, -v[q].y * a.scale);
      }
    }
  }
}

template <int R>
__device__ __forceinline__ void threshold(float2 (&v)[R], float scale, float tau) {
#pragma unroll
  for (int q = 0; q < R; ++q) {
    float ca = v[q].x * scale, cb = -v[q].y * scale;   // x_a, x_b
    if (fabsf(ca) < tau) ca = 0.f;
    if (fabsf(cb) < tau) cb = 0.f;
    v[q] = make_float2(ca, cb);
  }
}

// A line has one buffer: between reading it and writing it again stands a barrier
// (a second buffer would save it, and halve the CTAs on an SM).
//
// One line of a forward transform whose first-stage values v (radix R0) are in
// registers -> Z in natural order in the buffer; b is free on entry.
template <int R0, int R1, bool BL>
__device__ __forceinline__ void forward_rest(float2 (&v)[R0], const PairPlan& p, float2* b, int j,
                                             bool act, const float2* t01, const float2* t10) {
  const bool act0 = act && j < R1, act1 = act && j < R0;
  if (act0) {
    dft_n<R0>(v);
    put_first<R0, 1>(v, b, j);
  }
  __syncthreads();
  float2 u[R1];
  if (act1) {
    get_second<R0, R1, 1>(u, b, t01, j);
    dft_n<R1>(u);
    if constexpr (BL) {
      kern_turn(u, p, j, R0);
      dft_n<R1>(u);
    }
  }
  __syncthreads();
  if (act1) {
    if constexpr (BL) {
      put_first<R1, 1>(u, b, j);
    } else {
#pragma unroll
      for (int q = 0; q < R1; ++q) b[j + q * R0] = u[q];
    }
  }
  __syncthreads();
  if constexpr (BL) {
    if (act0) {
      get_second<R1, R0, 1>(v, b, t10, j);
      dft_n<R0>(v);
      chirp_out(v, p, j, R1);
    }
    __syncthreads();
    if (act0) {
#pragma unroll
      for (int q = 0; q < R0; ++q) b[j + q * R1] = v[q];
    }
    __syncthreads();
  }
}

enum RowKind : int { ROW_FWD = 0, ROW_INV = 1, ROW_SHRINK = 2 };

template <int A, int B, bool BL, int KIND>
__global__ void __launch_bounds__(PairT<A, B>::ROW_THREADS, (PairT<A, B>::ROW_CTAS)) k_pair_rows(const __grid_constant__ PairRowArgs a) {
  using T = PairT<A, B>;
  extern __shared__ __align__(16) float2 sm[];
  const PairPlan& p = a.p;
  const int M = p.L, Mh = M / 2 + 1, Np = (a.N + 1) / 2;   // lines per plane
  const int l = threadIdx.x / T::TL, j = threadIdx.x % T::TL;
  const int L0 = blockIdx.x * T::ROW_LINES;
  const int lines = min(T::ROW_LINES, Np * a.nplanes - L0);
  const bool act = l < lines;
  RowLine ln;
  {
    const int lg = L0 + min(l, lines - 1), pl = lg / Np, m = lg - pl * Np;
    ln.ra = (size_t)pl * a.N + 2 * m;
    ln.two = 2 * m + 1 < a.N;
    ln.tau = a.thresh ? __ldg(a.thresh + pl) : 0.f;
  }
  constexpr int LB = T::LINE;
  float2* b = sm + (size_t)min(l, T::ROW_LINES - 1) * LB;
  // order (A, B): twiddles ab; (B, A): ba
  if constexpr (KIND == ROW_FWD) {
    if constexpr (!BL) {                           // order (B, A): the shrink pass's second transform
      float2 v[B];
      if (act && j < A) load_real_rows(v, a, ln, j, A);
      forward_rest<B, A, false>(v, p, b, j, act, p.ba, p.ab);
    } else {
      float2 v[A];
      if (act && j < B) {
        load_real_rows(v, a, ln, j, B);
        chirp_in(v, p, j, B);
      }
      forward_rest<A, B, true>(v, p, b, j, act, p.ab, p.ba);
    }
  } else {
    float2 v[A], u[B];
    if (act && j < B) {
      load_half_rows(v, a, ln, j, B);
      if constexpr (BL) chirp_in(v, p, j, B);
      dft_n<A>(v);
      put_first<A, 1>(v, b, j);
    }
    __syncthreads();
    if (act && j < A) {
      get_second<A, B, 1>(u, b, p.ab, j);
      dft_n<B>(u);
      if constexpr (BL) {
        kern_turn(u, p, j, A);
        dft_n<B>(u);
      } else if constexpr (KIND == ROW_INV) {
        store_real_rows(u, a, ln, j, A);
      } else {
        threshold(u, a.scale, ln.tau);
      }
    }
    if constexpr (!BL && KIND == ROW_INV) return;
    __syncthreads();
    if constexpr (!BL) {
      forward_rest<B, A, false>(u, p, b, j, act, p.ba, p.ab);
    } else {
      if (act && j < A) put_first<B, 1>(u, b, j);
      __syncthreads();
      if (act && j < B) {
        get_second<B, A, 1>(v, b, p.ba, j);
        dft_n<A>(v);
        chirp_out(v, p, j, B);
        if constexpr (KIND == ROW_INV) {
          store_real_rows(v, a, ln, j, B);
        } else {
          threshold(v, a.scale, ln.tau);
          chirp_in(v, p, j, B);
        }
      }
      if constexpr (KIND == ROW_INV) return;
      __syncthreads();
      forward_rest<A, B, true>(v, p, b, j, act, p.ab, p.ba);
    }
  }
  if constexpr (KIND != ROW_INV) {
    // half spectra of both rows; forward_rest has ended with a barrier
    if (act) {
      float2 *za = a.z + ln.ra * Mh, *zb = za + Mh;
      for (int e = j; e < Mh; e += T::TL) {
        const float2 zk = b[e], zn = b[e ? M - e : 0];
        za[e] = make_float2(0.5f * (zk.x + zn.x), 0.5f * (zk.y - zn.y));
        if (ln.two) zb[e] = make_float2(0.5f * (zk.y + zn.y), 0.5f * (zn.x - zk.x));
      }
    }
  }
}

// --------------------------------------------------------------- columns
// A column CTA owns 8 adjacent columns of one plane: a row's 8 values are one
// 64-byte run in global and in shared memory.  Loads past row N (Bluestein) and
// past column W read the last one.
template <bool BL>
struct ColAt {               // offset of element j + m S of column `col`
  int e0, es, j, S, W, last;
  __device__ __forceinline__ ColAt(const PairColArgs& a, int j_, int S_, int col)
      : j(j_), S(S_), W(a.W), last(a.p.L - 1) {
    const int c = min(col, a.W - 1);
    e0 = BL ? c : j * W + c;
    es = S * W;
  }
  __device__ __forceinline__ int operator()(int m) const {
    return BL ? min(j + m * S, last) * W + e0 : e0 + m * es;
  }
};
template <int R, class At>
__device__ __forceinline__ void scale_by(float2 (&v)[R], const float* g, const At& at) {
#pragma unroll
  for (int m = 0; m < R; ++m) v[m] = cscale(v[m], __ldg(g + at(m)));
}
template <int R>
__device__ __forceinline__ void conj_all(float2 (&v)[R]) {
#pragma unroll
  for (int m = 0; m < R; ++m) v[m].y = -v[m].y;
}

// Subbands [sa, sb) of image b in the chunk s0 .. s0+S-1, and their group g
// of `groups`: [lo, hi) (possibly empty).
struct PairRange {
  int b, lo, hi;
  bool first, last;
};
__device__ __forceinline__ PairRange pair_range(const PairColArgs& a, int img, int g) {
  PairRange r;
  r.b = a.s0 / a.K + img;
  const int sa = max(a.s0, r.b * a.K), sb = min(a.s0 + a.S, (r.b + 1) * a.K);
  r.first = sa == r.b * a.K;
  r.last = sb == (r.b + 1) * a.K;
  r.lo = sa + (g * (sb - sa)) / a.groups;
  r.hi = sa + ((g + 1) * (sb - sa)) / a.groups;
  return r;
}

constexpr int REC_GROUPS = 16;   // most subband groups per image (rec_groups)

template <int A, int B, bool BL, int KIND>
__global__ void __launch_bounds__(PairT<A, B>::COL_THREADS, (PairT<A, B>::COL_CTAS)) k_pair_cols(const __grid_constant__ PairColArgs a) {
  using T = PairT<A, B>;
  constexpr int C = T::COLS;
  constexpr bool inv = KIND != PCOL_FWD;
  extern __shared__ __align__(16) float2 sm[];
  const PairPlan& p = a.p;
  const int N = p.L, W = a.W, c = threadIdx.x % C, j = threadIdx.x / C;
  const int col = blockIdx.x * C + c;
  const size_t plane = (size_t)N * W;
  float2* b = sm + c;
  float2* out;
  float2 v[A];
  const ColAt<BL> at(a, j, B, col);
  if constexpr (KIND == PCOL_FIN) {
    // the image's partial sum (unless the chunk holds its first subband), then the
    // groups' partials in group order
    const PairRange r0 = pair_range(a, blockIdx.y, 0);
    out = a.A + (size_t)r0.b * plane;
    if (!r0.last) {
      for (int y = j; y < N && col < W; y += T::TL) {
        const size_t e = (size_t)y * W + col;
        float2 s = r0.first ? make_float2(0.f, 0.f) : out[e];
        for (int g = 0; g < a.groups; ++g) {
          const PairRange r = pair_range(a, blockIdx.y, g);
          if (r.lo < r.hi) s = cadd(s, a.T[(size_t)(r.lo - a.s0) * plane + e]);
        }
        out[e] = s;
      }
      return;
    }
    // Bound by latency: few CTAs (columns / 8 per image) add up to 16 planes.  Four
    // elements of four groups are loaded at a time, in group order, and not one group
    // after the other with its range's division in between: the reconstruction's
    // column passes of 3 x 480 x 640 149.8 -> 111.1 us, of 1 x 500^2 78.8 -> 56.5 us,
    // of 16 x 480 x 640 393 -> 379 us.
    __shared__ int s_lo[REC_GROUPS];           // the groups' planes, -1: empty
    if (threadIdx.x < a.groups) {
      const PairRange r = pair_range(a, blockIdx.y, threadIdx.x);
      s_lo[threadIdx.x] = r.lo < r.hi ? r.lo - a.s0 : -1;
    }
    __syncthreads();
    if (j < B) {
#pragma unroll
      for (int m = 0; m < A; ++m) v[m] = r0.first ? make_float2(0.f, 0.f) : out[at(m)];
#pragma unroll
      for (int m0 = 0; m0 < A; m0 += 4) {
        for (int g = 0; g < a.groups; g += 4) {
          float2 q[4][4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int lo = g + k < a.groups ? s_lo[g + k] : -1;
            const float2* s = a.T + (size_t)max(lo, 0) * plane;
#pragma unroll
            for (int m = 0; m < 4; ++m)
              q[k][m] = lo >= 0 && m0 + m < A ? s[at(m0 + m)] : make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int m = 0; m < 4; ++m)
              if (m0 + m < A) v[m0 + m] = caddp(v[m0 + m], q[k][m]);
        }
      }
      if (a.invW) scale_by(v, a.invW, at);
    }
  } else if constexpr (KIND == PCOL_DEC) {
    const int s = a.s0 + blockIdx.y, b = s / a.K, i = s - b * a.K;
    out = a.T + (size_t)blockIdx.y * plane;
    if (j < B) {
      // eight elements at a time: the loads of all A at once (spectrum, filter and
      // weight) spill
      const float2* x = a.X + (size_t)b * plane;
      const float2* gc = static_cast<const float2*>(a.G) + (size_t)i * plane;
      const float* gr = static_cast<const float*>(a.G) + (size_t)i * plane;
#pragma unroll
      for (int m0 = 0; m0 < A; m0 += 8) {
        constexpr int E = 8;
#pragma unroll
        for (int m = m0; m < m0 + E && m < A; ++m) v[m] = x[at(m)];
        if (a.cplx) {
#pragma unroll
          for (int m = m0; m < m0 + E && m < A; ++m) v[m] = mul2(__ldg(gc + at(m)), v[m]);
        } else {
#pragma unroll
          for (int m = m0; m < m0 + E && m < A; ++m) v[m] = cscale(v[m], __ldg(gr + at(m)));
        }
        if (a.invW) {
#pragma unroll
          for (int m = m0; m < m0 + E && m < A; ++m) v[m] = cscale(v[m], __ldg(a.invW + at(m)));
        }
        asm volatile("" ::: "memory");
      }
    }
  } else {
    out = a.A + (size_t)blockIdx.y * plane;
    if (j < B) {
#pragma unroll
      for (int m = 0; m < A; ++m) v[m] = out[at(m)];
    }
  }
  if (j < B) {
    if (inv) conj_all(v);
    if constexpr (BL) chirp_in(v, p, j, B);
    dft_n<A>(v);
    put_first<A, C>(v, b, j);
  }
  __syncthreads();
  float2 u[B];
  if (j < A) {
    get_second<A, B, C>(u, b, p.ab, j);
    dft_n<B>(u);
    if constexpr (BL) {
      kern_turn(u, p, j, A);
      dft_n<B>(u);
    } else {
      if (inv) conj_all(u);
#pragma unroll
      for (int q = 0; q < B; ++q)
        if (col < W) out[(j + q * A) * W + col] = u[q];
    }
  }
  if constexpr (BL) {
    __syncthreads();
    if (j < A) put_first<B, C>(u, b, j);
    __syncthreads();
    if (j < B) {
      get_second<B, A, C>(v, b, p.ba, j);
      dft_n<A>(v);
      chirp_out(v, p, j, B);
      if (inv) conj_all(v);
#pragma unroll
      for (int q = 0; q < A; ++q)
        if (col < W && j + q * B < N) out[(j + q * B) * W + col] = v[q];
    }
  }
}

// Group blockIdx.z of image blockIdx.y: its subbands' column DFTs times conj(G_i),
// summed in order of i in registers, written over the columns of the group's first
// staging plane (which only this CTA reads).  Direct lines alternate between two
// line buffers, so that one barrier per subband is enough.
template <int A, int B, bool BL>
__global__ void __launch_bounds__(PairT<A, B>::COL_THREADS, (BL ? 1 : PairT<A, B>::REC_CTAS)) k_pair_rec(const __grid_constant__ PairColArgs a) {
  using T = PairT<A, B>;
  constexpr int C = T::COLS, RL = BL ? A : B, SL = BL ? B : A;   // last radix, its butterflies
  extern __shared__ __align__(16) float2 sm[];
  const PairPlan& p = a.p;
  const PairRange r = pair_range(a, blockIdx.y, blockIdx.z);
  if (r.lo >= r.hi) return;
  const int N = p.L, W = a.W, c = threadIdx.x % C, j = threadIdx.x / C;
  const int col = blockIdx.x * C + c;
  const size_t plane = (size_t)N * W;
  float2 acc[RL];
#pragma unroll
  for (int q = 0; q < RL; ++q) acc[q] = make_float2(0.f, 0.f);
  for (int s = r.lo; s < r.hi; ++s) {
    float2* b0 = sm + c + (!BL && ((s - r.lo) & 1) ? T::LINE * C : 0);
    const int i = s - r.b * a.K;
    float2 w[RL];
    if (j < B) {
      float2 v[A];
      const ColAt<BL> at(a, j, B, col);
      const float2* x = a.T + (size_t)(s - a.s0) * plane;
#pragma unroll
      for (int m = 0; m < A; ++m) v[m] = x[at(m)];
      if constexpr (BL) chirp_in(v, p, j, B);
      dft_n<A>(v);
      put_first<A, C>(v, b0, j);
    }
    __syncthreads();
    if constexpr (BL) {
      float2 u[B];
      if (j < A) {
        get_second<A, B, C>(u, b0, p.ab, j);
        dft_n<B>(u);
        kern_turn(u, p, j, A);
        dft_n<B>(u);
      }
      __syncthreads();
      if (j < A) put_first<B, C>(u, b0, j);
      __syncthreads();
      if (j < SL) {
        get_second<B, A, C>(w, b0, p.ba, j);
        dft_n<A>(w);
        chirp_out(w, p, j, B);
      }
      __syncthreads();
    } else {
      if (j < SL) {
        get_second<A, B, C>(w, b0, p.ab, j);
        dft_n<B>(w);
      }
    }
    if (j < SL) {
      const ColAt<BL> at(a, j, SL, col);
      if (a.cplx) {
        const float2* g = static_cast<const float2*>(a.G) + (size_t)i * plane;
#pragma unroll
        for (int q = 0; q < RL; ++q) acc[q] = cadd(acc[q], conj_mul(__ldg(g + at(q)), w[q]));
      } else {
        const float* g = static_cast<const float*>(a.G) + (size_t)i * plane;
#pragma unroll
        for (int q = 0; q < RL; ++q) {
          const float f = __ldg(g + at(q));
          acc[q].x = fmaf(f, w[q].x, acc[q].x);
          acc[q].y = fmaf(f, w[q].y, acc[q].y);
        }
      }
    }
  }
  float2* part = a.T + (size_t)(r.lo - a.s0) * plane;
  if (j < SL && col < W) {
#pragma unroll
    for (int q = 0; q < RL; ++q)
      if (j + q * SL < N) part[(size_t)(j + q * SL) * W + col] = acc[q];
  }
}

template <typename Args>
cudaError_t pair_launch(void (*k)(Args), dim3 grid, int threads, size_t smem, cudaStream_t st,
                        const Args& a) {
  if (grid.x == 0 || grid.y == 0) return cudaSuccess;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
  }
  k<<<grid, threads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int A, int B, bool BL>
cudaError_t pair_rows(int kind, const PairRowArgs& a, cudaStream_t st) {
  using T = PairT<A, B>;
  const long long lines = (long long)((a.N + 1) / 2) * a.nplanes;
  const dim3 grid((unsigned)((lines + T::ROW_LINES - 1) / T::ROW_LINES));
  const size_t buf = sizeof(float2) * (size_t)T::ROW_LINES * T::LINE;
  if (kind == ROW_INV)
    return pair_launch(k_pair_rows<A, B, BL, ROW_INV>, grid, T::ROW_THREADS, buf, st, a);
  if (kind == ROW_FWD)
    return pair_launch(k_pair_rows<A, B, BL, ROW_FWD>, grid, T::ROW_THREADS, buf, st, a);
  return pair_launch(k_pair_rows<A, B, BL, ROW_SHRINK>, grid, T::ROW_THREADS, buf, st, a);
}

template <int A, int B, bool BL>
cudaError_t pair_cols(bool rec, int planes, const PairColArgs& a0, cudaStream_t st) {
  using T = PairT<A, B>;
  PairColArgs a = a0;
  const size_t buf = sizeof(float2) * (size_t)T::COLS * T::LINE;
  const dim3 grid((a.W + T::COLS - 1) / T::COLS, planes, rec ? a.groups : 1);
  if (rec) return pair_launch(k_pair_rec<A, B, BL>, grid, T::COL_THREADS, BL ? buf : 2 * buf, st, a);
  if (a.kind == PCOL_DEC) return pair_launch(k_pair_cols<A, B, BL, PCOL_DEC>, grid, T::COL_THREADS, buf, st, a);
  if (a.kind == PCOL_FWD) return pair_launch(k_pair_cols<A, B, BL, PCOL_FWD>, grid, T::COL_THREADS, buf, st, a);
  return pair_launch(k_pair_cols<A, B, BL, PCOL_FIN>, grid, T::COL_THREADS, buf, st, a);
}

}  // namespace
}  // namespace gen
}  // namespace shl
