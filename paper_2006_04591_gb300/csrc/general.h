// general.h - the transform for any image size (1..4096 per side) and for
// complex Hermitian filter spectra: declarations shared by api.cpp and
// general.cu.
//
// The power-of-two kernels of fast.cu keep real, even spectra in transposed
// half-spectrum planes.  This path keeps row-major half-spectrum planes
// [N][M/2+1] (columns kx = 0..M/2 of the natural-order spectrum; the rest
// follows from Hermitian symmetry, which holds for real images and Hermitian
// filters), complex filter values where the bank has them, and computes
// every line DFT in shared memory with a mixed-radix Stockham FFT (all prime
// factors <= 61), or with Bluestein's chirp-z algorithm (a larger prime
// factor: the length-L DFT becomes a circular convolution of length P = the
// power of two >= 2L - 1).  Lengths that are products of two small radices, and
// lengths up to 512 with a prime factor above 19 (by Bluestein), run on the two-stage
// register kernels of general_pairs.cuh.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <vector>

namespace shl {
namespace gen {

constexpr int MAX_LEN = 4096;     // longest side
constexpr int MAX_STAGES = 16;
constexpr int MAX_DIRECT_PRIME = 61;

// Lines of the two-stage register kernels (general_pairs.cuh): length L = A B, or
// Bluestein's P = A B >= 2 L - 1.  A = 0: no pair, the kernels of general.cu.
struct PairPlan {
  int L, A, B, bluestein;
  const float2* ab;          // [(m - 1) A + k] = exp(-2 pi i m k / P), m < B, k < A
  const float2* ba;          // [(m - 1) B + k], m < A, k < B
  const float2* chirp;       // [L] exp(-i pi n^2 / L) (Bluestein)
  const float2* kern;        // [P] DFT_P(h) / P over the transform's mean gain (pair_gain),
                             // h[m] = conj chirp[|m|]
};

// Forward DFT of length L, X[k] = sum_n x[n] exp(-2 pi i n k / L); the
// inverse is taken as conj(DFT(conj(x))).  Pointers refer to device tables.
struct LinePlan {
  int L;                     // transform length
  int P;                     // working length (L, or Bluestein's power of two)
  int bluestein;             // 1: chirp-z through a length-P FFT
  int nst;                   // Stockham stages of the length-P FFT
  int radix[MAX_STAGES];     // their radices (product P)
  const float2* tw;          // [P]  exp(-2 pi i q / P)
  const float2* chirp;       // [L]  exp(-i pi n^2 / L)              (Bluestein)
  const float2* kern;        // [P]  DFT_P(h) / P, h[m] = conj chirp[|m|] (Bluestein)
  PairPlan pair;
};

// Host-side tables of one length, computed in float64 and rounded; offsets
// (in float2 units) of tw / chirp / kern inside `data`.
struct LineTables {
  LinePlan plan{};
  std::vector<float2> data;
  size_t off_tw = 0, off_chirp = 0, off_kern = 0, off_ab = 0, off_ba = 0;
};
// Builds the plan and tables of length L (1 <= L <= MAX_LEN).
LineTables make_line_tables(int L);
// Points the plan at the tables after `data` was copied to `dev`.
void place_line_tables(LineTables* t, const float2* dev);

// Real-row input of the forward row pass.
enum RowIn : int { RIN_F32 = 0, RIN_BF16 = 1, RIN_MASKED = 2 };

// Row passes (rows of length M, plan pm) between real planes [nplanes][N][M]
// and half-spectrum planes [nplanes][N][M/2+1].
//   rows_fwd:    real rows (thresholded on read when thresh != null, one
//                threshold per plane; masked: mask ? f_masked : f_est) ->
//                row DFTs, columns 0..M/2 -> out.
//   rows_inv:    Hermitian row spectra (from their halves) -> inverse row
//                DFT -> real part * scale -> float32 or bfloat16 out.
//   rows_shrink: in place: inverse row DFT -> real part * scale -> zero
//                |c| < thresh[plane] -> forward row DFT.
cudaError_t launch_rows_fwd(const LinePlan& pm, RowIn mode, const void* in, const uint8_t* mask,
                            const float* fest, const float* thresh, float2* out, int N,
                            int nplanes, cudaStream_t st);
cudaError_t launch_rows_inv(const LinePlan& pm, const float2* in, void* out, bool bf16,
                            float scale, int N, int nplanes, cudaStream_t st);
cudaError_t launch_rows_shrink(const LinePlan& pm, float2* z, const float* thresh, float scale,
                               int N, int nplanes, cudaStream_t st);

// The same passes on the two-stage register kernels (plans with pair.A > 0).
struct PairRowArgs {
  PairPlan p;                // rows: length M
  const void* in;            // forward: [nplanes][N][M] reals (f_masked when masked)
  const uint8_t* mask;       // forward, masked
  const float* fest;         // forward, masked
  const float* thresh;       // [nplanes] or null (forward), [nplanes] (shrink)
  float2* z;                 // half-spectrum planes [nplanes][N][M/2+1]
  void* out;                 // inverse: float32 / bfloat16 [nplanes][N][M]
  float scale;               // inverse, shrink
  int N, nplanes;
  int mode;                  // forward: RowIn; inverse: 1 = bfloat16 out
};
enum PairColKind : int { PCOL_FWD, PCOL_DEC, PCOL_REC, PCOL_FIN };
struct PairColArgs {
  PairPlan p;                // columns: length N
  const float2* X;           // PCOL_DEC: image spectra [B][N][W]
  float2* T;                 // PCOL_DEC out / PCOL_REC, PCOL_FIN in: staging [S][N][W]
  float2* A;                 // PCOL_FWD planes (in place) / PCOL_FIN accumulators [B][N][W]
  const void* G;             // float [K][N][W] or float2 [K][N][W]
  const float* invW;         // [N][W] or null
  int W, K, s0, S, cplx;     // W = M/2 + 1 stored columns
  int groups;                // PCOL_REC, PCOL_FIN: subband groups per image
  int kind;
};
// kind: 0 forward, 1 inverse, 2 shrink.
cudaError_t launch_pair_rows(int kind, const PairRowArgs& a, cudaStream_t st);
cudaError_t launch_pair_cols(int planes, const PairColArgs& a, cudaStream_t st);

// Column passes (columns of length N, plan pn) on half-spectrum planes of
// W = M/2 + 1 columns.
//   cols_fwd: in-place forward column DFT of nplanes planes.
//   cols_dec: T[s - s0] = inverse column DFT of G_i * X_b [* 1/W] for the
//             subbands s = s0 .. s0+S-1 (b = s / K, i = s % K).
//   cols_rec: for each image b with subbands in s0 .. s0+S-1, split into
//             groups of consecutive subbands (one CTA per column block,
//             image and group): the group's sum_i conj(G_i) * column
//             DFT(T[s - s0]) in order of i, written over its first staging
//             plane; then acc = (partial sum in A_b unless the chunk holds
//             the image's first subband) + the group sums in group order; on
//             the image's last subband acc is multiplied by 1/W (when invW)
//             and inverse column transformed into A_b, else stored there as
//             the new partial sum.  T is overwritten.
// G is float [K][N][W] (real spectra) or float2 [K][N][W] (complex), 1/W
// float [N][W]: the columns kx = 0..M/2 of the natural-order tables.
cudaError_t launch_cols_fwd(const LinePlan& pn, float2* X, int W, int nplanes, cudaStream_t st);
cudaError_t launch_cols_dec(const LinePlan& pn, const float2* X, float2* T, const void* G,
                            bool cplx, const float* invW, int W, int K, int s0, int S,
                            cudaStream_t st);
cudaError_t launch_cols_rec(const LinePlan& pn, float2* T, float2* A, const void* G,
                            bool cplx, const float* invW, int W, int K, int s0, int S,
                            cudaStream_t st);

}  // namespace gen
}  // namespace shl
