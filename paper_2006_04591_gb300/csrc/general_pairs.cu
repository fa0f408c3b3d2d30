// general_pairs.cu - instances of general_pairs.cuh.  Compiled once per part of the
// pair list (SHL_PART = 0..3) for the row passes and once for the column passes
// (SHL_PART = 4..7).
#include "general_pairs.cuh"
#include "general_pairs_list.h"

#define SHL_CAT2(a, b) a##b
#define SHL_CAT(a, b) SHL_CAT2(a, b)

namespace shl {
namespace gen {

#if SHL_PART < 4
#if SHL_PART == 0
#define SHL_LIST SHL_PAIRS_0
#elif SHL_PART == 1
#define SHL_LIST SHL_PAIRS_1
#elif SHL_PART == 2
#define SHL_LIST SHL_PAIRS_2
#else
#define SHL_LIST SHL_PAIRS_3
#endif
cudaError_t SHL_CAT(pair_rows_part, SHL_PART)(int kind, const PairRowArgs& a, cudaStream_t st) {
#define X(RA, RB, BL) \
  if (a.p.A == RA && a.p.B == RB && (a.p.bluestein != 0) == BL) return pair_rows<RA, RB, BL>(kind, a, st);
  SHL_LIST(X)
#undef X
  return cudaErrorInvalidValue;
}
#else
#if SHL_PART == 4
#define SHL_LIST SHL_PAIRS_0
#elif SHL_PART == 5
#define SHL_LIST SHL_PAIRS_1
#elif SHL_PART == 6
#define SHL_LIST SHL_PAIRS_2
#else
#define SHL_LIST SHL_PAIRS_3
#endif
cudaError_t SHL_CAT(pair_cols_part, SHL_PART)(int planes, const PairColArgs& a, cudaStream_t st) {
#define X(RA, RB, BL)                                                     \
  if (a.p.A == RA && a.p.B == RB && (a.p.bluestein != 0) == BL)           \
    return pair_cols<RA, RB, BL>(a.kind == PCOL_REC, planes, a, st);
  SHL_LIST(X)
#undef X
  return cudaErrorInvalidValue;
}
#endif

}  // namespace gen
}  // namespace shl
