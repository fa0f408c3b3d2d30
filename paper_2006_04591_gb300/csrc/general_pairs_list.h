// general_pairs_list.h - the pairs (A, B) that general_pairs.cuh is compiled for,
// in four parts (one translation unit each per pass kind).
//
// Direct: every product of two radices of {8, 10, 12, 15, 16, 20, 24, 25, 30, 32}
// (the register DFTs of at most 32 points that split into 2-, 3-, 4-, 5- and
// 8-point ones, from the length where two stages pay) in its most equal split,
// the larger radix first.  Bluestein (last argument true): the powers of two from 128
// to 1024, the smaller radix first (the radix that ends the second transform, whose
// outputs the reconstruction sums).
#pragma once

#define SHL_PAIRS_0(X) \
  X(12, 8, false) X(10, 10, false) X(16, 12, false) X(20, 10, false) X(20, 15, false) \
  X(20, 20, false) X(24, 20, false) X(32, 16, false) X(30, 24, false) X(8, 16, true) \
  X(32, 32, true)
#define SHL_PAIRS_1(X) \
  X(12, 12, false) X(16, 10, false) X(16, 15, false) X(25, 10, false) X(24, 16, false) \
  X(25, 20, false) X(32, 20, false) X(32, 24, false) X(30, 30, false) X(16, 16, true)
#define SHL_PAIRS_2(X) \
  X(8, 8, false) X(16, 8, false) X(15, 10, false) X(16, 16, false) X(24, 12, false) \
  X(25, 15, false) X(30, 15, false) X(25, 25, false) X(30, 25, false) X(32, 32, false)
#define SHL_PAIRS_3(X) \
  X(10, 8, false) X(12, 10, false) X(15, 12, false) X(15, 15, false) X(20, 16, false) \
  X(24, 15, false) X(24, 24, false) X(25, 24, false) X(32, 25, false) X(32, 30, false) \
  X(16, 32, true)
#define SHL_PAIRS_ALL(X) SHL_PAIRS_0(X) SHL_PAIRS_1(X) SHL_PAIRS_2(X) SHL_PAIRS_3(X)
