// Fixed-point copies of the FP64 links and clover blocks, for the FP64 stencil on the integer pipes.
//
// GB300 has two FP64 lanes per SM but 64 lanes of 32-bit integer multiply-add with a 64-bit
// accumulator, so a product of two 59-bit fixed-point numbers as three 32 x 32 -> 64-bit products
// costs 3/64 of a cycle per lane against 1/2 for one FP64 multiply-add.
//
// A number is kept as two limbs, value = h 2^30 + l with |l| <= 2^29. A matrix is scaled by a power of two
// so that the absolute real and imaginary parts of every row (and, for a link, of every column, the rows
// of its adjoint) sum to less than 2^59.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace tmamg {

constexpr int FX_BITS = 59;          // row sums of a scaled matrix are below 2^FX_BITS
constexpr int FX_BAD = 1 << 20;      // exponent of a matrix with a non-finite or out-of-range entry
constexpr int FX_ZERO = -(1 << 20);  // exponent of a zero matrix, or of a vector with no entry seen yet

struct FixedOp {
  int4* U = nullptr;   // [4 nu][9][V]: limbs (re.h, re.l, im.h, im.l) of the entries times 2^(59 - nU)
  int* nU = nullptr;   // [4 nu][V]: scaling exponents
  int2* C = nullptr;   // [2 chi][36][V]: limbs of the packed clover entries times 2^(59 - nC)
  int* nC = nullptr;   // [V]: scaling exponent of both chiralities
};

}  // namespace tmamg
