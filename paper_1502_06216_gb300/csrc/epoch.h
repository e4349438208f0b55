// epoch.h -- epochs of the exchanges between blocks (strip.cuh): the words of exchange e of a
// launch that starts at `first` carry first + e, e = 1, 2, ...; the launch leaves the epoch the
// next one starts at.  Plain C++ for both sides.
#pragma once

#ifndef JKO_HD
#ifdef __CUDACC__
#define JKO_HD __host__ __device__ __forceinline__
#else
#define JKO_HD inline
#endif
#endif

namespace jko {
namespace epoch {

// Exchanges a launch can make at most: a step on strips (one epoch a pair, one for the end),
// a step of its reverse pass (two before the solve, one an iteration, one after), and the
// heat kernel on tiles (per application one for v and one between phases of `h` Clenshaw
// steps; a block sends the next exchange's words ahead).
JKO_HD unsigned of_strip(unsigned pairs) { return pairs + 2u; }
JKO_HD unsigned of_adjoint(unsigned budget) { return budget + 3u; }
JKO_HD unsigned of_heat(unsigned pairs, unsigned degree, unsigned h) {
  return pairs * 2u * ((degree + h - 1u) / h) + 1u;
}

// The epoch the next launch starts at.  After a wait that gave up other blocks may have
// published exchanges beyond this block's `last`: the next launch starts behind all that the
// launch can have published, or it would take their words for its own.
JKO_HD unsigned after(unsigned first, unsigned last, unsigned most, bool gave_up) {
  return gave_up ? first + most : last;
}

}  // namespace epoch
}  // namespace jko
