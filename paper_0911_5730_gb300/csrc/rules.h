// rules.h - rules of the kernels that depend on sizes only, in plain C++ for
// the host and the device: a host compiler checks them over their whole range.
#pragma once

#ifdef __CUDACC__
#define BDDC_HD __host__ __device__
#else
#define BDDC_HD
#endif

namespace bddc {

// A product over the columns [0, b) of a block with a triangle of zeros, by
// threads of R rows k, k + h, ... (h = ceil(b / R)), is taken in R segments of
// columns: entry (row, c) is zero for c > row + d (low) or c < row - d, so
// segment `seg` serves the rows from number seg on (low) or up to it, and this
// is its end.  Within [0, b] for every b: R h exceeds small b (R = 4: 3 h > b
// for b = 1, 2 and 5).
BDDC_HD constexpr int tri_segment_end(int seg, int R, int h, int b, int d, bool low) {
    const int e = seg + 1 == R ? b : low ? (seg + 1) * h + d : (seg + 1) * h - d;
    return e < 0 ? 0 : e > b ? b : e;
}

// The batched stencil: up to kMarchMinK right-hand sides take a node tile, whose
// shape is timed at that width, the widest one that uses it; more march.
constexpr int kMarchMinK = 24, kTileTuneK = kMarchMinK;
BDDC_HD constexpr bool stencil_marches(int K) { return K > kMarchMinK; }

}  // namespace bddc
