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

// The FP64 batch Dirichlet kernels on levels of uniform blocks of bp rows where
// the lane-per-right-hand-side kernel fits; us for both corrections (m = 15
// blocks of 16 rows, 7 of 8 rows; 152 SMs; the streaming kernel and the staged
// one take the same within 5 % for fewer columns unless given):
//   blocks of 16 rows        169 subs.  256   576   1024
//     staged                       678   684  1373   2396
//     streaming, 17 to 32          544   556   848   1456
//     streaming, up to 16          543   545   596    809
//     lane                         755   758   776   1175
//   blocks of 8 rows         169 subs.  256   400   484   625   784  1024   4096  16384
//     staged                        95    98   132   166   204   243   307   1017   3986
//     streaming                    177   180   183   186   189   202   223    761   2664
//     lane                         136   136   137   141   206   214   216    677   2526
// Whether the staged kernel is timed beside the others: not where it lost
// wherever it was measured, which keeps the first use of a large problem short.
BDDC_HD constexpr bool fp64_staged_timed(int bp, int nsub, int sms, bool stream) {
    return bp == 16 ? !(stream && nsub >= sms) : nsub < 3 * sms;
}
// Whether K columns take the lane kernel where it was the fastest for 32: it
// costs the same for any K, and so does the streaming kernel with blocks of 8
// rows; with blocks of 16 rows that one is the faster up to 16 columns.
BDDC_HD constexpr bool fp64_lane_at(int K, int bp, int nsub, int sms, bool stream) {
    return K > 16 || !(bp == 16 && nsub >= sms && stream);
}

// The two direction buffers of a batch: lockstep step `step` reads one and
// writes the other, for the columns that iterate.  A column that sat out steps
// may find its latest direction in the one that its next step would write.
BDDC_HD constexpr int direction_read(int step) { return step & 1; }
BDDC_HD constexpr int direction_written(int step) { return 1 - (step & 1); }

// One thread's view of a ring of shared-memory slots filled by bulk copies, a
// barrier each (barrier s completes once per copy into slot s, with alternating
// parity).  wait_for(s, parity) polls barrier s a bounded number of times.
struct RingSlots {
    unsigned parity = 0;    // bit s: parity of the next completion of slot s
    unsigned pending = 0;   // bit s: a copy that this thread issued is in flight
    bool ok = true;         // false once a wait gave up: the thread waits and issues no more

    BDDC_HD void issued(int s) { pending |= 1u << s; }
    template <class F> BDDC_HD void wait(int s, F &&wait_for) {
        if (ok) {
            ok = wait_for(s, (parity >> s) & 1u);
            if (ok) pending &= ~(1u << s);
        }
        parity ^= (unsigned)ok << s;    // (a slot whose copy did not land keeps its parity for the drain)
    }
    // before the block exits: the copies in flight land
    template <class F> BDDC_HD void drain(int slots, F &&wait_for) const {
        for (int s = 0; s < slots; ++s)
            if ((pending >> s) & 1u) wait_for(s, (parity >> s) & 1u);
    }
};

// Whether a Cholesky pivot d of an n x n matrix that may be semidefinite to
// rounding counts as positive, d0 being the diagonal entry it came from: what
// is left of a dependent column is rounding of either sign, and a positive one
// divided by its own root spoils every later column (in 0.1 % of random Gram
// matrices of half rank, by more than the matrix itself).  Leaving out a pivot
// this small changes the matrix by at most its root, relatively.
BDDC_HD constexpr bool semi_pivot(double d, double d0, int n) { return d > n * 2.220446049250313e-16 * d0; }

}  // namespace bddc
