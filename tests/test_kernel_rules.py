"""The kernels' rules of sizes (csrc/rules.h), compiled by the host compiler
and checked over their whole range; no GPU."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0911_5730_gb300", "csrc")


@pytest.fixture
def run(tmp_path):
    def go(body, flags=()):
        """Compiles a program around `body` (statements that return the number
        of the first rule broken, 0 if none) and returns that number."""
        src, exe = tmp_path / "t.cpp", tmp_path / "t"
        src.write_text(body)
        subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, *flags, str(src), "-o", str(exe)], check=True)
        p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
        assert p.returncode == 0, p.stdout + p.stderr
    return go


def test_triangle_segments(run):
    """Products with a triangle of zeros, for every block size and offset: the
    segments stay within the block, follow one another, and every entry that
    may be nonzero lies in a segment that serves its row."""
    run(r"""
#include <cstdio>
#include <initializer_list>
#include "rules.h"
int main() {
    for (int R : {2, 4}) for (int b = 1; b <= 160; ++b) for (int d = 0; d <= b; ++d) for (int low = 0; low < 2; ++low) {
        const int h = (b + R - 1) / R;
        int from = 0, end[4];
        for (int s = 0; s < R; ++s) {
            end[s] = bddc::tri_segment_end(s, R, h, b, d, low);
            if (end[s] < from || end[s] > b) { printf("R %d b %d d %d low %d: segment %d [%d, %d)\n", R, b, d, low, s, from, end[s]); return 1; }
            from = end[s];
        }
        if (end[R - 1] != b) return 2;
        for (int r = 0; r < b; ++r) for (int c = 0; c < b; ++c) {
            if (low ? c > r + d : c < r - d) continue;
            int s = 0;
            while (c >= end[s]) ++s;
            if (low ? r / h < s : r / h > s) { printf("R %d b %d d %d low %d: (%d, %d) left out\n", R, b, d, low, r, c); return 3; }
        }
    }
}
""")


def test_stencil_tile_is_timed_where_it_runs(run):
    """The width at which the stencil's tiles are timed takes a tile, and no
    wider one does."""
    run(r"""
#include "rules.h"
int main() { return bddc::stencil_marches(bddc::kTileTuneK) ? 1 : !bddc::stencil_marches(bddc::kTileTuneK + 1) ? 2 : 0; }
""")


def test_fp64_dirichlet_routes(run):
    """FP64 batch Dirichlet kernels: the staged one is timed wherever it was
    not measured to lose (blocks of 8 rows with up to 2.6 substructures for an
    SM, where it is the fastest, among them), and narrow batches leave the lane
    kernel only where the streaming one was measured faster."""
    run(r"""
#include "rules.h"
using namespace bddc;
int main() {
    const int sms = 152;
    for (int nsub = 1; nsub <= 400; ++nsub) if (!fp64_staged_timed(8, nsub, sms, true)) return 1;
    for (int nsub = 1; nsub < sms; ++nsub) if (!fp64_staged_timed(16, nsub, sms, true)) return 2;
    for (int nsub = 1; nsub < 20000; ++nsub) if (!fp64_staged_timed(16, nsub, sms, false)) return 3;
    if (fp64_staged_timed(16, 169, sms, true) || fp64_staged_timed(8, 484, sms, true)) return 4;
    for (int K = 1; K <= 32; ++K) {
        if (!fp64_lane_at(K, 8, 4096, sms, true) || !fp64_lane_at(K, 16, 1024, sms, false) || !fp64_lane_at(K, 16, 100, sms, true)) return 5;
        if (fp64_lane_at(K, 16, 1024, sms, true) != (K > 16)) return 6;
    }
}
""")


def test_direction_buffers_of_a_resumed_column(run):
    """A column that stops at a step, sits out any number of steps and resumes
    finds the direction that it wrote last."""
    run(r"""
#include "rules.h"
using namespace bddc;
int main() {
    for (int stop = 0; stop < 8; ++stop) for (int missed = 0; missed < 8; ++missed) {
        int buf[2] = {-1, -2}, last = -1, step = 0;
        for (; step <= stop; ++step) {
            if (step > 0 && buf[direction_read(step)] != last) return 1;
            last = step;
            buf[direction_written(step)] = step;
        }
        step += missed;
        const int from = direction_written(last), to = direction_read(step);
        if (from != to) buf[to] = buf[from];
        if (buf[direction_read(step)] != stop) return 2;
        if (direction_read(step) == direction_written(step)) return 3;
    }
}
""")


def test_ring_drains_what_is_in_flight(run):
    """A ring whose copy number `late` does not land within a wait: the thread
    waits and issues no more, and the drain waits for every copy in flight, the
    late one among them."""
    run(r"""
#include <initializer_list>
#include "rules.h"
using namespace bddc;
int main() {
    for (int n : {2, 3, 4, 6}) for (int units = 1; units <= 14; ++units) for (int late = -1; late < units; ++late) {
        RingSlots R;
        unsigned done[8] = {0};                 // completions of each barrier
        bool flight[8] = {false};
        int copy[8], polls = 0;
        bool slow = true;                       // the late copy lands after the first wait for it
        auto wait_for = [&](int s, unsigned parity) {
            ++polls;
            if ((done[s] & 1u) != parity) return true;     // that phase has completed: no time passes
            if (flight[s] && copy[s] == late && slow) { slow = false; return false; }
            if (flight[s]) { ++done[s]; flight[s] = false; }
            return (done[s] & 1u) != parity;
        };
        auto issue = [&](int u) { flight[u % n] = true; copy[u % n] = u; R.issued(u % n); };
        for (int u = 0; u < n && u < units; ++u) issue(u);
        for (int u = 0; u < units; ++u) {
            const int before = polls;
            const bool had = R.ok;
            R.wait(u % n, wait_for);
            if (!had && polls != before) return 1;
            if (R.ok != (late < 0 || u < late)) return 2;
            if (R.ok && u + n < units) issue(u + n);
        }
        R.drain(n, wait_for);
        for (int s = 0; s < n; ++s) if (flight[s]) return 3;
    }
}
""")


def test_semidefinite_pivots(run):
    """Cholesky factors of Gram matrices of half rank: L L^T is the matrix up to
    n dropped pivots, each worth the root of its threshold."""
    run(r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "rules.h"
int main() {
    for (int n : {8, 16, 31}) {
        const int r = n / 2;
        std::mt19937_64 gen(1);
        for (int t = 0; t < 20000; ++t) {
            std::vector<double> B(n * r), G(n * n), A;
            for (auto &v : B) v = (double)(gen() >> 11) * 0x1p-52 - 1.0;
            double mx = 0.0;
            for (int i = 0; i < n; ++i)
                for (int j = 0; j < n; ++j) {
                    double s = 0.0;
                    for (int k = 0; k < r; ++k) s += B[i * r + k] * B[j * r + k];
                    G[i * n + j] = s;
                    if (i == j) mx = std::max(mx, s);
                }
            A = G;
            for (int j = 0; j < n; ++j) {
                const double d = A[j * n + j], l = bddc::semi_pivot(d, G[j * n + j], n) ? std::sqrt(d) : 0.0;
                A[j * n + j] = l;
                for (int i = j + 1; i < n; ++i) A[i * n + j] = l > 0.0 ? A[i * n + j] / l : 0.0;
                for (int i = j + 1; i < n; ++i)
                    for (int k = j + 1; k <= i; ++k) A[i * n + k] -= A[i * n + j] * A[k * n + j];
            }
            for (int i = 0; i < n; ++i)
                for (int j = 0; j <= i; ++j) {
                    double s = 0.0;
                    for (int k = 0; k <= j; ++k) s += A[i * n + k] * A[j * n + k];
                    if (!(std::fabs(s - G[i * n + j]) <= n * std::sqrt(n * 0x1p-52) * mx)) {
                        printf("n %d matrix %d: off by %g of %g\n", n, t, s - G[i * n + j], mx);
                        return 1;
                    }
                }
        }
    }
}
""", ["-O2"])
