// batch_kernels.cu - Algorithm 1 (eqs. 4-11) and the PCG recurrences for a
// batch of K <= 32 right-hand sides solved in lockstep.
//
// Every global vector of the batch is stored interleaved, entry (g, k) at
// g * K + k, so that the K values of one DOF are contiguous.  The operator
// blocks of a substructure are staged once in shared memory and used for all
// K right-hand sides, so operator bytes are read once per batch instead of
// once per right-hand side.  The Dirichlet kernel gives a block of four warps
// to one substructure (eight right-hand sides per warp, four lanes per
// right-hand side); the substructure-correction and averaging kernels give a
// warp to a substructure and a lane to a right-hand side.
//
// The PCG scalars are per right-hand side; a right-hand side that has
// converged keeps its state while the others iterate.
#include "internal.h"
#include "device_util.cuh"
#include "rules.h"

#include <algorithm>
#include <cstdlib>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

namespace bddc {

namespace {

constexpr int kChunksB = 4;   // bulk copies per factor

// The batch kernels are launched in plain stream order: with programmatic
// serialisation a batched solve of the 512 x 512 channel workload ran 47%
// slower (FP32, 32 right-hand sides), whereas the single right-hand-side
// kernels gain from it.  They still call pdl_wait(), which then returns at once.
template <class... KArgs, class... Args>
inline void launch_plain(void (*k)(KArgs...), int grid, int block, size_t smem, cudaStream_t s,
                         Args... args) {
    launch_k(false, k, grid, block, smem, s, args...);
}

// N consecutive storage elements (N * sizeof(T) bytes aligned) into accumulators.
template <class T, class ACC, int N>
__device__ __forceinline__ void load_vec(const T *src, ACC (&v)[N]) {
    if constexpr (N == 1) {
        v[0] = ld<T, ACC>(src);
    } else if constexpr (std::is_same<T, double>::value) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const double2 q = reinterpret_cast<const double2 *>(src)[i];
            v[2 * i] = q.x; v[2 * i + 1] = q.y;
        }
    } else if constexpr (std::is_same<T, float>::value) {
        if constexpr (N == 2) {
            const float2 q = *reinterpret_cast<const float2 *>(src);
            v[0] = q.x; v[1] = q.y;
        } else {
#pragma unroll
            for (int i = 0; i < N / 4; ++i) {
                const float4 q = reinterpret_cast<const float4 *>(src)[i];
                v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
            }
        }
    } else {
        unsigned u[N / 2];
        if constexpr (N == 2) {
            u[0] = *reinterpret_cast<const unsigned *>(src);
        } else if constexpr (N == 4) {
            const uint2 q = *reinterpret_cast<const uint2 *>(src);
            u[0] = q.x; u[1] = q.y;
        } else {
#pragma unroll
            for (int i = 0; i < N / 8; ++i) {
                const uint4 q = reinterpret_cast<const uint4 *>(src)[i];
                u[4 * i] = q.x; u[4 * i + 1] = q.y; u[4 * i + 2] = q.z; u[4 * i + 3] = q.w;
            }
        }
#pragma unroll
        for (int h = 0; h < N / 2; ++h) {
            v[2 * h] = __uint_as_float(u[h] << 16);
            v[2 * h + 1] = __uint_as_float(u[h] & 0xffff0000u);
        }
    }
}


// The batched Dirichlet kernel gives one block of LR warps to one
// substructure, LR lanes to a right-hand side: warp w takes right-hand sides
// (32/LR) w .. (32/LR)(w+1) - 1; lane LR g + h holds rows h*RPL .. h*RPL +
// RPL - 1 (RPL = BP / LR) of every block of right-hand side (32/LR) w + g.
// The block's warps only meet at the gathers and the coupling terms; the
// sweeps run without block barriers.  LR = 8 for BP >= 16 (eight warps per
// substructure), 4 for BP = 8.
constexpr int kMaxDW = 8;
template <int BP> __host__ __device__ constexpr int lanes_per_rhs() { return BP >= 16 ? 8 : 4; }

template <class T, class ACC, int BP> struct DirSmemB {
    static size_t bytes(const DevLevel &L) {
        return al16(sizeof(T) * (size_t)L.max_fac) + al16(sizeof(ACC) * (size_t)L.max_m * BP * 32) +
               al16(sizeof(ACC) * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32) + al16((size_t)L.max_irec) +
               al16(sizeof(ACC) * (size_t)(L.max_coo > 0 ? L.max_coo : 1)) + al16(8 * 32 * kMaxDW + 16) +
               8 * (kChunksB + 1) + 16;
    }
};

// (4)-(5) [pre] or (10)-(11) [post] for K right-hand sides.  Block factor
// storage as in the single right-hand-side kernel: per block j, [Linv_j |
// L_{j,j-1}] of BP x BP each, element (r, c) at c * BP + (r ^ c), Linv_j lower
// triangular (zeros stored above the diagonal).
template <class T, class ACC, int BP, bool POST>
__global__ void __launch_bounds__(32 * lanes_per_rhs<BP>()) k_dir_b(DevLevel L, BatchLevel B, const double *r,
                                                                    double *z, const int *skip, RzBatch rz) {
    constexpr int LR = lanes_per_rhs<BP>(), kDW = LR;
    constexpr int BB = BP * BP, RPL = BP / LR;
    extern __shared__ __align__(16) unsigned char smem_b[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int sub = blockIdx.x;
    const int K = B.K;
    const bool act = lane < K;
    unsigned char *p = smem_b;
    T *fac = reinterpret_cast<T *>(p);      p += al16(sizeof(T) * (size_t)L.max_fac);
    ACC *xs = reinterpret_cast<ACC *>(p);   p += al16(sizeof(ACC) * (size_t)L.max_m * BP * 32);
    ACC *vG = reinterpret_cast<ACC *>(p);   p += al16(sizeof(ACC) * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32);
    unsigned char *rec = p;                 p += al16((size_t)L.max_irec);
    ACC *cvs = reinterpret_cast<ACC *>(p);  p += al16(sizeof(ACC) * (size_t)(L.max_coo > 0 ? L.max_coo : 1));
    double *red = reinterpret_cast<double *>(p);   // [kDW][32] partials and a flag word
    int *flag = reinterpret_cast<int *>(red + 32 * kDW);
    p += al16(8 * 32 * kMaxDW + 16);
    unsigned long long *bars = reinterpret_cast<unsigned long long *>(p);   // kChunksB factor + 1 record

    const int nI = L.nI[sub], nG = L.nG[sub], m = L.nblk[sub];
    const int ncoo = L.ncoo[sub], nown = L.nown[sub];
    const T *F = Ops<T>::get(L).dir + L.offF[sub];
    const int nch = m < kChunksB ? m : kChunksB;
    const IRecLayout lay(nI, nG, ncoo, nown);
    if (tid == 0) {
        for (int c = 0; c < nch; ++c) mbar_init(&bars[c]);
        mbar_init(&bars[kChunksB]);
    }
    __syncthreads();
    if (tid == 0) {
        // the index record first: the gathers wait for it, the sweeps for the factor
        mbar_expect(&bars[kChunksB], (unsigned)lay.bytes);
        bulk_copy(rec, L.irec + L.irecOff[sub], (unsigned)lay.bytes, &bars[kChunksB]);
        for (int c = 0; c < nch; ++c) {
            const int b0 = c * m / nch, b1 = (c + 1) * m / nch;
            const unsigned bytes = (unsigned)((size_t)(b1 - b0) * 2 * BB * sizeof(T));
            mbar_expect(&bars[c], bytes);
            bulk_copy(fac + (size_t)b0 * 2 * BB, F + (size_t)b0 * 2 * BB, bytes, &bars[c]);
        }
    }
    const int *gI = reinterpret_cast<const int *>(rec + lay.iI);
    const int *gGi = reinterpret_cast<const int *>(rec + lay.iG);
    const int *gP = reinterpret_cast<const int *>(rec + lay.pr);
    const double *gC = reinterpret_cast<const double *>(rec + lay.cv);
    const int *gO = reinterpret_cast<const int *>(rec + lay.ow);
    pdl_wait();
    pdl_trigger();
    auto drain = [&](int from) {   // bounded: copies in flight land before the block exits
        if (tid == 0) {
            for (int c = from; c < nch; ++c) mbar_wait(&bars[c], 0);
            mbar_wait(&bars[kChunksB], 0);
        }
    };
    if (skip && *skip) { drain(0); return; }
    const bool rec_ok = mbar_wait(&bars[kChunksB], 0);
    if (!__syncthreads_and(rec_ok)) {
        if (tid == 0) atomicExch(L.err, 1);
        drain(0);
        return;
    }
    // right-hand sides (lane = right-hand side), sixteen row loads in flight per warp
    constexpr int kG = 16;
    for (int i0 = warp * kG; i0 < m * BP; i0 += kDW * kG) {
        double v[kG];
#pragma unroll
        for (int u = 0; u < kG; ++u) {
            const int i = i0 + u;
            v[u] = (i < nI && act) ? r[(int64_t)gI[i] * K + lane] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kG; ++u)
            if (i0 + u < m * BP) xs[(i0 + u) * 32 + lane] = from_f64<ACC>(v[u]);
    }
    for (int e = tid; e < ncoo; e += 32 * kDW) cvs[e] = from_f64<ACC>(gC[e]);
    if (POST) {
        for (int q0 = warp * kG; q0 < nG; q0 += kDW * kG) {
            double v[kG];
#pragma unroll
            for (int u = 0; u < kG; ++u)
                v[u] = (q0 + u < nG && act) ? B.uB[(int64_t)gGi[q0 + u] * K + lane] : 0.0;
#pragma unroll
            for (int u = 0; u < kG; ++u)
                if (q0 + u < nG) vG[(q0 + u) * 32 + lane] = from_f64<ACC>(v[u]);
        }
        __syncthreads();
        // interior right-hand side r_I - A_{I Gamma} u_B; warp w applies, in
        // entry order, the entries of the interior rows il = w (mod kDW), so
        // the sums do not depend on scheduling
        for (int e = 0; e < ncoo; ++e) {
            const int pr = gP[e];
            if (((pr & 0xffff) & (kDW - 1)) != warp) continue;
            xs[(pr & 0xffff) * 32 + lane] -= cvs[e] * vG[(pr >> 16) * 32 + lane];
        }
    } else {
        for (int q = warp; q < nG; q += kDW) {
            vG[q * 32 + lane] = 0;
            if (act) B.uB[(int64_t)gGi[q] * K + lane] = 0.0;   // consumed by the previous post-correction
        }
    }
    __syncthreads();

    const int g = lane / LR, h = lane % LR;
    const int kc = warp * (32 / LR) + g;   // column of xs: the right-hand side of this lane
    const int rb = h * RPL;                // first row of this lane within a block
    const int src0 = lane & ~(LR - 1);     // lane holding rows 0 .. RPL-1 of the same right-hand side
    int cw = 0;
    bool ok = true;
    ACC xp[RPL];
#pragma unroll
    for (int q = 0; q < RPL; ++q) xp[q] = 0;
    for (int j = 0; j < m; ++j) {
        while (cw < nch && cw * m / nch <= j) {
            if (!mbar_wait(&bars[cw], 0)) { ok = false; break; }
            ++cw;
        }
        if (!ok) break;
        const T *Li = fac + (size_t)j * 2 * BB;
        const T *Ls = Li + BB;
        ACC t[RPL];
#pragma unroll
        for (int q = 0; q < RPL; ++q) t[q] = xs[(j * BP + rb + q) * 32 + kc];
        if (j > 0) {
            // t -= L_{j,j-1} x_{j-1}: the whole x_{j-1} of this right-hand side by shuffles
            ACC xf[BP];
#pragma unroll
            for (int c = 0; c < BP; ++c) xf[c] = __shfl_sync(0xffffffffu, xp[c % RPL], src0 | (c / RPL));
#pragma unroll
            for (int c = 0; c < BP; ++c) {
                ACC cv[RPL];
                load_vec<T, ACC, RPL>(Ls + c * BP + (rb ^ (c & ~(RPL - 1))), cv);
#pragma unroll
                for (int q = 0; q < RPL; ++q) t[q ^ (c & (RPL - 1))] -= cv[q] * xf[c];
            }
        }
        ACC tf[BP];
#pragma unroll
        for (int c = 0; c < BP; ++c) tf[c] = __shfl_sync(0xffffffffu, t[c % RPL], src0 | (c / RPL));
#pragma unroll
        for (int q = 0; q < RPL; ++q) xp[q] = 0;
#pragma unroll
        for (int c = 0; c < BP; ++c) {
            ACC cv[RPL];
            load_vec<T, ACC, RPL>(Li + c * BP + (rb ^ (c & ~(RPL - 1))), cv);
#pragma unroll
            for (int q = 0; q < RPL; ++q) xp[q ^ (c & (RPL - 1))] += cv[q] * tf[c];
        }
#pragma unroll
        for (int q = 0; q < RPL; ++q) xs[(j * BP + rb + q) * 32 + kc] = xp[q];
    }
    if (ok) {
        // backward sweep: z_j = Linv_j^T (y_j - L_{j+1,j}^T z_{j+1}).  Each lane
        // forms the column partials of its own rows for all BP output rows and
        // the LR lanes of a right-hand side reduce-scatter them: in the round
        // with partner h ^ st a lane keeps the half of the rows whose bit st of
        // the lane index it carries, so it ends with its own RPL rows.
        auto reduce_scatter = [&](ACC (&part)[BP], ACC (&out)[RPL]) {
            ACC buf[BP];
#pragma unroll
            for (int i = 0; i < BP; ++i) buf[i] = part[i];
            int len = BP;
#pragma unroll
            for (int st = LR / 2; st >= 1; st /= 2) {
                len /= 2;
                const bool hi = (h & st) != 0;
#pragma unroll
                for (int i = 0; i < BP / 2; ++i) {
                    if (i < len) {
                        const ACC send = hi ? buf[i] : buf[len + i];
                        const ACC keep = hi ? buf[len + i] : buf[i];
                        buf[i] = keep + __shfl_xor_sync(0xffffffffu, send, st);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < RPL; ++i) out[i] = buf[i];
        };
        ACC zn[RPL];
#pragma unroll
        for (int q = 0; q < RPL; ++q) zn[q] = 0;
        for (int j = m - 1; j >= 0; --j) {
            const T *Li = fac + (size_t)j * 2 * BB;
            ACC t[RPL];
#pragma unroll
            for (int q = 0; q < RPL; ++q) t[q] = xs[(j * BP + rb + q) * 32 + kc];
            if (j < m - 1) {
                const T *Ls1 = fac + (size_t)(j + 1) * 2 * BB + BB;
                ACC part[BP];
#pragma unroll
                for (int rr = 0; rr < BP; ++rr) {
                    // L_{j+1,j}(c, rr) for this lane's c = rb + q' at rr * BP + (c ^ rr)
                    ACC v[RPL];
                    load_vec<T, ACC, RPL>(Ls1 + rr * BP + (rb ^ (rr & ~(RPL - 1))), v);
                    ACC a = 0;
#pragma unroll
                    for (int q = 0; q < RPL; ++q) a += v[q] * zn[q ^ (rr & (RPL - 1))];
                    part[rr] = a;
                }
                ACC red[RPL];
                reduce_scatter(part, red);
#pragma unroll
                for (int q = 0; q < RPL; ++q) t[q] -= red[q];
            }
            ACC part[BP];
#pragma unroll
            for (int rr = 0; rr < BP; ++rr) {
                ACC v[RPL];
                load_vec<T, ACC, RPL>(Li + rr * BP + (rb ^ (rr & ~(RPL - 1))), v);
                ACC a = 0;
#pragma unroll
                for (int q = 0; q < RPL; ++q) a += v[q] * t[q ^ (rr & (RPL - 1))];
                part[rr] = a;
            }
            reduce_scatter(part, zn);
#pragma unroll
            for (int q = 0; q < RPL; ++q) xs[(j * BP + rb + q) * 32 + kc] = zn[q];
        }
    }
    if (!__syncthreads_and(ok)) {
        if (tid == 0) atomicExch(L.err, 1);
        drain(0);
        return;
    }
    if (!POST) {
        // A_{Gamma I} u_I into vG (warp w: the rows gl = w (mod kDW), entry
        // order), then r_B -= it on Gamma
        for (int e = 0; e < ncoo; ++e) {
            const int pr = gP[e];
            if (((pr >> 16) & (kDW - 1)) != warp) continue;
            vG[(pr >> 16) * 32 + lane] += cvs[e] * xs[(pr & 0xffff) * 32 + lane];
        }
        __syncthreads();
        if (act) {
            for (int q = warp; q < nG; q += kDW) {
                const ACC v = vG[q * 32 + lane];
                if (v != (ACC)0) atomicAdd(&B.rB[(int64_t)gGi[q] * K + lane], -to_f64(v));
            }
        }
    } else {
        double acc = 0.0;   // r.z over the entries of z this substructure writes
        if (act) {
            for (int i = warp; i < nI; i += kDW) {
                const int64_t e = (int64_t)gI[i] * K + lane;
                const double zv = to_f64(xs[i * 32 + lane]);
                z[e] = zv;
                if (rz.sc) acc = fma(r[e], zv, acc);
            }
            for (int e = warp; e < nown; e += kDW) {
                const int owp = gO[2 * e];
                const int64_t o = (int64_t)gO[2 * e + 1] * K + lane;
                const double zv = to_f64(vG[owp * 32 + lane]);
                z[o] = zv;
                if (rz.sc) acc = fma(r[o], zv, acc);
            }
        }
        if (rz.sc) {
            // every entry of z is written once, by its owner: per-substructure
            // partials, summed over the substructures in a fixed order by the
            // block that finishes last
            red[warp * 32 + lane] = acc;
            __syncthreads();
            if (warp == 0) {
                double t = 0.0;
#pragma unroll
                for (int w = 0; w < kDW; ++w) t += red[w * 32 + lane];
                if (act) rz.part[(int64_t)sub * K + lane] = t;
                __threadfence();
            }
            __syncthreads();
            if (tid == 0) *flag = atomicAdd(rz.counter, 1u) == (unsigned)L.nsub - 1u;
            __syncthreads();
            if (!*flag) return;
            __threadfence();
            double t = 0.0;
            if (act) {
                for (int sb = warp; sb < L.nsub; sb += 8 * kDW) {   // eight loads in flight
                    double v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        v[u] = sb + u * kDW < L.nsub ? __ldcg(&rz.part[(int64_t)(sb + u * kDW) * K + lane]) : 0.0;
#pragma unroll
                    for (int u = 0; u < 8; ++u) t += v[u];
                }
            }
            red[warp * 32 + lane] = t;
            __syncthreads();
            if (warp == 0 && act) {
                double tot = 0.0;
#pragma unroll
                for (int w = 0; w < kDW; ++w) tot += red[w * 32 + lane];
                BatchScalars *sc = rz.sc;
                if (!sc->done[lane]) {
                    const double beta = sc->fresh[lane] ? 0.0 : tot / sc->rho[lane];
                    sc->fresh[lane] = 0;
                    sc->hold[lane] = 0;          // joins the next direction update
                    sc->beta[lane] = beta;
                    if (sc->it[lane] > 0) rz.betas[(int64_t)(sc->it[lane] - 1) * K + lane] = beta;
                    sc->rho[lane] = tot;
                }
            }
            if (tid == 0) *rz.counter = 0u;
        }
    }
}

// The Dirichlet corrections with a lane per right-hand side, streamed
// (blocks of up to 16 rows).  A block takes as many substructures as it has
// warps, one per warp, so every warp of the SM runs sweeps and little shared
// memory is needed per substructure: the factor blocks come through a ring of
// slots (unit u in slot u mod the slots, copied that many units ahead; the
// backward sweep starts from the units left in the ring), the right-hand side
// rows of block j are loaded into registers two steps ahead (FP64: one), and
// the forward sweep's y_j go to the sweep scratch (same thread writes and
// reads them back, as far ahead).  Each lane holds all rows of its right-hand side's
// block: a factor column is a broadcast read feeding BP multiply-adds per
// lane and no value crosses lanes.  The coupling entries A_{I Gamma} (post:
// b_I -= A_{I Gamma} u_B; pre: the product A_{Gamma I} x_I) are grouped by
// the block of their interior row at the start (a stable counting sort by
// ballots), so each step applies only its own.  The blocks' zero triangles are
// skipped exactly (TRI: those of L_{j,j-1} too), which a block's warps that
// share rows can do only by halves.
// The ring's unit is a block in FP32, half a block (the sequence Linv_0, Lsub_1,
// Linv_1, ...) in FP64.  There the double pipe bounds the kernel and a
// substructure of the 16 x 16-element kind takes 30 KB with three half blocks:
// seven of them share an SM, one wave of 1024 substructures: 436 us before and
// 462 us after the coarse solve for 32 right-hand sides, where the streaming
// kernel takes 535 and 594 (with two whole blocks in the ring six share an SM,
// and the second wave brought it to 598 and 649).
template <class ACC> __host__ __device__ constexpr int ls_ring() { return sizeof(ACC) == 4 ? 4 : 3; }
template <class ACC, int BP> __host__ __device__ constexpr int ls_max_warps() { return sizeof(ACC) == 8 && BP == 16 ? 7 : 4; }
// Rows of u_B (and half as many of r and z) in flight outside the sweeps, and
// blocks per SM: with blocks of 8 rows the registers of 32 rows in flight
// (166 a thread) left twelve warps per SM.  With half of them 24 warps: 16384
// substructures, post 291 -> 279 us, 1024^2 FP32 solve of 32 91.7 -> 84.5 ms.
template <class ACC> __host__ __device__ constexpr int ls_rows(int bp) { return bp == 8 || sizeof(ACC) == 8 ? 16 : 32; }
template <class ACC> __host__ __device__ constexpr int ls_blocks(int bp) { return bp == 8 && sizeof(ACC) == 4 ? 6 : 0; }

template <class T, class ACC, int BP> struct LaneSmem {
    size_t unit, ring, bsm, vg, rec, srt, bst, bars, warp, total;
    __host__ __device__ static LaneSmem of(const DevLevel &L, int warps) {
        LaneSmem m;
        m.unit = (sizeof(ACC) == 4 ? 2 : 1) * (size_t)BP * BP * sizeof(T);
        m.ring = ls_ring<ACC>() * m.unit;
        m.bsm = al16(sizeof(ACC) * BP * 32);
        m.vg = al16(sizeof(ACC) * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32);
        m.rec = al16((size_t)L.max_irec);
        m.srt = al16(2 * (size_t)(L.max_coo > 0 ? L.max_coo : 1));
        m.bst = al16(2 * (size_t)(L.max_m + 2));
        m.bars = al16(8 * (ls_ring<ACC>() + 1));
        m.warp = m.ring + m.bsm + m.vg + m.rec + m.srt + m.bst + m.bars;
        m.total = warps * m.warp + al16(8 * 32 * warps + 16);
        return m;
    }
};

// TRI: L.sub_tri
template <class T, class ACC, int BP, bool POST, bool TRI>
__global__ void __launch_bounds__(32 * ls_max_warps<ACC, BP>(), ls_blocks<ACC>(BP))
k_dir_ls(DevLevel L, BatchLevel B, const double *r, double *z, const int *skip, RzBatch rz) {
    constexpr int NS = ls_ring<ACC>(), BB = BP * BP;
    constexpr bool HALF = sizeof(ACC) == 8;
    constexpr int UE = HALF ? BB : 2 * BB;   // elements of a ring unit
    if (skip && *skip) return;
    extern __shared__ __align__(16) unsigned char smem_ls[];
    const int nwb = blockDim.x >> 5;
    const LaneSmem<T, ACC, BP> ly = LaneSmem<T, ACC, BP>::of(L, nwb);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = blockIdx.x * nwb + warp;
    const bool live = sub < L.nsub;
    const int K = B.K;
    const bool act = lane < K;
    unsigned char *p = smem_ls + (size_t)warp * ly.warp;
    T *ring = reinterpret_cast<T *>(p);          p += ly.ring;
    ACC *bsm = reinterpret_cast<ACC *>(p);       p += ly.bsm;
    ACC *vG = reinterpret_cast<ACC *>(p);        p += ly.vg;
    unsigned char *rec = p;                      p += ly.rec;
    unsigned short *srt = reinterpret_cast<unsigned short *>(p);   p += ly.srt;
    unsigned short *bst = reinterpret_cast<unsigned short *>(p);   p += ly.bst;
    unsigned long long *bars = reinterpret_cast<unsigned long long *>(p);   // ring slots, then the record
    double *red = reinterpret_cast<double *>(smem_ls + (size_t)nwb * ly.warp);   // [nwb][32]
    int *flag = reinterpret_cast<int *>(red + 32 * nwb);

    const int nI = live ? L.nI[sub] : 0, nG = live ? L.nG[sub] : 0, m = live ? L.nblk[sub] : 0;
    const int ncoo = live ? L.ncoo[sub] : 0, nown = live ? L.nown[sub] : 0;
    const IRecLayout lay(nI, nG, ncoo, nown);
    const unsigned unit_bytes = (unsigned)(UE * sizeof(T));
    const int nu = HALF ? 2 * m - 1 : m;
    const T *F = live ? Ops<T>::get(L).dir + L.offF[sub] : nullptr;
    unsigned ph = 0, pend = 0;      // per ring slot: parity of its next completion, a copy in flight
    bool ok = true;
    double acc = 0.0;               // post: r.z over the entries of z this substructure writes
    auto refill = [&](int u) {      // unit u into its slot, which every lane is done with
        const int s = u % NS;
        if (lane == 0) {
            const T *src = HALF ? F + (size_t)((u + 1) / 2 * 2 + (u & 1)) * BB : F + (size_t)u * UE;
            mbar_expect(&bars[s], unit_bytes);
            bulk_copy(ring + (size_t)s * UE, src, unit_bytes, &bars[s]);
        }
        pend |= 1u << s;
    };
    auto unit = [&](int u) -> const T * { return ring + (size_t)(u % NS) * UE; };
    if (live) {
        if (lane == 0) {
            for (int s = 0; s <= NS; ++s) mbar_init(&bars[s]);
            mbar_expect(&bars[NS], (unsigned)lay.bytes);
            bulk_copy(rec, L.irec + L.irecOff[sub], (unsigned)lay.bytes, &bars[NS]);
        }
        __syncwarp();
        for (int u = 0; u < nu && u < NS; ++u) refill(u);
    }
    pdl_wait();
    pdl_trigger();
    if (live) ok = __all_sync(0xffffffffu, mbar_wait(&bars[NS], 0));
    if (live && ok) {
        const double *gC = reinterpret_cast<const double *>(rec + lay.cv);
        const int *gI = reinterpret_cast<const int *>(rec + lay.iI);
        const int *gGi = reinterpret_cast<const int *>(rec + lay.iG);
        const int *gP = reinterpret_cast<const int *>(rec + lay.pr);
        const int *gO = reinterpret_cast<const int *>(rec + lay.ow);
        ACC *ys = reinterpret_cast<ACC *>(B.ys) + L.offY[sub] * 32;
        // post: the first UV rows of u_B in flight while the entries are sorted
        constexpr int UV = ls_rows<ACC>(BP);
        double uv[UV];
        if (POST) {
#pragma unroll
            for (int u = 0; u < UV; ++u) uv[u] = (u < nG && act) ? B.uB[(int64_t)gGi[u] * K + lane] : 0.0;
        }
        // FP32: the coupling values narrowed in place, entry e's binary32 in the
        // first half of its binary64 slot (read and written by one lane)
        constexpr int CS = 8 / sizeof(ACC);
        ACC *cvs = reinterpret_cast<ACC *>(rec + lay.cv);
        if (CS > 1)
            for (int e = lane; e < ncoo; e += 32) {
                const double v = gC[e];
                cvs[CS * e] = from_f64<ACC>(v);
            }
        {
            // entries by the block of their interior row, in entry order
            // within a block: counts (shared atomics), their prefix sums, then
            // each chunk of 32 entries placed in order (lanes of one block
            // found by __match_any_sync, ranked by lane)
            int *cnt = reinterpret_cast<int *>(bsm);   // [m + 1]; bsm is free until the sweeps
            for (int b = lane; b <= m; b += 32) cnt[b] = 0;
            __syncwarp();
            for (int e = lane; e < ncoo; e += 32) atomicAdd(&cnt[(gP[e] & 0xffff) / BP], 1);
            __syncwarp();
            if (lane == 0) {
                int run = 0;
                for (int b = 0; b < m; ++b) {
                    const int c = cnt[b];
                    bst[b] = (unsigned short)run;
                    cnt[b] = run;
                    run += c;
                }
                bst[m] = (unsigned short)run;
            }
            __syncwarp();
            for (int c0 = 0; c0 < ncoo; c0 += 32) {
                const int e = c0 + lane;
                const int key = e < ncoo ? (gP[e] & 0xffff) / BP : -1;
                const unsigned peers = __match_any_sync(0xffffffffu, key);
                const unsigned below = peers & ((1u << lane) - 1u);
                const int base = key >= 0 ? cnt[key] : 0;
                __syncwarp();
                if (key >= 0) {
                    srt[base + __popc(below)] = (unsigned short)e;
                    if (below == 0) cnt[key] = base + __popc(peers);
                }
                __syncwarp();
            }
        }
        if (POST) {
            for (int q0 = 0; q0 < nG; q0 += UV) {
#pragma unroll
                for (int u = 0; u < UV; ++u)
                    if (q0 + u < nG) vG[(q0 + u) * 32 + lane] = from_f64<ACC>(uv[u]);
                if (q0 + UV < nG) {
#pragma unroll
                    for (int u = 0; u < UV; ++u) {
                        const int q = q0 + UV + u;
                        uv[u] = (q < nG && act) ? B.uB[(int64_t)gGi[q] * K + lane] : 0.0;
                    }
                }
            }
        } else {
            for (int q = 0; q < nG; ++q) {
                vG[q * 32 + lane] = 0;
                if (act) B.uB[(int64_t)gGi[q] * K + lane] = 0.0;   // consumed by the previous post-correction
            }
        }
        __syncwarp();

        constexpr int AH = sizeof(ACC) == 4 ? 2 : 1;   // blocks of rows in flight
        auto load_rows = [&](double (&d)[BP], int j) {
#pragma unroll
            for (int q = 0; q < BP; ++q) {
                const int row = j * BP + q;
                d[q] = (j >= 0 && j < m && row < nI && act) ? r[(int64_t)gI[row] * K + lane] : 0.0;
            }
        };
        auto wait_unit = [&](int u) -> bool {
            const int s = u % NS;
            const bool w = warp_wait_copy(&bars[s], nullptr, lane, (ph >> s) & 1u);   // waits twice for a late copy
            ph ^= 1u << s;
            pend &= ~(1u << s);
            return w;
        };

        // forward sweep: y_j = Linv_j (b_j - L_{j,j-1} y_{j-1})
        ACC xp[BP];
#pragma unroll
        for (int q = 0; q < BP; ++q) xp[q] = 0;
        auto fstep = [&](int j, double (&d)[BP]) -> bool {
#pragma unroll
            for (int q = 0; q < BP; ++q) bsm[q * 32 + lane] = from_f64<ACC>(d[q]);
            load_rows(d, j + AH);
            if (POST) {
                const int e1 = bst[j + 1];
                for (int e = bst[j]; e < e1; ++e) {
                    const int k = srt[e], pr = gP[k];
                    bsm[((pr & 0xffff) - j * BP) * 32 + lane] -= cvs[CS * k] * vG[(pr >> 16) * 32 + lane];
                }
            }
            ACC t[BP];
#pragma unroll
            for (int q = 0; q < BP; ++q) t[q] = bsm[q * 32 + lane];
            if (!HALF && !wait_unit(j)) return false;
            if (j > 0) {
                if (HALF && !wait_unit(2 * j - 1)) return false;
                const T *Ls = HALF ? unit(2 * j - 1) : unit(j) + BB;
#pragma unroll
                for (int c = 0; c < BP; ++c) {
                    ACC col[BP];
                    load_vec<T, ACC, BP>(Ls + c * BP, col);
#pragma unroll
                    for (int q = 0; q < BP; ++q)
                        if (!TRI || q <= c) t[q] -= col[q ^ c] * xp[c];
                }
                if (HALF) {
                    __syncwarp();
                    if (2 * j - 1 + NS < nu) refill(2 * j - 1 + NS);
                }
            }
            if (HALF && !wait_unit(2 * j)) return false;
            const T *Li = unit(HALF ? 2 * j : j);
#pragma unroll
            for (int q = 0; q < BP; ++q) xp[q] = 0;
#pragma unroll
            for (int c = 0; c < BP; ++c) {
                ACC col[BP];
                load_vec<T, ACC, BP>(Li + c * BP, col);
#pragma unroll
                for (int q = c; q < BP; ++q) xp[q] += col[q ^ c] * t[c];
            }
#pragma unroll
            for (int q = 0; q < BP; ++q) ys[(j * BP + q) * 32 + lane] = xp[q];
            __syncwarp();
            if (const int u = (HALF ? 2 * j : j) + NS; u < nu) refill(u);
            return true;
        };
        {
            double da[BP];
            load_rows(da, 0);
            if constexpr (AH == 2) {
                double db[BP];
                load_rows(db, 1);
                for (int j = 0; j < m && ok; j += 2) {
                    ok = fstep(j, da);
                    if (ok && j + 1 < m) ok = fstep(j + 1, db);
                }
            } else {
                for (int j = 0; j < m && ok; ++j) ok = fstep(j, da);
            }
        }

        // backward sweep: z_j = Linv_j^T (y_j - L_{j+1,j}^T z_{j+1})
        if (ok) {
            ACC zn[BP];
#pragma unroll
            for (int q = 0; q < BP; ++q) zn[q] = 0;
            auto load_y = [&](ACC (&y)[BP], int j) {
#pragma unroll
                for (int q = 0; q < BP; ++q) y[q] = j >= 0 ? ys[(j * BP + q) * 32 + lane] : (ACC)0;
            };
            // column dot products in four partial sums (fixed order)
            auto dot4 = [](const ACC (&col)[BP], const ACC (&v)[BP], int c, int q0, int q1) -> ACC {
                ACC a[4] = {0, 0, 0, 0};
#pragma unroll
                for (int q = 0; q < BP; ++q)
                    if (q >= q0 && q < q1) a[q & 3] += col[q ^ c] * v[q];
                return (a[0] + a[1]) + (a[2] + a[3]);
            };
            auto bstep = [&](int j, ACC (&y)[BP]) -> bool {
                ACC t[BP];
#pragma unroll
                for (int q = 0; q < BP; ++q) t[q] = y[q];
                load_y(y, j - AH);
                if (!HALF && j < nu - NS && !wait_unit(j)) return false;
                if (j < m - 1) {
                    if (HALF && 2 * j + 1 < nu - NS && !wait_unit(2 * j + 1)) return false;
                    const T *Ls1 = HALF ? unit(2 * j + 1) : unit(j + 1) + BB;
#pragma unroll
                    for (int c = 0; c < BP; ++c) {
                        ACC col[BP];
                        load_vec<T, ACC, BP>(Ls1 + c * BP, col);
                        t[c] -= dot4(col, zn, c, 0, TRI ? c + 1 : BP);
                    }
                    if (HALF) {
                        __syncwarp();
                        if (2 * j + 1 >= NS) refill(2 * j + 1 - NS);
                    }
                }
                if (HALF && 2 * j < nu - NS && !wait_unit(2 * j)) return false;
                const T *Li = unit(HALF ? 2 * j : j);
#pragma unroll
                for (int c = 0; c < BP; ++c) {
                    ACC col[BP];
                    load_vec<T, ACC, BP>(Li + c * BP, col);
                    zn[c] = dot4(col, t, c, c, BP);
                }
                if (POST) {
#pragma unroll
                    for (int q = 0; q < BP; ++q) {
                        const int row = j * BP + q;
                        if (row < nI && act) z[(int64_t)gI[row] * K + lane] = to_f64(zn[q]);
                    }
                } else {
                    // A_{Gamma I} x_I: this block's entries
#pragma unroll
                    for (int q = 0; q < BP; ++q) bsm[q * 32 + lane] = zn[q];
                    const int e1 = bst[j + 1];
                    for (int e = bst[j]; e < e1; ++e) {
                        const int k = srt[e], pr = gP[k];
                        vG[(pr >> 16) * 32 + lane] += cvs[CS * k] * bsm[((pr & 0xffff) - j * BP) * 32 + lane];
                    }
                }
                __syncwarp();
                if (HALF) {
                    if (2 * j >= NS) refill(2 * j - NS);
                } else if (j <= m - 2 && j + 1 >= NS) {
                    refill(j + 1 - NS);
                }
                return true;
            };
            ACC ya[BP];
            load_y(ya, m - 1);
            if constexpr (AH == 2) {
                ACC yb[BP];
                load_y(yb, m - 2);
                for (int j = m - 1; j >= 0 && ok; j -= 2) {
                    ok = bstep(j, ya);
                    if (ok && j - 1 >= 0) ok = bstep(j - 1, yb);
                }
            } else {
                for (int j = m - 1; j >= 0 && ok; --j) ok = bstep(j, ya);
            }
        }
        if (ok && POST && rz.sc && act) {
            // r.z over the interior entries just written (read back by the
            // lane that wrote them), in four partial sums
            double a4[4] = {0.0, 0.0, 0.0, 0.0};
            constexpr int RU = BP == 8 ? 8 : ls_rows<ACC>(BP);
            for (int i0 = 0; i0 < nI; i0 += RU) {
                double rv[RU], zv[RU];
#pragma unroll
                for (int u = 0; u < RU; ++u) {
                    const bool in = i0 + u < nI;
                    const int64_t e = in ? (int64_t)gI[i0 + u] * K + lane : 0;
                    rv[u] = in ? r[e] : 0.0;
                    zv[u] = in ? z[e] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < RU; ++u) a4[u & 3] = fma(rv[u], zv[u], a4[u & 3]);
            }
            acc = (a4[0] + a4[1]) + (a4[2] + a4[3]);
        }
        if (ok) {
            if (POST) {
                if (act) {
                    for (int e0 = 0; e0 < nown; e0 += 8) {
                        double rv[8], zv[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int e = e0 + u;
                            const bool in = e < nown;
                            const int64_t o = in ? (int64_t)gO[2 * e + 1] * K + lane : 0;
                            zv[u] = in ? to_f64(vG[gO[2 * e] * 32 + lane]) : 0.0;
                            if (in) z[o] = zv[u];
                            rv[u] = in ? r[o] : 0.0;
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) acc = fma(rv[u], zv[u], acc);
                    }
                }
            } else if (act) {
                for (int q = 0; q < nG; ++q) {
                    const ACC v = vG[q * 32 + lane];
                    if (v != (ACC)0) atomicAdd(&B.rB[(int64_t)gGi[q] * K + lane], -to_f64(v));
                }
            }
        }
    }
    if (live && !ok) {
        if (lane == 0) atomicExch(L.err, 1);
        for (int s = 0; s < NS; ++s)   // bounded: copies in flight land before the warp exits
            if ((pend >> s) & 1u) mbar_wait(&bars[s], (ph >> s) & 1u);
        mbar_wait(&bars[NS], 0);
    }
    if (POST && rz.sc) {
        // per-block partials (the warps' in a fixed order), summed over the
        // blocks in a fixed order by the block that finishes last
        red[warp * 32 + lane] = (live && act) ? acc : 0.0;
        __syncthreads();
        if (warp == 0) {
            double t = 0.0;
            for (int w = 0; w < nwb; ++w) t += red[w * 32 + lane];
            if (act) rz.part[(int64_t)blockIdx.x * K + lane] = t;
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) *flag = atomicAdd(rz.counter, 1u) == gridDim.x - 1u;
        __syncthreads();
        if (!*flag) return;
        __threadfence();
        double t = 0.0;
        if (act) {
            constexpr int PU = 16;
            int sb = warp;
            for (; sb + (PU - 1) * nwb < (int)gridDim.x; sb += PU * nwb) {
                double v[PU];
#pragma unroll
                for (int u = 0; u < PU; ++u) v[u] = __ldcg(&rz.part[(int64_t)(sb + u * nwb) * K + lane]);
#pragma unroll
                for (int u = 0; u < PU; ++u) t += v[u];
            }
            for (; sb < (int)gridDim.x; sb += nwb) t += __ldcg(&rz.part[(int64_t)sb * K + lane]);
        }
        red[warp * 32 + lane] = t;
        __syncthreads();
        if (warp == 0 && act) {
            double tot = 0.0;
            for (int w = 0; w < nwb; ++w) tot += red[w * 32 + lane];
            BatchScalars *sc = rz.sc;
            if (!sc->done[lane]) {
                const double beta = sc->fresh[lane] ? 0.0 : tot / sc->rho[lane];
                sc->fresh[lane] = 0;
                sc->hold[lane] = 0;          // joins the next direction update
                sc->beta[lane] = beta;
                if (sc->it[lane] > 0) rz.betas[(int64_t)(sc->it[lane] - 1) * K + lane] = beta;
                sc->rho[lane] = tot;
            }
        }
        if (threadIdx.x == 0) *rz.counter = 0u;
    }
}

// Batched Dirichlet solves for substructures whose factor does not fit in
// shared memory (large or irregular cells).  Persistent blocks, one launch
// per size bucket (the substructures whose blocks take the same number of
// warps), each block taking the bucket's substructures largest first; per
// substructure all 32 right-hand-side columns go in one pass, so each sweep
// streams the factor once.  The unit of the stream is half a block: the
// forward sweep uses Linv_0, Lsub_1, Linv_1, Lsub_2, ... and the backward
// sweep the same sequence in reverse, so a ring of SBN halves (half s in slot
// s mod SBN, refilled SBN halves ahead as soon as it is used) needs no more
// than what is in use and in flight, and turns round on the halves left in
// it.  Thread t of a substructure with block size b owns column group
// g = t / h (columns 4g..4g+3) and the R rows k, k + h, ... (k = t mod h,
// h = ceil(b/R), R = bs_rows) of every block: an R-row x 4-column register
// tile, so a factor entry read from shared memory feeds four FMAs and a
// broadcast 4-column vector 4 R, with four factor columns in flight.  Rows of a block
// are ld apart (odd unless swizzled), so the transposed walks of the backward
// sweep are free of bank conflicts too.  The sweeps touch global memory only
// through the factor's copies and a scratch [8][rows][4] per substructure in
// L2 (each thread its own entries, one step ahead): a first pass of the block,
// a lane per column, gathers the right-hand side (with the post-correction's
// A_IG u_B terms) into it, and a last one writes z and sums r.z.  With those
// gathers inside the sweeps a warp waited on chains of dependent loads at
// every step (ncu: long scoreboard 2.4 of 5.6 cycles per instruction).
// 1024 Voronoi cells of 1000 DOFs, 21
// right-hand sides: solve 145.8 -> 133.3 ms; 1024 cells of 225 DOFs in FP64, 32
// right-hand sides: 600 and 667 us before, 617 and 684 with whole products, 535
// and 594 with the zeros of Lsub left out (which took the Voronoi solve from 130
// to 124 ms).
constexpr int kSBMaxT = 32 * kMaxBuckets;            // largest block
constexpr int kSBSmallT = 96;                        // the common block sizes: more blocks per SM
// Rows of a thread: four in the FP32 accumulator, so that a 4-column vector
// feeds sixteen multiply-adds; two in FP64, whose pipe is the limit anyway.
template <class ACC> __host__ __device__ constexpr int bs_rows() { return sizeof(ACC) == 4 ? 4 : 2; }
// Slots of the ring: three where shared memory limits the blocks of an SM.
template <class ACC> __host__ __device__ constexpr int bs_ring() { return sizeof(ACC) == 4 ? 3 : 4; }

__host__ __device__ inline size_t red_doubles(int nt) { return nt > 256 ? (size_t)nt : 256; }
struct StreamSmemB {
    size_t stage, ring, vec, red, total;
    template <class T, class ACC> __host__ __device__ static StreamSmemB of(const DevLevel &L, int nt) {
        constexpr int SBN = bs_ring<ACC>();
        StreamSmemB m;
        const size_t mb = L.max_b > 0 ? L.max_b : 1, mld = L.max_ld > 0 ? L.max_ld : 1;
        m.stage = al16(mb * mld * sizeof(T) + 32);
        m.ring = SBN * m.stage;
        m.vec = al16(sizeof(ACC) * mb * kMaxBatch);   // [8][b][4]
        m.red = al16(8 * red_doubles(nt) + 16);       // r.z partials per warp and column, a flag
        m.total = m.ring + 2 * m.vec + m.red + 8 * SBN + 16;
        return m;
    }
};

__device__ __forceinline__ void ld4(const float *p, float (&v)[4]) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void ld4(const double *p, double (&v)[4]) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0], c = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = c.x; v[3] = c.y;
}
__device__ __forceinline__ void st4(float *p, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void st4(double *p, const double (&v)[4]) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}

// a[i] (row rw[i], F <= i < E) -= (SUB) or += sum over c in [c0, c1) of
// M(row, c) v[c] for four columns.  COL: M(r, c) is the stored entry (r, c) (a
// column walk); else the stored entry (c, r) (a row walk, the transposed block).
template <class T, class ACC, bool SUB, bool COL, bool SWZ, int F, int E, int R>
__device__ __forceinline__ void prod(ACC (&a)[R][4], const T *M, int ldm, const ACC *v, int c0, int c1,
                                     const int (&rw)[R]) {
    auto at = [&](int r, int c) -> const T * {
        if (COL) return M + c * ldm + (SWZ ? (r ^ c) : r);
        return M + r * ldm + (SWZ ? (c ^ r) : c);
    };
    auto fma4 = [&](ACC (&y)[4], ACC l, const ACC (&x)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (SUB) y[q] -= l * x[q];
            else y[q] += l * x[q];
        }
    };
    int c = c0;
    for (; c + 4 <= c1; c += 4) {
        ACC x[4][4], l[4][R];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) ld4(v + (c + cc) * 4, x[cc]);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
            for (int i = F; i < E; ++i) l[cc][i] = ld<T, ACC>(at(rw[i], c + cc));
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
            for (int i = F; i < E; ++i) fma4(a[i], l[cc][i], x[cc]);
    }
    for (; c < c1; ++c) {
        ACC x[4];
        ld4(v + c * 4, x);
#pragma unroll
        for (int i = F; i < E; ++i) fma4(a[i], ld<T, ACC>(at(rw[i], c)), x);
    }
}
// The same over all columns of an M with a triangle of zeros, for the rows k,
// k + h, ... of a thread: M(row, c) is zero for c > row + d (LOW) or c < row - d,
// so row i of them has its columns below (i + 1) h + d or from i h - d on, taken
// in R segments.
template <class T, class ACC, bool SUB, bool COL, bool SWZ, bool LOW, int R, int SEG = 0>
__device__ __forceinline__ void prod_tri(ACC (&a)[R][4], const T *M, int ldm, const ACC *v, int h, int b, int d,
                                         const int (&rw)[R], int c0 = 0) {
    const int e = tri_segment_end(SEG, R, h, b, d, LOW);
    prod<T, ACC, SUB, COL, SWZ, LOW ? SEG : 0, LOW ? R : SEG + 1, R>(a, M, ldm, v, c0, e, rw);
    if constexpr (SEG + 1 < R) prod_tri<T, ACC, SUB, COL, SWZ, LOW, R, SEG + 1>(a, M, ldm, v, h, b, d, rw, e);
}

template <class T, class ACC, bool SWZ, bool POST, int NT>
__global__ void __launch_bounds__(NT, NT == kSBSmallT ? 6 : 1)
k_dir_bs(DevLevel L, BatchLevel B, const double *r, double *z, const int *skip, RzBatch rz, const int *perm,
         int count) {
    constexpr int R = bs_rows<ACC>(), SBN = bs_ring<ACC>();   // rows of a thread, slots
    extern __shared__ __align__(16) unsigned char smem_bs[];
    if (skip && *skip) return;
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = nt >> 5;
    const StreamSmemB ly = StreamSmemB::of<T, ACC>(L, nt);
    unsigned char *ring = smem_bs;
    ACC *ybuf = reinterpret_cast<ACC *>(smem_bs + ly.ring);
    ACC *tbuf = reinterpret_cast<ACC *>(smem_bs + ly.ring + ly.vec);
    double *red = reinterpret_cast<double *>(smem_bs + ly.ring + 2 * ly.vec);
    int *flag = reinterpret_cast<int *>(red + red_doubles(nt));
    unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem_bs + ly.ring + 2 * ly.vec + ly.red);
    const int K = B.K;
    const bool lact = lane < K;
    const OpSet<T> &O = Ops<T>::get(L);
    if (tid == 0)
        for (int s2 = 0; s2 < SBN; ++s2) mbar_init(&bars[s2]);
    __syncthreads();
    RingSlots slots;                      // copies in flight: thread 0's
    for (int ti = blockIdx.x; ti < count; ti += gridDim.x) {
        const int sub = perm[ti];
        const int nI = L.nI[sub], nG = L.nG[sub], b = L.bsz[sub], m = nI > 0 ? L.nblk[sub] : 0;
        const int mb = m * b, ldb = fld(b, SWZ), h = (b + R - 1) / R;
        const int dz = L.sub_over[sub];   // Lsub is zero left of column row - dz
        const T *F = O.dir + L.offF[sub];
        const size_t bsq = (size_t)b * ldb;
        const int *iI = L.idxI + L.offI[sub];
        const int *iG = L.idxG + L.offG[sub];
        ACC *Ysub = reinterpret_cast<ACC *>(B.ys) + L.offY[sub] * kMaxBatch;   // [8][mb][4]
        ACC *Yl = Ysub + (size_t)(lane >> 2) * mb * 4 + (lane & 3);            // this lane's column: row i at 4 i
        const bool act = tid < 8 * h;
        const int cg = act ? tid / h : 0, k = act ? tid - cg * h : 0;
        int rw[R];                        // its rows; beyond the block: computed on the last one, not kept
#pragma unroll
        for (int i = 0; i < R; ++i) rw[i] = k + i * h < b ? k + i * h : b - 1;
        auto kept = [&](int i) { return k + i * h < b; };
        const bool colact = act && 4 * cg < K;
        ACC *Yg = Ysub + (size_t)cg * mb * 4;
        ACC *yb = ybuf + (size_t)cg * b * 4, *tb = tbuf + (size_t)cg * b * 4;
        // half s of the sequence Linv_0, Lsub_1, Linv_1, ...: s = 2 j: Linv_j, s = 2 j - 1: Lsub_j
        const int ns = 2 * m - 1;
        auto half_of = [&](int s) { return F + ((size_t)(s + 1) / 2 * 2 + (s & 1)) * bsq; };
        auto issue = [&](int s) {         // thread 0: half s, its bytes rounded out to 16-byte boundaries
            const uintptr_t a = reinterpret_cast<uintptr_t>(half_of(s));
            const uintptr_t al = a & ~uintptr_t(15);
            const uintptr_t ae = (a + bsq * sizeof(T) + 15) & ~uintptr_t(15);
            mbar_expect(&bars[s % SBN], (unsigned)(ae - al));
            bulk_copy(ring + (size_t)(s % SBN) * ly.stage, reinterpret_cast<const void *>(al),
                      (unsigned)(ae - al), &bars[s % SBN]);
            slots.issued(s % SBN);
        };
        auto slot = [&](int s) {
            const uintptr_t a = reinterpret_cast<uintptr_t>(half_of(s));
            return reinterpret_cast<const T *>(ring + (size_t)(s % SBN) * ly.stage + (a & 15));
        };
        auto wait_half = [&](int s) {     // every thread sees the copy's completion itself
            slots.wait(s % SBN, [&](int q, unsigned parity) { return mbar_wait(&bars[q], parity); });
        };
        if (tid == 0 && slots.ok)
            for (int s = 0; s < SBN && s < ns; ++s) issue(s);
        {
            // the right-hand side into the scratch, a lane per column, four
            // rows in flight: interior rows of r, minus their A_{I Gamma} u_B
            // terms in the post-correction (the row's coupling entries in
            // increasing order); padding rows and columns are zero
            const int64_t i0 = L.offI[sub];
            constexpr int PU = 4;
            for (int q0 = w * PU; q0 < mb; q0 += nw * PU) {
                double v[PU];
                int e0[PU], e1[PU];
#pragma unroll
                for (int u = 0; u < PU; ++u) {
                    const int i = q0 + u;
                    v[u] = (i < nI && lact) ? r[(int64_t)iI[i] * K + lane] : 0.0;
                    e0[u] = e1[u] = 0;
                    if (POST && i < nI) {
                        e0[u] = (int)L.cooRptr[i0 + i];
                        e1[u] = (int)L.cooRptr[i0 + i + 1];
                    }
                }
#pragma unroll
                for (int u = 0; u < PU; ++u) {
                    if (q0 + u >= mb) break;
                    ACC x = from_f64<ACC>(v[u]);
                    if (POST && lact)
                        for (int p = e0[u]; p < e1[u]; ++p)
                            x -= ld<T, ACC>(O.aig + L.cooRowE[p]) *
                                 from_f64<ACC>(B.uB[(int64_t)L.cooRowId[p] * K + lane]);
                    Yl[(size_t)(q0 + u) * 4] = x;
                }
            }
        }
        __syncthreads();
        ACC nx[R][4];                     // the next step's rows, loaded a step ahead
        if (colact && m > 0)
#pragma unroll
            for (int i = 0; i < R; ++i) ld4(Yg + (size_t)rw[i] * 4, nx[i]);
        // forward: y_j = Linv_j (rhs_j - Lsub_j y_{j-1})
        for (int j = 0; j < m; ++j) {
            ACC a[R][4];
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[i][q] = nx[i][q];
                    if (j + 1 < m) ld4(Yg + ((size_t)(j + 1) * b + rw[i]) * 4, nx[i]);
                }
            }
            if (j > 0) {
                wait_half(2 * j - 1);
                if (colact) prod_tri<T, ACC, true, true, SWZ, false, R>(a, slot(2 * j - 1), ldb, yb, h, b, dz, rw);
            }
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (kept(i)) st4(tb + rw[i] * 4, a[i]);
            }
            wait_half(2 * j);
            __syncthreads();
            if (tid == 0 && slots.ok && j > 0 && 2 * j - 1 + SBN < ns) issue(2 * j - 1 + SBN);
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[i][q] = 0;
                prod_tri<T, ACC, false, true, SWZ, true, R>(a, slot(2 * j), ldb, tb, h, b, 0, rw);   // Linv_j
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    if (kept(i)) {
                        st4(yb + rw[i] * 4, a[i]);
                        st4(Yg + ((size_t)j * b + rw[i]) * 4, a[i]);
                    }
                    if (j + 1 == m)
#pragma unroll
                        for (int q = 0; q < 4; ++q) nx[i][q] = a[i][q];   // y_{m-1}
                }
            }
            __syncthreads();
            if (tid == 0 && slots.ok && 2 * j + SBN < ns) issue(2 * j + SBN);
        }
        // backward: x_j = Linv_j^T (y_j - Lsub_{j+1}^T x_{j+1}); halves ns-1 ..
        // ns-SBN are still in the ring
        for (int j = m - 1; j >= 0; --j) {
            ACC a[R][4];
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[i][q] = nx[i][q];
                    if (j > 0) ld4(Yg + ((size_t)(j - 1) * b + rw[i]) * 4, nx[i]);
                }
            }
            if (j < m - 1) {
                const int s = 2 * j + 1;
                if (s < ns - SBN) wait_half(s);
                if (colact) prod_tri<T, ACC, true, false, SWZ, true, R>(a, slot(s), ldb, yb, h, b, dz, rw);
            }
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (kept(i)) st4(tb + rw[i] * 4, a[i]);
            }
            if (2 * j < ns - SBN) wait_half(2 * j);
            __syncthreads();
            if (tid == 0 && slots.ok && j < m - 1 && 2 * j + 1 - SBN >= 0) issue(2 * j + 1 - SBN);
            if (colact) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[i][q] = 0;
                prod_tri<T, ACC, false, false, SWZ, false, R>(a, slot(2 * j), ldb, tb, h, b, 0, rw);   // its transpose
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (kept(i)) {
                        st4(yb + rw[i] * 4, a[i]);
                        st4(Yg + ((size_t)j * b + rw[i]) * 4, a[i]);
                    }
            }
            __syncthreads();
            if (tid == 0 && slots.ok && 2 * j - SBN >= 0) issue(2 * j - SBN);
        }
        if (!__syncthreads_and(slots.ok)) break;
        // every issued half has been waited for: the ring is idle from here
        if (!POST) {
            // r_B -= A_{Gamma I} x (Gamma entry q: warp q mod nw, lane: column;
            // the entry's couplings in order); u_B was consumed by the previous
            // post-correction
            const int64_t g0 = L.offG[sub];
            if (lact)
                for (int q = w; q < nG; q += nw) {
                    ACC acc = 0;
                    for (int64_t e = L.cooGptr[g0 + q]; e < L.cooGptr[g0 + q + 1]; ++e)
                        acc += ld<T, ACC>(O.aig + e) * Yl[(size_t)L.cooI[e] * 4];
                    const int64_t o = (int64_t)iG[q] * K + lane;
                    if (acc != (ACC)0) atomicAdd(&B.rB[o], -to_f64(acc));
                    B.uB[o] = 0.0;
                }
            __syncthreads();              // the scratch and the buffers are free for the next substructure
            continue;
        }
        // z: the interior rows from the scratch and the owned interface
        // entries (u_B), a lane per column; r.z over what is written
        double rzs = 0.0;
        constexpr int PU = 4;
        for (int q0 = w * PU; q0 < nI; q0 += nw * PU) {
            double zv[PU], rv[PU];
            int o[PU];                    // DOF
#pragma unroll
            for (int u = 0; u < PU; ++u) {
                const int i = q0 + u;
                const bool in = i < nI && lact;
                o[u] = in ? iI[i] : 0;
                zv[u] = in ? to_f64(Yl[(size_t)i * 4]) : 0.0;
                rv[u] = in && rz.sc ? r[(int64_t)o[u] * K + lane] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < PU; ++u) {
                if (q0 + u < nI && lact) z[(int64_t)o[u] * K + lane] = zv[u];
                rzs = fma(rv[u], zv[u], rzs);
            }
        }
        for (int64_t q0 = L.offOwn[sub] + w * PU; q0 < L.offOwn[sub + 1]; q0 += nw * PU) {
            double zv[PU], rv[PU];
            int o[PU];                    // DOF
#pragma unroll
            for (int u = 0; u < PU; ++u) {
                const bool in = q0 + u < L.offOwn[sub + 1] && lact;
                const int id = in ? L.own[q0 + u] : 0;
                o[u] = in ? L.ifaceDof[id] : 0;
                zv[u] = in ? B.uB[(int64_t)id * K + lane] : 0.0;
                rv[u] = in && rz.sc ? r[(int64_t)o[u] * K + lane] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < PU; ++u) {
                if (q0 + u < L.offOwn[sub + 1] && lact) z[(int64_t)o[u] * K + lane] = zv[u];
                rzs = fma(rv[u], zv[u], rzs);
            }
        }
        __syncthreads();                  // the scratch is free for the next substructure
        if (!rz.sc) continue;
        // r.z per column: the warps in order, then the substructures by the
        // block that finishes the last one, in order
        red[w * 32 + lane] = rzs;
        __syncthreads();
        if (w == 0 && lact) {
            double t = 0.0;
            for (int u = 0; u < nw; ++u) t += red[u * 32 + lane];
            rz.part[(int64_t)sub * K + lane] = t;
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) *flag = atomicAdd(rz.counter, 1u) == (unsigned)L.nsub - 1u;
        __syncthreads();
        if (*flag) {
            __threadfence();
            // eight fixed groups of substructures (sb mod 8), whatever the
            // bucket of the finishing block: the same order in every run
            for (int g = w; g < 8; g += nw) {
                double t = 0.0;
                if (lact) {
                    // sixteen loads in flight (one at a time, this tail took
                    // 25 us more at 1024 substructures)
                    for (int sb = g; sb < L.nsub; sb += 8 * 16) {
                        double v[16];
#pragma unroll
                        for (int u = 0; u < 16; ++u)
                            v[u] = sb + 8 * u < L.nsub ? __ldcg(&rz.part[(int64_t)(sb + 8 * u) * K + lane]) : 0.0;
#pragma unroll
                        for (int u = 0; u < 16; ++u) t += v[u];
                    }
                }
                red[g * 32 + lane] = t;
            }
            __syncthreads();
            if (w == 0 && lact) {
                double tot = 0.0;
                for (int v = 0; v < 8; ++v) tot += red[v * 32 + lane];
                BatchScalars *sc = rz.sc;
                if (!sc->done[lane]) {
                    const double beta = sc->fresh[lane] ? 0.0 : tot / sc->rho[lane];
                    sc->fresh[lane] = 0;
                    sc->hold[lane] = 0;
                    sc->beta[lane] = beta;
                    if (sc->it[lane] > 0) rz.betas[(int64_t)(sc->it[lane] - 1) * K + lane] = beta;
                    sc->rho[lane] = tot;
                }
            }
            if (tid == 0) *rz.counter = 0u;
        }
        __syncthreads();                  // red is free for the next substructure
    }
    if (!slots.ok) atomicExch(L.err, 1);
    if (tid == 0)                         // bounded: copies in flight land before the block exits
        slots.drain(SBN, [&](int q, unsigned parity) { return mbar_wait(&bars[q], parity); });
}

// (6)-(9) for K right-hand sides, a block of up to kNBW warps per
// substructure and a lane per right-hand side.  The record [Psi | D | ids] and
// the rows of N_i arrive by bulk copies that start before the vectors are
// touched; N_i streams through two stages of `chunk` bytes, so records of any
// size take this route.  Shared-memory reads bound the product (one per
// multiply-add when an entry feeds one row): a warp takes tiles of eight rows,
// so an entry of f and two vector reads of N feed eight multiply-adds, and RT
// tiles at once.  w_i is kept in the accumulator type (the value it was
// computed in; half the traffic of FP64 in the mixed path).
// Measured (solves of the benchmark cases, the kernels these replaced read one
// shared word per multiply-add): 21 right-hand sides on 1024 Voronoi cells
// 157.5 -> 145.8 ms, 32 on the 1024^2 three-level problem 107.4 -> 101.3 ms.
constexpr int kChunkBytes = 32 * 1024, kNBW = 8;   // chunk of N; most warps of a block

// chunk: bytes of N per stage (0: kChunkBytes), the autotuner's choice
template <class T> __host__ __device__ inline int neu_chunk_rows(int nG, int chunk = 0) {
    const int cb = chunk > 0 ? chunk : kChunkBytes;
    const int rows = cb / (int)(sizeof(T) * (nG > 0 ? (nG + 7) & ~7 : 8));
    return rows < 1 ? 1 : (rows > nG ? (nG > 0 ? nG : 1) : rows);
}
struct NeuSmem {
    size_t head, f, stage, total;
    template <class T, class ACC> __host__ __device__ static NeuSmem of(const DevLevel &L, int chunk, bool head = true) {
        NeuSmem m;
        const size_t mg = L.max_nG > 0 ? L.max_nG : 1, mc = L.max_nc > 0 ? L.max_nc : 1;
        const size_t row = sizeof(T) * ((mg + 7) & ~size_t(7));
        m.head = head ? (size_t)NRecLayout((int)mg, (int)mc, (int)sizeof(T)).N : 0;
        m.f = al16(sizeof(ACC) * ((mg + 7) & ~size_t(7)) * 32);
        const size_t cb = chunk > 0 ? (size_t)chunk : (size_t)kChunkBytes;
        // one stage when the whole operator fits in it and one pass covers its rows, else two
        const bool whole = mg * row <= cb && (mg + 7) / 8 <= kNBW * (sizeof(ACC) == 8 ? 2 : 3);
        m.stage = whole ? al16(mg * row) : al16(row > cb ? row : cb);
        m.total = m.head + m.f + (whole ? 1 : 2) * m.stage + 32;
        return m;
    }
};
template <class T, class ACC> __host__ inline size_t neu_bg_smem(const DevLevel &L, int chunk_bytes, bool head = true) {
    return NeuSmem::of<T, ACC>(L, chunk_bytes, head).total;
}

// HEAD: the record ahead of N is staged; else it is read where it lies (levels
// whose Psi leaves no room for N's stages: FP64 interfaces of 512 DOFs with 19
// coarse ones or more).
template <class T, class ACC, int RT, bool HEAD>
__global__ void __launch_bounds__(32 * kNBW, RT == 1 ? 4 : 3) k_neu_bg(DevLevel L, BatchLevel B, int pidx, const double *r,
                                                      const int *skip, int chunk) {
    extern __shared__ __align__(16) unsigned char smem_ng[];
    if (skip && *skip) return;
    const int sub = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    const int K = B.K;
    const bool act = lane < K;
    const int nG = L.nG[sub], nc = L.ncl[sub];
    const NeuSmem ly = NeuSmem::of<T, ACC>(L, chunk, HEAD);
    const NRecLayout lay(nG, nc, (int)sizeof(T));
    const unsigned char *rec = L.nrec[pidx] + L.nrecOff[pidx][sub];
    const unsigned char *head = HEAD ? smem_ng : rec;
    ACC *f = reinterpret_cast<ACC *>(smem_ng + ly.head);
    unsigned char *ring = smem_ng + ly.head + ly.f;
    unsigned long long *bars = reinterpret_cast<unsigned long long *>(smem_ng + ly.total - 32);   // stages, head
    const int ldn = lay.ld, CH = neu_chunk_rows<T>(nG, chunk);
    const int ntile = ldn >> 3, nch = nG > 0 ? (nG + CH - 1) / CH : 0;
    // N streams once per pass of nw * RT tiles; step s is chunk s % nch of pass s / nch
    const int npass = (ntile + nw * RT - 1) / (nw * RT), nstep = npass * nch;
    auto issue = [&](int s) {               // thread 0: step s into stage s & 1
        const int p0 = (s % nch) * CH, pn = nG - p0 < CH ? nG - p0 : CH;
        bulk_load(ring + (size_t)(s & 1) * ly.stage, rec + lay.N + (size_t)p0 * ldn * sizeof(T),
                  (unsigned)(al16((size_t)pn * ldn * sizeof(T))), &bars[s & 1]);
    };
    if (tid == 0) {
        for (int s = 0; s < 3; ++s) mbar_init(&bars[s]);
        if (HEAD && lay.N > 0) bulk_load(smem_ng, rec, (unsigned)lay.N, &bars[2]);
        for (int s = 0; s < 2 && s < nstep; ++s) issue(s);
    }
    __syncthreads();
    bool ok = !HEAD || lay.N == 0 || mbar_wait(&bars[2], 0);
    int waited = 0;                          // steps waited for
    if (__syncthreads_and(ok)) {
        const T *Ps = reinterpret_cast<const T *>(head + lay.psi);
        const T *wg = reinterpret_cast<const T *>(head + lay.wg);
        const int *iG = reinterpret_cast<const int *>(head + lay.iG);
        const int *rcs = reinterpret_cast<const int *>(head + lay.rc);
        const int *gG = reinterpret_cast<const int *>(head + lay.gG);
        constexpr int GU = 8;                // rows of r and r_B in flight per warp
        for (int q0 = warp; q0 < ldn; q0 += nw * GU) {
            double v[GU], c[GU];
#pragma unroll
            for (int u = 0; u < GU; ++u) {
                const int q = q0 + u * nw;
                const bool in = q < nG && act;
                v[u] = in ? r[(int64_t)gG[q] * K + lane] : 0.0;
                c[u] = in ? B.rB[(int64_t)iG[q] * K + lane] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < GU; ++u) {
                const int q = q0 + u * nw;
                if (q < ldn) f[q * 32 + lane] = q < nG ? ld<T, ACC>(wg + q) * from_f64<ACC>(v[u] + c[u]) : (ACC)0;
            }
        }
        __syncthreads();
        const int64_t g0 = L.offG[sub];
        ACC *W = reinterpret_cast<ACC *>(B.w);
        for (int pass = 0, s = 0; pass < npass && ok; ++pass) {
            const int t0 = pass * nw * RT + warp;      // tiles t0, t0 + nw, ...
            ACC acc[RT][8];
#pragma unroll
            for (int t = 0; t < RT; ++t)
#pragma unroll
                for (int u = 0; u < 8; ++u) acc[t][u] = 0;
            for (int c = 0; c < nch; ++c, ++s) {
                const bool got = mbar_wait(&bars[s & 1], (unsigned)(s >> 1) & 1u);
                waited = s + 1;
                if (!__syncthreads_and(got)) { ok = false; break; }
                const T *buf = reinterpret_cast<const T *>(ring + (size_t)(s & 1) * ly.stage);
                const int p0 = c * CH, pn = nG - p0 < CH ? nG - p0 : CH;
                if (t0 < ntile) {
#pragma unroll 2
                    for (int pp = 0; pp < pn; ++pp) {
                        const ACC fv = f[(p0 + pp) * 32 + lane];
#pragma unroll
                        for (int t = 0; t < RT; ++t) {
                            if (t0 + t * nw < ntile) {
                                ACC col[8];
                                load_vec<T, ACC, 8>(buf + pp * ldn + (t0 + t * nw) * 8, col);
#pragma unroll
                                for (int u = 0; u < 8; ++u) acc[t][u] += col[u] * fv;
                            }
                        }
                    }
                }
                __syncthreads();                       // the stage is free
                if (tid == 0 && s + 2 < nstep) issue(s + 2);
            }
            if (!ok) break;
            if (act) {
#pragma unroll
                for (int t = 0; t < RT; ++t)
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int q = (t0 + t * nw) * 8 + u;
                        if (q < nG) W[(g0 + q) * K + lane] = acc[t][u];
                    }
            }
        }
        if (ok) {
            // r_c += Psi^T f: a row per warp, eight entries per step
            for (int k = warp; k < nc; k += nw) {
                ACC s4[4] = {0, 0, 0, 0};
                for (int q = 0; q < ldn; q += 8) {
                    ACC row[8];
                    load_vec<T, ACC, 8>(Ps + (size_t)k * ldn + q, row);
#pragma unroll
                    for (int u = 0; u < 8; ++u) s4[u & 3] += row[u] * f[(q + u) * 32 + lane];
                }
                if (act) atomicAdd(&B.rcv[(int64_t)rcs[k] * K + lane], to_f64((s4[0] + s4[1]) + (s4[2] + s4[3])));
            }
            return;
        }
    }
    // a wait gave up: flag it, and let the copies in flight land (bounded)
    if (tid == 0) {
        atomicExch(L.err, 1);
        if (HEAD && lay.N > 0) mbar_wait(&bars[2], 0);
        const int s0 = waited > 0 ? waited - 1 : 0;          // in flight: the step that failed and the next
        for (int s = s0; s < s0 + 2 && s < nstep; ++s) mbar_wait(&bars[s & 1], (unsigned)(s >> 1) & 1u);
    }
}

// (9) for K right-hand sides: u_B += D_i (w_i + Psi_i u_c) on Gamma; clears
// the r_B and r_c entries it consumed.  Tiles of eight rows per warp as above.
__host__ __device__ inline size_t avg_head(const DevLevel &L, int esz) {
    return (size_t)NRecLayout(L.max_nG > 0 ? L.max_nG : 1, L.max_nc > 0 ? L.max_nc : 1, esz).avg_bytes;
}
template <class T, class ACC> __host__ inline size_t avg_bg_smem(const DevLevel &L) {
    return avg_head(L, (int)sizeof(T)) + al16(sizeof(ACC) * (size_t)(L.max_nc > 0 ? L.max_nc : 1) * 32) + 16;
}
template <class T, class ACC>
__global__ void __launch_bounds__(32 * kNBW) k_avg_bg(DevLevel L, BatchLevel B, int pidx, const int *skip) {
    extern __shared__ __align__(16) unsigned char smem_ag[];
    if (skip && *skip) return;
    const int sub = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    const int K = B.K;
    const bool act = lane < K;
    const int nG = L.nG[sub], nc = L.ncl[sub];
    const NRecLayout lay(nG, nc, (int)sizeof(T));
    const size_t mh = avg_head(L, (int)sizeof(T));
    unsigned char *head = smem_ag;
    ACC *uc = reinterpret_cast<ACC *>(smem_ag + mh);
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(
        smem_ag + mh + al16(sizeof(ACC) * (size_t)(L.max_nc > 0 ? L.max_nc : 1) * 32));
    if (tid == 0) {
        mbar_init(bar);
        if (lay.avg_bytes > 0) bulk_load(head, L.nrec[pidx] + L.nrecOff[pidx][sub], (unsigned)lay.avg_bytes, bar);
    }
    // w of the first tile in flight while the record arrives
    const int64_t g0 = L.offG[sub];
    const ACC *W = reinterpret_cast<const ACC *>(B.w);
    ACC v[8];
    auto load_w = [&](int t) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = t * 8 + u;
            v[u] = (act && q < nG) ? W[(g0 + q) * K + lane] : (ACC)0;
        }
    };
    const int ntile = lay.ld >> 3;
    load_w(warp);
    __syncthreads();
    const bool ok = lay.avg_bytes == 0 || mbar_wait(bar, 0);
    if (!__syncthreads_and(ok)) {
        if (tid == 0) {
            atomicExch(L.err, 1);
            mbar_wait(bar, 0);               // bounded: the copy lands before the block exits
        }
        return;
    }
    const T *Ps = reinterpret_cast<const T *>(head + lay.psi);
    const T *wg = reinterpret_cast<const T *>(head + lay.wg);
    const int *iG = reinterpret_cast<const int *>(head + lay.iG);
    const int *rcs = reinterpret_cast<const int *>(head + lay.rc);
    for (int k = warp; k < nc; k += nw)
        uc[k * 32 + lane] = act ? from_f64<ACC>(B.ucv[(int64_t)rcs[k] * K + lane]) : (ACC)0;
    __syncthreads();
    for (int t = warp; t < ntile; t += nw) {
        if (t != warp) load_w(t);
#pragma unroll 2
        for (int k = 0; k < nc; ++k) {
            const ACC ucv = uc[k * 32 + lane];
            ACC row[8];
            load_vec<T, ACC, 8>(Ps + (size_t)k * lay.ld + t * 8, row);
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] += row[u] * ucv;
        }
        if (act) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int q = t * 8 + u;
                if (q >= nG) break;
                const int64_t e = (int64_t)iG[q] * K + lane;
                atomicAdd(&B.uB[e], to_f64(ld<T, ACC>(wg + q) * v[u]));
                B.rB[e] = 0.0;            // consumed by the substructure correction
            }
        }
    }
    if (act)
        for (int k = warp; k < nc; k += nw) B.rcv[(int64_t)rcs[k] * K + lane] = 0.0;   // consumed
}

// (6)-(8) for K right-hand sides: f = D_i r_B on Gamma, w = N_i f,
// r_c += Psi_i^T f.
template <class T, class ACC>
__global__ void k_neu_b(DevLevel L, BatchLevel B, int pidx, const double *r, const int *skip,
                        unsigned slice) {
    extern __shared__ __align__(16) unsigned char smem_b[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = blockIdx.x * (blockDim.x >> 5) + warp;
    if (sub >= L.nsub) { pdl_wait(); return; }
    const int K = B.K;
    const bool act = lane < K;
    unsigned char *p = smem_b + (size_t)warp * slice;
    unsigned char *rec = p;                  p += al16((size_t)L.max_nrec[pidx]);
    ACC *f = reinterpret_cast<ACC *>(p);     p += al16(sizeof(ACC) * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32);
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(p);
    const int nG = L.nG[sub], nc = L.ncl[sub];
    const NRecLayout lay(nG, nc, (int)sizeof(T));
    if (lane == 0) mbar_init(bar);
    __syncwarp();
    if (lane == 0 && lay.bytes) {
        mbar_expect(bar, (unsigned)lay.bytes);
        bulk_copy(rec, L.nrec[pidx] + L.nrecOff[pidx][sub], (unsigned)lay.bytes, bar);
    }
    pdl_wait();
    pdl_trigger();
    if (skip && *skip) {
        if (lay.bytes) mbar_wait(bar, 0);   // bounded: the copy lands first
        return;
    }
    if (lay.bytes && !warp_wait_copy(bar, L.err, lane)) return;
    const T *Ps = reinterpret_cast<const T *>(rec + lay.psi);
    const T *wg = reinterpret_cast<const T *>(rec + lay.wg);
    const int *iG = reinterpret_cast<const int *>(rec + lay.iG);
    const int *rcs = reinterpret_cast<const int *>(rec + lay.rc);
    const int *gG = reinterpret_cast<const int *>(rec + lay.gG);
    const T *Ns = reinterpret_cast<const T *>(rec + lay.N);
    for (int q0 = 0; q0 < nG; q0 += 16) {
        double v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int q = q0 + u;
            v[u] = (q < nG && act) ? r[(int64_t)gG[q] * K + lane] + B.rB[(int64_t)iG[q] * K + lane] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 16; ++u)
            if (q0 + u < nG) f[(q0 + u) * 32 + lane] = ld<T, ACC>(wg + q0 + u) * from_f64<ACC>(v[u]);
    }
    const int64_t g0 = L.offG[sub];
    // w = N f, four output rows at a time (each f entry read once per four rows)
    for (int q0 = 0; q0 < nG; q0 += 4) {
        ACC s[4] = {0, 0, 0, 0};
        const int nq = nG - q0 < 4 ? nG - q0 : 4;
        for (int pp = 0; pp < nG; ++pp) {
            const ACC fv = f[pp * 32 + lane];
            const T *Nr = Ns + (size_t)pp * lay.ld + q0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < nq) s[u] += ld<T, ACC>(Nr + u) * fv;
        }
        if (act)
            for (int u = 0; u < nq; ++u) reinterpret_cast<ACC *>(B.w)[(g0 + q0 + u) * K + lane] = s[u];
    }
    for (int k0 = 0; k0 < nc; k0 += 4) {
        ACC s[4] = {0, 0, 0, 0};
        const int nk = nc - k0 < 4 ? nc - k0 : 4;
        for (int q = 0; q < nG; ++q) {
            const ACC fv = f[q * 32 + lane];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < nk) s[u] += ld<T, ACC>(Ps + (size_t)(k0 + u) * lay.ld + q) * fv;
        }
        if (act)
            for (int u = 0; u < nk; ++u) atomicAdd(&B.rcv[(int64_t)rcs[k0 + u] * K + lane], to_f64(s[u]));
    }
}

// (9) for K right-hand sides: u_B += D_i (w_i + Psi_i u_c) on Gamma; clears
// the r_B and r_c entries it consumed.
template <class T, class ACC>
__global__ void k_avg_b(DevLevel L, BatchLevel B, int pidx, const int *skip, unsigned slice) {
    extern __shared__ __align__(16) unsigned char smem_b[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = blockIdx.x * (blockDim.x >> 5) + warp;
    if (sub >= L.nsub) { pdl_wait(); return; }
    const int K = B.K;
    const bool act = lane < K;
    unsigned char *p = smem_b + (size_t)warp * slice;
    unsigned char *rec = p;                  p += al16((size_t)L.max_nrec[pidx]);
    ACC *uc = reinterpret_cast<ACC *>(p);    p += al16(sizeof(ACC) * (size_t)(L.max_nc > 0 ? L.max_nc : 1) * 32);
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(p);
    const int nG = L.nG[sub], nc = L.ncl[sub];
    const NRecLayout lay(nG, nc, (int)sizeof(T));
    if (lane == 0) mbar_init(bar);
    __syncwarp();
    if (lane == 0 && lay.avg_bytes) {
        mbar_expect(bar, (unsigned)lay.avg_bytes);
        bulk_copy(rec, L.nrec[pidx] + L.nrecOff[pidx][sub], (unsigned)lay.avg_bytes, bar);
    }
    pdl_wait();
    pdl_trigger();
    if (skip && *skip) {
        if (lay.avg_bytes) mbar_wait(bar, 0);   // bounded: the copy lands first
        return;
    }
    if (lay.avg_bytes && !warp_wait_copy(bar, L.err, lane)) return;
    const T *Ps = reinterpret_cast<const T *>(rec + lay.psi);
    const T *wg = reinterpret_cast<const T *>(rec + lay.wg);
    const int *iG = reinterpret_cast<const int *>(rec + lay.iG);
    const int *rcs = reinterpret_cast<const int *>(rec + lay.rc);
    for (int k = 0; k < nc; ++k) uc[k * 32 + lane] = act ? from_f64<ACC>(B.ucv[(int64_t)rcs[k] * K + lane]) : (ACC)0;
    const int64_t g0 = L.offG[sub];
    for (int q0 = 0; q0 < nG; q0 += 4) {
        const int nq = nG - q0 < 4 ? nG - q0 : 4;
        ACC v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = (act && u < nq) ? reinterpret_cast<const ACC *>(B.w)[(g0 + q0 + u) * K + lane] : (ACC)0;
        for (int k = 0; k < nc; ++k) {
            const ACC ucv = uc[k * 32 + lane];
            const T *Pr = Ps + (size_t)k * lay.ld + q0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < nq) v[u] += ld<T, ACC>(Pr + u) * ucv;
        }
        if (act) {
            for (int u = 0; u < nq; ++u) {
                const int64_t e = (int64_t)iG[q0 + u] * K + lane;
                atomicAdd(&B.uB[e], to_f64(ld<T, ACC>(wg + q0 + u) * v[u]));
                B.rB[e] = 0.0;            // consumed by the substructure correction
            }
        }
    }
    if (act)
        for (int k = 0; k < nc; ++k) B.rcv[(int64_t)rcs[k] * K + lane] = 0.0;   // consumed by the coarse solve
}

// Y = A X, A dense n x n row-major (leading dimension ld, a multiple of 4,
// zero padded), X and Y interleaved [ld][K] (X zero on rows [n, ld)).  FP64;
// the FP64 pipe bounds it.  A block of NW warps owns `rpb` <= NW RPW rows;
// the columns stream in chunks of GM_C through a GM_S-stage ring of bulk
// copies (the row segments of A and the GM_C x K block of X, contiguous in
// the interleaved layout), thread 0 refilling a stage once all warps have
// used it.  Warp w computes rows RPW w .. RPW w + RPW - 1 for all K columns
// (lane k: column k), reading the A entries by broadcast.  The variant is
// chosen per problem by the autotuner (gemm_tune): eight warps with 8, 16 or
// 32 rows per block, or sixteen warps with ceil(n / SMs) rows per block, one
// block per SM, so that no SM does more rows than another.
constexpr int GM_C = 64, GM_S = 3;
__host__ __device__ constexpr size_t gm_stage(int rows) {
    return (size_t)rows * GM_C * 8 + (size_t)GM_C * 32 * 8;
}

template <int RPW, int NW>
__global__ void __launch_bounds__(32 * NW) k_gemm_b(int n, int ld, const double *A, const double *X,
                                                    double *Y, int K, int rpb, const int *skip, int *err) {
    constexpr int GR = NW * RPW;
    constexpr size_t STAGE = gm_stage(GR);
    extern __shared__ __align__(16) unsigned char smem_g[];
    __shared__ __align__(8) unsigned long long full[GM_S];
    __shared__ int ok_all;
    pdl_wait();
    pdl_trigger();
    if (skip && *skip) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = blockIdx.x * rpb;
    const int nrow = n - row0 < rpb ? n - row0 : rpb;
    const int nchunk = (ld + GM_C - 1) / GM_C;
    if (threadIdx.x == 0) {
        for (int s = 0; s < GM_S; ++s) mbar_init(&full[s]);
        ok_all = 1;
    }
    __syncthreads();
    auto issue = [&](int c) {   // thread 0: chunk c into stage c % GM_S
        unsigned char *st = smem_g + (size_t)(c % GM_S) * STAGE;
        const int c0 = c * GM_C;
        const int w = ld - c0 < GM_C ? ld - c0 : GM_C;
        const unsigned abytes = (unsigned)(w * 8), xbytes = (unsigned)((size_t)w * K * 8);
        mbar_expect(&full[c % GM_S], abytes * nrow + xbytes);
        for (int r = 0; r < nrow; ++r)
            bulk_copy(st + (size_t)r * GM_C * 8, A + (int64_t)(row0 + r) * ld + c0, abytes, &full[c % GM_S]);
        bulk_copy(st + (size_t)GR * GM_C * 8, X + (int64_t)c0 * K, xbytes, &full[c % GM_S]);
    };
    if (threadIdx.x == 0)
        for (int c = 0; c < GM_S && c < nchunk; ++c) issue(c);
    const int rw = RPW * warp;
    double sacc[RPW], tacc[RPW];
#pragma unroll
    for (int q = 0; q < RPW; ++q) { sacc[q] = 0.0; tacc[q] = 0.0; }
    for (int c = 0; c < nchunk; ++c) {
        const unsigned phase = (unsigned)((c / GM_S) & 1);
        if (!mbar_wait(&full[c % GM_S], phase)) {
            if (lane == 0) { atomicExch(err, 1); ok_all = 0; }
        }
        __syncthreads();
        if (!ok_all) break;
        const unsigned char *st = smem_g + (size_t)(c % GM_S) * STAGE;
        const double *As = reinterpret_cast<const double *>(st) + rw * GM_C;
        const double *Xs = reinterpret_cast<const double *>(st + (size_t)GR * GM_C * 8);
        const int w = ld - c * GM_C < GM_C ? ld - c * GM_C : GM_C;
        if (rw < nrow) {
            int i = 0;
            for (; i + 1 < w; i += 2) {
                const double x0 = lane < K ? Xs[i * K + lane] : 0.0;
                const double x1 = lane < K ? Xs[(i + 1) * K + lane] : 0.0;
#pragma unroll
                for (int q = 0; q < RPW; ++q) {
                    sacc[q] = fma(As[q * GM_C + i], x0, sacc[q]);
                    tacc[q] = fma(As[q * GM_C + i + 1], x1, tacc[q]);
                }
            }
            for (; i < w; ++i) {
                const double x0 = lane < K ? Xs[i * K + lane] : 0.0;
#pragma unroll
                for (int q = 0; q < RPW; ++q) sacc[q] = fma(As[q * GM_C + i], x0, sacc[q]);
            }
        }
        __syncthreads();                                   // every warp is done with the stage
        if (threadIdx.x == 0 && c + GM_S < nchunk) issue(c + GM_S);
    }
    if (!ok_all) {
        // bounded: let the copies still in flight land before the block exits
        if (threadIdx.x == 0)
            for (int s = 0; s < GM_S; ++s) mbar_wait(&full[s], 0), mbar_wait(&full[s], 1);
        return;
    }
    if (lane < K) {
#pragma unroll
        for (int q = 0; q < RPW; ++q)
            if (rw + q < nrow) Y[(int64_t)(row0 + rw + q) * K + lane] = sacc[q] + tacc[q];
    }
}

// ---------------------------------------------------------------------------
// PCG for K right-hand sides (FP64).  Blocks have K * floor(256 / K) threads
// and the grid stride is a multiple of K, so a thread always serves the same
// right-hand side k = threadIdx.x % K.
// ---------------------------------------------------------------------------
constexpr int kRB = 256;

__host__ __device__ inline int bblock(int K) { return K * (kRB / K); }

// Sum of v over the threads of each right-hand side and over the grid; the
// last block to finish calls fin(k, total) for every k < K (deterministic:
// fixed partition and order), then post() once.
template <class Fin, class Post>
__device__ void grid_reduce_k(double v, int K, double *part, unsigned *counter, Fin fin, Post post) {
    __shared__ double red[kRB];
    __shared__ bool last;
    const int per = blockDim.x / K;     // threads per right-hand side in a block
    red[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int t = 0; t < per; ++t) s += red[t * K + threadIdx.x];
        part[(int64_t)blockIdx.x * K + threadIdx.x] = s;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // thread t sums blocks b = t / K, t / K + per, ... of right-hand side t % K,
    // sixteen loads in flight (with four, the 1216 blocks of a vector kernel
    // took 38 rounds of L2 latency)
    double s = 0.0;
    if ((int)threadIdx.x < per * K) {
        const int kk = threadIdx.x % K;
        for (int b = threadIdx.x / K; b < (int)gridDim.x; b += 16 * per) {
            double u[16];
#pragma unroll
            for (int q = 0; q < 16; ++q)
                u[q] = b + q * per < (int)gridDim.x ? __ldcg(&part[(int64_t)(b + q * per) * K + kk]) : 0.0;
#pragma unroll
            for (int q = 0; q < 16; q += 4) s += (u[q] + u[q + 1]) + (u[q + 2] + u[q + 3]);
        }
    }
    red[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < K) {
        double tot = 0.0;
        for (int t = 0; t < per; ++t) tot += red[t * K + threadIdx.x];
        fin(threadIdx.x, tot);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        post();
        *counter = 0u;
    }
}

struct NoPost { __device__ void operator()() const {} };

// Tiles of kTG DOFs x K columns between the caller's layout (column k at
// src + k * ld) and the interleaved one, through shared memory: both sides are
// read and written in full rows.  (A thread per interleaved entry touched 8
// bytes of every 32-byte sector of the caller's columns: 601 us for 32 columns
// of the 1024^2 problem, where the bytes take 79.)
constexpr int kTG = 64, kTT = 256;
struct TileTr {
    double v[kMaxBatch][kTG + 1];
};
// warp w loads the columns w, w + 8, ... of the DOFs [g0, g0 + kTG)
__device__ __forceinline__ void tile_load(TileTr &t, int n, int K, const double *__restrict__ src, int64_t ld, int g0) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < kMaxBatch / (kTT / 32); ++u) {
        const int k = w + u * (kTT / 32);
        if (k < K)
#pragma unroll
            for (int h = 0; h < kTG; h += 32)
                t.v[k][h + lane] = g0 + h + lane < n ? src[(int64_t)k * ld + g0 + h + lane] : 0.0;
    }
}

__global__ void __launch_bounds__(kTT) k_b_init(int n, int K, const double *b, int64_t ldb, double *x, double *r,
                                                double *p, double *part, unsigned *counter, BatchScalars *sc,
                                                double tol, int maxit) {
    __shared__ TileTr t;
    __shared__ bool last;
    pdl_wait();
    pdl_trigger();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NW = kTT / 32, PER = kMaxBatch / NW;
    double s[PER] = {};                     // sums of squares of this warp's columns
    for (int g0 = blockIdx.x * kTG; g0 < n; g0 += gridDim.x * kTG) {
        tile_load(t, n, K, b, ldb, g0);
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int k = w + u * NW;
            if (k < K)
#pragma unroll
                for (int h = 0; h < kTG; h += 32) s[u] = fma(t.v[k][h + lane], t.v[k][h + lane], s[u]);
        }
        __syncthreads();
        const int cnt = min(kTG, n - g0) * K;
        const int64_t e0 = (int64_t)g0 * K;
        for (int q = threadIdx.x; q < cnt; q += kTT) {
            x[e0 + q] = 0.0;
            r[e0 + q] = t.v[q % K][q / K];
            p[e0 + q] = 0.0;
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        for (int o = 16; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
        const int k = w + u * NW;
        if (lane == 0 && k < K) part[(int64_t)blockIdx.x * K + k] = s[u];
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // lane k: column k; the warps share the blocks, in a fixed order
    double tot = 0.0;
    if (lane < K)
        for (int q = w; q < (int)gridDim.x; q += 8 * NW) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = q + u * NW < (int)gridDim.x ? __ldcg(&part[(int64_t)(q + u * NW) * K + lane]) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) tot += v[u];
        }
    t.v[w][lane] = tot;
    __syncthreads();
    if (w == 0 && lane < K) {
        tot = 0.0;
#pragma unroll
        for (int u = 0; u < NW; ++u) tot += t.v[u][lane];
        sc->bb[lane] = tot; sc->rr[lane] = tot; sc->tol2[lane] = tol * tol * tot;
        sc->it[lane] = 0; sc->fresh[lane] = 1; sc->beta[lane] = 0.0; sc->hold[lane] = 0; sc->mx[lane] = maxit;
        sc->conv[lane] = tot == 0.0 ? 1 : 0;
        sc->done[lane] = tot == 0.0 ? 1 : 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sc->K = K; sc->maxit = maxit; sc->step = 0;
        int all = 1;
        for (int kk = 0; kk < K; ++kk) all &= sc->done[kk];
        sc->all_done = all;
        *counter = 0u;
    }
}

// First half of a batched PCG iteration: p_new = z + beta p_old, q = A p_new
// and alpha_k = rho_k / (p_new . q).  A block owns a BT_X x BT_Y tile of nodes
// (the tile shape is chosen per problem by the autotuner, dir_spmv_tune, at the
// widest K that takes a tile)
// for all K right-hand sides; p_new is formed once per entry of the tile and
// its halo in shared memory (the FP64 pipe is the limit), from p_old in one
// direction buffer, and written to the other.
__host__ __device__ constexpr size_t bt_smem(int tx, int ty, int K) { return (size_t)(ty + 2) * (tx + 2) * K * 8; }

template <int BT_X, int BT_Y>
__global__ void k_b_dir_spmv(int nx, int K, const double *__restrict__ w, const double *__restrict__ z,
                             double *p0, double *p1, double *__restrict__ q, double *part,
                             unsigned *counter, BatchScalars *sc, double *alphas) {
    extern __shared__ __align__(16) double ps[];     // [(BT_Y + 2) * (BT_X + 2)][K]
    pdl_wait();
    pdl_trigger();
    if (sc->all_done) return;
    const int n1 = nx - 1;
    const int n = n1 * n1;
    const int tiles_x = (n1 + BT_X - 1) / BT_X;
    const int i0 = (blockIdx.x % tiles_x) * BT_X, j0 = (blockIdx.x / tiles_x) * BT_Y;
    const bool odd = sc->step & 1;
    const double *po = odd ? p1 : p0;
    double *pn = odd ? p0 : p1;
    constexpr int HX = BT_X + 2;
    const int tot = (BT_Y + 2) * HX * K;
    // eight entries per thread in flight: the loads of one round are independent
    for (int e0 = threadIdx.x; e0 < tot; e0 += 8 * blockDim.x) {
        double a[8], b[8], bt[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * blockDim.x;
            a[u] = 0.0; b[u] = 0.0; bt[u] = 0.0;
            if (e < tot) {
                const int hn = e / K, kk = e - hn * K;
                const int hy = hn / HX, hx = hn - hy * HX;
                const int i = i0 + hx - 1, j = j0 + hy - 1;
                if (i >= 0 && i < n1 && j >= 0 && j < n1) {
                    const int64_t g = (int64_t)(j * n1 + i) * K + kk;
                    a[u] = po[g]; b[u] = z[g]; bt[u] = sc->beta[kk];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * blockDim.x;
            if (e < tot) ps[e] = fma(bt[u], a[u], b[u]);
        }
    }
    __syncthreads();
    const int k = threadIdx.x % K;
    const int per = blockDim.x / K;
    const bool live = !sc->done[k] && !sc->hold[k];
    double s = 0.0;
#pragma unroll 4
    for (int ln = threadIdx.x / K; ln < BT_X * BT_Y; ln += per) {
        const int lx = ln % BT_X, ly = ln / BT_X;
        const int i = i0 + lx, j = j0 + ly;
        if (i >= n1 || j >= n1) continue;
        const int g = j * n1 + i;
        const bool W = i > 0, E = i < n1 - 1, S = j > 0, N = j < n1 - 1;
        const double *c = ps + ((ly + 1) * HX + lx + 1) * K + k;
        // neighbours outside the domain hold zero in ps; their weights are not read
        const double pc = c[0];
        double v = w[g] * pc;
        if (E) v = fma(w[n + g], c[K], v);
        if (N) v = fma(w[2 * n + g], c[HX * K], v);
        if (N && E) v = fma(w[3 * n + g], c[(HX + 1) * K], v);
        if (N && W) v = fma(w[4 * n + g], c[(HX - 1) * K], v);
        if (W) v = fma(w[n + g - 1], c[-K], v);
        if (S) v = fma(w[2 * n + g - n1], c[-HX * K], v);
        if (S && W) v = fma(w[3 * n + g - n1 - 1], c[-(HX + 1) * K], v);
        if (S && E) v = fma(w[4 * n + g - n1 + 1], c[-(HX - 1) * K], v);
        const int64_t e = (int64_t)g * K + k;
        if (live) pn[e] = pc;
        q[e] = v;
        s = fma(v, pc, s);
    }
    grid_reduce_k(s, K, part, counter,
        [&](int kk, double tot) {
            if (sc->done[kk] || sc->hold[kk]) return;
            sc->pq[kk] = tot;
            sc->alpha[kk] = sc->rho[kk] / tot;
            alphas[(int64_t)sc->it[kk] * K + kk] = sc->alpha[kk];
        }, NoPost{});
}

// The same first half for more than kMarchMinK right-hand sides (a warp costs
// the FP64 pipe the same for 21 lanes as for 32: 650 against the tile's 531 us
// for 21 right-hand sides on 1024^2, 652 against 856 for 32), a lane per
// right-hand side and no tile: each warp marches up a strip of MW columns with
// three rows of p_new in registers, so nothing meets at a barrier, and the
// strips are cut into as many equal segments as there are resident warps (one
// wave).  The FP64 pipe bounds it: per node 9 products, 1 for the dot product
// and (MW + 2) / MW (and two rows per segment) for p_new, 11.4 in all, as with
// the tiles; those left a last wave of blocks partly filled and met at the
// end of their load phases.  Every weight read is in range (a missing
// neighbour's p_new is zero and reads a finite weight), so the products need
// no predicates, and their order is the tile kernel's: q is the same bit for
// bit.  32 right-hand sides: the 1024^2 three-level solve (46 iterations)
// 101 -> 92 ms (the kernel 856 -> 652 us), the 512^2 FP64 solve 75.6 -> 72.5 ms.
constexpr int MW = 8, kMarchT = 256, kMarchPerSm = 2;
__global__ void __launch_bounds__(kMarchT, kMarchPerSm)
k_b_dir_march(int nx, int K, const double *__restrict__ w, const double *__restrict__ z, double *p0, double *p1,
              double *__restrict__ q, double *part, unsigned *counter, BatchScalars *sc, double *alphas, int strips,
              int rows) {
    __shared__ double red[kMarchT / 32][32];
    __shared__ bool last;
    if (sc->all_done) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n1 = nx - 1;
    const int64_t n = (int64_t)n1 * n1;
    const bool odd = sc->step & 1;
    const double *__restrict__ po = odd ? p1 : p0;
    double *__restrict__ pn = odd ? p0 : p1;
    const bool act = lane < K;
    const int k = act ? lane : 0;
    const bool live = act && !sc->done[k] && !sc->hold[k];
    const double bt = sc->beta[k];
    const int unit = blockIdx.x * (kMarchT / 32) + warp;
    const int i0 = (unit % strips) * MW, j0 = (unit / strips) * rows;
    const int j1 = min(n1, j0 + rows);
    double s = 0.0;
    if (j0 < n1) {
        double A[MW + 2], B[MW + 2];
        auto fetch = [&](int j) {          // p_old and z of row j, zero outside the domain
#pragma unroll
            for (int c = 0; c < MW + 2; ++c) {
                const int i = i0 + c - 1;
                const bool in = act && j >= 0 && j < n1 && i >= 0 && i < n1;
                const int64_t g = ((int64_t)j * n1 + i) * K + k;
                A[c] = in ? po[g] : 0.0;
                B[c] = in ? z[g] : 0.0;
            }
        };
        auto form = [&](double (&R)[MW + 2]) {
#pragma unroll
            for (int c = 0; c < MW + 2; ++c) R[c] = fma(bt, A[c], B[c]);
        };
        // row j (C) from the rows below and above (S, N); forms N and fetches row j + 2
        auto step = [&](int j, const double (&S)[MW + 2], const double (&C)[MW + 2], double (&N)[MW + 2]) {
            form(N);
            if (j + 1 < j1) fetch(j + 2);
            const double *wr = w + (int64_t)j * n1 + i0;
#pragma unroll
            for (int c = 0; c < MW; ++c) {
                if (i0 + c >= n1) break;
                const double *wc = wr + c;
                double v = __ldg(wc) * C[c + 1];
                v = fma(__ldg(wc + n), C[c + 2], v);                    // E
                v = fma(__ldg(wc + 2 * n), N[c + 1], v);                // N
                v = fma(__ldg(wc + 3 * n), N[c + 2], v);                // NE
                v = fma(__ldg(wc + 4 * n), N[c], v);                    // NW
                v = fma(__ldg(wc + n - 1), C[c], v);                    // W
                v = fma(__ldg(wc + 2 * n - n1), S[c + 1], v);           // S
                v = fma(__ldg(wc + 3 * n - n1 - 1), S[c], v);           // SW
                v = fma(__ldg(wc + 4 * n - n1 + 1), S[c + 2], v);       // SE
                const int64_t e = ((int64_t)j * n1 + i0 + c) * K + k;
                if (live) pn[e] = C[c + 1];
                if (act) q[e] = v;
                s = fma(v, C[c + 1], s);
            }
        };
        double P0[MW + 2], P1[MW + 2], P2[MW + 2];
        fetch(j0 - 1);
        form(P0);
        fetch(j0);
        form(P1);
        fetch(j0 + 1);
        for (int j = j0; j < j1; j += 3) {
            step(j, P0, P1, P2);
            if (j + 1 < j1) step(j + 1, P1, P2, P0);
            if (j + 2 < j1) step(j + 2, P2, P0, P1);
        }
    }
    // block partials, added over the blocks in a fixed order by the last block
    red[warp][lane] = s;
    __syncthreads();
    constexpr int NWM = kMarchT / 32;
    if (warp == 0 && act) {
        double t = 0.0;
#pragma unroll
        for (int u = 0; u < NWM; ++u) t += red[u][lane];
        part[(int64_t)blockIdx.x * K + lane] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t = 0.0;
    if (act)
        for (int b = warp; b < (int)gridDim.x; b += 8 * NWM) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = b + u * NWM < (int)gridDim.x ? __ldcg(&part[(int64_t)(b + u * NWM) * K + lane]) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) t += v[u];
        }
    red[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && act) {
        double tot = 0.0;
#pragma unroll
        for (int u = 0; u < NWM; ++u) tot += red[u][lane];
        if (!sc->done[lane] && !sc->hold[lane]) {
            sc->pq[lane] = tot;
            sc->alpha[lane] = sc->rho[lane] / tot;
            alphas[(int64_t)sc->it[lane] * K + lane] = sc->alpha[lane];
        }
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// x += alpha p; r -= alpha q; rr_k; convergence; it_k += 1
__global__ void k_b_update(int64_t nK, int K, double *__restrict__ x, double *__restrict__ r,
                           const double *p0, const double *p1, const double *__restrict__ q,
                           double *part, unsigned *counter, BatchScalars *sc) {
    pdl_wait();
    pdl_trigger();
    if (sc->all_done) return;
    const double *__restrict__ p = (sc->step & 1) ? p0 : p1;   // p_new of this step
    const int k = threadIdx.x % K;
    const bool live = !sc->done[k] && !sc->hold[k];
    const double a = sc->alpha[k];
    double s = 0.0;
    if (live) {
        for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nK; e += (int64_t)gridDim.x * blockDim.x) {
            x[e] = fma(a, p[e], x[e]);
            const double ri = fma(-a, q[e], r[e]);
            r[e] = ri;
            s = fma(ri, ri, s);
        }
    }
    grid_reduce_k(s, K, part, counter,
        [&](int kk, double tot) {
            if (sc->done[kk] || sc->hold[kk]) return;
            sc->rr[kk] = tot;
            sc->it[kk] += 1;
            sc->last[kk] = sc->step;
            if (tot <= sc->tol2[kk]) { sc->conv[kk] = 1; sc->done[kk] = 1; }
            if (sc->it[kk] >= sc->mx[kk]) sc->done[kk] = 1;
        },
        [&]() {
            int all = 1;
            for (int kk = 0; kk < K; ++kk) all &= sc->done[kk];
            sc->all_done = all;
            sc->step += 1;   // every block has read step before the last one gets here
        });
}

// res = b - A x (b in the caller's layout, column k at b + k * ldb)
__global__ void k_b_residual(int nx, int K, const double *w, const double *b, int64_t ldb,
                             const double *x, double *res) {
    const int n1 = nx - 1;
    const int n = n1 * n1;
    const int64_t nK = (int64_t)n * K;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nK) return;
    const int k = (int)(e % K);
    const int g = (int)(e / K);
    const int jj = g / n1, ii = g - jj * n1;
    const bool W = ii > 0, E = ii < n1 - 1, S = jj > 0, N = jj < n1 - 1;
    auto X = [&](int gg) { return x[(int64_t)gg * K + k]; };
    double v = w[g] * X(g);
    if (E) v = fma(w[n + g], X(g + 1), v);
    if (N) v = fma(w[2 * n + g], X(g + n1), v);
    if (N && E) v = fma(w[3 * n + g], X(g + n1 + 1), v);
    if (N && W) v = fma(w[4 * n + g], X(g + n1 - 1), v);
    if (W) v = fma(w[n + g - 1], X(g - 1), v);
    if (S) v = fma(w[2 * n + g - n1], X(g - n1), v);
    if (S && W) v = fma(w[3 * n + g - n1 - 1], X(g - n1 - 1), v);
    if (S && E) v = fma(w[4 * n + g - n1 + 1], X(g - n1 + 1), v);
    res[e] = b[(int64_t)k * ldb + g] - v;
}

__global__ void k_b_norm2(int64_t nK, int K, const double *v, double *part, unsigned *counter,
                          double *out) {
    const int k = threadIdx.x % K;
    (void)k;
    double s = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nK; e += (int64_t)gridDim.x * blockDim.x)
        s = fma(v[e], v[e], s);
    grid_reduce_k(s, K, part, counter, [&](int kk, double tot) { out[kk] = tot; }, NoPost{});
}


// dst[g * K + k] = src[k * ld + g] and back
__global__ void __launch_bounds__(kTT) k_b_gather(int n, int K, const double *src, int64_t ld, double *dst) {
    __shared__ TileTr t;
    const int g0 = blockIdx.x * kTG;
    tile_load(t, n, K, src, ld, g0);
    __syncthreads();
    const int cnt = min(kTG, n - g0) * K;
    for (int q = threadIdx.x; q < cnt; q += kTT) dst[(int64_t)g0 * K + q] = t.v[q % K][q / K];
}
__global__ void __launch_bounds__(kTT) k_b_scatter(int n, int K, const double *src, double *dst, int64_t ld) {
    __shared__ TileTr t;
    const int g0 = blockIdx.x * kTG, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cnt = min(kTG, n - g0) * K;
    for (int q = threadIdx.x; q < cnt; q += kTT) t.v[q % K][q / K] = src[(int64_t)g0 * K + q];
    __syncthreads();
    for (int k = w; k < K; k += kTT / 32)
#pragma unroll
        for (int h = 0; h < kTG; h += 32)
            if (g0 + h + lane < n) dst[(int64_t)k * ld + g0 + h + lane] = t.v[k][h + lane];
}

// A new right-hand side in slot k of a running batch.  p: the direction buffer
// that the slot reads when it joins, cleared if the slot's last right-hand side
// may have left a NaN there (beta = 0 would keep it), else null.
__global__ void k_b_admit(int n, int K, int k, const double *__restrict__ b, double *x, double *r, double *p,
                          double *part, unsigned *counter, BatchScalars *sc, double tol, int maxit) {
    double s = 0.0;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
        const double v = b[g];
        x[(int64_t)g * K + k] = 0.0;
        r[(int64_t)g * K + k] = v;
        if (p) p[(int64_t)g * K + k] = 0.0;
        s = fma(v, v, s);
    }
    grid_reduce_k(s, 1, part, counter,
        [&](int, double tot) {
            sc->bb[k] = tot; sc->rr[k] = tot; sc->tol2[k] = tol * tol * tot;
            sc->it[k] = 0; sc->fresh[k] = 1; sc->beta[k] = 0.0; sc->mx[k] = maxit;
            sc->conv[k] = tot == 0.0 ? 1 : 0;
            sc->done[k] = tot == 0.0 ? 1 : 0;
            sc->hold[k] = tot == 0.0 ? 0 : 1;
        },
        [&]() {
            if (!sc->done[k]) sc->all_done = 0;
        });
}

__global__ void k_b_column(int n, int K, int k, const double *x, double *dst) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) dst[g] = x[(int64_t)g * K + k];
}

__global__ void k_b_move_column(int n, int K, int k, const double *src, double *dst) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) dst[(int64_t)g * K + k] = src[(int64_t)g * K + k];
}

// Both integer-operation conversions against the hardware ones, bit for bit
// (NaN results compared as NaN).
// FP64 fused multiply-add rate: kFmaChains independent chains per thread, so
// that neither latency nor issue of anything else limits the FP64 pipe.  The
// sum is written only if it takes a value it cannot reach (it keeps the
// chains live).  Launched kFmaBlocksPerSm x SMs blocks of 256 threads.
constexpr int kFmaChains = 8;
__global__ void __launch_bounds__(256) k_fp64_rate(int iters, double b, double c, double *out) {
    double a[kFmaChains];
#pragma unroll
    for (int j = 0; j < kFmaChains; ++j) a[j] = 1e-3 * threadIdx.x + j;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int j = 0; j < kFmaChains; ++j) a[j] = fma(a[j], b, c);
    }
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < kFmaChains; ++j) s += a[j];
    if (s == -1.0) out[0] = s;
}

__global__ void k_selftest_convert(const double *d, int64_t n, unsigned long long *bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = d[i];
    const float a = f64_to_f32(v), b = __double2float_rn(v);
    const bool nan1 = a != a && b != b;
    if (!nan1 && __float_as_uint(a) != __float_as_uint(b)) atomicAdd(bad, 1ull);
    // every low word, read as a binary32, widened
    const float f = __uint_as_float((unsigned)__double2loint(v));
    const double x = f32_to_f64(f), y = (double)f;
    const bool nan2 = x != x && y != y;
    if (!nan2 && __double_as_longlong(x) != __double_as_longlong(y)) atomicAdd(bad, 1ull);
}

constexpr size_t kSmemMaxB = 227 * 1024;

int num_sms_b() { return device_sms(); }

int warps_b(int nsub, size_t slice) {
    const int fit = (int)(kSmemMaxB / slice);
    int want = (nsub + num_sms_b() - 1) / num_sms_b();
    if (want < 1) want = 1;
    int w = want < fit ? want : fit;
    if (w > 8) w = 8;
    return w < 1 ? 1 : w;
}

int pidx_b(int prec) { return prec == BDDC_PREC_FP64 ? 0 : (prec == BDDC_PREC_FP32 ? 1 : 2); }

template <class T, class ACC, int BP>
void dir_b_launch(const DevLevel &L, const BatchLevel &B, bool post, const double *r, double *z,
                  const int *skip, cudaStream_t s, const RzBatch *rz) {
    const size_t sm = DirSmemB<T, ACC, BP>::bytes(L);
    const RzBatch none{nullptr, nullptr, nullptr, nullptr};
    constexpr int nt = 32 * lanes_per_rhs<BP>();
    if (!post) launch_plain(k_dir_b<T, ACC, BP, false>, L.nsub, nt, sm, s, L, B, r, z, skip, none);
    else launch_plain(k_dir_b<T, ACC, BP, true>, L.nsub, nt, sm, s, L, B, r, z, skip, rz ? *rz : none);
}

template <class T, class ACC>
void dir_b(const DevLevel &L, const BatchLevel &B, bool post, const double *r, double *z,
           const int *skip, cudaStream_t s, const RzBatch *rz = nullptr) {
    if (L.bp == 8) dir_b_launch<T, ACC, 8>(L, B, post, r, z, skip, s, rz);
    else if (L.bp == 16) dir_b_launch<T, ACC, 16>(L, B, post, r, z, skip, s, rz);
    else dir_b_launch<T, ACC, 32>(L, B, post, r, z, skip, s, rz);
}

// The lane-per-right-hand-side kernel (k_dir_ls) takes uniform blocks of 8 or
// 16 rows.
template <class T, class ACC> size_t lane_total(const DevLevel &L, int w) {
    return L.bp == 8 ? LaneSmem<T, ACC, 8>::of(L, w).total : LaneSmem<T, ACC, 16>::of(L, w).total;
}
// Warps of a block: one wave of blocks, up to the most that the kernel and
// the shared memory take.
template <class T, class ACC> int lane_warps(const DevLevel &L) {
    const int most = L.bp == 8 ? ls_max_warps<ACC, 8>() : ls_max_warps<ACC, 16>();
    int w = std::min(most, std::max(1, (L.nsub + num_sms_b() - 1) / num_sms_b()));
    while (w > 1 && lane_total<T, ACC>(L, w) > kSmemMaxB) --w;
    return w;
}
template <class T, class ACC> size_t lane_smem(const DevLevel &L) {
    if (!(L.bp == 8 || L.bp == 16) || !L.irec) return 0;
    if (L.max_m + 1 > 32 * L.bp) return 0;   // the sort's block counts live in the block buffer
    return lane_total<T, ACC>(L, lane_warps<T, ACC>(L));
}

template <class T, class ACC>
void dir_ls(const DevLevel &L, const BatchLevel &B, bool post, const double *r, double *z, const int *skip,
            cudaStream_t s, const RzBatch *rz = nullptr) {
    if (!B.ys) throw Error(BDDC_E_STATE, "lane Dirichlet kernel without its scratch");
    const RzBatch none{nullptr, nullptr, nullptr, nullptr};
    const RzBatch rzv = (post && rz) ? *rz : none;
    const int W = lane_warps<T, ACC>(L);
    const auto k8 = L.sub_tri ? (post ? k_dir_ls<T, ACC, 8, true, true> : k_dir_ls<T, ACC, 8, false, true>)
                              : (post ? k_dir_ls<T, ACC, 8, true, false> : k_dir_ls<T, ACC, 8, false, false>);
    const auto k16 = L.sub_tri ? (post ? k_dir_ls<T, ACC, 16, true, true> : k_dir_ls<T, ACC, 16, false, true>)
                               : (post ? k_dir_ls<T, ACC, 16, true, false> : k_dir_ls<T, ACC, 16, false, false>);
    launch_plain(L.bp == 8 ? k8 : k16, (L.nsub + W - 1) / W, 32 * W, lane_smem<T, ACC>(L), s, L, B, r, z, skip, rzv);
}

template <class T, class ACC>
void neu_b(const DevLevel &L, const BatchLevel &B, int prec, const double *r, const int *skip,
           cudaStream_t s) {
    const int pi = pidx_b(prec);
    const size_t slice = al16(al16((size_t)L.max_nrec[pi]) +
                              al16(sizeof(ACC) * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32) + 16);
    const int wpc = warps_b(L.nsub, slice);
    launch_plain(k_neu_b<T, ACC>, (L.nsub + wpc - 1) / wpc, 32 * wpc, slice * wpc, s, L, B, pi, r, skip,
               (unsigned)slice);
}

template <class T, class ACC>
void avg_b(const DevLevel &L, const BatchLevel &B, int prec, const int *skip, cudaStream_t s) {
    const int pi = pidx_b(prec);
    const size_t slice = al16(al16((size_t)L.max_nrec[pi]) +
                              al16(sizeof(ACC) * (size_t)(L.max_nc > 0 ? L.max_nc : 1) * 32) + 16);
    const int wpc = warps_b(L.nsub, slice);
    launch_plain(k_avg_b<T, ACC>, (L.nsub + wpc - 1) / wpc, 32 * wpc, slice * wpc, s, L, B, pi, skip,
               (unsigned)slice);
}

// Warps of a block: one per tile of eight rows of the largest interface, at
// most kNBW; and tiles per warp, so that the interfaces of up to 192 (FP64:
// 128) DOFs take one pass over N.
int neu_warps(const DevLevel &L) {
    const int t = (L.max_nG + 7) / 8;
    return t < 1 ? 1 : (t > kNBW ? kNBW : t);
}
// The form of a launch: the chunk asked for (tuned, in the context's precision
// then) where the level fits with it in this precision, else the largest of
// 32, 16 and 8 KB that fits, with the record staged if possible; chunk 0: none.
struct NeuForm { int chunk; bool head; };
template <class T, class ACC> NeuForm neu_form(const DevLevel &L, int asked) {
    for (bool head : {true, false})
        for (int c : {head ? asked : 0, kChunkBytes, kChunkBytes / 2, kChunkBytes / 4})
            if (c > 0 && neu_bg_smem<T, ACC>(L, c, head) <= kSmemMaxB) return {c, head};
    return {0, false};
}
template <class T, class ACC>
void neu_bg(const DevLevel &L, const BatchLevel &B, int prec, const double *r, const int *skip, cudaStream_t s) {
    const int nw = neu_warps(L), rt = ((L.max_nG + 7) / 8 + nw - 1) / nw;
    const NeuForm F = neu_form<T, ACC>(L, B.chunk);
    // without the staged record, interfaces that need all tiles of a warp only
    constexpr int most = sizeof(ACC) == 8 ? 2 : 3;
    const auto kern = !F.head                     ? k_neu_bg<T, ACC, most, false>
                      : rt <= 1                   ? k_neu_bg<T, ACC, 1, true>
                      : rt == 2 || most == 2      ? k_neu_bg<T, ACC, 2, true>
                                                  : k_neu_bg<T, ACC, 3, true>;
    launch_plain(kern, L.nsub, 32 * nw, neu_bg_smem<T, ACC>(L, F.chunk, F.head), s, L, B, pidx_b(prec), r, skip, F.chunk);
}
template <class T, class ACC>
void avg_bg(const DevLevel &L, const BatchLevel &B, int prec, const int *skip, cudaStream_t s) {
    launch_plain(k_avg_bg<T, ACC>, L.nsub, 32 * neu_warps(L), avg_bg_smem<T, ACC>(L), s, L, B, pidx_b(prec), skip);
}

template <class T, class ACC> size_t dir_slice_b(const DevLevel &L) {
    if (L.bp == 8) return DirSmemB<T, ACC, 8>::bytes(L);
    if (L.bp == 16) return DirSmemB<T, ACC, 16>::bytes(L);
    return DirSmemB<T, ACC, 32>::bytes(L);
}

int vgrid_b(int64_t nK, int K) {
    const int bd = bblock(K);
    int64_t g = (nK + 4 * (int64_t)bd - 1) / (4 * (int64_t)bd);
    const int cap = 8 * num_sms_b() < kMaxVecGrid ? 8 * num_sms_b() : kMaxVecGrid;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

namespace {

// Which batch kernels a level uses: the staged kernels when the operators
// fit in shared memory, else the streaming Dirichlet kernel and the chunked
// Neumann / averaging kernels.  A staged Neumann / averaging record must also
// leave room for three substructures per SM: with fewer warps resident the
// warp-per-substructure kernels wait on latency, and the block-per-
// substructure kernels are faster.
struct BatchRoute {
    bool dir_staged = false, neu_staged = false, avg_staged = false;
    bool dir_stream = false;   // the streaming Dirichlet kernel
    bool stream_fits = false, bg_fits = false;   // the streaming / chunked kernels could run
    bool pre_tc = false, post_tc = false;   // the tensor-core products (tc_kernels.cu)
    bool lane_fits = false, dir_lane = false;   // the lane-per-right-hand-side Dirichlet kernel
    bool ok = false;
};

// Bit of DevLevel::route_pref that selects the lane-per-right-hand-side
// Dirichlet kernel in precision index pi.
constexpr int lane_bit(int pi) { return 1 << (6 + pi); }

// BDDC_BATCH_STREAM=1 routes every level that the streaming / chunked
// kernels can take to them, also where the staged kernels fit (read when a
// batch is launched or captured).
bool force_stream() {
    const char *e = std::getenv("BDDC_BATCH_STREAM");
    return e && e[0] == '1';
}

template <class T, class ACC> BatchRoute route_t(const DevLevel &L, int prec) {
    BatchRoute R;
    const int pi = pidx_b(prec);
    const size_t a = sizeof(ACC);
    R.dir_staged = (L.bp == 8 || L.bp == 16 || L.bp == 32) && L.irec && dir_slice_b<T, ACC>(L) <= kSmemMaxB;
    R.neu_staged = 3 * (al16((size_t)L.max_nrec[pi]) + al16(a * (size_t)(L.max_nG > 0 ? L.max_nG : 1) * 32) + 16) <= kSmemMaxB;
    R.avg_staged = 3 * (al16((size_t)L.max_nrec[pi]) + al16(a * (size_t)(L.max_nc > 0 ? L.max_nc : 1) * 32) + 16) <= kSmemMaxB;
    // the largest bucket's layout bounds every bucket's
    const int nw_max = ((L.max_b + 1) / 2 + 3) / 4;
    const bool stream = L.bk.n > 0 && L.bperm && nw_max <= kMaxBuckets &&
                        StreamSmemB::of<T, ACC>(L, 32 * nw_max).total <= kSmemMaxB;
    const bool bg = neu_form<T, ACC>(L, 0).chunk > 0 && avg_bg_smem<T, ACC>(L) <= kSmemMaxB;
    R.dir_stream = !R.dir_staged && stream;
    R.stream_fits = stream;
    R.bg_fits = bg;
    const bool pdir = (L.route_pref >> (2 * pi)) & 1, pneu = (L.route_pref >> (2 * pi + 1)) & 1;
    if ((force_stream() || pdir) && stream) R.dir_staged = false, R.dir_stream = true;
    if ((force_stream() || pneu) && bg) R.neu_staged = R.avg_staged = false;
    R.pre_tc = tc_route(L, prec, false);
    R.post_tc = tc_route(L, prec, true);
    const size_t ls = lane_smem<T, ACC>(L);
    R.lane_fits = ls > 0 && ls <= kSmemMaxB;
    R.dir_lane = R.lane_fits && (L.route_pref & lane_bit(pi));
    if (const char *e = std::getenv("BDDC_DIR_LANE")) {   // "1" / "0": the lane kernel where it fits, or never
        if (e[0] == '1') R.dir_lane = R.lane_fits && batch_lane(L);
        if (e[0] == '0') R.dir_lane = false;
    }
    if (R.dir_lane) R.dir_staged = R.dir_stream = false;
    R.ok = (R.dir_staged || R.dir_stream || R.dir_lane || (R.pre_tc && R.post_tc)) && (R.neu_staged || bg) && (R.avg_staged || bg);
    return R;
}

BatchRoute route(const DevLevel &L, int prec) {
    if (prec == BDDC_PREC_FP64) return route_t<double, double>(L, prec);
    if (prec == BDDC_PREC_FP32) return route_t<float, float>(L, prec);
    return route_t<__nv_bfloat16, float>(L, prec);
}

}  // namespace

bool batch_path(const DevLevel &L, int prec) { return route(L, prec).ok; }

bool batch_lane(const DevLevel &L) {
    auto fits = [](size_t b) { return b > 0 && b <= kSmemMaxB; };
    return fits(lane_smem<float, float>(L)) || fits(lane_smem<__nv_bfloat16, float>(L)) || fits(lane_smem<double, double>(L));
}

bool batch_streams(const DevLevel &L) {
    for (int prec : {BDDC_PREC_FP64, BDDC_PREC_FP32, BDDC_PREC_BF16}) {
        const BatchRoute R = route(L, prec);
        if (R.ok && (R.dir_stream || R.stream_fits)) return true;
    }
    return false;
}

namespace {

// Resident blocks per SM of a kernel at a block size and shared-memory size,
// queried once and cached: the query may load the kernel's module, which a
// stream capture does not allow, so batch_prepare_level asks for every
// bucket before the first capture and a capturing stream only reads the
// cache (an entry missing there gives one block per SM).
int resident_blocks(const void *kern, int nt, size_t sm, cudaStream_t s) {
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, size_t>, int> cache;
    const auto key = std::make_tuple(kern, nt, sm);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
    }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (s && cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) return 1;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, nt, sm) != cudaSuccess || per < 1) {
        cudaGetLastError();
        per = 1;
    }
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = per;
    return per;
}

// The buckets one after another on s, or (B.bucket_par) at once: bucket 0
// on s, the others on the fork's streams, joined back into s.
template <class T, class ACC, bool SWZ, bool POST>
void dir_bs_buckets(const DevLevel &L, const BatchLevel &B, const double *r, double *z, const int *skip,
                    const RzBatch &rz, cudaStream_t s, bool launch = true) {
    const BucketFork *F = (launch && B.bucket_par && B.fork && L.bk.n > 1) ? B.fork : nullptr;
    if (F) BDDC_CUDA_TRY(cudaEventRecord(F->fork, s));
    for (int i = 0; i < L.bk.n; ++i) {
        DevLevel Lb = L;                  // the bucket's maxima size its shared memory
        Lb.max_b = L.bk.max_b[i];
        Lb.max_ld = L.bk.max_ld[i];
        Lb.max_nG = L.bk.max_nG[i];
        // the bucket's warps are those of two rows a thread
        const int nt = bs_rows<ACC>() == 2 ? 32 * L.bk.nw[i] : 32 * ((L.bk.nw[i] + 1) / 2);
        const size_t sm = StreamSmemB::of<T, ACC>(Lb, nt).total;
        auto kern = k_dir_bs<T, ACC, SWZ, POST, kSBMaxT>;
        if constexpr (sizeof(ACC) == 4)       // (FP64 wants the 128 registers)
            if (nt <= kSBSmallT) kern = k_dir_bs<T, ACC, SWZ, POST, kSBSmallT>;
        const int per = resident_blocks(reinterpret_cast<const void *>(kern), nt, sm, s);
        if (!launch) continue;
        const int grid = std::min(L.bk.count[i], per * num_sms_b());
        cudaStream_t si = s;
        if (F && i > 0) {
            si = F->st[i - 1];
            BDDC_CUDA_TRY(cudaStreamWaitEvent(si, F->fork, 0));
        }
        launch_plain(kern, grid, nt, sm, si, Lb, B, r, z, skip, rz,
                     (const int *)(L.bperm + L.bk.first[i]), L.bk.count[i]);
        if (F && i > 0) BDDC_CUDA_TRY(cudaEventRecord(F->join[i - 1], si));
    }
    if (F)
        for (int i = 1; i < L.bk.n; ++i) BDDC_CUDA_TRY(cudaStreamWaitEvent(s, F->join[i - 1], 0));
}

template <class T, class ACC> void prepare_bs(const DevLevel &L) {
    const RzBatch none{nullptr, nullptr, nullptr, nullptr};
    const BatchLevel B;
    if (L.bp != 0) {
        dir_bs_buckets<T, ACC, true, false>(L, B, nullptr, nullptr, nullptr, none, nullptr, false);
        dir_bs_buckets<T, ACC, true, true>(L, B, nullptr, nullptr, nullptr, none, nullptr, false);
    } else {
        dir_bs_buckets<T, ACC, false, false>(L, B, nullptr, nullptr, nullptr, none, nullptr, false);
        dir_bs_buckets<T, ACC, false, true>(L, B, nullptr, nullptr, nullptr, none, nullptr, false);
    }
}

template <class T, class ACC>
void dir_bs(const DevLevel &L, const BatchLevel &B, bool post, const double *r, double *z, const int *skip,
            const RzBatch *rz, cudaStream_t s) {
    if (!B.ys) throw Error(BDDC_E_STATE, "streaming Dirichlet kernel without its scratch");
    const RzBatch none{nullptr, nullptr, nullptr, nullptr};
    const RzBatch rzv = (post && rz) ? *rz : none;
    const bool swz = L.bp != 0;
    if (swz) {
        if (post) dir_bs_buckets<T, ACC, true, true>(L, B, r, z, skip, rzv, s);
        else dir_bs_buckets<T, ACC, true, false>(L, B, r, z, skip, rzv, s);
    } else {
        if (post) dir_bs_buckets<T, ACC, false, true>(L, B, r, z, skip, rzv, s);
        else dir_bs_buckets<T, ACC, false, false>(L, B, r, z, skip, rzv, s);
    }
}

// Whether a level whose route is the lane kernel uses it for this batch.
template <class ACC> bool lane_wide(const DevLevel &L, const BatchRoute &R, const BatchLevel &B) {
    return sizeof(ACC) == 4 || fp64_lane_at(B.K, L.bp, L.nsub, num_sms_b(), R.stream_fits);
}

template <class T, class ACC>
void pre_b(const DevLevel &L, const BatchLevel &B, int prec, const double *r, const int *skip, cudaStream_t s,
           cudaEvent_t *ev) {
    const BatchRoute R = route_t<T, ACC>(L, prec);
    if (ev) cudaEventRecord(ev[0], s);
    if (R.pre_tc) tc_dir_b(L, B, prec, false, r, nullptr, skip, nullptr, s);
    else if (R.dir_lane && lane_wide<ACC>(L, R, B)) dir_ls<T, ACC>(L, B, false, r, nullptr, skip, s);
    else if (R.dir_staged) dir_b<T, ACC>(L, B, false, r, nullptr, skip, s);
    else dir_bs<T, ACC>(L, B, false, r, nullptr, skip, nullptr, s);
    if (ev) cudaEventRecord(ev[1], s);
    if (R.neu_staged) neu_b<T, ACC>(L, B, prec, r, skip, s);
    else neu_bg<T, ACC>(L, B, prec, r, skip, s);
    if (ev) cudaEventRecord(ev[2], s);
}

template <class T, class ACC>
void post_b(const DevLevel &L, const BatchLevel &B, int prec, const double *r, double *z, const int *skip,
            cudaStream_t s, cudaEvent_t *ev, const RzBatch *rz) {
    const BatchRoute R = route_t<T, ACC>(L, prec);
    if (ev) cudaEventRecord(ev[0], s);
    if (R.avg_staged) avg_b<T, ACC>(L, B, prec, skip, s);
    else avg_bg<T, ACC>(L, B, prec, skip, s);
    if (ev) cudaEventRecord(ev[1], s);
    if (R.post_tc) tc_dir_b(L, B, prec, true, r, z, skip, rz, s);
    else if (R.dir_lane && lane_wide<ACC>(L, R, B)) dir_ls<T, ACC>(L, B, true, r, z, skip, s, rz);
    else if (R.dir_staged) dir_b<T, ACC>(L, B, true, r, z, skip, s, rz);
    else dir_bs<T, ACC>(L, B, true, r, z, skip, rz, s);
    if (ev) cudaEventRecord(ev[2], s);
}

}  // namespace

namespace {

// mean ms of three runs of f after one untimed
template <class F> double time3(cudaStream_t s, F &&f) {
    cudaEvent_t e0, e1;
    BDDC_CUDA_TRY(cudaEventCreate(&e0));
    BDDC_CUDA_TRY(cudaEventCreate(&e1));
    f();
    BDDC_CUDA_TRY(cudaEventRecord(e0, s));
    for (int i = 0; i < 3; ++i) f();
    BDDC_CUDA_TRY(cudaEventRecord(e1, s));
    BDDC_CUDA_TRY(cudaEventSynchronize(e1));
    float ms = 0.0f;
    BDDC_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ms / 3.0;
}

// staged against streaming / chunked routes of one precision (L.route_pref)
template <class T, class ACC>
void tune_route_t(DevLevel &L, BatchLevel &B, int prec, const double *r, double *z, cudaStream_t s) {
    const int pi = pidx_b(prec);
    const char *forced = std::getenv("BDDC_ROUTE");   // "staged" or "stream": no timing
    if (const char *bits = std::getenv("BDDC_ROUTE_PREF")) {   // the route bits themselves, every level
        L.route_pref = std::atoi(bits);
        return;
    }
    auto steps = [&] {            // the level's pre- and post-correction steps
        pre_b<T, ACC>(L, B, prec, r, nullptr, s, nullptr);
        post_b<T, ACC>(L, B, prec, r, z, nullptr, s, nullptr, nullptr);
    };
    {
        // Dirichlet kernel: staged, lane per right-hand side, or streaming,
        // among those that fit
        const int sbit = 1 << (2 * pi), lbit = lane_bit(pi);
        L.route_pref &= ~(sbit | lbit);
        const BatchRoute R0 = route_t<T, ACC>(L, prec);
        if (R0.dir_staged && !(R0.pre_tc && R0.post_tc)) {
            int cand[3] = {0, 0, 0}, nc = 0;
            const bool lane = R0.lane_fits && B.ys, stream = R0.stream_fits && B.ys;
            if (prec != BDDC_PREC_FP64 || !lane || fp64_staged_timed(L.bp, L.nsub, num_sms_b(), stream)) cand[nc++] = 0;
            if (lane) cand[nc++] = lbit;
            if (stream) cand[nc++] = sbit;
            int pick = forced ? 0 : cand[0];
            if (forced) {
                if (forced[0] == 's' && forced[1] == 't' && forced[2] == 'r' && stream) pick = sbit;
            } else if (nc > 1) {
                double best = 1e30;
                for (int i = 0; i < nc; ++i) {
                    L.route_pref = (L.route_pref & ~(sbit | lbit)) | cand[i];
                    const double t = time3(s, steps);
                    if (t < best) best = t, pick = cand[i];
                }
            }
            L.route_pref = (L.route_pref & ~(sbit | lbit)) | pick;
        }
    }
    {
        // Neumann and averaging kernels: staged or chunked
        const int bit = 1 << (2 * pi + 1);
        L.route_pref &= ~bit;
        const BatchRoute R0 = route_t<T, ACC>(L, prec);
        if ((R0.neu_staged || R0.avg_staged) && R0.bg_fits) {
            if (forced) {
                if (forced[0] == 's' && forced[1] == 't' && forced[2] == 'r') L.route_pref |= bit;
            } else {
                double t[2];
                for (int v = 0; v < 2; ++v) {
                    if (v) L.route_pref |= bit;
                    else L.route_pref &= ~bit;
                    t[v] = time3(s, steps);
                }
                if (t[1] < t[0]) L.route_pref |= bit;
                else L.route_pref &= ~bit;
            }
        }
    }
}

template <class T, class ACC> void tune_t(const DevLevel &L, BatchLevel &B, int prec, const double *r, double *z,
                                       cudaStream_t s) {
    const BatchRoute R = route_t<T, ACC>(L, prec);
    // The streaming kernel's buckets, for the correction that takes it (FP32
    // levels with a tensor-core pre-correction stream the post-correction only;
    // sixteen large level-2 substructures in three buckets: 318 us one after
    // another, 128 the longest).
    const bool bs_pre = R.dir_stream && !R.pre_tc, bs_post = R.dir_stream && !R.post_tc;
    if ((bs_pre || bs_post) && L.bk.n > 1 && B.fork && B.ys) {
        double t[2];
        for (int par = 0; par < 2; ++par) {
            B.bucket_par = par;
            t[par] = time3(s, [&] { dir_bs<T, ACC>(L, B, !bs_pre, r, z, nullptr, nullptr, s); });
        }
        B.bucket_par = t[1] < t[0] ? 1 : 0;
        if (const char *e = std::getenv("BDDC_BUCKETS")) {   // "serial" or "parallel"
            if (e[0] == 's') B.bucket_par = 0;
            if (e[0] == 'p') B.bucket_par = 1;
        }
    }
    if (!R.neu_staged) {
        const int cand[3] = {16 * 1024, 32 * 1024, 64 * 1024};
        double best = 1e30;
        int pick = 0;
        for (int c : cand) {
            if (neu_bg_smem<T, ACC>(L, c) > kSmemMaxB) continue;
            B.chunk = c;
            const double t = time3(s, [&] { neu_bg<T, ACC>(L, B, prec, r, (const int *)nullptr, s); });
            if (t < best) best = t, pick = c;
        }
        B.chunk = pick;
        if (const char *e = std::getenv("BDDC_NEU_CHUNK")) {   // bytes: this chunk
            const int c = std::atoi(e);
            if (c > 0 && neu_bg_smem<T, ACC>(L, c) <= kSmemMaxB) B.chunk = c;
        }
    }
}

}  // namespace

void tune_level_b(DevLevel &L, BatchLevel &B, int prec, const double *r, double *z, cudaStream_t s) {
    tune_route_t<double, double>(L, B, BDDC_PREC_FP64, r, z, s);
    tune_route_t<float, float>(L, B, BDDC_PREC_FP32, r, z, s);
    tune_route_t<__nv_bfloat16, float>(L, B, BDDC_PREC_BF16, r, z, s);
    if (prec == BDDC_PREC_FP64) tune_t<double, double>(L, B, prec, r, z, s);
    else if (prec == BDDC_PREC_FP32) tune_t<float, float>(L, B, prec, r, z, s);
    else tune_t<__nv_bfloat16, float>(L, B, prec, r, z, s);
    BDDC_CUDA_TRY(cudaStreamSynchronize(s));
}

void batch_prepare_level(const DevLevel &L) {
    if (L.bk.n == 0) return;
    prepare_bs<double, double>(L);
    prepare_bs<float, float>(L);
    prepare_bs<__nv_bfloat16, float>(L);
}

void prepare_batch_kernels() {
    const int big = (int)kSmemMaxB;
#define BDDC_SMEM_ATTR_B(k) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, big)
#define BDDC_DIR_B(T, A, BPV)                                   \
    BDDC_SMEM_ATTR_B((k_dir_b<T, A, BPV, false>));              \
    BDDC_SMEM_ATTR_B((k_dir_b<T, A, BPV, true>));
#define BDDC_DIR_LS(T, ACC, BPV)                                     \
    BDDC_SMEM_ATTR_B((k_dir_ls<T, ACC, BPV, false, false>));         \
    BDDC_SMEM_ATTR_B((k_dir_ls<T, ACC, BPV, true, false>));          \
    BDDC_SMEM_ATTR_B((k_dir_ls<T, ACC, BPV, false, true>));          \
    BDDC_SMEM_ATTR_B((k_dir_ls<T, ACC, BPV, true, true>));
    BDDC_DIR_LS(double, double, 8) BDDC_DIR_LS(double, double, 16)
    BDDC_DIR_LS(float, float, 8) BDDC_DIR_LS(float, float, 16)
    BDDC_DIR_LS(__nv_bfloat16, float, 8) BDDC_DIR_LS(__nv_bfloat16, float, 16)
#undef BDDC_DIR_LS
    BDDC_DIR_B(double, double, 8) BDDC_DIR_B(double, double, 16) BDDC_DIR_B(double, double, 32)
    BDDC_DIR_B(float, float, 8) BDDC_DIR_B(float, float, 16) BDDC_DIR_B(float, float, 32)
    BDDC_DIR_B(__nv_bfloat16, float, 8) BDDC_DIR_B(__nv_bfloat16, float, 16) BDDC_DIR_B(__nv_bfloat16, float, 32)
    BDDC_SMEM_ATTR_B((k_neu_b<double, double>)); BDDC_SMEM_ATTR_B((k_neu_b<float, float>));
    BDDC_SMEM_ATTR_B((k_neu_b<__nv_bfloat16, float>));
    // (k_gemm_b and k_b_dir_spmv also have static shared memory: their
    // dynamic limits are their own sizes)
#define BDDC_TILE_ATTR(X, Y) \
    cudaFuncSetAttribute(k_b_dir_spmv<X, Y>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt_smem(X, Y, kMaxBatch));
    BDDC_TILE_ATTR(16, 8) BDDC_TILE_ATTR(32, 4) BDDC_TILE_ATTR(32, 8) BDDC_TILE_ATTR(8, 16)
#undef BDDC_TILE_ATTR
    cudaFuncSetAttribute(k_gemm_b<1, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(GM_S * gm_stage(8)));
    cudaFuncSetAttribute(k_gemm_b<2, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(GM_S * gm_stage(16)));
    cudaFuncSetAttribute(k_gemm_b<4, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(GM_S * gm_stage(32)));
    cudaFuncSetAttribute(k_gemm_b<1, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(GM_S * gm_stage(16)));
#define BDDC_DIR_BS(T, A, SW)                                   \
    BDDC_SMEM_ATTR_B((k_dir_bs<T, A, SW, false, kSBMaxT>));     \
    BDDC_SMEM_ATTR_B((k_dir_bs<T, A, SW, true, kSBMaxT>));
#define BDDC_DIR_BS_SMALL(T, SW)                                    \
    BDDC_SMEM_ATTR_B((k_dir_bs<T, float, SW, false, kSBSmallT>));   \
    BDDC_SMEM_ATTR_B((k_dir_bs<T, float, SW, true, kSBSmallT>));
    BDDC_DIR_BS(double, double, false) BDDC_DIR_BS(double, double, true)
    BDDC_DIR_BS(float, float, false) BDDC_DIR_BS(float, float, true)
    BDDC_DIR_BS(__nv_bfloat16, float, false) BDDC_DIR_BS(__nv_bfloat16, float, true)
    BDDC_DIR_BS_SMALL(float, false) BDDC_DIR_BS_SMALL(float, true)
    BDDC_DIR_BS_SMALL(__nv_bfloat16, false) BDDC_DIR_BS_SMALL(__nv_bfloat16, true)
#undef BDDC_DIR_BS_SMALL
#undef BDDC_DIR_BS
#define BDDC_NEU_BG(T, A)                                       \
    BDDC_SMEM_ATTR_B((k_neu_bg<T, A, 1, true>));                \
    BDDC_SMEM_ATTR_B((k_neu_bg<T, A, 2, true>));                \
    BDDC_SMEM_ATTR_B((k_neu_bg<T, A, 3, true>));                \
    BDDC_SMEM_ATTR_B((k_neu_bg<T, A, sizeof(A) == 8 ? 2 : 3, false>));
    BDDC_NEU_BG(double, double) BDDC_NEU_BG(float, float) BDDC_NEU_BG(__nv_bfloat16, float)
#undef BDDC_NEU_BG
    BDDC_SMEM_ATTR_B((k_avg_bg<double, double>)); BDDC_SMEM_ATTR_B((k_avg_bg<float, float>));
    BDDC_SMEM_ATTR_B((k_avg_bg<__nv_bfloat16, float>));
    BDDC_SMEM_ATTR_B((k_avg_b<double, double>)); BDDC_SMEM_ATTR_B((k_avg_b<float, float>));
    BDDC_SMEM_ATTR_B((k_avg_b<__nv_bfloat16, float>));
    prepare_tc_kernels();
#undef BDDC_DIR_B
#undef BDDC_SMEM_ATTR_B
}

void apply_level_pre_b(const DevLevel &L, const BatchLevel &B, int prec, const double *r,
                       const int *skip, cudaStream_t s, cudaEvent_t *ev) {
    if (prec == BDDC_PREC_FP64) pre_b<double, double>(L, B, prec, r, skip, s, ev);
    else if (prec == BDDC_PREC_FP32) pre_b<float, float>(L, B, prec, r, skip, s, ev);
    else pre_b<__nv_bfloat16, float>(L, B, prec, r, skip, s, ev);
}

void apply_level_post_b(const DevLevel &L, const BatchLevel &B, int prec, const double *r, double *z,
                        const int *skip, cudaStream_t s, cudaEvent_t *ev, const RzBatch *rz) {
    if (prec == BDDC_PREC_FP64) post_b<double, double>(L, B, prec, r, z, skip, s, ev, rz);
    else if (prec == BDDC_PREC_FP32) post_b<float, float>(L, B, prec, r, z, skip, s, ev, rz);
    else post_b<__nv_bfloat16, float>(L, B, prec, r, z, skip, s, ev, rz);
}

// Variants the autotuner chooses from.
constexpr int kTiles[][2] = {{16, 8}, {32, 4}, {32, 8}, {8, 16}};
constexpr int kNTiles = 4;
constexpr int kNGemm = 4;          // product variants (launch_gemm_b)

void launch_gemm_b(int n, int ld, const double *A, const double *X, double *Y, int K, const int *skip,
                   int *err, cudaStream_t s, int variant) {
    if (n <= 0) return;
    switch (variant) {
    case 0: launch_plain(k_gemm_b<1, 8>, (n + 7) / 8, 256, GM_S * gm_stage(8), s, n, ld, A, X, Y, K, 8, skip, err); break;
    case 2: launch_plain(k_gemm_b<4, 8>, (n + 31) / 32, 256, GM_S * gm_stage(32), s, n, ld, A, X, Y, K, 32, skip, err); break;
    case 3: {
        const int rpb = gemm_rows(3, n);
        launch_plain(k_gemm_b<1, 16>, (n + rpb - 1) / rpb, 512, GM_S * gm_stage(16), s, n, ld, A, X, Y, K, rpb, skip,
                     err);
        break;
    }
    default: launch_plain(k_gemm_b<2, 8>, (n + 15) / 16, 256, GM_S * gm_stage(16), s, n, ld, A, X, Y, K, 16, skip, err);
    }
}

// Mean device time of `reps` launches of f (one untimed launch first).
template <class F> float time_launches(F f, int reps, cudaStream_t s) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    f();
    cudaEventRecord(e0, s);
    for (int i = 0; i < reps; ++i) f();
    cudaEventRecord(e1, s);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ms / reps;
}

int gemm_tune(int n, int ld, const double *A, const double *X, double *Y, int K, int *err, cudaStream_t s) {
    // BDDC_GEMM_VARIANT=0..3 fixes the variant instead of timing them.  The
    // timing covers 0..2 only: variant 3 (one sixteen-warp block per SM) is
    // the fastest alone but takes each SM's slot from the other batches in
    // flight (measured on the 512^2 channel problem: 0.864 against 0.846 of
    // the FP64 pipe alone, 1375 against 1426 solves/s with three groups)
    if (const char *e = std::getenv("BDDC_GEMM_VARIANT"))
        if (e[0] >= '0' && e[0] < '0' + kNGemm && e[1] == 0) return e[0] - '0';
    int best = 1;
    float tb = 1e30f;
    for (int v = 0; v < kNGemm - 1; ++v) {
        const float t = time_launches([&] { launch_gemm_b(n, ld, A, X, Y, K, nullptr, err, s, v); }, 3, s);
        if (t < tb) { tb = t; best = v; }
    }
    return best;
}
int gemm_rows(int variant, int n) {
    if (variant == 3) {                // one block per SM, sixteen warps
        const int r = (n + num_sms_b() - 1) / num_sms_b();
        return r < 1 ? 1 : (r > 16 ? 16 : r);
    }
    return variant == 0 ? 8 : (variant == 2 ? 32 : 16);
}

void launch_b_init(int n, int K, const double *b, int64_t ldb, double *x, double *r, double *p,
                   double *part, unsigned *counter, BatchScalars *sc, double tol, int maxit,
                   cudaStream_t s) {
    int g = (n + kTG - 1) / kTG;
    const int cap = 8 * num_sms_b() < kMaxVecGrid ? 8 * num_sms_b() : kMaxVecGrid;
    if (g > cap) g = cap;
    k_b_init<<<g < 1 ? 1 : g, kTT, 0, s>>>(n, K, b, ldb, x, r, p, part, counter, sc, tol, maxit);
}
template <int TX, int TY> int tile_blocks(int nx) {
    const int n1 = nx - 1;
    return ((n1 + TX - 1) / TX) * ((n1 + TY - 1) / TY);
}
// Strips, rows per segment and blocks of k_b_dir_march: the segments that the
// resident warps can take at once, at least kMarchRows rows each.
struct MarchShape { int strips, rows, blocks; };
MarchShape march_shape(int nx) {
    constexpr int kMarchRows = 4;
    const int n1 = nx - 1, warps = kMarchT / 32;
    MarchShape m;
    m.strips = (n1 + MW - 1) / MW;
    int segs = kMarchPerSm * num_sms_b() * warps / m.strips;
    const int most = (n1 + kMarchRows - 1) / kMarchRows;
    segs = segs < 1 ? 1 : (segs > most ? most : segs);
    m.rows = (n1 + segs - 1) / segs;
    segs = (n1 + m.rows - 1) / m.rows;
    m.blocks = (m.strips * segs + warps - 1) / warps;
    return m;
}
int launch_b_dir_spmv_blocks(int nx) {   // the most blocks any variant launches
    return std::max(std::max(std::max(tile_blocks<16, 8>(nx), tile_blocks<32, 4>(nx)),
                             std::max(tile_blocks<32, 8>(nx), tile_blocks<8, 16>(nx))),
                    march_shape(nx).blocks);
}
template <int TX, int TY>
void dir_spmv_v(int nx, int K, const double *w, const double *z, double *p0, double *p1, double *q,
                double *part, unsigned *counter, BatchScalars *sc, double *alphas, cudaStream_t s) {
    launch_plain(k_b_dir_spmv<TX, TY>, tile_blocks<TX, TY>(nx), bblock(K), bt_smem(TX, TY, K), s, nx, K, w, z,
                 p0, p1, q, part, counter, sc, alphas);
}
void launch_b_dir_tile(int nx, int K, const double *w, const double *z, double *p0, double *p1, double *q,
                       double *part, unsigned *counter, BatchScalars *sc, double *alphas, cudaStream_t s,
                       int variant) {
    switch (variant) {
    case 1: dir_spmv_v<32, 4>(nx, K, w, z, p0, p1, q, part, counter, sc, alphas, s); break;
    case 2: dir_spmv_v<32, 8>(nx, K, w, z, p0, p1, q, part, counter, sc, alphas, s); break;
    case 3: dir_spmv_v<8, 16>(nx, K, w, z, p0, p1, q, part, counter, sc, alphas, s); break;
    default: dir_spmv_v<16, 8>(nx, K, w, z, p0, p1, q, part, counter, sc, alphas, s);
    }
}
void launch_b_dir_spmv(int nx, int K, const double *w, const double *z, double *p0, double *p1,
                       double *q, double *part, unsigned *counter, BatchScalars *sc, double *alphas,
                       cudaStream_t s, int variant) {
    if (!stencil_marches(K)) {
        launch_b_dir_tile(nx, K, w, z, p0, p1, q, part, counter, sc, alphas, s, variant);
        return;
    }
    const MarchShape m = march_shape(nx);
    launch_plain(k_b_dir_march, m.blocks, kMarchT, 0, s, nx, K, w, z, p0, p1, q, part, counter, sc, alphas,
                 m.strips, m.rows);
}
int dir_spmv_tune(int nx, const double *w, const double *z, double *p0, double *p1, double *q, double *part,
                  unsigned *counter, BatchScalars *sc, double *alphas, cudaStream_t s) {
    static_assert(!stencil_marches(kTileTuneK), "the tiles are timed at a width that takes one");
    if (const char *e = std::getenv("BDDC_TILE_VARIANT")) {   // 0..3: this tile, no timing
        const int v = std::atoi(e);
        if (v >= 0 && v < kNTiles) return v;
    }
    int best = 0;
    float tb = 1e30f;
    for (int v = 0; v < kNTiles; ++v) {
        const float t = time_launches(
            [&] { launch_b_dir_tile(nx, kTileTuneK, w, z, p0, p1, q, part, counter, sc, alphas, s, v); }, 3, s);
        if (t < tb) { tb = t; best = v; }
    }
    return best;
}
void dir_spmv_tile(int variant, int *tx, int *ty) {
    const int v = variant < 0 || variant >= kNTiles ? 0 : variant;
    *tx = kTiles[v][0];
    *ty = kTiles[v][1];
}
void launch_b_update(int n, int K, double *x, double *r, const double *p0, const double *p1,
                     const double *q, double *part, unsigned *counter, BatchScalars *sc, cudaStream_t s) {
    const int64_t nK = (int64_t)n * K;
    launch_plain(k_b_update, vgrid_b(nK, K), bblock(K), 0, s, nK, K, x, r, p0, p1, q, part, counter, sc);
}
void launch_b_residual(int nx, int K, const double *w, const double *b, int64_t ldb, const double *x,
                       double *res, cudaStream_t s) {
    const int64_t nK = (int64_t)(nx - 1) * (nx - 1) * K;
    k_b_residual<<<(int)((nK + 255) / 256), 256, 0, s>>>(nx, K, w, b, ldb, x, res);
}
void launch_b_norm2(int n, int K, const double *v, double *part, unsigned *counter, double *out,
                    cudaStream_t s) {
    const int64_t nK = (int64_t)n * K;
    k_b_norm2<<<vgrid_b(nK, K), bblock(K), 0, s>>>(nK, K, v, part, counter, out);
}
void launch_b_admit(int n, int K, int k, const double *b, double *x, double *r, double *p, double *part,
                    unsigned *counter, BatchScalars *sc, double tol, int maxit, cudaStream_t s) {
    int g = (n + kRB - 1) / kRB;
    if (g > 4 * num_sms_b()) g = 4 * num_sms_b();
    k_b_admit<<<g, kRB, 0, s>>>(n, K, k, b, x, r, p, part, counter, sc, tol, maxit);
}
void launch_b_column(int n, int K, int k, const double *x, double *dst, cudaStream_t s) {
    if (n > 0) k_b_column<<<(n + 255) / 256, 256, 0, s>>>(n, K, k, x, dst);
}
void launch_b_move_column(int n, int K, int k, const double *src, double *dst, cudaStream_t s) {
    if (n > 0) k_b_move_column<<<(n + 255) / 256, 256, 0, s>>>(n, K, k, src, dst);
}
void launch_selftest_convert(const double *d, int64_t n, unsigned long long *bad, cudaStream_t s) {
    if (n > 0) k_selftest_convert<<<(int)((n + 255) / 256), 256, 0, s>>>(d, n, bad);
}
void launch_fp64_rate(int iters, double *out, cudaStream_t s) {
    k_fp64_rate<<<kFmaBlocksPerSm * num_sms_b(), 256, 0, s>>>(iters, 0.9999999, 1e-9, out);
}
void launch_b_gather(int n, int K, const double *src, int64_t ld, double *dst, cudaStream_t s) {
    if (n > 0) k_b_gather<<<(n + kTG - 1) / kTG, kTT, 0, s>>>(n, K, src, ld, dst);
}
void launch_b_scatter(int n, int K, const double *src, double *dst, int64_t ld, cudaStream_t s) {
    if (n > 0) k_b_scatter<<<(n + kTG - 1) / kTG, kTT, 0, s>>>(n, K, src, dst, ld);
}

}  // namespace bddc
