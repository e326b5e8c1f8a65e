// What the team kernel (chm_team.cuh) and the solve kernel (chm_solve.cu)
// share: thread blocks of four warps that run the steps of blocked
// substitutions, each step a task, with the inverse of every 32 x 32
// diagonal block and its products with the two tiles next to it prepared
// beforehand, so that a chain's step is one product with the step before.
#pragma once

#include "chm_device.cuh"
#include "chm_layout.h"
#include "chm_pass.cuh"

namespace chm {
namespace sub {

constexpr int kThreads = 128;
constexpr int kWarps = 4;
constexpr int kPer = kW / kWarps;  // rows of a split 32 x 32 product per warp

constexpr unsigned kFull = 0xffffffffu;
struct PrepSmem {
    double D[kW][kW + 1];
    double U[kW][kW + 1];
    double F[kW][kW + 1];
    double M[kW / 2][kW / 2 + 1];
    double rd[kW];
};
// Stage the 32 x 32 tile at row r0, column c0 into dst[column][Stride], read
// through L2 (an earlier pass of the launch may have written it on another
// SM): 16-byte asynchronous copies if `vec`, else loads of one element,
// sixteen in flight per lane (a 4- or 8-byte cp.async would go through L1; with
// eight a substitution step's tiles take 5 % longer).  `diag`: the diagonal
// tile, rows <= column only; the rest is zero.  stage_columns: the columns
// first .. last - 1, N loads in flight.
template <int N, typename T>
__device__ __forceinline__ void stage_columns(const SyncArgs &sy, T *dst, const T *L, long long ld, long long r0,
                                              long long c0, long long n, bool diag, int lane, int first, int last)
{
    constexpr int SD = pass::Stride<T>::value;
#pragma unroll 1
    for (int c = first; c < last; c += N) {
        T x[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const long long o = (r0 + lane) + (c0 + c + i) * ld;
            x[i] = (c0 + c + i < n && (!diag || lane <= c + i) && CHK_TRI(sy, o, n, ld)) ? __ldcg(L + o) : T(0);
        }
#pragma unroll
        for (int i = 0; i < N; ++i) dst[(c + i) * SD + lane] = x[i];
    }
}
template <typename T>
__device__ __forceinline__ void stage_tile(const SyncArgs &sy, T *dst, const T *L, long long ld, long long r0,
                                           long long c0, long long n, bool vec, bool diag, int lane)
{
    if (vec) pass::stage_tile(sy, dst, L, ld, r0, c0, n, kW, true, lane);
    else stage_columns<16>(sy, dst, L, ld, r0, c0, n, diag, lane, 0, kW);
}

// S.U = S.D^{-1}, upper triangular, with `d` the diagonal to use (lane = row,
// read from warp 0).  S.U is zero on entry.  The inverse is built up from 8 x 8 diagonal blocks: with
// D = [[D1, B], [0, D2]], U = [[U1, -U1 B U2], [0, U2]].  The four 8 x 8
// inverses take one warp (a column per lane, 36 dependent FP64 instructions),
// the products of the two levels above all four warps: 116 instructions in
// a row instead of the 560 of a column-per-lane substitution (3.6 against
// 17 us at one FP64 instruction per 64 cycles and warp).
__device__ __forceinline__ void invert_block(PrepSmem &S, double d)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        S.rd[lane] = rcp_refined(d);
        __syncwarp();
        const int h = lane & 24, col = lane & 7;
        double u[8];
#pragma unroll
        for (int i = 7; i >= 0; --i) {
            double s = (i == col) ? 1.0 : 0.0;
#pragma unroll
            for (int m = i + 1; m < 8; ++m) s = fma(-S.D[h + i][h + m], u[m], s);
            u[i] = s * S.rd[h + i];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) S.U[h + i][h + col] = u[i];
    }
    __syncthreads();
    {
        // 8 to 16: thread = (half, row, column)
        const int h = (tid >> 6) * 16, i = (tid >> 3) & 7, j = tid & 7;
        double s = 0.0;
#pragma unroll
        for (int m = 0; m < 8; ++m) s = fma(S.D[h + i][h + 8 + m], S.U[h + 8 + m][h + 8 + j], s);
        S.M[(tid >> 6) * 8 + i][j] = s;
        __syncthreads();
        s = 0.0;
#pragma unroll
        for (int m = 0; m < 8; ++m) s = fma(S.U[h + i][h + m], S.M[(tid >> 6) * 8 + m][j], s);
        S.U[h + i][h + 8 + j] = -s;
        __syncthreads();
    }
    {
        // 16 to 32: two rows a thread
        constexpr int kH = kW / 2;
        const int i = tid / kH, j = tid & (kH - 1);
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int m = 0; m < kH; ++m) {
            const double u = S.U[kH + m][kH + j];
            s0 = fma(S.D[i][kH + m], u, s0);
            s1 = fma(S.D[i + 8][kH + m], u, s1);
        }
        S.M[i][j] = s0;
        S.M[i + 8][j] = s1;
        __syncthreads();
        s0 = s1 = 0.0;
#pragma unroll
        for (int m = 0; m < kH; ++m) {
            const double x = S.M[m][j];
            s0 = fma(S.U[i][m], x, s0);
            s1 = fma(S.U[i + 8][m], x, s1);
        }
        S.U[i][kH + j] = -s0;
        S.U[i + 8][kH + j] = -s1;
        __syncthreads();
    }
}

// out[j kW + i] = G[i][j] = sum_{m<=i} U[m][i] F[j][m]; rows i = warp,
// warp + 4, ... (so that the four warps' triangles weigh the same: 144
// FMAs each, with U's zeros in the rows' last groups of four), lane = j.
__device__ __forceinline__ void form_g(const PrepSmem &S, double *out)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc[kPer];
#pragma unroll
    for (int ii = 0; ii < kPer; ++ii) acc[ii] = 0.0;
#pragma unroll
    for (int m = 0; m < kW; ++m) {
        const double f = S.F[lane][m];
#pragma unroll
        for (int ii = m / kWarps; ii < kPer; ++ii) acc[ii] = fma(S.U[m][ii * kWarps + warp], f, acc[ii]);
    }
#pragma unroll
    for (int ii = 0; ii < kPer; ++ii) __stcg(out + (size_t)lane * kW + ii * kWarps + warp, acc[ii]);
}
// Every store of the block's threads so far, then the flag.
__device__ __forceinline__ void publish(int *flag, int epoch)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) st_release_gpu(flag, epoch);
}

// Warp-wide bounded wait for R tagged doubles per lane; zeros if it gave up,
// so that the task reaches its barriers.  With `probe` the wait is not one of
// the chain's next steps: it polls that one word (the last one written) with
// pauses of up to 128 ns and takes the values once it is there.  Dozens of
// warps wait on the newest step, and a poll of all its words by each would
// slow the L2 slices that the chain's own stores and loads go to.  Without
// it the warp polls the values themselves, without a pause.
template <int R>
__device__ __forceinline__ void wait_vals(const SyncArgs &sy, const long long *w2, const long long *probe, long long ep64,
                                          long long who, double (&x)[R])
{
    auto have = [&]() {
        bool ok = true;
#pragma unroll
        for (int r = 0; r < R; ++r) ok = get_tagged(w2 + 2 * r, ep64, &x[r]) && ok;
        return __all_sync(kFull, ok) != 0;
    };
    if (have()) return;
    const long long t0 = global_ns();
    unsigned ns = 16;
    for (unsigned it = 1;; ++it) {
        bool look = true;
        if (probe) {
            look = __any_sync(kFull, (ld_relaxed_gpu(probe) & ~0xffffffffll) == ep64);
            if (!look) {
                __nanosleep(ns);
                if (ns < 128) ns <<= 1;
            }
        }
        if (look && have()) return;
        // (looked at by all lanes alike: a branch of lane 0 alone would leave
        // the warp split, and every later shuffle would wait for the halves)
        if ((it & 31u) == 0u) {
            const bool late = global_ns() - t0 > sy.timeout_ns || it > (1u << 28);
            if (__any_sync(kFull, late || aborted(sy))) {
                if ((threadIdx.x & 31) == 0 && late) record_error(sy, kStatusTimeout, who);
#pragma unroll
                for (int r = 0; r < R; ++r) x[r] = 0.0;
                return;
            }
        }
    }
}
__device__ __forceinline__ double wait_p(const SyncArgs &sy, const long long *w2, const long long *probe, long long ep64,
                                         long long who)
{
    double x[1] = {0.0};
    wait_vals<1>(sy, w2, probe, ep64, who, x);
    return x[0];
}
// Warp-wide bounded wait for the flags f[first .. last] (last - first < 32 per
// look, one a lane), the warp staying together.
__device__ __forceinline__ void wait_flags(const SyncArgs &sy, const int *f, int first, int last, long long who)
{
    for (int r0 = first; r0 <= last; r0 += 32) {
        const int r = min(r0 + ((int)threadIdx.x & 31), last);
        const long long t0 = global_ns();
        unsigned ns = 16;
        for (unsigned it = 1; !__all_sync(kFull, ld_acquire_gpu(f + r) == sy.epoch); ++it) {
            __nanosleep(ns);
            if (ns < 256) ns <<= 1;
            if ((it & 15u) == 0u) {
                const bool late = global_ns() - t0 > sy.timeout_ns || it > (1u << 26);
                if (__any_sync(kFull, late || aborted(sy))) {
                    if ((threadIdx.x & 31) == 0 && late) record_error(sy, kStatusTimeout, who);
                    return;
                }
            }
        }
    }
}

}  // namespace sub
}  // namespace chm
