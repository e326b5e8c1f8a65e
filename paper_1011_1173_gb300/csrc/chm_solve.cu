// Solve with a factor: B <- (L^T L)^{-1} B, the use a maintained Cholesky
// factor serves (Sec. 1).  A forward substitution with L^T (lower) followed
// by a back substitution with L (upper), both blocked by kW = 32 rows, in
// one persistent launch per group of right-hand sides.
//
// A launch runs C chains of R right-hand sides each.  Tasks are taken in
// order from a launch-wide counter by blocks of four warps:
//   t < nb: prepare block b = t: U_b = D_b^{-1}, G_b = U_b^T L_{b-1,b}^T and
//     H_b = U_b L_{b,b+1} (D_b the diagonal block, L_{p,b} the 32 x 32 tile in
//     row block p and column block b), shared by every chain;
//   then, dealt round-robin to the chains, step s = 0 .. 2 nb - 1 of each:
//     s <  nb: y_b = D_b^{-T} (b_b - sum_{p<b} L_{p,b}^T y_p), b = s
//     s >= nb: x_b = D_b^{-1} (y_b - sum_{q>b} L_{b,q} x_q), b = 2 nb - 1 - s
// A task waits only on tasks taken before it, so the launch cannot deadlock
// whatever the number of resident blocks.
//
// A forward step sums the tiles whose y is already published, forms
// z_b = U_b^T (b_b - sum over p <= b-2) once y_{b-2} is in, and then
// y_b = z_b - G_b y_{b-1}; a backward step mirrors it with H_b.  Between one
// block's result and the next block's there is one 32 x 32 product (eight
// FMAs per warp and right-hand side), one barrier and a four-way sum.
// Results pass between blocks as epoch-tagged doubles (no fence, no flag).
//
// Why chains: right-hand sides do not depend on each other, and a step is
// bound by FP64 issue (one FP64 instruction per 64 cycles and warp), so a
// step of four right-hand sides takes three times a step of one.  C chains
// side by side fill the SMs that one chain leaves idle; the tiles they share
// meet in L2, and U, G and H are formed once instead of once per four
// right-hand sides.  n = 5000, float64, 16 right-hand sides: 1.13 ms in 16
// chains against 6.96 ms as four launches of four right-hand sides each; the
// FP64 rate allows 0.76 ms (400 M FMAs).
#include <float.h>

#include <algorithm>

#include "chm.h"
#include "chm_device.cuh"
#include "chm_internal.h"
#include "chm_layout.h"

namespace chm {
namespace {

constexpr int kSolveThreads = 128;
constexpr int kSolveWarps = kSolveThreads / 32;
constexpr int kSolveRhs = 4;                       // right-hand sides per chain (largest)
constexpr int kSolveChains = 16;                   // chains per launch (largest)
constexpr int kRowsPerWarp = kW / kSolveWarps;     // rows (or columns) of a split tile per warp
constexpr int kPrepMats = 3;                       // U_b, G_b and H_b
constexpr unsigned kFull = 0xffffffffu;

template <typename T>
struct SolveArgs {
    const T *L;
    long long n, ld;
    T *B;
    long long ldb;
    int nb;           // blocks of kW rows
    int nr;           // right-hand sides of this launch (1 .. C R)
    int chains;       // C: chain c takes right-hand sides c R .. c R + R - 1
    // back substitution only: y = L^{-T} b is given, row i of right-hand
    // side r at Y[i * ys + r * cs] (chm_modify_solve's pass forms it)
    const T *Y;
    long long ys, cs;
    int back_only;
    double *inv;      // [nb][kPrepMats][kW][kW]: U_b = D_b^{-1} (row i at i * kW), G_b and H_b
                      // (transposed: element (i, j) at j * kW + i)
    int *uflag;       // [nb]: U_b, G_b and H_b published (== epoch)
    long long *ytag;  // [C][nb][kW][R][2]: y_b as tagged doubles
    long long *xtag;  // [C][nb][kW][R][2]: x_b as tagged doubles
    int *ctl;
    long long *status;
    long long timeout_ns;
    // the workspace allocations inv, uflag and ytag / xtag are carved from (bounds-checked builds)
    const char *ws_data;
    size_t ws_data_bytes;
    const int *ws_iflags;
    size_t ws_iflags_n;
    const long long *ws_progress;
    size_t ws_progress_n;
    long long chk_cut;
};

// Shared memory of a block: a preparation task's matrices or a step's
// partial sums.
struct PrepSmem {
    double D[kW][kW + 1];  // diagonal block (row, column); identity beyond the order
    double U[kW][kW + 1];  // its inverse
    double T[kW][kW + 1];  // the tile above it, then the tile to its right
    double M[kW / 2][kW / 2 + 1];
    double rd[kW];         // 1 / D_ii
};
template <int R>
struct SolveSmem {
    union {
        PrepSmem prep;
        double part[2][kSolveWarps][R][kW];
    };
};

template <int R>
__device__ __forceinline__ size_t tag_at(int blk, int i, int r)
{
    return (((size_t)blk * kW + i) * R + r) * 2;
}

// The whole warp waits for the R tagged values of block `blk` (lane i gets
// row i).  `next_step` marks the wait on the previous block's result, the
// one step of the chain: it polls at short fixed intervals (only the next
// block's four warps wait on a fresh result, and each step gains the time a
// longer sleep would add); every other wait backs off up to 256 ns, since
// hundreds of warps may be waiting on older results at once.  A wait that
// gives up (recorded as a timeout, or the launch is aborted) yields zeros,
// so that every warp still reaches the block's barriers; the result is then
// unspecified and the status says so.
template <int R>
__device__ __forceinline__ void wait_block(const SyncArgs &sy, const long long *tags, long long ep64, int blk,
                                           long long who, double *v, bool next_step = false)
{
    const int lane = threadIdx.x & 31;
    const long long *w = tags + tag_at<R>(blk, lane, 0);
    const long long t0 = global_ns();
    unsigned ns = next_step ? 32 : 16;
    for (unsigned it = 0;; ++it) {
        bool ok = true;
#pragma unroll
        for (int r = 0; r < R; ++r) ok = get_tagged(w + 2 * r, ep64, &v[r]) && ok;
        if (__all_sync(kFull, ok)) return;
        // (looked at by all lanes alike: a branch of lane 0 alone would leave
        // the warp split, and every later shuffle would wait for the halves)
        if ((it & 15u) == 15u) {
            const bool late = global_ns() - t0 > sy.timeout_ns || it > (1u << 28);
            if (__any_sync(kFull, late || aborted(sy))) {
                if (lane == 0 && late) record_error(sy, kStatusTimeout, who);
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = 0.0;
                return;
            }
        }
        __nanosleep(ns);
        if (!next_step && ns < 256) ns <<= 1;
    }
}

// Sum of the four warps' partial products of row `lane`, for each r.
template <int R>
__device__ __forceinline__ double part_sum(const SolveSmem<R> &S, int buf, int r, int lane)
{
    return (S.part[buf][0][r][lane] + S.part[buf][1][r][lane]) + (S.part[buf][2][r][lane] + S.part[buf][3][r][lane]);
}

// U_b, G_b and H_b of block b.  The inverse goes by halves: with
// D = [[D1, B], [0, D2]], U = [[U1, -U1 B U2], [0, U2]]; the two 16 x 16
// inverses take one warp (a column per lane, 136 dependent FMAs instead of
// the 528 of a whole column each) and the products all four.
template <typename T>
__device__ void prep_task(const SolveArgs<T> &a, const SyncArgs &sy, int b, PrepSmem &S)
{
    constexpr int kH = kW / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = a.n, ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool above = b >= 1 && !a.back_only;  // G_b serves the forward steps only

    // the diagonal block (identity beyond the order) and the tile above it,
    // S.T[j][m] = L[(b-1) kW + j, c0 + m]
    for (int e = threadIdx.x; e < kW * kW; e += kSolveThreads) {
        const int i = e & (kW - 1), j = e / kW;
        double v = 0.0;
        if (j < nc) {
            if (i <= j && CHK_TRI(sy, c0 + i + (c0 + j) * ld, n, ld)) v = (double)__ldg(a.L + c0 + i + (c0 + j) * ld);
        } else if (i == j) {
            v = 1.0;
        }
        S.D[i][j] = v;
        if (above)
            S.T[i][j] = (j < nc && CHK_TRI(sy, c0 - kW + i + (c0 + j) * ld, n, ld))
                            ? (double)__ldg(a.L + c0 - kW + i + (c0 + j) * ld) : 0.0;
    }
    __syncthreads();
    if (warp == 0) {
        double d = S.D[lane][lane];
        if (!(d > 0.0 && d <= DBL_MAX)) {  // not a Cholesky factor
            record_error(sy, kStatusNotPD, c0 + lane);
            d = 1.0;
        }
        S.rd[lane] = 1.0 / d;
        __syncwarp();
        // column `col` of the inverse of diagonal half h: back substitution on D_h u = e_col
        const int h = lane & kH, col = lane & (kH - 1);
        double u[kH];
#pragma unroll
        for (int i = kH - 1; i >= 0; --i) {
            double s = (i == col) ? 1.0 : 0.0;
#pragma unroll
            for (int m = i + 1; m < kH; ++m) s = fma(-S.D[h + i][h + m], u[m], s);
            u[i] = s * S.rd[h + i];
        }
#pragma unroll
        for (int i = 0; i < kH; ++i) {
            S.U[h + i][h + col] = u[i];
            if (h) S.U[h + i][col] = 0.0;
        }
    }
    __syncthreads();
    // M = B U2, then U12 = -U1 M: two outputs a thread, a row pair per half warp
    const int mi = threadIdx.x / kH, mj = threadIdx.x & (kH - 1);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        const int i = mi + 8 * v;
        double s = 0.0;
#pragma unroll
        for (int m = 0; m < kH; ++m) s = fma(S.D[i][kH + m], S.U[kH + m][kH + mj], s);
        S.M[i][mj] = s;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        const int i = mi + 8 * v;
        double s = 0.0;
#pragma unroll
        for (int m = 0; m < kH; ++m) s = fma(S.U[i][m], S.M[m][mj], s);
        S.U[i][kH + mj] = -s;
    }
    __syncthreads();
    double *inv = a.inv + (size_t)b * kPrepMats * kW * kW;
    for (int e = threadIdx.x; e < kW * kW; e += kSolveThreads) __stcg(inv + e, S.U[e / kW][e & (kW - 1)]);
    // G: G[i][j] = sum_{m<=i} U[m][i] T[j][m]; rows i = warp, warp + 4, ... (so
    // that the four warps' triangles weigh the same), lane = j
    if (above) {
        for (int ii = 0; ii < kRowsPerWarp; ++ii) {
            const int i = ii * kSolveWarps + warp;
            double s0 = 0.0, s1 = 0.0;
            for (int m = 0; m <= i; m += 2) {
                s0 = fma(S.U[m][i], S.T[lane][m], s0);
                if (m < i) s1 = fma(S.U[m + 1][i], S.T[lane][m + 1], s1);
            }
            __stcg(inv + kW * kW + (size_t)lane * kW + i, s0 + s1);
        }
    }
    // H: H[i][j] = sum_{m>=i} U[i][m] T[m][j], T the tile to the right of the diagonal block
    if (b + 1 < a.nb) {
        __syncthreads();
        const long long q1 = c0 + kW;
        const int nc1 = (int)min((long long)kW, n - q1);
        for (int e = threadIdx.x; e < kW * kW; e += kSolveThreads) {
            const int i = e & (kW - 1), j = e / kW;
            S.T[i][j] = (j < nc1 && CHK_TRI(sy, c0 + i + (q1 + j) * ld, n, ld)) ? (double)__ldg(a.L + c0 + i + (q1 + j) * ld)
                                                                                : 0.0;
        }
        __syncthreads();
        for (int ii = 0; ii < kRowsPerWarp; ++ii) {
            const int i = ii * kSolveWarps + warp;
            double s0 = 0.0, s1 = 0.0;
            for (int m = kW - 1; m >= i; m -= 2) {
                s0 = fma(S.U[i][m], S.T[m][lane], s0);
                if (m > i) s1 = fma(S.U[i][m - 1], S.T[m - 1][lane], s1);
            }
            __stcg(inv + 2 * kW * kW + (size_t)lane * kW + i, s0 + s1);
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) st_release_gpu(a.uflag + b, sy.epoch);
}

// The block's four warps wait for U_b, G_b and H_b; false if the wait gave up.
template <typename T>
__device__ __forceinline__ bool wait_prep(const SolveArgs<T> &a, const SyncArgs &sy, int b)
{
    const bool ok = __all_sync(kFull, wait_eq(sy, a.uflag + b, sy.epoch, b));
    __syncwarp();
    return ok;
}

// Chain c's step at block b, forward.
template <typename T, int R>
__device__ void forward_task(const SolveArgs<T> &a, const SyncArgs &sy, long long ep64, int c, int b, SolveSmem<R> &S)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, a.n - c0);
    const bool active = lane < nc;
    const long long who = b;
    const int r0 = c * R;  // this chain's first right-hand side
    long long *ytag = a.ytag + (size_t)c * a.nb * kW * R * 2;

    double rhs[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        rhs[r] = (active && r0 + r < a.nr && CHK_RECT(sy, c0 + lane + (r0 + r) * a.ldb, a.n, a.nr, a.ldb))
                     ? (double)a.B[c0 + lane + (r0 + r) * a.ldb] : 0.0;
    // tiles p <= b - 3 of column block b, dealt round-robin to the warps (a
    // fixed order of the sums: results do not depend on timing); lane =
    // column of the block, the tile's 32 rows read down the column
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    const long long colo = (c0 + (active ? lane : 0)) * ld;
    const T *col = a.L + colo;
    for (int p = warp; p <= b - 3; p += kSolveWarps) {
        const T *src = col + (long long)p * kW;
        double t[kW];
#pragma unroll
        for (int j = 0; j < kW; ++j)
            t[j] = (active && CHK_TRI(sy, colo + (long long)p * kW + j, a.n, ld)) ? (double)__ldg(src + j) : 0.0;
        double yv[R];
        wait_block<R>(sy, ytag, ep64, p, who, yv);
#pragma unroll
        for (int j = 0; j < kW; ++j)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t[j], __shfl_sync(kFull, yv[r], j), acc[r]);
    }
    // this warp's rows of U_b and columns of G_b (see the products below)
    const bool ok = wait_prep(a, sy, b);
    const double *inv = a.inv + (size_t)b * kPrepMats * kW * kW;
    double u[kRowsPerWarp], g[kRowsPerWarp];
#pragma unroll
    for (int jj = 0; jj < kRowsPerWarp; ++jj) {
        const int j = warp * kRowsPerWarp + jj;
        u[jj] = ok ? __ldcg(inv + j * kW + lane) : 0.0;
        g[jj] = (ok && b >= 1) ? __ldcg(inv + kW * kW + j * kW + lane) : 0.0;
    }
    // tile b - 2: its rows split over the warps
    if (b >= 2) {
        const T *src = col + (long long)(b - 2) * kW + warp * kRowsPerWarp;
        double t[kRowsPerWarp];
#pragma unroll
        for (int jj = 0; jj < kRowsPerWarp; ++jj) t[jj] = active ? (double)__ldg(src + jj) : 0.0;
        double yv[R];
        wait_block<R>(sy, ytag, ep64, b - 2, who, yv);
#pragma unroll
        for (int jj = 0; jj < kRowsPerWarp; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r)
                acc[r] = fma(t[jj], __shfl_sync(kFull, yv[r], warp * kRowsPerWarp + jj), acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = acc[r];
    __syncthreads();
    double rv[R];  // b_b - sum_{p <= b-2} L_{p,b}^T y_p, row `lane`
#pragma unroll
    for (int r = 0; r < R; ++r) rv[r] = rhs[r] - part_sum(S, 0, r, lane);
    // z_b = U^T r: z_i = sum_{j <= i} U_ji r_j, the j split over the warps
    double pz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) pz[r] = 0.0;
#pragma unroll
    for (int jj = 0; jj < kRowsPerWarp; ++jj) {
        const int j = warp * kRowsPerWarp + jj;
#pragma unroll
        for (int r = 0; r < R; ++r) pz[r] = fma(u[jj], __shfl_sync(kFull, rv[r], j), pz[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[1][warp][r][lane] = pz[r];
    __syncthreads();
    double z[R];
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = part_sum(S, 1, r, lane);
    // (part[0] is free again: every warp read it before the barrier above)
    // y_b = z_b - G_b y_{b-1}: the step that waits on the previous block
    double py[R];
#pragma unroll
    for (int r = 0; r < R; ++r) py[r] = 0.0;
    if (b >= 1) {
        double yv[R];
        wait_block<R>(sy, ytag, ep64, b - 1, who, yv, true);
#pragma unroll
        for (int jj = 0; jj < kRowsPerWarp; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r)
                py[r] = fma(g[jj], __shfl_sync(kFull, yv[r], warp * kRowsPerWarp + jj), py[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = py[r];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) put_tagged(ytag + tag_at<R>(b, lane, r), z[r] - part_sum(S, 0, r, lane), ep64);
    }
}

// Chain c's step at block b, backward.
template <typename T, int R>
__device__ void backward_task(const SolveArgs<T> &a, const SyncArgs &sy, long long ep64, int c, int b,
                              SolveSmem<R> &S)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = a.n, ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool active = lane < nc;
    const long long who = b;
    const bool has_next = b + 1 < a.nb;
    const int r0 = c * R;
    long long *xtag = a.xtag + (size_t)c * a.nb * kW * R * 2;

    // this warp's columns of U_b and H_b (see the products below)
    const bool ok = wait_prep(a, sy, b);
    const double *inv = a.inv + (size_t)b * kPrepMats * kW * kW;
    double u[kRowsPerWarp], h[kRowsPerWarp];
#pragma unroll
    for (int jj = 0; jj < kRowsPerWarp; jj += 2) {
        const int j = warp * kRowsPerWarp + jj;
        const double2 v = ok ? __ldcg(reinterpret_cast<const double2 *>(inv + lane * kW + j)) : make_double2(0.0, 0.0);
        u[jj] = v.x;
        u[jj + 1] = v.y;
    }
#pragma unroll
    for (int jj = 0; jj < kRowsPerWarp; ++jj)
        h[jj] = (ok && has_next) ? __ldcg(inv + 2 * kW * kW + (warp * kRowsPerWarp + jj) * kW + lane) : 0.0;

    // tiles q >= b + 3 of row block b, from the last one up, dealt
    // round-robin to the warps; lane = row of the block, so each column of a
    // tile is one coalesced read
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    const long long rowo = c0 + (active ? lane : 0);
    const T *row = a.L + rowo;
    for (int q = a.nb - 1 - warp; q >= b + 3; q -= kSolveWarps) {
        const long long q0 = (long long)q * kW;
        const int ncq = (int)min((long long)kW, n - q0);
        double t[kW];
#pragma unroll
        for (int i = 0; i < kW; ++i)
            t[i] = (active && i < ncq && CHK_TRI(sy, rowo + (q0 + i) * ld, n, ld)) ? (double)__ldg(row + (q0 + i) * ld) : 0.0;
        double xv[R];
        wait_block<R>(sy, xtag, ep64, q, who, xv);
#pragma unroll
        for (int i = 0; i < kW; ++i)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t[i], __shfl_sync(kFull, xv[r], i), acc[r]);
    }
    // tile b + 2: its columns split over the warps
    if (b + 2 < a.nb) {
        const long long q0 = (long long)(b + 2) * kW;
        const int ncq = (int)min((long long)kW, n - q0);
        double t[kRowsPerWarp];
#pragma unroll
        for (int cc = 0; cc < kRowsPerWarp; ++cc) {
            const int i = warp * kRowsPerWarp + cc;
            t[cc] = (active && i < ncq && CHK_TRI(sy, rowo + (q0 + i) * ld, n, ld)) ? (double)__ldg(row + (q0 + i) * ld) : 0.0;
        }
        double xv[R];
        wait_block<R>(sy, xtag, ep64, b + 2, who, xv);
#pragma unroll
        for (int cc = 0; cc < kRowsPerWarp; ++cc)
#pragma unroll
            for (int r = 0; r < R; ++r)
                acc[r] = fma(t[cc], __shfl_sync(kFull, xv[r], warp * kRowsPerWarp + cc), acc[r]);
    }
    // y_b: this chain's forward result, or the caller's
    double yv[R];
    if (a.back_only) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            yv[r] = (active && r0 + r < a.nr) ? (double)__ldcg(a.Y + (c0 + lane) * a.ys + (r0 + r) * a.cs) : 0.0;
    } else {
        wait_block<R>(sy, a.ytag + (size_t)c * a.nb * kW * R * 2, ep64, b, who, yv);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = acc[r];
    __syncthreads();
    double rv[R];  // y_b - sum_{q >= b+2} L_{b,q} x_q, row `lane`
#pragma unroll
    for (int r = 0; r < R; ++r) rv[r] = yv[r] - part_sum(S, 0, r, lane);
    // z'_b = U r: z_i = sum_{j >= i} U_ij r_j, the j split over the warps
    double pz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) pz[r] = 0.0;
#pragma unroll
    for (int jj = 0; jj < kRowsPerWarp; ++jj) {
        const int j = warp * kRowsPerWarp + jj;
#pragma unroll
        for (int r = 0; r < R; ++r) pz[r] = fma(u[jj], __shfl_sync(kFull, rv[r], j), pz[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[1][warp][r][lane] = pz[r];
    __syncthreads();
    double z[R];
#pragma unroll
    for (int r = 0; r < R; ++r) z[r] = part_sum(S, 1, r, lane);
    // x_b = z'_b - H_b x_{b+1}: the step that waits on the previous block
    double px[R];
#pragma unroll
    for (int r = 0; r < R; ++r) px[r] = 0.0;
    if (has_next) {
        double xv[R];
        wait_block<R>(sy, xtag, ep64, b + 1, who, xv, true);
#pragma unroll
        for (int jj = 0; jj < kRowsPerWarp; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r)
                px[r] = fma(h[jj], __shfl_sync(kFull, xv[r], warp * kRowsPerWarp + jj), px[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = px[r];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double x = z[r] - part_sum(S, 0, r, lane);
            put_tagged(xtag + tag_at<R>(b, lane, r), x, ep64);
            if (active && r0 + r < a.nr && CHK_RECT(sy, c0 + lane + (r0 + r) * a.ldb, a.n, a.nr, a.ldb))
                a.B[c0 + lane + (r0 + r) * a.ldb] = (T)x;
        }
    }
}

template <typename T, int R>
__global__ void __launch_bounds__(kSolveThreads) solve_kernel(SolveArgs<T> a)
{
    __shared__ SolveSmem<R> S;
    __shared__ int s_task, s_last;
    SyncArgs sy;
    sy.abort_flag = a.ctl + kCtlAbort;
    sy.status = a.status;
    sy.user_info = nullptr;
    sy.epoch = ld_relaxed_gpu(a.ctl + kCtlEpoch);
    sy.timeout_ns = a.timeout_ns;
    sy.chk_cut = a.chk_cut;
    const long long ep64 = (long long)sy.epoch << 32;
    const size_t tags = (size_t)a.chains * a.nb * kW * R * 2;
    // bounds-checked builds: the workspace regions inside their allocations
    const bool ws_in = CHK_REGION(sy, a.inv, (size_t)a.nb * kPrepMats * kW * kW * sizeof(double), a.ws_data, a.ws_data_bytes) &&
                       CHK_REGION(sy, a.uflag, (size_t)a.nb * sizeof(int), a.ws_iflags, a.ws_iflags_n * sizeof(int)) &&
                       CHK_REGION(sy, a.ytag, tags * sizeof(long long), a.ws_progress, a.ws_progress_n * sizeof(long long)) &&
                       CHK_REGION(sy, a.xtag, tags * sizeof(long long), a.ws_progress, a.ws_progress_n * sizeof(long long));
    (void)tags;

    const int nb = a.nb, steps = a.back_only ? nb : 2 * nb;
    for (;;) {
        if (threadIdx.x == 0) s_task = (!ws_in || aborted(sy)) ? -1 : atomicAdd(a.ctl + kCtlPairNext, 1);
        __syncthreads();
        const int t = s_task;
        if (t < 0 || t >= nb + a.chains * steps) break;
        if (t < nb) {
            // a back substitution starts at the last block
            prep_task<T>(a, sy, a.back_only ? nb - 1 - t : t, S.prep);
        } else {
            const int c = (t - nb) % a.chains, s = (t - nb) / a.chains + (a.back_only ? nb : 0);
            if (s < nb) forward_task<T, R>(a, sy, ep64, c, s, S);
            else backward_task<T, R>(a, sy, ep64, c, 2 * nb - 1 - s, S);
        }
        __syncthreads();
    }

    // The last block to finish zeroes the control words for the next launch
    // and advances the epoch.
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.ctl + kCtlExited, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int i = threadIdx.x; i < kCtlInts; i += blockDim.x)
            if (i != kCtlEpoch) a.ctl[i] = 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            a.ctl[kCtlEpoch] = a.ctl[kCtlEpoch] + 1;
            __threadfence();
        }
    }
}

// Right-hand sides of one launch, at most: 64 (their tagged words take
// 2 KB per row block and right-hand side), 16 above order 8192, where 16
// chains of one already keep the FP64 pipes busy.
int solve_group(long long n) { return n > 8192 ? kSolveChains : kSolveChains * kSolveRhs; }
// Right-hand sides per chain: one while the chains suffice for all (a step
// is shortest then), else as few as do.
int solve_rhs(int nr) { return nr <= kSolveChains ? 1 : nr <= 2 * kSolveChains ? 2 : kSolveRhs; }

template <typename T, int R>
int launch_solve(const void *L, long long n, long long ld, void *B, long long ldb, int nr, const Scratch &sc,
                 cudaStream_t stream, const T *Y, long long ys, long long cs)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return CHM_ERR_CUDA;
    static int occ[64] = {0};
    if (!occ[dev]) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, solve_kernel<T, R>, kSolveThreads, 0) !=
                cudaSuccess ||
            b < 1)
            return CHM_ERR_CUDA;
        occ[dev] = b;
    }
    const int nb = (int)((n + kW - 1) / kW);
    SolveArgs<T> a;
    a.L = static_cast<const T *>(L);
    a.n = n;
    a.ld = ld;
    a.B = static_cast<T *>(B);
    a.ldb = ldb;
    a.nb = nb;
    a.nr = nr;
    a.chains = (nr + R - 1) / R;
    a.Y = Y;
    a.ys = ys;
    a.cs = cs;
    a.back_only = Y != nullptr;
    a.inv = reinterpret_cast<double *>(sc.data);
    a.uflag = sc.iflags;
    a.ytag = sc.progress;
    a.xtag = sc.progress + (size_t)a.chains * nb * kW * R * 2;
    a.ctl = sc.ctl;
    a.status = sc.status;
    a.timeout_ns = timeout_ns();
    a.ws_data = sc.data;
    a.ws_data_bytes = sc.data_bytes;
    a.ws_iflags = sc.iflags;
    a.ws_iflags_n = sc.iflags_cap;
    a.ws_progress = sc.progress;
    a.ws_progress_n = sc.progress_cap;
    a.chk_cut = check_cut();
    const long long tasks = nb + (long long)a.chains * (a.back_only ? nb : 2 * nb);
    const int grid = (int)std::min<long long>(tasks, (long long)sm_count(dev) * occ[dev]);
    solve_kernel<T, R><<<grid, kSolveThreads, 0, stream>>>(a);
    return cudaGetLastError() == cudaSuccess ? CHM_OK : CHM_ERR_CUDA;
}

// Both substitutions, or (Y given) the back substitution alone.
template <typename T>
int solve_all(const void *L, long long n, long long ld, void *B, long long ldb, long long nrhs, const Scratch &sc,
              cudaStream_t stream, const T *Y = nullptr, long long ys = 0, long long cs = 0)
{
    T *b = static_cast<T *>(B);
    const int most = solve_group(n);
    for (long long r0 = 0; r0 < nrhs; r0 += most) {
        const int nr = (int)std::min<long long>(most, nrhs - r0);
        const T *y = Y ? Y + r0 * cs : nullptr;
        const int R = solve_rhs(nr);
        const int rc = R == 1   ? launch_solve<T, 1>(L, n, ld, b + r0 * ldb, ldb, nr, sc, stream, y, ys, cs)
                       : R == 2 ? launch_solve<T, 2>(L, n, ld, b + r0 * ldb, ldb, nr, sc, stream, y, ys, cs)
                                : launch_solve<T, kSolveRhs>(L, n, ld, b + r0 * ldb, ldb, nr, sc, stream, y, ys, cs);
        if (rc != CHM_OK) return rc;
    }
    return CHM_OK;
}

}  // namespace

ScratchNeed solve_need(long long n, long long nrhs)
{
    const size_t nb = (size_t)((n + kW - 1) / kW);
    const size_t nr = (size_t)std::min<long long>(std::max(1ll, nrhs), solve_group(n));
    const size_t R = (size_t)solve_rhs((int)nr), cols = (nr + R - 1) / R * R;
    ScratchNeed need;
    need.iflags = (nb + 63) & ~(size_t)63;
    need.progress = 2 * nb * kW * cols * 2;
    need.data = nb * kPrepMats * kW * kW * sizeof(double);
    return need;
}

int solve_enqueue(const void *L, long long n, long long ld, void *B, long long ldb, long long nrhs, int dtype,
                  const Scratch &sc, cudaStream_t stream)
{
    if (n <= 0 || nrhs <= 0) return CHM_OK;
    return dtype == CHM_F64 ? solve_all<double>(L, n, ld, B, ldb, nrhs, sc, stream)
                            : solve_all<float>(L, n, ld, B, ldb, nrhs, sc, stream);
}

int solve_back_enqueue(const void *L, long long n, long long ld, void *B, long long ldb, long long nrhs,
                       const void *Y, long long ys, long long cs, int dtype, const Scratch &sc, cudaStream_t stream)
{
    if (n <= 0 || nrhs <= 0) return CHM_OK;
    return dtype == CHM_F64
               ? solve_all<double>(L, n, ld, B, ldb, nrhs, sc, stream, static_cast<const double *>(Y), ys, cs)
               : solve_all<float>(L, n, ld, B, ldb, nrhs, sc, stream, static_cast<const float *>(Y), ys, cs);
}

namespace {

int solve_dispatch(const void *L, long long n, long long ld, void *B, long long ldb, long long nrhs, int dtype,
                   cudaStream_t stream)
{
    if (n < 0 || nrhs < 0 || n > (1ll << 26)) return CHM_ERR_ARG;
    if (dtype != CHM_F64 && dtype != CHM_F32_MIXED) return CHM_ERR_ARG;
    if (ld < std::max(1ll, n) || ldb < std::max(1ll, n)) return CHM_ERR_ARG;
    const size_t elt = dtype == CHM_F64 ? 8 : 4;
    if (n > 0 && (!L || (uintptr_t)L % elt)) return CHM_ERR_ARG;
    if (n > 0 && nrhs > 0 && (!B || (uintptr_t)B % elt)) return CHM_ERR_ARG;
    if (n == 0 || nrhs == 0) return CHM_OK;
    int rc = check_reachable(L);
    if (rc == CHM_OK) rc = check_reachable(B);
    if (rc != CHM_OK) return rc;
    return with_stream_scratch(stream, solve_need(n, nrhs), [&](const Scratch &sc) {
        return dtype == CHM_F64 ? solve_all<double>(L, n, ld, B, ldb, nrhs, sc, stream)
                                : solve_all<float>(L, n, ld, B, ldb, nrhs, sc, stream);
    });
}

}  // namespace
}  // namespace chm

extern "C" int chm_solve(const void *L, int64_t n, int64_t ld, void *B, int64_t ldb, int64_t nrhs, int dtype,
                         chm_stream_t stream)
{
    return chm::solve_dispatch(L, n, ld, B, ldb, nrhs, dtype, (cudaStream_t)stream);
}
