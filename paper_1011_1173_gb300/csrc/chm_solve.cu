// Solve with a factor: B <- (L^T L)^{-1} B, the use a maintained Cholesky
// factor serves (Sec. 1).  A forward substitution with L^T (lower) followed
// by a back substitution with L (upper), both blocked by kW = 32 rows, in
// one persistent launch per group of right-hand sides.
//
// A launch runs C chains of R right-hand sides each.  Tasks are taken in
// order from a launch-wide counter by blocks of four warps: in stage t of the
// forward half
//   PREP(t + 4)  U_b = D_b^{-1} and G1_b = U_b^T L_{b-1,b}^T (D_b the diagonal
//                block, L_{p,b} the 32 x 32 tile in row block p and column
//                block b), shared by every chain;
//   PREP2(t + 4) G2_b = U_b^T L_{b-2,b}^T;
//   each chain's y_b = U_b^T (b_b - sum_{p<=b-3} L_{p,b}^T y_p) - G2_b y_{b-2} - G1_b y_{b-1}, b = t;
//   PREPH(t)     H1_b = U_b L_{b,b+1} and H2_b = U_b L_{b,b+2};
// and in the backward half, b = nb - 1 .. 0,
//   each chain's x_b = U_b (y_b - sum_{q>=b+3} L_{b,q} x_q) - H2_b x_{b+2} - H1_b x_{b+1}.
// A task waits only on tasks taken before it, so the launch cannot deadlock
// whatever the number of resident blocks.
//
// A step sums the tiles whose y is already published, staged through shared
// memory (a lane reads down its column; tile_sum), the third and fourth tiles back
// split over the four warps, and multiplies by U; between one block's result and the next
// block's there is one 32 x 32 product (eight FMAs per warp and right-hand
// side), one barrier and a four-way sum.  With the two nearest tiles
// multiplied by U beforehand a step has three steps' time from y_{b-3} on
// (with one, y_{b-2}'s way through the tile and U set the pace: 1.7 us a step
// at n = 5000).  Results pass between blocks as epoch-tagged doubles (no
// fence, no flag).
//
// Why chains: right-hand sides do not depend on each other, and a step is
// bound by FP64 issue (one FP64 instruction per 64 cycles and warp), so a
// step of four right-hand sides takes three times a step of one.  C chains
// side by side fill the SMs that one chain leaves idle; the tiles they share
// meet in L2, and U, G and H are formed once instead of once per four
// right-hand sides.  n = 5000, float64: 16 right-hand sides 0.91 ms in 16
// chains against 6.96 ms as four launches of four right-hand sides each (the
// FP64 rate allows 0.76 ms: 400 M FMAs), one right-hand side 0.41 against
// 0.53 ms, bound by the chain: 314 steps of 1.3 us.
#include <float.h>

#include <algorithm>

#include "chm.h"
#include "chm_internal.h"
#include "chm_sub.cuh"

namespace chm {
namespace {

using namespace chm::sub;

constexpr int kSolveRhs = 4;      // right-hand sides per chain (largest)
constexpr int kSolveChains = 16;  // chains per launch (largest)
constexpr int kAhead = 4;         // stages by which PREP runs ahead of the chains
constexpr int kPrepMats = 5;      // U_b, G1_b, G2_b, H1_b and H2_b
constexpr size_t kMat = kW * kW;

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
    double *inv;      // [nb][kPrepMats][kW][kW]: U_b = D_b^{-1} (row i at i * kW), G1_b, G2_b, H1_b and
                      // H2_b (transposed: element (i, j) at j * kW + i)
    int *uflag, *gflag, *g2flag, *hflag;  // [nb] each: U, G1, G2, both H published (== epoch)
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

// Shared memory of a block: a preparation task's matrices or a step's tiles
// and partial sums.
template <typename T, int R>
union SolveSmem {
    PrepSmem prep;
    struct {
        T tile[kWarps][2][kW * pass::Stride<T>::value];
        alignas(16) double y[kWarps][R][kW][sizeof(T) == 4 ? 2 : 1];  // a tile's values (in float, as three floats)
        double part[2][kWarps][R][kW];
    };
    __device__ SolveSmem() {}
};

template <int R>
__device__ __forceinline__ size_t tag_at(int blk, int i, int r)
{
    return (((size_t)blk * kW + i) * R + r) * 2;
}

// Sum of the four warps' partial products of row `lane`, for each r.
template <typename T, int R>
__device__ __forceinline__ double part_sum(const SolveSmem<T, R> &S, int buf, int r, int lane)
{
    return (S.part[buf][0][r][lane] + S.part[buf][1][r][lane]) + (S.part[buf][2][r][lane] + S.part[buf][3][r][lane]);
}

// The tile at row block p, column block q: F[j][m] = L[p kW + j, q kW + m] (`rows`), or
// F[j][m] = L[p kW + m, q kW + j]; zero past the order.
template <typename T>
__device__ __forceinline__ void load_tile(const SolveArgs<T> &a, const SyncArgs &sy, int p, int q, bool rows, PrepSmem &S)
{
    (void)sy;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads, i = e & (kW - 1), j = e / kW;
        const long long r = (long long)p * kW + i, c = (long long)q * kW + j, o = r + c * a.ld;
        const double v = (r < a.n && c < a.n && CHK_TRI(sy, o, a.n, a.ld)) ? (double)__ldg(a.L + o) : 0.0;
        if (rows) S.F[i][j] = v;
        else S.F[j][i] = v;
    }
}

// U_b, and for the forward half G1_b.
template <typename T>
__device__ void prep_task(const SolveArgs<T> &a, const SyncArgs &sy, int b, PrepSmem &S)
{
    const int lane = threadIdx.x & 31;
    const long long n = a.n, ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool above = b >= 1 && !a.back_only;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads, i = e & (kW - 1), j = e / kW;
        double d = i == j ? 1.0 : 0.0;  // identity beyond the order
        if (j < nc && i <= j) d = CHK_TRI(sy, c0 + i + (c0 + j) * ld, n, ld) ? (double)__ldg(a.L + c0 + i + (c0 + j) * ld) : 0.0;
        S.D[i][j] = d;
        S.U[i][j] = 0.0;
    }
    if (above) load_tile(a, sy, b - 1, b, true, S);
    __syncthreads();
    double d = S.D[lane][lane];
    if (threadIdx.x < 32 && !(d > 0.0 && d <= DBL_MAX)) {  // not a Cholesky factor
        record_error(sy, kStatusNotPD, c0 + lane);
        d = 1.0;
    }
    __syncwarp();
    invert_block(S, d);
    double *inv = a.inv + (size_t)b * kPrepMats * kMat;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads;
        __stcg(inv + e, S.U[e / kW][e & (kW - 1)]);
    }
    publish(a.uflag + b, sy.epoch);
    if (above) {
        form_g(S, inv + kMat);
        publish(a.gflag + b, sy.epoch);
    }
}

// U_b from PREP(b).
template <typename T>
__device__ __forceinline__ const double *take_u(const SolveArgs<T> &a, const SyncArgs &sy, int b, PrepSmem &S)
{
    wait_flags(sy, a.uflag, b, b, b);
    const double *inv = a.inv + (size_t)b * kPrepMats * kMat;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads;
        S.U[e / kW][e & (kW - 1)] = __ldcg(inv + e);
    }
    return inv;
}

// G2_b.
template <typename T>
__device__ void prep2_task(const SolveArgs<T> &a, const SyncArgs &sy, int b, PrepSmem &S)
{
    if (b < 2) return;
    load_tile(a, sy, b - 2, b, true, S);
    take_u(a, sy, b, S);
    __syncthreads();
    form_g(S, a.inv + ((size_t)b * kPrepMats + 2) * kMat);
    publish(a.g2flag + b, sy.epoch);
}

// H1_b and H2_b: out[j kW + i] = H[i][j] = sum_{m>=i} U[i][m] L[m, j]; rows
// i = warp, warp + 4, ..., lane = j (see form_g).
template <typename T>
__device__ void preph_task(const SolveArgs<T> &a, const SyncArgs &sy, int b, PrepSmem &S)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    take_u(a, sy, b, S);
    for (int h = 1; h <= 2 && b + h < a.nb; ++h) {
        load_tile(a, sy, b, b + h, false, S);
        __syncthreads();
        double acc[kPer];
#pragma unroll
        for (int ii = 0; ii < kPer; ++ii) acc[ii] = 0.0;
#pragma unroll
        for (int m = 0; m < kW; ++m) {
            const double f = S.F[lane][m];
#pragma unroll
            for (int ii = 0; ii <= m / kWarps; ++ii) acc[ii] = fma(S.U[ii * kWarps + warp][m], f, acc[ii]);
        }
        double *out = a.inv + ((size_t)b * kPrepMats + 2 + h) * kMat;
#pragma unroll
        for (int ii = 0; ii < kPer; ++ii) __stcg(out + (size_t)lane * kW + ii * kWarps + warp, acc[ii]);
        __syncthreads();
    }
    publish(a.hflag + b, sy.epoch);
}

// t[j] = L[row j, column lane] of a staged tile.
template <typename T>
__device__ __forceinline__ void tile_column(const T *tl, T (&t)[kW])
{
    constexpr int E = 16 / (int)sizeof(T);
    using V16 = typename pass::Vec16<T>::type;
#pragma unroll
    for (int j = 0; j < kW; j += E) {
        const V16 x = *reinterpret_cast<const V16 *>(tl + j);
#pragma unroll
        for (int e = 0; e < E; ++e) t[j + e] = pass::vget<T>(x, e);
    }
}
// acc[r] += sum over a tile's 32 entries of t[j] v_j[r], lane j holding v_j;
// y is the warp's space for them.
template <int R>
__device__ __forceinline__ void tile_sum(const double (&t)[kW], const double (&v)[R], double (*y)[kW][1], int lane,
                                         double (&acc)[R])
{
#pragma unroll
    for (int r = 0; r < R; ++r) y[r][lane][0] = v[r];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kW; j += 2)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double2 u = *reinterpret_cast<const double2 *>(y[r][j]);
            acc[r] = fma(t[j], u.x, acc[r]);
            acc[r] = fma(t[j + 1], u.y, acc[r]);
        }
    __syncwarp();
}
// For a factor in float: a conversion is as slow as an FMA in double (64
// cycles a warp instruction), and together they bound every solve but the
// smallest.  The values are scaled by a power of two to below 2^-5 (so that
// no sum of products with the factor's entries overflows) and split into three
// floats that hold all of their 53 bits; the products are split exactly, and
// the tile's sum is kept in three floats, two of them added to exactly
// (two-sum): to about 2^-70 of the sum of its terms' sizes, against 2^-50 in double.  The
// tiles' sums are added up in double.  A tile costs 1090 FP32 and 15 FP64
// instructions a right-hand side instead of 64 FP64 ones: n = 16384, 1 / 8
// right-hand sides 1.70 / 4.11 ms against 2.18 / 8.96.
//
// What a float cannot hold is lost below 2^-150: of each value, so 2^-145 max
// |t| of the sum, and of each product's parts, 2^-143.  A double sum is off by
// 2^-53 of its largest term or more, which is at least the smallest value
// (that is not zero) times max |t| (over those).  Where that is not above
// 2^-88 or the smallest value not above 2^-90 (values or entries that differ by
// tens of orders of magnitude, entries next to a float's smallest), and where a
// value is not finite, the warp sums the tile in double (n = 16384 with columns
// between 1e-18 and 1e18: 1.88 / 6.78 ms).  The test costs 3 to 5 % where the
// FP32 rate binds.
__device__ __forceinline__ void two_sum(float &s, float x, float &err)
{
    const float u = __fadd_rn(s, x), b = __fsub_rn(u, s);
    err = __fadd_rn(__fsub_rn(s, __fsub_rn(u, b)), __fsub_rn(x, b));
    s = u;
}
template <int R>
__device__ __forceinline__ void tile_sum(const float (&t)[kW], const double (&v)[R], double (*y)[kW][2], int lane,
                                         double (&acc)[R])
{
    double up[R];
    bool plain = false;  // the tile is summed in double
    // (four entries are large enough nearly always)
    const float four = fmaxf(fmaxf(fabsf(t[0]), fabsf(t[9])), fmaxf(fabsf(t[18]), fabsf(t[27])));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // the largest value's exponent, kept where both powers of two are finite, and the smallest's
        const unsigned hi = (unsigned)__double2hiint(v[r]) & 0x7fffffffu;
        const bool some = (hi | (unsigned)__double2loint(v[r])) != 0u;
        const int top = (int)(__reduce_max_sync(kFull, hi) >> 20), ex = min(max(top, 64), 2000);
        const int low = (int)(__reduce_min_sync(kFull, some ? hi : 0x7fffffffu) >> 20) - ex - 6;
        auto above = [&](float m) { return low >= -90 && (__float_as_int(m) >> 23) - 127 + low >= -88; };
        const unsigned which = __ballot_sync(kFull, some);
        if (top == 0x7ff || which != kFull || !__all_sync(kFull, above(four))) {
            float m = 0.0f;
#pragma unroll
            for (int j = 0; j < kW; ++j)
                if (which >> j & 1u) m = fmaxf(m, fabsf(t[j]));
            if (top == 0x7ff || !__all_sync(kFull, m == 0.0f || above(m))) plain = true;
        }
        up[r] = __hiloint2double((ex + 6) << 20, 0);
        double x = v[r] * __hiloint2double((2040 - ex) << 20, 0);
        const float h = (float)x;
        x -= (double)h;
        const float l = (float)x;
        *reinterpret_cast<float4 *>(y[r][lane]) = make_float4(h, l, (float)(x - (double)l), 0.0f);
    }
    __syncwarp();
    if (plain) {
#pragma unroll
        for (int r = 0; r < R; ++r) y[r][lane][0] = v[r];
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kW; ++j) {
            const double f = (double)t[j];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(f, y[r][j][0], acc[r]);
        }
        __syncwarp();
        return;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float s = 0.0f, e = 0.0f, l = 0.0f;
#pragma unroll
        for (int j = 0; j < kW; ++j) {
            const float4 u = *reinterpret_cast<const float4 *>(y[r][j]);
            const float p = __fmul_rn(t[j], u.x), d = fmaf(t[j], u.x, -p);
            const float q = __fmul_rn(t[j], u.y), g = fmaf(t[j], u.z, fmaf(t[j], u.y, -q));
            float e0, e1, e2, e3;
            two_sum(s, p, e0);
            two_sum(e, d, e1);
            two_sum(e, q, e2);
            two_sum(e, e0, e3);
            l = __fadd_rn(l, __fadd_rn(__fadd_rn(g, e1), __fadd_rn(e2, e3)));
        }
        acc[r] = fma((double)s + ((double)e + (double)l), up[r], acc[r]);
    }
    __syncwarp();
}

// Chain c's step at block b, forward.
template <typename T, int R>
__device__ void forward_task(const SolveArgs<T> &a, const SyncArgs &sy, long long ep64, int c, int b, SolveSmem<T, R> &S)
{
    constexpr int SD = pass::Stride<T>::value;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = a.n, ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool active = lane < nc;
    const int r0 = c * R;  // this chain's first right-hand side
    long long *ytag = a.ytag + (size_t)c * a.nb * kW * R * 2;
    const bool vec = ((ld * (long long)sizeof(T)) & 15) == 0 && (reinterpret_cast<uintptr_t>(a.L) & 15) == 0;

    double rhs[R];
#pragma unroll
    for (int r = 0; r < R; ++r)
        rhs[r] = (active && r0 + r < a.nr && CHK_RECT(sy, c0 + lane + (r0 + r) * a.ldb, n, a.nr, a.ldb))
                     ? (double)a.B[c0 + lane + (r0 + r) * a.ldb] : 0.0;
    const int far = b - 4;  // tiles 0 .. far - 1; tiles b - 4 and b - 3 are split over the warps below
    auto stage = [&](int p, int slot) {
        if (p < far) stage_tile(sy, S.tile[warp][slot], a.L, ld, (long long)p * kW, c0, n, vec, false, lane);
        pass::cp_commit();
    };
    stage(warp, 0);
    // this warp's columns of G1_b and G2_b, taken before the tiles so that
    // behind y_{b-4} nothing but the chain's own values is waited for
    wait_flags(sy, a.uflag, b, b, b);
    if (b >= 1) wait_flags(sy, a.gflag, b, b, b);
    if (b >= 2) wait_flags(sy, a.g2flag, b, b, b);
    const double *inv = a.inv + (size_t)b * kPrepMats * kMat + warp * kPer * kW + lane;
    double g1[kPer], g2[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) {
        g1[jj] = b >= 1 ? __ldcg(inv + kMat + jj * kW) : 0.0;
        g2[jj] = b >= 2 ? __ldcg(inv + 2 * kMat + jj * kW) : 0.0;
    }
    // tiles p <= b - 5 of column block b, dealt round-robin to the warps (a
    // fixed order of the sums: results do not depend on timing)
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    int slot = 0;
    for (int p = warp; p < far; p += kWarps) {
        stage(p + kWarps, slot ^ 1);
        // (the tile's column in registers before y is waited for)
        pass::cp_wait<1>();
        __syncwarp();
        T t[kW];
        tile_column<T>(S.tile[warp][slot] + lane * SD, t);
        const long long *w = ytag + tag_at<R>(p, 0, 0);
        double y[R];
        // (a warp's last tile is waited for as closely as the chain's next steps)
        wait_vals<R>(sy, w + tag_at<R>(0, lane, 0), p + kWarps < far ? w + tag_at<R>(1, 0, 0) - 1 : nullptr, ep64, b, y);
        tile_sum<R>(t, y, S.y[warp], lane, acc);
        slot ^= 1;
    }
    pass::cp_wait<0>();
    // the steps before: a lane takes the values of one of its warp's eight rows
    auto tag_of = [&](int up) { return ytag + tag_at<R>(b - up, warp * kPer + (lane & (kPer - 1)), 0); };
    // this warp's rows of tiles b - 4 and b - 3, and of U_b
    const long long o4 = (long long)(b - 4) * kW + warp * kPer + (c0 + (active ? lane : 0)) * ld;
    double t4[kPer], t3[kPer], u[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) {
        t4[jj] = (b >= 4 && active && CHK_TRI(sy, o4 + jj, n, ld)) ? (double)__ldg(a.L + o4 + jj) : 0.0;
        t3[jj] = (b >= 3 && active && CHK_TRI(sy, o4 + kW + jj, n, ld)) ? (double)__ldg(a.L + o4 + kW + jj) : 0.0;
    }
    if (b >= 4) {
        double y[R];
        wait_vals<R>(sy, tag_of(4), nullptr, ep64, b, y);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t4[jj], __shfl_sync(kFull, y[r], jj), acc[r]);
    }
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) u[jj] = __ldcg(inv + jj * kW);
    if (b >= 3) {
        double y[R];
        wait_vals<R>(sy, tag_of(3), nullptr, ep64, b, y);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t3[jj], __shfl_sync(kFull, y[r], jj), acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = acc[r];
    __syncthreads();
    double pz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double rv = rhs[r] - part_sum(S, 0, r, lane);
        pz[r] = 0.0;
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj) pz[r] = fma(u[jj], __shfl_sync(kFull, rv, warp * kPer + jj), pz[r]);
    }
    if (b >= 2) {
        double y[R];
        wait_vals<R>(sy, tag_of(2), nullptr, ep64, b, y);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) pz[r] = fma(-g2[jj], __shfl_sync(kFull, y[r], jj), pz[r]);
    }
    if (b >= 1) {
        double y[R];
        wait_vals<R>(sy, tag_of(1), nullptr, ep64, b, y);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) pz[r] = fma(-g1[jj], __shfl_sync(kFull, y[r], jj), pz[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[1][warp][r][lane] = pz[r];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) put_tagged(ytag + tag_at<R>(b, lane, r), part_sum(S, 1, r, lane), ep64);
    }
}

// Chain c's step at block b, backward.
template <typename T, int R>
__device__ void backward_task(const SolveArgs<T> &a, const SyncArgs &sy, long long ep64, int c, int b, SolveSmem<T, R> &S)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = a.n, ld = a.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool active = lane < nc;
    const int r0 = c * R, nb = a.nb;
    long long *xtag = a.xtag + (size_t)c * nb * kW * R * 2;

    // this warp's columns of H1_b and H2_b
    wait_flags(sy, a.uflag, b, b, b);
    wait_flags(sy, a.hflag, b, b, b);
    const double *inv = a.inv + (size_t)b * kPrepMats * kMat;
    double h1[kPer], h2[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) {
        const int j = warp * kPer + jj;
        h1[jj] = b + 1 < nb ? __ldcg(inv + 3 * kMat + j * kW + lane) : 0.0;
        h2[jj] = b + 2 < nb ? __ldcg(inv + 4 * kMat + j * kW + lane) : 0.0;
    }
    // tiles q >= b + 5 of row block b, from the last one up, dealt
    // round-robin to the warps; lane = row of the block, so each column of a
    // tile is one coalesced read
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    const long long rowo = c0 + (active ? lane : 0);
    const T *row = a.L + rowo;
    for (int q = nb - 1 - warp; q >= b + 5; q -= kWarps) {
        const long long q0 = (long long)q * kW;
        const int ncq = (int)min((long long)kW, n - q0);
        T t[kW];
#pragma unroll
        for (int i = 0; i < kW; ++i)
            t[i] = (active && i < ncq && CHK_TRI(sy, rowo + (q0 + i) * ld, n, ld)) ? __ldg(row + (q0 + i) * ld) : T(0);
        const long long *w = xtag + tag_at<R>(q, 0, 0);
        double x[R];
        wait_vals<R>(sy, w + tag_at<R>(0, lane, 0), q - kWarps >= b + 5 ? w + tag_at<R>(1, 0, 0) - 1 : nullptr, ep64, b, x);
        tile_sum<R>(t, x, S.y[warp], lane, acc);
    }
    // y_b: this chain's forward result, or the caller's
    double yv[R];
    if (a.back_only) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            yv[r] = (active && r0 + r < a.nr) ? (double)__ldcg(a.Y + (c0 + lane) * a.ys + (r0 + r) * a.cs) : 0.0;
    } else {
        wait_vals<R>(sy, a.ytag + (size_t)c * nb * kW * R * 2 + tag_at<R>(b, lane, 0), nullptr, ep64, b, yv);
    }
    auto tag_of = [&](int dn) { return xtag + tag_at<R>(b + dn, warp * kPer + (lane & (kPer - 1)), 0); };
    // this warp's columns of tiles b + 4 and b + 3, and of U_b
    double t4[kPer], t3[kPer], u[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) {
        const long long q3 = (long long)(b + 3) * kW + warp * kPer + jj, q4 = q3 + kW;
        t4[jj] = (active && q4 < n && CHK_TRI(sy, rowo + q4 * ld, n, ld)) ? (double)__ldg(row + q4 * ld) : 0.0;
        t3[jj] = (active && q3 < n && CHK_TRI(sy, rowo + q3 * ld, n, ld)) ? (double)__ldg(row + q3 * ld) : 0.0;
    }
    if (b + 4 < nb) {
        double x[R];
        wait_vals<R>(sy, tag_of(4), nullptr, ep64, b, x);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t4[jj], __shfl_sync(kFull, x[r], jj), acc[r]);
    }
#pragma unroll
    for (int jj = 0; jj < kPer; jj += 2) {
        const double2 x = __ldcg(reinterpret_cast<const double2 *>(inv + lane * kW + warp * kPer + jj));
        u[jj] = x.x;
        u[jj + 1] = x.y;
    }
    if (b + 3 < nb) {
        double x[R];
        wait_vals<R>(sy, tag_of(3), nullptr, ep64, b, x);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(t3[jj], __shfl_sync(kFull, x[r], jj), acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[0][warp][r][lane] = acc[r];
    __syncthreads();
    double pz[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double rv = yv[r] - part_sum(S, 0, r, lane);
        pz[r] = 0.0;
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj) pz[r] = fma(u[jj], __shfl_sync(kFull, rv, warp * kPer + jj), pz[r]);
    }
    if (b + 2 < nb) {
        double x[R];
        wait_vals<R>(sy, tag_of(2), nullptr, ep64, b, x);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) pz[r] = fma(-h2[jj], __shfl_sync(kFull, x[r], jj), pz[r]);
    }
    if (b + 1 < nb) {
        double x[R];
        wait_vals<R>(sy, tag_of(1), nullptr, ep64, b, x);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
#pragma unroll
            for (int r = 0; r < R; ++r) pz[r] = fma(-h1[jj], __shfl_sync(kFull, x[r], jj), pz[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) S.part[1][warp][r][lane] = pz[r];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double x = part_sum(S, 1, r, lane);
            put_tagged(xtag + tag_at<R>(b, lane, r), x, ep64);
            if (active && r0 + r < a.nr && CHK_RECT(sy, c0 + lane + (r0 + r) * a.ldb, n, a.nr, a.ldb))
                a.B[c0 + lane + (r0 + r) * a.ldb] = (T)x;
        }
    }
}

// Tasks of a launch: 2 kAhead to start with, then per stage kStageExtra and
// one per chain (in the backward half of both: the chains' alone).
constexpr int kStageExtra = 3;
__host__ __device__ inline int solve_tasks(int nb, int chains, bool back_only)
{
    return 2 * kAhead + nb * (kStageExtra + chains) + (back_only ? 0 : nb * chains);
}

template <typename T, int R>
__global__ void __launch_bounds__(kThreads, R == 1 ? 3 : 2) solve_kernel(SolveArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char raw[];
    SolveSmem<T, R> &S = *reinterpret_cast<SolveSmem<T, R> *>(raw);
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
                       CHK_REGION(sy, a.uflag, 4 * (size_t)a.nb * sizeof(int), a.ws_iflags, a.ws_iflags_n * sizeof(int)) &&
                       CHK_REGION(sy, a.ytag, tags * sizeof(long long), a.ws_progress, a.ws_progress_n * sizeof(long long)) &&
                       CHK_REGION(sy, a.xtag, tags * sizeof(long long), a.ws_progress, a.ws_progress_n * sizeof(long long));
    (void)tags;

    const int nb = a.nb, total = solve_tasks(nb, a.chains, a.back_only);
    const int per = kStageExtra + a.chains;
    for (;;) {
        if (threadIdx.x == 0) s_task = (!ws_in || aborted(sy)) ? -1 : atomicAdd(a.ctl + kCtlPairNext, 1);
        __syncthreads();
        const int t = s_task;
        if (t < 0 || t >= total) break;
        // the task: a preparation (0 PREP, 1 PREP2, 2 PREPH) of the i-th block the
        // launch comes to, or chain c's step
        int prep = -1, i = 0, c = 0, s = 0;
        if (t < 2 * kAhead) {
            prep = t & 1;
            i = t >> 1;
        } else if (t < 2 * kAhead + nb * per) {
            const int x = t - 2 * kAhead, r = x % per;
            s = x / per;
            if (r < 2) {
                prep = r;
                i = s + kAhead;
            } else if (r < 2 + a.chains) {
                c = r - 2;
            } else {
                prep = 2;
                i = s;
            }
        } else {
            const int x = t - 2 * kAhead - nb * per;
            c = x % a.chains;
            s = nb + x / a.chains;
        }
        if (a.back_only) {
            // a back substitution comes to the last block first and needs no G
            const int b = nb - 1 - i;
            if (prep == 0 && b >= 0) prep_task<T>(a, sy, b, S.prep);
            else if (prep == 1 && b >= 0) preph_task<T>(a, sy, b, S.prep);
            else if (prep < 0) backward_task<T, R>(a, sy, ep64, c, nb - 1 - s, S);
        } else if (prep >= 0) {
            if (i < nb) {
                if (prep == 0) prep_task<T>(a, sy, i, S.prep);
                else if (prep == 1) prep2_task<T>(a, sy, i, S.prep);
                else preph_task<T>(a, sy, i, S.prep);
            }
        } else if (s < nb) {
            forward_task<T, R>(a, sy, ep64, c, s, S);
        } else {
            backward_task<T, R>(a, sy, ep64, c, 2 * nb - 1 - s, S);
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
constexpr long long kSolveWide = 8192;
int solve_group(long long n) { return n > kSolveWide ? kSolveChains : kSolveChains * kSolveRhs; }
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
    const int smem = (int)sizeof(SolveSmem<T, R>);
    if (!occ[dev]) {
        int b = 0;
        if (cudaFuncSetAttribute(solve_kernel<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, solve_kernel<T, R>, kThreads, smem) != cudaSuccess ||
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
    a.gflag = a.uflag + nb;
    a.g2flag = a.gflag + nb;
    a.hflag = a.g2flag + nb;
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
    const int grid = (int)std::min<long long>(solve_tasks(nb, a.chains, a.back_only), (long long)sm_count(dev) * occ[dev]);
    solve_kernel<T, R><<<grid, kThreads, smem, stream>>>(a);
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

// What this solve takes or, where more, what a smaller one does: up to order
// 8192 a launch holds four times the right-hand sides, so that the tagged words
// of an order above it can be fewer (a stream's workspace, once it served a
// solve, serves every smaller one without growing).
ScratchNeed solve_need(long long n, long long nrhs)
{
    const size_t nb = (size_t)((n + kW - 1) / kW);
    auto tags = [&](long long m) {
        const size_t nr = (size_t)std::min<long long>(std::max(1ll, nrhs), solve_group(m));
        const size_t R = (size_t)solve_rhs((int)nr), cols = (nr + R - 1) / R * R;
        return 2 * (size_t)((m + kW - 1) / kW) * kW * cols * 2;
    };
    ScratchNeed need;
    need.iflags = (4 * nb + 63) & ~(size_t)63;
    need.progress = std::max(tags(n), tags(std::min(n, kSolveWide)));
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
