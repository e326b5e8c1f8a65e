// Team kernel of the rank-k up/downdate (Walder 2010, Algorithm 1): one
// persistent launch that carries one or many independent factors, for
// factors that stay in L2.  It evaluates the same exact identities as the
// pass kernels (chm_pass.cuh), in passes of up to kTeamKb = 8 vectors:
//   P = F^{-T} V;  the prefix Grams H_r = Sigma + sum_{i<r} p_i p_i^T and
//   their factors L |D| Sigma L^T, which fix every rotation's coefficients
//   (Compute);  and the scaled Apply sweep, two FMAs per element and vector.
//
// Work split.  Every piece of a pass is a task of one thread block (four
// warps), and the tasks of a factor are numbered in an order in which each
// waits only on tasks before it, so that a launch of any number of resident
// blocks progresses.  Blocks take a factor's tasks from its ticket word; a
// factor is worked on by a team of blocks, and the launch holds G teams.
//   PREP(b)   U_b = D_b^{-1} and G1_b = U_b^T F_{b-1,b}^T of diagonal block b,
//             and whether D_b is so ill-conditioned that SUB substitutes
//             through it instead (see is_hard)
//   PREP2(b)  G2_b = U_b^T F_{b-2,b}^T
//   SUB(c, b) step b of the forward substitution of vector c:
//               p_b = U_b^T (v_b - sum_{r<=b-3} F_{r,b}^T p_r) - G2_b p_{b-2} - G1_b p_{b-1}.
//             The tiles above are summed as their p arrive, and what is left
//             of v at the start of every sweep segment is kept.  After
//             p_{b-1} there is one 32 x 32 product, eight FMAs a warp.
//   COEF(b)   the prefix Grams of row block b's rows, their LDL^T (where that
//             would cancel, factors carried from row to row) and the rows'
//             sweep coefficients
//   SWEEP(b, s) segments of column block b (`seg` row blocks each): the
//             carries restart from the kept residual, and every tile is
//             read, rotated and written once per pass
// A column is swept only after its substitution step, which is the last
// reader of its tiles as they entered the pass, so no tile needs a flag of
// its own; the next pass of a factor enters column b once b's sweep is done.
//
// What bounds it.  A vector's substitution is the serial chain: nb steps of
// 1.3 us (a value through L2, 8 FMAs at one FP64 instruction per 64 cycles
// and warp, a barrier, a four-way sum; up to 2 us where sweeps share the FP64
// pipes).  Vectors do not wait for each other, and nothing else is on the
// chain: the sweep trails it by one segment, whatever the number of vectors.
// With many vectors or factors the FP64 rate binds (three FMAs per element
// and vector: one in the substitution, two in the sweep).  n = 5000 in double,
// one call: k = 1 0.38 ms (the wave kernel 1.04), k = 16 1.69 ms (1.93), of
// which the FMAs are 0.05 and 1.1 ms.
//
// Precision: CHM_F64 is double throughout; what the identities would lose
// where Grams or diagonal blocks are ill-conditioned is avoided (Carried,
// is_hard).  CHM_F32_MIXED substitutes in double (P, U, G) with the far sums in
// pairs of floats (48 bits), forms the coefficients in double, and sweeps in
// float; the diagonal is carried in double through all passes of the launch and
// rounded to float at the end of each.
#pragma once

#include "chm_sub.cuh"
#include "chm_team_layout.h"

namespace chm {
namespace team {

using namespace chm::sub;

template <typename T>
struct Launch {
    const Prob *probs;  // device array [nprobs]; null: the one problem is prob0
    Prob prob0;
    int nprobs, nteams;
    int *ctl;           // kCtlInts control words
    long long *status;  // sticky {status, row} of the scratch owner
    long long *trace;   // optional timestamps of the one problem, [k][nb][kTracePoints]
    long long timeout_ns;
    int skip_publish;   // test hook: vector 0's step at this block is never published (-1: none)
    // the workspace allocations the problems' regions are carved from (bounds-checked builds)
    const char *ws_data;
    size_t ws_data_bytes;
    const int *ws_iflags;
    size_t ws_iflags_n;
    const long long *ws_progress;
    size_t ws_progress_n;
    long long chk_cut;  // bounds-checked build: columns taken off each factor's declared extent
};

// One pass of one problem, in shared memory: written by thread 0 when the
// block takes up the problem or its next pass.
template <typename T>
struct View {
    T *L;
    const T *V;  // the pass's first vector
    long long n, ld, ldv;
    int nb, pass, npass, kb, KB, seg, nbound, look, units;
    unsigned down_mask;  // bit q: vector q of the pass is a downdate
    bool vec;            // 16-byte column segments
    double *ug;          // [nb][3][kW][kW]: U_b (row i at i * kW), G1_b and G2_b (element (i, j) at j * kW + i)
    T *coef;             // [nb * kW][2 KB]
    T *escale;           // [nb * kW]
    double *dfac;        // [nb * kW]
    T *snap;             // [nbound][nb * kW][KB]
    double *rst;         // [nbound][KB (KB + 1) / 2]: packed unit lower factor, 1 / |D_q| on the diagonal
    double *dcar;        // [nb * kW]: the diagonal, carried in double from pass to pass
    long long *ptag;     // [kb][nb][kW][2]
    long long *htag;     // [nb][KB (KB + 1) / 2][2]: the Gram before block b + 1
    long long *ftag;     // [nb][KB (KB + 1) / 2][2]: its factor, where the Gram is ill-conditioned (else infinity)
    int *uflag, *gflag, *g2flag, *cflag;  // [nb] each: U, G1, G2, coefficients published (== epoch)
    int *hflag;          // [nb]: whether block b is multiplied by U (epoch) or substituted (-epoch)
    long long *sdone;    // [nb]: sweep tasks of a column finished, all passes (epoch-tagged count)
    SyncArgs sync;
};

// A block's cursor in the list of a pass's tasks.
struct Stage {
    int t;        // stage
    int first;    // its first task
    int passes;   // tasks of the passes before
    int segs;     // segments of column t - look (once that is a column)
    int left;     // columns until there is one more
};

template <typename T>
struct SubSmem {
    T tile[2][kWarps][kW * pass::Stride<T>::value];  // two groups of four tiles, [column][row]
    double part[4][kWarps][kW];        // the warps' sums at segment starts, in turn
    double fin[kWarps][kW];            // and behind the tiles
    double y[kWarps][kW];              // a group's values of p, or their float pairs
    double z[kW];                      // the entries of v
};
struct CoefSmem {
    static constexpr int ne = kTeamKb * (kTeamKb + 1) / 2;
    static constexpr int hs = ne | 1;
    double H[kW][hs];       // row r: its prefix Gram, then its factor
    double g[8][ne];        // the Grams of the threads' shares of the rows
    double p[kW][kTeamKb + 1];
    double z[kW][kTeamKb + 1];
    double p0[kW][kTeamKb + 1];  // p again (p becomes z = L^{-1} p)
    double size[kTeamKb];        // the sizes of the Gram's diagonal behind the block
    double l0[ne];               // the factor handed on by the block before, |D_q| on its diagonal
    unsigned ill[kWarps];        // per warp: four bits a row, set where its Gram is ill-conditioned
    double M[ne];                // from l0 on: the Gram behind the block, then its factor, |D_q| on the diagonal
    int have;                    // what the block before has handed on
};
// A sweep task's segments: NV warps pass a tile on, so NV + 1 tiles are in
// flight per segment.
template <typename T, int KB, int NV>
struct SweepSmem {
    static constexpr int NS = NV + 1, UNITS = kWarps / NV;
    struct Unit {
        T tile[NS][kW * pass::Stride<T>::value];
        T cf[NS][kW * 2 * KB];
        T e[NS][kW];
    } unit[UNITS];
};
template <typename T>
union TaskSmem {
    PrepSmem prep;
    SubSmem<T> sub;
    CoefSmem coef;
    SweepSmem<T, 1, 1> sweep1;
    SweepSmem<T, 1, 2> sweep12;
    SweepSmem<T, 2, 2> sweep2;
    SweepSmem<T, 4, 4> sweep4;
    SweepSmem<T, 8, 4> sweep8;
    __device__ TaskSmem() {}
};


// Stamp `pt` of column block b of vector c (diagnostics): 0 SUB taken, 1 its
// tiles summed, 2 what is left multiplied by U, 3 the previous step seen, 4
// its result put; for the pass's first vector 5 COEF's inputs in, 6 its
// results out, 7 the column's last segment swept.
#define TEAM_TRACE(c, b, pt)                                                                                     \
    do {                                                                                                         \
        if (P.trace && threadIdx.x == 0)                                                                         \
            P.trace[((size_t)(v.pass * kTeamKb + (c)) * v.nb + (b)) * kTracePoints + (pt)] = global_ns();        \
    } while (0)

// ---------------------------------------------------------------- PREP

// The next pass may enter column block b once the last one has swept it
// (every pass but the last has kTeamKb vectors, one column per task).
template <typename T>
__device__ __forceinline__ bool wait_column(const View<T> &v, int b)
{
    if (v.pass == 0) return true;
    const long long want = ((long long)v.sync.epoch << 32) + (long long)v.pass * segs_of(b, seg_of(v.nb, kTeamKb, sizeof(T) == 8));
    const bool ok = __all_sync(kFull, wait_ge(v.sync, v.sdone + b, want, b));
    __syncwarp();
    return ok;
}

// The tile `up` blocks above diagonal block b: F[j][m] = L[(b - up) kW + j, b kW + m].
template <typename T>
__device__ __forceinline__ void load_above(const View<T> &v, int b, int up, PrepSmem &S)
{
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, v.n - c0);
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads, i = e & (kW - 1), j = e / kW;
        const long long o = c0 - up * kW + i + (c0 + j) * v.ld;
        S.F[i][j] = (j < nc && CHK_TRI(v.sync, o, v.n, v.ld)) ? (double)__ldcg(v.L + o) : 0.0;
    }
}
// The size of x in units of 2^e, e the exponent in the high word e0 (`inverse`:
// of 2^-e), to 20 bits on the integer pipe; beyond float's range 0 or its largest.
__device__ __forceinline__ float coarse(double x, int e0, bool inverse)
{
    const int e = e0 & 0x7ff00000, h = __double2hiint(x) & 0x7fffffff;
    const int u = inverse ? min(h - 0x77f00000, 0x000fffff) + e : min(h - e, 0x10000000) + 0x07f00000;
    return __int_as_float(min(max(u, 0), 0x0fefffff) << 3);
}
// Whether p = U^T r would be less accurate than substituting through D: the
// product's residual D^T p - r is up to kappa = max_i sum_l (|D^T| |U^T|)_il
// roundings of |D^T| |p|, the substitution's one or two whatever D is.  kappa
// is 3 to 50 for the blocks of well-conditioned factors, where both leave the
// same error; from about 100 on the factor's error grows with it (smooth rows
// over a diagonal of 1e-4: kappa 900, 2e-13 instead of 9e-15).  Uses S.M.
__device__ __forceinline__ bool is_hard(PrepSmem &S)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float(*part)[kW] = reinterpret_cast<float(*)[kW]>(&S.M[0][0]);
    const int e0 = __double2hiint(S.D[0][0]);
    float s = 0.0f;
#pragma unroll
    for (int m = 0; m < kPer; ++m) s += coarse(S.U[warp * kPer + m][lane], e0, true);
    part[warp][lane] = s;
    __syncthreads();
    const float g = (part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]);
    s = 0.0f;
#pragma unroll
    for (int m = 0; m < kPer; ++m)
        s = fmaf(coarse(S.D[warp * kPer + m][lane], e0, false), __shfl_sync(kFull, g, warp * kPer + m), s);
    part[kWarps + warp][lane] = s;
    __syncthreads();
    const float kappa = (part[4][lane] + part[5][lane]) + (part[6][lane] + part[7][lane]);
    return __any_sync(kFull, !(kappa <= 64.0f)) != 0;
}
// U_b and G1_b, then the block's kind, which nothing waits for before its far
// tiles are summed.
template <typename T>
__device__ void prep_task(const Launch<T> &P, const View<T> &v, int b, PrepSmem &S)
{

    const SyncArgs &sy = v.sync;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long n = v.n, ld = v.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    (void)wait_column(v, b);
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = tid + x * kThreads, i = e & (kW - 1), j = e / kW;
        double d = 0.0;
        if (j < nc) {
            if (i == j && v.pass > 0) d = __ldcg(v.dcar + c0 + j);
            else if (i <= j && CHK_TRI(sy, c0 + i + (c0 + j) * ld, n, ld)) d = (double)__ldcg(v.L + c0 + i + (c0 + j) * ld);
        } else if (i == j) {
            d = 1.0;
        }
        S.D[i][j] = d;
        S.U[i][j] = 0.0;
    }
    if (b >= 1) load_above(v, b, 1, S);
    __syncthreads();
    double d = S.D[lane][lane];
    if (warp == 0) {
        const bool bad = lane < nc && !(d > 0.0 && d <= DBL_MAX);
        const unsigned badm = __ballot_sync(kFull, bad);
        if (badm && lane == 0) record_error(sy, kStatusNotPD, c0 + (__ffs(badm) - 1));
        if (bad) d = 1.0;
        if (v.pass == 0 && lane < nc) __stcg(v.dcar + c0 + lane, d);
    }
    invert_block(S, d);
    double *ug = v.ug + (size_t)b * 3 * kW * kW;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = tid + x * kThreads;
        __stcg(ug + e, S.U[e / kW][e & (kW - 1)]);
    }
    publish(v.uflag + b, sy.epoch);
    if (b >= 1) {
        form_g(S, ug + kW * kW);
        publish(v.gflag + b, sy.epoch);
    }
    const bool hard = is_hard(S);
    if (tid == 0) st_release_gpu(v.hflag + b, hard ? -sy.epoch : sy.epoch);
}

// G2_b, from PREP(b)'s U_b.
template <typename T>
__device__ void prep2_task(const View<T> &v, int b, PrepSmem &S)
{
    if (b < 2) return;
    (void)wait_column(v, b);
    load_above(v, b, 2, S);
    (void)__all_sync(kFull, wait_eq(v.sync, v.uflag + b, v.sync.epoch, b));
    __syncwarp();
    double *ug = v.ug + (size_t)b * 3 * kW * kW;
#pragma unroll
    for (int x = 0; x < kW * kW / kThreads; ++x) {
        const int e = threadIdx.x + x * kThreads;
        S.U[e / kW][e & (kW - 1)] = __ldcg(ug + e);
    }
    __syncthreads();
    form_g(S, ug + 2 * kW * kW);
    publish(v.g2flag + b, v.sync.epoch);
}

// ---------------------------------------------------------------- SUB

// s + e += F_{row, column} y over the eight rows of a tile a warp holds,
// column = lane.  float: y comes as pairs (hi + lo = y to 48 bits) and the
// sum is kept as s + e: products split exactly, the running sum compensated
// (two-sum), so that the far sums lose about 2^-46 relative to their terms at
// FP32 speed instead of a conversion and an FMA at the FP64 rate.
__device__ __forceinline__ void rows_dot(const double (&f)[kPer], const double *y, double &s, double &)
{
#pragma unroll
    for (int j = 0; j < kPer; j += 2) {
        const double2 u = *reinterpret_cast<const double2 *>(y + j);
        s = fma(f[j], u.x, s);
        s = fma(f[j + 1], u.y, s);
    }
}
__device__ __forceinline__ void pair_fma(float f, float hi, float lo, float &s, float &e)
{
    const float p = __fmul_rn(f, hi);
    const float d = fmaf(f, hi, -p);
    const float u = __fadd_rn(s, p);
    const float b = __fsub_rn(u, s);
    const float r = __fadd_rn(__fsub_rn(s, __fsub_rn(u, b)), __fsub_rn(p, b));
    s = u;
    e = __fadd_rn(e, __fadd_rn(fmaf(f, lo, d), r));
}
__device__ __forceinline__ void rows_dot(const float (&f)[kPer], const double *y, float &s, float &e)
{
#pragma unroll
    for (int j = 0; j < kPer; j += 2) {
        const float4 u = *reinterpret_cast<const float4 *>(y + j);  // (hi, lo) of two rows
        pair_fma(f[j], u.x, u.y, s, e);
        pair_fma(f[j + 1], u.z, u.w, s, e);
    }
}
__device__ __forceinline__ void put_y(double *y, double x, double) { *y = x; }
__device__ __forceinline__ void put_y(double *y, double x, float)
{
    const float hi = (float)x;
    *reinterpret_cast<float2 *>(y) = make_float2(hi, (float)(x - (double)hi));
}

// What is left of SUB(c, b) where block b is substituted; false if it turns
// out not to be (`kind`: an early look at hflag, which is waited for here).
// `rv` is what the far tiles left of v: the two tiles next to the block come
// off it as they are, then D^T p = rv goes one row at a time.  32 FMAs in a
// row instead of eight, and nothing taken beforehand: n = 5000 with every block
// like this, one vector 0.77 instead of 0.38 ms, 16 vectors 1.90 instead of 1.69.
template <typename T>
__device__ __noinline__ bool sub_hard(const Launch<T> &P, const View<T> &v, int c, int b, double rv, int kind, SubSmem<T> &S)
{
    const SyncArgs &sy = v.sync;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = v.n, ld = v.ld, c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const long long ep64 = (long long)sy.epoch << 32;
    long long *ptag = v.ptag + (size_t)c * v.nb * kW * 2;
    const long long t0 = global_ns();
    for (unsigned it = 1; !__all_sync(kFull, kind == sy.epoch || kind == -sy.epoch); ++it) {
        if ((it & 31u) == 0u) {
            const bool late = global_ns() - t0 > sy.timeout_ns || it > (1u << 28);
            if (__any_sync(kFull, late || aborted(sy))) {
                if (lane == 0 && late) record_error(sy, kStatusTimeout, b);
                break;
            }
        }
        kind = ld_relaxed_gpu(v.hflag + b);
    }
    // (every warp decides the same, but for one that gave up, whose way has as many barriers)
    if (!__any_sync(kFull, kind == -sy.epoch)) return false;
    // dr[i kW + j] = D_ij / D_ii above the diagonal, 1 / D_ii on it (the tiles are done with)
    double *const dr = reinterpret_cast<double *>(&S.tile[1][0][0]);
    const long long o = c0 + lane + c0 * ld;
    double d = 1.0;
    if (lane < nc && v.pass > 0) d = __ldcg(v.dcar + c0 + lane);
    else if (lane < nc && CHK_TRI(sy, o + lane * ld, n, ld)) d = (double)__ldcg(v.L + o + lane * ld);
    const double rd = rcp_refined(d);
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
        const int j = warp + x * kWarps;
        double f = lane == j ? rd : 0.0;
        if (lane < j && j < nc && CHK_TRI(sy, o + j * ld, n, ld)) f = (double)__ldcg(v.L + o + j * ld) * rd;
        dr[lane * kW + j] = f;
    }
    // this warp's rows of the two tiles
    double x = warp == 0 ? rv : 0.0;
    for (int up = 2; up >= 1; --up) {
        if (b < up) continue;
        const long long r0 = c0 - up * kW + warp * kPer + (c0 + lane) * ld;
        double f[kPer];
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj)
            f[jj] = (lane < nc && CHK_TRI(sy, r0 + jj, n, ld)) ? (double)__ldcg(v.L + r0 + jj) : 0.0;
        const double y = wait_p(sy, ptag + ((size_t)(b - up) * kW + warp * kPer + (lane & (kPer - 1))) * 2, nullptr, ep64, b);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj) x = fma(-f[jj], __shfl_sync(kFull, y, jj), x);
    }
    double(*sum)[kW] = reinterpret_cast<double(*)[kW]>(&S.tile[0][0][0]);
    sum[warp][lane] = x;
    __syncthreads();
    if (warp == 0 && !(c == 0 && b == P.skip_publish)) {
        x = (sum[0][lane] + sum[1][lane]) + (sum[2][lane] + sum[3][lane]);
#pragma unroll 4
        for (int i = 0; i < kW; ++i) {
            const double xi = __shfl_sync(kFull, x, i);
            if (lane > i) x = fma(-dr[i * kW + lane], xi, x);
        }
        x *= dr[lane * kW + lane];
        put_tagged(ptag + ((size_t)b * kW + lane) * 2, lane < nc ? x : 0.0, ep64);
    }
    return true;
}

template <typename T>
__device__ void sub_task(const Launch<T> &P, const View<T> &v, int c, int b, SubSmem<T> &S)
{
    constexpr int SD = pass::Stride<T>::value;
    constexpr int E = 16 / (int)sizeof(T);  // elements of a 16-byte chunk
    using V16 = typename pass::Vec16<T>::type;
    const SyncArgs &sy = v.sync;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = v.n, ld = v.ld;
    const long long c0 = (long long)b * kW;
    const int nc = (int)min((long long)kW, n - c0);
    const bool active = lane < nc;
    const long long ep64 = (long long)sy.epoch << 32;
    long long *ptag = v.ptag + (size_t)c * v.nb * kW * 2;
    TEAM_TRACE(c, b, 0);
    (void)wait_column(v, b);
    if (warp == 0) {
        // (read by other warps behind the first barrier)
        const long long o = c0 + lane + c * v.ldv;
        S.z[lane] = (active && CHK_RECT(sy, o, n, v.kb, v.ldv)) ? (double)v.V[o] : 0.0;
    }
    // The tiles p <= b - 3 of column block b, in groups of four (the first of
    // two, so that segments start between groups).  A warp takes eight rows
    // of every tile, so that the newest step costs it eight FMAs; the order
    // of its sums depends on nothing but the order of the factor.  A group is
    // staged one group ahead, a tile by each warp (whole columns: a warp that
    // fetched its own rows of each would touch four times the lines), and
    // its 32 values of p come in one look, a lane each.
    const int far = b - 2;  // tiles 0 .. far - 1
    // this warp's columns of G1_b and G2_b, taken before the tiles so that
    // nothing but the chain's own values is waited for behind p_{b-4}
    const double *ug = v.ug + (size_t)b * 3 * kW * kW + warp * kPer * kW + lane;
    wait_flags(sy, v.uflag, b, b, b);
    if (b >= 1) wait_flags(sy, v.gflag, b, b, b);
    if (b >= 2) wait_flags(sy, v.g2flag, b, b, b);
    int kind = ld_relaxed_gpu(v.hflag + b);
    double g1[kPer], g2[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) {
        g1[jj] = b >= 1 ? __ldcg(ug + kW * kW + jj * kW) : 0.0;
        g2[jj] = b >= 2 ? __ldcg(ug + 2 * kW * kW + jj * kW) : 0.0;
    }
    auto stage = [&](int i) {
        const int p = 4 * i - 2 + warp;
        if (p >= 0 && p < far) stage_tile(sy, S.tile[i & 1][warp], v.L, ld, (long long)p * kW, c0, n, v.vec, false, lane);
        pass::cp_commit();
    };
    // this lane's row of the four tiles' p it looks for
    const long long *const mytag = ptag + ((size_t)(lane / kPer) * kW + warp * kPer + lane % kPer) * 2;
    // What is left of v at a segment's start, for the sweep: one warp (another
    // each time) adds the warps' sums behind the next barrier, while the
    // others go on; four buffers in turn (a group holds at most two starts)
    // keep them from overwriting what it reads.
    int mid = 0, end = 0;  // the segments whose starts' sums are in S.part: within and behind the last group
    int next = 1, at = seg_start(1, v.seg);  // the next segment and where it starts
    auto keep = [&](int sg) {
        double(*part)[kW] = S.part[sg & 3];
        const double z = S.z[lane] - ((part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]));
        __stcg(v.snap + ((size_t)(sg - 1) * v.nb * kW + c0 + lane) * v.KB + c, (T)z);
        __threadfence();  // before the step's result, which the sweep's inputs follow from
    };
    stage(0);
    T s = T(0), e = T(0), sm = T(0), em = T(0);  // the sums, and as they stood behind a group's second tile
    for (int i = 0; 4 * i - 2 < far; ++i) {
        pass::cp_wait<0>();
        __syncthreads();  // group i is staged, group i - 1 is done with
        stage(i + 1);
        if (mid > 0 && warp == (i & (kWarps - 1))) keep(mid);
        if (end > 0 && warp == ((i + 2) & (kWarps - 1))) keep(end);
        const int p0 = 4 * i - 2, t1 = min(4, far - p0);
        // segments that start at the group's third tile and behind it
        mid = end = 0;
        if (at == 4 * i && at < far) mid = next++, at += v.seg;
        if (at == 4 * i + 2 && at < far) end = next++, at += v.seg;
        const bool nearby = p0 + 8 >= far;  // the last tiles are waited for without a pause
        int t = i == 0 ? 2 : 0;
        double y = 0.0;
        bool have = p0 + lane / kPer < 0 || lane / kPer >= t1;
        long long t0 = 0;
        for (unsigned it = 0;; ++it) {
            if (!have) {
                have = get_tagged(mytag + (long long)p0 * kW * 2, ep64, &y);
                if (have) put_y(&S.y[warp][lane], y, T(0));
            }
            const unsigned m = __ballot_sync(kFull, have);
            __syncwarp();
            for (; t < t1 && ((m >> (8 * t)) & 0xffu) == 0xffu; ++t) {
                T f[kPer];
                const V16 *rows = reinterpret_cast<const V16 *>(S.tile[i & 1][t] + lane * SD + warp * kPer);
#pragma unroll
                for (int ch = 0; ch < kPer / E; ++ch) {
                    const V16 x = rows[ch];
#pragma unroll
                    for (int w = 0; w < E; ++w) f[ch * E + w] = pass::vget<T>(x, w);
                }
                rows_dot(f, S.y[warp] + t * kPer, s, e);
                if (t == 1) {
                    sm = s;
                    em = e;
                }
            }
            if (t >= t1) break;
            if (!nearby) __nanosleep(100);
            if (it == 0) t0 = global_ns();
            if ((it & 31u) == 31u) {
                const bool late = global_ns() - t0 > sy.timeout_ns || it > (1u << 28);
                if (__any_sync(kFull, late || aborted(sy))) {
                    if (lane == 0 && late) record_error(sy, kStatusTimeout, b);
                    break;  // (the launch is being aborted)
                }
            }
        }
        __syncwarp();
        if (mid > 0) S.part[mid & 3][warp][lane] = (double)sm + (double)em;
        if (end > 0) S.part[end & 3][warp][lane] = (double)s + (double)e;
    }
    pass::cp_wait<0>();
    TEAM_TRACE(c, b, 1);
    // the steps before: a lane takes the tagged value of one of its warp's eight rows
    auto tag_of = [&](int up) { return ptag + ((size_t)(b - up) * kW + warp * kPer + (lane & (kPer - 1))) * 2; };
    double u[kPer];
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) u[jj] = __ldcg(ug + jj * kW);
    S.fin[warp][lane] = (double)s + (double)e;
    // (a first look at p_{b-2}, before the barrier hides its latency)
    double y2 = 0.0, y1 = 0.0;
    const bool have2 = b >= 2 && get_tagged(tag_of(2), ep64, &y2);
    __syncthreads();
    const double rv = S.z[lane] - ((S.fin[0][lane] + S.fin[1][lane]) + (S.fin[2][lane] + S.fin[3][lane]));
    double pz = 0.0;
#pragma unroll
    for (int jj = 0; jj < kPer; ++jj) pz = fma(u[jj], __shfl_sync(kFull, rv, warp * kPer + jj), pz);
    TEAM_TRACE(c, b, 2);
    // U^T (what is left) - G2 p_{b-2} - G1 p_{b-1}: this warp's share of each
    const bool have1 = b >= 1 && get_tagged(tag_of(1), ep64, &y1);
    // (the fences pass while the warps would wait for p_{b-1})
    if (mid > 0 && warp == 1) keep(mid);
    if (end > 0 && warp == 2) keep(end);
    if (at == b - 2 && warp == kWarps - 1) {
        // what is left at the start of the column's last segment, row block b - 2
        __stcg(v.snap + ((size_t)(next - 1) * v.nb * kW + c0 + lane) * v.KB + c, (T)rv);
        __threadfence();
    }
    if (!__all_sync(kFull, kind == sy.epoch) && sub_hard(P, v, c, b, rv, kind, S)) return;
    if (b >= 2) {
        if (!__all_sync(kFull, have2)) y2 = wait_p(sy, tag_of(2), nullptr, ep64, b);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj) pz = fma(-g2[jj], __shfl_sync(kFull, y2, jj), pz);
    }
    if (b >= 1) {
        if (!__all_sync(kFull, have1)) y1 = wait_p(sy, tag_of(1), nullptr, ep64, b);
        TEAM_TRACE(c, b, 3);
#pragma unroll
        for (int jj = 0; jj < kPer; ++jj) pz = fma(-g1[jj], __shfl_sync(kFull, y1, jj), pz);
    }
    double(*sum)[kW] = reinterpret_cast<double(*)[kW]>(&S.tile[0][0][0]);  // (the tiles are done with)
    sum[warp][lane] = pz;
    __syncthreads();
    if (warp == 0 && !(c == 0 && b == P.skip_publish)) {
        const double x = (sum[0][lane] + sum[1][lane]) + (sum[2][lane] + sum[3][lane]);
        put_tagged(ptag + ((size_t)b * kW + lane) * 2, active ? x : 0.0, ep64);
    }
    TEAM_TRACE(c, b, 4);
}

// ---------------------------------------------------------------- COEF

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }  // j <= i

// Bounded wait of one thread for a tagged double; 0 if it gave up.  `next`:
// the Grams' chain, polled without a pause first.
__device__ __forceinline__ double wait_one(const SyncArgs &sy, const long long *w2, long long ep64, long long who, bool next)
{
    double x = 0.0;
    for (int it = 0; next && it < 32; ++it)
        if (get_tagged(w2, ep64, &x)) return x;
    if (!bounded_wait(sy, [&] { return get_tagged(w2, ep64, &x); }, [] {}, who, 128)) x = 0.0;
    return x;
}

// Signs and comparisons on the integer pipe: an FP64 instruction takes its own
// for 64 cycles.
__device__ __forceinline__ double signed_by(double x, unsigned down) { return __hiloint2double(__double2hiint(x) ^ (int)(down << 31), __double2loint(x)); }
__device__ __forceinline__ bool positive_finite(double x)
{
    const long long u = __double_as_longlong(x);
    return u > 0 && u < 0x7ff0000000000000ll;
}

// A Gram is ill-conditioned if a pivot |D_q| is below this fraction of the
// sums that it is left of, 1 + sum_i p_iq^2: subtracting costs the pivot that
// factor in relative accuracy, so that three bits may go in double; in float,
// whose coefficients are rounded to 24 bits, twenty of the Gram's 53.
// Compared by the numbers' high words; a NaN is not found here, but as a row
// that has failed.
template <typename T>
__device__ __forceinline__ bool ill_pivot(double ad, double size)
{
    constexpr int bits = sizeof(T) == 8 ? 3 : 20;
    return __double2hiint(ad) < __double2hiint(size) - (bits << 20);
}

// The factor of an ill-conditioned Gram is not taken from the Gram, whose small
// pivots are rounding errors (a factor 1e-4 I and eight vectors of size 1: the
// result off by 1e-8).  A block whose first Gram is ill-conditioned starts
// from the factor L0 D0 L0^T that the block before hands on, and sums the
// Grams of L0^{-1} p on top of D0: only what these rows add counts there, so
// that vectors which are large and alike all the way cost a chain of 2 to 9 us
// a block (n = 5000, 2 / 8 vectors 0.79 / 1.94 ms instead of 0.44 / 0.95).
// Where rows are still ill-conditioned (the first ones of an estimator that
// starts from a small multiple of the identity) the factor is carried from row
// to row, L D L^T + p p^T:
//   z = L^{-1} p,  D~_q = D_q Dc_q / Dc_{q-1},  L~_iq = L_iq + sigma_q b_q w_iq,
// w_iq what is left of p_i behind z_q.  These are the rotations that the sweep
// applies, with the coefficients that it applies, so that the factor and the
// carries stay consistent, as they do where vector after vector is rotated
// (and as they do not with a Gram of more bits).  A serial chain of up to 40 FP64
// instructions and two dozen shuffles a row, 2.9 us with eight vectors.
// Lane i (one of eight; the others repeat them) holds row i.
struct Carried {
    double l[kTeamKb], ad;  // L_iq, |D_i|
};
__device__ __forceinline__ Carried carried_at(const CoefSmem &S, int row, int kb, unsigned down_mask)
{
    const int i = threadIdx.x & (kTeamKb - 1);
    Carried c;
    c.ad = 1.0;
#pragma unroll
    for (int q = 0; q < kTeamKb; ++q) c.l[q] = (i < kb && q < i) ? S.H[row][tri(i, q)] : 0.0;
    if (i < kb) c.ad = signed_by(S.H[row][tri(i, i)], (down_mask >> i) & 1u);
    return c;
}
// `c` is row `row`'s factor: its z and the terms of its Dc to S, and (`store`) itself; then the next row's.
__device__ __forceinline__ void carry_row(CoefSmem &S, Carried &c, int row, int kb, unsigned down_mask, bool store)
{
    const int lane = threadIdx.x & 31, i = lane & (kTeamKb - 1);
    const unsigned down = (down_mask >> i) & 1u;
    double w = i < kb ? S.p0[row][i] : 0.0, wq[kTeamKb];
#pragma unroll
    for (int q = 0; q < kTeamKb; ++q) {
        if (q < kb) {
            const double zq = __shfl_sync(kFull, w, q);
            if (q < i) w = fma(-zq, c.l[q], w);
        }
        wq[q] = w;
    }
    const double term = signed_by(w * w, down) * rcp_refined(c.ad);
    double Dc = 1.0, before = 1.0;
#pragma unroll
    for (int q = 0; q < kTeamKb; ++q) {
        if (q < kb) {
            const double t = __shfl_sync(kFull, term, q);
            if (q == i) before = Dc;
            if (q <= i) Dc += t;
        }
    }
    if (store && lane < kb) {
#pragma unroll
        for (int q = 0; q < kTeamKb; ++q)
            if (q < i) S.H[row][tri(i, q)] = c.l[q];
        S.H[row][tri(i, i)] = signed_by(c.ad, down);
        S.p[row][i] = w;
        S.z[row][i] = term;
    }
    const double b = signed_by(w * rcp_refined(c.ad * Dc), down);
#pragma unroll
    for (int q = 0; q < kTeamKb; ++q) {
        if (q < kb) {
            const double bq = __shfl_sync(kFull, b, q);
            if (q < i) c.l[q] = fma(bq, wq[q], c.l[q]);
        }
    }
    c.ad = c.ad * Dc * rcp_refined(before);
}

// One warp: rows first .. last are carried from row first's Gram on.
__device__ __noinline__ void carry_rows(CoefSmem &S, int first, int last, int kb, unsigned down_mask)
{
    Carried c = carried_at(S, first, kb, down_mask);
    __syncwarp();
    for (int m = first; m <= last; ++m) carry_row(S, c, m, kb, down_mask, true);
}
// One warp: S.M becomes the factor behind the block, one row on from the last.
__device__ __noinline__ void carry_end(CoefSmem &S, int kb, unsigned down_mask)
{
    const int lane = threadIdx.x & 31;
    Carried c = carried_at(S, kW - 1, kb, down_mask);
    carry_row(S, c, kW - 1, kb, down_mask, false);
    if (lane < kb) {
#pragma unroll
        for (int q = 0; q < kTeamKb; ++q)
            if (q < lane) S.M[tri(lane, q)] = c.l[q];
        S.M[tri(lane, lane)] = c.ad;
    }
    __syncwarp();
}
// One warp: S.M, the Gram behind the block on top of D0, becomes its factor;
// false if that is ill-conditioned.  Lane i (one of eight) holds row i.
template <typename T>
__device__ __noinline__ bool factor_end(CoefSmem &S, int kb, unsigned down_mask)
{
    const int lane = threadIdx.x & 31, i = lane & (kTeamKb - 1);
    const unsigned down = (down_mask >> i) & 1u;
    double a[kTeamKb];
#pragma unroll
    for (int m = 0; m < kTeamKb; ++m) a[m] = (i < kb && m <= i) ? S.M[tri(i, m)] : 0.0;
    const double size = i < kb ? S.M[tri(i, i)] + (down ? 2.0 * S.l0[tri(i, i)] : 0.0) : 0.0;
    double ad = 1.0;
#pragma unroll
    for (int j = 0; j < kTeamKb; ++j) {
        if (j >= kb) continue;
        if (i == j) ad = signed_by(a[j], down);
        const double l = a[j] * rcp_refined(__shfl_sync(kFull, a[j], j));
#pragma unroll
        for (int m = j + 1; m < kTeamKb; ++m) {
            if (m >= kb) continue;
            const double x = __shfl_sync(kFull, a[j], m);
            if (m <= i) a[m] = fma(-l, x, a[m]);
        }
        if (i > j) a[j] = l;
    }
    const bool ok = __all_sync(kFull, i >= kb || !ill_pivot<T>(ad, size)) != 0;
    if (lane < kb) {
#pragma unroll
        for (int m = 0; m < kTeamKb; ++m)
            if (m < i) S.M[tri(i, m)] = a[m];
        S.M[tri(i, i)] = ad;
    }
    __syncwarp();
    return ok;
}
// One warp: the factor L0 M (`handed`) or M to the next block.
__device__ __noinline__ void put_factor(const CoefSmem &S, long long *w, int kb, int ne, bool handed, long long ep64)
{
    for (int e = threadIdx.x & 31; e < ne; e += 32) {
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        const int j = e - i * (i + 1) / 2;
        double f = i < kb ? S.M[e] : 0.0;
        if (handed && j < i && i < kb) {
            f += S.l0[e];
            for (int m = j + 1; m < i; ++m) f = fma(S.l0[tri(i, m)], S.M[tri(m, j)], f);
        }
        put_tagged(w + 2 * e, f, ep64);
    }
}

// Row r of the block: H_r = H_b + sum_{i<r} p_i p_i^T = L D L^T, z = L^{-1} p_r and,
// with |D_q| = sigma_q D_q,
//   Dc_q = 1 + sum_{q'<=q} sigma_q' z_q'^2 / |D_q'|,  a_q = sigma_q z_q,
//   b_q = z_q / (|D_q| Dc_q),  e = Dc_kb^{-1/2},  the diagonal factor Dc_kb^{1/2}.
// The Grams of the blocks form a chain (H_{b+1} = H_b + the block's Gram)
// that is handed on before the factors are formed; where H_{b+1} is
// ill-conditioned, its factor is handed on too (see Carried).  Four lanes share a row:
// its factor's rows are dealt to them, so that a block of eight vectors
// takes about 60 FP64 instructions a warp and step group instead of 250.
template <typename T>
__device__ void coef_task(const Launch<T> &P, const View<T> &v, int b, CoefSmem &S)
{
    const SyncArgs &sy = v.sync;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long ep64 = (long long)sy.epoch << 32;
    const int kb = v.kb, KB = v.KB, ne = KB * (KB + 1) / 2;
    const long long r0 = (long long)b * kW;
    const int rows = (int)min((long long)kW, v.n - r0);
    for (int x = threadIdx.x; x < kW * kb; x += kThreads) {
        const int q = x / kW, i = x & (kW - 1);
        const double p = wait_one(sy, v.ptag + (((size_t)q * v.nb + b) * kW + i) * 2, ep64, b, false);
        S.p[i][q] = p;
        S.p0[i][q] = p;
    }
    __syncthreads();
    TEAM_TRACE(0, b, 5);
    // rows threadIdx.x / 4; the four lanes of a row take the factor's rows i = sub, sub + 4, ...;
    // row kb of the elimination is p itself, which becomes z
    const int row = threadIdx.x >> 2, sub = threadIdx.x & 3;
    double *h = S.H[row], *t = S.p[row];
    // entry x of the packed triangle: each of `ng` threads sums its share of the rows
    const int ng = KB <= 4 ? 8 : 2, nr = kW / ng;
    const int x = threadIdx.x % ne, part = threadIdx.x / ne, i0 = part * nr;
    const bool mine = part < ng;
    int q = 0;
    while ((q + 1) * (q + 2) / 2 <= x) ++q;
    const int r = x - q * (q + 1) / 2;
    const bool in = mine && q < kb;
    enum { kHanded, kTakeGram, kFailed };
    int from = kHanded;
    bool handed = false;  // the block starts from a factor handed on, S.l0
    bool early = false;   // (last warp) the next block has its factor
    for (;;) {
        // the prefix Grams: each thread's share, then what comes before it
        double acc = 0.0;
        if (mine) {
#pragma unroll 4
            for (int i = i0; i < i0 + nr; ++i) {
                S.H[i][x] = acc;
                if (in) acc = fma(S.p[i][q], S.p[i][r], acc);
            }
            S.g[part][x] = acc;
        }
        __syncthreads();
        if (mine) {
            double before = 0.0, all = 0.0;
            for (int m = 0; m < ng; ++m) {
                if (m == part) before = all;
                all += S.g[m][x];
            }
            const bool down = (v.down_mask >> q) & 1u;
            double h = (q == r) ? (down ? -1.0 : 1.0) : 0.0;
            if (handed) {
                if (in) h *= S.l0[x];
                if (part == 0) S.M[x] = h + all;
            } else {
                if (b > 0 && in) h = wait_one(sy, v.htag + ((size_t)(b - 1) * ne + x) * 2, ep64, b, true);
                if (in && part == 0 && b + 1 < v.nb) put_tagged(v.htag + ((size_t)b * ne + x) * 2, h + all, ep64);
                if (in && part == 0 && q == r) S.size[q] = h + all + (down ? 2.0 : 0.0);
            }
            h += before;
#pragma unroll 4
            for (int i = i0; i < i0 + nr; ++i) S.H[i][x] += h;
        }
        __syncthreads();
        // where the blocks' factors form a chain, the next block's goes first
        if (handed && warp == kWarps - 1 && b + 1 < v.nb && factor_end<T>(S, kb, v.down_mask)) {
            put_factor(S, v.ftag + (size_t)b * ne * 2, kb, ne, true, ep64);
            early = true;
        }
        // the sizes of the diagonal's sums (the elimination's pivots q are this lane's own rows)
        double size[kTeamKb / 4];
#pragma unroll
        for (int u = 0; u < kTeamKb / 4; ++u) {
            const int q = sub + 4 * u;
            size[u] = 0.0;
            if (q < kb) size[u] = h[tri(q, q)] + ((v.down_mask >> q) & 1u ? 2.0 * (handed ? S.l0[tri(q, q)] : 1.0) : 0.0);
        }
        for (int j = 0; j < kb; ++j) {
            const double id = rcp_refined(h[tri(j, j)]);
            for (int i = sub; i <= kb; i += 4) {
                if (i <= j) continue;
                const double lij = (i == kb ? t[j] : h[tri(i, j)]) * id;
                if (i == kb) {
                    for (int m = j + 1; m < kb; ++m) t[m] = fma(-lij, h[tri(m, j)], t[m]);
                } else {
                    for (int m = j + 1; m <= i; ++m) h[tri(i, m)] = fma(-lij, h[tri(m, j)], h[tri(i, m)]);
                }
            }
            __syncwarp();
            for (int i = sub; i < kb; i += 4)
                if (i > j) h[tri(i, j)] *= id;
            __syncwarp();
        }
        // the terms of Dc, and which rows' Grams are ill-conditioned
        bool ill = false;
#pragma unroll
        for (int u = 0; u < kTeamKb / 4; ++u) {
            const int q = sub + 4 * u;
            if (q >= kb) continue;
            const unsigned down = (v.down_mask >> q) & 1u;
            const double ad = signed_by(h[tri(q, q)], down);
            ill = ill || ill_pivot<T>(ad, size[u]);
            S.z[row][q] = signed_by(t[q] * t[q], down) * rcp_refined(ad);
        }
        const unsigned illm = __ballot_sync(kFull, ill && row < rows);
        if (lane == 0) S.ill[warp] = illm;
        __syncthreads();
        if (handed || b == 0 || (S.ill[0] & 0xfu) == 0u) break;
        if (warp == 0) {
            // NaN: a row of the block before has failed, the rest is unspecified;
            // infinity: it found its last pivots just large enough, so take the Gram
            bool nan = false, inf = false;
            for (int e = lane; e < ne; e += 32) {
                const double f = wait_one(sy, v.ftag + ((size_t)(b - 1) * ne + e) * 2, ep64, b, true);
                S.l0[e] = f;
                nan = nan || f != f;
                inf = inf || fabs(f) > DBL_MAX;
            }
            nan = __any_sync(kFull, nan);
            inf = __any_sync(kFull, inf);
            if (lane == 0) S.have = nan ? kFailed : inf ? kTakeGram : kHanded;
        }
        __syncthreads();
        from = S.have;
        if (from != kHanded) break;
        // p becomes L0^{-1} p
        double *y = S.p0[row];
        for (int j = 0; j + 1 < kb; ++j) {
            for (int i = sub; i < kb; i += 4)
                if (i > j) y[i] = fma(-S.l0[tri(i, j)], y[j], y[i]);
            __syncwarp();
        }
        for (int i = sub; i < kb; i += 4) t[i] = y[i];
        handed = true;
        __syncthreads();
    }
    int first = kW, last = -1;
#pragma unroll
    for (int m = kWarps - 1; m >= 0; --m) {
        const unsigned rowm = S.ill[m] & (m == 0 && from == kTakeGram ? ~0xfu : ~0u);
        if (!rowm) continue;
        first = m * 8 + ((__ffs(rowm) - 1) >> 2);
        last = max(last, m * 8 + ((31 - __clz(rowm)) >> 2));
    }
    if (first > 0 && last >= 0) {
        // (row 0 is ill-conditioned only behind a row that has failed)
        if (warp == 0) carry_rows(S, first - 1, last, kb, v.down_mask);
        __syncthreads();
    }
    // the prefix sums and the coefficients
    bool bad = false, next = false;
    const int start = seg_at(b, v.seg);
    double Dc = 1.0;
    T *cf = v.coef + (size_t)(r0 + row) * 2 * KB;
    for (int q = 0; q < KB; ++q) {
        const double before = Dc;
        if (q < kb) {
            Dc += S.z[row][q];
            bad = bad || !positive_finite(Dc);
        }
        if ((q & 3) != sub || row >= rows) continue;
        if (q < kb) {
            const unsigned down = (v.down_mask >> q) & 1u;
            const double ad = signed_by(h[tri(q, q)], down);
            bad = bad || !positive_finite(ad);
            cf[2 * q] = (T)signed_by(t[q], down);
            cf[2 * q + 1] = (T)(t[q] * rcp_refined(ad * Dc));
            next = next || (row == kW - 1 && ill_pivot<T>(ad * Dc, S.size[q] * before));
            if (row == 0 && start > 0 && start <= v.nbound) {
                // a segment starts at this block: the factor of H_b for its carries
                double *dst = v.rst + (size_t)(start - 1) * ne;
                for (int m = 0; m < q; ++m) __stcg(dst + tri(q, m), handed ? S.l0[tri(q, m)] : h[tri(q, m)]);
                __stcg(dst + tri(q, q), rcp_refined(ad));
            }
        } else {
            cf[2 * q] = T(0);
            cf[2 * q + 1] = T(0);
        }
    }
    if (sub == 0 && row < rows) {
        const double rD = rsqrt_refined(Dc);
        v.escale[r0 + row] = (T)rD;
        v.dfac[r0 + row] = Dc * rD;
    }
    const unsigned badm = __ballot_sync(kFull, bad && row < rows);
    if (badm && lane == 0) record_error(sy, kStatusNotPD, r0 + ((threadIdx.x + __ffs(badm) - 1) >> 2));
    __threadfence();
    const bool failed = __syncthreads_or(badm != 0u) != 0;
    if (threadIdx.x == 0) st_release_gpu(v.cflag + b, sy.epoch);
    TEAM_TRACE(0, b, 6);
    if (warp == kWarps - 1 && b + 1 < v.nb && !early) {
        // the next block's factor, if its Gram is ill-conditioned, else
        // infinity, or NaN where a row has failed
        long long *w = v.ftag + (size_t)b * ne * 2;
        if (!failed && __any_sync(kFull, next)) {
            carry_end(S, kb, v.down_mask);
            put_factor(S, w, kb, ne, handed, ep64);
        } else {
            const double none = __longlong_as_double(failed ? 0x7ff8000000000000ll : 0x7ff0000000000000ll);
            for (int e = lane; e < ne; e += 32) put_tagged(w + 2 * e, none, ep64);
        }
    }
}

// ---------------------------------------------------------------- SWEEP

// The warps that share a segment.
template <int NV>
__device__ __forceinline__ void unit_sync(int unit)
{
    static_assert(NV == 1 || NV == 2 || NV == kWarps, "warps of a segment");
    if (NV == 1) __syncwarp();
    else if (NV == kWarps) __syncthreads();
    else if (unit == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
    else asm volatile("bar.sync 2, 64;" ::: "memory");
}

// Segments sg0 .. sg0 + UNITS - 1 of column block j.  NV warps share a
// segment, VW of its KB vectors each: a tile passes from warp to warp in
// shared memory, each applying its vectors' rotations (lane = column, the
// carries in registers), so that NV tiles are in work at once and a tile's
// step takes the time of VW vectors, not of KB (in double 64 cycles per FMA
// and warp: 4 us instead of 16 with eight vectors).  The order of the
// operations on an element is that of one warp doing all vectors.  For one
// vector in double and a short column a second warp scales and stores what
// the first has rotated (a tile 4.0 instead of 6.3 us).  Tiles and coefficients are staged one step ahead.  The warps'
// places are turned from task to task, so that the last place, which also
// scales and stores the tile, falls on each of the SM's four FP64 pipes in
// turn.  A wait that runs out leaves the task running on whatever it has
// (the launch is being aborted), so that the warps' barriers stay matched.
template <typename T, int VW, int NV, int KB>
__device__ void sweep_task(const Launch<T> &P, const View<T> &v, int j, int task, SweepSmem<T, KB, NV> &S)
{
    using SS = SweepSmem<T, KB, NV>;
    constexpr int NR = KB / VW;  // places that rotate; with NR < NV the last one only scales and stores
    static_assert(KB % VW == 0 && (NR == NV || NR == NV - 1), "places of a segment");
    using V16 = typename pass::Vec16<T>::type;
    constexpr int NS = SS::NS;
    constexpr int SD = pass::Stride<T>::value;
    constexpr int E = 16 / (int)sizeof(T);
    constexpr int CPC = kW / E;  // 16-byte chunks per column segment
    const SyncArgs &sy = v.sync;
    const int lane = threadIdx.x & 31;
    const int place = ((threadIdx.x >> 5) + j + task) & (kWarps - 1);
    const int unit = place / NV, part = place % NV;
    const int sg = task * SS::UNITS + unit, nseg = segs_of(j, v.seg);
    if (NV < kWarps && sg >= nseg) return;  // (whole segments' warps; they share no barrier with the others)
    typename SS::Unit &U = S.unit[unit];
    const long long n = v.n, ld = v.ld;
    const bool last = sg == nseg - 1;
    const int rb = seg_start(sg, v.seg);
    const int re = last ? j : seg_start(sg + 1, v.seg) - 1;
    const long long c0 = (long long)j * kW;
    const bool active = c0 + lane < n;
    // the coefficients of the segment's rows, and of row block j: column j's
    // substitution steps were the last readers of its tiles as they entered
    wait_flags(sy, v.cflag, rb, re, j);
    if (!last) wait_flags(sy, v.cflag, j, j, j);
    // the diagonal's row block: the diagonal as it enters the pass, its
    // factors, and what the 16-byte chunk with the diagonal holds above it
    double dc = 0.0, df = 0.0;
    T dch[E];
#pragma unroll
    for (int w = 0; w < E; ++w) dch[w] = T(0);
    if (last && active) {
        if (part == NV - 1) {
            dc = __ldcg(v.dcar + c0 + lane);
            df = __ldcg(v.dfac + c0 + lane);
        }
        if (part == 0) {
            const long long o = c0 + (lane & ~(E - 1)) + (c0 + lane) * ld;
#pragma unroll
            for (int w = 0; w < E; ++w)
                if (w < (lane & (E - 1)) && CHK_TRI(sy, o + w, n, ld)) dch[w] = __ldcg(v.L + o + w);
        }
    }
    // 16-byte chunk `ch` of the columns cc0, cc0 + cstep, ... is this lane's to copy
    constexpr int cstep = NV * 32 / CPC;
    const int ch = lane % CPC, cc0 = part * (32 / CPC) + lane / CPC;
    const int ncol = (int)min((long long)kW, n - c0);
    const T *const lcol = v.L + ch * E + (c0 + cc0) * ld;
    auto stage = [&](int t) {  // tile and coefficients of row block rb + t
        const int r = rb + t, slot = t % NS;
        const long long r0 = (long long)r * kW;
        T *tl = U.tile[slot];
        if (v.vec) {
            // this lane's chunk of every cstep-th column (of the diagonal tile
            // the chunks above the diagonal's)
            const int first = r == j ? (ch + 1) * E : 0;
            const T *src = lcol + r0;
            T *d = tl + cc0 * SD + ch * E;
#pragma unroll
            for (int cc = cc0; cc < kW; cc += cstep, src += cstep * ld, d += cstep * SD) {
                if (cc < first) continue;
                if (cc < ncol && CHK_TRI(sy, src - v.L, n, ld) && CHK_TRI(sy, src - v.L + E - 1, n, ld)) {
                    pass::cp16(d, src);
                } else {
#pragma unroll
                    for (int w = 0; w < E; ++w) d[w] = T(0);
                }
            }
        } else {
            stage_columns<8>(sy, tl, v.L, ld, r0, c0, n, r == j, lane, part * (kW / NV), (part + 1) * (kW / NV));
        }
        const T *cf = v.coef + (size_t)r0 * 2 * KB;
        for (int x = part * 32 + lane; x < kW * 2 * KB / E; x += NV * 32) pass::cp16(U.cf[slot] + x * E, cf + x * E);
        if (part == NV - 1 && lane < kW / E) pass::cp16(U.e[slot] + lane * E, v.escale + r0 + lane * E);
    };
    stage(0);
    pass::cp_commit();
    T uh[VW];
#pragma unroll
    for (int w = 0; w < VW; ++w) uh[w] = T(0);
    if (NR < NV && part >= NR) {
        // (this place rotates nothing)
    } else if (sg == 0) {
#pragma unroll
        for (int w = 0; w < VW; ++w) {
            const int q = part * VW + w;
            const long long o = c0 + lane + q * v.ldv;
            uh[w] = (active && q < v.kb && CHK_RECT(sy, o, n, v.kb, v.ldv)) ? v.V[o] : T(0);
        }
    } else {
        // the carry entering row block rb is |D|^{-1} L^{-1} w of the residual w kept there
        const T *w = v.snap + ((size_t)(sg - 1) * v.nb * kW + c0 + lane) * KB;
        const double *h = v.rst + (size_t)(sg - 1) * (KB * (KB + 1) / 2);
        double z[KB];
#pragma unroll
        for (int q = 0; q < KB; ++q) z[q] = (active && q < v.kb && q < (part + 1) * VW) ? (double)__ldcg(w + q) : 0.0;
#pragma unroll
        for (int q = 1; q < KB; ++q) {
            if (q < v.kb && q < (part + 1) * VW) {
#pragma unroll
                for (int m = 0; m < q; ++m) z[q] = fma(-__ldcg(h + tri(q, m)), z[m], z[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < KB; ++q)
            if (q / VW == part) uh[q % VW] = q < v.kb ? (T)(z[q] * __ldcg(h + tri(q, q))) : T(0);
    }
    const int ntile = re - rb + 1;
    for (int i = 0; i < ntile + NV - 1; ++i) {
        if (i + 1 < ntile) stage(i + 1);
        pass::cp_commit();
        pass::cp_wait<1>();
        unit_sync<NV>(unit);
        const int t = i - part, r = rb + t;
        if (t >= 0 && t < ntile) {
            const bool diag = r == j;
            const int slot = t % NS;
            T *tl = U.tile[slot];
            V16 *colv = reinterpret_cast<V16 *>(tl + lane * SD);
            const T *cf = U.cf[slot] + 2 * VW * part;
            T *mycol = tl + lane * SD;
            if (diag && part == 0 && v.vec) {
                const int i0 = lane & ~(E - 1);
#pragma unroll
                for (int w = 0; w < E; ++w) mycol[i0 + w] = dch[w];
            }
            if (NR == NV || part < NR) {
                T x[kW];
#pragma unroll
                for (int k = 0; k < CPC; ++k) {
                    const V16 y = colv[k];
#pragma unroll
                    for (int w = 0; w < E; ++w) x[k * E + w] = pass::vget<T>(y, w);
                }
                // (a lane past the order, and a row at or below the diagonal, keeps what it has)
                const int rows = !active ? 0 : diag ? lane : kW;
#pragma unroll
                for (int k = 0; k < kW; ++k) {
                    T a[VW], b[VW];
#pragma unroll
                    for (int w = 0; w < VW; ++w) {
                        a[w] = cf[k * 2 * KB + 2 * w];
                        b[w] = cf[k * 2 * KB + 2 * w + 1];
                    }
                    if (k < rows) {
#pragma unroll
                        for (int w = 0; w < VW; ++w) {
                            x[k] = fma(a[w], uh[w], x[k]);
                            uh[w] = fma(-b[w], x[k], uh[w]);
                        }
                    }
                }
                if (NR == NV && part == NV - 1) {
#pragma unroll
                    for (int k = 0; k < kW; ++k)
                        if (k < rows) x[k] *= U.e[slot][k];
                }
#pragma unroll
                for (int k = 0; k < CPC; ++k) {
                    V16 y;
                    T *yp = reinterpret_cast<T *>(&y);
#pragma unroll
                    for (int w = 0; w < E; ++w) yp[w] = x[k * E + w];
                    colv[k] = y;
                }
            }
            if (diag && part == NV - 1) mycol[lane] = (T)(dc * df);
            if (part == NV - 1) {
                const long long r0 = (long long)r * kW;
                if (diag && active) __stcg(v.dcar + c0 + lane, dc * df);
                __syncwarp();
                constexpr bool scale = NR < NV;  // the rows' scales are still to be applied
                const T *er = U.e[slot];
                if (v.vec) {
                    // whole chunks above the diagonal, then, one column a lane, the
                    // diagonal's chunk
                    const int first = diag ? (ch + 1) * E : 0;
                    constexpr int step = 32 / CPC;
                    const int k0 = lane / CPC;
                    T *g = v.L + r0 + ch * E + (c0 + k0) * ld;
                    const T *d = tl + k0 * SD + ch * E;
#pragma unroll
                    for (int cc = k0; cc < kW; cc += step, g += step * ld, d += step * SD)
                        if (cc >= first && cc < ncol && CHK_TRI(sy, g - v.L, n, ld) && CHK_TRI(sy, g - v.L + E - 1, n, ld)) {
                            V16 y = *reinterpret_cast<const V16 *>(d);
                            if (scale) {
                                T *yp = reinterpret_cast<T *>(&y);
#pragma unroll
                                for (int w = 0; w < E; ++w) yp[w] *= er[ch * E + w];
                            }
                            __stcg(reinterpret_cast<V16 *>(g), y);
                        }
                    const int i0 = lane & ~(E - 1);
                    if (diag && active) {
#pragma unroll
                        for (int w = 0; w < E; ++w)
                            if (i0 + w <= lane && CHK_TRI(sy, r0 + i0 + w + (c0 + lane) * ld, n, ld))
                                __stcg(v.L + r0 + i0 + w + (c0 + lane) * ld,
                                       tl[lane * SD + i0 + w] * (scale && i0 + w < lane ? er[i0 + w] : T(1)));
                    }
                }
            }
        }
        unit_sync<NV>(unit);  // the next step's copies may take the slot of the tile that left
        const int left = i - (NV - 1);
        if (!v.vec && left >= 0) {
            // (or, where columns do not start on 16 bytes, the segment's warps
            // store it first, each its share, as they fetched it: one warp for
            // either kept the others waiting, n = 6001 with 64 vectors 10.3 ms
            // instead of 9.05, n = 511 1.20 instead of 1.03)
            const int r = rb + left, slot = left % NS;
            const bool diag = r == j;
            const long long r0 = (long long)r * kW;
            const T *tl = U.tile[slot], e = NR < NV ? U.e[slot][lane] : T(1);
#pragma unroll
            for (int x = 0; x < kW / NV; ++x) {
                const int cc = part * (kW / NV) + x;
                if (c0 + cc < n && (!diag || lane <= cc) && CHK_TRI(sy, (r0 + lane) + (c0 + cc) * ld, n, ld))
                    __stcg(v.L + (r0 + lane) + (c0 + cc) * ld, tl[cc * SD + lane] * (diag && lane == cc ? T(1) : e));
            }
            unit_sync<NV>(unit);
        }
    }
    pass::cp_wait<0>();
    if (P.trace && last && part == 0 && lane == 0)
        P.trace[((size_t)v.pass * kTeamKb * v.nb + j) * kTracePoints + 7] = global_ns();
    if (v.pass + 1 < v.npass) {
        // count the segment done for the problem's next pass; a count left by
        // an earlier launch is first lifted to (epoch << 32)
        __threadfence();
        unit_sync<NV>(unit);
        if (part == 0 && lane == 0) {
            unsigned long long *d = reinterpret_cast<unsigned long long *>(v.sdone + j);
            atomicMax(d, (unsigned long long)sy.epoch << 32);
            __threadfence();
            atomicAdd(d, 1ull);
        }
    }
}

// ---------------------------------------------------------------- entry

template <typename T>
__device__ __forceinline__ const Prob &prob_of(const Launch<T> &P, int i)
{
    return P.probs ? P.probs[i] : P.prob0;
}
template <typename T>
__device__ __forceinline__ unsigned long long *ticket_of(const Launch<T> &P, int i)
{
    const Prob &pr = prob_of(P, i);
    return reinterpret_cast<unsigned long long *>(pr.progress + prob_ticket(pr.nb, pr.k));
}

// Fill the view of pass s of problem i; false if a region fails its bounds check.
template <typename T>
__device__ bool set_view(const Launch<T> &P, int i, int s, int epoch, View<T> &v)
{
    const Prob &pr = prob_of(P, i);
    const int nb = pr.nb, kb = min(kTeamKb, pr.k - s * kTeamKb), KB = kb_inst(kb);
    const PassRec rc = pass_rec(nb, kb);
    char *d = pr.data + pass_data_off(nb, s);
    v.L = static_cast<T *>(pr.L);
    v.ldv = pr.ldv;
    v.V = static_cast<const T *>(pr.V) + (long long)s * kTeamKb * pr.ldv;
    v.n = pr.n;
    v.ld = pr.ld;
    v.nb = nb;
    v.pass = s;
    v.npass = passes_of(pr.k);
    v.units = units_of(nb, KB, sizeof(T) == 8);
    v.kb = kb;
    v.KB = KB;
    v.seg = seg_of(nb, KB, sizeof(T) == 8);
    v.nbound = bounds_of(nb, KB, sizeof(T) == 8);
    v.look = look_of(kb);
    v.down_mask = (unsigned)(pr.down_mask >> (s * kTeamKb)) & ((1u << kb) - 1u);
    v.vec = ((pr.ld * (long long)sizeof(T)) & 15) == 0 && (reinterpret_cast<uintptr_t>(pr.L) & 15) == 0;
    v.ug = reinterpret_cast<double *>(d + rc.ug);
    v.coef = reinterpret_cast<T *>(d + rc.coef);
    v.escale = reinterpret_cast<T *>(d + rc.escale);
    v.dfac = reinterpret_cast<double *>(d + rc.dfac);
    v.snap = reinterpret_cast<T *>(d + rc.snap);
    v.rst = reinterpret_cast<double *>(d + rc.rst);
    v.dcar = reinterpret_cast<double *>(pr.data + prob_dcar(nb, pr.k));
    v.ptag = pr.progress + pass_tag_off(nb, s);
    v.htag = v.ptag + (size_t)kb * nb * kW * 2;
    v.ftag = v.htag + (size_t)nb * KB * (KB + 1);
    v.uflag = pr.iflags + (size_t)s * kPassFlags * nb;
    v.gflag = v.uflag + nb;
    v.g2flag = v.gflag + nb;
    v.cflag = v.g2flag + nb;
    v.hflag = v.cflag + nb;
    v.sdone = pr.progress + prob_ticket(nb, pr.k) + 1;
    v.sync.abort_flag = P.ctl + kCtlAbort;
    v.sync.status = P.status;
    v.sync.user_info = pr.info;
    v.sync.epoch = epoch;
    v.sync.timeout_ns = P.timeout_ns;
    v.sync.chk_cut = P.chk_cut;
#ifdef CHM_CHECK
    return CHK_REGION(v.sync, pr.data, prob_data(nb, pr.k), P.ws_data, P.ws_data_bytes) &&
           CHK_REGION(v.sync, pr.iflags, prob_flags(nb, pr.k) * sizeof(int), P.ws_iflags, P.ws_iflags_n * sizeof(int)) &&
           CHK_REGION(v.sync, pr.progress, prob_tags(nb, pr.k) * sizeof(long long), P.ws_progress,
                      P.ws_progress_n * sizeof(long long)) &&
           CHK_REGION(v.sync, d, rc.bytes, pr.data, prob_data(nb, pr.k)) &&
           CHK_REGION(v.sync, v.dcar, (size_t)nb * kW * sizeof(double), pr.data, prob_data(nb, pr.k)) &&
           CHK_REGION(v.sync, v.ptag, pass_tags(nb, kb) * sizeof(long long), pr.progress,
                      prob_tags(nb, pr.k) * sizeof(long long)) &&
           CHK_RECT(v.sync, (long long)s, (long long)passes_of(pr.k), 1, 1 << 30);
#else
    return true;
#endif
}

// What thread 0 hands the block: a task of the problem in the view.
enum : int { kTaskNone = 0, kTaskPrep, kTaskPrep2, kTaskSub, kTaskCoef, kTaskSweep };
struct Picked {
    int kind, a, b;
};

// Task number x of the pass in `v` (x counts from the pass's first task),
// walking the block's stage cursor forward; kTaskNone past the last stage
// (the cursor then holds the pass's task count in `first`).
template <typename T>
__device__ Picked task_at(const View<T> &v, int x, Stage &st)
{
    Picked p{kTaskNone, 0, 0};
    const int stages = stage_count(v.nb, v.look);
    // (the column's segments are counted along: a division per stage and block
    // would cost microseconds)
    if (st.t == 0) {
        st.segs = 1;
        st.left = v.seg + 2 - seg_off(v.seg);  // segs_of grows where b - 2 + off is a multiple of seg
    }
    const int ush = v.units >> 1;  // units 1, 2, 4: a shift by 0, 1, 2
    for (; st.t < stages; ++st.t) {
        int c = 0;
        if (st.t == 0) c += 2 * min(v.nb, kPrepAhead);
        if (st.t + kPrepAhead < v.nb) c += 2;
        if (st.t < v.nb) c += v.kb;
        if (st.t >= v.look) c += 1 + ((st.segs + v.units - 1) >> ush);
        if (x < st.first + c) break;
        st.first += c;
        if (st.t >= v.look && --st.left == 0) {
            ++st.segs;
            st.left = v.seg;
        }
    }
    if (st.t >= stages) return p;
    int y = x - st.first;
    const int t = st.t;
    if (t == 0) {
        const int c = 2 * min(v.nb, kPrepAhead);
        if (y < c) return Picked{(y & 1) ? kTaskPrep2 : kTaskPrep, y >> 1, 0};
        y -= c;
    }
    if (t + kPrepAhead < v.nb) {
        if (y < 2) return Picked{y ? kTaskPrep2 : kTaskPrep, t + kPrepAhead, 0};
        y -= 2;
    }
    if (t < v.nb) {
        if (y < v.kb) return Picked{kTaskSub, y, t};
        y -= v.kb;
    }
    const int u = t - v.look;
    if (y == 0) return Picked{kTaskCoef, u, 0};
    return Picked{kTaskSweep, u, y - 1};
}

// One ticket of problem i: the task number, or -1 if none is left.  The
// ticket word is read first, so that an exhausted one is not counted up.
template <typename T>
__device__ __forceinline__ long long take_ticket(const Launch<T> &P, int i, long long ep64)
{
    const long long total = prob_of(P, i).ntasks;
    unsigned long long *w = ticket_of(P, i);
    const long long seen = ld_relaxed_gpu(reinterpret_cast<const long long *>(w));
    if (seen >= ep64 + total) return -1;
    if (seen < ep64) atomicMax(w, (unsigned long long)ep64);
    const long long x = (long long)atomicAdd(w, 1ull) - ep64;
    return x < total ? x : -1;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 8 ? 3 : 4) team_kernel(Launch<T> P)
{
    extern __shared__ __align__(16) unsigned char raw[];
    TaskSmem<T> &S = *reinterpret_cast<TaskSmem<T> *>(raw);
    __shared__ View<T> v;
    __shared__ Picked s_task;
    __shared__ int s_last, s_abort;
    int *ctl = P.ctl;
    const int epoch = ld_relaxed_gpu(ctl + kCtlEpoch);
    const long long ep64 = (long long)epoch << 32;
    // thread 0's scheduling state
    const int team = blockIdx.x % P.nteams;
    int prob = -1;      // the problem in the view
    Stage st{0, 0, 0, 0, 0};  // cursor in its task list
    if (threadIdx.x == 0) {
        v.pass = -1;
        s_task.kind = kTaskNone;
    }
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            s_task.kind = kTaskNone;
            int want = -1;
            long long x = -1;
            if (ld_relaxed_gpu(ctl + kCtlAbort) == 0 && P.nprobs == 1) {
                want = 0;
                x = take_ticket(P, 0, ep64);
            } else if (ld_relaxed_gpu(ctl + kCtlAbort) == 0) {
                // the problem at hand, then the team's (a new one once its
                // own is handed out), then, when no problem is left, another team's
                if (prob >= 0) {
                    x = take_ticket(P, prob, ep64);
                    want = prob;
                }
                int *word = ctl + kCtlTeam + team;
                for (unsigned it = 0; x < 0 && it < (1u << 22); ++it) {
                    const int cur = ld_relaxed_gpu(word);  // problem + 1; 0: none yet, -1: one is being named
                    if (cur < 0) {
                        __nanosleep(64);
                        continue;
                    }
                    if (cur > 0 && cur - 1 != prob) {
                        want = cur - 1;
                        x = take_ticket(P, want, ep64);
                        if (x >= 0) break;
                    }
                    if (ld_relaxed_gpu(ctl + kCtlPairNext) >= P.nprobs) break;
                    if (atomicCAS(word, cur, -1) != cur) continue;
                    const int next = atomicAdd(ctl + kCtlPairNext, 1);
                    atomicExch(word, next < P.nprobs ? next + 1 : cur);
                    prob = -1;  // (its tickets are all taken)
                }
                for (int d = 1; d < P.nteams && x < 0; ++d) {
                    int h = team + d;
                    if (h >= P.nteams) h -= P.nteams;
                    const int cur = ld_relaxed_gpu(ctl + kCtlTeam + h);
                    if (cur <= 0) continue;
                    want = cur - 1;
                    x = take_ticket(P, want, ep64);
                }
            }
            if (x >= 0) {
                if (want != prob) {
                    prob = want;
                    st = Stage{0, 0, 0, 0, 0};
                    v.pass = -1;
                }
                bool ok = true;
                const int np = passes_of(prob_of(P, prob).k);
                if (v.pass < 0) ok = set_view(P, prob, 0, epoch, v);
                Picked pk = ok ? task_at(v, (int)x - st.passes, st) : Picked{kTaskNone, 0, 0};
                while (ok && pk.kind == kTaskNone && v.pass + 1 < np) {
                    st = Stage{0, 0, st.passes + st.first, 0, 0};
                    ok = set_view(P, prob, v.pass + 1, epoch, v);
                    if (ok) pk = task_at(v, (int)x - st.passes, st);
                }
                s_task = pk;
            }
        }
        __syncthreads();
        const Picked pk = s_task;
        if (pk.kind == kTaskNone) break;
        if (pk.kind == kTaskPrep) {
            prep_task<T>(P, v, pk.a, S.prep);
        } else if (pk.kind == kTaskPrep2) {
            prep2_task<T>(v, pk.a, S.prep);
        } else if (pk.kind == kTaskSub) {
            sub_task<T>(P, v, pk.a, pk.b, S.sub);
        } else if (pk.kind == kTaskCoef) {
            coef_task<T>(P, v, pk.a, S.coef);
        } else {
            switch (v.KB) {
            case 1:
                if (sizeof(T) == 8 && v.units == 2) sweep_task<T, 1, 2, 1>(P, v, pk.a, pk.b, S.sweep12);
                else sweep_task<T, 1, 1, 1>(P, v, pk.a, pk.b, S.sweep1);
                break;
            case 2: sweep_task<T, 1, 2, 2>(P, v, pk.a, pk.b, S.sweep2); break;
            case 4: sweep_task<T, 1, 4, 4>(P, v, pk.a, pk.b, S.sweep4); break;
            default: sweep_task<T, 2, 4, 8>(P, v, pk.a, pk.b, S.sweep8); break;
            }
        }
    }

    // The last block to finish zeroes the control words for the next launch
    // and advances the epoch.
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(ctl + kCtlExited, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        // A wait that ran out aborted the whole launch: every problem that
        // recorded nothing stopped unfinished, so it is marked too (info -5:
        // stopped by another problem's failure) and none reads as complete.
        if (threadIdx.x == 0) s_abort = ld_relaxed_gpu(ctl + kCtlAbort);
        __syncthreads();
        if (s_abort) {
            for (int i = threadIdx.x; i < P.nprobs; i += blockDim.x) {
                long long *info = prob_of(P, i).info;
                if (info) record_one(info, kStatusTimeout, -5);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kCtlTeam + kMaxTeams; i += blockDim.x)
            if (i != kCtlEpoch) ctl[i] = 0;  // (the words this kernel uses; the others stay zero)
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            ctl[kCtlEpoch] = epoch + 1;
            __threadfence();
        }
    }
}

#undef TEAM_TRACE

}  // namespace team
}  // namespace chm
