// Scratch layout of the team kernel (chm_team.cuh), shared by the device
// code and the host side that carves scratch memory for one or many
// problems.  Plain C++ usable from host and device translation units.
#pragma once

#include "chm_layout.h"

namespace chm {
namespace team {

// Update vectors of one pass.  Eight keep a sweep task's coefficients and
// carries small enough for two blocks per SM in double, and a modification
// of more vectors runs its passes in a pipeline: pass s + 1 enters a column
// as soon as pass s has swept it.
constexpr int kTeamKb = 8;
// The kernels' instantiation for kb vectors: the next power of two.
CHM_HD inline int kb_inst(int kb) { return kb <= 1 ? 1 : kb <= 2 ? 2 : kb <= 4 ? 4 : 8; }
CHM_HD inline int passes_of(int k) { return (k + kTeamKb - 1) / kTeamKb; }

// Segments of a column swept by one task of four warps: one of four or eight
// vectors, two of two, four of one; in double up to 64 row blocks two of one,
// with a second warp each that scales and stores (see sweep_task).
CHM_HD inline bool store_warp(int nb, int KB, bool f64) { return f64 && KB == 1 && nb <= 64; }
CHM_HD inline int units_of(int nb, int KB, bool f64) { return KB >= 4 ? 1 : KB == 2 || store_warp(nb, KB, f64) ? 2 : 4; }

// Row blocks per sweep segment.  One or two vectors: two up to 64 row blocks
// in double (n = 512 0.094 to 0.070 ms; in float, whose tiles take a third of
// the time, no gain), else four, while that takes at most 64 segments of a column (whose starts'
// residuals are kept, n values per vector each): the last segment is what
// is left to do when the substitution ends.  More vectors: a twelfth of the
// column, at least four, since a task of `seg` tiles fills and drains its
// four warps' pipeline in seg + 3 steps (n = 5000, 16 vectors, double: 2.06 ms
// with segments of four, 1.69 with sixteen).  A multiple of four from four on.
CHM_HD inline int seg_of(int nb, int KB, bool f64)
{
    if (f64 && KB <= 2 && nb <= 64) return 2;
    const int s = (KB <= 2 ? (nb + 63) / 64 : (nb + 11) / 12) + 3;
    return s < 7 ? 4 : s & ~3;
}
// Segment s >= 1 starts at row block s seg - off: where a group of four tiles
// of the substitution (4 i - 2 .. 4 i + 1) begins, and for segments of two
// also in its middle.  A start needs the residual a SUB step keeps, which
// covers row blocks up to b - 2 of column block b, so b's last segment is the
// one that starts at or before row block b - 2.
CHM_HD inline int seg_off(int seg) { return seg == 2 ? 0 : 2; }
CHM_HD inline int seg_start(int s, int seg) { return s > 0 ? s * seg - seg_off(seg) : 0; }
CHM_HD inline int segs_of(int b, int seg)
{
    const int x = b - 2 + seg_off(seg);
    return 1 + (x > 0 ? x / seg : 0);
}
// Segment s if one starts at row block r (> 0), else 0.
CHM_HD inline int seg_at(int r, int seg) { return r > 0 && (r + seg_off(seg)) % seg == 0 ? (r + seg_off(seg)) / seg : 0; }
// Segment starts of the last column (the most any has); in double there are at
// least as many as in float.
CHM_HD inline int bounds_of(int nb, int KB, bool f64) { return segs_of(nb - 1, seg_of(nb, KB, f64)) - 1; }

// Byte offsets inside the data record of one pass of kb vectors (element
// sizes are the double's, so that one size serves both types).
struct PassRec {
    size_t ug;      // [nb][3][kW][kW]
    size_t coef;    // [nb * kW][2 KB]
    size_t escale;  // [nb * kW]
    size_t dfac;    // [nb * kW]
    size_t snap;    // [bounds][nb * kW][KB]
    size_t rst;     // [bounds][KB (KB + 1) / 2]
    size_t bytes;
};
CHM_HD inline PassRec pass_rec(int nb, int kb)
{
    const size_t rows = (size_t)nb * kW, KB = (size_t)kb_inst(kb), nd = (size_t)bounds_of(nb, kb_inst(kb), true);
    PassRec r;
    size_t x = 0;
    r.ug = x;     x += rows * 3 * kW * 8;
    r.coef = x;   x += rows * 2 * KB * 8;
    r.escale = x; x += rows * 8;
    r.dfac = x;   x += rows * 8;
    r.snap = x;   x += nd * rows * KB * 8;
    r.rst = x;    x += nd * KB * (KB + 1) / 2 * 8;
    r.bytes = align256(x);
    return r;
}
// A problem's passes all have kTeamKb vectors but the last; the diagonal
// carried from pass to pass ([nb * kW] doubles) follows them.
CHM_HD inline size_t pass_data_off(int nb, int s) { return (size_t)s * pass_rec(nb, kTeamKb).bytes; }
CHM_HD inline size_t prob_dcar(int nb, int k)
{
    const int np = passes_of(k);
    return pass_data_off(nb, np - 1) + pass_rec(nb, k - (np - 1) * kTeamKb).bytes;
}
CHM_HD inline size_t prob_data(int nb, int k) { return align256(prob_dcar(nb, k) + (size_t)nb * kW * 8); }
// A problem's data region is not the larger the larger n or k: a last pass of
// two vectors can keep more segment starts than one of eight, and the segments
// grow in steps with n.  A workspace that serves more than the one shape it was
// sized for (a modification's launches of 64 vectors and of what is left, a
// stream's later, smaller calls) is therefore sized by bounds that never
// fall: at least the segment starts of every order up to this one,
CHM_HD inline size_t bounds_cap(int nb, int KB)
{
    const int x = KB <= 2 ? nb / 2 : nb / 4, most = KB <= 2 ? 64 : 12;
    return (size_t)(x < most ? x : most);
}
// and at least the data region of every problem of up to nb blocks and k vectors.
CHM_HD inline size_t prob_data_cap(int nb, int k)
{
    const size_t rows = (size_t)nb * kW;
    size_t pass = 0;
    for (int KB = 1; KB <= kb_inst(k < kTeamKb ? k : kTeamKb); KB *= 2) {
        const size_t snap = bounds_cap(nb, KB) * (rows * KB + KB * (KB + 1) / 2) * 8;
        const size_t b = align256(rows * (3 * kW + 2 * KB + 2) * 8 + snap);
        if (b > pass) pass = b;
    }
    return align256((size_t)passes_of(k) * pass + rows * 8);
}
// Int flags: per pass, U, G1, G2, a block's kind and the coefficients published ([nb] each).
constexpr int kPassFlags = 5;
CHM_HD inline size_t prob_flags(int nb, int k) { return ((size_t)passes_of(k) * kPassFlags * nb + 63) & ~(size_t)63; }
// Epoch-tagged 64-bit words: per pass P ([kb][nb][kW][2]), the prefix Grams
// and the factors handed on in their place ([nb][KB (KB + 1) / 2][2] each) as
// tagged doubles; then the problem's ticket word and, per column block, the
// count of its segments swept ((epoch << 32) + count each).
CHM_HD inline size_t pass_tags(int nb, int kb)
{
    const int KB = kb_inst(kb);
    return (size_t)kb * nb * kW * 2 + 2 * (size_t)nb * KB * (KB + 1);
}
CHM_HD inline size_t pass_tag_off(int nb, int s) { return (size_t)s * pass_tags(nb, kTeamKb); }
CHM_HD inline size_t prob_ticket(int nb, int k)
{
    const int np = passes_of(k);
    return pass_tag_off(nb, np - 1) + pass_tags(nb, k - (np - 1) * kTeamKb);
}
CHM_HD inline size_t prob_tags(int nb, int k) { return (prob_ticket(nb, k) + 1 + (size_t)nb + 31) & ~(size_t)31; }

// ---------------------------------------------------------------- tasks

constexpr int kPrepAhead = 4;  // stages by which PREP runs ahead of SUB

// Blocks by which the substitution runs ahead of the coefficients and the
// sweep in the task order, so that the thread blocks holding its next steps
// have summed their tiles when the chain reaches them.
CHM_HD inline int look_of(int kb) { return kb >= 8 ? 12 : kb >= 4 ? 20 : 32; }
// Stage t of a pass hands out PREP and PREP2(t + kPrepAhead) (stage 0 also
// the first kPrepAhead), the kb SUB steps of block t, and for block
// u = t - look COEF(u) and column u's SWEEPs.
CHM_HD inline int stage_count(int nb, int look) { return nb + look; }
CHM_HD inline int stage_tasks(int t, int nb, int kb, int seg, int look, int units)
{
    int c = 0;
    if (t == 0) c += 2 * (nb < kPrepAhead ? nb : kPrepAhead);
    if (t + kPrepAhead < nb) c += 2;
    if (t < nb) c += kb;
    const int u = t - look;
    if (u >= 0 && u < nb) c += 1 + (segs_of(u, seg) + units - 1) / units;
    return c;
}
// All tasks of a problem.
inline int prob_tasks(int nb, int k, bool f64)
{
    int total = 0;
    for (int s = 0; s < passes_of(k); ++s) {
        const int kb = k - s * kTeamKb < kTeamKb ? k - s * kTeamKb : kTeamKb;
        const int KB = kb_inst(kb), look = look_of(kb), units = units_of(nb, KB, f64), seg = seg_of(nb, KB, f64);
        for (int t = 0; t < stage_count(nb, look); ++t) total += stage_tasks(t, nb, kb, seg, look, units);
    }
    return total;
}

}  // namespace team
}  // namespace chm
