// rqr.cu -- the QR iteration for a REAL Hessenberg matrix in FP32 (Algorithm
// 2, step 1, for real A): small-bulge multishift double-shift QR in real
// arithmetic down to a block triangular matrix with diagonal blocks of at
// most kQrTiny rows, then the complex Schur form of those blocks alone.  The
// result is the complex Schur form A_s = Q T Q^H that the rest of Algorithm 2
// takes.
//
// Why real: a pair of conjugate shifts costs one 3 x 3 Householder reflector
// per step on real entries (10 flops per 3-entry segment) where two complex
// single shifts cost two rotations on complex pairs (40 flops), a sweep of 16
// bulges carries 32 shifts instead of 16 (half the sweeps, the serial chain
// of the iteration: 13.9 k steps instead of 26.5 k for 3I + G/sqrt(n) at
// n = 512), and every deferred product is real (a quarter of the flops, half
// of the bytes).
//
// Chase.  Bulge g of a sweep sits at p_g = lo + t - 3 g in step t: its
// reflector P = I - tau v v^T, v = (1, v1, v2), acts on rows and columns
// p_g .. p_g + 2.  Bulges three positions apart tile the chain's rows (and
// columns) without gaps, so one step is a set of independent 3 x 3 tiles
// (row triple of bulge i, column triple of bulge j), each updated from both
// sides by one thread, with ONE barrier per step: the thread of a diagonal
// tile holds exactly the entries that define its bulge's next reflector and
// forms it before the barrier.  Every thread keeps the overlap of its
// consecutive tiles in registers: a tile moves down the diagonal by one per
// step, reads the row and column that come in and stores those that go out.
// Columns the chain has not reached take only left reflectors, as tiles that
// move with the chain; rows it has left take only right ones, and as nothing
// in the chain reads them again, they join the window's out-of-block rows
// with a later first step.  A step is bound by the latency of the diagonal
// tiles (loads, the two updates, a reciprocal square root and a reciprocal,
// the barrier); no conditional lies on that path while all bulges are on
// their way.
//
// Windows of W steps form dense tables of reflectors (W x NB), applied
// outside the window's block by rows and columns: by the chase CTA (one CTA
// per matrix), by helper CTAs (one large matrix), or in shared memory when
// the whole matrix fits there (n <= kRqrResident).  Everything outside the
// active block is deferred as in the complex iteration (qr.cu): a window's
// reflectors are multiplied into an orthogonal U_w, and two passes apply
// x <- x U_w to rows (Schur vectors, rows of T above the block) and
// y <- U_w^T y to columns right of it.
//
// Shifts: the eigenvalues of the trailing 2 nb x 2 nb block by the
// Ehrlich-Aberth iteration (see qr_small.cuh for the method) on the real
// block less the mean of its diagonal, started from the previous sweep's, taken
// in conjugate pairs.
// Deflation, exceptional shifts and the iteration cap are those of qr.cu.
#include <algorithm>

#include "internal.h"
#include "qr_small.cuh"
#include "tc_common.cuh"

namespace sqm {

namespace {

constexpr int NB = 16;               // bulges per sweep (2 NB shifts)
constexpr int W = 32;                // steps per window
constexpr int NS2 = 2 * NB;          // shifts
constexpr int MLD = NS2 + 1;         // leading dimension of the shift block
constexpr int RR = W - 1 + 3 * NB;   // largest index range of a window's reflectors (79)
constexpr int BW = RR + 2;           // largest window block: one row above, one below
constexpr int BLD = 81;              // its leading dimension: 17 mod 32 puts the 120 tiles beside
                                     // the diagonal into 4 warps without bank conflicts
constexpr int TS = 52;               // a table row: (v1, v2)[NB], tau[NB], padding
constexpr int kCta = 512;            // threads of every chase CTA and helper
constexpr int kStep = 352;           // threads that take part in a step (11 warps)
constexpr int kQuad = 128;           // threads of a group that applies a window to 32 segments
constexpr int KB = 4;                // steps between two barriers of such a group
constexpr int NAH = 11;              // column triples ahead of the chain
constexpr int kShiftIt = 12;         // iterations of the shift refinement
constexpr float kShiftTol = 3e-2f;   // and its tolerance relative to the spread of the estimates
constexpr int kShiftSlow = 6;        // after this many sweeps without deflation the refinement starts anew
constexpr int kShiftItSlow = 30;     // and may take this many iterations
constexpr int kRqrPostMin = 64;      // fewer out-of-window rows + columns: the chase CTA does them
constexpr int SLD = 81;              // staged segments: leading dimension (odd, >= RR)
constexpr int kStage = kCta / kQuad * 32 * SLD;  // staged floats: 32 segments per group of four warps
constexpr int TLD = 117;             // new columns: W of them, up to RR + W + 2 rows
static_assert(RR + W + 2 <= TLD && BW <= BLD && RR <= SLD && 3 * NAH > W && W % KB == 0, "shared-memory geometry");

constexpr size_t kTableBytes = 2 * (size_t)W * TS * sizeof(float);  // two windows' tables

template <int MODE>
constexpr size_t window_smem()
{
    return kTableBytes + (size_t)kStage * sizeof(float) + (size_t)BLD * BW * sizeof(float) * (MODE == 1 ? 2 : 1) +
           (MODE == 1 ? (size_t)TLD * W * sizeof(float) : 0);
}

// leading dimension of a resident matrix: 1 mod 4 and not 1 mod 32 (at most
// five tiles of the chain per bank, see BLD)
__host__ __device__ constexpr int resident_ld(int n)
{
    const int l = n <= 5 ? 5 : ((n + 2) & ~3) + 1;
    return l % 32 == 1 ? l + 4 : l;
}
constexpr size_t resident_smem(int n)
{
    return kTableBytes + (size_t)resident_ld(n) * n * sizeof(float);
}

// Warp roles in a step, spread over the SM's four sub-partitions (warp mod
// 4): 0: the diagonal tiles; 1, 2, 3, 5: the other chain tiles; 4, 6 .. 10:
// tiles ahead of the chain; 11 .. 15 take no part (in the cooperative chase
// 11 .. 14 follow on the next block's columns).
enum Role { R_DIAG, R_CHAIN, R_AHEAD, R_SIDE, R_NONE };
__device__ __forceinline__ int warp_role(int warp, int &idx)
{
    idx = 0;
    if (warp == 0) return R_DIAG;
    if (warp == 4) return R_AHEAD;
    if (warp <= 5) { idx = warp == 5 ? 3 : warp - 1; return R_CHAIN; }
    if (warp <= 10) { idx = warp - 5; return R_AHEAD; }
    idx = warp - 11;
    return idx < 4 ? R_SIDE : R_NONE;
}

__device__ __forceinline__ void quad_bar(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kQuad) : "memory"); }

// rows x cols elements by `nw` warps, the lanes along a column, U columns'
// loads in flight per lane: a copy of a window's block from L2 one load at a
// time took longer than the chase of the window
template <int U = 8, class LD, class ST>
__device__ __forceinline__ void copy_cols(int rows, int cols, int warp, int nw, LD load, ST store)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int b0 = warp * U; b0 < cols; b0 += nw * U)
#pragma unroll 1
        for (int a = lane; a < rows; a += 32) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = b0 + u < cols ? load(a, b0 + u) : 0.0f;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (b0 + u < cols) store(a, b0 + u, v[u]);
        }
}

struct Refl {
    float x, y, z;  // v1, v2, tau
};
__device__ __forceinline__ Refl table_get(const float *row, int g)
{
    const float2 v = *reinterpret_cast<const float2 *>(row + 2 * g);
    return Refl{v.x, v.y, row[2 * NB + g]};
}
__device__ __forceinline__ void table_put(float *row, int g, Refl v)
{
    *reinterpret_cast<float2 *>(row + 2 * g) = make_float2(v.x, v.y);
    row[2 * NB + g] = v.z;
}

__device__ __forceinline__ void step_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kStep) : "memory"); }

__device__ __forceinline__ float rcp_approx(float v)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float v)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
    return y;
}

// P = I - tau v v^T with v = (1, v1, v2) and P (x0, x1, x2)^T = (beta, 0, 0)^T:
// d = x0 + sign(x0) ||x||, v = x / d, tau = |d| / ||x||.  The reciprocal
// square root y of nn = ||x||^2 and the reciprocal of d take one Newton step
// each (see rsqrt_refined), folded into the products that follow: with e = 1 -
// nn y^2, ||x|| = nn y (1 + e / 2).  P is orthogonal to the rounding of one
// number only if tau is 2 / (1 + v1^2 + v2^2) for the v that was rounded, so
// |d| y takes a Newton step towards that: with tau = |d| / ||x|| as it came (its
// own three roundings beside those of v) the backward error of the Schur form
// was 1.5 times as large, 7.5e-6 / 5.0e-6 of ||A|| for 3 I + G / sqrt(n), n = 400.
// Tiny or huge nn take the scaled form; the
// test comes last, off the path of the result.
__device__ __forceinline__ void reflector3(float x0, float x1, float x2, Refl &v, float &beta)
{
    const float nn = fmaf(x0, x0, fmaf(x1, x1, x2 * x2));
    const float y = rsqrt_approx(nn);
    const float ns = copysignf(nn, x0);
    const float t = ns * y, h = 0.5f * t;
    const float e = fmaf(-nn * y, y, 1.0f);
    const float d = fmaf(h, e, x0 + t);
    const float z = rcp_approx(d);
    const float e2 = fmaf(-d, z, 1.0f);
    const float p1 = x1 * z, p2 = x2 * z;
    const float tau = fabsf(d) * y, ht = 0.5f * tau;
    v.x = fmaf(p1, e2, p1);
    v.y = fmaf(p2, e2, p2);
    const float g = fmaf(v.x, v.x, v.y * v.y);
    v.z = fmaf(tau, fmaf(-ht, g, 1.0f - ht), tau);
    beta = -fmaf(h, e, t);
    if (!(nn >= 1e-28f && nn <= 1e28f)) {
        const float m = fmaxf(fabsf(x0), fmaxf(fabsf(x1), fabsf(x2)));
        v = Refl{0.0f, 0.0f, 0.0f};
        beta = x0;
        if (m > 0.0f) {
            const float a0 = x0 / m, a1 = x1 / m, a2 = x2 / m;
            const float s = sqrtf(fmaf(a0, a0, fmaf(a1, a1, a2 * a2)));
            const float dd = a0 + copysignf(s, a0);
            v = Refl{a1 / dd, a2 / dd, fabsf(dd) / s};
            beta = -copysignf(s, a0) * m;
        }
    }
}

// one 3 x 3 tile at e (leading dimension ld): left reflector l, right
// reflector r
template <bool LEFT, bool RIGHT>
__device__ __forceinline__ void tile_update(float a[3][3], Refl l, Refl r)
{
    if (LEFT) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float w = l.z * fmaf(l.y, a[2][c], fmaf(l.x, a[1][c], a[0][c]));
            a[0][c] -= w;
            a[1][c] = fmaf(-w, l.x, a[1][c]);
            a[2][c] = fmaf(-w, l.y, a[2][c]);
        }
    }
    if (RIGHT) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float w = r.z * fmaf(r.y, a[q][2], fmaf(r.x, a[q][1], a[q][0]));
            a[q][0] -= w;
            a[q][1] = fmaf(-w, r.x, a[q][1]);
            a[q][2] = fmaf(-w, r.y, a[q][2]);
        }
    }
}
// First reflector of a bulge with shifts alpha +- i r (r >= 0) or alpha +- r
// (r < 0): from the first column of (H - s1)(H - s2) for the block starting at
// lo.  B(i, j) is element (i, j) at B[i + j ld].  The entries are scaled by a
// power of two to a largest of about 1 among those squared, so that the
// products of a block far below the matrix's scale do not underflow.
__device__ __noinline__ Refl intro_reflector(const float *B, int ld, int lo, float alpha, float r)
{
    const float a = B[lo + lo * ld], b = B[lo + (lo + 1) * ld], c = B[(lo + 1) + lo * ld],
                d = B[(lo + 1) + (lo + 1) * ld], e = B[(lo + 2) + (lo + 1) * ld];
    const float big = fmaxf(fabsf(a - alpha), fmaxf(fabsf(r), fabsf(c)));
    const float sc = __uint_as_float((254u - min(max(__float_as_uint(big) >> 23, 30u), 253u)) << 23);
    const float am = (a - alpha) * sc, dm = (d - alpha) * sc, rs = r * sc, cs = c * sc;
    const float x0 = fmaf(am, am, fmaf(b * sc, cs, rs * fabsf(rs))), x1 = cs * (am + dm), x2 = cs * (e * sc);
    const float m = fmaxf(fabsf(x0), fmaxf(fabsf(x1), fabsf(x2)));
    Refl v{0.0f, 0.0f, 0.0f};
    if (m > 0.0f) {
        float beta;
        const float im = 1.0f / m;
        reflector3(x0 * im, x1 * im, x2 * im, v, beta);
    }
    return v;
}

// how many rows of the current window's table are complete
__device__ __forceinline__ void prog_set(int *p, int v)
{
    asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int prog_get(const int *p)
{
    int v;
    asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
    return v;
}

// The diagonal tiles during a window (steps t0 .. t1 - 1; element (i, j) at
// B[i + j ld]), lane g: bulge g.  rt: the window's table, row 0 given; every
// step writes the next one's row, the last one rt_next's row 0.  Entries
// below the subdiagonal that a bulge has left are not cleared: nothing uses
// them.  One path for every step, entering and leaving bulges included: the
// chase kernels' code has to stay within the instruction caches (as separate
// steady and general paths, 130 KB in all, a step took 600 cycles in the
// kernel and the first iteration of each shift computation 40 k).
__device__ __forceinline__ void diag_window(float *B, int ld, int lo, int hi, int t0, int t1, int nb, float *rt,
                                            float *rt_next, const float2 *s_sh)
{
    const int g = threadIdx.x & 31;
    float a[3][3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) a[q][c] = 0.0f;
    Refl v{0.0f, 0.0f, 0.0f};
    if (g < NB) v = table_get(rt, g);
    // a holds columns p, p + 1 of the tile with the left reflector already
    // applied to them (before the barrier, in the shadow of the stores), s the
    // sums a_q0 + v1 a_q1
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
    bool held = false;
#pragma unroll 1
    for (int t = t0; t < t1; ++t) {
        if (g < NB) {
            const int p = lo + t - 3 * g;
            float *row = t + 1 < t1 ? rt + (t + 1 - t0) * TS : rt_next;
            float *e = B + p + p * ld;
            const bool act = g < nb && p >= lo && p < hi, k2 = act && p + 2 <= hi, k3 = act && p + 3 <= hi;
            if (act && !held) {
#pragma unroll
                for (int c = 0; c < 2; ++c)
#pragma unroll
                    for (int q = 0; q < 3; ++q) a[q][c] = (k2 || q < 2) ? e[q + c * ld] : 0.0f;
                if (p == lo) a[2][0] = 0.0f;  // (a bulge that enters: not cleared by the one before)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float w = v.z * fmaf(v.y, a[2][c], fmaf(v.x, a[1][c], a[0][c]));
                    a[0][c] -= w;
                    a[1][c] = fmaf(-w, v.x, a[1][c]);
                    a[2][c] = fmaf(-w, v.y, a[2][c]);
                }
                s0 = fmaf(v.x, a[0][1], a[0][0]);
                s1 = fmaf(v.x, a[1][1], a[1][0]);
                s2 = fmaf(v.x, a[2][1], a[2][0]);
                held = true;
            }
            // column p + 2 and the right reflector; f: the subdiagonal entry below
            float f = 0.0f;
#pragma unroll
            for (int q = 0; q < 3; ++q) a[q][2] = 0.0f;
            if (k2) {
#pragma unroll
                for (int q = 0; q < 3; ++q) a[q][2] = e[q + 2 * ld];
            }
            if (k3) f = e[3 + 2 * ld];
            const float w = v.z * fmaf(v.y, a[2][2], fmaf(v.x, a[1][2], a[0][2]));
            a[1][2] = fmaf(-w, v.x, a[1][2]);
            a[2][2] = fmaf(-w, v.y, a[2][2]);
            a[0][2] -= w;
            const float w1 = v.z * fmaf(v.y, a[1][2], s1), w2 = v.z * fmaf(v.y, a[2][2], s2),
                        w0 = v.z * fmaf(v.y, a[0][2], s0);
            a[1][0] -= w1;
            a[2][0] -= w2;
            const float u = v.z * v.y * f;
            // column p defines the next reflector
            Refl nxt;
            float beta;
            reflector3(a[1][0], a[2][0], -u, nxt, beta);
            a[0][0] -= w0;
            a[0][1] = fmaf(-w0, v.x, a[0][1]);
            a[0][2] = fmaf(-w0, v.y, a[0][2]);
            a[1][1] = fmaf(-w1, v.x, a[1][1]);
            a[1][2] = fmaf(-w1, v.y, a[1][2]);
            a[2][1] = fmaf(-w2, v.x, a[2][1]);
            a[2][2] = fmaf(-w2, v.y, a[2][2]);
            const float f1 = -u * v.x, f2 = fmaf(-u, v.y, f);
            if (!k2) {  // no further step of this bulge (or none at all)
                nxt = Refl{0.0f, 0.0f, 0.0f};
                beta = a[1][0];
                if (g < nb && t + 1 == 3 * g) nxt = intro_reflector(B, ld, lo, s_sh[g].x, s_sh[g].y);
            }
            table_put(row, g, nxt);
            if (act) {  // row p and column p leave the tile
                e[0] = a[0][0];
                e[ld] = a[0][1];
                e[1] = beta;
                if (k2) e[2 * ld] = a[0][2];
                if (!k2 || t + 1 == t1) {  // and the rest of it
                    e[1 + ld] = a[1][1];
                    if (k2) {
                        e[2 + ld] = a[2][1];
                        e[1 + 2 * ld] = a[1][2];
                        e[2 + 2 * ld] = a[2][2];
                    }
                    if (k3) {
                        e[3 + ld] = f1;
                        e[3 + 2 * ld] = f2;
                    }
                }
            }
            // the next tile: its columns p + 1, p + 2 with the left reflector
            v = nxt;
            const float b00 = a[1][1], b01 = a[1][2], b10 = a[2][1], b11 = a[2][2];
            const float x0 = v.z * fmaf(v.y, f1, fmaf(v.x, b10, b00)), x1 = v.z * fmaf(v.y, f2, fmaf(v.x, b11, b01));
            a[0][0] = b00 - x0;
            a[0][1] = b01 - x1;
            a[1][0] = fmaf(-x0, v.x, b10);
            a[1][1] = fmaf(-x1, v.x, b11);
            a[2][0] = fmaf(-x0, v.y, f1);
            a[2][1] = fmaf(-x1, v.y, f2);
            s0 = fmaf(v.x, a[0][1], a[0][0]);
            s1 = fmaf(v.x, a[1][1], a[1][0]);
            s2 = fmaf(v.x, a[2][1], a[2][0]);
        }
        step_bar();
    }
}

// A tile beside the diagonal during a window: rows of bulge gi; columns of
// bulge gj < gi (!AHEAD) or the gj-th triple right of the first bulge (AHEAD:
// left reflectors only, columns up to r1).  A lane keeps the overlap of its
// consecutive tiles.  extra (one warp's lanes 0 .. 15, bulge = lane): !AHEAD:
// while bulges are still entering at lo, the up to two rows between lo and the
// last one take the right reflectors here; AHEAD: once the first bulges have
// left at hi, the up to two columns right of the rest.  prog: one thread's
// step count for the warps that follow the chase.
template <bool AHEAD>
__device__ __forceinline__ void tile_window(float *B, int ld, int lo, int hi, int r1, int t0, int t1, int nb, int gi,
                                            int gj, bool extra, const float *rt, int *prog)
{
    float a[3][3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) a[q][c] = 0.0f;
    bool held = false;
    const int last = AHEAD ? r1 : hi;
#pragma unroll 1
    for (int t = t0; t < t1; ++t) {
        const float *row = rt + (t - t0) * TS;
        const int pi = lo + t - 3 * gi;
        const int pj = AHEAD ? lo + t + 3 + 3 * gj : lo + t - 3 * gj;
        if (gi < nb && pi >= lo && (AHEAD ? pj <= r1 && lo + t < hi : pj < hi)) {
            float *e = B + pi + pj * ld;
            const Refl l = table_get(row, gi);
            Refl r{0.0f, 0.0f, 0.0f};
            if (!AHEAD) r = table_get(row, gj);
            const bool c1 = !AHEAD || pj + 1 <= last, c2 = pj + 2 <= last;
            if (!held) {
                a[0][0] = e[0];
                a[1][0] = e[1];
                if (c1) {
                    a[0][1] = e[ld];
                    a[1][1] = e[1 + ld];
                }
                held = true;
            }
            a[2][0] = e[2];
            if (c1) a[2][1] = e[2 + ld];
            if (c2) {
                a[0][2] = e[2 * ld];
                a[1][2] = e[1 + 2 * ld];
                a[2][2] = e[2 + 2 * ld];
            } else {
                a[0][2] = a[1][2] = a[2][2] = 0.0f;
                if (AHEAD && !c1) a[0][1] = a[1][1] = a[2][1] = 0.0f;
            }
            tile_update<true, !AHEAD>(a, l, r);
            e[0] = a[0][0];
            e[1] = a[1][0];
            e[2] = a[2][0];
            if (c1) e[ld] = a[0][1];
            if (c2) e[2 * ld] = a[0][2];
            if (t + 1 == t1 || !c2) {  // the last step with this tile, or columns end: everything goes out
                if (c1) {
                    e[1 + ld] = a[1][1];
                    e[2 + ld] = a[2][1];
                }
                if (c2) {
                    e[1 + 2 * ld] = a[1][2];
                    e[2 + 2 * ld] = a[2][2];
                }
                held = false;
            } else {
                a[0][0] = a[1][1];
                a[0][1] = a[1][2];
                a[1][0] = a[2][1];
                a[1][1] = a[2][2];
            }
        }
        if (extra) {
            const int over = t - (hi - 1 - lo);
            const int ga = over > 0 ? (over + 2) / 3 : 0, gb = min(nb - 1, t / 3);  // bulges ga .. gb are on the way
            const int g = threadIdx.x & 31, pg = lo + t - 3 * g;
            if (g >= ga && g <= gb) {
                if (!AHEAD && t < 3 * (nb - 1)) {
                    const Refl v = table_get(row, g);
                    const bool k2 = pg + 2 <= hi;
#pragma unroll 1
                    for (int i = lo; i < lo + t - 3 * gb; ++i) {
                        float *e = B + i + pg * ld;
                        const float x0 = e[0], x1 = e[ld], x2 = k2 ? e[2 * ld] : 0.0f;
                        const float w = v.z * fmaf(v.y, x2, fmaf(v.x, x1, x0));
                        e[0] = x0 - w;
                        e[ld] = fmaf(-w, v.x, x1);
                        if (k2) e[2 * ld] = fmaf(-w, v.y, x2);
                    }
                }
                if (AHEAD && ga > 0) {
                    const Refl v = table_get(row, g);
#pragma unroll 1
                    for (int j = lo + t - 3 * ga + 3; j <= hi; ++j) {
                        float *e = B + pg + j * ld;
                        const float x0 = e[0], x1 = e[1], x2 = e[2];
                        const float w = v.z * fmaf(v.y, x2, fmaf(v.x, x1, x0));
                        e[0] = x0 - w;
                        e[1] = fmaf(-w, v.x, x1);
                        e[2] = fmaf(-w, v.y, x2);
                    }
                }
            }
        }
        step_bar();
        if (AHEAD && prog && threadIdx.x == 10 * 32) prog_set(prog, t - t0 + 2);
    }
}

// Which chain tile a lane of the chain warps w = 0 .. 3 takes: the pairs (i,
// j) of one shared-memory bank (3 i + 3 ld j mod 32) go to different warps as
// far as possible.  s_pair: 128 entries, i << 8 | j (i = NB: no tile); cnt: 4
// ints.  Every thread of the CTA calls it.
__device__ void assign_pairs(int ld, int *s_pair, int *cnt)
{
    const int tid = threadIdx.x;
    if (tid < 128) s_pair[tid] = NB << 8;
    if (tid < 4) cnt[tid] = 0;
    __syncthreads();
    if (tid < NB * (NB - 1) / 2) {
        int i = 1;
        while ((i + 1) * i / 2 <= tid) ++i;
        const int j = tid - i * (i - 1) / 2;
        const int bank = (3 * i + 3 * (ld & 31) * j) & 31;
        int rank = 0;
        for (int a = 1; a < NB; ++a)
            for (int b = 0; b < a; ++b)
                if ((((3 * a + 3 * (ld & 31) * b) & 31) == bank) && a * (a - 1) / 2 + b < tid) ++rank;
        int w = (rank + bank) & 3;
        while (true) {  // 120 tiles, 128 places
            const int k = atomicAdd(&cnt[w], 1);
            if (k < 32) {
                s_pair[w * 32 + k] = i << 8 | j;
                break;
            }
            w = (w + 1) & 3;
        }
    }
    __syncthreads();
}

// Apply one window's reflectors (table rt, steps 0 .. ns - 1) to 32 segments
// of rr indices at vec[i * stride] in shared memory (columns or rows: P is
// symmetric, so both take the same form); bulge g of step q acts on indices
// off + q + 3 (NB - 1 - g) .. + 2.  Lane = segment; the four warps sub = 0 ..
// 3 of a group (barrier id `bar`) take four bulges each, which span 12
// adjacent indices that move by one per step and that the lane holds in
// registers, KB steps at a time; warp sub runs one block of KB steps behind
// warp sub - 1, whose final entries it reads, so one barrier per block orders
// them.  Steps before qs are skipped (zero: a table row of zeros).  All table
// reads of a warp are the same for its lanes (but for qs).  TRAIL: a block
// waits for its table rows (prog_get(prog)).  All four warps call it.
template <bool TRAIL>
__device__ __noinline__ bool quad_window(float *vec, int stride, bool on, const float *rt, const float *zero, int qs,
                                         int ns, int off, int rr, int sub, int bar, const int *prog)
{
    constexpr int NG = NB / 4, L = 3 * NG, N = L - 1 + KB;
    __builtin_assume(__isShared(vec));
    __builtin_assume(__isShared(rt));
    __builtin_assume(__isShared(zero));
    float x[N];
    bool ok = true;
    if (!on) rr = 0;
    int A = off + 3 * (NB - NG * (sub + 1));
#pragma unroll
    for (int i = 0; i < L - 1; ++i) x[i] = ((unsigned)(A + i) < (unsigned)rr) ? vec[(A + i) * stride] : 0.0f;
    const int nblk = (ns + KB - 1) / KB;
#pragma unroll 1
    for (int st = 0; st < nblk + 3; ++st) {
        const int q0 = (st - sub) * KB;
        if (st >= sub && q0 < ns) {
            if (TRAIL) {
                int spins = 0;
                const int need = min(q0 + KB, ns);
                while (prog_get(prog) < need && ok) {
                    __nanosleep(40);
                    if (++spins > (1 << 22)) ok = false;  // the chase never takes this long
                }
            }
#pragma unroll
            for (int i = 0; i < KB; ++i) {
                const int r = A + L - 1 + i;
                x[L - 1 + i] = ((unsigned)r < (unsigned)rr) ? vec[r * stride] : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < KB; ++k) {
                const int q = q0 + k;
                const float *row = (q < ns && q >= qs) ? rt + q * TS : zero;
                const float4 a = *reinterpret_cast<const float4 *>(row + 2 * NG * sub);
                const float4 b = *reinterpret_cast<const float4 *>(row + 2 * NG * sub + 4);
                const float4 c = *reinterpret_cast<const float4 *>(row + 2 * NB + NG * sub);
                const float v1[4] = {a.x, a.z, b.x, b.z}, v2[4] = {a.y, a.w, b.y, b.w}, tau[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int j = 0; j < NG; ++j) {
                    const int m = k + 3 * (NG - 1 - j);
                    const float w = tau[j] * fmaf(v2[j], x[m + 2], fmaf(v1[j], x[m + 1], x[m]));
                    x[m] -= w;
                    x[m + 1] = fmaf(-w, v1[j], x[m + 1]);
                    x[m + 2] = fmaf(-w, v2[j], x[m + 2]);
                }
            }
#pragma unroll
            for (int i = 0; i < KB; ++i)
                if ((unsigned)(A + i) < (unsigned)rr) vec[(A + i) * stride] = x[i];
            A += KB;
#pragma unroll
            for (int i = 0; i < L - 1; ++i) x[i] = x[i + KB];
            if (q0 + KB >= ns) {
#pragma unroll
                for (int i = 0; i < L - 1; ++i)
                    if ((unsigned)(A + i) < (unsigned)rr) vec[(A + i) * stride] = x[i];
            }
        }
        quad_bar(bar);
    }
    return ok;
}

// Eigenvalue estimates of the real unreduced Hessenberg block M (m x m, m <=
// 32, leading dimension MLD) refined together by the Ehrlich-Aberth
// iteration with Hyman's recurrence (the method of cta_aberth_shifts in
// qr_small.cuh, here for real M: the running sums take two multiply-adds per
// entry instead of four).  M is the trailing block as centre_block leaves it,
// mnrm its largest entry.  The QR iteration does not see a translation, so
// every tolerance here and in the two functions below is relative to the
// spread of the estimates, max|z|, and not to the eigenvalues' distance from
// zero: relative to that, matrices as near to a multiple of I as 300 I + G /
// sqrt(n) ran into the iteration cap.  (Nor is it relative to mnrm, which in a
// graded M lies far above the eigenvalues: with 10^(10 (j - i) / n) on the
// entries they ran into it as well.)  On entry z holds m distinct estimates;
// true: the last corrections were at most kShiftTol max|z|.  Shifts need not
// be eigenvalues to rounding: the correction that passes the test is itself
// applied, and the iteration converges cubically.  An iteration costs about eight
// steps of a sweep; a resident matrix, whose sweeps are short, takes at most
// 6 + (rows of the active block) / 32 of them up to kShiftIt, the others kShiftIt
// (ms of chase, means over 80 to 100 matrices, this rule everywhere / kShiftIt
// everywhere: n = 101 0.805 / 0.813, 256 3.57 / 3.53, 300 4.60 / 4.51, 512 9.91 / 9.73).
//
// A half-warp per estimate (warps 0 .. 15 take 32), lane r of it keeping the
// sums of rows r and r + 16, as packed pairs (re, im): the packed FP32
// instructions and one broadcast for both estimates of a warp keep the issue
// slots down, which bound the iteration (32 estimates x 32 rows).
struct f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 f2_mk(float x, float y)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 f2_get(f2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
// largest of a warp's non-negative values
__device__ __forceinline__ float warp_max(float v)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
// 1 / (x + i y) to about 1e-6 (an estimate of an estimate: shifts only);
// a zero or overflowing modulus gives zero
__device__ __forceinline__ float2 crcp_approx(float x, float y)
{
    const float m = fmaxf(fabsf(x), fabsf(y));
    if (!(m > 1e-30f && m < 1e30f)) return make_float2(0.0f, 0.0f);
    float im;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(im) : "f"(m));
    const float xs = x * im, ys = y * im;
    float d;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(d) : "f"(fmaf(xs, xs, ys * ys)));
    return make_float2(xs * im * d, -ys * im * d);
}

__device__ __noinline__ bool cta_aberth_real(const float *M, int m, float2 *z, float mnrm, int kmax)
{
    __shared__ float s_inv[NS2];
    __shared__ float2 s_w[NS2];
    __shared__ int s_bad;
    __builtin_assume(__isShared(M));
    __builtin_assume(__isShared(z));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float floor_sub = mnrm * 1e-20f;
    if (tid < m) {
        float sb = tid ? M[tid + (tid - 1) * MLD] : 1.0f;
        if (!(fabsf(sb) > floor_sub)) sb = floor_sub;
        s_inv[tid] = -1.0f / sb;
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    static_assert(kCta >= 32 * 16, "warps 0 .. 15 take the estimates");
    const int r = lane & 15, j = 2 * warp + (lane >> 4);  // row (and row + 16), estimate
#pragma unroll 1
    for (int it = 0; it < kmax; ++it) {
        if (2 * warp < m) {  // (m is even)
            const float2 mu = z[j];
            const f2 zero2 = f2_mk(0.0f, 0.0f), nmx = f2_mk(-mu.x, -mu.x), nmy = f2_mk(mu.y, -mu.y);
            f2 s0 = zero2, ds0 = zero2, s1 = zero2, ds1 = zero2, dx = zero2, x = f2_mk(1.0f, 0.0f);
            const float *c0 = M + min(r, m - 1), *c1 = M + min(r + 16, m - 1);
#pragma unroll 1
            for (int i = m - 1;; --i) {
                // column i of (M - mu I) into rows 0 .. i (rows below are done)
                const float a0 = c0[i * MLD], a1 = c1[i * MLD], iv = s_inv[i];
                const f2 p0 = f2_mk(a0, a0), p1 = f2_mk(a1, a1);
                s0 = f2_fma(p0, x, s0);
                ds0 = f2_fma(p0, dx, ds0);
                s1 = f2_fma(p1, x, s1);
                ds1 = f2_fma(p1, dx, ds1);
                // row i with the diagonal's -mu x_i (and -x_i in the derivative),
                // over -M(i, i-1): x_{i-1} and its derivative
                const float2 xv = f2_get(x), dv = f2_get(dx);
                f2 cc = f2_fma(nmx, x, i < 16 ? s0 : s1);
                f2 dd = f2_fma(nmx, dx, i < 16 ? ds0 : ds1);
                cc = f2_fma(nmy, f2_mk(xv.y, xv.x), cc);
                dd = f2_fma(nmy, f2_mk(dv.y, dv.x), dd);
                dd = f2_add(dd, f2_mk(-xv.x, -xv.y));
                const f2 iv2 = f2_mk(iv, iv);
                cc = f2_mul(cc, iv2);
                dd = f2_mul(dd, iv2);
                float2 c = f2_get(cc), d = f2_get(dd);
                c.x = __shfl_sync(0xffffffffu, c.x, i & 15, 16);
                c.y = __shfl_sync(0xffffffffu, c.y, i & 15, 16);
                d.x = __shfl_sync(0xffffffffu, d.x, i & 15, 16);
                d.y = __shfl_sync(0xffffffffu, d.y, i & 15, 16);
                x = f2_mk(c.x, c.y);
                dx = f2_mk(d.x, d.y);
                if (i == 0) break;
                if ((i & 3) == 0) {  // back into range by powers of two (the same in every lane of the half)
                    const float mag = fmaxf(fmaxf(fabsf(c.x), fabsf(c.y)), fmaxf(fabsf(d.x), fabsf(d.y)));
                    const int e = min(max((int)((__float_as_uint(mag) >> 23) & 255), 1), 253);
                    const float sc = mag > 1.0e6f || mag < 1.0e-6f ? __uint_as_float((unsigned)(254 - e) << 23) : 1.0f;
                    const f2 sc2 = f2_mk(sc, sc);
                    x = f2_mul(x, sc2);
                    dx = f2_mul(dx, sc2);
                    s0 = f2_mul(s0, sc2);
                    ds0 = f2_mul(ds0, sc2);
                    s1 = f2_mul(s1, sc2);
                    ds1 = f2_mul(ds1, sc2);
                }
            }
            // x, dx: the residual of row 0 and its derivative, p and p' up to a
            // factor (s_inv[0] = -1 in both)
            const float2 xv = f2_get(x), dv = f2_get(dx);
            const float2 id = crcp_approx(dv.x, dv.y);
            const float nx = xv.x * id.x - xv.y * id.y, ny = xv.x * id.y + xv.y * id.x;
            float2 part = make_float2(0.0f, 0.0f);
#pragma unroll 1
            for (int q = r; q < m; q += 16)
                if (q != j) {
                    const float2 zr = z[q], t = crcp_approx(mu.x - zr.x, mu.y - zr.y);
                    part.x += t.x;
                    part.y += t.y;
                }
            for (int o = 8; o > 0; o >>= 1) {
                part.x += __shfl_xor_sync(0xffffffffu, part.x, o);
                part.y += __shfl_xor_sync(0xffffffffu, part.y, o);
            }
            const float2 iq = crcp_approx(1.0f - (nx * part.x - ny * part.y), -(nx * part.y + ny * part.x));
            if (r == 0) s_w[j] = make_float2(nx * iq.x - ny * iq.y, nx * iq.y + ny * iq.x);
        }
        __syncthreads();
        bool done = true;
        if (warp == 0) {  // (m <= 32)
            const float2 w = lane < m ? s_w[lane] : make_float2(0.0f, 0.0f);
            float2 zn = make_float2(0.0f, 0.0f);
            if (lane < m) {
                zn = make_float2(z[lane].x - w.x, z[lane].y - w.y);
                if (!(isfinite(zn.x) && isfinite(zn.y))) s_bad = 1;
                z[lane] = zn;
            }
            done = fmaxf(fabsf(w.x), fabsf(w.y)) <= kShiftTol * warp_max(fmaxf(fabsf(zn.x), fabsf(zn.y)));
        }
        const int all = __syncthreads_and(done);
        if (s_bad) return false;
        if (all) return true;
    }
    return false;
}

// M (m x m) less the mean of its diagonal, times a power of two that takes its
// largest entry to [1, 2).  Every thread of the CTA calls it, behind a barrier;
// mnrm (shared) is 0 on entry.  Returns the mean, that power's inverse and
// the largest entry.
__device__ __noinline__ float3 centre_block(float *M, int m, float *mnrm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kCta / 32;
    const float ctr = warp_sum(lane < m ? M[lane + lane * MLD] : 0.0f) * rcp_approx((float)m);
    float mx = 0.0f;
#pragma unroll 1
    for (int j = warp; j < m; j += nw)
        if (lane < m) mx = fmaxf(mx, fabsf(M[lane + j * MLD] - (lane == j ? ctr : 0.0f)));
    mx = warp_max(mx);
    if (lane == 0) atomicMax(reinterpret_cast<int *>(mnrm), __float_as_int(mx));  // (non-negative: ordered as integers)
    __syncthreads();
    mx = *mnrm;
    const unsigned ex = min(max(__float_as_uint(mx) >> 23, 1u), 253u);
    const float sc = __uint_as_float((254u - ex) << 23);
#pragma unroll 1
    for (int j = warp; j < m; j += nw)
        if (lane < m) M[lane + j * MLD] = (M[lane + j * MLD] - (lane == j ? ctr : 0.0f)) * sc;
    __syncthreads();
    return make_float3(ctr, __uint_as_float(ex << 23), mx * sc);
}

// Starting estimates (one warp; lane q holds the q-th previous estimate).  prev
// and defl are eigenvalues of the matrix, ctr the mean that centre_block took
// from M, 1 / isc its scale.
// Warm start: the np estimates of the previous sweep, whose trailing block
// ended dh rows lower; for each of the dh eigenvalues deflated since (defl)
// the nearest is dropped, and at most m stay; the remaining places (all for a
// cold start, np = 0) take eigenvalues of M's 2 x 2 diagonal blocks.
__device__ __noinline__ void warp_shift_start(const float *M, int m, float mnrm, float ctr, float isc, const float2 *prev, int np,
                                              const float2 *defl, int dh, float2 *z)
{
    const int lane = threadIdx.x & 31;
    float2 c = lane < np ? prev[lane] : make_float2(0.0f, 0.0f);
    const float sc = rcp_approx(isc);  // (a power of two)
    c = make_float2((c.x - ctr) * sc, c.y * sc);
    bool alive = lane < np;
    for (int q = 0; q < dh; ++q) {
        const float ex = c.x - (defl[q].x - ctr) * sc, ey = c.y - defl[q].y * sc;
        // the distance's leading bits with the lane below them
        const unsigned key = alive ? (__float_as_uint(fmaf(ex, ex, ey * ey)) & ~31u) | lane : 0xffffffffu;
        const unsigned best = __reduce_min_sync(0xffffffffu, key);
        if (best != 0xffffffffu && lane == (int)(best & 31u)) alive = false;
    }
    {  // at most m stay
        const unsigned am = __ballot_sync(0xffffffffu, alive);
        if (__popc(am & ((1u << lane) - 1u)) >= m) alive = false;
    }
    const int cnt = __popc(__ballot_sync(0xffffffffu, alive));
    const unsigned am = __ballot_sync(0xffffffffu, alive);
    if (alive) z[__popc(am & ((1u << lane) - 1u))] = c;
    // the spread as the 2 x 2 blocks show it (a diagonal scaling of M does not
    // change it, where the largest entry of a graded M says nothing)
    float spread = 0.0f;
    if (lane < m) {
        spread = fabsf(M[lane + lane * MLD]);
        if (lane + 1 < m) spread = fmaxf(spread, sqrtf(fabsf(M[lane + (lane + 1) * MLD] * M[(lane + 1) + lane * MLD])));
    }
    spread = 5e-2f * fmaxf(warp_max(spread), 1e-6f * mnrm);
    const int q = lane - cnt;  // places cnt .. m-1
    if (q >= 0 && lane < m) {
        // an eigenvalue of the 2 x 2 diagonal block (q & ~1, q | 1), the
        // places moved apart along the m-th roots of unity
        const int b0 = q & ~1, b1 = min(b0 + 1, m - 1);
        const float a = M[b0 + b0 * MLD], d = M[b1 + b1 * MLD], h = 0.5f * (a - d);
        const float disc = b1 > b0 ? fmaf(h, h, M[b0 + b1 * MLD] * M[b1 + b0 * MLD]) : 0.0f;
        const float r = ((q & 1) ? -1.0f : 1.0f) * sqrtf(fabsf(disc)), mid = 0.5f * (a + d);
        float sn, cs;
        sincospif((2.0f * q + 0.5f) / (float)m, &sn, &cs);
        sn *= spread;
        cs *= spread;
        z[lane] = disc < 0.0f ? make_float2(mid + cs, r + sn) : make_float2(mid + r + cs, sn);
    }
    __syncwarp();
}

// The m estimates z (of M, see above) as bulges: sh[g] = (alpha, r) for
// intro_reflector, in the matrix's own scale (isc = 1 / sc): a conjugate pair
// alpha +- i beta gives r = beta, two real estimates r = -|a - b| / 2.  One
// warp; returns the number of bulges (at most nb, at least 1).
__device__ __noinline__ int warp_pair_shifts(const float2 *z, int m, float ctr, float isc, float2 *sh, int nb)
{
    const int lane = threadIdx.x & 31;
    const float2 c = lane < m ? z[lane] : make_float2(0.0f, 0.0f);
    const bool in = lane < m;
    const float thr = 1e-3f * warp_max(fmaxf(fabsf(c.x), fabsf(c.y)));
    unsigned up = __ballot_sync(0xffffffffu, in && c.y > thr);
    const unsigned dn = __ballot_sync(0xffffffffu, in && c.y < -thr);
    const unsigned re = __ballot_sync(0xffffffffu, in && fabsf(c.y) <= thr);
    const bool use_dn = __popc(dn) > __popc(up);
    if (use_dn) up = dn;
    const int nu = __popc(up), nr = __popc(re);
    const unsigned lt = (1u << lane) - 1u;
    if ((up >> lane) & 1u) {
        const int k = __popc(up & lt);
        if (k < nb) sh[k] = make_float2(fmaf(c.x, isc, ctr), fabsf(c.y) * isc);
    }
    // the r-th real estimate pairs with the (r ^ 1)-th
    __shared__ float s_re[32];
    const bool isr = (re >> lane) & 1u;
    const int rk = __popc(re & lt);
    if (isr) s_re[rk] = c.x;
    __syncwarp();
    const float other = isr && (rk ^ 1) < nr ? s_re[rk ^ 1] : c.x;
    if (isr && !(rk & 1)) {
        const int k = nu + (rk >> 1);
        if (k < nb) sh[k] = make_float2(fmaf(0.5f * (c.x + other), isc, ctr), -0.5f * fabsf(c.x - other) * isc);
    }
    __syncwarp();
    return max(1, min(nb, nu + (nr + 1) / 2));
}

constexpr int kMaxHelpers = 64;  // the sync array holds 4 + this many ints

constexpr uint64_t kWaitNs = 2000000000ull;  // bounded inter-CTA waits (~2 s) unless the descriptor sets one

__device__ __forceinline__ uint64_t wait_lim(const SchurDesc<float> &d) { return d.wait_ns ? (uint64_t)d.wait_ns : kWaitNs; }

// One warp waits until each of the H helpers has finished `target` windows,
// each lane watching two; false (warp-uniform) if a helper failed or the wait gave up.
__device__ bool poll_helpers(const SchurDesc<float> &d, int H, int target)
{
    const int lane = threadIdx.x & 31;
    bool ok = true;
    static_assert(kMaxHelpers <= 64, "two helpers per lane");
    if (lane < H) {
        volatile int *sy = d.sync;
        const int second = lane + 32 < H ? lane + 32 : lane;
        const uint64_t t0 = globaltimer_ns(), lim = wait_lim(d);
        while (sy[4 + lane] < target || sy[4 + second] < target) {
            if (sy[2] || globaltimer_ns() - t0 > lim) { ok = false; break; }
            __nanosleep(64);  // keep the polls off the helpers' L2 lines
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    __threadfence();
    return ok;
}

// every thread of the CTA
__device__ bool wait_all_helpers(const SchurDesc<float> &d, int H, int target)
{
    __shared__ int s_ok;
    if (threadIdx.x < 32) {
        const bool ok = poll_helpers(d, H, target);
        if (threadIdx.x == 0) s_ok = ok;
    }
    __syncthreads();
    const bool ok = s_ok != 0;
    __syncthreads();
    return ok;
}

// The out-of-window segments of one window, staged in shared memory: columns
// c0 .. c1 (left reflectors) and rows ra .. rb - 1 (right reflectors; row i >=
// r0 is one the chain left during the window and starts at step i + qoff), in
// groups of 8 consecutive indices.  With H > 0 only the groups g = h (mod H);
// H = 0: all of them.  A warp stages a group (all of its loads in flight at
// once: one at a time they took longer than the chase of the window), four
// warps apply the window to four groups.
constexpr int kQuads = kCta / kQuad;

__device__ __noinline__ void staged_window(float *T, int64_t ld, float *stage, const float *rt, const float *zero, int ns, int off,
                              int kmin, int rr, int c0, int c1, int ra, int rb, int r0, int qoff, int H, int h)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m = H > 0 ? H : 1, hh = H > 0 ? h : 0;
    auto first = [&](int i) {  // first owned group at or after index i's
        const int g = i >> 3;
        return g + ((hh - g % m) % m + m) % m;
    };
    auto count = [&](int g, int last) { return g > (last >> 3) ? 0 : ((last >> 3) - g) / m + 1; };
    const int gc = first(c0), gr = first(ra);
    const int nc = c1 < c0 ? 0 : count(gc, c1), nr = rb <= ra ? 0 : count(gr, rb - 1);
    constexpr int NG8 = 4 * kQuads;  // groups at a time
    for (int b0 = 0; b0 < nc + nr; b0 += NG8) {
        __syncthreads();
        const int k = b0 + warp;  // this warp's group
        const bool has = warp < NG8 && k < nc + nr, col = k < nc;
        const int i0 = col ? 8 * (gc + k * m) : 8 * (gr + (k - nc) * m);
        float *sg = stage + warp * 8 * SLD;
        if (has && col) {
#pragma unroll 1
            for (int z = 0; z < (RR + 31) / 32; ++z) {
                const int v = lane + 32 * z;
                float x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    x[u] = (v < rr && i0 + u >= c0 && i0 + u <= c1) ? __ldcg(T + kmin + v + (i0 + u) * ld) : 0.0f;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (v < rr) sg[u * SLD + v] = x[u];
            }
        } else if (has) {
            const int r = lane & 7, i = i0 + r;
            const bool in = i >= ra && i < rb;
                constexpr int NV = (RR + 3) / 4;  // 20
#pragma unroll 1
            for (int z = 0; z < 2; ++z) {
                float x[NV / 2];
#pragma unroll
                for (int u = 0; u < NV / 2; ++u) {
                    const int v = (lane >> 3) + 4 * (u + z * (NV / 2));
                    x[u] = (in && v < rr) ? __ldcg(T + i + (kmin + v) * ld) : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < NV / 2; ++u) {
                    const int v = (lane >> 3) + 4 * (u + z * (NV / 2));
                    if (v < rr) sg[r * SLD + v] = x[u];
                }
            }
        }
        __syncthreads();
        const int quad = warp >> 2;
        if (quad < kQuads && b0 + 4 * quad < nc + nr) {  // groups b0 + 4 quad .. + 3, lane = segment
            const int kk = b0 + 4 * quad + (lane >> 3);
            const bool cc = kk < nc;
            const int i = (cc ? 8 * (gc + kk * m) : 8 * (gr + (kk - nc) * m)) + (lane & 7);
            quad_window<false>(stage + (quad * 32 + lane) * SLD, 1, kk < nc + nr, rt, zero,
                               cc || i < r0 ? 0 : max(0, i + qoff), ns, off, rr, warp & 3, 2 + quad, nullptr);
        }
        __syncthreads();
        if (has && col) {
            for (int u = 0; u < 8; ++u)
                if (i0 + u >= c0 && i0 + u <= c1)
                    for (int v = lane; v < rr; v += 32) T[kmin + v + (i0 + u) * ld] = sg[u * SLD + v];
        } else if (has) {
            const int r = lane & 7, i = i0 + r;
            if (i >= ra && i < rb)
                for (int v = lane >> 3; v < rr; v += 4) T[i + (kmin + v) * ld] = sg[r * SLD + v];
        }
    }
}

// Helper CTA h of the cooperative chase (the protocol of qr_helper in
// qr.cu): for every posted window, in order, the left reflectors on the
// columns right of the next window's block and the right ones on the rows
// above it, on the groups of 8 indices it owns (no other CTA writes them, so
// the windows need no ordering between helpers).  Then it publishes its
// count.  One thread's fence after a barrier covers the CTA's stores (a
// fence by every warp took most of a window's time).
__device__ __noinline__ void helper_cta(const SchurDesc<float> &d, float *T, int H, int h, float *stage, float *rt, const float *zero)
{
    const int nt = (int)blockDim.x;
    __shared__ int s_go, s_nwin;
    __shared__ int s_win[12];
    const int tid = threadIdx.x;
    for (int w = 0;; ++w) {
        if (tid == 0) {
            volatile int *sy = d.sync;
            const uint64_t t0 = globaltimer_ns(), lim = wait_lim(d);
            int go = 0;
            while (true) {
                // the last post: its count and, above, its window record
                const unsigned v = (unsigned)sy[0];
                const int cnt = (int)(v & 0xffffu);
                if (cnt > w) {
                    go = 1;
                    s_nwin = cnt == w + 1 ? (int)(v >> 16) : -1;
                    break;
                }
                if (sy[1]) { go = 2; break; }
                if (sy[2] || globaltimer_ns() - t0 > lim) { go = 3; break; }
            }
            __threadfence();
            s_go = go;
        }
        __syncthreads();
        const int go = s_go;
        if (go != 1) {
            if (go == 3 && tid == 0) atomicExch(&d.sync[2], 1);
            return;
        }
        const int nwin = s_nwin >= 0 ? s_nwin : __ldcg(d.postlist + w);
        if (tid < 12) s_win[tid] = __ldcg(reinterpret_cast<const int *>(&d.win[nwin]) + tid);
        // (the whole table of the window, whatever its number of steps: the
        // record and the table come in one round trip)
        const float4 *lg = reinterpret_cast<const float4 *>(d.log) + (int64_t)nwin * (W * NB);
        for (int e = tid; e < W * (TS / 4); e += nt) reinterpret_cast<float4 *>(rt)[e] = __ldcg(lg + e);
        __syncthreads();
        const int kbase = s_win[1], ns = s_win[2], kmin = s_win[3], rr = s_win[4];
        const int lo = s_win[5], hi = s_win[6], t0w = s_win[7], nb = s_win[8], r0 = s_win[9], rnext = s_win[10];
        const int r0n = max(lo, max(lo, lo + t0w + ns - 3 * (nb - 1)) - 1);
        staged_window(T, d.n, stage, rt, zero, ns, kbase - kmin, kmin, rr, rnext + 1, hi, lo, r0n, r0,
                      -lo + 3 * (nb - 1) + 1 - t0w, H, h);
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            atomicExch(&d.sync[4 + h], w + 1);
        }
    }
}

}  // namespace

// The chase.  MODE 0: one CTA per matrix, windows staged from global memory;
// 1: CTA 0 chases and posts its windows to the helper CTAs 1 .. H, one of its
// warps follows the chase on the next block's new columns, and the next block
// is assembled in shared memory; 2: one CTA per matrix with the
// whole matrix in shared memory.  Matrices with n outside (nlo, nhi] return
// at once (the size classes of a batch).
// Bound by the serial chain of steps (one barrier each, about 300 cycles of
// dependent arithmetic in the diagonal tiles) and by instruction supply: one
// warp's code runs once a step, so it misses the instruction cache unless each
// role has a single path.  One path for every step, loops left rolled outside
// the steps and an estimate of the shifts per half-warp, against a fast and a
// general copy and an estimate per warp, ms of chase: n = 64 0.35 / 0.54, 101
// 0.83 / 0.99, 200 2.14 / 2.85, 256 3.38 / 5.48, 512 10.1 / 12.5, 1024 31.4 /
// 32.6, 2048 97.5 / 112.9.  (Since then, with shifts relative to the spread and tau
// from the rounded v, means over 4 to 12 matrices before / after: n = 64 0.44 /
// 0.44, 101 0.79 / 0.80, 200 2.32 / 2.38, 512 9.6 / 9.7, 1024 30.2 / 30.7, 2048 100 to
// 103 / 100 to 106.)
template <int MODE>
__global__ void __launch_bounds__(kCta, 1)
rqr_chase_kernel(const SchurDesc<float> *__restrict__ descs, int H, int nlo, int nhi)
{
    constexpr int nt = kCta;
    extern __shared__ __align__(16) unsigned char smraw[];
    float *tab = reinterpret_cast<float *>(smraw);        // two tables of W rows, used in turn
    float *dyn = tab + 2 * W * TS;
    __shared__ float2 s_sh[NB];                           // the sweep's shifts (alpha, r)
    __shared__ float s_m[NS2 * MLD];
    __shared__ float2 s_z[NS2], s_prev[NS2], s_defl[NS2];
    __shared__ int s_pair[128], s_cnt[4];
    __shared__ __align__(16) float s_zero[TS];
    __shared__ float s_mnrm, s_sub;
    __shared__ int s_prevn, s_prevhi, s_fail;
    __shared__ int s_prog;
    __shared__ int s_lo, s_hi, s_iter, s_status, s_done, s_nb, s_sweeps, s_stop, s_multi;
    __shared__ long long s_rots, s_work;

    const SchurDesc<float> d = descs[MODE == 1 ? 0 : blockIdx.x];
    if (MODE != 1 && (d.n <= nlo || d.n > nhi)) return;
    float *T = reinterpret_cast<float *>(d.w);
    int *bst = reinterpret_cast<int *>(d.v);
    float *stage = dyn;                                   // MODE 0, 1
    float *blk0 = dyn + kStage;                            // window block(s)
    float *tile = dyn + kStage + 2 * BLD * BW;             // MODE 1
    if (threadIdx.x < TS) s_zero[threadIdx.x] = 0.0f;
    if (MODE == 1 && blockIdx.x > 0) {
        helper_cta(d, T, H, (int)blockIdx.x - 1, stage, tab, s_zero);
        return;
    }
    const int n = d.n, ld = n;
    float *S = dyn;                                       // MODE 2: the whole matrix
    const int lds = resident_ld(n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int ridx;
    const int role = warp_role(warp, ridx);
    const float eps = num<float>::eps;
    int *st = d.state;
    auto at = [&](int i, int j) -> float {
        if (MODE == 2) return S[i + j * lds];
        if (MODE == 1) return __ldcg(T + i + (int64_t)j * ld);
        return T[i + (int64_t)j * ld];
    };
    auto put = [&](int i, int j, float v) {
        if (MODE == 2) S[i + j * lds] = v;
        else T[i + (int64_t)j * ld] = v;
    };
    if (st[2]) {  // already finished: nothing new in the log
        if (tid == 0) {
            st[3] = 0; st[7] = 0; d.rstate[0] = 0;
            if (MODE == 1) atomicExch(&d.sync[1], 1);
        }
        return;
    }
    if (tid == 0) {
        s_hi = (st[0] < -1) ? n - 1 : st[0];
        s_iter = st[1];
        s_status = 0;
        s_done = 0;
        s_sweeps = st[4];
        s_rots = (long long)st[5] + ((long long)st[6] << 31);
        s_work = (long long)st[8] + ((long long)st[9] << 31);
        s_stop = 0;
        s_prevn = 0;
        s_prevhi = 0;
        s_fail = 0;
    }
    assign_pairs(MODE == 2 ? lds : BLD, s_pair, s_cnt);
    const int pair = role == R_CHAIN ? s_pair[ridx * 32 + lane] : NB << 8;
    if (MODE == 2)
        copy_cols(n, n, warp, nt / 32, [&](int i, int j) { return T[i + (int64_t)j * ld]; },
                  [&](int i, int j, float v) { S[i + j * lds] = v; });
    __syncthreads();

    // log, window, U and posted-window counts: the same in every thread
    int nlog = 0, nwin = 0, npost = 0, par = 0;
    long long uoff = 0;
    while (true) {
        const int hi = s_hi;
        if (hi < 0) { if (tid == 0) s_done = 1; break; }
        if (tid == 0) s_lo = 0;
        __syncthreads();
        for (int k = 1 + tid; k <= hi; k += nt) {
            const float as = fabsf(at(k, k - 1));
            if (as == 0.0f || as <= eps * (fabsf(at(k, k)) + fabsf(at(k - 1, k - 1)))) atomicMax(&s_lo, k);
        }
        __syncthreads();
        const int lo = s_lo, m = hi - lo + 1;
        if (m <= kQrTiny) {
            // a small active block is final for the real iteration: the
            // complex Schur form of its diagonal block comes at the end
            if (tid < m) bst[lo + tid] = lo;
            if (tid == 0) {
                if (lo > 0) put(lo, lo - 1, 0.0f);
                s_hi = lo - 1;
                s_iter = 0;
            }
            __syncthreads();
            continue;
        }
        if (tid == 0) {
            int nb = min(NB, max(1, (m - 2) / 6));
            const long long nwin_sweep = ((hi - lo) + 3 * (nb - 1) + W - 1) / W;
            const bool fits = nlog + nwin_sweep * (W * NB) <= d.log_cap && nwin + nwin_sweep <= d.win_cap &&
                              uoff + nwin_sweep * (long long)(RR * RR) <= 2 * d.u_cap;
            s_multi = 0;
            if (!fits) {
                s_stop = 1;  // drain the log first
                if (nlog == 0 && nwin == 0 && uoff == 0) s_status = 7;  // can never fit
            } else {
                if (lo > 0) put(lo, lo - 1, 0.0f);
                const int it = ++s_iter;
                ++s_sweeps;
                if (it > kItMax) s_status = 3;
                if (it % 10 == 0) {  // exceptional: a double real shift off the bottom entry
                    nb = 1;
                    s_sh[0] = make_float2(fmaf(0.75f, fabsf(at(hi, hi - 1)), at(hi, hi)), 0.0f);
                } else {
                    s_multi = 1;
                }
                s_nb = nb;
            }
        }
        __syncthreads();
        if (s_stop || s_status) break;
        if (s_multi) {
            const int nb0 = s_nb, ms = 2 * nb0, b0 = hi - ms + 1;
            if (tid == 0) s_mnrm = 0.0f;
            copy_cols(ms, ms, warp, nt / 32, [&](int i, int j) { return i <= j + 1 ? at(b0 + i, b0 + j) : 0.0f; },
                      [&](int i, int j, float v) { s_m[i + j * MLD] = v; });
            const int dh = s_prevhi - hi;
            const bool slow = s_iter > kShiftSlow;
            const bool warm = s_prevn > 0 && dh >= 0 && dh < ms && !slow;
            if (warm && tid < dh) {
                // an eigenvalue estimate of each deflated row: its diagonal
                // entry, or the pair of the 2 x 2 block it heads or ends
                const int i = hi + 1 + tid;
                float re = at(i, i), im = 0.0f;
                if (i + 1 < n && tid + 1 < dh) {
                    const float bc = at(i, i + 1) * at(i + 1, i);
                    if (bc < 0.0f) im = sqrtf(-bc);
                }
                if (im == 0.0f && tid > 0) {
                    const float bc = at(i - 1, i) * at(i, i - 1);
                    if (bc < 0.0f) im = -sqrtf(-bc);
                }
                s_defl[tid] = make_float2(re, im);
            }
            __syncthreads();
            const float3 cb = centre_block(s_m, ms, &s_mnrm);
            const float ctr = cb.x, isc = cb.y, mnrm = cb.z;
            if (warp == 0)
                warp_shift_start(s_m, ms, mnrm, ctr, isc, s_prev, warm ? s_prevn : 0, s_defl, warm ? dh : 0, s_z);
            __syncthreads();
            // Unconverged estimates are shifts all the same (and non-finite ones
            // are replaced by the block's diagonal) while the iteration gets on
            cta_aberth_real(s_m, ms, s_z, mnrm, slow ? kShiftItSlow : MODE == 2 ? min(kShiftIt, 6 + m / 32) : kShiftIt);
            if (tid < ms) {
                if (!(isfinite(s_z[tid].x) && isfinite(s_z[tid].y))) s_z[tid] = make_float2(s_m[tid + tid * MLD], 0.0f);
                s_prev[tid] = make_float2(fmaf(s_z[tid].x, isc, ctr), s_z[tid].y * isc);
            }
            __syncthreads();
            if (warp == 0) {
                const int k = warp_pair_shifts(s_z, ms, ctr, isc, s_sh, nb0);
                if (lane == 0) {
                    s_nb = k;
                    s_prevn = ms;
                    s_prevhi = hi;
                }
            }
            __syncthreads();
        }
        const int nb = s_nb;
        if (tid == 0) {
            s_rots += (long long)(hi - lo) * nb;
            // in-block work: each reflector updates about m 3-entry segments
            s_work += (long long)(hi - lo) * nb * (long long)m;
        }
        const int nsteps = (hi - lo) + 3 * (nb - 1);
        int cur = 0;  // MODE 1: block buffer in use

        for (int t0 = 0; t0 < nsteps; t0 += W) {
            const int t1 = min(t0 + W, nsteps), ns = t1 - t0;
            const int kmin = max(lo, lo + t0 - 3 * (nb - 1));
            const int kmax = min(hi - 1, lo + t1 - 1);
            const int r0 = max(lo, kmin - 1);
            const int r1 = min(hi, kmax + 3);
            const int bw = r1 - r0 + 1, rr = min(kmax + 2, hi) - kmin + 1;
            const int kbase = lo + t0 - 3 * (NB - 1), off = kbase - kmin;
            if (bw > BW || rr > RR) {  // cannot happen; guards the shared-memory bounds
                if (tid == 0) s_status = 7;
                __syncthreads();
                break;
            }
            // next window's block: its last column, its first row
            const bool last = t1 >= nsteps;
            const int rnext = last ? hi : min(hi, min(hi - 1, lo + min(t1 + W, nsteps) - 1) + 3);
            const int r0n = max(lo, max(lo, lo + t1 - 3 * (nb - 1)) - 1);
            const bool post = MODE == 1 && (hi - rnext) + (r0n - lo) > kRqrPostMin;
            float *B;
            int bld;
            if (MODE == 2) {
                B = S;
                bld = lds;
            } else {
                B = blk0 + cur * (BLD * BW) - r0 - r0 * BLD;
                bld = BLD;
                if (MODE == 0 || t0 == 0)
                    copy_cols(bw, bw, warp, nt / 32,
                              [&](int a, int b) { return a <= b + 3 ? at(r0 + a, r0 + b) : 0.0f; },
                              [&](int a, int b, float v) { blk0[cur * (BLD * BW) + a + b * BLD] = v; });
            }
            float *rt = tab + par * (W * TS), *rt_next = tab + (par ^ 1) * (W * TS);
            if (t0 == 0) {
                if (MODE != 2) __syncthreads();
                if (tid < NB)
                    table_put(rt, tid, tid == 0 ? intro_reflector(B, bld, lo, s_sh[0].x, s_sh[0].y)
                                                : Refl{0.0f, 0.0f, 0.0f});
            }
            if (MODE == 1 && t0 == 0 && tid == 0) s_prog = 1;
            if (MODE != 1 || t0 == 0) __syncthreads();
            const int cn = MODE == 1 ? rnext - r1 : 0;  // the next block's new columns
            if (role == R_DIAG) {
                diag_window(B, bld, lo, hi, t0, t1, nb, rt, rt_next, s_sh);
            } else if (role == R_CHAIN) {
                tile_window<false>(B, bld, lo, hi, r1, t0, t1, nb, pair >> 8, pair & 255, ridx == 3, rt, nullptr);
            } else if (role == R_AHEAD) {
                const int b = 2 * ridx + (lane >> 4);
                tile_window<true>(B, bld, lo, hi, b < NAH ? r1 : -1, t0, t1, nb, lane & 15, b, ridx == 0, rt,
                                  MODE == 1 ? &s_prog : nullptr);
            } else if (MODE == 1 && role == R_SIDE && cn > 0) {
                // four warps: once the helpers are done with every window
                // posted before this one, the new columns are read and follow
                // the chase, a lane per column
                if (ridx == 0 && !poll_helpers(d, H, npost) && lane == 0) s_fail = 1;
                quad_bar(2);
                if (!s_fail) {
                    const int rows = rnext - kmin + 1;
                    copy_cols(rows, cn, ridx, 4,
                              [&](int v, int j) {
                                  return kmin + v <= r1 + 2 + j ? __ldcg(&T[(kmin + v) + (int64_t)(r1 + 1 + j) * ld]) : 0.0f;
                              },
                              [&](int v, int j, float x) { tile[v + j * TLD] = x; });
                    if (ridx == 1 && lane == 0) s_sub = __ldcg(&T[(r1 + 1) + (int64_t)r1 * ld]);
                    quad_bar(2);
                    if (!quad_window<true>(tile + lane * TLD, 1, lane < cn, rt, s_zero, 0, ns, off, rr, ridx, 2, &s_prog))
                        s_fail = 1;
                    for (int j = ridx; j < cn; j += 4)
                        for (int v = lane; v < min(rows, r1 + 2 + j - kmin + 1); v += 32)
                            T[(kmin + v) + (int64_t)(r1 + 1 + j) * ld] = tile[v + j * TLD];
                }
            }
            __syncthreads();
            if (MODE == 1 && s_fail) {
                if (tid == 0) s_status = 6;
                __syncthreads();
                break;
            }
            float4 *lg = reinterpret_cast<float4 *>(d.log) + nlog;
            for (int e = tid; e < ns * (TS / 4); e += nt) lg[e] = reinterpret_cast<const float4 *>(rt)[e];
            if (MODE != 2) {
                // cooperative: the rows that leave the block; else all of it
                const float *bk = blk0 + cur * (BLD * BW);
                const int rows = MODE == 1 && !last ? r0n - r0 : bw;
                for (int b = warp; b < bw; b += nt / 32)
                    for (int a = lane; a < (MODE == 1 && !last ? min(b + 2, rows + (b + 1 == rows)) : min(b + 4, bw)); a += 32)
                        T[(r0 + a) + (int64_t)(r0 + b) * ld] = bk[a + b * BLD];
            }
            if (tid == 0) {
                WinRec wr;
                wr.start = nlog; wr.kbase = kbase; wr.nsteps = ns; wr.kmin = kmin; wr.rr = rr;
                wr.lo = lo; wr.hi = hi; wr.t0 = t0; wr.nb = nb; wr.r0 = r0; wr.rnext = rnext; wr.pad = 0;
                wr.uoff = uoff;
                d.win[nwin] = wr;
                if (post) d.postlist[npost] = nwin;
                if (MODE == 1) s_prog = 1;  // for the next window
            }
            if (MODE == 1 && !last) {
                // the next block: the chain's part of this one, the new
                // columns, and the subdiagonal entry between them
                const float *bk = blk0 + cur * (BLD * BW);
                float *nbk = blk0 + (cur ^ 1) * (BLD * BW);
                const int keep = r1 - r0n + 1, sh = r0n - r0;
                copy_cols<4>(keep, keep, warp, nt / 32, [&](int a, int b) { return bk[(a + sh) + (b + sh) * BLD]; },
                             [&](int a, int b, float v) { nbk[a + b * BLD] = v; });
                copy_cols<4>(rnext - r0n + 1, cn, nt / 32 - 1 - warp, nt / 32,
                             [&](int a, int b) { return tile[(r0n - kmin + a) + b * TLD]; },
                             [&](int a, int b, float v) { nbk[a + (keep + b) * BLD] = v; });
                // below the kept part: zeros (never used, but multiplied by zeros)
                // and the subdiagonal entry before the new columns
                for (int b = warp; b < keep; b += nt / 32)
                    for (int a = keep + lane; a < keep + cn; a += 32)
                        nbk[a + b * BLD] = a == keep && b == keep - 1 ? s_sub : 0.0f;
            }
            if (MODE == 1) {
                __syncthreads();
                if (post && tid == kCta - 1) {  // (no thread that the next steps wait for)
                    __threadfence();
                    atomicExch(&d.sync[0], (npost + 1) | (nwin << 16));
                }
                if (!post && (hi > rnext || r0n > lo) && !wait_all_helpers(d, H, npost)) {
                    if (tid == 0) s_status = 6;
                    __syncthreads();
                    break;
                }
            }
            const int qoff = -lo + 3 * (nb - 1) + 1 - t0;  // first step of a row the chain has left
            if (MODE == 2) {
                // the rest of the active block, in place: columns r1+1 .. hi
                // and the rows behind the chain, a lane each
                const int nc = hi - r1, nr = r0n - lo;
                for (int s0 = (warp >> 2) * 32; s0 < nc + nr && (warp >> 2) < kQuads; s0 += kQuads * 32) {
                    const int sg = s0 + lane, i = lo + sg - nc;
                    const bool on = sg < nc + nr, col = sg < nc;
                    quad_window<false>(col ? S + kmin + (r1 + 1 + sg) * lds : S + (on ? i : lo) + kmin * lds, col ? 1 : lds, on,
                                       rt, s_zero, col || i < r0 ? 0 : max(0, i + qoff), ns, off, rr, warp & 3,
                                       2 + (warp >> 2), nullptr);
                }
            } else if (!post) {
                // columns right of the block (cooperative: beyond the new
                // columns) and rows behind the chain, staged
                staged_window(T, ld, stage, rt, s_zero, ns, off, kmin, rr, (MODE == 1 ? rnext : r1) + 1, hi, lo, r0n, r0, qoff, 0, 0);
                if (MODE == 1) __syncthreads();
            }
            if (MODE != 1) __syncthreads();
            if (post) ++npost;
            nwin += 1;
            uoff += (long long)rr * rr;
            nlog += W * NB;
            par ^= 1;
            cur ^= MODE == 1 ? 1 : 0;
        }
        __syncthreads();
        // cooperative chase: the sweep's out-of-window updates are done
        // before the next sweep reads T
        if (MODE == 1 && !s_status && !wait_all_helpers(d, H, npost)) {
            if (tid == 0) s_status = 6;
            __syncthreads();
        }
        if (s_status) break;
    }
    __syncthreads();
    if (MODE == 2)
        for (int j = warp; j < n; j += nt / 32)
            for (int i = lane; i < n; i += 32) T[i + (int64_t)j * ld] = S[i + j * lds];
    if (tid == 0) {
        st[0] = s_hi;
        st[1] = s_iter;
        st[2] = (s_done || s_status) ? 1 : 0;
        st[3] = nlog;
        st[7] = nwin;
        d.rstate[0] = nwin;
        st[4] = s_sweeps;
        st[5] = (int)(s_rots & 0x7fffffff);
        st[6] = (int)(s_rots >> 31);
        st[8] = (int)(s_work & 0x7fffffff);
        st[9] = (int)(s_work >> 31);
        if (s_status) *d.status = s_status;
        if (MODE == 1) {
            __threadfence();
            atomicExch(&d.sync[1], 1);  // helpers leave once every posted window is done
        }
        if (d.counters) {
            d.counters[0] = s_sweeps;
            d.counters[1] = st[5];
            d.counters[2] = st[6];
            d.counters[3] = st[8];
            d.counters[4] = st[9];
        }
    }
}

namespace {

// Accumulated product of one window's reflectors, U = I P_1 P_2 ... (in log
// order), stored row by row: the segment x of a row that receives the
// window's right reflectors becomes x U, the segment y of a column that
// receives its left ones U^T y.
constexpr int kBuildThreads = 3 * kQuad;  // 32 rows of U per group
constexpr size_t kBuildSmem = (size_t)W * TS * sizeof(float) + (size_t)96 * SLD * sizeof(float);
static_assert(RR <= 96, "three groups cover U");

__global__ void __launch_bounds__(kBuildThreads) rqr_build_u_kernel(const SchurDesc<float> *__restrict__ descs)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ __align__(16) float s_zero[TS];
    float *rt = reinterpret_cast<float *>(smraw);
    float *u = rt + W * TS;
    const SchurDesc<float> d = descs[blockIdx.y];
    const int nwin = d.rstate[0];
    if (threadIdx.x < TS) s_zero[threadIdx.x] = 0.0f;
    for (int wi = blockIdx.x; wi < nwin; wi += gridDim.x) {
        __syncthreads();  // the previous window's shared-memory reads are done
        const WinRec w = d.win[wi];
        const int rr = w.rr, ns = w.nsteps;
        if (rr > RR || rr < 2 || ns < 1 || ns > W) {
            if (threadIdx.x == 0) atomicExch(d.status, 7);
            continue;
        }
        const float4 *src = reinterpret_cast<const float4 *>(d.log) + w.start;
        for (int e = threadIdx.x; e < ns * (TS / 4); e += blockDim.x) reinterpret_cast<float4 *>(rt)[e] = src[e];
        for (int e = threadIdx.x; e < rr * rr; e += blockDim.x) u[(e % rr) + (e / rr) * SLD] = (e % rr == e / rr) ? 1.0f : 0.0f;
        __syncthreads();
        const int q = threadIdx.x / kQuad, r = 32 * q + (threadIdx.x & 31);
        quad_window<false>(u + r * SLD, 1, r < rr, rt, s_zero, 0, ns, w.kbase - w.kmin, rr, (threadIdx.x >> 5) & 3, 1 + q,
                           nullptr);
        __syncthreads();
        float *U = reinterpret_cast<float *>(d.ubuf) + w.uoff;
        for (int e = threadIdx.x; e < rr * rr; e += blockDim.x) U[e] = u[(e % rr) + (e / rr) * SLD];  // U(q, c) at q rr + c
    }
}

// The deferred passes: x <- x U_w for each window in order, a CTA holding
// `per` vectors of length n in shared memory (buf[v + c PL], v fastest).
// !COLS: rows of T (grid x < ctas_t; only rows above the window's block,
// i < lo) and of the Schur vectors (every window); COLS: columns of T right
// of the block (j > hi).  A thread takes one column c of U and RV vectors:
// one load of U and one vector load of x give RV multiply-adds.  Only
// entries a window changed are written back (the rest may belong to a later
// active block that the chase is updating meanwhile).
constexpr int kDefThreads = 256;
constexpr int kUPad = 96;  // columns of U, padded to whole warps

template <bool COLS, int RV>
__global__ void __launch_bounds__(kDefThreads)
rqr_deferred_kernel(const SchurDesc<float> *__restrict__ descs, int per, int ctas_t)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const SchurDesc<float> d = descs[blockIdx.y];
    const int n = d.n, ld = n;
    const int nwin = d.rstate[0];
    if (nwin == 0) return;
    const bool isT = COLS || blockIdx.x < (unsigned)ctas_t;
    const int cb = isT ? blockIdx.x : blockIdx.x - ctas_t;
    const int i0 = cb * per;
    if (i0 >= n) return;
    const int rn = min(per, n - i0);
    float *M = reinterpret_cast<float *>(d.w) + (isT ? 0 : (size_t)n * n);
    const int PL = per;                                        // a multiple of RV
    float *ub[2] = {reinterpret_cast<float *>(smraw), reinterpret_cast<float *>(smraw) + RR * RR};
    int *mask = reinterpret_cast<int *>(ub[1] + RR * RR + 2);  // per entry c: rows below mask / columns above it changed
    float *buf = reinterpret_cast<float *>(smraw) + ((2 * RR * RR + 2 + n + 3) & ~3);
    for (int c = threadIdx.x; c < n; c += kDefThreads) mask[c] = COLS ? n : 0;
    for (int e = threadIdx.x; e < PL * n; e += kDefThreads) {
        int a, b;
        if (COLS) { b = e % n; a = e / n; }
        else { a = e % PL; b = e / PL; }
        buf[a + (size_t)b * PL] = a < rn ? (COLS ? M[b + (int64_t)(i0 + a) * ld] : M[(i0 + a) + (int64_t)b * ld]) : 0.0f;
    }
    auto next_win = [&](int wi) {
        while (wi < nwin && isT && (COLS ? i0 + rn - 1 <= d.win[wi].hi : i0 >= d.win[wi].lo)) ++wi;
        return wi;
    };
    auto fetch_u = [&](int wi, float *dst) {
        const WinRec w = d.win[wi];
        const float *src = reinterpret_cast<const float *>(d.ubuf) + w.uoff;
        for (int e = threadIdx.x; e < w.rr * w.rr; e += kDefThreads) {
            unsigned sa = (unsigned)__cvta_generic_to_shared(dst + e);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(src + e) : "memory");
        }
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int groups = PL / RV, tasks = groups * (kUPad / 32);
    constexpr int MAXT = (32 / RV * (kUPad / 32) + kDefThreads / 32 - 1) / (kDefThreads / 32);
    int wi = next_win(0), par = 0;
    if (wi < nwin) fetch_u(wi, ub[0]);
    while (wi < nwin) {
        const WinRec w = d.win[wi];
        const int rr = w.rr;
        cp_async_wait_all();
        __syncthreads();
        const int wn = next_win(wi + 1);
        if (wn < nwin) fetch_u(wn, ub[par ^ 1]);
        const float *us = ub[par];
        float acc[MAXT][RV];
#pragma unroll
        for (int k = 0; k < MAXT; ++k) {
            const int task = warp + k * (kDefThreads / 32);
#pragma unroll
            for (int v = 0; v < RV; ++v) acc[k][v] = 0.0f;
            if (task < tasks) {
                const int c = (task % (kUPad / 32)) * 32 + lane, g = task / (kUPad / 32);
                const float *x = buf + g * RV + (size_t)w.kmin * PL;
                const float *uc = us + min(c, rr - 1);
#pragma unroll 4
                for (int q = 0; q < rr; ++q) {
                    const float uq = uc[q * rr];
                    float xv[RV];
                    if (RV == 4) *reinterpret_cast<float4 *>(xv) = *reinterpret_cast<const float4 *>(x + (size_t)q * PL);
                    else
#pragma unroll
                        for (int v = 0; v < RV; ++v) xv[v] = x[(size_t)q * PL + v];
#pragma unroll
                    for (int v = 0; v < RV; ++v) acc[k][v] = fmaf(xv[v], uq, acc[k][v]);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < MAXT; ++k) {
            const int task = warp + k * (kDefThreads / 32);
            const int c = (task % (kUPad / 32)) * 32 + lane, g = task / (kUPad / 32);
            if (task < tasks && c < rr) {
#pragma unroll
                for (int v = 0; v < RV; ++v) {
                    const int a = i0 + g * RV + v;
                    if (!isT || (COLS ? a > w.hi : a < w.lo)) buf[g * RV + v + (size_t)(w.kmin + c) * PL] = acc[k][v];
                }
                if (g == 0) mask[w.kmin + c] = COLS ? min(mask[w.kmin + c], w.hi) : max(mask[w.kmin + c], w.lo);
            }
        }
        wi = wn;
        par ^= 1;
    }
    cp_async_wait_all();
    __syncthreads();
    for (int e = threadIdx.x; e < rn * n; e += kDefThreads) {
        int a, b;
        if (COLS) { b = e % n; a = e / n; }
        else { a = e % rn; b = e / rn; }
        if (!isT || (COLS ? i0 + a > mask[b] : i0 + a < mask[b])) {
            if (COLS) M[b + (int64_t)(i0 + a) * ld] = buf[a + (size_t)b * PL];
            else M[(i0 + a) + (int64_t)b * ld] = buf[a + (size_t)b * PL];
        }
    }
}

// real copies of H and the Hessenberg stage's Q, block starts, QR state
__global__ void rqr_begin_kernel(const SchurDesc<float> *__restrict__ descs)
{
    const SchurDesc<float> d = descs[blockIdx.y];
    const int n = d.n;
    float *T = reinterpret_cast<float *>(d.w), *Q = T + (size_t)n * n;
    int *bst = reinterpret_cast<int *>(d.v);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)n * n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t % n), j = (int)(t / n);
        T[t] = i <= j + 1 ? d.T[i + (int64_t)j * d.ld].x : 0.0f;
        Q[t] = d.Q[i + (int64_t)j * d.ld].x;
        if (j == 0) bst[i] = i;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        d.state[0] = -2;  // fresh: start from hi = n - 1
        for (int q = 1; q < kQrStateInts; ++q) d.state[q] = 0;
        if (d.counters) d.counters[5] = d.counters[6] = 0;
    }
}

// The complex Schur form of each diagonal block (rows i with bst[i] = its
// first row; at most kQrTiny of them), one warp each: its unitary factor
// into ub (n x kQrTiny, row i of a block's U at ub + i kQrTiny), its upper
// triangular T_II into T.
__global__ void __launch_bounds__(32) rqr_blocks_kernel(const SchurDesc<float> *__restrict__ descs)
{
    __shared__ cplx<float> M[kQrTiny * kQrTinyLd], U[kQrTiny * kQrTinyLd];
    const SchurDesc<float> d = descs[blockIdx.y];
    const int n = d.n, lane = threadIdx.x;
    const float *T = reinterpret_cast<const float *>(d.w);
    const int *bst = reinterpret_cast<const int *>(d.v);
    cplx<float> *ub = d.ubuf;
    for (int i0 = blockIdx.x; i0 < n; i0 += gridDim.x) {
        if (bst[i0] != i0) continue;
        const int m = __popc(__ballot_sync(0xffffffffu, lane < kQrTiny && i0 + lane < n && bst[min(i0 + lane, n - 1)] == i0));
        // scaled by a power of two to a largest entry in [1, 2): the shifts of a
        // block far below the matrix's scale are roots of products of its entries
        float mx = 0.0f;
        for (int e = lane; e < m * m; e += 32) {
            const int a = e % m, b = e / m;
            const float t = a <= b + 1 ? T[(i0 + a) + (int64_t)(i0 + b) * n] : 0.0f;
            M[a + b * kQrTinyLd] = cplx<float>{t, 0.0f};
            U[a + b * kQrTinyLd] = cplx<float>{a == b ? 1.0f : 0.0f, 0.0f};
            mx = fmaxf(mx, fabsf(t));
        }
        const unsigned ex = min(max(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)) >> 23, 1u), 253u);
        const float sc = __uint_as_float((254u - ex) << 23), isc = __uint_as_float(ex << 23);
        for (int e = lane; e < m * m; e += 32) M[e % m + (e / m) * kQrTinyLd].x *= sc;
        __syncwarp();
        int nsw = 0, nrot = 0;
        const bool ok = warp_tiny_schur<float, kQrTinyLd>(M, U, m, &nsw, &nrot);
        __syncwarp();
        for (int e = lane; e < m * m; e += 32) {
            const int a = e % m, b = e / m;
            d.T[(i0 + a) + (int64_t)(i0 + b) * d.ld] = a <= b ? isc * M[a + b * kQrTinyLd] : cplx<float>{0.0f, 0.0f};
            ub[(i0 + a) * kQrTiny + b] = U[a + b * kQrTinyLd];
        }
        if (lane == 0) {
            if (!ok) atomicExch(d.status, 3);
            if (d.counters && nsw) {
                atomicAdd(&d.counters[5], nsw);
                atomicAdd(&d.counters[6], nrot);
            }
        }
        __syncwarp();
    }
}

// T_IJ = U_I^H T_IJ U_J (J > I), zeros below, and Q_J = Q_J U_J as complex
// matrices: CTA (x, y) takes the diagonal blocks that start in columns
// 32 x .. 32 x + 31 and the row blocks that start in rows 128 y .. 128 y +
// 127; z: T or Q of each matrix.
constexpr int kFinThreads = 256, kFinRows = 128;

__global__ void __launch_bounds__(kFinThreads) rqr_finish_kernel(const SchurDesc<float> *__restrict__ descs)
{
    __shared__ cplx<float> uj[kQrTiny * kQrTiny];
    __shared__ cplx<float> Y[(kFinRows + kQrTiny) * kQrTiny];
    const SchurDesc<float> d = descs[blockIdx.z >> 1];
    const bool isQ = blockIdx.z & 1;
    const int n = d.n, tid = threadIdx.x;
    const int j0 = blockIdx.x * 32, i0 = blockIdx.y * kFinRows;
    if (j0 >= n || i0 >= n) return;
    const int *bst = reinterpret_cast<const int *>(d.v);
    const float *M = reinterpret_cast<const float *>(d.w) + (isQ ? (size_t)n * n : 0);
    const cplx<float> *ub = d.ubuf;
    cplx<float> *out = isQ ? d.Q : d.T;
    // rows of this CTA: whole blocks for T
    int ra = i0, rb = min(n, i0 + kFinRows);
    if (!isQ) {
        while (ra < n && bst[ra] != ra) ++ra;
        while (rb < n && bst[rb] != rb) ++rb;
    }
    if (ra >= rb) return;
    for (int c0 = j0; c0 < min(n, j0 + 32);) {
        if (bst[c0] != c0) { ++c0; continue; }
        int m = 1;
        while (m < kQrTiny && c0 + m < n && bst[c0 + m] == c0) ++m;
        // T: row blocks above this one; the diagonal block is done, zeros below
        const int rt = isQ ? rb : min(rb, c0), nr = max(0, rt - ra);
        __syncthreads();
        for (int e = tid; e < m * m; e += kFinThreads) uj[e] = ub[(c0 + e / m) * kQrTiny + e % m];  // U(q, c) at q m + c
        __syncthreads();
        for (int e = tid; e < nr * m; e += kFinThreads) {
            const int r = e % nr, c = e / nr;
            float yx = 0.0f, yy = 0.0f;
            for (int q = 0; q < m; ++q) {
                const float a = M[(ra + r) + (int64_t)(c0 + q) * n];
                const cplx<float> uv = uj[q * m + c];
                yx = fmaf(a, uv.x, yx);
                yy = fmaf(a, uv.y, yy);
            }
            if (isQ) out[(ra + r) + (int64_t)(c0 + c) * d.ld] = cplx<float>{yx, yy};
            else Y[r + c * (kFinRows + kQrTiny)] = cplx<float>{yx, yy};
        }
        if (!isQ) {
            __syncthreads();
            for (int e = tid; e < nr * m; e += kFinThreads) {
                const int r = e % nr, c = e / nr;
                const int b = bst[ra + r], a = ra + r - b;
                cplx<float> acc{0.0f, 0.0f};
                for (int q = b; q < n && q < b + kQrTiny && bst[q] == b; ++q)
                    cfma(acc, conj(ub[q * kQrTiny + a]), Y[(q - ra) + c * (kFinRows + kQrTiny)]);
                out[(ra + r) + (int64_t)(c0 + c) * d.ld] = acc;
            }
            const int z0 = max(ra, c0 + m);
            for (int e = tid; e < max(0, rb - z0) * m; e += kFinThreads) {
                const int r = e % (rb - z0), c = e / (rb - z0);
                out[(z0 + r) + (int64_t)(c0 + c) * d.ld] = cplx<float>{0.0f, 0.0f};
            }
        }
        c0 += m;
    }
}

// A matrix whose iteration did not finish within the round limit gets the
// iteration-cap status.
__global__ void rqr_mark_unfinished_kernel(const SchurDesc<float> *__restrict__ descs, int batch)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < batch; b += gridDim.x * blockDim.x)
        if (!descs[b].state[2]) atomicExch(descs[b].status, 3);
}

// largest matrix kept whole in shared memory: 224 columns of 225 + 4 floats
// and the two reflector tables, 213 KB
constexpr int kRqrResident = 224;
static_assert(resident_smem(kRqrResident) <= 220 * 1024, "resident matrix");

struct Deferred {
    int per, rv;
    size_t smem;
};
// vectors per CTA of the deferred passes: one matrix: about 128 CTAs per
// pass (the last round's passes overlap with no chase and should spread over
// many SMs); a batch: about 8 CTAs per SM over all matrices, since every CTA
// reads each window's U once, whatever its number of vectors
Deferred deferred_shape(int nmax, int batch)
{
    const int64_t n = std::max(nmax, 1);
    const size_t fixed = (size_t)(2 * RR * RR + 2 + n + 8) * sizeof(float);
    const size_t avail = 220 * 1024 > fixed ? 220 * 1024 - fixed : 0;
    const int64_t cap = std::min<int64_t>(32, (int64_t)(avail / (n * sizeof(float))));
    const int64_t want = batch > 1 ? cdiv_i(n * batch, 152 * 8) : cdiv_i(n, 128);
    int64_t per = std::max<int64_t>(1, std::min(want, cap));
    Deferred r;
    r.rv = cap >= 4 ? 4 : 1;
    if (r.rv == 4) per = std::min<int64_t>((per + 3) & ~(int64_t)3, cap & ~(int64_t)3);
    r.per = (int)per;
    r.smem = fixed + (size_t)r.per * n * sizeof(float);
    return r;
}

cudaError_t allow_rqr_smem()
{
    cudaError_t err;
    if ((err = allow_max_smem((const void *)rqr_chase_kernel<0>))) return err;
    if ((err = allow_max_smem((const void *)rqr_chase_kernel<1>))) return err;
    if ((err = allow_max_smem((const void *)rqr_chase_kernel<2>))) return err;
    if ((err = allow_max_smem((const void *)rqr_deferred_kernel<false, 1>))) return err;
    if ((err = allow_max_smem((const void *)rqr_deferred_kernel<false, 4>))) return err;
    if ((err = allow_max_smem((const void *)rqr_deferred_kernel<true, 1>))) return err;
    return allow_max_smem((const void *)rqr_deferred_kernel<true, 4>);
}

// window products and the two deferred passes of one round
cudaError_t enqueue_deferred(const SchurDesc<float> *dd, int batch, int nmax, int wins, cudaStream_t s)
{
    const Deferred f = deferred_shape(nmax, batch);
    const int ctas = (int)cdiv_i(nmax, f.per);
    rqr_build_u_kernel<<<dim3(wins, batch), kBuildThreads, kBuildSmem, s>>>(dd); count_launch();
    if (f.rv == 4) {
        rqr_deferred_kernel<false, 4><<<dim3(2 * ctas, batch), kDefThreads, f.smem, s>>>(dd, f.per, ctas); count_launch();
        rqr_deferred_kernel<true, 4><<<dim3(ctas, batch), kDefThreads, f.smem, s>>>(dd, f.per, ctas); count_launch();
    } else {
        rqr_deferred_kernel<false, 1><<<dim3(2 * ctas, batch), kDefThreads, f.smem, s>>>(dd, f.per, ctas); count_launch();
        rqr_deferred_kernel<true, 1><<<dim3(ctas, batch), kDefThreads, f.smem, s>>>(dd, f.per, ctas); count_launch();
    }
    return cudaGetLastError();
}

cudaError_t enqueue_begin(const SchurDesc<float> *dd, int batch, int nmax, cudaStream_t s)
{
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(batch > 1 ? 16 : 592, cdiv_i((int64_t)nmax * nmax, 1024)));
    rqr_begin_kernel<<<dim3(g, batch), 256, 0, s>>>(dd); count_launch();
    return cudaGetLastError();
}

cudaError_t enqueue_finish(const SchurDesc<float> *dd, int batch, int nmax, cudaStream_t s)
{
    rqr_blocks_kernel<<<dim3(std::min(nmax, batch > 1 ? 16 : 1024), batch), 32, 0, s>>>(dd); count_launch();
    for (int b0 = 0; b0 < batch; b0 += 16384) {  // (grid z is limited to 65535)
        const int bc = std::min(16384, batch - b0);
        rqr_finish_kernel<<<dim3((unsigned)cdiv_i(nmax, 32), (unsigned)cdiv_i(nmax, kFinRows), 2 * bc), kFinThreads, 0,
                            s>>>(dd + b0);
        count_launch();
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rqr_sweeps(const SchurDesc<float> *d_desc, int n, int *h_state, const int *d_state, cudaStream_t s,
                              float *ms_chase, const SchurDesc<float> *d_desc_alt, cudaStream_t side,
                              const cudaEvent_t *qev, int *d_sync, int helpers)
{
    cudaError_t err;
    if ((err = allow_rqr_smem())) return err;
    const bool resident = n <= kRqrResident;
    // cooperative chase (one chase CTA + H helper CTAs) for one large matrix
    const bool coop = !resident && d_sync != nullptr && helpers != 0;
    // a helper per 32 rows or columns (one group of four warps each), unless
    // the caller sets their number: with 8 (16 from n = 1024) the chase waited
    // for them, 20 k of a window's 45 k cycles at n = 512
    int H = helpers > 0 ? std::min(helpers, kMaxHelpers) : std::max(8, std::min(kMaxHelpers, n / 32));
    if ((err = enqueue_begin(d_desc, 1, n, s))) return err;
    bool all = false;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (ms_chase) {
        *ms_chase = 0.0f;
        if ((err = cudaEventCreate(&ev[0])) || (err = cudaEventCreate(&ev[1]))) return err;
    }
    // a resident round writes the whole matrix back, so its deferred passes
    // run before the next round instead of beside it
    const bool overlap = !resident && d_desc_alt && side && qev;
    bool used[2] = {false, false};
    // round r's deferred passes go to the side stream after round r + 1's chase
    // has been launched: the chase's CTAs, which have to be resident together,
    // then find their SMs free
    int pend = -1, pend_wins = 0;  // buffer set with deferred passes to launch
    auto flush = [&]() -> cudaError_t {
        if (pend < 0) return cudaSuccess;
        const SchurDesc<float> *dd = pend ? d_desc_alt : d_desc;
        const int par = pend;
        pend = -1;
        cudaError_t e;
        if (!overlap) return enqueue_deferred(dd, 1, n, pend_wins, s);
        if ((e = cudaStreamWaitEvent(side, qev[par], 0)) || (e = enqueue_deferred(dd, 1, n, pend_wins, side))) return e;
        used[par] = true;
        return cudaEventRecord(qev[2 + par], side);
    };
    for (int round = 0; round < 256 && !all; ++round) {
        const int par = overlap ? (round & 1) : 0;
        const SchurDesc<float> *dd = par ? d_desc_alt : d_desc;
        if (!overlap && (err = flush())) break;
        // this buffer set's deferred passes from two rounds ago must be done
        if (used[par] && (err = cudaStreamWaitEvent(s, qev[2 + par], 0))) break;
        if (ms_chase && (err = cudaEventRecord(ev[0], s))) break;
        if (coop) {
            if ((err = cudaMemsetAsync(d_sync, 0, (4 + H) * sizeof(int), s))) break;
            const SchurDesc<float> *arg0 = dd;
            int z = 0;
            void *args[4] = {(void *)&arg0, (void *)&H, (void *)&z, (void *)&z};
            if ((err = cudaLaunchCooperativeKernel((const void *)rqr_chase_kernel<1>, dim3(1 + H), dim3(kCta),
                                                   args, window_smem<1>(), s))) break;
        } else if (resident) {
            rqr_chase_kernel<2><<<1, kCta, resident_smem(n), s>>>(dd, 0, 0, n);
        } else {
            rqr_chase_kernel<0><<<1, kCta, window_smem<0>(), s>>>(dd, 0, 0, n);
        }
        count_launch();
        if (ms_chase && (err = cudaEventRecord(ev[1], s))) break;
        if (overlap && (err = cudaEventRecord(qev[par], s))) break;
        if ((err = cudaMemcpyAsync(h_state, d_state, sizeof(int) * kQrStateInts, cudaMemcpyDeviceToHost, s))) break;
        if (overlap && (err = flush())) break;
        if ((err = cudaStreamSynchronize(s))) break;
        if (ms_chase) {
            float ms = 0.0f;
            if ((err = cudaEventElapsedTime(&ms, ev[0], ev[1]))) break;
            *ms_chase += ms;
        }
        all = h_state[2] != 0;
        if (h_state[7] > 0) {
            pend = par;
            pend_wins = h_state[7];
        }
    }
    if (!err) err = flush();
    // every deferred pass finishes before T is read again
    for (int q = 0; q < 2; ++q)
        if (used[q]) {
            cudaError_t e2 = cudaStreamWaitEvent(s, qev[2 + q], 0);
            if (!err) err = e2;
        }
    if (ev[0]) cudaEventDestroy(ev[0]);
    if (ev[1]) cudaEventDestroy(ev[1]);
    if (err) return err;
    if (!all) { rqr_mark_unfinished_kernel<<<1, 32, 0, s>>>(d_desc, 1); count_launch(); }
    return enqueue_finish(d_desc, 1, n, s);
}

// Device-driven rounds for a batch: after each round a single CTA reads every
// matrix's done flag and sets the WHILE condition of the enclosing graph;
// after max_rounds rounds the unfinished matrices get status 3.
__global__ void rqr_round_decide_kernel(const SchurDesc<float> *__restrict__ descs, int batch, int *round,
                                        cudaGraphConditionalHandle cond, int max_rounds)
{
    __shared__ int s_open;
    if (threadIdx.x == 0) s_open = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < batch; b += blockDim.x)
        if (!descs[b].state[2]) atomicOr(&s_open, 1);
    __syncthreads();
    const int r = *round + 1;
    const bool more = s_open && r < max_rounds;
    if (s_open && !more)
        for (int b = threadIdx.x; b < batch; b += blockDim.x)
            if (!descs[b].state[2]) atomicExch(descs[b].status, 3);
    __syncthreads();
    if (threadIdx.x == 0) {
        *round = r;
        cudaGraphSetConditional(cond, more ? 1u : 0u);
    }
}

namespace {
struct RoundCtx {
    const SchurDesc<float> *desc;
    int batch, nmax, nmin, *round;
};

// size classes of the chase: a matrix up to 64 rows takes 27 KB of shared
// memory, up to 128 rows 75 KB, so that several share an SM
cudaError_t enqueue_round(void *p, cudaStream_t s, cudaGraphConditionalHandle cond)
{
    const RoundCtx *c = (const RoundCtx *)p;
    const int edge[4] = {0, 64, 128, kRqrResident};
    if (c->nmax > kRqrResident) {
        rqr_chase_kernel<0><<<c->batch, kCta, window_smem<0>(), s>>>(c->desc, 0, kRqrResident, INT32_MAX);
        count_launch();
    }
    for (int q = 2; q >= 0; --q) {
        if (c->nmax <= edge[q] || c->nmin > edge[q + 1]) continue;
        rqr_chase_kernel<2><<<c->batch, kCta, resident_smem(std::min(edge[q + 1], c->nmax)), s>>>(c->desc, 0, edge[q],
                                                                                               edge[q + 1]);
        count_launch();
    }
    cudaError_t err;
    // windows of a round: at most the window capacity of the largest matrix
    const int ubx = (int)std::min<int64_t>(qr_win_capacity(c->nmax), 64);
    if ((err = enqueue_deferred(c->desc, c->batch, c->nmax, ubx, s))) return err;
    rqr_round_decide_kernel<<<1, 256, 0, s>>>(c->desc, c->batch, c->round, cond, 256); count_launch();
    return cudaGetLastError();
}
}  // namespace

cudaError_t enqueue_rqr_sweeps_device(const SchurDesc<float> *d_desc, int batch, int nmax, int nmin, int *d_round,
                                      cudaStream_t s, cudaStream_t body_stream)
{
    if (batch <= 0) return cudaSuccess;
    cudaError_t err;
    if ((err = allow_rqr_smem())) return err;
    if ((err = enqueue_begin(d_desc, batch, nmax, s))) return err;
    if ((err = cudaMemsetAsync(d_round, 0, sizeof(int), s))) return err;
    RoundCtx ctx{d_desc, batch, nmax, nmin, d_round};
    if ((err = capture_while(s, body_stream, 1u, enqueue_round, &ctx))) return err;
    return enqueue_finish(d_desc, batch, nmax, s);
}

}  // namespace sqm
