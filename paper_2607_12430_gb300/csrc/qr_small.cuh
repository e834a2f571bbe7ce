// qr_small.cuh -- warp- and CTA-level pieces shared by the complex (qr.cu)
// and the real (rqr.cu) QR iterations: complex Givens rotations, single-shift
// sweeps and complete Schur forms of small blocks by one warp, and the
// starting estimates of the shift iteration.
#pragma once

#include "internal.h"

namespace sqm {

static constexpr int kItMax = 60;        // sweeps per eigenvalue
static constexpr int kQrTiny = 24;       // active blocks up to this size: one warp, dense U
static constexpr int kQrTinyLd = 33;     // leading dimension of its shared-memory block and U
static constexpr int kAberthIt = 24;     // iteration limit of the simultaneous shift refinement

// Complex Givens G = [c s; -conj(s) c] with c real and G [x; y] = [r; 0].
// c^2 + |s|^2 = 1 to rounding only if the phase x / |x| has modulus 1, and a
// subnormal |x| has too few bits for that (c^2 + |s|^2 came out between 0.89 and
// 1.04 where a shift met an eigenvalue exactly), so a small x is scaled up
// for the phase, and both where y is small too.
template <class R>
__device__ __forceinline__ void givens(cplx<R> x, cplx<R> y, R &c, cplx<R> &s, cplx<R> &r)
{
    const R up = R(1.2676506002282294e30);  // 2^100
    const R low = sizeof(R) == 4 ? R(1e-28) : R(1e-280);
    R ax = hypot(x.x, x.y), ay = hypot(y.x, y.y);
    if (ay == R(0)) { c = 1; s = {0, 0}; r = x; return; }
    const cplx<R> yu = up * y;
    if (ax == R(0)) {
        r = {ay, 0};
        if (ay < low) { y = yu; ay = hypot(y.x, y.y); }
        c = 0;
        s = {y.x / ay, -y.y / ay};
        return;
    }
    cplx<R> ph{x.x / ax, x.y / ax};
    R back = R(1);
    if (ax < low) {
        const cplx<R> xu = up * x;
        const R au = hypot(xu.x, xu.y);
        ph = cplx<R>{xu.x / au, xu.y / au};
        if (ay < low) { ax = au; y = yu; ay = hypot(y.x, y.y); back = R(1) / up; }
    }
    R nrm = hypot(ax, ay);
    c = ax / nrm;
    cplx<R> cy = conj(y);
    s = cplx<R>{(ph.x * cy.x - ph.y * cy.y) / nrm, (ph.x * cy.y + ph.y * cy.x) / nrm};
    r = (back * nrm) * ph;
}

// Eigenvalue of [a b; c d] closer to d, written without cancellation:
// d + h -/+ disc = d - bc / (h +/- disc), h = (a - d)/2, disc = sqrt(h^2 + bc).
template <class R>
__device__ cplx<R> wilkinson(cplx<R> a, cplx<R> b, cplx<R> c, cplx<R> d)
{
    cplx<R> h = R(0.5) * (a - d);
    cplx<R> bc = b * c;
    cplx<R> disc = csqrt_(h * h + bc);
    cplx<R> p1 = h + disc, p2 = h - disc;
    bool ok1 = abs2(p1) > R(0), ok2 = abs2(p2) > R(0);
    cplx<R> m1 = ok1 ? d - cdiv(bc, p1) : d;
    cplx<R> m2 = ok2 ? d - cdiv(bc, p2) : d;
    ok1 = ok1 && isfinite(m1.x) && isfinite(m1.y);
    ok2 = ok2 && isfinite(m2.x) && isfinite(m2.y);
    if (ok1 && (!ok2 || abs2(m1 - d) <= abs2(m2 - d))) return m1;
    if (ok2) return m2;
    return d;
}

// The same rotation for FP32 from |x|^2 and |y|^2 and two reciprocal square
// roots, each refined by one Newton step written with fused multiply-adds:
// e = 1 - v y0^2 (one rounding), y1 = y0 + (y0 / 2) e (one rounding).  The
// refinement squares away the systematic part of the hardware reciprocal
// square root's error, which would otherwise accumulate over the thousands
// of rotations applied to each Schur vector (an unrefined form measured ten
// times worse orthogonality); the remaining error is rounding of either
// sign, as with correctly rounded square roots and divisions, at a fraction
// of their latency on the chase's critical path.  Tiny or huge arguments
// take the scaled path.
__device__ __forceinline__ float rsqrt_refined(float v)
{
    const float y0 = rsqrtf(v);
    const float e = fmaf(-(v * y0), y0, 1.0f);
    return fmaf(0.5f * y0, e, y0);
}
template <class R>
__device__ __forceinline__ void givens_fast(cplx<R> x, cplx<R> y, R &c, cplx<R> &s, cplx<R> &r)
{
    givens(x, y, c, s, r);
}
template <>
__device__ __forceinline__ void givens_fast<float>(cplx<float> x, cplx<float> y, float &c, cplx<float> &s,
                                                   cplx<float> &r)
{
    const float ax2 = fmaf(x.x, x.x, x.y * x.y), ay2 = fmaf(y.x, y.x, y.y * y.y);
    const float nrm2 = ax2 + ay2;
    if (!(ax2 >= 1e-30f) || !(nrm2 <= 1e30f)) {
        givens(x, y, c, s, r);
        return;
    }
    const float inv = rsqrt_refined(nrm2), invx = rsqrt_refined(ax2);
    const float f = invx * inv;  // 1 / (|x| ||(x, y)||)
    c = ax2 * f;
    s = cplx<float>{(x.x * y.x + x.y * y.y) * f, (x.y * y.x - x.x * y.y) * f};  // x conj(y) f
    const float gsc = nrm2 * f;                                                // ||(x, y)|| / |x|
    r = cplx<float>{x.x * gsc, x.y * gsc};
}

// Cheaper rotation for the shift computation only (eigenvalue estimates,
// never applied to T or Z): reciprocal square roots instead of correctly
// rounded square roots and divisions.
template <class R>
__device__ __forceinline__ void givens_approx(cplx<R> x, cplx<R> y, R &c, cplx<R> &s, cplx<R> &r)
{
    givens(x, y, c, s, r);
}
template <>
__device__ __forceinline__ void givens_approx<float>(cplx<float> x, cplx<float> y, float &c, cplx<float> &s,
                                                     cplx<float> &r)
{
    const float ax2 = fmaf(x.x, x.x, x.y * x.y), ay2 = fmaf(y.x, y.x, y.y * y.y);
    const float nrm2 = ax2 + ay2;
    if (!(ax2 >= 1e-30f) || !(nrm2 <= 1e30f)) {
        givens(x, y, c, s, r);
        return;
    }
    const float inv = rsqrtf(nrm2), invx = rsqrtf(ax2);
    const float f = invx * inv;
    c = ax2 * f;
    s = cplx<float>{(x.x * y.x + x.y * y.y) * f, (x.y * y.x - x.x * y.y) * f};
    const float gsc = nrm2 * f;
    r = cplx<float>{x.x * gsc, x.y * gsc};
}

// Eigenvalues of a small upper Hessenberg matrix M (nb x nb, nb <= 32,
// column-major, leading dimension LDM) by single-shift QR without vectors,
// one warp: lane j updates column j of a row rotation and row j of a column
// rotation.  Only the active block is updated.  M is destroyed; out[0..nb-1]
// receives the eigenvalues.
template <class R>
__device__ __forceinline__ cplx<R> shfl_c(cplx<R> v, int src)
{
    return cplx<R>{__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src)};
}

// One implicit single-shift sweep on rows / columns lo .. hi of the small
// Hessenberg matrix M (ld LDM, one warp, lane j = column j in the row half
// and row j in the column half of each rotation), optionally accumulating
// the rotations into U (U <- U G^H).  The shared-memory copy is kept up to
// date, but the entries the next step needs -- its rotation's x and y, the
// 2 x 2 block where the row and column halves overlap, the next pair of rows
// -- travel between lanes by shuffles from the lanes that computed them, so
// a rotation costs no shared-memory round trip on the critical path.  The
// arithmetic (and hence every value) is that of the plain two-phase sweep.
template <class R, int LDM, bool ACC, bool APPROX>
__device__ __forceinline__ void warp_sweep(cplx<R> *M, cplx<R> *U, int m, int lo, int hi, cplx<R> mu, int *nrot)
{
    const int lane = threadIdx.x & 31;
    const int ccols = ACC ? m : hi + 1;  // the row half runs to this column (exclusive)
    // row half of rotation k: lane j >= js holds p = M(k, j), q = M(k+1, j)
    cplx<R> p{0, 0}, q{0, 0};
    if (lane >= lo && lane < ccols) {
        p = M[lo + lane * LDM];
        q = M[(lo + 1) + lane * LDM];
    }
    cplx<R> x = shfl_c(p, lo), y = shfl_c(q, lo);
    x = x - mu;
    for (int k = lo; k < hi; ++k) {
        const int js = (k == lo) ? k : k - 1;
        // row k+2 of the columns right of k+1 is untouched until rotation k+1
        cplx<R> nxt{0, 0};
        if (k + 2 <= hi && lane >= k + 2 && lane < ccols) nxt = M[(k + 2) + lane * LDM];
        const cplx<R> sub2 = (k + 2 <= hi) ? M[(k + 2) + (k + 1) * LDM] : cplx<R>{0, 0};
        R c;
        cplx<R> s, r;
        if (APPROX) givens_approx(x, y, c, s, r);
        else givens_fast(x, y, c, s, r);
        const bool lj = lane >= js && lane < ccols;
        cplx<R> np = c * p + s * q, nq = c * q - conj(s) * p;
        if (lane == js && k > lo) {
            np = r;
            nq = cplx<R>{0, 0};
        }
        if (lj) {
            M[k + lane * LDM] = np;
            M[(k + 1) + lane * LDM] = nq;
        }
        // column half: rows lo .. min(k+2, hi) of columns k, k+1
        const cplx<R> np_k1 = shfl_c(np, k + 1), nq_k = shfl_c(nq, k);
        const int rmax = min(k + 2, hi);
        cplx<R> pp{0, 0}, qq{0, 0};
        if (lane == k) {
            pp = np;
            qq = np_k1;
        } else if (lane == k + 1) {
            pp = nq_k;
            qq = nq;
        } else if (lane == k + 2) {
            pp = cplx<R>{0, 0};
            qq = sub2;
        } else if (lane >= (ACC ? 0 : lo) && lane < k) {
            pp = M[lane + k * LDM];
            qq = M[lane + (k + 1) * LDM];
        }
        const cplx<R> npp = c * pp + conj(s) * qq, nqq = c * qq - s * pp;
        __syncwarp();  // the row half's stores land before the column half's
        if (lane >= (ACC ? 0 : lo) && lane <= rmax) {
            M[lane + k * LDM] = npp;
            M[lane + (k + 1) * LDM] = nqq;
        }
        if (ACC && lane < m) {
            const cplx<R> up = U[lane + k * LDM], uq = U[lane + (k + 1) * LDM];
            U[lane + k * LDM] = c * up + conj(s) * uq;
            U[lane + (k + 1) * LDM] = c * uq - s * up;
        }
        // the next rotation: x = M(k+1, k), y = M(k+2, k) as the column half
        // left them; rows k+1, k+2 of columns k, k+1 from the column half
        const cplx<R> a1 = shfl_c(npp, k + 1), b1 = shfl_c(nqq, k + 1);
        const cplx<R> a2 = shfl_c(npp, k + 2), b2 = shfl_c(nqq, k + 2);
        x = a1;
        y = (k + 2 <= hi) ? a2 : cplx<R>{0, 0};
        if (lane == k) {
            p = a1;
            q = a2;
        } else if (lane == k + 1) {
            p = b1;
            q = b2;
        } else {
            p = nq;
            q = nxt;
        }
        __syncwarp();
        if (nrot) ++*nrot;
    }
}

// Eigenvalues of a small upper Hessenberg matrix M (nb x nb, nb <= 32,
// column-major, leading dimension LDM) by single-shift QR without vectors,
// one warp (warp_sweep).  Only the active block is updated.  M is
// destroyed; out[0..nb-1] receives the eigenvalues.
template <class R, int LDM>
__device__ void warp_small_eigvals(cplx<R> *M, int nb, cplx<R> *out)
{
    const int lane = threadIdx.x & 31;
    const R eps = num<R>::eps;
    int hi = nb - 1, it = 0;
    while (hi > 0) {
        bool small = false;
        if (lane >= 1 && lane <= hi) {
            const cplx<R> sub = M[lane + (lane - 1) * LDM];
            const R as = hypot(sub.x, sub.y);
            const cplx<R> a = M[lane + lane * LDM], b = M[(lane - 1) + (lane - 1) * LDM];
            small = as == R(0) || as <= eps * (hypot(a.x, a.y) + hypot(b.x, b.y));
        }
        const unsigned bal = __ballot_sync(0xffffffffu, small);
        const int lo = bal ? 31 - __clz(bal) : 0;
        if (lo == hi) {
            if (lane == 0) out[hi] = M[hi + hi * LDM];
            --hi;
            it = 0;
            __syncwarp();
            continue;
        }
        if (++it > 40) {  // give up: the diagonal of the unreduced block
            for (int i = lo + lane; i <= hi; i += 32) out[i] = M[i + i * LDM];
            hi = lo - 1;
            it = 0;
            __syncwarp();
            continue;
        }
        const cplx<R> mu = wilkinson(M[(hi - 1) + (hi - 1) * LDM], M[(hi - 1) + hi * LDM],
                                     M[hi + (hi - 1) * LDM], M[hi + hi * LDM]);
        __syncwarp();
        warp_sweep<R, LDM, false, true>(M, nullptr, nb, lo, hi, mu, nullptr);
    }
    if (hi == 0 && lane == 0) out[0] = M[0];
    __syncwarp();
}

// Shifts by simultaneous refinement of all nb eigenvalue estimates of the
// small unreduced Hessenberg block M (nb x nb, nb <= 32, leading dimension
// LDM): the Ehrlich-Aberth iteration (O. Aberth, Math. Comp. 27 (1973)),
//   z_j <- z_j - N_j / (1 - N_j sum_{k != j} 1 / (z_j - z_k)),
// with every estimate updated at once, where N_j = p(z_j) / p'(z_j) and
// p(z) = det(M - z I).  The Newton ratio comes from Hyman's recurrence
// (Wilkinson, The Algebraic Eigenvalue Problem, 1965, Ch. 7): with
// x_{nb-1} = 1, row i of (M - z I) x = 0 fixes x_{i-1} through the
// subdiagonal entry M(i, i-1), for i = nb-1 down to 1; the residual of row 0
// is then p(z) times a product of subdiagonal entries that does not depend
// on z, so differentiating the recurrence gives the same multiple of p'(z)
// and the ratio of the two is N.  A segment of lanes per estimate (16 while
// nb <= 16, so a warp takes two): lane r keeps the running sums of row r for
// the residual and its derivative, and each new x_i (formed by lane i) is
// broadcast and added into the rows above it.  x, its derivative and the
// sums are rescaled together by powers of two to stay in range, which
// leaves the ratio unchanged.  No CTA-wide state other than z changes; M is
// not modified.  On entry z (shared memory) holds nb distinct starting
// estimates; true means every correction of the last
// iteration was at most tol (|z_j| + 1e-3 max|M_ij|) and z holds the
// shifts; false (no convergence within kmax iterations, or a non-finite
// value) leaves z unusable.  Every thread of the CTA calls it.
template <class R> __device__ __forceinline__ R aberth_tol();
template <> __device__ __forceinline__ float aberth_tol<float>() { return 1e-6f; }
template <> __device__ __forceinline__ double aberth_tol<double>() { return 1e-11; }

template <class R, int LDM>
__device__ bool cta_aberth_shifts(const cplx<R> *M, int nb, cplx<R> *z, R mnrm, int kmax)
{
    __shared__ cplx<R> s_inv[32], s_w[32];
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = (int)(blockDim.x >> 5);
    // seg lanes per estimate (a half-warp while nb <= 16, so a warp takes two)
    const int seg = nb <= 16 ? 16 : 32, per = 32 / seg, r = lane % seg, half = lane / seg;
    const R tol = aberth_tol<R>();
    const R floor_sub = mnrm * R(1e-20);
    if (tid < nb) {  // 1 / M(i, i-1) for i = tid >= 1; a vanishing entry is raised to floor_sub
        cplx<R> sb = tid ? M[tid + (tid - 1) * LDM] : cplx<R>{R(1), R(0)};
        if (!(fmax(fabs(sb.x), fabs(sb.y)) > floor_sub)) sb = cplx<R>{floor_sub, R(0)};
        s_inv[tid] = cdiv(cplx<R>{R(1), R(0)}, sb);
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int it = 0; it < kmax; ++it) {
        // every lane of a warp runs the same trip counts (the shuffles span the
        // warp); a segment past nb computes on a copy of estimate nb - 1 and
        // stores nothing
        for (int j0 = warp * per; j0 < nb; j0 += nw * per) {
            const int j = j0 + half;
            const cplx<R> mu = z[min(j, nb - 1)];
            cplx<R> s{0, 0}, ds{0, 0}, x{R(1), R(0)}, dx{0, 0};
#pragma unroll 2
            for (int i = nb - 1;; --i) {
                if (r <= i) {  // column i of (M - mu I) into rows 0 .. i
                    cplx<R> a = M[r + i * LDM];
                    if (r == i) a = a - mu;
                    cfma(ds, a, dx);
                    if (r == i) ds = ds - x;
                    cfma(s, a, x);
                }
                if (i == 0) break;
                const cplx<R> iv = s_inv[i];
                const cplx<R> xn = -(s * iv), dxn = -(ds * iv);  // meaningful on lane i of the segment
                x = cplx<R>{__shfl_sync(0xffffffffu, xn.x, i, seg), __shfl_sync(0xffffffffu, xn.y, i, seg)};
                dx = cplx<R>{__shfl_sync(0xffffffffu, dxn.x, i, seg), __shfl_sync(0xffffffffu, dxn.y, i, seg)};
                const R mag = fmax(fmax(fabs(x.x), fabs(x.y)), fmax(fabs(dx.x), fabs(dx.y)));
                const R f = mag > R(1099511627776.0) ? R(1.0 / 1099511627776.0)  // 2^40
                            : (mag > R(0) && mag < R(1.0 / 1099511627776.0)) ? R(1099511627776.0) : R(1);
                x = f * x; dx = f * dx; s = f * s; ds = f * ds;
            }
            const cplx<R> q = cdiv(s, ds);  // row 0 (lane 0 of the segment): p / p'
            const cplx<R> N{__shfl_sync(0xffffffffu, q.x, 0, seg), __shfl_sync(0xffffffffu, q.y, 0, seg)};
            cplx<R> part{0, 0};
            if (r < nb && r != j) part = cdiv(cplx<R>{R(1), R(0)}, mu - z[r]);
            for (int o = seg >> 1; o > 0; o >>= 1) {
                part.x += __shfl_xor_sync(0xffffffffu, part.x, o);
                part.y += __shfl_xor_sync(0xffffffffu, part.y, o);
            }
            const cplx<R> w = cdiv(N, cplx<R>{R(1), R(0)} - N * part);
            if (r == 0 && j < nb) s_w[j] = w;
        }
        __syncthreads();
        bool done = true;
        if (tid < nb) {
            const cplx<R> w = s_w[tid];
            const cplx<R> zn = z[tid] - w;
            if (!(isfinite(zn.x) && isfinite(zn.y))) s_bad = 1;
            done = hypot(w.x, w.y) <= tol * (hypot(zn.x, zn.y) + R(1e-3) * mnrm);
            z[tid] = zn;
        }
        const int all = __syncthreads_and(done);
        if (s_bad) return false;
        if (all) return true;
    }
    return false;
}

// Starting estimates for cta_aberth_shifts (one warp; lane q holds the
// q-th previous shift).  Warm start: the np shifts of the previous
// multishift sweep, whose trailing block ended dh rows lower (0 <= dh < nb);
// for each of the dh eigenvalues deflated since (defl) the nearest previous
// shift is dropped, then while more than nb remain the one farthest from
// every diagonal entry of M; the remaining places take diagonal entries of
// M moved apart by multiples of 1e-4 mnrm.  Cold start (np = 0): the
// diagonal of M moved by 1e-3 mnrm along the nb-th roots of unity.
template <class R>
__device__ __forceinline__ void warp_argbest(R &d, int &l, bool want_min)
{
    for (int o = 16; o > 0; o >>= 1) {
        const R od = __shfl_xor_sync(0xffffffffu, d, o);
        const int ol = __shfl_xor_sync(0xffffffffu, l, o);
        if ((want_min ? od < d : od > d) || (od == d && ol < l)) { d = od; l = ol; }
    }
}
template <class R, int LDM>
__device__ void warp_aberth_start(const cplx<R> *M, int nb, R mnrm, const cplx<R> *prev, int np, const cplx<R> *defl,
                                  int dh, cplx<R> *z)
{
    const int lane = threadIdx.x & 31;
    const cplx<R> c = lane < np ? prev[lane] : cplx<R>{0, 0};
    bool alive = lane < np;
    for (int q = 0; q < dh; ++q) {
        R d = alive ? abs2(c - defl[q]) : R(INFINITY);
        int l = lane;
        warp_argbest(d, l, true);
        if (d < R(INFINITY) && lane == l) alive = false;
    }
    int cnt = __popc(__ballot_sync(0xffffffffu, alive));
    while (cnt > nb) {
        R d = R(-1);
        if (alive) {
            d = abs2(c - M[0]);
            for (int i = 1; i < nb; ++i) d = fmin(d, abs2(c - M[i + i * LDM]));
        }
        int l = lane;
        warp_argbest(d, l, false);
        if (lane == l) alive = false;
        --cnt;
    }
    const unsigned am = __ballot_sync(0xffffffffu, alive);
    if (alive) z[__popc(am & ((1u << lane) - 1u))] = c;
    const int q = lane - cnt;  // places cnt .. nb-1
    if (q >= 0 && lane < nb) {
        const cplx<R> d = M[q + q * LDM];
        if (np > 0) {
            z[lane] = cplx<R>{d.x + R(q + 1) * R(1e-4) * mnrm, d.y};
        } else {
            R sn, cs;
            sincospi(R(2 * q) / R(nb), &sn, &cs);
            z[lane] = cplx<R>{d.x + R(1e-3) * mnrm * cs, d.y + R(1e-3) * mnrm * sn};
        }
    }
    __syncwarp();
}

// Complete Schur form of a small active block (m <= 32), one warp: single-
// shift QR with Wilkinson shifts (an exceptional shift every 10 sweeps
// without deflation) on the m x m block M in shared memory (leading
// dimension LDM), every rotation applied to the whole block (rows k, k+1
// from column k-1 on; columns k, k+1 down to row k+2) and accumulated into
// U (U <- U G^H, U = I on entry), until every subdiagonal entry is
// negligible (set to zero).  Then the rest of T needs only x <- x U (rows
// above the block, Schur vectors) and y <- U^H y (columns right of it).
// Returns false if some eigenvalue took more than kItMax sweeps.
template <class R, int LDM>
__device__ bool warp_tiny_schur(cplx<R> *M, cplx<R> *U, int m, int *sweeps, int *rots, const cplx<R> *cand = nullptr,
                                int ncand = 0)
{
    const int lane = threadIdx.x & 31;
    const R eps = num<R>::eps;
    int hi = m - 1, it = 0, nsw = 0, nrot = 0;
    bool ok = true;
    while (hi > 0) {
        bool small = false;
        if (lane >= 1 && lane <= hi) {
            const cplx<R> sub = M[lane + (lane - 1) * LDM];
            const R as = hypot(sub.x, sub.y);
            const cplx<R> a = M[lane + lane * LDM], b = M[(lane - 1) + (lane - 1) * LDM];
            small = as == R(0) || as <= eps * (hypot(a.x, a.y) + hypot(b.x, b.y));
        }
        const unsigned bal = __ballot_sync(0xffffffffu, small);
        const int lo = bal ? 31 - __clz(bal) : 0;
        __syncwarp();
        if (lo == hi) {
            if (lane == 0) M[hi + (hi - 1) * LDM] = cplx<R>{0, 0};
            --hi;
            it = 0;
            __syncwarp();
            continue;
        }
        if (lo > 0 && lane == 0) M[lo + (lo - 1) * LDM] = cplx<R>{0, 0};
        if (++it > kItMax) { ok = false; break; }
        ++nsw;
        cplx<R> mu;
        if (it % 10 == 0) {
            const cplx<R> sb = M[hi + (hi - 1) * LDM];
            mu = M[hi + hi * LDM];
            mu.x += R(0.75) * hypot(sb.x, sb.y);
        } else {
            mu = wilkinson(M[(hi - 1) + (hi - 1) * LDM], M[(hi - 1) + hi * LDM], M[hi + (hi - 1) * LDM],
                           M[hi + hi * LDM]);
            if (it == 1 && ncand > 0) {
                // first sweep on this bottom entry: the nearest of the given
                // estimates (shifts of the sweep that split this block off,
                // eigenvalue estimates of the whole matrix) replaces the
                // Wilkinson shift when both point at the same eigenvalue
                R db = R(INFINITY);
                cplx<R> zb = mu;
                for (int q = 0; q < ncand; ++q) {
                    const R dq = abs2(cand[q] - mu);
                    if (dq < db) { db = dq; zb = cand[q]; }
                }
                if (db <= R(1e-4) * abs2(mu)) mu = zb;
            }
        }
        __syncwarp();
        warp_sweep<R, LDM, true, false>(M, U, m, lo, hi, mu, &nrot);
    }
    *sweeps = nsw;
    *rots = nrot;
    return ok;
}

}  // namespace sqm
