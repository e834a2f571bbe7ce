// xsplit.cu -- the FP64 residual R = (A - X Y) 2^-s of small and middling
// matrices, one, a batch or one complex one (Y = X, or X X for the cube root),
// the product from exact digit products on the BF16
// tensor cores (the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// Numer. Algorithms 59 (2012)), with the digits formed in the kernel.
//
// Row i of X is scaled by 2^-rho_i and column j of Y by 2^-sig_j (the smallest
// powers of two above their largest magnitudes) and every entry rounded to a
// 62-bit fixed-point integer, cut into 8 balanced base-256 digits by adding
// 128 to every byte and reading the bytes:
//   x = 2^(rho - 6) sum_s m_s 2^(-8 s),  |m_0| <= 64, -128 <= m_s <= 127,
// every digit exact in BF16.  The products of digits s and t carry 2^(-8 (s +
// t)); the eight sums over s + t = d, d = 0 .. 7, each have a TMEM accumulator:
//   A_d = sum_k sum_{s+t=d} m_s(i, k) m_t(k, j),
// an integer of at most 2 2^13 + 6 2^14 = 7 2^14 a term (d = 7, the largest),
// below 2^24 for 128 terms in k, so the FP32 accumulation is exact; every 128
// terms the accumulators are drained into two 64-bit integers an entry, hi for
// d < 4 and lo for the others.  Left out are the pairs with s + t > 7, below n 2^(rho +
// sig - 59) in sum, and the rounding to 62 bits, below n 2^(rho + sig - 62):
// the FP64 product's own error bound is n 2^-53 sum |x| |y|.  The two integers
// then leave A in two fused multiply-adds, so that the cancellation in A - X Y
// rounds once, where an FP64 product rounds at every term.
//
// One CTA per 128 x 64 tile of R; for each 64 terms in k its 16 warps form the
// digit tiles (8 x 16 KB of X, 8 x 8 KB of Y, 128-byte swizzle) in shared
// memory, one thread issues 36 x 4 tcgen05.mma (M = 128, N = 64, K = 16), and
// the next 64 terms are split when those are done.  TMEM: 8 accumulators of 64
// columns, all 512; the 192 KB of digits keep it to one CTA an SM.
//
// The error above is relative to the largest entry of a row of X and of a
// column of Y, the FP64 product's to the entries that meet.  It is of the order
// of sqrt(n) 2^-62 ||2^rho|| ||2^sig|| (the digits left out are as good as
// random), the FP64 product's about 0.3 sqrt(n) 2^-53 ||A|| where X X is near A:
// measured on Gaussian and uniform X, n = 16 .. 511, 4.6e-18 .. 1.8e-16 of ||A||
// against 1.4e-16 .. 7.9e-16.  A tile takes the digit products where
//   ||2^rho|| ||2^sig|| <= 128 ||A|| / sqrt(number of tiles)
// over its own rows and columns, so that their error stays below the FP64
// product's, and FP64 products where not (graded or far from normal X, entries
// that are not finite) and for n <= 32, where there is less to do than the
// digits cost.  FP64 products are bound by an SM's FP64 units (2 multiply-adds a
// cycle), and 128 x 64 tiles leave most SMs idle, so where they do the launch has
// up to 4 CTAs a tile, each for its own columns; those beyond the first leave
// after the test where the tile takes the digits.
//
// A complex product is two real ones with 2 n terms each, the imaginary parts of
// a row after its real ones: Re = [Xr, -Xi] [Yr; Yi], Im = [Xr, Xi] [Yi; Yr].
//
// A tile of a matrix of n = 256 takes about 150 k cycles: 51 k to form the
// digits, 52 k in the products (89 cycles each; an M = 128, N = 64 product reads
// 6 KB of shared memory), 33 k in the FP64 units at the end, the rest in the
// exponents and drains; FP64 products take 128 x 64 x 256 / 2 = 1.05 M.  The
// residual alone, us with its host call (about 50): n = 101 90 / 158, 256 127 /
// 316, 512 182 / 600 against FP64 products; against tc_split.cu's kernels 512
// 182 / 313, 800 253 / 416, 1024 305 / 461 (1025).  Three residuals of a batch of
// 2048 matrices of 16 to 256 rows: 13 ms, 60 with FP64 products.
// Refinement of a complex matrix with these and with FP64 products, ms: n = 40
// 0.48 / 0.95, 101 1.04 / 2.17, 301 2.95 / 6.07; cube root (one of its two
// products) n = 200 3.76 / 4.26.
#include <cuda_bf16.h>

#include "internal.h"
#include "tc_common.cuh"

namespace sqm {

namespace {

constexpr int XM = 128, XN = 64, XK = 64, XS = 8, XT = 512;
constexpr int XA_BYTES = XM * XK * 2, XB_BYTES = XN * XK * 2;  // one digit's tile
constexpr int X_SMEM = XS * (XA_BYTES + XB_BYTES) + 1024;

// instruction descriptor: D = F32, A = B = BF16, both K-major, M = 128, N = 64
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);

struct XArgs {
    const double *A, *X, *Y;
    int64_t lda, ldx, ldy;
    float *Rhat;
    int ldr;
    double *partials;
    double sc;
    double norm_a;  // ||A||_F: decides between the digit and the FP64 product
    int n;
    int slices;     // CTAs per tile
};

// the scaling exponent from the largest high word of |x|: 2^r > |x| for every
// finite x of the row; kNonFinite where an entry is an infinity or a NaN
constexpr int kNonFinite = 1 << 20;
__device__ __forceinline__ int scale_exp(unsigned hi)
{
    const int ef = (int)(hi >> 20);
    return ef == 0x7FF ? kNonFinite : (ef > 0 ? ef : 1) - 1022;
}

// round(x 2^(62 - r)) for |x| < 2^r, plus 128 in every byte
__device__ __forceinline__ unsigned long long biased_fixed(double x, int r)
{
    const long long vb = __double_as_longlong(x);
    const int ef = (int)((vb >> 52) & 0x7FF);
    const unsigned long long mant = (vb & 0x000FFFFFFFFFFFFFull) | (ef ? (1ull << 52) : 0ull);
    // 1 .. (0 or less: an infinity or NaN, whose tile does not come here)
    const int right = r + 1075 - 62 + 10 - (ef ? ef : 1);
    unsigned long long f = ((mant << 10) + (1ull << ((right - 1) & 63))) >> (right & 63);
    if (right > 63) f = 0;
    const unsigned long long sg = (unsigned long long)(vb >> 63);
    return (f ^ sg) - sg + 0x8080808080808080ull;
}

// byte j of two biased integers' words as a pair of BF16 digits: with u = m +
// 128 = 128 h + l, m = (128 + l) - (256 - 128 h); both terms and m are exact
template <int j>
__device__ __forceinline__ uint32_t digit_pair(uint32_t a, uint32_t b)
{
    const uint32_t p = __byte_perm(a, b, j | (j << 4) | ((4 + j) << 8) | ((4 + j) << 12));
    const uint32_t lo = (p & 0x007F007Fu) | 0x43004300u, hi = (p & 0x00800080u) ^ 0x43804380u;
    __nv_bfloat162 x, y;
    memcpy(&x, &lo, 4);
    memcpy(&y, &hi, 4);
    x = __hsub2(x, y);
    uint32_t r;
    memcpy(&r, &x, 4);
    return r;
}

// digit 7 - byte of 8 consecutive k to its 16-byte chunk of every digit's tile
template <int j>
__device__ __forceinline__ void store_digit(unsigned char *dst, int digit_stride, const unsigned long long (&g)[8])
{
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned long long a = g[2 * q], b = g[2 * q + 1];
        w[q] = j < 4 ? digit_pair<(j & 3)>((uint32_t)a, (uint32_t)b)
                     : digit_pair<(j & 3)>((uint32_t)(a >> 32), (uint32_t)(b >> 32));
    }
    *reinterpret_cast<uint4 *>(dst + (7 - j) * digit_stride) = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void store_digits(unsigned char *dst, int digit_stride, const double (&x)[8], int r)
{
    unsigned long long g[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) g[q] = biased_fixed(x[q], r);
    store_digit<0>(dst, digit_stride, g);
    store_digit<1>(dst, digit_stride, g);
    store_digit<2>(dst, digit_stride, g);
    store_digit<3>(dst, digit_stride, g);
    store_digit<4>(dst, digit_stride, g);
    store_digit<5>(dst, digit_stride, g);
    store_digit<6>(dst, digit_stride, g);
    store_digit<7>(dst, digit_stride, g);
}

// 16 columns of two accumulators (warp-collective)
__device__ __forceinline__ void tmem_ld16x2(uint32_t t0, uint32_t t1, uint32_t (&a)[16], uint32_t (&b)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15},"
        " [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29,"
        " %30, %31}, [%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]),
          "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(b[0]),
          "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]),
          "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15])
        : "r"(t0), "r"(t1)
        : "memory");
}

// old - v 2^e; the power of two is exact, so this rounds once
__device__ __forceinline__ double sub_scaled(double old, long long v, int e)
{
    if (e >= -1022 && e <= 1023) return fma(-__ll2double_rn(v), __longlong_as_double((long long)(e + 1023) << 52), old);
    return old - ldexp(__ll2double_rn(v), e);
}

// whether the digit products of a tile are as accurate as FP64 ones (see the
// head of the file); one warp, every lane gets the answer
__device__ __forceinline__ bool digits_accurate(const int *ri, const int *sj, int nr, int nc, int lane, double norm_a,
                                                float tiles)
{
    int mr = INT32_MIN, mc = INT32_MIN;
    for (int i = lane; i < nr; i += 32) mr = max(mr, ri[i]);
    for (int j = lane; j < nc; j += 32) mc = max(mc, sj[j]);
    mr = __reduce_max_sync(0xffffffffu, mr);
    mc = __reduce_max_sync(0xffffffffu, mc);
    if (mr == kNonFinite || mc == kNonFinite) return false;
    float sr = 0.0f, sc = 0.0f;  // sums of squares in units of the largest
    for (int i = lane; i < nr; i += 32) sr += ldexpf(1.0f, max(2 * (ri[i] - mr), -120));
    for (int j = lane; j < nc; j += 32) sc += ldexpf(1.0f, max(2 * (sj[j] - mc), -120));
    sr = warp_sum(sr);
    sc = warp_sum(sc);
    return (double)(mr + mc) + 0.5 * (double)log2f(sr * sc * tiles) <= 7.0 + log2(norm_a);
}

// jn <= NJ columns from c0 on of one row of R by FP64 products, in the order of
// residual_f64_kernel and zresidual_f64_kernel; their sum of squares
template <bool CPLX, int NJ>
__device__ __forceinline__ double fp64_columns(const XArgs &a, int row, int c0, int jn, int im)
{
    constexpr int ES = CPLX ? 2 : 1;
    double acc[NJ], ss = 0.0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = 0.0;
    const double *x = a.X + ES * row;
    const double *y = a.Y + ES * (int64_t)c0 * a.ldy;
#pragma unroll 2
    for (int k = 0; k < a.n; ++k) {
        const double xv = x[ES * (int64_t)k * a.ldx];
        const double xi = CPLX ? (im ? 1.0 : -1.0) * x[ES * (int64_t)k * a.ldx + 1] : 0.0;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const double *yj = y + ES * (k + (int64_t)min(j, jn - 1) * a.ldy);
            acc[j] = fma(xv, yj[im], acc[j]);
            if (CPLX) acc[j] = fma(xi, yj[1 - im], acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        if (j >= jn) continue;
        const int64_t col = c0 + j;
        const double r = (a.A[ES * (row + col * a.lda) + im] - acc[j]) * a.sc;
        a.Rhat[ES * (row + col * a.ldr) + im] = (float)r;
        ss = fma(r, r, ss);
    }
    return ss;
}

// CPLX: complex A, X, Y and Rhat (interleaved), part blockIdx.z / slices (0 real, 1
// imaginary) of R; leading dimensions in elements.  CTA blockIdx.z % slices of a
// tile.
template <bool CPLX>
__global__ void __launch_bounds__(XT, 1)
xsplit_residual_kernel(XArgs a, const ResJob *__restrict__ jobs)
{
    extern __shared__ unsigned char smraw[];
    __shared__ uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    __shared__ bool s_go;
    __shared__ int s_ri[XM], s_sj[XN];
    __shared__ unsigned s_mx[4][XM];
    __shared__ double s_red[XT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = blockIdx.x * XM, n0 = blockIdx.y * XN;
    const int slices = a.slices, slice = (int)blockIdx.z % slices, zi = (int)blockIdx.z / slices;
    if (jobs) {
        const ResJob jb = jobs[zi];
        if (!*jb.active) return;
        a = XArgs{jb.A, jb.X, jb.X, jb.lda, jb.ldx, jb.ldx, jb.Rhat, jb.n, jb.partials, ldexp(1.0, -2 * *jb.e),
                  *jb.norm_a, jb.n, slices};
    }
    const int n = a.n;
    if (m0 >= n || n0 >= n) return;
    constexpr int ES = CPLX ? 2 : 1;  // doubles per element
    const int im = CPLX ? zi : 0;
    const int part = (blockIdx.x + (blockIdx.y + im * cdiv_i(n, XN)) * cdiv_i(n, XM)) * slices + slice;
    const int cz = XN / slices;  // FP64 products: columns per CTA
    if (slice > 0 && n0 + slice * cz >= n) {
        if (tid == 0) a.partials[part] = 0.0;
        return;
    }
    unsigned char *sA = (unsigned char *)(((uintptr_t)smraw + 1023) & ~(uintptr_t)1023);
    unsigned char *sB = sA + XS * XA_BYTES;
    // the scaling exponents of the tile's rows of X and columns of Y
    {
        const int row = m0 + (tid & (XM - 1)), g = tid / XM;
        unsigned mx = 0;
        if (row < n) {
            const double *x = a.X + ES * row;
#pragma unroll 8
            for (int k = g; k < n; k += XT / XM)
#pragma unroll
                for (int p = 0; p < ES; ++p)
                    mx = max(mx, (unsigned)__double2hiint(x[ES * (int64_t)k * a.ldx + p]) & 0x7FFFFFFFu);
        }
        s_mx[g][tid & (XM - 1)] = mx;
        const int col = n0 + (tid >> 3);
        mx = 0;
        if (col < n) {
            const double *y = a.Y + ES * (int64_t)col * a.ldy;
#pragma unroll 8
            for (int k = tid & 7; k < ES * n; k += 8) mx = max(mx, (unsigned)__double2hiint(y[k]) & 0x7FFFFFFFu);
        }
#pragma unroll
        for (int o = 4; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((tid & 7) == 0) s_sj[tid >> 3] = scale_exp(mx);
    }
    __syncthreads();
    if (tid < XM) s_ri[tid] = scale_exp(max(max(s_mx[0][tid], s_mx[1][tid]), max(s_mx[2][tid], s_mx[3][tid])));
    __syncthreads();
    const int qw = warp & 3, cg = warp >> 2;  // TMEM lanes 32 qw .., columns 16 cg .. of an accumulator
    const int row = m0 + 32 * qw + lane;
    if (warp == 0) {
        const bool go = n > kXsplitMinN && digits_accurate(s_ri, s_sj, min(XM, n - m0), min(XN, n - n0), lane,
                                                           a.norm_a, (float)(ES * cdiv_i(n, XM) * cdiv_i(n, XN)));
        if (lane == 0) s_go = go;
    }
    __syncthreads();
    if (!s_go) {
        // FP64 products: columns c0 .. c0 + jn - 1 of this thread's row
        const int c0 = n0 + slice * cz + cg * (cz / 4), jn = min(cz / 4, n - c0);
        double ss = 0.0;
        if (row < n && jn > 0) {
            switch (cz / 4) {
            case 16: ss = fp64_columns<CPLX, 16>(a, row, c0, jn, im); break;
            case 8: ss = fp64_columns<CPLX, 8>(a, row, c0, jn, im); break;
            default: ss = fp64_columns<CPLX, 4>(a, row, c0, jn, im); break;
            }
        }
        ss = warp_sum(ss);
        if (lane == 0) s_red[warp] = ss;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < XT / 32; ++w) t += s_red[w];
            a.partials[part] = t;
        }
        return;
    }
    if (slice > 0) {  // the tile's first CTA forms it
        if (tid == 0) a.partials[part] = 0.0;
        return;
    }
    if (tid == 0) {
        mbar_init(&s_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(XS * XN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    long long hi[16], lo[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) hi[j] = lo[j] = 0;
    const int KS = (n + XK - 1) / XK, KT = ES * KS;  // steps of 64 terms, real parts first
    bool ok = true;
    int kt = 0;
    for (; kt < KT; ++kt) {
        const int seg = CPLX && kt >= KS, k0 = (kt - seg * KS) * XK, kc = min(XK, n - k0), ksteps = (kc + 15) / 16;
        // digits of the rows of X and the columns of Y; rows and columns past
        // n are left as they are: they reach only outputs that are not stored
#pragma unroll 1
        for (int u = tid; u < XM * (XK / 8); u += XT) {
            const int r = u & (XM - 1), c = u / XM;
            if (m0 + r >= n || c >= 2 * ksteps) continue;
            const double *x = a.X + ES * (m0 + r + (int64_t)(k0 + 8 * c) * a.ldx) + seg;
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                v[q] = 8 * c + q < kc ? x[ES * (int64_t)q * a.ldx] : 0.0;
                if (CPLX && seg && !im) v[q] = -v[q];
            }
            store_digits(sA + r * 128 + ((c ^ (r & 7)) << 4), XA_BYTES, v, s_ri[r]);
        }
        {
            const int j = tid >> 3, c = tid & 7;
            if (n0 + j < n && c < 2 * ksteps) {
                const double *y = a.Y + ES * ((int64_t)(n0 + j) * a.ldy + k0 + 8 * c) + (seg ^ im);
                double v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = 8 * c + q < kc ? y[ES * q] : 0.0;
                store_digits(sB + j * 128 + ((c ^ (j & 7)) << 4), XB_BYTES, v, s_sj[j]);
            }
        }
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        if (warp == 0) {
            if (lane == 0) {
                tc_fence_after();
                const uint64_t a0 = smem_desc_sw128(smem_u32(sA)), b0 = smem_desc_sw128(smem_u32(sB));
#pragma unroll 1
                for (int d = 0; d < XS; ++d)
#pragma unroll 1
                    for (int s = 0; s <= d; ++s) {
                        // (the descriptors count in 16 bytes; 16 BF16 values = 32 bytes along k)
                        const uint64_t da = a0 + s * (XA_BYTES >> 4), db = b0 + (d - s) * (XB_BYTES >> 4);
                        const uint32_t t = tmem + (uint32_t)(d * XN);
                        mma_bf16(t, da, db, kIdesc, ((kt & 1) || s > 0) ? 1u : 0u);
                        if (ksteps > 1) mma_bf16(t, da + 2, db + 2, kIdesc, 1u);
                        if (ksteps > 2) mma_bf16(t, da + 4, db + 4, kIdesc, 1u);
                        if (ksteps > 3) mma_bf16(t, da + 6, db + 6, kIdesc, 1u);
                    }
                mma_commit(&s_bar);
            }
            __syncwarp();
        }
        // every thread waits (bounded); the block goes on or gives up as one
        if (!__syncthreads_and(mbar_wait(&s_bar, kt & 1))) {
            ok = false;
            break;
        }
        tc_fence_after();
        if ((kt & 1) || kt == KT - 1) {
            const uint32_t t0 = tmem + ((uint32_t)(32 * qw) << 16) + (uint32_t)(16 * cg);
#pragma unroll
            for (int d = 0; d < XS; d += 2) {
                uint32_t p[16], q[16];
                tmem_ld16x2(t0 + d * XN, t0 + (d + 1) * XN, p, q);
                const int w = 1 << (8 * (3 - (d & 3)));
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const long long v = (long long)__float2int_rn(__uint_as_float(p[j])) * w +
                                        (long long)__float2int_rn(__uint_as_float(q[j])) * (w >> 8);
                    if (d < 4) hi[j] += v;
                    else lo[j] += v;
                }
            }
        }
    }
    double ss = 0.0;
    if (ok && row < n) {
        const int ri = s_ri[row - m0];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int c = 16 * cg + j, col = n0 + c;
            if (col >= n) continue;
            const int e = ri + s_sj[c];
            double r = a.A[ES * (row + (int64_t)col * a.lda) + im];
            r = sub_scaled(sub_scaled(r, hi[j], e - 36), lo[j], e - 68);
            const double rs = r * a.sc;
            a.Rhat[ES * (row + (int64_t)col * a.ldr) + im] = (float)rs;
            ss = fma(rs, rs, ss);
        }
    }
    ss = warp_sum(ss);
    if (lane == 0) s_red[warp] = ss;
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
        double t = ok ? 0.0 : __longlong_as_double(0x7FF8000000000000ll);  // gave up: the norm says so
        for (int w = 0; w < XT / 32; ++w) t += s_red[w];
        a.partials[part] = t;
        // products still in flight finish (bounded) before TMEM is freed
        if (!ok) mbar_wait(&s_bar, kt & 1);
    }
    __syncthreads();
    tc_fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(XS * XN) : "memory");
}

}  // namespace

// CTAs per tile, at most 4 (with 16 the ones that leave cost a residual by digits
// 6 % at n = 384): as many as fill the SMs once; for one matrix, whose tiles
// come first in the launch and hide them, as many as give an SM the fewest
// columns of FP64 products in a row.  A matrix of FP64 tiles alone, us with the
// host call (about 50), one CTA a tile / this many / residual_f64_kernel: n = 64
// 138 / 87 / 99, 128 334 / 136 / 170, 256 594 / 209 / 307, 512 1123 / 358 / 590, 640 1391
// / 751 / 726, 777 1672 / 1111 / 1640, 1024 2181 / 2180 / 2137.
static int xsplit_slices(int64_t tiles, bool one)
{
    int best = 1;
    for (int z = 2; z <= 4; z *= 2)
        if (z * tiles <= (one ? 4 * 152 : 152) && cdiv_i(z * tiles, 152) * best < cdiv_i(best * tiles, 152) * z) best = z;
    return best;
}
static int64_t xsplit_tiles(int n) { return n <= 0 ? 0 : cdiv_i(n, XM) * cdiv_i(n, XN); }

int xsplit_parts(int n, int nmax, int batch) { return (int)xsplit_tiles(n) * xsplit_slices(xsplit_tiles(nmax) * batch, false); }
int xsplit_parts_cap(int n) { return 4 * (int)xsplit_tiles(n); }

cudaError_t launch_xsplit_residual(const double *A, int64_t lda, const double *X, int64_t ldx, const double *Y,
                                   int64_t ldy, int n, int shift, double norm_a, float *Rhat, int ldr, double *partials,
                                   int *nparts, cudaStream_t s)
{
    const int z = xsplit_slices(xsplit_tiles(n), true);
    *nparts = (int)xsplit_tiles(n) * z;
    if (n <= 0) return cudaSuccess;
    cudaError_t err = allow_max_smem((const void *)xsplit_residual_kernel<false>);
    if (err) return err;
    xsplit_residual_kernel<false><<<dim3((unsigned)cdiv_i(n, XM), (unsigned)cdiv_i(n, XN), (unsigned)z), XT, X_SMEM, s>>>(
        XArgs{A, X, Y, lda, ldx, ldy, Rhat, ldr, partials, ldexp(1.0, -shift), norm_a, n, z}, nullptr);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_xsplit_zresidual(const double *A, int64_t lda, const double *X, int64_t ldx, int n, int shift,
                                    double norm_a, cplx<float> *Rhat, int ldr, double *partials, int *nparts,
                                    cudaStream_t s)
{
    const int z = xsplit_slices(2 * xsplit_tiles(n), true);
    *nparts = 2 * (int)xsplit_tiles(n) * z;
    if (n <= 0) return cudaSuccess;
    cudaError_t err = allow_max_smem((const void *)xsplit_residual_kernel<true>);
    if (err) return err;
    xsplit_residual_kernel<true><<<dim3((unsigned)cdiv_i(n, XM), (unsigned)cdiv_i(n, XN), 2u * z), XT, X_SMEM, s>>>(
        XArgs{A, X, X, lda, ldx, ldx, reinterpret_cast<float *>(Rhat), ldr, partials, ldexp(1.0, -shift), norm_a, n, z},
        nullptr);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_xsplit_residual_batched(const ResJob *jobs, int batch, int nmax, cudaStream_t s)
{
    if (nmax <= 0 || batch <= 0) return cudaSuccess;
    cudaError_t err = allow_max_smem((const void *)xsplit_residual_kernel<false>);
    if (err) return err;
    XArgs a{};
    a.slices = xsplit_slices(xsplit_tiles(nmax) * batch, false);
    xsplit_residual_kernel<false><<<dim3((unsigned)cdiv_i(nmax, XM), (unsigned)cdiv_i(nmax, XN), (unsigned)(batch * a.slices)),
                                    XT, X_SMEM, s>>>(a, jobs);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sqm
