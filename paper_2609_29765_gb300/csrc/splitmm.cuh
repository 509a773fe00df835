// splitmm.cuh -- FP64 tile products on the tensor cores by an error-free split.
//
// sm_103a has no FP64 tensor kind worth using (DMMA shares the 2-DFMA/clk/SM FP64 pipe),
// so C -= A B^T is formed from exact integer products (the error-free transformation of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): each operand row of a
// 16-column chunk is scaled by a power of two to 62-bit fixed point, cut into eight
// balanced base-256 digits, and the digit pairs (i, j), i + j <= 7, are multiplied by
// mma.sync f16 with f32 accumulators, one accumulator per i + j.  A digit is at most 128
// in magnitude, so a sum over 16 columns and 8 pairs stays below 2^21 and every f32 sum
// is exact.  The eight sums are put together in integers (one rounding to 2^-58 of the
// largest product the rows allow), rounded to a double and subtracted from C: two
// roundings per 16 columns where sixteen fused multiply-adds made sixteen.
//
// What bounds it: 36 tensor products per FP64 product at 605 TFLOP/s (mma.sync f16,
// measured) are 16.8 TFLOP/s of FP64 work against 1.26 on the DFMA pipe; the split, the
// digit expansion and the epilogue issue about as long as the tensor pipe runs.  Measured,
// supernodal route: one factorization at n = 180,020 517 -> 251 ms, a 48^3 FEM operator
// 180 -> 98 ms, 16 sets at n = 22,520 95 -> 57 ms, and the products and their staging no
// more than 37 % of the CTAs' time (the rest waits for other tasks).
//
// Rows whose largest entry is not finite or lies outside 2^[-400, 400] (where the scale
// arithmetic could leave the exponent range), and rows of subnormals, are reported by the
// staging pass; the caller then multiplies that chunk with DFMAs, so infinities, NaN and
// extreme scales keep IEEE semantics.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace stc {
namespace {

constexpr int kSpK = 16;                   // inner columns per chunk (one k16 mma step)
constexpr int kSpRows = 128;               // operand rows a digit buffer holds
// a digit buffer: kSpRows rows of 16 columns x 8 digits (one byte each), then an exponent
// per row
constexpr int kSpDoubles = kSpRows * kSpK + kSpRows / 2;

__device__ __forceinline__ uint4* sp_digits(double* S) { return reinterpret_cast<uint4*>(S); }
__device__ __forceinline__ int* sp_exp(double* S) { return reinterpret_cast<int*>(S + kSpRows * kSpK); }

// Place of column pair kp (columns 2 kp, 2 kp + 1) of row r: a row is 128 bytes, eight
// 16-byte pairs, permuted so that eight consecutive rows of one pair (the staging stores)
// and two rows of four pairs (the fragment loads) both touch every bank once.
__device__ __forceinline__ int sp_slot(int r, int kp) { return r * 8 + (kp ^ (((r & 1) << 2) | ((r >> 1) & 3))); }

// Biased exponent of the largest entry of a chunk row v[0..15]; ok: the row can take this
// path (see above).
__device__ __forceinline__ int sp_row_exp(const double (&v)[kSpK], bool& ok) {
    unsigned m = 0u, any = 0u;
#pragma unroll
    for (int k = 0; k < kSpK; ++k) {
        const unsigned h = (unsigned)__double2hiint(v[k]) & 0x7fffffffu;
        m = max(m, h);
        any |= h | (unsigned)__double2loint(v[k]);
    }
    const int e = (int)(m >> 20);
    ok = any == 0u || (e >= 1023 - 400 && e <= 1023 + 400);
    return e;
}

// The digits of row r, v[0..15] (zero from K on), e its exponent.
__device__ __forceinline__ void sp_split_row(const double (&v)[kSpK], int e, int K, double* S, int r) {
    sp_exp(S)[r] = e;
    uint4* D = sp_digits(S);
#pragma unroll
    for (int kp = 0; kp < kSpK / 2; ++kp) {
        if (2 * kp >= K) {  // no such columns (K is the same for the whole CTA): digits of zero
            D[sp_slot(r, kp)] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
            continue;
        }
        unsigned hi[2], lo[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned h = (unsigned)__double2hiint(v[2 * kp + q]);
            const int ex = (int)((h >> 20) & 0x7ffu);
            // 53-bit mantissa at bit 9 (below 2^62 for the row's largest), aligned to the row
            unsigned long long f = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) |
                                   (unsigned)__double2loint(v[2 * kp + q]);
            f = ex ? f : 0ull;
            f = (f << 9) >> min(e - ex, 63);
            f = ((int)h < 0 ? 0ull - f : f) + 0x8080808080808080ull;  // digit bytes, each + 128
            hi[q] = (unsigned)(f >> 32);
            lo[q] = (unsigned)f;
        }
        // word w holds digits 2 w and 2 w + 1 of both columns: bytes (d1, d0, d1', d0')
        D[sp_slot(r, kp)] = make_uint4(__byte_perm(hi[0], hi[1], 0x7632), __byte_perm(hi[0], hi[1], 0x5410),
                                       __byte_perm(lo[0], lo[1], 0x7632), __byte_perm(lo[0], lo[1], 0x5410));
    }
}

// Whether a chunk's product is worth the split: 2 x 2 DFMA micro-tiles take 256 clocks per
// column and 512 entries, splitting and multiplying at least about kSpWorth times that
// whatever the size.  Measured at thresholds 0 / 8 / 24 / 80: one small grid (n = 1,026)
// 596 / 594 / 625 / 627 us, a 48^3 FEM operator - / 71.1 / 72.2 / 80.9 ms, 16 spatio-temporal
// precisions (n = 22,520) - / 42.6 / 44.0 / 49.2 ms.
constexpr int kSpWorth = 8;
__device__ __forceinline__ bool sp_worth(int entries, int K) { return K * ((entries + 511) >> 9) >= kSpWorth; }

// Operands A (R x K, entries ga(r, k)) and B (Cn x K, gb(c, k)) of a chunk into the digit
// buffers SA and SB, a thread per row (R + Cn <= blockDim.x); returns on every thread
// whether all rows can take the tensor path, after a barrier.  IN_PLACE: ga or gb may read
// SA or SB; nothing is written unless the result is true.
template <bool IN_PLACE, class GetA, class GetB>
__device__ __forceinline__ bool sp_stage_t(double* SA, int R, GetA ga, double* SB, int Cn, GetB gb, int K) {
    const int i = threadIdx.x;
    double v[kSpK];
#pragma unroll
    for (int k = 0; k < kSpK; ++k) v[k] = 0.0;
    if (i < R) {
#pragma unroll
        for (int k = 0; k < kSpK; ++k)
            if (k < K) v[k] = ga(i, k);
    } else if (i < R + Cn) {
#pragma unroll
        for (int k = 0; k < kSpK; ++k)
            if (k < K) v[k] = gb(i - R, k);
    }
    bool ok = true;
    const int e = sp_row_exp(v, ok);
    if (IN_PLACE && !__syncthreads_and(ok)) return false;
    if (i < R + Cn) sp_split_row(v, e, K, i < R ? SA : SB, i < R ? i : i - R);
    return __syncthreads_and(ok);
}
template <class GetA, class GetB>
__device__ __forceinline__ bool sp_stage_ab(double* SA, int R, GetA ga, double* SB, int Cn, GetB gb, int K) {
    return sp_stage_t<false>(SA, R, ga, SB, Cn, gb, K);
}
template <class GetA>
__device__ __forceinline__ bool sp_stage_a(double* SA, int R, GetA ga, int K) {
    return sp_stage_t<false>(SA, R, ga, SA, 0, ga, K);
}

// Digits of one 16-byte pair as eight f16x2 registers (the two columns of digit d), exact:
// byte b = digit + 128 becomes f16 1024 + b, minus 1152.
__device__ __forceinline__ void sp_expand(uint4 p, unsigned (&f)[8]) {
    const unsigned w[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        unsigned a = __byte_perm(w[q], 0x64646464u, 0x4341), b = __byte_perm(w[q], 0x64646464u, 0x4240);
        asm("sub.f16x2 %0, %1, %2;" : "=r"(f[2 * q]) : "r"(a), "r"(0x64806480u));
        asm("sub.f16x2 %0, %1, %2;" : "=r"(f[2 * q + 1]) : "r"(b), "r"(0x64806480u));
    }
}

__device__ __forceinline__ void sp_mma(float (&d)[4], const float (&c)[4], unsigned a0, unsigned a1, unsigned a2,
                                       unsigned a3, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// The double nearest T 2^(10 + E - 2046 - 66) for |T| < 2^63 (E: sum of the two biased row
// exponents), T = 0 giving +0.
__device__ __forceinline__ double sp_double(long long T, int E) {
    const unsigned long long mag = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
    if (mag == 0ull) return 0.0;
    const int lz = __clzll((long long)mag);
    const unsigned long long nrm = mag << lz;
    // biased exponent of the leading bit: 1023 + 63 - lz + E - 2102; the hidden bit adds one
    // (rounded after the shift: a mantissa of ones carries into the exponent)
    const unsigned long long bits =
        ((unsigned long long)(unsigned)(E - 1016 - lz - 1) << 52) + (nrm >> 11) + ((nrm >> 10) & 1ull);
    return __longlong_as_double((long long)(bits | ((unsigned long long)T & 0x8000000000000000ull)));
}

// sum over the chunk of A(a0 + r, k) B(b0 + c, k) for every r < R, c < Cn (LOWER: at least every
// r >= c), one call epi(r, c, value) per entry; 16 x 8 units of the product spread over the
// CTA's warps in contiguous runs, so that a warp expands a strip of A once.  epi must not
// synchronise.
template <bool LOWER, class Epi>
__device__ __forceinline__ void sp_product(double* SA, int a0, int R, double* SB, int b0, int Cn, Epi epi) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const uint4 *A = sp_digits(SA), *B = sp_digits(SB);
    const int *ea = sp_exp(SA), *eb = sp_exp(SB);
    const int MR = (R + 15) >> 4, NC = (Cn + 7) >> 3;
    // LOWER: strip s holds the units c < min(2 s + 2, NC) (rows and columns index one range)
    const int units = LOWER ? (MR - 1) * MR + min(2 * MR, NC) : MR * NC;
    int u = units * warp / nwarps;
    const int uend = units * (warp + 1) / nwarps;
    if (u >= uend) return;
    int s, c;
    if (LOWER) {
        s = 0;
        while ((s + 1) * (s + 2) <= u) ++s;
        c = u - s * (s + 1);
    } else {
        s = u / NC;
        c = u - s * NC;
    }
    const float kM = 12582912.0f;  // 1.5 2^23: an integer n is then the bits 0x4B400000 + n
    const float m4[4] = {kM, kM, kM, kM};
    while (u < uend) {
        unsigned fa[4][8];
        const int r0 = s * 16 + g;
        const int ra = a0 + min(r0, R - 1), rb = a0 + min(r0 + 8, R - 1);  // rows past the end: not used
        sp_expand(A[sp_slot(ra, t)], fa[0]);
        sp_expand(A[sp_slot(rb, t)], fa[1]);
        sp_expand(A[sp_slot(ra, t + 4)], fa[2]);
        sp_expand(A[sp_slot(rb, t + 4)], fa[3]);
        const int e0 = ea[ra], e1 = ea[rb];
        const int cend = LOWER ? min(2 * s + 2, NC) : NC;
        for (; c < cend && u < uend; ++c, ++u) {
            unsigned fb[2][8];
            const int cb = b0 + min(c * 8 + g, Cn - 1);
            sp_expand(B[sp_slot(cb, t)], fb[0]);
            sp_expand(B[sp_slot(cb, t + 4)], fb[1]);
            float acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8 - i; ++j) {
                    if (i == 0) sp_mma(acc[j], m4, fa[0][0], fa[1][0], fa[2][0], fa[3][0], fb[0][j], fb[1][j]);
                    else sp_mma(acc[i + j], acc[i + j], fa[0][i], fa[1][i], fa[2][i], fa[3][i], fb[0][j], fb[1][j]);
                }
            const int c0 = c * 8 + 2 * t;
            const int f0 = eb[b0 + min(c0, Cn - 1)], f1 = eb[b0 + min(c0 + 1, Cn - 1)];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + (q >> 1) * 8, cc = c0 + (q & 1);
                if (r >= R || cc >= Cn || (LOWER && r < cc)) continue;
                int n[8];
#pragma unroll
                for (int d = 0; d < 8; ++d) n[d] = __float_as_int(acc[d][q]) - 0x4B400000;
                const long long hi = (long long)(n[0] * 256 + n[1]) * 65536 + (n[2] * 256 + n[3]);
                const long long lo = (long long)(n[4] * 256 + n[5]) * 65536 + (n[6] * 256 + n[7]);
                const long long T = hi * (1ll << 22) + ((lo + 512) >> 10);
                epi(r, cc, sp_double(T, ((q >> 1) ? e1 : e0) + ((q & 1) ? f1 : f0)));
            }
        }
        ++s;
        c = 0;
    }
}

}  // namespace
}  // namespace stc
