// splitmm.cuh -- FP64 tile products on the tensor cores by a split into digits.
//
// sm_103a has no FP64 tensor kind worth using (DMMA shares the 2-DFMA/clk/SM FP64 pipe),
// so C -= A B^T is formed from integer products of digits (after the error-free
// transformation of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): each operand
// row of a 16-column chunk is scaled by a power of two to 62-bit fixed point, cut into eight
// balanced base-256 digits, and the digit pairs (i, j), i + j <= 7, are multiplied by
// mma.sync f16 with f32 accumulators, one accumulator per i + j.  A digit is at most 128
// in magnitude, so a sum over 16 columns and 8 pairs stays below 2^21 and every f32 sum
// is exact.  The eight sums are put together in integers, rounded to a double and subtracted
// from C.
//
// What is exact and what is not: the sums of the 36 pairs are.  An entry more than 2^9 below
// its row's largest of the chunk loses its last bits (truncated), one 2^62 below all of them;
// the 28 pairs beyond are left out; the sum is rounded twice.  All of it is at most 2^-53 of
// (largest of A's row) x (largest of B's row) per chunk, with digits of one sign throughout;
// with the digits of ordinary data about 2^-58.  That is relative to the row maxima, not to
// sum |a_k b_k| as the roundings of FMAs are.  For rows of L over the same columns it is what
// the factorization's error is measured in (|L_ik| <= sqrt(a_ii), units of the variables scale
// whole rows); products of other operands have to be balanced first (Balance below).
//
// What bounds it: 36 tensor products per FP64 product at 605 TFLOP/s (mma.sync f16,
// measured) are 16.8 TFLOP/s of FP64 work against 1.26 on the DFMA pipe; the split, the
// digit expansion and the epilogue issue about as long as the tensor pipe runs.  Measured,
// supernodal route: one factorization at n = 180,020 517 -> 251 ms by the products alone
// (107 with two CTAs per SM and the scheduled queue), a 48^3 FEM operator 180 -> 98 (33) ms,
// 16 sets at n = 22,520 95 -> 57 (35) ms; of the CTAs' time at n = 180,020 the products then
// take 55 %, their staging 17 %.  Tile routes: 64 bands (n = 50,000, half-bandwidth 200)
// 178 -> 89 ms with the 16-column panels of POTRF and TRSM.
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

// Balance of the inner index.  A row keeps 62 bits below its largest entry of the chunk, so
// both operands need rows whose entries matter alike: rows of L do (|L_ik| <= sqrt(a_ii) for
// every k), rows of a selected inverse times L do not (Sigma_ri ~ 1 / d_i against L_ic ~ d_i
// for a variable i in units 1 / d_i).  There the caller gives the power of two b(i, k) that
// entry k of operand row i is multiplied by before the cut, opposite for the two operands, so
// the products stay what they are.  It is added to the exponents only: no entry is formed.
// A balance outside 2^+-kSpBalMax (entries that are not finite have to stay out of range)
// becomes one that puts every row of the other operand out of range: DFMAs take the chunk.
constexpr int kSpBalMax = 300, kSpUnbalanced = 3000;
__device__ __forceinline__ int sp_balance(int e) { return abs(e) <= kSpBalMax ? e : kSpUnbalanced; }
struct NoBalance {
    static constexpr bool kNone = true, late = false;
};
struct Balance {  // A's rows (i < R) times 2^-e[k], B's times 2^e[k]
    static constexpr bool kNone = false;
    const int* e;  // 16 readable values from a 16-byte boundary on, those from K on unused
    int R, K;
    bool late;  // e was written since the last barrier (the same for the whole CTA)
};
// The balances of columns 4 g .. 4 g + 3 in row i.
__device__ __forceinline__ void sp_bal4(const Balance& b, int i, int g, int (&s)[4]) {
    const int4 x = reinterpret_cast<const int4*>(b.e)[g];
    const int v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = 4 * g + q >= b.K ? 0 : i < b.R ? -v[q] : v[q];
}
__device__ __forceinline__ void sp_bal4(const NoBalance&, int, int, int (&s)[4]) { s[0] = s[1] = s[2] = s[3] = 0; }

// Biased exponent of the largest entry of a chunk row v[0..15], balanced as operand row i;
// ok: the row can take this path (see above; a subnormal entry counts as 2^-1023, far below
// the cut of a row in range).
template <class Bal>
__device__ __forceinline__ int sp_row_exp(const double (&v)[kSpK], bool& ok, int i, Bal bal) {
    int m = Bal::kNone ? 0 : -kSpUnbalanced;
    unsigned any = 0u;
#pragma unroll
    for (int g = 0; g < kSpK / 4; ++g) {
        int s[4];
        sp_bal4(bal, i, g, s);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned h = (unsigned)__double2hiint(v[4 * g + q]) & 0x7fffffffu;
            m = max(m, Bal::kNone ? (int)h : (int)(h >> 20) + s[q]);
            any |= h | (unsigned)__double2loint(v[4 * g + q]);
        }
    }
    const int e = Bal::kNone ? m >> 20 : m;
    ok = any == 0u || (e >= 1023 - 400 && e <= 1023 + 400);
    return e;
}

// The digits of v[0..15] (zero from K on), balanced as operand row i, e their exponent, as row r.
template <class Bal>
__device__ __forceinline__ void sp_split_row(const double (&v)[kSpK], int e, int K, double* S, int r, int i, Bal bal) {
    sp_exp(S)[r] = e;
    uint4* D = sp_digits(S);
#pragma unroll
    for (int kp = 0; kp < kSpK / 2; ++kp) {
        if (2 * kp >= K) {  // no such columns (K is the same for the whole CTA): digits of zero
            D[sp_slot(r, kp)] = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
            continue;
        }
        int s[4];
        sp_bal4(bal, i, kp >> 1, s);
        unsigned hi[2], lo[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned h = (unsigned)__double2hiint(v[2 * kp + q]);
            const int ex = (int)((h >> 20) & 0x7ffu);
            // 53-bit mantissa at bit 9 (below 2^62 for the row's largest), aligned to the row
            unsigned long long f = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32) |
                                   (unsigned)__double2loint(v[2 * kp + q]);
            f = ex ? f : 0ull;
            f = (f << 9) >> min(e - ex - s[2 * (kp & 1) + q], 63);
            f = ((int)h < 0 ? 0ull - f : f) + 0x8080808080808080ull;  // digit bytes, each + 128
            hi[q] = (unsigned)(f >> 32);
            lo[q] = (unsigned)f;
        }
        // word w holds digits 2 w and 2 w + 1 of both columns: bytes (d1, d0, d1', d0')
        D[sp_slot(r, kp)] = make_uint4(__byte_perm(hi[0], hi[1], 0x7632), __byte_perm(hi[0], hi[1], 0x5410),
                                       __byte_perm(lo[0], lo[1], 0x7632), __byte_perm(lo[0], lo[1], 0x5410));
    }
}

// Whether a chunk's product is worth the split: with an entry per thread DFMAs take 64 clocks
// per column and 128 entries, splitting and multiplying about kSpWorth times that at least.
// At thresholds 32 / 64 / 96: three FEM operators (dense tiles) 88.1 / 84.1 / 83.6 ms, 16
// bands with marginals 147 / 142 / 141 ms, 64 small grids 1.08 / 1.05 / 1.04 ms, one 48^3 FEM
// operator (supernodal) 49.1 / 49.4 / 50.5 ms, 16 spatio-temporal precisions 34.3 / 35.0 /
// 35.8 ms.  (Below it 2 x 2 micro-tiles in place of an entry per thread: 64 grids 1.53 ms.)
constexpr int kSpWorth = 64;
__device__ __forceinline__ bool sp_worth(int entries, int K) { return K * ((entries + 127) >> 7) >= kSpWorth; }

// Operands A (R x K, entries ga(r, k)) and B (Cn x K, gb(c, k)) of a chunk into the digit
// buffers SA and SB, a thread per row (R + Cn <= blockDim.x); returns on every thread
// whether all rows can take the tensor path, after a barrier.  bal: the balance of the inner
// index.  IN_PLACE: ga or gb may read SA or SB; nothing is written unless
// the result is true.
template <bool IN_PLACE, class GetA, class GetB, class Bal = NoBalance>
__device__ __forceinline__ bool sp_stage_t(double* SA, int R, GetA ga, double* SB, int Cn, GetB gb, int K,
                                           Bal bal = Bal()) {
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
    if (!Bal::kNone && bal.late) __syncthreads();  // the balance was written while the rows were loaded
    bool ok = true;
    const int e = sp_row_exp(v, ok, i, bal);
    if (IN_PLACE && !__syncthreads_and(ok)) return false;
    if (i < R + Cn) sp_split_row(v, e, K, i < R ? SA : SB, i < R ? i : i - R, i, bal);
    return __syncthreads_and(ok);
}
template <class GetA, class GetB, class Bal = NoBalance>
__device__ __forceinline__ bool sp_stage_ab(double* SA, int R, GetA ga, double* SB, int Cn, GetB gb, int K,
                                            Bal bal = Bal()) {
    return sp_stage_t<false>(SA, R, ga, SB, Cn, gb, K, bal);
}
template <class GetA, class Bal = NoBalance>
__device__ __forceinline__ bool sp_stage_a(double* SA, int R, GetA ga, int K, Bal bal = Bal()) {
    return sp_stage_t<false>(SA, R, ga, SA, 0, ga, K, bal);
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

// sum_d n_d 2^(8 (7 - d)) / 2^10, rounded, from the accumulators 1.5 2^23 + n_d: their bits
// are 0x4B400000 + n_d and go in as they are (wide integer multiply-adds, which leave the
// busier ALU pipe alone), the biases come off in one constant.
__device__ __forceinline__ long long sp_sum(float n0, float n1, float n2, float n3, float n4, float n5, float n6,
                                            float n7) {
    constexpr unsigned long long kB = 0x4B400000ull;
    constexpr unsigned long long kOff =
        0ull - (((kB * (1u << 14) + kB * (1u << 6)) << 32) + kB * ((1ull << 30) + (1ull << 22) + (1ull << 14) + (1ull << 6)));
    unsigned long long T;
    asm("{\n\t"
        ".reg .u64 a;\n\t"
        ".reg .u32 lo, hi;\n\t"
        "mad.wide.u32 a, %3, 0x40000000, %9;\n\t"
        "mad.wide.u32 a, %4, 0x400000, a;\n\t"
        "mad.wide.u32 a, %5, 0x4000, a;\n\t"
        "mad.wide.u32 a, %6, 0x40, a;\n\t"
        "mov.b64 {lo, hi}, a;\n\t"
        "mad.lo.u32 hi, %1, 0x4000, hi;\n\t"
        "mad.lo.u32 hi, %2, 0x40, hi;\n\t"
        "mov.b64 a, {lo, hi};\n\t"
        "mad.lo.u32 lo, %7, 0x100, %8;\n\t"
        "add.u32 lo, lo, %10;\n\t"
        "shr.s32 lo, lo, 10;\n\t"
        "mad.wide.s32 %0, lo, 1, a;\n\t"
        "}"
        : "=l"(T)
        : "r"(__float_as_uint(n0)), "r"(__float_as_uint(n1)), "r"(__float_as_uint(n2)), "r"(__float_as_uint(n3)),
          "r"(__float_as_uint(n4)), "r"(__float_as_uint(n5)), "r"(__float_as_uint(n6)), "r"(__float_as_uint(n7)),
          "l"(kOff), "n"(512u - 0x4B400000u * 257u));
    return (long long)T;
}

// The double nearest T 2^(E - 2102) for |T| < 2^63 (E: sum of the two biased row exponents),
// T = 0 giving +0.
__device__ __forceinline__ double sp_double(long long T, int E) {
    const long long sg = T >> 63;
    const unsigned long long mag = (unsigned long long)((T ^ sg) - sg);
    const int lz = __clzll((long long)mag);
    const unsigned long long nrm = mag << (lz & 63);
    // biased exponent of the leading bit: 1023 + 63 - lz + E - 2102; the hidden bit adds one
    // (rounded after the shift: a mantissa of ones carries into the exponent)
    unsigned long long bits =
        ((unsigned long long)(unsigned)(E - 1016 - lz - 1) << 52) + (nrm >> 11) + ((nrm >> 10) & 1ull);
    bits = mag ? bits | ((unsigned long long)sg & 0x8000000000000000ull) : 0ull;
    return __longlong_as_double((long long)bits);
}

// Units (16 rows x 8 columns) of a product: row strips in order, LOWER only the units that
// reach r >= c (rows and columns index one range; strip s then starts at unit s (s + 1)).
template <bool LOWER>
__device__ __forceinline__ int sp_units(int R, int Cn) {
    const int MR = (R + 15) >> 4, NC = (Cn + 7) >> 3;
    return LOWER ? (MR - 1) * MR + min(2 * MR, NC) : MR * NC;
}

// One warp: at(r, c) -= sum_k A(a0 + r, k) B(b0 + c, k) over the units [u, uend), for r < R,
// c < Cn (LOWER: r >= c); at(r, c) is a reference to the entry.  A strip of A is expanded
// once.  A unit is 330 instructions, half of them on the ALU pipe and 36 on the tensor pipe,
// which take about 330 clocks of an SM sub-partition each: a 64 x 128 chunk takes 9,500
// clocks of an SM with two CTAs (65,500 on the DFMA pipe).  The four entries of a lane side
// by side without branches take 8,100 where every entry is wanted, but ragged units then pay
// for entries nobody wants (one factorization at n = 180,020: 158 -> 176 ms).
template <bool LOWER, class At>
__device__ __forceinline__ void sp_run(double* SA, int a0, int R, double* SB, int b0, int Cn, int u, int uend, At at) {
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const uint4 *A = sp_digits(SA), *B = sp_digits(SB);
    const int *ea = sp_exp(SA), *eb = sp_exp(SB);
    const int NC = (Cn + 7) >> 3;
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
                const long long T = sp_sum(acc[0][q], acc[1][q], acc[2][q], acc[3][q], acc[4][q], acc[5][q],
                                           acc[6][q], acc[7][q]);
                at(r, cc) -= sp_double(T, ((q >> 1) ? e1 : e0) + ((q & 1) ? f1 : f0));
            }
        }
        ++s;
        c = 0;
    }
}

// The whole product, its units spread over the CTA's warps in contiguous runs.
template <bool LOWER, class At>
__device__ __forceinline__ void sp_product(double* SA, int a0, int R, double* SB, int b0, int Cn, At at) {
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, units = sp_units<LOWER>(R, Cn);
    sp_run<LOWER>(SA, a0, R, SB, b0, Cn, units * warp / nwarps, units * (warp + 1) / nwarps, at);
}

}  // namespace
}  // namespace stc
