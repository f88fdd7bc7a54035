// tc_f64.cuh -- FP64 products on the tensor cores, in fixed point.
//
// A GB300 SM retires about 1.6 FP64 multiply-adds a clock and 0.47 FP16
// 16 x 8 x 16 tile products (2,048 multiply-adds each), so the Gram block and
// the rotation update of FP64 and complex128 split every operand into digits that the
// FP16 units multiply exactly (the scheme of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", Numer. Algorithms 59, 2012):
//   x = 2^(E - 52) sum_i d_i 512^(5 - i),  d_i in [-256, 256], i = 0 .. 5,
// E the largest exponent of the row (or column) the product sums over; an
// entry keeps 53 bits below that exponent, rounded to nearest.  A product of
// two digits is below 2^16 and a sum of 32 times the up to six digit products
// of equal weight i + j below 2^24: the digit products and their sums are exact
// in the FP32 accumulator.  The result is not: weights up to 6 are kept (26 of
// the 36 digit products), and the operands are rounded.  In units of the row's
// largest entry times the column's, what is dropped is below 2^-59 a term and
// 2^-54 over 32, the operands' rounding (2^-53 on either side) below 2^-52 a
// term and 2^-47 over 32; 32 chained multiply-adds, each rounding a partial
// sum, may lose 2^-44 on the same entries.  Accumulators are converted and
// combined as integers and rounded once to FP64; no FP64 instruction is used
// at all.
//
// Fragments (PTX ISA, mma.sync.m16n8k16 .f16), g = lane / 4, t = lane % 4:
//   A (16 x 16)  a0 (g, 2t..2t+1)  a1 (g+8, 2t..)  a2 (g, 2t+8..)  a3 (g+8, 2t+8..)
//   B (16 x 8)   b0 (2t..2t+1, g)  b1 (2t+8.., g)
//   C (16 x 8)   c0 c1 (g, 2t..2t+1)  c2 c3 (g+8, 2t..)
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

#include "jacobi_common.cuh"

namespace bsvd {

constexpr int kDigits = 6, kWeights = 7;       // weights i + j = 0 .. 6
constexpr int kNoExp = -4000;                  // exponent of a zero

// Biased exponent of x (denormals count as zero).
__device__ __forceinline__ int exp_f64(double x) {
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    return e ? e : kNoExp;
}

// x as a 54-bit integer relative to exponent E = exp(x) + sh (sh >= 0), rounded
// to nearest even (an entry one binary order below E drops one bit, a tie half
// of the time: rounding those one way moves every column a quarter of a unit
// per update), plus 256 in every digit: digit i is bits 9 (5 - i) .. of the
// result less 256 (the leading one takes ten bits).
__device__ __forceinline__ unsigned long long fixed_f64(double x, int sh) {
    const long long b = __double_as_longlong(x);
    long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    if (((b >> 52) & 0x7ff) == 0) m = 0;
    if (b < 0) m = -m;
    const int s = min(sh, 60);
    const long long v = s > 0 ? (m + (1ll << (s - 1)) - 1 + ((m >> s) & 1)) >> s : m;
    // sum of 256 * 512^i, i < 6
    return (unsigned long long)v + 0x20100804020100ull;
}

// digit i of two fixed-point values as an FP16 pair (x0 in the low half)
template <int I>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long x0, unsigned long long x1) {
    constexpr int S = 9 * (5 - I);
    const uint32_t u0 = I == 0 ? (uint32_t)(x0 >> S) : (uint32_t)(x0 >> S) & 511u;
    const uint32_t u1 = I == 0 ? (uint32_t)(x1 >> S) : (uint32_t)(x1 >> S) & 511u;
    // 0x6400 + u is 1024 + u in FP16; less 1280
    const uint32_t h = (u0 | (u1 << 16)) + 0x64006400u;
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6500)));
    return *reinterpret_cast<const uint32_t*>(&r);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The weights' sums as one integer in units of 512^4 / 2^21 (weight 2's unit
// is 512^8): sum_o acc_o 512^(10 - o) = T 2^51, T below 2^62.
__device__ __forceinline__ long long combine_weights(const float (&c)[kWeights]) {
    const int i0 = __float2int_rn(c[0]), i1 = __float2int_rn(c[1]), i2 = __float2int_rn(c[2]), i3 = __float2int_rn(c[3]),
              i4 = __float2int_rn(c[4]), i5 = __float2int_rn(c[5]), i6 = __float2int_rn(c[6]);
    const long long hi = (long long)i0 * 262144 + ((long long)i1 * 512 + i2);
    const long long lo = ((long long)i3 * 512 + i4) * 262144 + ((long long)i5 * 512 + i6);
    return (hi << 21) + ((lo + (1 << 14)) >> 15);
}

// T 2^s to FP64, rounded to nearest; zero below the normal range.
__device__ __forceinline__ double fixed_to_f64(long long T, int s) {
    const unsigned long long a = T < 0 ? (unsigned long long)-T : (unsigned long long)T;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const int e = 1023 + 63 - lz + s;
    if (e < 1) return 0.0;
    const unsigned long long m = a << lz;                  // leading one at bit 63
    // the leading one adds itself to the exponent field; a rounding carry too
    const unsigned long long r = ((unsigned long long)(e - 1) << 52) + (m >> 11) + ((m >> 10) & 1);
    return __longlong_as_double((long long)(r | ((unsigned long long)T & 0x8000000000000000ull)));
}

// Largest biased exponent of each of the 2 NB columns of a panel (columns [cbi,
// cbi + NB) and [cbj, cbj + NB) of W, M rows) into ec.  GT threads (a multiple of
// 2 NB); the caller synchronises.
template <int NB, int GT>
__device__ __forceinline__ void column_exponents_f64(const double* W, long long ldw, int M, int cbi, int cbj, int* ec,
                                                     int gt) {
    constexpr int P = GT / (2 * NB);                       // threads a column
    static_assert(P >= 1 && P <= 32 && (P & (P - 1)) == 0, "threads a column");
    const int c = gt / P, q = gt % P;
    const double* x = W + (c < NB ? cbi + c : cbj + c - NB) * ldw;
    int e = kNoExp;
    for (int r = q; r < M; r += P) e = max(e, exp_f64(x[r]));
#pragma unroll
    for (int o = 1; o < P; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (q == 0) ec[c] = e;
}

// S2: G = P^T P (2 NB x 2 NB, column stride LDG) for the panel P of
// column_exponents.  Four warps (NB = 8: two) take 16 rows in turn, whatever the
// group's size, so that the bits do not depend on it; each forms the 16 x 8
// tiles that meet the upper triangle from one set of digits (a column's digits serve as A and as B
// fragment), converts them to FP64 and sums its own; the warps' sums are added
// in warp order.  Upper entries are written and mirrored.  GT threads, named
// barrier `bar`; synchronised on return.
template <int NB, int GT, int LDG>
__device__ __forceinline__ void gram_f64_split(const double* W, long long ldw, int M, int cbi, int cbj, const int* ec,
                                               double* G, int gt, int bar) {
    constexpr int NBM = 2 * NB / 16, NTL = NBM == 2 ? 6 : 2, NWS = NBM == 2 ? 4 : 2;
    static_assert(NB == 8 || NB == 16, "one or two blocks of 16 columns");
    static_assert(GT >= 32 * NWS, "the summing warps");
    const int warp = gt >> 5, lane = gt & 31, g = lane >> 2, t = lane & 3;
    auto col = [&](int c) { return (c < NB ? cbi + c : cbj + c - NB) * ldw; };
    double sum[NTL][4];
#pragma unroll
    for (int u = 0; u < NTL; ++u)
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[u][i] = 0.0;
    for (int k0 = warp < NWS ? 16 * warp : M; k0 < M; k0 += 16 * NWS) {
        uint32_t D[kDigits][NBM][4];
#pragma unroll
        for (int bm = 0; bm < NBM; ++bm)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = 16 * bm + 8 * h + g;
                const double* x = W + col(c);
                const int E = ec[c];
                unsigned long long v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = k0 + 2 * t + (i & 1) + 8 * (i >> 1);
                    const double y = r < M ? x[r] : 0.0;
                    v[i] = fixed_f64(y, E - exp_f64(y));
                }
                D[0][bm][h] = digit_pair<0>(v[0], v[1]); D[0][bm][2 + h] = digit_pair<0>(v[2], v[3]);
                D[1][bm][h] = digit_pair<1>(v[0], v[1]); D[1][bm][2 + h] = digit_pair<1>(v[2], v[3]);
                D[2][bm][h] = digit_pair<2>(v[0], v[1]); D[2][bm][2 + h] = digit_pair<2>(v[2], v[3]);
                D[3][bm][h] = digit_pair<3>(v[0], v[1]); D[3][bm][2 + h] = digit_pair<3>(v[2], v[3]);
                D[4][bm][h] = digit_pair<4>(v[0], v[1]); D[4][bm][2 + h] = digit_pair<4>(v[2], v[3]);
                D[5][bm][h] = digit_pair<5>(v[0], v[1]); D[5][bm][2 + h] = digit_pair<5>(v[2], v[3]);
            }
#pragma unroll
        for (int u = 0; u < NTL; ++u) {
            const int bm = u < 4 ? 0 : 1, nt = u < 4 ? u : u - 2, bn = nt >> 1, h = nt & 1;
            float acc[kWeights][4];
#pragma unroll
            for (int o = 0; o < kWeights; ++o)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[o][i] = 0.f;
#pragma unroll
            for (int j = 0; j < kDigits; ++j)
#pragma unroll
                for (int i = 0; i < kDigits; ++i)
                    if (i + j < kWeights) mma_f16(acc[i + j], D[i][bm], D[j][bn][h], D[j][bn][2 + h]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float c[kWeights];
#pragma unroll
                for (int o = 0; o < kWeights; ++o) c[o] = acc[o][i];
                const int rr = 16 * bm + g + 8 * (i >> 1), cc = 8 * nt + 2 * t + (i & 1);
                sum[u][i] += fixed_to_f64(combine_weights(c), ec[rr] + ec[cc] - 2150 + 51);
            }
        }
    }
    for (int w = 0; w < NWS; ++w) {
        if (warp == w) {
#pragma unroll
            for (int u = 0; u < NTL; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int bm = u < 4 ? 0 : 1, nt = u < 4 ? u : u - 2;
                    const int rr = 16 * bm + g + 8 * (i >> 1), cc = 8 * nt + 2 * t + (i & 1);
                    if (rr > cc) continue;                 // lower entries: the mirror of an upper one
                    const double x = w ? G[rr + cc * LDG] + sum[u][i] : sum[u][i];
                    G[rr + cc * LDG] = x;
                    G[cc + rr * LDG] = x;
                }
        }
        named_sync(bar, GT);
    }
}

// Exponents of the columns' norms from the Gram block's diagonal (of 2^-511
// where the square underflows): the scales of the update.
__device__ __forceinline__ int norm_exponent_f64(double gkk) { return (max(exp_f64(gkk), 1) + 1023) / 2; }

// J (2 NB x 2 NB, column stride ldj) for the update of columns scaled by 2^-ek[k]
// (ek null: unscaled): B fragments of the digits of J_kc 2^(ek[k] - fc[c]), fc[c]
// the largest exponent of column c.  Jd[((d * KS + ks) * NT + nt) * 32 + lane], KS
// = NB / 8 steps of 16, NT = NB / 4 tiles of 8 columns: 12 KB (NB = 8: 3 KB; complex:
// twice that).  GT threads; the caller synchronises.
template <class T, int NB>
__host__ __device__ constexpr int j_digit_bytes() {
    return (Traits<T>::kComplex ? 2 : 1) * kDigits * (NB / 8) * (NB / 4) * 32 * 8;
}
template <int NB, int GT>
__device__ __forceinline__ void j_digits_f64(const double* J, int ldj, const int* ek, uint2* Jd, int* fc, int gt) {
    const int warp = gt >> 5, lane = gt & 31, g = lane >> 2, t = lane & 3;
    constexpr int KS = NB / 8, NT = NB / 4;
    for (int nt = warp; nt < NT; nt += GT / 32) {
        const int c = 8 * nt + g;
        double x[4 * KS];
        int e[4 * KS], f = kNoExp;
#pragma unroll
        for (int i = 0; i < 4 * KS; ++i) {
            const int k = 16 * (i >> 2) + 2 * t + (i & 1) + 8 * ((i >> 1) & 1);
            x[i] = J[k + c * ldj];
            e[i] = exp_f64(x[i]) + (ek ? ek[k] : 0);
            f = max(f, e[i]);
        }
        f = max(f, __shfl_xor_sync(0xffffffffu, f, 1));
        f = max(f, __shfl_xor_sync(0xffffffffu, f, 2));
        if (t == 0) fc[c] = f;
        unsigned long long v[4 * KS];
#pragma unroll
        for (int i = 0; i < 4 * KS; ++i) v[i] = fixed_f64(x[i], f - e[i]);
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            uint2* o = Jd + (ks * NT + nt) * 32 + lane;
            o[0 * KS * NT * 32] = make_uint2(digit_pair<0>(v[4 * ks], v[4 * ks + 1]), digit_pair<0>(v[4 * ks + 2], v[4 * ks + 3]));
            o[1 * KS * NT * 32] = make_uint2(digit_pair<1>(v[4 * ks], v[4 * ks + 1]), digit_pair<1>(v[4 * ks + 2], v[4 * ks + 3]));
            o[2 * KS * NT * 32] = make_uint2(digit_pair<2>(v[4 * ks], v[4 * ks + 1]), digit_pair<2>(v[4 * ks + 2], v[4 * ks + 3]));
            o[3 * KS * NT * 32] = make_uint2(digit_pair<3>(v[4 * ks], v[4 * ks + 1]), digit_pair<3>(v[4 * ks + 2], v[4 * ks + 3]));
            o[4 * KS * NT * 32] = make_uint2(digit_pair<4>(v[4 * ks], v[4 * ks + 1]), digit_pair<4>(v[4 * ks + 2], v[4 * ks + 3]));
            o[5 * KS * NT * 32] = make_uint2(digit_pair<5>(v[4 * ks], v[4 * ks + 1]), digit_pair<5>(v[4 * ks + 2], v[4 * ks + 3]));
        }
    }
}

// A warp's 16 rows of an operand times the 2 NB x 2 NB matrix of j_digits_f64 (for
// the same ek).  load(h, k): entry k of row g + 8 h; store(nt, i, y): element i of
// the 16 x 8 output tile nt in the C layout.  All loads come before the first
// store.  U: tiles unrolled (NT where the caller indexes registers by nt).
template <int NB, int U, class Load, class Store>
__device__ __forceinline__ void rows_times_digits(Load load, Store store, const int* ek, const uint2* Jd, const int* fc,
                                                  int lane) {
    const int t = lane & 3;
    constexpr int KS = NB / 8, NT = NB / 4;
    uint32_t A[kDigits][KS][4];
    int Ea = kNoExp, Eb = kNoExp;
    {
        double x[2][4 * KS];                               // [row][entry]
        int e[2][4 * KS];
#pragma unroll
        for (int i = 0; i < 4 * KS; ++i) {
            const int k = 16 * (i >> 2) + 2 * t + (i & 1) + 8 * ((i >> 1) & 1);
            x[0][i] = load(0, k);
            x[1][i] = load(1, k);
            const int sc = ek ? ek[k] : 0;
            e[0][i] = exp_f64(x[0][i]);
            e[1][i] = exp_f64(x[1][i]);
            if (e[0][i] != kNoExp) e[0][i] -= sc;          // a zero does not count, whatever its column's scale
            if (e[1][i] != kNoExp) e[1][i] -= sc;
            Ea = max(Ea, e[0][i]);
            Eb = max(Eb, e[1][i]);
        }
        Ea = max(Ea, __shfl_xor_sync(0xffffffffu, Ea, 1));
        Eb = max(Eb, __shfl_xor_sync(0xffffffffu, Eb, 1));
        Ea = max(Ea, __shfl_xor_sync(0xffffffffu, Ea, 2));
        Eb = max(Eb, __shfl_xor_sync(0xffffffffu, Eb, 2));
#pragma unroll
        for (int p = 0; p < 2 * KS; ++p) {                 // entry pairs (2p, 2p + 1): k-step p / 2, half p % 2
            const unsigned long long a0 = fixed_f64(x[0][2 * p], Ea - e[0][2 * p]), a1 = fixed_f64(x[0][2 * p + 1], Ea - e[0][2 * p + 1]);
            const unsigned long long b0 = fixed_f64(x[1][2 * p], Eb - e[1][2 * p]), b1 = fixed_f64(x[1][2 * p + 1], Eb - e[1][2 * p + 1]);
            const int ks = p >> 1, h = 2 * (p & 1);
            A[0][ks][h] = digit_pair<0>(a0, a1); A[0][ks][h + 1] = digit_pair<0>(b0, b1);
            A[1][ks][h] = digit_pair<1>(a0, a1); A[1][ks][h + 1] = digit_pair<1>(b0, b1);
            A[2][ks][h] = digit_pair<2>(a0, a1); A[2][ks][h + 1] = digit_pair<2>(b0, b1);
            A[3][ks][h] = digit_pair<3>(a0, a1); A[3][ks][h + 1] = digit_pair<3>(b0, b1);
            A[4][ks][h] = digit_pair<4>(a0, a1); A[4][ks][h + 1] = digit_pair<4>(b0, b1);
            A[5][ks][h] = digit_pair<5>(a0, a1); A[5][ks][h + 1] = digit_pair<5>(b0, b1);
        }
    }
    __syncwarp();
#pragma unroll U
    for (int nt = 0; nt < NT; ++nt) {
        float acc[kWeights][4];
#pragma unroll
        for (int o = 0; o < kWeights; ++o)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[o][i] = 0.f;
#pragma unroll
        for (int j = 0; j < kDigits; ++j) {
            uint2 bj[KS];
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) bj[ks] = Jd[((j * KS + ks) * NT + nt) * 32 + lane];
#pragma unroll
            for (int i = 0; i < kDigits; ++i) {
                if (i + j >= kWeights) continue;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) mma_f16(acc[i + j], A[i][ks], bj[ks].x, bj[ks].y);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float c[kWeights];
#pragma unroll
            for (int o = 0; o < kWeights; ++o) c[o] = acc[o][i];
            const int cc = 8 * nt + 2 * t + (i & 1);
            // x = int 2^(E - 1075), J = int 2^(f - 1075), the integers' product T 2^51
            const double y = fixed_to_f64(combine_weights(c), (i < 2 ? Ea : Eb) + fc[cc] - 2150 + 51);
            store(nt, i, y);
        }
    }
}

// Rows [r0, r0 + 16) of a column-major X (rows valid below `rows`), columns
// [cbi, cbi + NB) and [cbj, cbj + NB), times J in place, with the fragments of
// j_digits_f64 for the same ek.  One warp; it reads all its inputs before it
// writes any output, and no other warp touches these rows.
template <int NB>
__device__ __forceinline__ void update_rows_f64(double* X, long long ld, int rows, int r0, int cbi, int cbj, const int* ek,
                                                const uint2* Jd, const int* fc, int lane) {
    const int t = lane & 3, ra = r0 + (lane >> 2), rb = ra + 8;
    auto col = [&](int c) { return (long long)(c < NB ? cbi + c : cbj + c - NB) * ld; };
    rows_times_digits<NB, 1>(
        [&](int h, int k) { const int r = h ? rb : ra; return r < rows ? X[r + col(k)] : 0.0; },
        [&](int nt, int i, double y) {
            const int r = i < 2 ? ra : rb;
            if (r < rows) X[r + col(8 * nt + 2 * t + (i & 1))] = y;
        },
        ek, Jd, fc, lane);
}

// ---- complex128 -----------------------------------------------------------------
// The same with real and imaginary parts, one exponent for both:
//   G = P^H P:  Re = Pr^T Pr + Pi^T Pi,  Im = Pr^T Pi - Pi^T Pr
//   P J:        Re = Pr Jr - Pi Ji,      Im = Pr Ji + Pi Jr
// Each real product has its own accumulators (two together could pass 2^24); the
// two integers of a part are added before the one rounding.  500 of 75x50 on chip: 48.5 ms on
// the FP64 pipe, 30.0 ms; 1000 of 64x64 in rounds 94.9 -> 53.4 ms.
__device__ __forceinline__ int exp_c128(double2 x) { return max(exp_f64(x.x), exp_f64(x.y)); }
// x's two parts relative to exponent E (each with its own distance to it)
__device__ __forceinline__ unsigned long long fixed_part(double x, int E, int sc) { return fixed_f64(x, E - (exp_f64(x) - sc)); }

template <int NB, int GT>
__device__ __forceinline__ void column_exponents_f64(const double2* W, long long ldw, int M, int cbi, int cbj, int* ec,
                                                     int gt) {
    constexpr int P = GT / (2 * NB);
    static_assert(P >= 1 && P <= 32 && (P & (P - 1)) == 0, "threads a column");
    const int c = gt / P, q = gt % P;
    const double2* x = W + (c < NB ? cbi + c : cbj + c - NB) * ldw;
    int e = kNoExp;
    for (int r = q; r < M; r += P) e = max(e, exp_c128(x[r]));
#pragma unroll
    for (int o = 1; o < P; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if (q == 0) ec[c] = e;
}

// the digits of four values (a fragment's two pairs) into words h and 2 + h
template <int I = 0>
__device__ __forceinline__ void digits4(const unsigned long long (&v)[4], uint32_t (&lo)[kDigits], uint32_t (&hi)[kDigits]) {
    if constexpr (I < kDigits) {
        lo[I] = digit_pair<I>(v[0], v[1]);
        hi[I] = digit_pair<I>(v[2], v[3]);
        digits4<I + 1>(v, lo, hi);
    }
}

// acc <- all digit products of weight below kWeights of fragments A and B
template <int KS>
__device__ __forceinline__ void digit_products(float (&acc)[kWeights][4], const uint32_t (&A)[kDigits][KS][4],
                                               const uint2* Bd, int bstride, int kstride, int lane) {
#pragma unroll
    for (int o = 0; o < kWeights; ++o)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[o][i] = 0.f;
#pragma unroll
    for (int j = 0; j < kDigits; ++j)
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            const uint2 b = Bd[j * bstride + ks * kstride + lane];
#pragma unroll
            for (int i = 0; i < kDigits; ++i)
                if (i + j < kWeights) mma_f16(acc[i + j], A[i][ks], b.x, b.y);
        }
}
__device__ __forceinline__ long long combined(const float (&acc)[kWeights][4], int i) {
    float c[kWeights];
#pragma unroll
    for (int o = 0; o < kWeights; ++o) c[o] = acc[o][i];
    return combine_weights(c);
}

// One pass of the Gram block: the tiles of 16-row block BM (columns 8 nt, nt from
// 2 BM on), as gram_f64_split.  Two passes keep a warp's sums in registers.
template <int NB, int GT, int LDG, int BM>
__device__ __forceinline__ void gram_c128_pass(const double2* W, long long ldw, int M, int cbi, int cbj, const int* ec,
                                               double2* G, int gt, int bar) {
    constexpr int NBM = 2 * NB / 16, NT0 = 2 * BM, NTL = 2 * (NBM - BM), NWS = NBM == 2 ? 4 : 2;
    static_assert(GT >= 32 * NWS, "the summing warps");
    const int warp = gt >> 5, lane = gt & 31, g = lane >> 2, t = lane & 3;
    auto col = [&](int c) { return (c < NB ? cbi + c : cbj + c - NB) * ldw; };
    double sr[NTL][4], si[NTL][4];
#pragma unroll
    for (int u = 0; u < NTL; ++u)
#pragma unroll
        for (int i = 0; i < 4; ++i) sr[u][i] = si[u][i] = 0.0;
    for (int k0 = warp < NWS ? 16 * warp : M; k0 < M; k0 += 16 * NWS) {
        uint32_t Dr[kDigits][NBM - BM][4], Di[kDigits][NBM - BM][4];
#pragma unroll
        for (int bm = BM; bm < NBM; ++bm)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = 16 * bm + 8 * h + g, E = ec[c];
                const double2* x = W + col(c);
                unsigned long long vr[4], vi[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = k0 + 2 * t + (i & 1) + 8 * (i >> 1);
                    const double2 y = r < M ? x[r] : make_double2(0.0, 0.0);
                    vr[i] = fixed_part(y.x, E, 0);
                    vi[i] = fixed_part(y.y, E, 0);
                }
                uint32_t lo[kDigits], hi[kDigits];
                digits4(vr, lo, hi);
#pragma unroll
                for (int d = 0; d < kDigits; ++d) { Dr[d][bm - BM][h] = lo[d]; Dr[d][bm - BM][2 + h] = hi[d]; }
                digits4(vi, lo, hi);
#pragma unroll
                for (int d = 0; d < kDigits; ++d) { Di[d][bm - BM][h] = lo[d]; Di[d][bm - BM][2 + h] = hi[d]; }
            }
        auto product = [&](float (&acc)[kWeights][4], const uint32_t (&A)[kDigits][NBM - BM][4],
                           const uint32_t (&B)[kDigits][NBM - BM][4], int bn, int h) {
#pragma unroll
            for (int o = 0; o < kWeights; ++o)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[o][i] = 0.f;
#pragma unroll
            for (int j = 0; j < kDigits; ++j)
#pragma unroll
                for (int i = 0; i < kDigits; ++i)
                    if (i + j < kWeights) mma_f16(acc[i + j], A[i][0], B[j][bn][h], B[j][bn][2 + h]);
        };
#pragma unroll
        for (int u = 0; u < NTL; ++u) {
            const int nt = NT0 + u, bn = (nt >> 1) - BM, h = nt & 1;
            float a1[kWeights][4], a2[kWeights][4];
            product(a1, Dr, Dr, bn, h);
            product(a2, Di, Di, bn, h);
            int s[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rr = 16 * BM + g + 8 * (i >> 1), cc = 8 * nt + 2 * t + (i & 1);
                s[i] = ec[rr] + ec[cc] - 2150 + 51;
                sr[u][i] += fixed_to_f64(combined(a1, i) + combined(a2, i), s[i]);
            }
            product(a1, Dr, Di, bn, h);
            product(a2, Di, Dr, bn, h);
#pragma unroll
            for (int i = 0; i < 4; ++i) si[u][i] += fixed_to_f64(combined(a1, i) - combined(a2, i), s[i]);
        }
    }
    for (int w = 0; w < NWS; ++w) {
        if (warp == w) {
#pragma unroll
            for (int u = 0; u < NTL; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int rr = 16 * BM + g + 8 * (i >> 1), cc = 8 * (NT0 + u) + 2 * t + (i & 1);
                    if (rr > cc) continue;                 // lower entries: the mirror of an upper one
                    double2 x = make_double2(sr[u][i], rr == cc ? 0.0 : si[u][i]);
                    if (w) x = add(G[rr + cc * LDG], x);
                    G[rr + cc * LDG] = x;
                    G[cc + rr * LDG] = conj_s(x);
                }
        }
        named_sync(bar, GT);
    }
}
template <int NB, int GT, int LDG>
__device__ __forceinline__ void gram_f64_split(const double2* W, long long ldw, int M, int cbi, int cbj, const int* ec,
                                               double2* G, int gt, int bar) {
    gram_c128_pass<NB, GT, LDG, 0>(W, ldw, M, cbi, cbj, ec, G, gt, bar);
    if constexpr (NB == 16) gram_c128_pass<NB, GT, LDG, 1>(W, ldw, M, cbi, cbj, ec, G, gt, bar);
}

// Digits of Jr, then of Ji, each in the layout of the real form.
template <int NB, int GT>
__device__ __forceinline__ void j_digits_f64(const double2* J, int ldj, const int* ek, uint2* Jd, int* fc, int gt) {
    constexpr int KS = NB / 8, NT = NB / 4, F = kDigits * KS * NT * 32;
    const int warp = gt >> 5, lane = gt & 31, g = lane >> 2, t = lane & 3;
    for (int nt = warp; nt < NT; nt += GT / 32) {
        const int c = 8 * nt + g;
        double2 x[4 * KS];
        int sc[4 * KS], f = kNoExp;
#pragma unroll
        for (int i = 0; i < 4 * KS; ++i) {
            const int k = 16 * (i >> 2) + 2 * t + (i & 1) + 8 * ((i >> 1) & 1);
            x[i] = J[k + c * ldj];
            sc[i] = ek ? -ek[k] : 0;
            f = max(f, exp_c128(x[i]) - sc[i]);
        }
        f = max(f, __shfl_xor_sync(0xffffffffu, f, 1));
        f = max(f, __shfl_xor_sync(0xffffffffu, f, 2));
        if (t == 0) fc[c] = f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                unsigned long long v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    v[i] = fixed_part(part ? x[4 * ks + i].y : x[4 * ks + i].x, f, sc[4 * ks + i]);
                uint32_t lo[kDigits], hi[kDigits];
                digits4(v, lo, hi);
#pragma unroll
                for (int d = 0; d < kDigits; ++d) Jd[part * F + ((d * KS + ks) * NT + nt) * 32 + lane] = make_uint2(lo[d], hi[d]);
            }
    }
}

template <int NB>
__device__ __forceinline__ void update_rows_f64(double2* X, long long ld, int rows, int r0, int cbi, int cbj, const int* ek,
                                                const uint2* Jd, const int* fc, int lane) {
    constexpr int KS = NB / 8, NT = NB / 4, F = kDigits * KS * NT * 32;
    const int g = lane >> 2, t = lane & 3, ra = r0 + g, rb = r0 + g + 8;
    auto col = [&](int c) { return (long long)(c < NB ? cbi + c : cbj + c - NB) * ld; };
    uint32_t Ar[kDigits][KS][4], Ai[kDigits][KS][4];
    int E[2] = {kNoExp, kNoExp};
    {
        double2 x[2][4 * KS];
        int sc[4 * KS];
#pragma unroll
        for (int i = 0; i < 4 * KS; ++i) {
            const int k = 16 * (i >> 2) + 2 * t + (i & 1) + 8 * ((i >> 1) & 1);
            const long long o = col(k);
            sc[i] = ek ? ek[k] : 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = h ? rb : ra;
                x[h][i] = r < rows ? X[r + o] : make_double2(0.0, 0.0);
                const int e = exp_c128(x[h][i]);
                if (e != kNoExp) E[h] = max(E[h], e - sc[i]);      // a zero does not count, whatever its column's scale
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            E[h] = max(E[h], __shfl_xor_sync(0xffffffffu, E[h], 1));
            E[h] = max(E[h], __shfl_xor_sync(0xffffffffu, E[h], 2));
        }
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned long long vr[4], vi[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    vr[i] = fixed_part(x[h][4 * ks + i].x, E[h], sc[4 * ks + i]);
                    vi[i] = fixed_part(x[h][4 * ks + i].y, E[h], sc[4 * ks + i]);
                }
                uint32_t lo[kDigits], hi[kDigits];
                digits4(vr, lo, hi);
#pragma unroll
                for (int d = 0; d < kDigits; ++d) { Ar[d][ks][h] = lo[d]; Ar[d][ks][2 + h] = hi[d]; }
                digits4(vi, lo, hi);
#pragma unroll
                for (int d = 0; d < kDigits; ++d) { Ai[d][ks][h] = lo[d]; Ai[d][ks][2 + h] = hi[d]; }
            }
    }
    __syncwarp();
    for (int nt = 0; nt < NT; ++nt) {
        const uint2* Jr = Jd + nt * 32;
        const uint2* Ji = Jr + F;
        float a1[kWeights][4], a2[kWeights][4];
        double yr[4];
        int s[4];
        digit_products<KS>(a1, Ar, Jr, KS * NT * 32, NT * 32, lane);
        digit_products<KS>(a2, Ai, Ji, KS * NT * 32, NT * 32, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            s[i] = E[i >> 1] + fc[8 * nt + 2 * t + (i & 1)] - 2150 + 51;
            yr[i] = fixed_to_f64(combined(a1, i) - combined(a2, i), s[i]);
        }
        digit_products<KS>(a1, Ar, Ji, KS * NT * 32, NT * 32, lane);
        digit_products<KS>(a2, Ai, Jr, KS * NT * 32, NT * 32, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int cc = 8 * nt + 2 * t + (i & 1), r = i < 2 ? ra : rb;
            const double yi = fixed_to_f64(combined(a1, i) + combined(a2, i), s[i]);
            if (r < rows) X[r + col(cc)] = make_double2(yr[i], yi);
        }
    }
}

// S4/S5: [W_i W_j] <- [W_i W_j] J for rowsW rows of W (its columns scaled by
// their exponents ek) and [V_i V_j] <- [V_i V_j] J for rowsV rows of V (0: V not
// kept; unscaled), 16-row tiles tile0, tile0 + step .. dealt to the group's
// warps.  Jd: j_digit_bytes, fc: 2 NB ints, both in shared memory.
template <int NB, int GT, class T>
__device__ __forceinline__ void update_f64_split(T* W, long long ldw, int rowsW, T* V, long long ldv, int rowsV,
                                                 int cbi, int cbj, const T* J, int ldj, const int* ek, uint2* Jd,
                                                 int* fc, int gt, int bar, int block = 0, int blocks = 1) {
    constexpr int NWG = GT / 32;
    const int warp = gt >> 5, lane = gt & 31, tw = (rowsW + 15) / 16, tv = (rowsV + 15) / 16, step = NWG * blocks;
    if (block * NWG < tw) {
        j_digits_f64<NB, GT>(J, ldj, ek, Jd, fc, gt);
        named_sync(bar, GT);
        for (int t = block * NWG + warp; t < tw; t += step)
            update_rows_f64<NB>(W, ldw, rowsW, 16 * t, cbi, cbj, ek, Jd, fc, lane);
    }
    if (block * NWG < tv) {
        named_sync(bar, GT);
        j_digits_f64<NB, GT>(J, ldj, nullptr, Jd, fc, gt);
        named_sync(bar, GT);
        for (int t = block * NWG + warp; t < tv; t += step)
            update_rows_f64<NB>(V, ldv, rowsV, 16 * t, cbi, cbj, nullptr, Jd, fc, lane);
    }
}

// ---- matrices the digits do not serve -------------------------------------------
// The update's error in an entry is 2^-53 of its row's largest entry over its
// column's norm times the norm of the output column: small relative to each
// column, not to each row.  Where the rows' sizes differ that takes the relative
// accuracy of the smallest singular values, which multiply-adds keep.  Median
// over 24 matrices D B, 40 x 40, of the largest relative error of a singular value in
// units of u, with digits and on the FP64 pipe: D over 2^6 45 and 45, 2^10 85 and
// 49, 2^20 608 and 67, 2^40 5.8e3 and 76, 2^100 2.4e6 and 76.  So a matrix whose
// rows span more than 2^6 keeps the FP64 pipe (not inlined: the digit path keeps
// its registers).  So does a matrix with a column shorter than 2^-400: the update
// scales columns by their norms, which the Gram block's diagonal gives down to
// 2^-511 only; a column of 2^-540 kept 24 bits per update and one of 2^-570 none.
constexpr int kDigitRowSpan = 6;

// Whether a column of W (M x N, largest entry between 1 and 2) is shorter than
// 2^-400 and not zero.  Called by all NT threads; synchronised.
template <class T, int NT>
__device__ __forceinline__ bool short_column(const T* W, long long ldw, int M, int N) {
    const int lane = threadIdx.x & 31;
    bool any = false;
    for (int j = threadIdx.x >> 5; j < N; j += NT / 32) {
        double mx = 0;
        for (int r = lane; r < M; r += 32) mx = fmax(mx, maxabs(W[r + j * ldw]));
        mx = warp_max(mx);
        any |= mx > 0 && mx < 0x1p-400;
    }
    return __syncthreads_or(any) != 0;
}

template <class T, int NB, int GT>
__device__ __noinline__ void gram_f64_fma(const T* W, long long ldw, int M, int cbi, int cbj, T* G, int ldg, int gt) {
    gram_tiles_fma<T, NB, GT>(W, ldw, M, cbi, cbj, G, ldg, gt);
}
template <class T, int NB, int GT>
__device__ __noinline__ void update_f64_fma(T* W, long long ldw, int rowsW, T* V, long long ldv, int rowsV, int cbi, int cbj,
                                            const T* J, int ldj, int gt, int block, int blocks) {
    update_rows_fma<T, NB, GT>(W, ldw, rowsW, V, ldv, rowsV, cbi, cbj, J, ldj, gt, block, blocks);
}

}  // namespace bsvd
