// mixed.cu -- kernels of the mixed-precision path for FP64 output.
//
// FP64 results from mostly-FP32 work: the FP32 solver runs on an FP32 copy
// of A until its own convergence test passes, giving V32; this file's
// kernels then restore an orthonormal V in FP64 (Newton-Schulz steps
// V <- V - V (V^H V - I) / 2 from the widened V32, in real FP64 from 33 to 127 columns with a
// preconditioning and a first-order diagonalisation step between them) and
// form A_hat = A V in FP64; FP64 polish sweeps on A_hat, starting from that V, win the accuracy
// back (the FP64 test decides convergence).  On a GB300, whose FP64 rate is
// about 1/64 of its FP32 rate, the polish needs a few FP64 sweeps instead of
// the full count.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "jacobi_common.cuh"
#include "precondition.cuh"
#include "tc_f64.cuh"

namespace bsvd {

__device__ __forceinline__ float narrow_s(double x) { return __double2float_rn(x); }
__device__ __forceinline__ float2 narrow_s(double2 x) { return make_float2(__double2float_rn(x.x), __double2float_rn(x.y)); }
__device__ __forceinline__ double widen_s(float x) { return (double)x; }
__device__ __forceinline__ double2 widen_s(float2 x) { return make_double2((double)x.x, (double)x.y); }

constexpr int kMxThreads = 256;

// Matrix b of the launch: the caller's strided batch, or by id through the
// pointer array.
template <class T64>
__device__ __forceinline__ const T64* mixed_a(const MixedArgs& a, int b) {
    return a.Ap ? static_cast<const T64*>(a.Ap[a.index[b]]) : static_cast<const T64*>(a.A) + (long long)b * a.sA;
}

// A32 (M x N, ld M) = fl32(2^-ex A) or fl32(2^-ex A^H) when m < n, ex the
// exponent of max |a_ij| (exact scaling: FP32's range holds the result); plain64.
template <class T64, class T32>
__global__ void __launch_bounds__(kMxThreads) mx_convert(const MixedArgs a) {
    using R = Real<T64>;
    constexpr int NT = kMxThreads, NW = NT / 32;
    __shared__ R red[NW];
    __shared__ int ex_s, span_s[2 * NW];
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T64* A = mixed_a<T64>(a, b);
    const int lda = a.Ap ? a.ldap[a.index[b]] : a.lda;
    R mx = 0;
    for (int e = tid; e < a.m * a.n; e += NT) {
        const T64 x = A[(e % a.m) + (long long)(e / a.m) * lda];
        if (finite_s(x)) mx = fmax(mx, maxabs(x));
    }
    mx = warp_max(mx);
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    if (tid == 0) {
        R m2 = 0;
        for (int w = 0; w < NW; ++w) m2 = fmax(m2, red[w]);
        ex_s = m2 > 0 ? ilogb_r(m2) : 0;
    }
    __syncthreads();
    const int ex = ex_s;
    T32* A32 = static_cast<T32*>(a.A32) + (long long)b * a.M * a.N;
    for (int e = tid; e < a.m * a.n; e += NT) {
        const int i = e % a.m, j = e / a.m;
        const T64 x = scalb_s(A[i + (long long)j * lda], -ex);
        if (a.trans) A32[j + (long long)i * a.M] = narrow_s(conj_s(x));
        else         A32[i + (long long)j * a.M] = narrow_s(x);
    }
    const int span = row_span<T64, NT>(A, a.trans ? lda : 1, a.trans ? 1 : lda, a.M, a.N, span_s);
    if (tid == 0) a.plain64[b] = span > kDigitRowSpan;
}

// V <- V - V (V^H V - I) / 2 (N x N, ld N), from Vin to Vout; E is scratch.
// Synchronised on return.
template <class T64, int NT>
__device__ __forceinline__ void mx_newton_schulz(const T64* Vin, T64* Vout, T64* E, int N) {
    using R = Real<T64>;
    const int tid = threadIdx.x;
    for (int e = tid; e < N * (N + 1) / 2; e += NT) {
        int ca, cb;
        tri_index(e, ca, cb);
        T64 acc = make_s<T64>(0);
        for (int i = 0; i < N; ++i) acc = cfma(Vin[i + (long long)ca * N], Vin[i + (long long)cb * N], acc);
        if (ca == cb) acc = make_s<T64>(re(acc) - R(1));
        E[ca + (long long)cb * N] = acc;
        E[cb + (long long)ca * N] = conj_s(acc);
    }
    __syncthreads();
    for (int e = tid; e < N * N; e += NT) {
        const int i = e % N, k = e / N;
        T64 acc = make_s<T64>(0);
        for (int j = 0; j < N; ++j) acc = fma_s(Vin[i + (long long)j * N], E[j + (long long)k * N], acc);
        Vout[i + (long long)k * N] = sub(Vin[i + (long long)k * N], scale(acc, R(0.5)));
    }
    __syncthreads();
}

// V (N x N) orthonormal in FP64 from V32, close to the right singular vectors
// of A' = A or A^H; A_hat (M x N, ld M) = A' V.  One CTA per matrix on
// L2-resident buffers: V = widen(V32), two Newton-Schulz steps, A_hat = A' V.
template <class T64, class T32>
__global__ void __launch_bounds__(kMxThreads) mx_restore(const MixedArgs a) {
    constexpr int NT = kMxThreads;
    const int b = blockIdx.x, tid = threadIdx.x;
    const int M = a.M, N = a.N;
    const long long nn = (long long)N * N;
    const T32* V32 = static_cast<const T32*>(a.V32) + b * nn;
    T64* Va = static_cast<T64*>(a.V64) + b * nn;
    T64* Vb = static_cast<T64*>(a.Vtmp) + b * nn;
    T64* E = static_cast<T64*>(a.E) + b * nn;
    T64* Ah = static_cast<T64*>(a.Ahat) + (long long)b * M * N;
    const T64* A = mixed_a<T64>(a, b);
    const int lda = a.Ap ? a.ldap[a.index[b]] : a.lda;
    auto product = [&](const T64* V) {                     // A_hat = A' V
        for (int e = tid; e < M * N; e += NT) {
            const int i = e % M, k = e / M;
            T64 acc = make_s<T64>(0);
            for (int j = 0; j < N; ++j) {
                const T64 aij = a.trans ? conj_s(A[j + (long long)i * lda]) : A[i + (long long)j * lda];
                acc = fma_s(aij, V[j + (long long)k * N], acc);
            }
            Ah[i + (long long)k * M] = acc;
        }
        __syncthreads();
    };
    for (int e = tid; e < N * N; e += NT) Va[e] = widen_s(V32[e]);
    __syncthreads();
    mx_newton_schulz<T64, NT>(Va, Vb, E, N);
    mx_newton_schulz<T64, NT>(Vb, Va, E, N);
    product(Va);
}

// ---- the restoration tiled over the whole GPU (complex128, N >= kMxTiledN) ------
// For large N one CTA per matrix leaves most SMs idle for O(N^3) work, so the
// same steps run as 64 x 64 output tiles over (matrix, tile, tile) grids:
// widen, E = V^H V - I, V <- V - V E / 2 (twice), A_hat = A' V.  Each output
// keeps one accumulator summed over the contraction index in increasing
// order with the same multiply-adds as mx_restore.
constexpr int kMxBT = 64, kMxKC = 16, kMxTiledN = 128;

template <class T64, class T32>
__global__ void __launch_bounds__(kMxThreads) mx_widen(const MixedArgs a) {
    const long long nn = (long long)a.N * a.N;
    const T32* V32 = static_cast<const T32*>(a.V32) + blockIdx.x * nn;
    T64* Va = static_cast<T64*>(a.V64) + blockIdx.x * nn;
    for (long long e = blockIdx.y * (long long)kMxThreads + threadIdx.x; e < nn; e += (long long)gridDim.y * kMxThreads)
        Va[e] = widen_s(V32[e]);
}

// acc[u][v] += sum over the chunk of X(r0 + tr + 16u, k) Y(k, c0 + tc + 16v),
// X and Y staged as Xs[k][row], Ys[k][col]; conj_x: X entries conjugated.
template <class T, bool ConjX>
__device__ __forceinline__ void mx_mac(T (&acc)[4][4], const T (*Xs)[kMxBT + 1], const T (*Ys)[kMxBT + 1], int tr,
                                       int tc, int kc) {
    for (int k = 0; k < kc; ++k) {
        T x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = Xs[k][tr + 16 * u];
#pragma unroll
        for (int v = 0; v < 4; ++v) y[v] = Ys[k][tc + 16 * v];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = ConjX ? cfma(x[u], y[v], acc[u][v]) : fma_s(x[u], y[v], acc[u][v]);
    }
}

// E (N x N) = V^H V - I for V = V64 (it = 0, 2: the buffer holding the
// current iterate), upper tiles computed and mirrored.
template <class T64>
__global__ void __launch_bounds__(kMxThreads) mx_gram_tiled(const MixedArgs a, int cur) {
    using R = Real<T64>;
    const int b = blockIdx.x, ta = blockIdx.y, tb = blockIdx.z, tid = threadIdx.x, tr = tid & 15, tc = tid >> 4;
    if (ta > tb) return;
    const int N = a.N, r0 = ta * kMxBT, c0 = tb * kMxBT;
    const long long nn = (long long)N * N;
    const T64* V = static_cast<const T64*>(cur ? a.Vtmp : a.V64) + b * nn;
    T64* E = static_cast<T64*>(a.E) + b * nn;
    __shared__ T64 Xs[kMxKC][kMxBT + 1], Ys[kMxKC][kMxBT + 1];
    const T64 zero = make_s<T64>(0);
    T64 acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = zero;
    for (int i0 = 0; i0 < N; i0 += kMxKC) {
        for (int e = tid; e < kMxKC * kMxBT; e += kMxThreads) {
            const int kk = e % kMxKC, cc = e / kMxKC, i = i0 + kk;
            Xs[kk][cc] = (i < N && r0 + cc < N) ? V[i + (long long)(r0 + cc) * N] : zero;
            Ys[kk][cc] = (i < N && c0 + cc < N) ? V[i + (long long)(c0 + cc) * N] : zero;
        }
        __syncthreads();
        mx_mac<T64, true>(acc, Xs, Ys, tr, tc, min(kMxKC, N - i0));
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int r = r0 + tr + 16 * u, c = c0 + tc + 16 * v;
            if (r >= N || c >= N || r > c) continue;
            T64 x = acc[u][v];
            if (r == c) x = make_s<T64>(re(x) - R(1));
            E[r + (long long)c * N] = x;
            E[c + (long long)r * N] = conj_s(x);
        }
}

// Vnext = Vcur - Vcur E / 2 (cur = 0: V64 -> Vtmp; 1: Vtmp -> V64)
template <class T64>
__global__ void __launch_bounds__(kMxThreads) mx_ns_tiled(const MixedArgs a, int cur) {
    using R = Real<T64>;
    const int b = blockIdx.x, ti = blockIdx.y, tk = blockIdx.z, tid = threadIdx.x, tr = tid & 15, tc = tid >> 4;
    const int N = a.N, r0 = ti * kMxBT, c0 = tk * kMxBT;
    const long long nn = (long long)N * N;
    const T64* V = static_cast<const T64*>(cur ? a.Vtmp : a.V64) + b * nn;
    T64* Vn = static_cast<T64*>(cur ? a.V64 : a.Vtmp) + b * nn;
    const T64* E = static_cast<const T64*>(a.E) + b * nn;
    __shared__ T64 Xs[kMxKC][kMxBT + 1], Ys[kMxKC][kMxBT + 1];
    const T64 zero = make_s<T64>(0);
    T64 acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = zero;
    for (int j0 = 0; j0 < N; j0 += kMxKC) {
        for (int e = tid; e < kMxKC * kMxBT; e += kMxThreads) {
            const int kk = e / kMxBT, cc = e % kMxBT, j = j0 + kk;
            Xs[kk][cc] = (j < N && r0 + cc < N) ? V[(r0 + cc) + (long long)j * N] : zero;
            Ys[kk][cc] = (j < N && c0 + cc < N) ? E[j + (long long)(c0 + cc) * N] : zero;
        }
        __syncthreads();
        mx_mac<T64, false>(acc, Xs, Ys, tr, tc, min(kMxKC, N - j0));
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int i = r0 + tr + 16 * u, k = c0 + tc + 16 * v;
            if (i >= N || k >= N) continue;
            Vn[i + (long long)k * N] = sub(V[i + (long long)k * N], scale(acc[u][v], R(0.5)));
        }
}

// A_hat (M x N) = A' V64, A' = A or A^H
template <class T64>
__global__ void __launch_bounds__(kMxThreads) mx_ahat_tiled(const MixedArgs a) {
    const int b = blockIdx.x, ti = blockIdx.y, tk = blockIdx.z, tid = threadIdx.x, tr = tid & 15, tc = tid >> 4;
    const int M = a.M, N = a.N, r0 = ti * kMxBT, c0 = tk * kMxBT;
    const long long nn = (long long)N * N;
    const T64* A = mixed_a<T64>(a, b);
    const int lda = a.Ap ? a.ldap[a.index[b]] : a.lda;
    const T64* V = static_cast<const T64*>(a.V64) + b * nn;
    T64* Ah = static_cast<T64*>(a.Ahat) + (long long)b * M * N;
    __shared__ T64 Xs[kMxKC][kMxBT + 1], Ys[kMxKC][kMxBT + 1];
    const T64 zero = make_s<T64>(0);
    T64 acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = zero;
    for (int j0 = 0; j0 < N; j0 += kMxKC) {
        for (int e = tid; e < kMxKC * kMxBT; e += kMxThreads) {
            const int kk = e / kMxBT, cc = e % kMxBT, j = j0 + kk, i = r0 + cc;
            T64 x = zero;
            if (j < N && i < M) x = a.trans ? conj_s(A[j + (long long)i * lda]) : A[i + (long long)j * lda];
            Xs[kk][cc] = x;
            Ys[kk][cc] = (j < N && c0 + cc < N) ? V[j + (long long)(c0 + cc) * N] : zero;
        }
        __syncthreads();
        mx_mac<T64, false>(acc, Xs, Ys, tr, tc, min(kMxKC, N - j0));
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int i = r0 + tr + 16 * u, k = c0 + tc + 16 * v;
            if (i < M && k < N) Ah[i + (long long)k * M] = acc[u][v];
        }
}

template <class T64, class T32>
cudaError_t mixed_restore_tiled(const MixedArgs& a, int batch, cudaStream_t st) {
    const int tn = (a.N + kMxBT - 1) / kMxBT, tm = (a.M + kMxBT - 1) / kMxBT;
    const long long nn = (long long)a.N * a.N;
    const int wblocks = (int)std::min<long long>((nn + kMxThreads - 1) / kMxThreads, 1024);
    mx_widen<T64, T32><<<dim3(batch, wblocks), kMxThreads, 0, st>>>(a);
    for (int it = 0; it < 2; ++it) {      // two Newton-Schulz steps: V64 -> Vtmp -> V64
        mx_gram_tiled<T64><<<dim3(batch, tn, tn), kMxThreads, 0, st>>>(a, it);
        mx_ns_tiled<T64><<<dim3(batch, tn, tn), kMxThreads, 0, st>>>(a, it);
    }
    mx_ahat_tiled<T64><<<dim3(batch, tm, tn), kMxThreads, 0, st>>>(a);
    return cudaGetLastError();
}

// ---- the restoration in real FP64: products as FP16 digits ---------------------
// The steps of mx_restore, and up to 127 columns between a first Newton-Schulz
// step and three more:
//   A_hat = A' V (off-diagonal to 1e-7, FP32's accuracy, but O(1) relative to
//   short columns of a graded matrix); A_hat P = Q L Z^T, V <- V P Z
//   (precondition.cuh: contracts those by the squared ratio of the singular
//   values); V <- V (I + Omega), the first-order diagonalisation of L^T L
//   (antisymmetric, omega_ij = g_ij / (g_jj - g_ii) where that is below 1e-2;
//   closer pairs, and pairs of a row whose entries sum to more than 0.1, are
//   left to the sweeps): one product instead of a sweep's dependent rotations,
//   off-diagonals of 1e-7 become 1e-14.  V^T V - I is then Omega^T Omega, at
//   most 1e-2 in norm by the row sums, and the three Newton-Schulz steps that
//   follow (e -> 3/4 e^2) take it to 8e-5, 4e-9 and rounding.  The entries'
//   own limit does not bound it: with many nearly equal singular values
//   |Omega| reached 0.08, and two steps left V off by 1e-9.
// The FP64 sweeps that follow then need 2 sweeps instead of 4 on 128 x 64 with
// kappa = 1e6, 3.5 instead of 8 on the clustered 96 x 96 set.  Up to kMxPlainN
// columns the sweep saved costs less than the launches and that step: 2,000 of
// 16 x 16 1.25 ms plain and 1.80 so, of 32 x 32 3.68 and 4.59, one 32 x 32 0.56
// and 0.81; 40 x 40 10.5 (the first version) and 9.7, one 1.55 and 1.51.
// complex128 stays plain: in one CTA on the FP64 pipe the step made one 96 x 96
// 17.1 ms instead of 11.5.  Every product is a digit product
// (tc_f64.cuh) over (matrix, 64 rows, 32 columns) grids, 32 terms of the
// contraction at a time; the chunks' sums are added in FP64 in increasing
// order.  Per chunk a CTA stages both operands in shared memory, splits the
// right one into digits once, and each of its four warps splits and multiplies
// 16 rows.  A matrix whose rows span more than 2^6 takes multiply-adds on the same
// tiles (kDigitRowSpan: V's small entries count there).  2,000 of 96x96: the
// restoration 42 ms as one CTA a matrix on the FP64 pipe, 29.7 so: 9.9 in these
// products, 0.6 in mx_omega, 19.1 in mx_precondition.
enum MxOp {
    kMxGram,      // E = V^T V - I
    kMxGramL,     // E = L^T L, L the lower triangle in A_hat
    kMxNs,        // Vn = V - V E / 2
    kMxRefine,    // Vn = V (I + Omega), Omega in A_hat (mx_omega)
    kMxAhat,      // A_hat = A' V
};
constexpr int kMxDT = 64, kMxDC = 32, kMxDThreads = 128, kMxPlainN = 32;

// cur: 1 where the current V is Vtmp (the next one then goes to V64)
template <int OP>
__global__ void __launch_bounds__(kMxDThreads, 3) mx_digits(const MixedArgs a, int cur) {
    constexpr int LDA = kMxDT + 2, LDB = kMxDC + 1, NT = 4;
    static_assert(kMxDC == 32, "a chunk is 2 x 16 columns");
    __shared__ double As[kMxDC * LDA], Bs[kMxDC * LDB];
    __shared__ uint2 Jd[j_digit_bytes<double, 16>() / sizeof(uint2)];
    __shared__ int ek[kMxDC], fc[kMxDC], range;
    const int b = blockIdx.x, c0 = blockIdx.z * kMxDC, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = a.N, M = OP == kMxAhat ? a.M : N;
    const bool plain = a.plain64[b] != 0;
    const long long nn = (long long)N * N;
    const double* V = static_cast<const double*>(cur ? a.Vtmp : a.V64) + b * nn;
    double* Vn = static_cast<double*>(cur ? a.V64 : a.Vtmp) + b * nn;
    double* E = static_cast<double*>(a.E) + b * nn;
    double* Ah = static_cast<double*>(a.Ahat) + (long long)b * a.M * N;
    const double* A = mixed_a<double>(a, b);
    const int lda = a.Ap ? a.ldap[a.index[b]] : a.lda;
    auto left = [&](int r, int k) -> double {              // entry (r, k) of the left operand
        if (r >= M || k >= N) return 0.0;
        if (OP == kMxGram) return V[k + (long long)r * N];
        if (OP == kMxGramL) return k >= r ? Ah[k + (long long)r * a.M] : 0.0;
        if (OP == kMxAhat) return a.trans ? A[k + (long long)r * lda] : A[r + (long long)k * lda];
        return V[r + (long long)k * N];
    };
    auto right = [&](int k, int c) -> double {
        if (k >= N || c >= N) return 0.0;
        if (OP == kMxGram || OP == kMxAhat) return V[k + (long long)c * N];
        if (OP == kMxGramL) return k >= c ? Ah[k + (long long)c * a.M] : 0.0;
        if (OP == kMxNs) return E[k + (long long)c * N];
        return Ah[k + (long long)c * N];
    };
    const bool along_k = OP == kMxGram || OP == kMxGramL || (OP == kMxAhat && a.trans);   // the left operand's contiguous index
    for (int r0 = blockIdx.y * kMxDT; r0 < M; r0 += gridDim.y * kMxDT) {
        if ((OP == kMxGram || OP == kMxGramL) && r0 > c0 + kMxDC - 1) break;   // below the diagonal
        double sum[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) sum[nt][i] = 0.0;
        bool bad = false;                                  // not finite: the digits would hide it
        for (int k0 = OP == kMxGramL ? c0 / kMxDC * kMxDC : 0; k0 < N; k0 += kMxDC) {   // L: zero above row c0
            if (tid == 0) range = 0;
            __syncthreads();
            int big = 0;                                   // 1: entries near overflow, 2: some not tiny
            for (int e = tid; e < kMxDC * kMxDT; e += kMxDThreads) {
                const int k = along_k ? e % kMxDC : e / kMxDT, r = along_k ? e / kMxDC : e % kMxDT;
                const double x = left(r0 + r, k0 + k);
                As[k * LDA + r] = x;
                const int ex = exp_f64(x);
                big |= (ex > 2000 ? 1 : 0) | (ex > 300 ? 2 : 0);
                bad |= ex == 0x7ff;
            }
            for (int e = tid; e < kMxDC * kMxDC; e += kMxDThreads) {
                const int k = e % kMxDC, c = e / kMxDC;
                const double x = right(k0 + k, c0 + c);
                Bs[c * LDB + k] = x;
                bad |= exp_f64(x) == 0x7ff;
            }
            if (plain) {                                   // uniform over the CTA: multiply-adds, in order
                __syncthreads();
                const int rw = 16 * warp + (lane >> 2), t2 = 2 * (lane & 3);
                for (int k = 0; k < kMxDC; ++k) {
                    const double x0 = As[k * LDA + rw], x1 = As[k * LDA + rw + 8];
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const double y0 = Bs[(8 * nt + t2) * LDB + k], y1 = Bs[(8 * nt + t2 + 1) * LDB + k];
                        sum[nt][0] = fma(x0, y0, sum[nt][0]);
                        sum[nt][1] = fma(x0, y1, sum[nt][1]);
                        sum[nt][2] = fma(x1, y0, sum[nt][2]);
                        sum[nt][3] = fma(x1, y1, sum[nt][3]);
                    }
                }
                __syncthreads();
                continue;
            }
            if (OP == kMxAhat) {
                big = __reduce_or_sync(0xffffffffu, big);
                if (lane == 0 && big) atomicOr(&range, big);
            }
            __syncthreads();
            bool scaled = false;
            double down = 1.0;
            if (OP == kMxAhat) {
                // A carries the caller's scale: a power of two takes entries near either
                // end of FP64's range, whose digits or products would leave it, inside
                const int rg = range;
                scaled = (rg & 1) || !(rg & 2);
                down = rg & 1 ? 0x1p64 : 0x1p-600;
                if (scaled) {
                    const double up = rg & 1 ? 0x1p-64 : 0x1p600;
                    for (int e = tid; e < kMxDC * kMxDT; e += kMxDThreads) As[e / kMxDT * LDA + e % kMxDT] *= up;
                    __syncthreads();
                }
                // columns of A on one scale, V's rows on its inverse: A_hat keeps short columns
                const int k = tid >> 2;
                int e = kNoExp;
                for (int r = tid & 3; r < kMxDT; r += 4) e = max(e, exp_f64(As[k * LDA + r]));
                e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
                e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
                if ((tid & 3) == 0) ek[k] = e;
                __syncthreads();
            }
            const int* const es = OP == kMxAhat ? ek : nullptr;
            j_digits_f64<16, kMxDThreads>(Bs, LDB, es, Jd, fc, tid);
            __syncthreads();
            const int rw = 16 * warp + (lane >> 2);
            if (r0 + 16 * warp < M && !((OP == kMxGram || OP == kMxGramL) && r0 + 16 * warp > c0 + kMxDC - 1))
                rows_times_digits<16, NT>([&](int h, int k) { return As[k * LDA + rw + 8 * h]; },
                                          [&](int nt, int i, double y) {
                                              if (OP == kMxAhat && scaled) y *= down;
                                              sum[nt][i] += y;
                                          },
                                          es, Jd, fc, lane);
            __syncthreads();
        }
        bad = __syncthreads_or(bad);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r0 + 16 * warp + (lane >> 2) + (i < 2 ? 0 : 8), c = c0 + 8 * nt + 2 * (lane & 3) + (i & 1);
                if (r >= M || c >= N) continue;
                const double y = bad ? __longlong_as_double(0x7ff8000000000000ll) : sum[nt][i];
                if (OP == kMxGram || OP == kMxGramL) {
                    if (r > c) continue;
                    const double x = OP == kMxGram && r == c ? y - 1.0 : y;
                    E[r + (long long)c * N] = x;
                    E[c + (long long)r * N] = x;
                } else if (OP == kMxAhat) {
                    Ah[r + (long long)c * M] = y;
                } else {
                    const double v = V[r + (long long)c * N];
                    Vn[r + (long long)c * N] = OP == kMxNs ? v - 0.5 * y : v + y;
                }
            }
    }
}

// A_hat P = Q L Z^T with V64 -> Vtmp = V64 P Z, L in A_hat.  Declined (or A_hat too
// large to square, or V's small entries count): Vtmp = V64 and L = 0, for which the
// first-order step is none.  Only V is kept of it, orthonormal whatever the rows of
// A_hat span: its rows may.
// On L2-resident buffers: about half of its 19.1 ms on 2,000 of 96x96 is the FP64
// pipe's; with A_hat in shared memory (two CTAs an SM instead of four) 19.5 ms.
__global__ void __launch_bounds__(kMxThreads) mx_precondition(const MixedArgs a) {
    constexpr int NT = kMxThreads;
    extern __shared__ __align__(16) unsigned char smem[];
    const int b = blockIdx.x, tid = threadIdx.x, M = a.M, N = a.N;
    const long long nn = (long long)N * N;
    double* V = static_cast<double*>(a.V64) + b * nn;
    double* Vn = static_cast<double*>(a.Vtmp) + b * nn;
    double* Ah = static_cast<double*>(a.Ahat) + (long long)b * M * N;
    int wide = 0;
    for (int e = tid; e < M * N; e += NT) wide |= !(fabs(Ah[e]) < 1e100);
    if (!__syncthreads_or(wide) && !a.plain64[b] &&
        precondition<double, NT>(Ah, M, M, N, Vn, N, V, N, nullptr, 0, PreScratch<double>(smem, N)) == Pre::kDone)
        return;
    __syncthreads();
    for (int e = tid; e < N * N; e += NT) {
        Vn[e] = V[e];
        Ah[e % N + (long long)(e / N) * M] = 0.0;
    }
}

// Omega (N x N, ld N) of E = L^T L into A_hat, whose L is no longer needed: the
// entries below 1e-2, without the rows and columns whose entries sum to more
// than 0.1.  One CTA per matrix; dynamic shared memory: 2 N doubles.
constexpr double kMxOmegaEntry = 1e-2, kMxOmegaRow = 0.1;
__global__ void __launch_bounds__(kMxThreads) mx_omega(const MixedArgs a) {
    constexpr int NT = kMxThreads, NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    double* const diag = reinterpret_cast<double*>(smem);
    double* const sum = diag + a.N;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, N = a.N;
    const double* E = static_cast<const double*>(a.E) + b * (long long)N * N;
    double* Om = static_cast<double*>(a.Ahat) + (long long)b * a.M * N;
    for (int i = tid; i < N; i += NT) diag[i] = E[i + (long long)i * N];
    __syncthreads();
    bool large = false;
    for (int c = warp; c < N; c += NW) {                   // a column's sum is its row's: |Omega| is symmetric
        double s = 0;
        for (int k = lane; k < N; k += 32) {
            const double g = E[k + (long long)c * N], den = diag[c] - diag[k];
            const double w = k != c && fabs(g) < kMxOmegaEntry * fabs(den) ? g / den : 0.0;
            Om[k + (long long)c * N] = w;
            s += fabs(w);
        }
        s = warp_sum(s);
        if (lane == 0) sum[c] = s;
        large |= !(s <= kMxOmegaRow);
    }
    if (!__syncthreads_or(large)) return;
    for (int e = tid; e < N * N; e += NT)
        if (!(sum[e % N] <= kMxOmegaRow && sum[e / N] <= kMxOmegaRow)) Om[e] = 0.0;
}

template <class T64, class T32>
cudaError_t mixed_restore_digits(const MixedArgs& a, int batch, cudaStream_t st) {
    const int tn = (a.N + kMxDT - 1) / kMxDT, tc = (a.N + kMxDC - 1) / kMxDC, tm = std::min((a.M + kMxDT - 1) / kMxDT, 65535);
    const long long nn = (long long)a.N * a.N;
    const int wblocks = (int)std::min<long long>((nn + kMxThreads - 1) / kMxThreads, 1024);
    const dim3 sq(batch, tn, tc), rect(batch, tm, tc);
    MixedArgs w = a;                                       // V64 and Vtmp the other way round
    w.V64 = a.Vtmp;
    w.Vtmp = a.V64;
    auto newton_schulz = [&](const MixedArgs& x, int cur) {
        mx_digits<kMxGram><<<sq, kMxDThreads, 0, st>>>(x, cur);
        mx_digits<kMxNs><<<sq, kMxDThreads, 0, st>>>(x, cur);
    };
    mx_widen<T64, T32><<<dim3(batch, wblocks), kMxThreads, 0, st>>>(a);
    if (a.N < kMxTiledN) {
        newton_schulz(a, 0);                               // -> Vtmp
        mx_digits<kMxAhat><<<rect, kMxDThreads, 0, st>>>(w, 0);
        mx_precondition<<<batch, kMxThreads, (size_t)PreScratch<double>::bytes(a.N), st>>>(w);   // -> V64
        mx_digits<kMxGramL><<<sq, kMxDThreads, 0, st>>>(a, 0);
        mx_omega<<<batch, kMxThreads, 2 * a.N * sizeof(double), st>>>(a);
        mx_digits<kMxRefine><<<sq, kMxDThreads, 0, st>>>(a, 0);                                   // -> Vtmp
        newton_schulz(a, 1);                               // -> V64
    }
    newton_schulz(a, 0);
    newton_schulz(a, 1);
    mx_digits<kMxAhat><<<rect, kMxDThreads, 0, st>>>(a, 0);
    return cudaGetLastError();
}

template <class T64, class T32>
cudaError_t mixed_prepare(const MixedArgs& a, int batch, cudaStream_t st) {
    mx_convert<T64, T32><<<batch, kMxThreads, 0, st>>>(a);
    return cudaGetLastError();
}

template <class T64, class T32>
cudaError_t mixed_restore(const MixedArgs& a, int batch, cudaStream_t st) {
    if constexpr (sizeof(T64) == 8)
        if (a.N > kMxPlainN) return mixed_restore_digits<T64, T32>(a, batch, st);
    if constexpr (sizeof(T64) == 16)
        if (a.N >= kMxTiledN) return mixed_restore_tiled<T64, T32>(a, batch, st);
    mx_restore<T64, T32><<<batch, kMxThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t mixed_prepare_d(const MixedArgs& a, int batch, cudaStream_t st) { return mixed_prepare<double, float>(a, batch, st); }
cudaError_t mixed_prepare_z(const MixedArgs& a, int batch, cudaStream_t st) { return mixed_prepare<double2, float2>(a, batch, st); }
cudaError_t mixed_restore_d(const MixedArgs& a, int batch, cudaStream_t st) { return mixed_restore<double, float>(a, batch, st); }
cudaError_t mixed_restore_z(const MixedArgs& a, int batch, cudaStream_t st) { return mixed_restore<double2, float2>(a, batch, st); }

}  // namespace bsvd
