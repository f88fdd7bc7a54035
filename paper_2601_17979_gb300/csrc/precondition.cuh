// precondition.cuh -- orthogonal preconditioning of the one-sided Jacobi
// sweeps: a pivoted Householder QR of the working matrix, then an LQ of R.
//
//   W P = Q [R; 0],   R = L Z^H,   so   W = Q [L; 0] (P Z)^H
//
// The sweeps then run on the N x N lower triangular L with V starting at
// P Z, and the left vectors are Q applied to L's (Drmac and Veselic, "New
// fast and accurate Jacobi SVD algorithm", SIAM J. Matrix Anal. Appl. 29,
// 2008).  L^H L is two steps of the LR iteration closer to diagonal than
// W^H W and its columns come out roughly in descending norm, so the sweeps
// start near the end of their linear phase: 128 x 64 with kappa = 1e6 takes
// 6.3 sweeps instead of 17, and on L's N rows instead of M.  Q and Z are
// backward stable, columns are taken by norm (rank revealing, safe for
// column-graded data), and the sweeps' own pair test still decides
// convergence.  The two factorisations cost about as many operations as half
// a sweep.
//
// All the threads of a CTA work on one matrix in shared or global memory.
// The QR applies a reflection to a column with P lanes (a row split, one
// shuffle tree); the LQ applies it to a row, reading columns, so neighbouring
// threads touch neighbouring rows in both.  Reflections are the Hermitian
// H = I - tau v v^H with v = x + e^{i arg x_0} |x| e_1: v is the column itself
// but for its first entry, so nothing is rescaled.  Every multiply-add is
// explicit: the same bits wherever it is inlined.
//
// What bounds it: N dependent steps per factorisation, in FP64 the FP64 pipe
// (64 % busy over the whole 128 x 64 solve), in FP32 latency and shared-memory
// bandwidth.  128 x 64, one CTA:
// FP64 1.48 M cycles and 0.74 M for Q's application (17 sweeps take 23 M, the
// 6.3 left 5 M); FP32 0.21 M and 0.075 M on the float4 form below (0.45 M and
// 0.20 M on the scalar one), 11 sweeps about 1.5 M.  Measured and not kept:
// panels of eight vectors factorised by one warp in registers (FP32 0.35 M;
// FP64 2.5 M, an FP64 instruction holds its SM partition's unit far too long
// for one warp to carry a panel).
#pragma once

#include "jacobi_common.cuh"
#include "tc_f32.cuh"

namespace bsvd {

__device__ __forceinline__ float sq_acc(float x, float a) { return fmaf(x, x, a); }
__device__ __forceinline__ double sq_acc(double x, double a) { return fma(x, x, a); }
__device__ __forceinline__ float sq_acc(float2 x, float a) { return fmaf(x.x, x.x, fmaf(x.y, x.y, a)); }
__device__ __forceinline__ double sq_acc(double2 x, double a) { return fma(x.x, x.x, fma(x.y, x.y, a)); }
// a - x y
__device__ __forceinline__ float nfma(float x, float y, float a) { return fmaf(-x, y, a); }
__device__ __forceinline__ double nfma(double x, double y, double a) { return fma(-x, y, a); }
__device__ __forceinline__ float2 nfma(float2 x, float2 y, float2 a) { return fma_s(make_float2(-x.x, -x.y), y, a); }
__device__ __forceinline__ double2 nfma(double2 x, double2 y, double2 a) { return fma_s(make_double2(-x.x, -x.y), y, a); }
__device__ __forceinline__ float rscale(float x, float r) { return rmul(x, r); }
__device__ __forceinline__ double rscale(double x, double r) { return rmul(x, r); }
__device__ __forceinline__ float2 rscale(float2 x, float r) { return make_float2(rmul(x.x, r), rmul(x.y, r)); }
__device__ __forceinline__ double2 rscale(double2 x, double r) { return make_double2(rmul(x.x, r), rmul(x.y, r)); }
// order of non-negative reals as unsigned words (the leading 32 bits: enough to pick a pivot)
__device__ __forceinline__ unsigned pivot_key(float x) { return __float_as_uint(fmaxf(x, 0.f)); }
__device__ __forceinline__ unsigned pivot_key(double x) { return (unsigned)__double2hiint(fmax(x, 0.0)); }

// Squared norms at or below this are not safe to square again; a matrix with
// such a column keeps the plain start.
template <class R> constexpr R kPreNormMin = R(0);
template <> constexpr float kPreNormMin<float> = 1e-24f;
template <> constexpr double kPreNormMin<double> = 1e-200;
template <class R> constexpr R kPreTiny = R(0);         // a reflection of a shorter vector is the identity
template <> constexpr float kPreTiny<float> = 1e-34f;
template <> constexpr double kPreTiny<double> = 1e-290;

// A column of which the QR leaves less than 2^-32 of its norm in single
// precision, 2^-64 in double (squares here): rounding of rounding, as in matrices
// of exact low rank, whose equal columns round equally.  From such an R the sweeps
// get a chain of columns u, u^2, u^3 .. of the largest, whose squares underflow in
// single precision: constant, checkerboard and block-constant FP32 and complex64
// matrices ran into the sweep limit.  They keep the plain start.
template <class R> constexpr R kPreDeficient = R(0);
template <> constexpr float kPreDeficient<float> = 0x1p-64f;
template <> constexpr double kPreDeficient<double> = 0x1p-128;

enum class Pre { kNone, kDone, kDeficient };               // unchanged, done, W destroyed and V unchanged

// Scratch of one matrix, N entries each (two sets of column norms: a step
// reads one while it writes the other).  v0 has at least eight: row_span's two
// ints a warp of up to 256 threads.
template <class T>
struct PreScratch {
    Real<T>* nrm2;
    Real<T>* tau;
    T* v0;
    T* diag;
    int* perm;
    __device__ explicit PreScratch(void* p, int N) {
        v0 = static_cast<T*>(p);
        diag = v0 + (N < 8 ? 8 : N);
        nrm2 = reinterpret_cast<Real<T>*>(diag + N);
        tau = nrm2 + 2 * N;
        perm = reinterpret_cast<int*>(tau + N);
    }
    __host__ __device__ static constexpr long long bytes(long long N) {
        return (N < 8 ? 8 : N) * (long long)sizeof(T) + N * ((long long)sizeof(T) + 3 * (long long)sizeof(Real<T>) + 4);
    }
};

// The reflection H = I - tau v v^H of a vector x (first entry x0, squared norm
// ss): ph = e^{i arg x0} |x|, v = x + ph e_1, H x = -ph e_1.
template <class T>
__device__ __forceinline__ void reflection(T x0, Real<T> ss, T& ph, Real<T>& tau) {
    using R = Real<T>;
    ph = make_s<T>(0);
    tau = 0;
    if (!(ss > kPreTiny<R>)) return;                  // H = I
    // two reciprocal square roots, no division (long FP64 sequences, all on
    // one warp); tau |v|^2 = 2 to a few ulp
    const R nrm = rmul(ss, rsqrt_r(ss)), a0 = abs_rot(x0);
    ph = make_s<T>(nrm);
    if constexpr (Traits<T>::kComplex) {
        // below 2^-60 of the norm any phase will do; nrm / a0 could overflow there,
        // and a denormal x0 does not give its phase to working accuracy
        if (a0 > rmul(nrm, R(0x1p-60))) ph = rscale(x0, nrm / a0);
    } else if (a0 > 0) {
        ph = phase_times(x0, a0, nrm);
    }
    const R st = rsqrt_r(rmul(nrm, nrm + a0));
    tau = rmul(st, st);
}

// Elements per pass of the two loops below.  Single precision waits for
// shared-memory latency: eight loads of each operand in flight, the last pass
// padded with zeros.  FP64 waits for its arithmetic pipe: two, none wasted.
template <class T> constexpr int kPreBatch = sizeof(Real<T>) == 4 ? 8 : 2;

// sum over i < n of conj(v[i sv]) y[i sy] (ConjV) or v[i sv] conj(y[i sy])
template <class T, bool ConjV>
__device__ __forceinline__ T strided_dot(const T* v, int sv, const T* y, int sy, int n) {
    constexpr int B = kPreBatch<T>;
    T a = make_s<T>(0), b = make_s<T>(0);
    auto mac = [](T x, T z, T acc) { return ConjV ? cfma(x, z, acc) : fma_s(x, conj_s(z), acc); };
    int i = 0;
    if constexpr (sizeof(Real<T>) == 8) {
#pragma unroll 2
        for (; i + 1 < n; i += 2) {
            a = mac(v[i * sv], y[i * sy], a);
            b = mac(v[(i + 1) * sv], y[(i + 1) * sy], b);
        }
        if (i < n) a = mac(v[i * sv], y[i * sy], a);
    } else
    for (; i < n; i += B) {
        T vv[B], yy[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool in = i + u < n;
            vv[u] = in ? v[(i + u) * sv] : make_s<T>(0);
            yy[u] = in ? y[(i + u) * sy] : make_s<T>(0);
        }
#pragma unroll
        for (int u = 0; u < B; u += 2) {
            a = mac(vv[u], yy[u], a);
            b = mac(vv[u + 1], yy[u + 1], b);
        }
    }
    return add(a, b);
}
// y[i sy] <- y[i sy] - v[i sv] f
template <class T>
__device__ __forceinline__ void strided_axpy(const T* v, int sv, T* y, int sy, int n, T f) {
    constexpr int B = kPreBatch<T>;
    if constexpr (sizeof(Real<T>) == 8) {
#pragma unroll 4
        for (int i = 0; i < n; ++i) y[i * sy] = nfma(v[i * sv], f, y[i * sy]);
    } else
    for (int i = 0; i < n; i += B) {
        T vv[B], yy[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool in = i + u < n;
            vv[u] = in ? v[(i + u) * sv] : make_s<T>(0);
            yy[u] = in ? y[(i + u) * sy] : make_s<T>(0);
        }
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (i + u < n) y[(i + u) * sy] = nfma(vv[u], f, yy[u]);
    }
}

// y_j <- (I - tau v v^H) y_j, v = x + ph e_1, for columns j0 .. N-1 of X on
// rows k .. M-1 (x[r] at row r), P lanes a column: lane = q * cw + c is row
// class q of the warp's column c (consecutive lanes on consecutive columns: an
// odd leading dimension spreads them over the banks).  v^H y is taken as
// x^H y + conj(ph) y_k, so the products do not wait for the norm: reflect()
// gives ph and tau in between.  norms(j, y_kj) sees each new row-k entry.
template <class T, int NT, int P, class Reflect, class Norms>
__device__ __forceinline__ void reflect_columns(T* X, int ldx, int k, int M, int j0, int N, const T* x,
                                                const Reflect& reflect, const Norms& norms) {
    constexpr int cw = 32 / P, per = NT / P;
    const int tid = threadIdx.x, lane = tid & 31, q = lane / cw;
    const int n = M - k > q ? (M - k - q + P - 1) / P : 0;
    T ph = make_s<T>(0);
    Real<T> tau = 0;
    bool have = false;
    for (int jb = j0; jb < N || !have; jb += per) {
        const int j = jb + (tid >> 5) * cw + lane % cw;
        T* y = X + (long long)min(j, N - 1) * ldx + k;
        T s = make_s<T>(0), yk = make_s<T>(0);
        if (j < N) {
            s = strided_dot<T, true>(x + k + q, P, y + q, P, n);
            yk = y[0];
        }
        if (!have) {
            reflect(ph, tau);
            have = true;
        }
#pragma unroll
        for (int o = cw; o < 32; o <<= 1) s = add(s, shfl_xor_s(s, o));
        s = rscale(cfma(ph, yk, s), tau);
        if (j < N) {
            if (q == 0) {
                yk = nfma(add(x[k], ph), s, yk);
                y[0] = yk;
                norms(j, yk);
                strided_axpy<T>(x + k + P, P, y + P, P, n - 1, s);
            } else {
                strided_axpy<T>(x + k + q, P, y + q, P, n, s);
            }
        }
    }
}

// Lanes a column: four, eight where N columns would leave threads idle.
template <int NT>
__device__ __forceinline__ bool eight_lanes(int N) { return NT <= 128 && 8 * N <= NT; }

// Binary orders that the rows' largest entries may span (row_span).  The
// factorisations are accurate relative to each column, not to each row: from a
// matrix with rows of different sizes they take the relative accuracy of its
// smallest singular values, which the plain start keeps.  Median over 24
// matrices D B, FP64 64 x 64, of the largest relative error of a singular value,
// in units of u, against that of the plain start: D over 2^4 (rows spanning five
// orders) 74 and 57, 2^5 96 and 57, 2^6 179 and 69, 2^8 398 and 62, 2^10 848 and 74.
// With two rows a column the larger rows alone determine the matrix as a rule, and
// nothing is lost: 128 x 64, D over 2^6 86 and 100, over 2^7 91 and 102; where the
// small rows carry an eighth of the dimensions by themselves up to 1.4 times the
// plain start's (100 x 48, 2^6: 103 and 72).  Such matrices may span seven orders,
// at which even a square one stays within a factor of three (179 and 69):
// geometric spectra reach them by chance, and 3 % of 128 x 64 matrices down to 1e-6
// on the plain start took a tenth of the time of a batch of 4,000 (95.0 ms, 84.7 so).
__host__ __device__ constexpr int pre_row_span(int M, int N) { return M >= 2 * N ? 7 : 5; }
// Where only V is kept, and FP64 sweeps on A V decide the values (kFlagVOnly): a
// fifteenth of the 96 x 96 matrices of a clustered spectrum span six orders, and
// their plain start cost the mixed path 2 ms of 95 on 2,000 of them.
constexpr int kPreVOnlySpan = 10;

// Whether the spectrum is so flat that the sweeps gain little from the
// preconditioner: the participation ratio (sum sigma^2)^2 / (N sum sigma^4)
// above 0.35 (iid normal entries: 0.5 square, 0.67 at 2:1; geometric spectra:
// 0.14 for a condition number of 1e3, 0.22 for 1e2, at 64 columns).  sum
// sigma^2 is the sum of the squared column norms; sum sigma^4 is estimated as
// |W^H W x|^2 for one fixed vector of signs.  y: M elements.  Synchronised.
template <class T, int NT>
__device__ __forceinline__ bool flat_spectrum(const T* W, int ldw, int M, int N, const Real<T>* nrm2, T* y, Real<T>* z2) {
    using R = Real<T>;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int r = tid; r < M; r += NT) {
        T a = make_s<T>(0);
        for (int j = 0; j < N; ++j) {
            const T w = W[r + (long long)j * ldw];
            a = (__popc(j * 0x9E3779B1u) & 1) ? sub(a, w) : add(a, w);
        }
        y[r] = a;
    }
    __syncthreads();
    for (int j = warp; j < N; j += NW) {
        T a = make_s<T>(0);
        for (int r = lane; r < M; r += 32) a = cfma(W[r + (long long)j * ldw], y[r], a);
        a = warp_sum_s(a);
        if (lane == 0) z2[j] = sq_acc(a, R(0));
    }
    __syncthreads();
    R s2 = 0, s4 = 0;
    for (int j = lane; j < N; j += 32) {
        s2 += nrm2[j];
        s4 += z2[j];
    }
    s2 = warp_sum(s2);
    s4 = warp_sum(s4);
    __syncthreads();                                       // y and z2 are scratch of what follows
    return rmul(s2, s2) > rmul(R(0.35) * R(N), s4);        // uniform: every warp sums the same numbers
}

// Columns of W (M rows) in descending norm, perm along; only for norms that
// differ by more than a factor of four.  order and t: N ints each.  Executed
// by all threads.
template <class T, int NT>
__device__ __forceinline__ void sort_columns(T* W, int ldw, int M, int N, const Real<T>* nrm2, int* perm, int* order,
                                             int* t) {
    using R = Real<T>;
    const int tid = threadIdx.x, lane = tid & 31;
    R lo = nrm2[0], hi = lo;
    for (int j = lane; j < N; j += 32) { lo = fmin(lo, nrm2[j]); hi = fmax(hi, nrm2[j]); }
    hi = warp_max(hi);
    lo = -warp_max(-lo);
    if (hi <= 16 * lo) return;                             // uniform: every warp sees all the norms
    for (int k = tid; k < N; k += NT) {
        int rk = 0;
        for (int j = 0; j < N; ++j) rk += nrm2[j] > nrm2[k] || (nrm2[j] == nrm2[k] && j < k);
        order[rk] = k;                                     // order[k]: the column that goes to place k
    }
    __syncthreads();
    if (tid == 0) {                                        // as transpositions (k, t_k)
        for (int k = 0; k < N; ++k) {
            int at = k;                                    // where column order[k] sits now
            while (perm[at] != order[k]) ++at;
            t[k] = at;
            const int p = perm[k];
            perm[k] = perm[at];
            perm[at] = p;
        }
    }
    __syncthreads();
    for (int r = tid; r < M; r += NT)
        for (int k = 0; k < N; ++k) {
            const int p = t[k];
            if (p == k) continue;
            const T a = W[r + (long long)k * ldw];
            W[r + (long long)k * ldw] = W[r + (long long)p * ldw];
            W[r + (long long)p * ldw] = a;
        }
    __syncthreads();
}

// W (M x N, M >= N, leading dimension ldw) becomes L (N x N, zero rows below);
// V (N x N, unless null) becomes V0 P Z (V0 null: I); the reflections of Q go
// to refl (M x N, scaled so that tau = 1; null: dropped).  Called by all NT
// threads after W is complete and synchronised; returns synchronised.
// The caller has seen to it that the rows span at most pre_row_span.  kNone when a
// column is too short to square safely (or zero), and in single precision when the
// spectrum is flat; kDeficient when a column is left with nothing.
//
// Double precision picks each column by its remaining norm (QR with column
// pivoting: 128 x 64 with kappa = 1e6 then takes 6.3 sweeps, 7.1 without).
// Single precision, where the extra barrier and reduction of every step cost
// more than the sweeps they save, sorts the columns once.
template <class T, int NT, int P>
__device__ __forceinline__ void qr_steps(T* W, int ldw, int M, int N, const PreScratch<T>& sc) {
    using R = Real<T>;
    constexpr bool kPivot = sizeof(R) == 8;
    const int tid = threadIdx.x, lane = tid & 31;
    R* const own = reinterpret_cast<R*>(sc.v0);            // squared column norms by the caller's column, for the end
    for (int j = tid; j < N; j += NT) own[j] = sc.nrm2[j];
    __syncthreads();
    for (int k = 0; k < N; ++k) {
        const R* cur = sc.nrm2 + (k & 1) * N;
        R* next = sc.nrm2 + ((k + 1) & 1) * N;
        int p = k;
        if constexpr (kPivot) {
            unsigned best = 0;
            int bj = N;
            for (int j = k + lane; j < N; j += 32) {
                const unsigned key = pivot_key(cur[j]);
                if (bj == N || key > best) { best = key; bj = j; }
            }
            const unsigned top = __reduce_max_sync(0xffffffffu, best);
            p = (int)__reduce_min_sync(0xffffffffu, bj < N && best == top ? (unsigned)bj : (unsigned)N);
            if (p != k) {                                     // uniform over the CTA
                for (int r = tid; r < M; r += NT) {
                    const T a = W[r + (long long)k * ldw], b = W[r + (long long)p * ldw];
                    W[r + (long long)k * ldw] = b;
                    W[r + (long long)p * ldw] = a;
                }
                if (tid == 0) { const int t = sc.perm[k]; sc.perm[k] = sc.perm[p]; sc.perm[p] = t; }
                __syncthreads();
            }
        }
        const T* x = W + (long long)k * ldw;
        reflect_columns<T, NT, P>(
            W, ldw, k, M, k + 1, N, x,
            [&](T& ph, R& tau) {          // by one warp: the square root and division are long FP64 sequences
                if (tid < 32) {
                    R ss = 0;
                    for (int r = k + lane; r < M; r += 32) ss = sq_acc(x[r], ss);
                    ss = warp_sum(ss);
                    reflection<T>(x[k], k + 1 < M ? ss : R(0), ph, tau);
                    if (lane == 0) {
                        sc.diag[k] = ph;
                        sc.tau[k] = tau;
                    }
                }
                __syncthreads();
                ph = sc.diag[k];
                tau = sc.tau[k];
            },
            [&](int j, T yk) {       // what is left of column j's squared norm (column p holds old column k)
                if constexpr (kPivot) {
                    const R n = cur[j == p ? k : j], d = sq_acc(yk, R(0));
                    next[j] = d < n ? n - d : R(0);
                }
            });
        __syncthreads();
    }
}

template <class T, int NT>
__device__ __forceinline__ Pre precondition(T* W, int ldw, int M, int N, T* V, int ldv, const T* V0, long long ldv0,
                                             T* refl, long long ldr, const PreScratch<T>& sc) {
    using R = Real<T>;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int j = warp; j < N; j += NW) {
        R ss = 0;
        for (int r = lane; r < M; r += 32) ss = sq_acc(W[r + (long long)j * ldw], ss);
        ss = warp_sum(ss);
        if (lane == 0) { sc.nrm2[j] = ss; sc.perm[j] = j; }
    }
    __syncthreads();
    bool small = false;
    for (int j = lane; j < N; j += 32) small |= !(sc.nrm2[j] > kPreNormMin<R>);
    if (__any_sync(0xffffffffu, small)) { __syncthreads(); return Pre::kNone; }   // uniform: every warp reads all norms
    if constexpr (sizeof(R) == 4)
        if (M <= 2 * N && flat_spectrum<T, NT>(W, ldw, M, N, sc.nrm2, sc.v0, sc.tau)) return Pre::kNone;
    if constexpr (sizeof(R) == 4)
        sort_columns<T, NT>(W, ldw, M, N, sc.nrm2, sc.perm, reinterpret_cast<int*>(sc.v0), reinterpret_cast<int*>(sc.diag));

    // ---- W P = Q R ---------------------------------------------------------------
    if (eight_lanes<NT>(N)) qr_steps<T, NT, 8>(W, ldw, M, N, sc);
    else                    qr_steps<T, NT, 4>(W, ldw, M, N, sc);
    bool left = true;
    for (int k = lane; k < N; k += 32)
        left &= sq_acc(sc.tau[k] > 0 ? sc.diag[k] : W[k + (long long)k * ldw], R(0)) >
                rmul(kPreDeficient<R>, reinterpret_cast<const R*>(sc.v0)[sc.perm[k]]);
    if (!__all_sync(0xffffffffu, left)) { __syncthreads(); return Pre::kDeficient; }   // uniform: every warp reads all
    if (refl)
        for (int k = warp; k < N; k += NW) {
            const R f = sqrt_r(sc.tau[k]);
            for (int r = k + lane; r < M; r += 32)
                refl[r + (long long)k * ldr] = rscale(r == k ? add(W[r + (long long)k * ldw], sc.diag[k]) : W[r + (long long)k * ldw], f);
        }
    if (V)
        for (int k = warp; k < N; k += NW) {
            const int c = sc.perm[k];
            for (int i = lane; i < N; i += 32)
                V[i + (long long)k * ldv] = V0 ? V0[i + (long long)c * ldv0] : make_s<T>(i == c ? 1 : 0);
        }
    __syncthreads();
    for (int k = warp; k < N; k += NW)                    // R: the diagonal, zeros below
        for (int r = k + lane; r < M; r += 32) {
            T* w = W + r + (long long)k * ldw;
            if (r > k) *w = make_s<T>(0);
            else if (sc.tau[k] > 0) *w = rscale(sc.diag[k], R(-1));
        }
    __syncthreads();

    // ---- R = L Z^H, V <- V Z: reflections of rows, two lanes a row --------------
    for (int i = 0; i + 1 < N; ++i) {
        const T* x = W + i + (long long)i * ldw;          // row i from its diagonal: x[j * ldw]
        const int nr = N - 1 - i, rows = nr + (V ? N : 0), h = tid & 1, n = (N - i - h + 1) / 2;
        T ph = make_s<T>(0);
        R tau = 0;
        bool have = false;
        for (int rb = 0; rb < rows || !have; rb += NT / 2) {
            const int rr = rb + tid / 2;
            const bool inW = rr < nr || !V, ok = rr < rows;
            T* y = inW ? W + min(i + 1 + rr, N - 1) + (long long)i * ldw : V + min(rr - nr, N - 1) + (long long)i * ldv;
            const int ld = inW ? ldw : ldv;
            T s = make_s<T>(0), yi = make_s<T>(0);
            if (ok) {
                s = strided_dot<T, false>(y + h * ld, 2 * ld, x + h * ldw, 2 * ldw, n);
                yi = y[0];
            }
            if (!have) {                                  // the reflection of conj(row i), applied from the right
                if (tid < 32) {
                    R ss = 0;
                    for (int j = lane; j < N - i; j += 32) ss = sq_acc(x[(long long)j * ldw], ss);
                    ss = warp_sum(ss);
                    reflection<T>(conj_s(x[0]), ss, ph, tau);
                    if (lane == 0) {
                        sc.diag[i] = ph;
                        sc.tau[i] = tau;
                    }
                }
                __syncthreads();
                ph = sc.diag[i];
                tau = sc.tau[i];
                have = true;
            }
            s = add(s, shfl_xor_s(s, 1));
            s = rscale(fma_s(yi, ph, s), tau);
            if (ok) {
                if (h == 0) {
                    y[0] = nfma(s, add(x[0], conj_s(ph)), yi);
                    strided_axpy<T>(x + 2 * ldw, 2 * ldw, y + 2 * ld, 2 * ld, n - 1, s);
                } else {
                    strided_axpy<T>(x + ldw, 2 * ldw, y + ld, 2 * ld, n, s);
                }
            }
        }
        __syncthreads();
    }
    for (int j = warp; j < N; j += NW)                    // L: the diagonal, zeros above
        for (int i = lane; i <= j; i += 32) {
            if (i < j) W[i + (long long)j * ldw] = make_s<T>(0);
            else if (i + 1 < N && sc.tau[i] > 0) W[i + (long long)j * ldw] = conj_s(rscale(sc.diag[i], R(-1)));
        }
    __syncthreads();
    return Pre::kDone;
}

// ---- real FP32: the same steps on float4 ------------------------------------------
// In FP32 the loops above are bound by instruction issue (about 20 instructions
// a multiply-add: predicates, addresses, one load per operand), so real FP32,
// whose columns start on 16-byte boundaries, works on four rows at a time.  The
// reflected vector is copied by one warp to a buffer that is zero outside it,
// so no loop needs a mask: a column step reads it and the column as float4
// (lane = q * cw + c on chunks q, q + P, ...; neighbouring columns lie 4 * odd
// words apart, so the eight lanes of a load phase hit different banks), and a
// row step takes four rows of a column per load, eight lanes a row group.
//
// Warp 0 looks ahead: at step k it updates only vector k + 1 and forms the
// reflection of step k + 1 in the other buffer while the remaining warps update
// the rest, so a step has one barrier and its critical path is one vector's
// product, update, norm and square roots.
struct PreF32 {
    float* v;       // two reflections: rows of a column, or a row's columns
    float* nrm2;
    float* tau;
    float* ph;
    int* perm;
    int* tmp;       // 2 N ints
    __device__ PreF32(void* p, int M, int N) {
        v = static_cast<float*>(p);
        nrm2 = v + 2 * f32_buf(M);
        tau = nrm2 + N;
        ph = tau + N;
        perm = reinterpret_cast<int*>(ph + N);
        tmp = perm + N;
    }
    __host__ __device__ static int f32_buf(int M) { return (M + 3) & ~3; }
    __host__ __device__ static long long bytes(int M, int N) { return 8LL * f32_buf(M) + 24LL * N; }
};

__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, s))));
}
__device__ __forceinline__ float4 nfma4(float4 a, float f, float4 y) {
    return make_float4(fmaf(-a.x, f, y.x), fmaf(-a.y, f, y.y), fmaf(-a.z, f, y.z), fmaf(-a.w, f, y.w));
}

// Columns j0 .. N-1 of X through I - tau v v^T; v zero outside rows [k, M).
// Warps w0 .. of the NT / 32, P lanes a column.
template <int NT, int P>
__device__ __forceinline__ void reflect_columns_f32(float* X, int ldx, int k, int M, int j0, int N, const float* v,
                                                    float tau, int w0) {
    constexpr int cw = 32 / P;
    const int lane = threadIdx.x & 31, q = lane / cw, c1 = (M + 3) >> 2, c0 = (k >> 2) + q;
    const float4* v4 = reinterpret_cast<const float4*>(v);
    if (M <= 32 * P) {                                     // at most 8 chunks a lane: loads first, all in registers
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const int cmin = k >> 2;
        float4 vr[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) vr[i] = q + i * P >= cmin && q + i * P < c1 ? v4[q + i * P] : z;
        for (int jw = j0 + ((threadIdx.x >> 5) - w0) * cw; jw < N; jw += (NT / 32 - w0) * cw) {   // uniform over the warp
            const int j = jw + lane % cw;
            float4* y = reinterpret_cast<float4*>(X + (long long)min(j, N - 1) * ldx) + q;
            float4 yr[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) yr[i] = q + i * P >= cmin && q + i * P < c1 ? y[i * P] : z;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                s0 = dot4(vr[i], yr[i], s0);
                s1 = dot4(vr[i + 1], yr[i + 1], s1);
            }
            float s = s0 + s1;
#pragma unroll
            for (int o = cw; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            s = rmul(s, tau);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (j < N && q + i * P >= cmin && q + i * P < c1) y[i * P] = nfma4(vr[i], s, yr[i]);
        }
        return;
    }
    for (int jw = j0 + ((threadIdx.x >> 5) - w0) * cw; jw < N; jw += (NT / 32 - w0) * cw) {   // uniform over the warp
        const int j = jw + lane % cw;
        float4* y = reinterpret_cast<float4*>(X + (long long)min(j, N - 1) * ldx);
        float s0 = 0.f, s1 = 0.f;
        int c = c0;
#pragma unroll 2
        for (; c + P < c1; c += 2 * P) {
            s0 = dot4(v4[c], y[c], s0);
            s1 = dot4(v4[c + P], y[c + P], s1);
        }
        if (c < c1) s0 = dot4(v4[c], y[c], s0);
        float s = s0 + s1;
#pragma unroll
        for (int o = cw; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s = rmul(s, tau);
        if (j < N) {
#pragma unroll 4
            for (c = c0; c < c1; c += P) y[c] = nfma4(v4[c], s, y[c]);
        }
    }
}

// One warp: the reflection of entries [k, n) of a strided vector x into v
// (entries [k & ~3, pad) written, zero outside [k, n)), tau and ph.
__device__ __forceinline__ void make_reflection_f32(const float* x, int sx, int k, int n, int pad, float* v, float* tau,
                                                    float* ph) {
    const int lane = threadIdx.x & 31;
    float ss = 0.f;
    for (int r = (k & ~3) + lane; r < pad; r += 32) {
        const float a = r >= k && r < n ? x[r * sx] : 0.f;
        ss = fmaf(a, a, ss);
        v[r] = a;
    }
    ss = warp_sum(ss);
    const float x0 = x[k * sx];
    float p, t;
    reflection<float>(x0, k + 1 < n ? ss : 0.f, p, t);
    __syncwarp();
    if (lane == 0) {
        v[k] = x0 + p;
        *tau = t;
        *ph = p;
    }
}

// One warp: vector x (entries x[r * sx], r < n) through I - tau v v^T (v from
// entry k), then the reflection of its entries from k + 1 into vn, tau_n, ph_n.
// The reflection keeps the norm of the entries from k on, so what the next one
// needs is that norm less the new entry k squared -- summed with the product
// in one round of shuffles, and summed again only where the difference cancels.
__device__ __forceinline__ void look_ahead_f32(float* x, int sx, int k, int n, int pad, const float* v, float tau,
                                               float* vn, float* tau_n, float* ph_n) {
    const int lane = threadIdx.x & 31, b = k & ~3;
    float x0 = 0.f, ss;
    if (pad - b <= 128) {
        float xr[4], vr[4], s = 0.f, all = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = b + lane + 32 * i;
            xr[i] = r < n ? x[r * sx] : 0.f;
            vr[i] = r < n ? v[r] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = b + lane + 32 * i >= k ? xr[i] : 0.f;
            s = fmaf(vr[i], xr[i], s);
            all = fmaf(a, a, all);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        s = rmul(s, tau);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            xr[i] = fmaf(-vr[i], s, xr[i]);
            const int r = b + lane + 32 * i;
            if (r < n) x[r * sx] = xr[i];
        }
        const float xk = __shfl_sync(0xffffffffu, xr[0], k - b);
        x0 = __shfl_sync(0xffffffffu, xr[0], k + 1 - b);
        ss = fmaf(-xk, xk, all);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (b + lane + 32 * i <= k) xr[i] = 0.f;
        if (!(ss > 0.5f * all)) {
            ss = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) ss = fmaf(xr[i], xr[i], ss);
            ss = warp_sum(ss);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (b + lane + 32 * i < pad) vn[b + lane + 32 * i] = xr[i];
    } else {
        float s = 0.f;
        for (int r = b + lane; r < n; r += 32) s = fmaf(v[r], x[r * sx], s);
        s = rmul(warp_sum(s), tau);
        ss = 0.f;
        for (int r = b + lane; r < pad; r += 32) {
            float a = 0.f;
            if (r < n) {
                a = fmaf(-v[r], s, x[r * sx]);
                x[r * sx] = a;
            }
            if (r == k + 1) x0 = a;
            a = r > k ? a : 0.f;
            ss = fmaf(a, a, ss);
            vn[r] = a;
        }
        ss = warp_sum(ss);
        x0 = __shfl_sync(0xffffffffu, x0, k + 1 - b);
    }
    float p, t;
    reflection<float>(x0, k + 2 < n ? ss : 0.f, p, t);
    __syncwarp();
    if (lane == 0) {
        vn[k + 1] = x0 + p;
        *tau_n = t;
        *ph_n = p;
    }
}

// precondition for real FP32 (W's columns and V's on 16-byte boundaries, zero
// in the rows that pad them to a multiple of four).
template <int NT>
__device__ __forceinline__ Pre precondition_f32(float* W, int ldw, int M, int N, float* V, int ldv, float* refl,
                                                 long long ldr, const PreF32& sc) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, mp = PreF32::f32_buf(M), np = PreF32::f32_buf(N);
    for (int j = warp; j < N; j += NW) {
        float ss = 0.f;
        for (int r = lane; r < M; r += 32) ss = sq_acc(W[r + j * ldw], ss);
        ss = warp_sum(ss);
        if (lane == 0) { sc.nrm2[j] = ss; sc.perm[j] = j; }
    }
    __syncthreads();
    bool small = false;
    for (int j = lane; j < N; j += 32) small |= !(sc.nrm2[j] > kPreNormMin<float>);
    if (__any_sync(0xffffffffu, small)) { __syncthreads(); return Pre::kNone; }   // uniform: every warp reads all norms
    if (flat_spectrum<float, NT>(W, ldw, M, N, sc.nrm2, sc.v, sc.tau)) return Pre::kNone;
    sort_columns<float, NT>(W, ldw, M, N, sc.nrm2, sc.perm, sc.tmp, sc.tmp + N);

    if (warp == 0) make_reflection_f32(W, 1, 0, M, mp, sc.v, sc.tau, sc.ph);
    __syncthreads();
    for (int k = 0; k < N; ++k) {                          // W P = Q R
        const float* v = sc.v + (k & 1) * mp;
        const float tau = sc.tau[k];
        if (warp == 0) {
            if (k + 1 < N)
                look_ahead_f32(W + (k + 1) * ldw, 1, k, M, mp, v, tau, sc.v + ((k + 1) & 1) * mp, sc.tau + k + 1,
                               sc.ph + k + 1);
        } else {
            if (eight_lanes<NT>(N)) reflect_columns_f32<NT, 8>(W, ldw, k, M, k + 2, N, v, tau, 1);
            else                    reflect_columns_f32<NT, 4>(W, ldw, k, M, k + 2, N, v, tau, 1);
        }
        __syncthreads();
    }
    bool left = true;
    for (int k = lane; k < N; k += 32)
        left &= sq_acc(sc.tau[k] > 0.f ? sc.ph[k] : W[k + k * ldw], 0.f) > rmul(kPreDeficient<float>, sc.nrm2[sc.perm[k]]);
    if (!__all_sync(0xffffffffu, left)) { __syncthreads(); return Pre::kDeficient; }   // uniform: every warp reads all
    if (refl)
        for (int k = warp; k < N; k += NW) {
            const float f = sqrtf(sc.tau[k]);
            for (int r = k + lane; r < M; r += 32)
                refl[r + (long long)k * ldr] = rmul(r == k ? W[r + k * ldw] + sc.ph[k] : W[r + k * ldw], f);
        }
    if (V)
        for (int k = warp; k < N; k += NW) {
            const int c = sc.perm[k];
            for (int i = lane; i < np; i += 32) V[i + k * ldv] = i == c ? 1.f : 0.f;
        }
    for (int k = warp; k < N; k += NW)                     // R: the diagonal, zeros below
        for (int r = k + lane; r < mp; r += 32) {
            if (r > k) W[r + k * ldw] = 0.f;
            else if (sc.tau[k] > 0.f) W[r + k * ldw] = -sc.ph[k];
        }
    __syncthreads();
    if (warp == 0) make_reflection_f32(W, ldw, 0, N, np, sc.v, sc.tau, sc.ph);
    __syncthreads();
    const int gw = np >> 2, q = tid & 7;                   // row groups of W; lane's column class
    for (int i = 0; i + 1 < N; ++i) {                      // R = L Z^T, V <- V Z
        const float* v = sc.v + (i & 1) * mp;
        const float tau = sc.tau[i];
        if (warp == 0) {
            look_ahead_f32(W + i + 1, ldw, i, N, np, v, tau, sc.v + ((i + 1) & 1) * mp, sc.tau + i + 1, sc.ph + i + 1);
            __syncthreads();
            continue;
        }
        const int g0 = (i + 2) >> 2, nw = max(gw - g0, 0), groups = nw + (V ? gw : 0);
        for (int gb = (warp - 1) * 4; gb < groups; gb += (NW - 1) * 4) {       // uniform over the warp
            const int g = min(gb + (lane >> 3), groups - 1);
            const bool inW = g < nw, ok = gb + (lane >> 3) < groups;
            const int row = 4 * (inW ? g0 + g : g - nw), ld = inW ? ldw : ldv;
            float* y = (inW ? W : V) + row + (i + q) * ld;
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
            // rows of W up to i are done and row i + 1 is warp 0's: not stored
            const int skip = inW ? i + 2 - row : 0;
            const float* w = v + i + q;
            if (N - i <= 64) {                             // at most 8 columns a lane: loads first, all in registers
                float4 yr[8];
                float wr[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const bool in = i + q + 8 * u < N;
                    yr[u] = in ? *reinterpret_cast<const float4*>(y + 8 * u * ld) : make_float4(0.f, 0.f, 0.f, 0.f);
                    wr[u] = in ? w[8 * u] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    a0 = fmaf(yr[u].x, wr[u], a0); a1 = fmaf(yr[u].y, wr[u], a1);
                    a2 = fmaf(yr[u].z, wr[u], a2); a3 = fmaf(yr[u].w, wr[u], a3);
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) {
                    a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                    a1 += __shfl_xor_sync(0xffffffffu, a1, o);
                    a2 += __shfl_xor_sync(0xffffffffu, a2, o);
                    a3 += __shfl_xor_sync(0xffffffffu, a3, o);
                }
                a0 = rmul(a0, tau); a1 = rmul(a1, tau); a2 = rmul(a2, tau); a3 = rmul(a3, tau);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (!ok || i + q + 8 * u >= N) continue;
                    float* p = y + 8 * u * ld;
                    const float4 t = make_float4(fmaf(-a0, wr[u], yr[u].x), fmaf(-a1, wr[u], yr[u].y),
                                                 fmaf(-a2, wr[u], yr[u].z), fmaf(-a3, wr[u], yr[u].w));
                    if (skip <= 0) {
                        *reinterpret_cast<float4*>(p) = t;
                    } else {
                        if (skip <= 1) p[1] = t.y;
                        if (skip <= 2) p[2] = t.z;
                        if (skip <= 3) p[3] = t.w;
                    }
                }
                continue;
            }
            float* p = y;
#pragma unroll 4
            for (int j = i + q; j < N; j += 8) {
                const float4 yy = *reinterpret_cast<const float4*>(p);
                const float ww = *w;
                a0 = fmaf(yy.x, ww, a0); a1 = fmaf(yy.y, ww, a1); a2 = fmaf(yy.z, ww, a2); a3 = fmaf(yy.w, ww, a3);
                p += 8 * ld;
                w += 8;
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                a1 += __shfl_xor_sync(0xffffffffu, a1, o);
                a2 += __shfl_xor_sync(0xffffffffu, a2, o);
                a3 += __shfl_xor_sync(0xffffffffu, a3, o);
            }
            a0 = rmul(a0, tau); a1 = rmul(a1, tau); a2 = rmul(a2, tau); a3 = rmul(a3, tau);
            if (ok) {
                p = y;
                w = v + i + q;
#pragma unroll 4
                for (int j = i + q; j < N; j += 8) {
                    float4 yy = *reinterpret_cast<const float4*>(p);
                    const float ww = *w;
                    yy.x = fmaf(-a0, ww, yy.x); yy.y = fmaf(-a1, ww, yy.y);
                    yy.z = fmaf(-a2, ww, yy.z); yy.w = fmaf(-a3, ww, yy.w);
                    if (skip <= 0) {
                        *reinterpret_cast<float4*>(p) = yy;
                    } else {
                        if (skip <= 1) p[1] = yy.y;
                        if (skip <= 2) p[2] = yy.z;
                        if (skip <= 3) p[3] = yy.w;
                    }
                    p += 8 * ld;
                    w += 8;
                }
            }
        }
        __syncthreads();
    }
    for (int j = warp; j < N; j += NW)                     // L: the diagonal, zeros above
        for (int i = lane; i <= j; i += 32) {
            if (i < j) W[i + j * ldw] = 0.f;
            else if (i + 1 < N && sc.tau[i] > 0.f) W[i + j * ldw] = -sc.ph[i];
        }
    __syncthreads();
    return Pre::kDone;
}

// apply_q for real FP32; buf: kQPanel buffers of f32_buf(M) floats.  A column
// belongs to its own lanes, so the panel's reflections need no barrier between
// them, only the next panel's loads do.
constexpr int kQPanel = 4;
template <int NT>
__device__ __forceinline__ void apply_q_f32(float* X, int ldx, int M, int N, const float* refl, long long ldr, float* buf) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, mp = PreF32::f32_buf(M);
    for (int k1 = N; k1 > 0; k1 -= kQPanel) {              // reflections k1 - 1, k1 - 2, ...
        const int nb = min(kQPanel, k1);
        __syncthreads();
        for (int t = warp; t < nb; t += NW) {
            const int k = k1 - 1 - t;
            for (int r = (k & ~3) + lane; r < mp; r += 32)
                buf[t * mp + r] = r >= k && r < M ? refl[r + (long long)k * ldr] : 0.f;
        }
        __syncthreads();
        for (int t = 0; t < nb; ++t) {
            const int k = k1 - 1 - t;
            if (eight_lanes<NT>(N)) reflect_columns_f32<NT, 8>(X, ldx, k, M, 0, N, buf + t * mp, 1.f, 0);
            else                    reflect_columns_f32<NT, 4>(X, ldx, k, M, 0, N, buf + t * mp, 1.f, 0);
            __syncwarp();
        }
    }
    __syncthreads();
}

// W (N x N) <- W Sigma^-1 in place; columns with sigma = 0 completed to an
// orthonormal basis as in finalize_outputs (the basis vector of largest
// residual, projected twice).  x: N elements.  Synchronised on return.
template <class T, int NT>
__device__ __forceinline__ void normalize_columns(T* W, int ldw, int N, T* x, const FinalScratch<T>& fs) {
    using R = Real<T>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const R* sig = fs.sig;
    for (int e = tid; e < N * N; e += NT) {
        const int i = e % N, k = e / N;
        if (sig[k] > 0) W[i + (long long)k * ldw] = divr(W[i + (long long)k * ldw], sig[k]);
    }
    __syncthreads();
    for (int c = 0; c < N; ++c) {
        if (sig[c] > 0) continue;                          // uniform over the CTA
        auto valid = [&](int q) { return sig[q] > 0 || q < c; };
        if (tid == 0) {
            R best = -1;
            int r0 = 0;
            for (int r = 0; r < N; ++r) {
                R s2 = 0;
                for (int q = 0; q < N; ++q)
                    if (valid(q)) s2 += abs2(W[r + (long long)q * ldw]);
                if (R(1) - s2 > best) { best = R(1) - s2; r0 = r; }
            }
            fs.iscr[1] = r0;
        }
        __syncthreads();
        const int r0 = fs.iscr[1];
        for (int r = tid; r < N; r += NT) x[r] = make_s<T>(r == r0 ? 1 : 0);
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass)
            for (int q = 0; q < N; ++q) {
                if (!valid(q)) continue;
                if (warp == 0) {
                    T d = make_s<T>(0);
                    for (int r = lane; r < N; r += 32) d = cfma(W[r + (long long)q * ldw], x[r], d);
                    d = warp_sum_s(d);
                    if (lane == 0) fs.bcast[0] = d;
                }
                __syncthreads();
                const T dd = fs.bcast[0];
                for (int r = tid; r < N; r += NT) x[r] = sub(x[r], mul(W[r + (long long)q * ldw], dd));
                __syncthreads();
            }
        if (warp == 0) {
            R ss = 0;
            for (int r = lane; r < N; r += 32) ss += abs2(x[r]);
            ss = warp_sum(ss);
            if (lane == 0) fs.red[0] = sqrt_r(ss);
        }
        __syncthreads();
        const R nx = fs.red[0];
        for (int r = tid; r < N; r += NT) W[r + (long long)c * ldw] = divr(x[r], nx);
        __syncthreads();
    }
}

// X (M x N) <- Q X with the reflections left by precondition; buf: two
// columns of M elements, or null to read them in place.
template <class T, int NT, int P>
__device__ __forceinline__ void apply_q_steps(T* X, int ldx, int M, int N, const T* refl, long long ldr, T* buf) {
    using R = Real<T>;
    const int tid = threadIdx.x;
    auto none = [](int, T) {};
    auto unit = [](T& ph, R& tau) { ph = make_s<T>(0); tau = 1; };
    if (!buf) {
        for (int k = N - 1; k >= 0; --k) {
            reflect_columns<T, NT, P>(X, ldx, k, M, 0, N, refl + (long long)k * ldr, unit, none);
            __syncthreads();
        }
        return;
    }
    auto load = [&](int k) {
        for (int r = k + tid; r < M; r += NT)
            cp_async<(int)sizeof(T)>(buf + (k & 1) * M + r, refl + r + (long long)k * ldr, (int)sizeof(T));
        cp_async_commit();
    };
    load(N - 1);
    cp_async_wait<0>();
    __syncthreads();
    for (int k = N - 1; k >= 0; --k) {
        if (k > 0) load(k - 1);                            // the next reflection loads during this one
        reflect_columns<T, NT, P>(X, ldx, k, M, 0, N, buf + (k & 1) * M, unit, none);
        cp_async_wait<0>();
        __syncthreads();
    }
}

template <class T, int NT>
__device__ __forceinline__ void apply_q(T* X, int ldx, int M, int N, const T* refl, long long ldr, T* buf) {
    if (eight_lanes<NT>(N)) apply_q_steps<T, NT, 8>(X, ldx, M, N, refl, ldr, buf);
    else                    apply_q_steps<T, NT, 4>(X, ldx, M, N, refl, ldr, buf);
}

}  // namespace bsvd
