// FP64 m x m kernels of the block Lanczos process and of the per-shift
// recurrences (Sec. 3): a few CTAs reduce the Gram partials and the last to
// arrive does the shared m x m work; the recurrences take one CTA per shift.
//
// Block form.  The Lanczos blocks V_1, V_2, ... (widths m_k, shrinking on
// deflation) satisfy
//     A V_k = V_{k-1} beta_k^H + V_k alpha_k + V_{k+1} beta_{k+1},
// so T = V^H A V is block tridiagonal with diagonal blocks alpha_k and
// sub-diagonal blocks beta_{k+1} (m_{k+1} x m_k): a hermitian band matrix of
// semi-bandwidth <= m (Eq. 3.1).  For each shift the root-free block
// Cholesky factorisation sigma_j I + T = L Delta L^H (L block unit lower
// bidiagonal with blocks Lambda_k, Delta block diagonal) is extended by one
// block row per step:
//     Delta_1 = alpha_1 + sigma I,
//     Lambda_{k+1} = beta_{k+1} Delta_k^{-1},
//     Delta_{k+1} = alpha_{k+1} + sigma I - Lambda_{k+1} beta_{k+1}^H,
// and with U = L^{-1} [rho; 0] (B = V_1 rho), P = V L^{-H}:
//     U_1 = rho, U_{k+1} = -Lambda_{k+1} U_k,  Ut_k = Delta_k^{-1} U_k,
//     P_1 = V_1, P_{k+1} = V_{k+1} - P_k Lambda_{k+1}^H,
//     X^(k) = X^(k-1) + P_k Ut_k,
// the block counterpart of the paper's scalar update with d^(k), p^(k),
// u^(k) (Sec. 3).  From the Lanczos relation the residual is
//     R^(k) = B - (sigma + A) X^(k) = -V_{k+1} beta_{k+1} Ut_k = V_{k+1} C_k,
// so with orthonormal V_{k+1} the residual norm of right-hand side i is the
// norm of column i of C_k = -beta_{k+1} Ut_k (Sec. 3, R^(k) = W^(k) C^(k)).
//
// Deflation (Sec. 1 and Sec. 3): the new block W is orthonormalised by a
// pivoted Cholesky factorisation of its FP64 Gram matrix.  Columns whose
// remaining squared norm falls to <= dtol^2 times their norm when created
//
// Arithmetic.  With FP64 storage these kernels run in FP64.  With the
// reduced storages they run in double-float (dd: pairs of FP32 words, 48-bit
// significands) unless FP64 is requested: GB300 issues FP64 at 1/64 of its
// FP32 rate, so one FP64
// instruction occupies an SM sub-partition for about 64 cycles and these
// latency-bound m x m kernels were dominated by it; the double-float forms
// run on the FP32 pipes and keep far more accuracy than the FP32 Gram
// partials they start from.  Both scalars take 16 bytes per complex entry,
// so the device state has one layout.
#include <math.h>

#include "fx.cuh"
#include "kernels.h"

namespace dsbcg {

// group sums of one reduction: at most 1024 groups x slots, or 36 slots of
// each of the 36 upper tiles of a 32 x 32 Gram matrix
constexpr int RED_SLOTS = 36 * 36;

template <class T>
struct SmallSharedT {
    T alpha[M_MAX * M_MAX];          // alpha_k (hermitised)
    T betak[M_MAX * M_MAX];          // beta_k    (m_k x m_{k-1})
    T betan[M_MAX * M_MAX];          // beta_{k+1} (m_{k+1} x m_k)
    T S[M_MAX * M_MAX];              // V_{k+1} = W S (m_k x m_{k+1})
    T yy[M_MAX / 2];                 // ||A v_i||^2 (real scalars, two per entry)
    double red[RED_SLOTS];           // group sums of the Gram partials (reduce_partials)
    unsigned ticket[3];              // arrival counters of the multi-CTA kernels (zero between launches)
    unsigned qr_step;                // the block step whose QR is published (released by small_qr_kernel)
};
template <class T>
struct SmallShiftT {
    T Lam[M_MAX * M_MAX];            // Lambda_k (m_k x m_{k-1})
    T U[M_MAX * M_MAX];              // U_k (m_k x m)
    int conv[M_MAX];                 // right-hand side i frozen
    int alive;                       // some column not converged
    int pad[M_MAX - 1];
};
template <class T>
struct SmallStateT {
    SmallSharedT<T> sh;
    SmallShiftT<T> sf[1];            // [s]
};
// the opaque type of kernels.h: the same bytes for both scalars
struct SmallState : SmallStateT<double2> {};
static_assert(sizeof(ddc) == sizeof(double2), "one state layout for both scalars");

size_t small_state_bytes(int s) {
    return sizeof(SmallSharedT<double2>) + (size_t)s * sizeof(SmallShiftT<double2>);
}
const double2* small_state_S(const SmallState* ss) { return ss->sh.S; }

namespace {

constexpr int WS = 32;
constexpr int QW = 4;              // warps of the pivoted QR: one per SM sub-partition
constexpr int GSL = 36;            // slots per 4 x 4 tile in the Gram partials
constexpr int RED_GROUPS = 1024;   // groups x slots of a reduction aim at this many chains
constexpr int NRC = 8;             // CTAs of the kernels that reduce Gram partials
constexpr int NT = 8 * GSL;        // threads per CTA: eight slot groups of a reduction, nine warps for the m x m work

// ------------------------------------------------------------ scalars --
// Sc<T>: real type R, complex T, and the operations the m x m algebra needs.
template <class T>
struct Sc;

template <>
struct Sc<double2> {
    using R = double;
    static __device__ __forceinline__ R r(double v) { return v; }
    static __device__ __forceinline__ double d(R v) { return v; }
    static __device__ __forceinline__ double2 z() { return make_double2(0.0, 0.0); }
    static __device__ __forceinline__ double2 c(R a, R b) { return make_double2(a, b); }
    static __device__ __forceinline__ R re(double2 a) { return a.x; }
    static __device__ __forceinline__ R im(double2 a) { return a.y; }
    static __device__ __forceinline__ R add(R a, R b) { return a + b; }
    static __device__ __forceinline__ R sub(R a, R b) { return a - b; }
    static __device__ __forceinline__ R mul(R a, R b) { return a * b; }
    static __device__ __forceinline__ R neg(R a) { return -a; }
    static __device__ __forceinline__ R rcp(R a) { return 1.0 / a; }
    static __device__ __forceinline__ R sqrt_(R a) { return sqrt(a); }
    static __device__ __forceinline__ bool gt(R a, R b) { return a > b; }
    static __device__ __forceinline__ float2 f2(double2 a) { return make_float2((float)a.x, (float)a.y); }
    // sum of a Kahan-compensated FP32 sum (value s - c)
    static __device__ __forceinline__ R kahan(float s, float c) { return widen(s) - widen(c); }
};

// double-float reciprocal and square root: FP32 estimate refined by one
// Newton-Raphson step in double-float (Karp & Markstein, "High-precision
// division and square root", ACM TOMS 23(4), 1997)
__device__ __forceinline__ dd dd_rcp(dd a) {
    const float q = 1.0f / a.hi;
    // e = 1 - a q, with a.hi q exact as p + pe
    const float p = a.hi * q;
    const float pe = fmaf(a.hi, q, -p);
    const float e = ((1.0f - p) - pe) - a.lo * q;
    return quick_two_sum(q, q * e);
}
__device__ __forceinline__ dd dd_sqrt(dd a) {
    if (!(a.hi > 0.f)) return dd(0.f);
    const float s = sqrtf(a.hi);
    const float p = s * s;
    const float pe = fmaf(s, s, -p);
    const float e = ((a.hi - p) - pe) + a.lo;            // a - s^2
    return quick_two_sum(s, e * (0.5f / s));
}

template <>
struct Sc<ddc> {
    using R = dd;
    static __device__ __forceinline__ R r(double v) { return dd::from_double(v); }
    static __device__ __forceinline__ double d(R v) { return (double)v.hi + (double)v.lo; }
    static __device__ __forceinline__ ddc z() { return ddc{dd(0.f), dd(0.f)}; }
    static __device__ __forceinline__ ddc c(R a, R b) { return ddc{a, b}; }
    static __device__ __forceinline__ R re(ddc a) { return a.x; }
    static __device__ __forceinline__ R im(ddc a) { return a.y; }
    static __device__ __forceinline__ R add(R a, R b) { return a + b; }
    static __device__ __forceinline__ R sub(R a, R b) { return a - b; }
    static __device__ __forceinline__ R mul(R a, R b) { return a * b; }
    static __device__ __forceinline__ R neg(R a) { return -a; }
    static __device__ __forceinline__ R rcp(R a) { return dd_rcp(a); }
    static __device__ __forceinline__ R sqrt_(R a) { return dd_sqrt(a); }
    static __device__ __forceinline__ bool gt(R a, R b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }
    static __device__ __forceinline__ float2 f2(ddc a) { return make_float2(a.x.hi, a.y.hi); }
    static __device__ __forceinline__ R kahan(float s, float c) { return dd(s) - dd(c); }
};

template <class T> __host__ __device__ constexpr bool is_fp64() { return false; }
template <> __host__ __device__ constexpr bool is_fp64<double2>() { return true; }

// complex helpers on Sc<T> (all normalised)
template <class T> __device__ __forceinline__ T cz() { return Sc<T>::z(); }
template <class T> __device__ __forceinline__ T cconj(T a) { return Sc<T>::c(Sc<T>::re(a), Sc<T>::neg(Sc<T>::im(a))); }
template <class T> __device__ __forceinline__ T cplus(T a, T b) {
    return Sc<T>::c(Sc<T>::add(Sc<T>::re(a), Sc<T>::re(b)), Sc<T>::add(Sc<T>::im(a), Sc<T>::im(b)));
}
template <class T> __device__ __forceinline__ T cminus(T a, T b) {
    return Sc<T>::c(Sc<T>::sub(Sc<T>::re(a), Sc<T>::re(b)), Sc<T>::sub(Sc<T>::im(a), Sc<T>::im(b)));
}
template <class T> __device__ __forceinline__ T ctimes(T a, T b) {
    using S = Sc<T>;
    return S::c(S::sub(S::mul(S::re(a), S::re(b)), S::mul(S::im(a), S::im(b))),
                S::add(S::mul(S::re(a), S::im(b)), S::mul(S::im(a), S::re(b))));
}
template <class T> __device__ __forceinline__ T cscal(T a, typename Sc<T>::R s) {
    return Sc<T>::c(Sc<T>::mul(Sc<T>::re(a), s), Sc<T>::mul(Sc<T>::im(a), s));
}
template <class T> __device__ __forceinline__ typename Sc<T>::R cnorm2(T a) {
    using S = Sc<T>;
    return S::add(S::mul(S::re(a), S::re(a)), S::mul(S::im(a), S::im(a)));
}

__device__ __forceinline__ void bsync() { __syncthreads(); }
__device__ __forceinline__ void wsync() { __syncwarp(); }

// True in the CTA of the grid that arrives last; every other CTA's earlier
// writes are then visible to it (through ld_cg).  No CTA waits for another.
// The counter wraps to zero for the next launch.
__device__ __forceinline__ bool last_arrival(unsigned* ticket) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
}
__device__ __forceinline__ double ld_cg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ dd ld_cg(const dd* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return dd(v.x, v.y);
}

// dst (r x c valid, R x Cc written, leading dim ld) <- src (M_MAX layout)
template <class T>
__device__ void ld_mat(T* dst, int ld, const T* src, int r, int c, int Rr, int Cc) {
    for (int t = threadIdx.x; t < Rr * Cc; t += blockDim.x) {
        int i = t / Cc, j = t % Cc;
        dst[i * ld + j] = (i < r && j < c) ? src[i * M_MAX + j] : cz<T>();
    }
}
// full M_MAX x M_MAX tile in the work precision (FP64 only for FP64 state),
// zero outside r x c
template <class T>
__device__ void st_mat_work(int wprec, void* dst, const T* src, int ld, int r, int c) {
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        int i = t / M_MAX, j = t % M_MAX;
        const bool in = i < r && j < c;
        if constexpr (is_fp64<T>()) {
            if (wprec == P64) {
                reinterpret_cast<double2*>(dst)[t] = in ? src[i * ld + j] : cz<T>();
                continue;
            }
        }
        reinterpret_cast<float2*>(dst)[t] = in ? Sc<T>::f2(src[i * ld + j]) : make_float2(0.f, 0.f);
    }
}

// The M_MAX x M_MAX tile get(i, j) (zero outside r x c) as limbs with one
// exponent per column (fx.cuh): the coefficient form of the fixed-point
// kernels.  All threads of the CTA.
template <class F>
__device__ void st_mat_fx(int4* dst, int* ce, int r, int c, F get) {
    __shared__ int es[M_MAX];
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < M_MAX; j += blockDim.x >> 5) {
        int mx = 0;
        if (lane < r && j < c) {
            const double2 v = get(lane, j);
            mx = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) {
            const int eb = max(mx >> 20, 1);
            es[j] = eb;
            ce[j] = mx == 0 ? FX_ZERO : eb == 0x7ff ? FX_NAN : eb - 1079;
        }
    }
    bsync();
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        const int i = t / M_MAX, j = t % M_MAX;
        int4 q = make_int4(0, 0, 0, 0);
        if (i < r && j < c) {
            const double2 v = get(i, j);
            const int2 re = fx_split(fx_of_double(v.x, es[j])), im = fx_split(fx_of_double(v.y, es[j]));
            q = make_int4(re.x, re.y, im.x, im.y);
        }
        dst[t] = q;
    }
    bsync();
}

// real (0) or imaginary (1) part of an entry
template <class T>
__device__ __forceinline__ typename Sc<T>::R& part_of(T& a, int part) {
    return reinterpret_cast<typename Sc<T>::R*>(&a)[part];
}
// x + a b and x - a b, one part of a complex entry (the expressions of cplus
// and cminus with ctimes)
template <class T>
__device__ __forceinline__ typename Sc<T>::R plus_times(typename Sc<T>::R x, T a, T b, int part) {
    using S = Sc<T>;
    if (part == 0) return S::add(x, S::sub(S::mul(S::re(a), S::re(b)), S::mul(S::im(a), S::im(b))));
    return S::add(x, S::add(S::mul(S::re(a), S::im(b)), S::mul(S::im(a), S::re(b))));
}
template <class T>
__device__ __forceinline__ typename Sc<T>::R minus_times(typename Sc<T>::R x, T a, T b, int part) {
    using S = Sc<T>;
    if (part == 0) return S::sub(x, S::sub(S::mul(S::re(a), S::re(b)), S::mul(S::im(a), S::im(b))));
    return S::sub(x, S::add(S::mul(S::re(a), S::im(b)), S::mul(S::im(a), S::re(b))));
}
// item t of 2 n: entry and part, the parts in different warps (up to one)
__device__ __forceinline__ int item_of(int t, int n, int* part) {
    *part = t >= n;
    return t >= n ? t - n : t;
}

// C (r x c) = +-op(A) op(B), or C +- op(A) op(B) (accumulate); op: plain (0)
// or conjugate transpose (1).  One thread per real number of the result, so
// that the FP64 work spreads over the SM's sub-partitions.
template <class T>
__device__ void gemm(T* Cm, int ldc, const T* A, int lda, int ta, const T* B, int ldb, int tb, int r, int q, int c,
                     bool negate, bool accumulate) {
    using S = Sc<T>;
    for (int t = threadIdx.x; t < 2 * r * c; t += blockDim.x) {
        int part;
        const int e = item_of(t, r * c, &part), i = e / c, j = e % c;
        typename S::R s = S::r(0.0);
        for (int l = 0; l < q; ++l) {
            const T a = ta ? cconj(A[l * lda + i]) : A[i * lda + l];
            const T b = tb ? cconj(B[j * ldb + l]) : B[l * ldb + j];
            s = plus_times<T>(s, a, b, part);
        }
        typename S::R& o = part_of(Cm[i * ldc + j], part);
        if (accumulate) o = negate ? S::sub(o, s) : S::add(o, s);
        else o = negate ? S::sub(S::r(0.0), s) : s;
    }
    bsync();
}

// In-place inverse of a hermitian positive definite n x n matrix by
// Gauss-Jordan elimination without pivoting (its pivots are the Schur
// complement diagonals, positive for hpd).  Returns 0 if a pivot is <= 0.
// The first warp alone forms each pivot's reciprocal and scales its row (an
// FP64 division in all warps of the CTA cost 3 us per pivot); the elimination
// takes one thread per real number.
template <class T>
__device__ int gj_inverse(T* A, int ld, int n, T* col, typename Sc<T>::R* inv_s) {
    using S = Sc<T>;
    using R = typename S::R;
    __shared__ int ok_s;
    if (threadIdx.x == 0) ok_s = 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int p = 0; p < n; ++p) {
        if (warp == 0) {
            R d = S::re(A[p * ld + p]);
            if (!S::gt(d, S::r(0.0))) {
                if (lane == 0) ok_s = 0;
                d = S::r(1.0);
            }
            const R inv = S::rcp(d);
            wsync();
            for (int t = lane; t < 2 * n; t += WS) {
                const int c = t >> 1, part = t & 1;
                R& o = part_of(A[p * ld + c], part);
                o = c == p ? (part ? S::r(0.0) : inv) : S::mul(o, inv);
            }
            if (lane == 0) *inv_s = inv;
        } else if (warp == 1) {
            for (int r = lane; r < n; r += WS)
                if (r != p) col[r] = A[r * ld + p];
        }
        bsync();
        const R inv = *inv_s;
        for (int t = threadIdx.x; t < 2 * n * n; t += blockDim.x) {
            int part;
            const int e = item_of(t, n * n, &part), r = e / n, c = e % n;
            if (r == p) continue;
            R& o = part_of(A[r * ld + c], part);
            if (c == p) o = S::mul(part_of(col[r], part), S::neg(inv));
            else o = minus_times<T>(o, col[r], A[p * ld + c], part);
        }
        bsync();
    }
    return ok_s;
}

// barrier of the QR's QW warps
__device__ __forceinline__ void qsync() { asm volatile("bar.sync 1, %0;" ::"n"(QW * WS) : "memory"); }

// Pivoted Cholesky of the hermitian Gram matrix G (n x n, smem, ld; its upper
// and lower triangles are overwritten by the remainders) with the deflation
// test: remaining squared norm <= dtol^2 * ref (the column's squared norm when
// it was created).  Pivot: the largest remaining relative squared norm, ties
// to the lowest position.  Produces the rank r, S = Pi_r R11^{-1} (n x r) and
// beta = R Pi^T (r x n), both in smem with leading dimension ld (beta zeroed by
// the caller).  R is kept in original column order.
// Runs on QW warps (threads 0 .. QW * 32 - 1): a warp-wide FP64 instruction
// occupies an SM sub-partition for 64 clocks, so the work is spread over the
// four of them and over the lanes: the pairwise pivot comparisons (whose
// outcomes every warp then scans as bits), the right-looking update of the
// remainder (the subtractions per entry in the order of the pivots), and the
// real and imaginary parts of the back substitution.
template <class T>
__device__ int pivoted_qr(T* G, int ld, int n, const typename Sc<T>::R* ref, typename Sc<T>::R dtol2, T* Rm, T* Sm,
                          T* beta, int* perm, typename Sc<T>::R* dd_, typename Sc<T>::R* irp, unsigned* bits) {
    using S = Sc<T>;
    using R = typename S::R;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    unsigned* wb = bits + w * 16;              // this warp's comparison bits: pair (q, b < q) at q (q - 1) / 2 + b
    if (tid < n) {
        perm[tid] = tid;
        dd_[tid] = S::re(G[tid * ld + tid]);
    }
    for (int t = tid; t < n * n; t += QW * WS) {
        Rm[t] = cz<T>();
        Sm[t / n * ld + t % n] = cz<T>();
    }
    const unsigned valid = __ballot_sync(0xffffffffu, lane < n && S::gt(ref[lane < n ? lane : 0], S::r(0.0)));
    qsync();
    int rank = n;
    for (int p = 0; p < n; ++p) {
        // dd[q] / ref[q] > dd[b] / ref[b] is tested as dd[q] ref[b] > dd[b] ref[q]
        const int rem = n - p, np = rem * (rem - 1) / 2;
        for (int base = 0; base < np; base += WS) {
            const int idx = min(base + lane, np - 1);
            int q = (int)((1.f + sqrtf(8.f * (float)idx + 1.f)) * 0.5f);
            while (q * (q - 1) / 2 > idx) --q;
            while (q * (q + 1) / 2 <= idx) ++q;
            const int oq = perm[p + q], ob = perm[p + idx - q * (q - 1) / 2];
            const unsigned m = __ballot_sync(0xffffffffu, S::gt(S::mul(dd_[oq], ref[ob]), S::mul(dd_[ob], ref[oq])));
            if (lane == 0) wb[base / WS] = m;
        }
        wsync();
        int best = -1;
        for (int q = 0; q < rem; ++q) {
            if (!(valid >> perm[p + q] & 1u)) continue;
            const int at = q * (q - 1) / 2 + best;
            if (best < 0 || (wb[at / WS] >> (at % WS) & 1u)) best = q;
        }
        bool stop = best < 0;
        if (!stop) {
            const R bd = dd_[perm[p + best]];
            stop = !S::gt(bd, S::mul(dtol2, ref[perm[p + best]])) || !S::gt(bd, S::r(0.0));
        }
        if (stop) {
            rank = p;
            break;
        }
        qsync();                               // every warp has chosen
        if (tid == 0 && best != 0) {
            const int tp = perm[p];
            perm[p] = perm[p + best];
            perm[p + best] = tp;
        }
        qsync();
        const int gp = perm[p];
        if (w == 0) {
            const R rpp = S::sqrt_(dd_[gp]);
            const R irpp = S::rcp(rpp);
            if (lane == 0) {
                Rm[p * n + gp] = S::c(rpp, S::r(0.0));
                irp[p] = irpp;
            }
            if (p + 1 + lane < n) {
                const int gr = perm[p + 1 + lane];
                const T v = cscal(G[gp * ld + gr], irpp);
                Rm[p * n + gr] = v;
                dd_[gr] = S::sub(dd_[gr], cnorm2(v));
            }
        }
        qsync();
        const int m2 = n - 1 - p;
        for (int e = tid; e < 2 * m2 * m2; e += QW * WS) {
            int part;
            const int t = item_of(e, m2 * m2, &part), a = t / m2, b = t % m2;
            if (a == b) continue;
            const int ga = perm[p + 1 + a], gb = perm[p + 1 + b];
            R& o = part_of(G[ga * ld + gb], part);
            o = minus_times<T>(o, cconj(Rm[p * n + ga]), Rm[p * n + gb], part);
        }
    }
    qsync();
    // beta = R Pi^T
    for (int t = tid; t < rank * n; t += QW * WS) {
        const int cp = t / n, c = t % n;
        if (c >= cp) beta[cp * ld + perm[c]] = Rm[cp * n + perm[c]];
    }
    // S = Pi_r R11^{-1}: column c solves R11 y = e_c by back substitution, a
    // lane per column; even and odd columns and their real and imaginary
    // parts in different warps
    const int c = 2 * lane + (w & 1), part = w >> 1;
    for (int i = rank - 1; i >= 0; --i) {
        if (c < rank && i <= c) {
            R s = S::r(i == c && part == 0 ? 1.0 : 0.0);
            for (int q = i + 1; q <= c; ++q) s = minus_times<T>(s, Rm[i * n + perm[q]], Sm[perm[q] * ld + c], part);
            part_of(Sm[perm[i] * ld + c], part) = S::mul(s, irp[i]);
        }
        qsync();
    }
    return rank;
}

__device__ inline void tile_ij(int t, int T, int herm, int* ti, int* tj) {
    if (!herm) {
        *ti = t / T;
        *tj = t % T;
        return;
    }
    int i = 0;
    while (t >= T - i) {
        t -= T - i;
        ++i;
    }
    *ti = i;
    *tj = i + t;
}

// write the reduced slot `it` ([tile][36] order) into G / diag
template <class T>
__device__ __forceinline__ void reduce_store(T* G, int ld, typename Sc<T>::R* diag, int Tt, int herm, int nf_max,
                                             int it, typename Sc<T>::R s) {
    using S = Sc<T>;
    const int tile = it / GSL, q = it % GSL;
    int ti, tj;
    tile_ij(tile, Tt, herm, &ti, &tj);
    if (q < 32) {
        const int i = ti * 4 + ((q >> 1) >> 2), j = tj * 4 + ((q >> 1) & 3);
        if (i < nf_max && j < nf_max) {
            if (q & 1) {
                G[i * ld + j].y = s;
                if (herm && ti != tj) G[j * ld + i].y = S::neg(s);
            } else {
                G[i * ld + j].x = s;
                if (herm && ti != tj) G[j * ld + i].x = s;
            }
        }
    } else if (diag && ti == tj) {
        const int j = tj * 4 + (q - 32);
        if (j < nf_max) diag[j] = s;
    }
}

// Sum the per-CTA Gram partials ([tile][blk][36], fixed order).  FP64
// partials (FP64 storage) are summed in FP64; FP32 partials (reduced storage;
// they carry FP32 accuracy) with compensated (Kahan) FP32 additions, the
// chains combined in the state's scalar.  The CTAs' range is split into
// red_groups groups per tile, whose sums are added in group order by
// reduce_combine; RC interleaved accumulators per thread keep several loads in
// flight (the partials come from L2, so the sum is latency-bound).
// The NRC CTAs of the launch share the (tile, group) units: the scalar
// additions that close the chains are FP64, 64 clocks per warp and
// sub-partition, which on one SM cost 8 us for three tiles.  Returns true in the CTA that
// arrives last, with every group sum in red[group * slots + slot].
// Fixed order: bitwise reproducible.
__host__ __device__ inline int red_groups(int ntiles) {
    const int items = ntiles * GSL, g = RED_GROUPS / items;
    return g < 1 ? 1 : g;
}

template <class T>
__device__ bool reduce_partials(const double* part, int nblk, int nf_max, typename Sc<T>::R* red,
                                unsigned* ticket, bool fp64_part) {
    using S = Sc<T>;
    using R = typename S::R;
    const int Tt = (nf_max + 3) / 4;
    const int ntiles = Tt * (Tt + 1) / 2;
    const int items = ntiles * GSL;
    const int ng = red_groups(ntiles);
    const int chunk = (nblk + ng - 1) / ng;
    const int q = threadIdx.x % GSL;
    for (int u = blockIdx.x + NRC * (threadIdx.x / GSL); u < ntiles * ng; u += NRC * (NT / GSL)) {
        const int tile = u % ntiles, grp = u / ntiles;
        const int b0 = grp * chunk, b1 = min(nblk, b0 + chunk);
        const size_t off = (size_t)tile * nblk * GSL + q;
        constexpr int RC = 8;
        R s;
        if (fp64_part) {
            const double* p = part + off;
            double a[RC];
#pragma unroll
            for (int r = 0; r < RC; ++r) a[r] = 0.0;
            int b = b0;
            for (; b + RC <= b1; b += RC)
#pragma unroll
                for (int r = 0; r < RC; ++r) a[r] += p[(size_t)(b + r) * GSL];
            for (; b < b1; ++b) a[0] += p[(size_t)b * GSL];
            double t = 0.0;
#pragma unroll
            for (int r = 0; r < RC; ++r) t += a[r];
            s = S::r(t);
        } else {
            const float* p = reinterpret_cast<const float*>(part) + off;
            float sum[RC], comp[RC];
#pragma unroll
            for (int r = 0; r < RC; ++r) sum[r] = comp[r] = 0.f;
            int b = b0;
            for (; b + RC <= b1; b += RC) {
                float y[RC];
#pragma unroll
                for (int r = 0; r < RC; ++r) y[r] = p[(size_t)(b + r) * GSL];
#pragma unroll
                for (int r = 0; r < RC; ++r) {
                    const float yy = y[r] - comp[r];
                    const float t = sum[r] + yy;
                    comp[r] = (t - sum[r]) - yy;
                    sum[r] = t;
                }
            }
            for (; b < b1; ++b) {
                const float yy = p[(size_t)b * GSL] - comp[0];
                const float t = sum[0] + yy;
                comp[0] = (t - sum[0]) - yy;
                sum[0] = t;
            }
            s = S::kahan(sum[0], comp[0]);
#pragma unroll
            for (int r = 1; r < RC; ++r) s = S::add(s, S::kahan(sum[r], comp[r]));
        }
        red[grp * items + tile * GSL + q] = s;
    }
    return last_arrival(ticket);
}
// G (ld, hermitian fill) and the |y|^2 diagonal from the group sums
template <class T>
__device__ void reduce_combine(const typename Sc<T>::R* red, int nf_max, T* G, int ld, typename Sc<T>::R* diag) {
    using S = Sc<T>;
    using R = typename S::R;
    const int Tt = (nf_max + 3) / 4;
    const int ntiles = Tt * (Tt + 1) / 2, items = ntiles * GSL, ng = red_groups(ntiles);
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        R s = ld_cg(red + it);
        for (int g = 1; g < ng; ++g) s = S::add(s, ld_cg(red + g * items + it));
        reduce_store<T>(G, ld, diag, Tt, 1, nf_max, it, s);
    }
}

// ---------------------------------------------------------------------------
// init: G0 = B^H B -> rank m_1, S0 (V_1 = B S0), rho = R Pi^T; U_{j,1} = rho
template <class T>
__global__ void small_init_kernel(SmallStateT<T>* ss, Ctl* ctl, const double2* __restrict__ G0,
                                  const double* __restrict__ ref, int m, int s, double dtol) {
    using S = Sc<T>;
    using R = typename S::R;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ unsigned bits[QW * 16];
    T* G = (T*)sm;
    T* Rm = G + m * m;
    T* Sm = Rm + m * m;
    T* rho = Sm + m * m;
    int* perm = (int*)(rho + m * m);
    R* dd_ = (R*)(perm + M_MAX);
    R* rf = dd_ + M_MAX;
    R* irp = rf + M_MAX;
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
        const double2 g = G0[(t / m) * M_MAX + t % m];
        G[t] = S::c(S::r(g.x), S::r(g.y));
        rho[t] = cz<T>();
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x) rf[i] = S::r(ref[i]);
    bsync();
    const int r = pivoted_qr<T>(G, m, m, rf, S::r(dtol * dtol), Rm, Sm, rho, perm, dd_, irp, bits);
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        const int i = t / M_MAX, j = t % M_MAX;
        ss->sh.S[t] = (i < m && j < m) ? Sm[i * m + j] : cz<T>();
        const T v = (i < r && j < m) ? rho[i * m + j] : cz<T>();
        for (int q = 0; q < s; ++q) {
            ss->sf[q].U[t] = v;
            ss->sf[q].Lam[t] = cz<T>();
        }
    }
    for (int t = threadIdx.x; t < s * M_MAX; t += blockDim.x) ss->sf[t / M_MAX].conv[t % M_MAX] = 0;
    for (int q = threadIdx.x; q < s; q += blockDim.x) ss->sf[q].alive = 1;
    if (threadIdx.x < 3) ss->sh.ticket[threadIdx.x] = 0;
    if (threadIdx.x == 3) ss->sh.qr_step = 0;
    if (threadIdx.x == 0) {
        ctl->k = 1;
        ctl->mk = r;
        ctl->mprev = 0;
        ctl->mnext = 0;
        ctl->done = (r == 0);
        ctl->status = 0;
        ctl->nact = s;
        ctl->deflations = m - r;
        ctl->mvms = 0;
        ctl->last_step = 0;
        ctl->f_dslash = ctl->f_gram = ctl->f_update = ctl->f_shift_s = ctl->f_shift_w = ctl->f_shift_cmac = 0;
    }
}

// alpha_k from the Gram partials of the upper tiles of V_k^H Y (alpha_k =
// V_k^H A V_k is hermitian; the lower tiles are the conjugates of the upper
// ones, the diagonal tiles are hermitised); coef_a = alpha and
// coef_bh = beta_k^H in the work precision (M_MAX tiles); ||y_i||^2.  NRC
// CTAs reduce, the last one to arrive forms the result.
template <class T>
__global__ void __launch_bounds__(NT) small_alpha_kernel(SmallStateT<T>* ss, const Ctl* ctl,
                                                         const double* part, int nblk, int nf_max,
                                                         int wprec, void* coef_a, void* coef_bh, int* ce) {
    step_begin();
    using S = Sc<T>;
    using R = typename S::R;
    if (cget(ctl->done)) return;
    R* red = reinterpret_cast<R*>(ss->sh.red);
    if (!reduce_partials<T>(part, nblk, nf_max, red, &ss->sh.ticket[0], wprec == P64)) return;
    __shared__ T A[M_MAX * M_MAX];
    __shared__ R yy[M_MAX];
    reduce_combine<T>(red, nf_max, A, M_MAX, yy);
    __syncthreads();
    const int mk_ = cget(ctl->mk), mp = cget(ctl->k) > 1 ? cget(ctl->mprev) : 0;
    const R half = S::r(0.5);
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        int i = t / M_MAX, j = t % M_MAX;
        const bool ina = i < mk_ && j < mk_, inb = i < mp && j < mk_;
        T v = cz<T>(), bh = cz<T>();
        if (ina) v = cscal(cplus(A[i * M_MAX + j], cconj(A[j * M_MAX + i])), half);
        if (inb) bh = cconj(ss->sh.betak[j * M_MAX + i]);
        ss->sh.alpha[t] = v;
        if constexpr (is_fp64<T>()) {
            if (wprec == P64) {
                if (ce) continue;
                ((double2*)coef_a)[t] = v;
                ((double2*)coef_bh)[t] = bh;
                continue;
            }
        }
        ((float2*)coef_a)[t] = ina ? S::f2(v) : make_float2(0.f, 0.f);
        ((float2*)coef_bh)[t] = inb ? S::f2(bh) : make_float2(0.f, 0.f);
    }
    R* yys = reinterpret_cast<R*>(ss->sh.yy);
    for (int t = threadIdx.x; t < M_MAX; t += blockDim.x) yys[t] = t < mk_ ? yy[t] : S::r(0.0);
    if constexpr (is_fp64<T>()) {
        if (ce) {
            st_mat_fx((int4*)coef_a, ce, mk_, mk_, [&](int i, int j) {
                return cscal(cplus(A[i * M_MAX + j], cconj(A[j * M_MAX + i])), half);
            });
            st_mat_fx((int4*)coef_bh, ce + M_MAX, mp, mk_, [&](int i, int j) { return cconj(ss->sh.betak[j * M_MAX + i]); });
        }
    }
}

// The block step's QR: G = W^H W from the partials (NRC CTAs), pivoted QR with
// deflation in the CTA that arrives last, which publishes S, beta_{k+1} and
// m_{k+1}.
template <class T>
__global__ void __launch_bounds__(NT) small_qr_kernel(SmallStateT<T>* ss, Ctl* ctl, const double* part,
                                                      int nblk, int m, double dtol, int wprec, void* coefS_w, int* ce, int MM) {
    step_begin();
    using S = Sc<T>;
    using R = typename S::R;
    if (cget(ctl->done)) return;
    R* red = reinterpret_cast<R*>(ss->sh.red);
    if (!reduce_partials<T>(part, nblk, m, red, &ss->sh.ticket[1], wprec == P64)) return;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ unsigned bits[QW * 16];
    __shared__ int mn_s;
    T* G = (T*)sm;
    T* Rm = G + MM * MM;
    T* Bn = Rm + MM * MM;       // beta_{k+1} (mn x mk)
    T* Sm = Bn + MM * MM;       // mk x mn
    R* dd_ = (R*)(Sm + MM * MM);
    R* rf = dd_ + MM;
    R* irp = rf + MM;
    int* perm = (int*)(irp + MM);
    const int mk_ = cget(ctl->mk);
    reduce_combine<T>(red, m, G, MM, nullptr);
    const R* yys = reinterpret_cast<const R*>(ss->sh.yy);
    for (int i = threadIdx.x; i < mk_; i += blockDim.x) rf[i] = yys[i];
    for (int t = threadIdx.x; t < MM * MM; t += blockDim.x) Bn[t] = cz<T>();
    bsync();
    if (threadIdx.x < QW * WS) {
        const int r = pivoted_qr<T>(G, MM, mk_, rf, S::r(dtol * dtol), Rm, Sm, Bn, perm, dd_, irp, bits);
        if (threadIdx.x == 0) mn_s = r;
    }
    bsync();
    const int mn = mn_s;
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        const int a = t / M_MAX, b = t % M_MAX;
        ss->sh.S[t] = (a < mk_ && b < mn) ? Sm[a * MM + b] : cz<T>();
        ss->sh.betan[t] = (a < mn && b < mk_) ? Bn[a * MM + b] : cz<T>();
    }
    if (threadIdx.x == 0) {
        ctl->mnext = mn;
        ctl->deflations = cget(ctl->deflations) + mk_ - mn;
    }
    // everything that the recurrences take from here, published for those that
    // run beside V = W S
    bsync();
    if (threadIdx.x == 0) st_release(&ss->sh.qr_step, (unsigned)cget(ctl->k));
    bool fx = false;
    if constexpr (is_fp64<T>()) {
        fx = ce != nullptr;
        if (fx) st_mat_fx((int4*)coefS_w, ce + 2 * M_MAX, mk_, mn, [&](int i, int j) { return Sm[i * MM + j]; });
    }
    if (!fx) st_mat_work<T>(wprec, coefS_w, Sm, MM, mk_, mn);
}

// One shift's recurrences of block step k (a CTA per shift).
template <class T>
__device__ void shift_recurrence(SmallStateT<T>* ss, Ctl* ctl, int j, int m, const double* __restrict__ sigma,
                                 const double* __restrict__ target, int freeze, int wprec, void* coefU_w,
                                 void* coefL_w, int* ce, int* active, int* conv_step, double* res_out, int MM,
                                 unsigned char* sm) {
    using S = Sc<T>;
    using R = typename S::R;
    SmallShiftT<T>& sf = ss->sf[j];
    if (!sf.alive) {
        if (threadIdx.x == 0) active[j] = 0;
        return;
    }
    T* Bn = (T*)sm;             // beta_{k+1} (mn x mk)
    T* Dl = Bn + MM * MM;       // Delta -> Delta^{-1}
    T* T1 = Dl + MM * MM;
    T* Ut = T1 + MM * MM;
    T* LH = Ut + MM * MM;
    T* Cc = LH + MM * MM;
    T* Bk = Cc + MM * MM;       // beta_k (mk x mp)
    T* col = Bk + MM * MM;
    R* res = (R*)(col + MM);
    R* inv = res + MM;
    const int k = cget(ctl->k), mk_ = cget(ctl->mk), mp = k > 1 ? cget(ctl->mprev) : 0, mn = cget(ctl->mnext);
    const size_t tile = (size_t)M_MAX * M_MAX;
    const size_t cb = wprec == P64 ? 16 : 8;
    // Delta_k = alpha_k + sigma I - Lambda_k beta_k^H
    ld_mat<T>(Dl, MM, ss->sh.alpha, mk_, mk_, mk_, mk_);
    ld_mat<T>(Bn, MM, ss->sh.betan, mn, mk_, mn, mk_);
    if (k > 1 && mp > 0) {
        ld_mat<T>(T1, MM, sf.Lam, mk_, mp, mk_, mp);
        ld_mat<T>(Bk, MM, ss->sh.betak, mk_, mp, mk_, mp);
    }
    bsync();
    if (k > 1 && mp > 0) gemm<T>(Dl, MM, T1, MM, 0, Bk, MM, 1, mk_, mp, mk_, true, true);
    const R sj = S::r(sigma[j]);
    for (int i = threadIdx.x; i < mk_; i += blockDim.x) Dl[i * MM + i].x = S::add(Dl[i * MM + i].x, sj);
    ld_mat<T>(T1, MM, sf.U, mk_, m, mk_, m);
    bsync();
    const R half = S::r(0.5);
    for (int t = threadIdx.x; t < mk_ * mk_; t += blockDim.x) {      // exact hermitian symmetry
        int a = t / mk_, b = t % mk_;
        if (b < a) {
            const T h = cscal(cplus(Dl[a * MM + b], cconj(Dl[b * MM + a])), half);
            Dl[a * MM + b] = h;
            Dl[b * MM + a] = cconj(h);
        }
    }
    bsync();
    if (!gj_inverse<T>(Dl, MM, mk_, col, inv)) {
        if (threadIdx.x == 0) {
            atomicCAS(&ctl->status, 0, ST_NOT_HPD);
            active[j] = 0;
            sf.alive = 0;
        }
        return;
    }
    // Ut = Delta^{-1} U_k (mk x m); Lambda_{k+1}^H = Delta^{-1} beta_{k+1}^H (mk x mn)
    gemm<T>(Ut, MM, Dl, MM, 0, T1, MM, 0, mk_, mk_, m, false, false);
    gemm<T>(LH, MM, Dl, MM, 0, Bn, MM, 1, mk_, mk_, mn, false, false);
    // C = -beta_{k+1} Ut (mn x m) gives the residual estimates, and it is also
    // U_{k+1} = -Lambda_{k+1} U_k = -beta_{k+1} Delta_k^{-1} U_k
    gemm<T>(Cc, MM, Bn, MM, 0, Ut, MM, 0, mn, mk_, m, true, false);
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        R s2 = S::r(0.0);
        for (int c = 0; c < mn; ++c) s2 = S::add(s2, cnorm2(Cc[c * MM + i]));
        res[i] = S::sqrt_(s2);
    }
    // shift-update coefficients: Ut with the columns frozen before this step zeroed
    for (int t = threadIdx.x; t < mk_ * m; t += blockDim.x) {
        int a = t / m, i = t % m;
        if (freeze && sf.conv[i]) Ut[a * MM + i] = cz<T>();
    }
    bsync();
    bool fx = false;
    if constexpr (is_fp64<T>()) {
        fx = ce != nullptr;
        if (fx) {
            int* e = ce + (size_t)j * 2 * M_MAX;
            st_mat_fx((int4*)coefU_w + (size_t)j * tile, e, mk_, m, [&](int a, int b) { return Ut[a * MM + b]; });
            st_mat_fx((int4*)coefL_w + (size_t)j * tile, e + M_MAX, mk_, mn, [&](int a, int b) { return LH[a * MM + b]; });
        }
    }
    if (!fx) {
        st_mat_work<T>(wprec, (char*)coefU_w + (size_t)j * tile * cb, Ut, MM, mk_, m);
        st_mat_work<T>(wprec, (char*)coefL_w + (size_t)j * tile * cb, LH, MM, mk_, mn);
    }
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) {
        int c = t / M_MAX, a = t % M_MAX;
        sf.Lam[t] = (c < mn && a < mk_) ? cconj(LH[a * MM + c]) : cz<T>();
        sf.U[t] = (c < mn && a < m) ? Cc[c * MM + a] : cz<T>();
    }
    if (threadIdx.x < WS) {
        const int i = threadIdx.x;
        int was = 1, now = 1;
        if (i < m) {
            was = sf.conv[i];
            const double ri = S::d(res[i]);
            res_out[(size_t)j * m + i] = ri;
            now = was || ri <= target[(size_t)j * m + i];
            if (now && !was) {
                sf.conv[i] = 1;
                if (conv_step) conv_step[(size_t)j * m + i] = k;
            }
        }
        const int any_before = __any_sync(0xffffffffu, !was), any_after = __any_sync(0xffffffffu, !now);
        if (i == 0) {
            active[j] = freeze ? any_before : 1;
            sf.alive = any_after;
        }
    }
}

// The recurrences of every shift; the CTA that arrives last closes the block
// step: counters, beta_k <- beta_{k+1}, k++.
template <class T>
__global__ void __launch_bounds__(NT) small_recur_kernel(SmallStateT<T>* ss, Ctl* ctl, int s, int m,
                                                         const double* __restrict__ sigma,
                                                         const double* __restrict__ target, int freeze, int wprec,
                                                         void* coefU_w, void* coefL_w, int* ce, int* active,
                                                         int* conv_step, double* res_out, int MM, int step, int ahead) {
    // Launched ahead of v_update's end: the recurrences of this step need the
    // QR, not V = W S.  The QR releases the step's number after it has written
    // what they take (all earlier kernels were complete for it); a CTA that
    // acquires that number runs beside v_update, any other waits for v_update's
    // end.  (It let this kernel in after its own wait, so the number is normally
    // there.)  The last CTA waits for v_update before it closes the step, whose
    // widths v_update reads, so this kernel ends after it.  The release and the
    // acquire take 0.1-0.2 of the 7.3 ms of a 4^4 FP64 solve with m = 4.
    const bool beside = ahead && __syncthreads_or(threadIdx.x == 0 && ld_acquire(&ss->sh.qr_step) == (unsigned)step);
    if (!beside) step_begin();
    if (cget(ctl->done)) return;
    extern __shared__ __align__(16) unsigned char sm[];
    shift_recurrence<T>(ss, ctl, (int)blockIdx.x, m, sigma, target, freeze, wprec, coefU_w, coefL_w, ce, active,
                        conv_step, res_out, MM, sm);
    if (!last_arrival(&ss->sh.ticket[2])) return;
    if (beside) step_begin();
    const int j = threadIdx.x;                     // s <= S_MAX shifts
    const int nalive = __syncthreads_count(j < s && __ldcg(&ss->sf[j < s ? j : 0].alive));
    const int nkd = __syncthreads_count(j < s && __ldcg(&active[j < s ? j : 0]));
    const int mk_ = cget(ctl->mk), mn = cget(ctl->mnext), mp = cget(ctl->k) > 1 ? cget(ctl->mprev) : 0;
    for (int t = threadIdx.x; t < M_MAX * M_MAX; t += blockDim.x) ss->sh.betak[t] = ss->sh.betan[t];
    __syncthreads();
    if (threadIdx.x == 0) {
        const int k = cget(ctl->k);
        ctl->mvms = cget(ctl->mvms) + mk_;
        ctl->f_dslash = cget(ctl->f_dslash) + 4LL * mk_;                 // D: V in, Z out; D^H: Z in, Y out
        ctl->f_gram = cget(ctl->f_gram) + 3LL * mk_;                     // V, Y for alpha; W for W^H W
        // Y, V_k, V_{k-1} in, W out; V_{k+1} = W S
        ctl->f_update = cget(ctl->f_update) + 3LL * mk_ + mp + mk_ + mn;
        if (nkd > 0) ctl->f_shift_s = cget(ctl->f_shift_s) + mn;         // V_{k+1} rows, read once per row tile
        // X_j += P_j Ut_j, P_j <- V - P_j Lh_j
        ctl->f_shift_cmac = cget(ctl->f_shift_cmac) + (long long)nkd * mk_ * (m + mn);
        ctl->hmk[(k - 1) & (CTL_HIST - 1)] = mk_;
        ctl->hmn[(k - 1) & (CTL_HIST - 1)] = mn;
        ctl->last_step = k;
        ctl->nact = nalive;
        ctl->k = k + 1;
        ctl->mprev = mk_;
        ctl->mk = mn;
        if (mn == 0 || nalive == 0 || __ldcg(&ctl->status) != 0) ctl->done = 1;
    }
}

size_t qr_smem(int MM) { return 4 * (size_t)MM * MM * sizeof(double2) + 3 * MM * sizeof(double) + M_MAX * sizeof(int); }
size_t recur_smem(int MM) { return 7 * (size_t)MM * MM * sizeof(double2) + MM * sizeof(double2) + (MM + 2) * sizeof(double); }

template <class T>
SmallStateT<T>* as_state(SmallState* ss) { return reinterpret_cast<SmallStateT<T>*>(ss); }

}  // namespace

// sfp64: FP64 m x m scalar (FP64 storage, or reduced storage on request),
// otherwise double-float; wprec: precision of the Gram partials (FP64 for
// FP64 storage, else FP32) and of the coefficient copies
void launch_small_init(SmallState* ss, Ctl* ctl, const double2* G0, const double* ref, int m, int s, double dtol,
                       int sfp64, cudaStream_t st) {
    auto bytes = [](int w) {
        return 4 * (size_t)w * w * sizeof(double2) + M_MAX * sizeof(int) + 3 * M_MAX * sizeof(double);
    };
    // above 48 KB from m = 28 on
    static std::atomic<unsigned long long> devs64{0}, devsdd{0};
    max_dyn_smem_once(small_init_kernel<double2>, (int)bytes(M_MAX), devs64);
    max_dyn_smem_once(small_init_kernel<ddc>, (int)bytes(M_MAX), devsdd);
    if (sfp64)
        small_init_kernel<double2><<<1, QW * WS, bytes(m), st>>>(as_state<double2>(ss), ctl, G0, ref, m, s, dtol);
    else
        small_init_kernel<ddc><<<1, QW * WS, bytes(m), st>>>(as_state<ddc>(ss), ctl, G0, ref, m, s, dtol);
}

void launch_small_alpha(SmallState* ss, const Ctl* ctl, const double* partials, int nblk, int nf_max, int wprec,
                        int sfp64, void* coef_a, void* coef_bh, int* ce, Stream st) {
    if (sfp64)
        launch_step(small_alpha_kernel<double2>, NRC, NT, 0, st, as_state<double2>(ss), ctl, partials, nblk, nf_max, wprec,
                                                        coef_a, coef_bh, ce);
    else
        launch_step(small_alpha_kernel<ddc>, NRC, NT, 0, st, as_state<ddc>(ss), ctl, partials, nblk, nf_max, wprec, coef_a,
                                                    coef_bh, ce);
}

void launch_small_qr(SmallState* ss, Ctl* ctl, const double* partials, int nblk, int m, double dtol, int wprec,
                     int sfp64, void* coefS_w, int* ce, Stream st) {
    static std::atomic<unsigned long long> devs64{0}, devsdd{0};
    max_dyn_smem_once(small_qr_kernel<double2>, (int)qr_smem(M_MAX), devs64);
    max_dyn_smem_once(small_qr_kernel<ddc>, (int)qr_smem(M_MAX), devsdd);
    // matrices at the initial width m, which block widths never exceed
    if (sfp64)
        launch_step(small_qr_kernel<double2>, NRC, NT, qr_smem(m), st, as_state<double2>(ss), ctl, partials, nblk, m, dtol,
                                                              wprec, coefS_w, ce, m);
    else
        launch_step(small_qr_kernel<ddc>, NRC, NT, qr_smem(m), st, as_state<ddc>(ss), ctl, partials, nblk, m, dtol, wprec,
                                                          coefS_w, ce, m);
}

void launch_small_recur(SmallState* ss, Ctl* ctl, int s, int m, const double* sigma_dev, const double* target_dev,
                        int freeze, int wprec, int sfp64, void* coefU_w, void* coefL_w, int* ce, int* active,
                        int* conv_step, double* res_out, int step, Stream st) {
    static std::atomic<unsigned long long> devs64{0}, devsdd{0};
    max_dyn_smem_once(small_recur_kernel<double2>, (int)recur_smem(M_MAX), devs64);
    max_dyn_smem_once(small_recur_kernel<ddc>, (int)recur_smem(M_MAX), devsdd);
    if (sfp64)
        launch_step(small_recur_kernel<double2>, s, NT, recur_smem(m), st, as_state<double2>(ss), ctl, s, m, sigma_dev,
                                                                  target_dev, freeze, wprec, coefU_w, coefL_w, ce, active,
                                                                  conv_step, res_out, m, step, st.ahead);
    else
        launch_step(small_recur_kernel<ddc>, s, NT, recur_smem(m), st, as_state<ddc>(ss), ctl, s, m, sigma_dev, target_dev,
                                                              freeze, wprec, coefU_w, coefL_w, ce, active, conv_step,
                                                              res_out, m, step, st.ahead);
}

}  // namespace dsbcg
