// The Wilson stencil of FP64 fields in block fixed point, on the integer
// multiply-add pipe.
//
// GB300 retires 2 FP64 FMA per SM and clock but 64 32 x 32 -> 64 bit integer
// multiply-adds (measured: 2.0 and 63.4), so the products of the stencil are
// formed in integers: a real number is two limbs h 2^29 + l with |l| <= 2^28,
// and a real multiply-add is three mad.wide (h h, h l, l h; the l l product
// is below the last bit kept).  Limbs add without carries, so the spin
// projections are 32-bit adds.
//
// Format of a field ("FX"): [32-site tile][spin-colour component 12][site of
// the tile] int4 (re.h, re.l, im.h, im.l), so that a hop's loads are one
// address and immediate offsets, and one exponent per site: component value =
// (h 2^29 + l) 2^E with |h 2^29 + l| <= 2^57, the largest component of the
// site above 2^56.  Links: the limbs of -k' u 2^58, where kappa = k' 2^-ks with
// |k'| < 1, [mu][entry][site]; links in SU(3) only (|u| <= 1).  The factor
// 2^-ks is an exponent offset of the hopping term.
//
// Error.  A unit is 2^Em, Em the largest exponent of the terms of a site.  A
// hop is exact to 10 units at most: 2.5 from components rounded in the
// conversion, 3.8 from the rounding of k' u, 1.5 from the dropped l l products
// and 2 from shifts that round down (all of one sign); the diagonal term to 9
// and a result kept in the format to 32.  Together 120 units in the worst case
// and about 8 typically, a unit being at most 2^-57 of the largest component of
// the nine sites times kappa.  That is an error bound per SITE: relative to the
// largest component around it, below that of an FP64 chain.
//
// Components.  An FP64 chain of 16 operations has every single complex component
// to 16 x 2^-53 of T, the sum of the magnitudes of its terms, also where all of
// them are far below the site's largest component (a colour or spin that the
// links do not mix with a larger one, a single site between zeros).  The format
// does not.  An application that a caller sees (flag given, CHECK) therefore adds
// up T, as |re| + |im| of the diagonal term and of each hop's share, and sets
// *flag where T is below FX_LOW = 2^55 units and the nine sites are not all zero:
// then the error can exceed 120 / 2^55 = 30 x 2^-53 of T, and dsbcg_apply repeats
// the call with the FP64 kernels.  Dense fields do not come near: the smallest T
// of 1.6 million components of Gaussian fields was 2^56.3 to 2^57.4 units (kappa
// 0.11 to 0.13; half lattice 2^56.0), and the tail falls with the 16th power.
// Sparse sources and fields that fall by decades from site to site do.  The check
// takes 2% of an application (A to 12 fields of 16^3 x 32: 1.12 -> 1.14 ms), and
// a call that fails it 0.05 to 1.1 ms more than the FP64 kernels (4^4: 0.095 ->
// 0.144 ms, 16^3 x 32: 5.26 -> 6.35).
// A solve's applications do not check: its contract is the norm of the residual.
//
// Overflow.  The limbs of a projected half spinor are at most 2^29 (sums of
// two), those of a link at most 2^29 and 2^28.  A link row has norm <= 1, so
// the h h sums of a component stay below 2^29 2^29 sqrt(6) < 2^60, the mixed
// sums below 2^61, a hop's result below 2^59.3 (sqrt(6) 2^58).  The diagonal term
// may lie 2^4 above the accumulators' unit, so that it reaches 2^61: the sum over
// eight hops (2^62.3) and the diagonal term stays below 2^62.8, and no term may
// take another bit.
//
// A site that is all zero has exponent FX_ZERO.  A component that the
// conversion holds as zero beside larger ones sets *flag.  A site with a NaN, an
// infinity or a largest exponent outside the range in which every result is
// a normal FP64 number sets *flag and turns its neighbourhood into NaN
// (FX_NAN) or, when tiny, counts as zero; dsbcg_apply then repeats the
// application with the FP64 kernels.
#include "fx.cuh"
#include "kernels.h"

namespace dsbcg {

namespace {

// biased exponents of a site's largest component for which the FX path holds
constexpr int FX_EB_MIN = 300, FX_EB_MAX = 1800;
constexpr int FX_TILE = 12 * 32;               // int4 per 32-site tile

// element of component 0 of site y
__device__ __forceinline__ size_t fx_at(int y) { return (size_t)(y >> 5) * FX_TILE + (y & 31); }

// FP64 field block -> FX fields and site exponents.  One thread per (site,
// field).  Bound by HBM: 16 bytes per complex in and out.  Canonical input (192
// contiguous bytes per thread: a sector serves two of a thread's loads, from
// L1) takes 101 us for 12 fields of 16^3 x 32, pair-chunk input 84; the packing
// pass that it spares takes 90, and as much again on the output side, where
// the stencil writes the canonical layout itself at no cost that could be
// measured.  A to those fields through dsbcg_apply: 1.28 -> 1.12 ms; to 4 of
// 4^4: 57 -> 53 us.
__global__ void __launch_bounds__(128) fx_convert_kernel(int4* __restrict__ out, int* __restrict__ eo,
                                                         const double2* in, Lay64 li, size_t ld,
                                                         int V, const Ctl* ctl, int nf_static,
                                                         int* __restrict__ flag, int ahead) {
    step_begin();
    int nf = nf_static;
    if (ctl) {
        if (cget(ctl->done, ahead)) return;
        nf = cget(ctl->mk, ahead);
    }
    const int x = (int)(blockIdx.x * 128u + threadIdx.x), f = (int)blockIdx.y;
    if (f >= nf || x >= V) return;
    const double2* p = in + (size_t)f * li.fs + (size_t)x * li.xs;
    double2 v[12];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const double2* q = p + c * li.cs;
        v[2 * c] = q[0];
        v[2 * c + 1] = q[1];
    }
    int mx = 0;
    unsigned any = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const int a = __double2hiint(v[c].x) & 0x7fffffff, b = __double2hiint(v[c].y) & 0x7fffffff;
        mx = max(mx, max(a, b));
        any |= (unsigned)(a | b) | (unsigned)__double2loint(v[c].x) | (unsigned)__double2loint(v[c].y);
    }
    const int eb = mx >> 20;
    int E = eb - 1079;
    if (!any) {
        E = FX_ZERO;
    } else if (eb > FX_EB_MAX) {
        E = FX_NAN;
        if (flag) atomicOr(flag, 1);
    } else if (eb < FX_EB_MIN) {
        E = FX_ZERO;
        if (flag) atomicOr(flag, 1);
    }
    const bool live = E != FX_ZERO && E != FX_NAN;
    eo[(size_t)f * V + x] = E;
    int4* o = out + (size_t)f * ld + fx_at(x);
    bool lost = false;                         // a component that the format holds as zero
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const int2 re = fx_split(live ? fx_of_double(v[c].x, eb) : 0ll);
        const int2 im = fx_split(live ? fx_of_double(v[c].y, eb) : 0ll);
        o[c * 32] = make_int4(re.x, re.y, im.x, im.y);
        lost |= !(re.x | re.y | im.x | im.y) && (v[c].x != 0.0 || v[c].y != 0.0);
    }
    if (flag && lost && live) atomicOr(flag, 1);
}

// canonical links -> FX links [mu][entry][site]; kfix = -k' 2^63.  The product
// k' u is formed from u 2^62 (exact above 2^-9) in 128 bits.
__global__ void fx_pack_links_kernel(int4* __restrict__ dst, const double2* __restrict__ src, size_t V,
                                     long long kfix) {
    const size_t total = V * 36;
    auto limbs = [&](double u) {
        const long long p = __mul64hi(__double2ll_rn(ldexp(u, 62)), kfix);      // -k' u 2^61
        return fx_split((p + 4) >> 3);
    };
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
         t += (size_t)gridDim.x * blockDim.x) {
        const size_t x = t % V;
        const int r = (int)(t / V);                       // mu * 9 + entry
        const double2 u = src[x * 36 + r];
        const int2 re = limbs(u.x), im = limbs(u.y);
        dst[t] = make_int4(re.x, re.y, im.x, im.y);
    }
}

__device__ __forceinline__ int4 iadd(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ int4 isub(int4 a, int4 b) { return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
// a + i b, a - i b
__device__ __forceinline__ int4 iaddi(int4 a, int4 b) { return make_int4(a.x - b.z, a.y - b.w, a.z + b.x, a.w + b.y); }
__device__ __forceinline__ int4 isubi(int4 a, int4 b) { return make_int4(a.x + b.z, a.y + b.w, a.z - b.x, a.w - b.y); }

struct ll2 {
    long long x, y;
};
// |v| 2^-32, to one unit
__device__ __forceinline__ unsigned fx_high(long long v) { return (unsigned)abs((int)(v >> 32)); }
// a += s q, s = +1 (PLUS) or -1, or s i q (ROT)
template <bool PLUS, bool ROT>
__device__ __forceinline__ void lacc(ll2& a, ll2 q) {
    const long long x = ROT ? -q.y : q.x, y = ROT ? q.x : q.y;
    if (PLUS) { a.x += x; a.y += y; }
    else { a.x -= x; a.y -= y; }
}

// One hop, for the half-spinor component (spin) S of a site: p the
// neighbour's components (stride 32), su the hop's link in shared memory
// (entry stride 32; U^H already for a backward hop), sh the shift from the
// hop's exponent to the accumulators'.  MINUS: projector 1 - gamma_MU, else
// 1 + gamma_MU.  The result goes to spin S (up) and to the lower spin it
// rebuilds (lo): the other thread's for mu = x, y, this thread's for z, t.
// CHECK: mg[a] += |re| + |im| of the component's share (high words).
template <int MU, bool MINUS, int S, bool AHEAD, bool CHECK>
__device__ __forceinline__ void fx_hop(const int4* p, const int4* su, int sh, ll2 up[3], ll2 lo[3], unsigned mg[3]) {
    constexpr int T = MU < 2 ? 1 - S : S;                 // lower spin of the projection
    constexpr bool NEG = (MU == 1 || MU == 2) && S == 1 ? !MINUS : MINUS;
    int4 h[3];
    int2 ni[3];                                           // minus the imaginary parts
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int4 u = ld_prev<AHEAD>(p + (S * 3 + a) * 32), l = ld_prev<AHEAD>(p + ((2 + T) * 3 + a) * 32);
        if (MU == 0 || MU == 2) h[a] = NEG ? isubi(u, l) : iaddi(u, l);
        else h[a] = NEG ? isub(u, l) : iadd(u, l);
        ni[a] = make_int2(-h[a].z, -h[a].w);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        long long hr = 0, hi = 0, mr = 0, mi = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 u = su[(a * 3 + b) * 32];
            const int4 v = h[b];
            hr += (long long)u.x * v.x;
            hi += (long long)u.x * v.z;
            mr += (long long)u.x * v.y;
            mi += (long long)u.x * v.w;
            hr += (long long)u.z * ni[b].x;
            hi += (long long)u.z * v.x;
            mr += (long long)u.y * v.x;
            mi += (long long)u.y * v.z;
            mr += (long long)u.z * ni[b].y;
            mi += (long long)u.z * v.y;
            mr += (long long)u.w * ni[b].x;
            mi += (long long)u.w * v.x;
        }
        ll2 q;
        q.x = (hr + (mr >> FX_BASE)) >> sh;
        q.y = (hi + (mi >> FX_BASE)) >> sh;
        if (CHECK) mg[a] += fx_high(q.x) + fx_high(q.y);
        lacc<true, false>(up[a], q);
        // lower spins of 1 - gamma_mu: i q for x, (q1, -q0) for y, (i q0, -i q1)
        // for z and -q for t; the opposite for 1 + gamma_mu
        if (MU == 0) lacc<MINUS, true>(lo[a], q);
        if (MU == 1) lacc<(S == 1) == MINUS, false>(lo[a], q);
        if (MU == 2) lacc<(S == 0) == MINUS, true>(lo[a], q);
        if (MU == 3) lacc<!MINUS, false>(lo[a], q);
    }
}

// the four hops in x, y (HALFH = 0) or z, t (1); sy: their neighbour sites
// (stride 32), sh: their shifts, six bits each
template <bool DAG, int S, int HALFH, bool AHEAD, bool CHECK>
__device__ __forceinline__ void fx_hops(const int4* fin, const int* sy, const int4* sl, unsigned sh,
                                        ll2 up[3], ll2 lo[3], unsigned mg[3]) {
    constexpr int HS = 9 * 32, M = 2 * HALFH;
    sy += 4 * 32 * HALFH;
    sl += 4 * HS * HALFH;
    fx_hop<M, !DAG, S, AHEAD, CHECK>(fin + fx_at(sy[0]), sl, (int)sh & 63, up, lo, mg);
    fx_hop<M, DAG, S, AHEAD, CHECK>(fin + fx_at(sy[32]), sl + HS, (int)(sh >> 6) & 63, up, lo, mg);
    fx_hop<M + 1, !DAG, S, AHEAD, CHECK>(fin + fx_at(sy[64]), sl + 2 * HS, (int)(sh >> 12) & 63, up, lo, mg);
    fx_hop<M + 1, DAG, S, AHEAD, CHECK>(fin + fx_at(sy[96]), sl + 3 * HS, (int)(sh >> 18) & 63, up, lo, mg);
}

// out = src - kappa H in (H the hopping term; DAG: gamma_5 H gamma_5), fields
// in FX; out FP64 (laid out by lo, OUT64) or FX.  src = in gives D (D^H).
// HALF: in on the other parity of the even-odd lattice, src and out on
// `parity`.  src NULL and neg: out = kappa H in.
//
// A CTA covers 32 sites of FX_FIELDS fields, two warps per field (one per
// spin of the half spinor: half the accumulators and operands per thread),
// with the tile's eight links per site staged in shared memory once (36 KB;
// backward links as U^H, the time-boundary sign folded in).  A thread first
// takes the x and y hops, whose lower-spin sums belong to the other warp and
// go to it through shared memory, then the z and t hops, so that only one set
// of lower-spin sums is in registers.
//
// Bound: per site and field 1728 mad.wide at 64 per SM and clock, 27 clocks,
// beside about as many adds, shifts and shared-memory loads; latency-bound at
// 16 warps per SM (IPC 1.6).  Measured, 16^3 x 32, 12 fields, one D: 0.47 ms
// against 2.51 ms of the FP64 kernel; 4^4, 4 fields: 12 against 36 us.  Other
// shapes: one thread per site and field 0.60 ms; 80 registers and 24 warps
// 0.50 (spills); 2 or 3 fields per CTA 0.57-0.60 (links staged more often).
constexpr int FX_FIELDS = 4;
constexpr unsigned FX_LOW = 1u << 23;                          // 2^55 units
static_assert(2 * FX_FIELDS <= 8, "the exchange of leading-zero counts reuses the 8 x 32 words of the sites");

template <bool DAG, bool OUT64, bool HALF, bool AHEAD, bool CHECK>
__global__ void __launch_bounds__(64 * FX_FIELDS, 2) fx_stencil_kernel(
    void* __restrict__ outv, int* __restrict__ eo, const int4* in, const int* ei,
    const int4* src, const int* es, size_t ld, const int4* __restrict__ links, Geom g,
    int kshift, int neg, int parity, Lay64 lo64, int* flag, const Ctl* ctl, int nf_static, int ngrp) {
    if (!AHEAD) step_begin();                                  // else after staging the links (as dslash_cta_kernel)
    extern __shared__ __align__(16) unsigned char fx_smem[];
    int4* sl = reinterpret_cast<int4*>(fx_smem);               // [hop][entry][lane]
    ll2* ex = reinterpret_cast<ll2*>(sl + 8 * 9 * 32);         // [warp][colour][lane]
    int* sy = reinterpret_cast<int*>(ex + 2 * FX_FIELDS * 3 * 32);     // [hop][lane]
    unsigned* sg = reinterpret_cast<unsigned*>(sy + 8 * 32);           // CHECK: [warp][colour][lane], twice
    int nf = nf_static;
    const int nw = (int)(blockDim.x >> 5), nfc = nw >> 1;      // warps, fields of the CTA
    const int grp = (int)(blockIdx.x % (unsigned)ngrp);
    auto idle = [&]() {                                        // CTA-uniform
        if (ctl) {
            if (cget(ctl->done, AHEAD)) return true;
            nf = cget(ctl->mk, AHEAD);
        }
        return grp * nfc >= nf;
    };
    if (!AHEAD && idle()) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const size_t V = (size_t)g.V;
    const int Vf = HALF ? g.V / 2 : g.V;
    const int k = (int)(blockIdx.x / (unsigned)ngrp) * 32 + lane;
    const int ks = k < Vf ? k : Vf - 1;
    int c[4], x;
    if (HALF) {
        const int hx = g.L[0] / 2;
        const int row = ks / hx;
        c[1] = row % g.L[1];
        c[2] = (row / g.L[1]) % g.L[2];
        c[3] = row / (g.L[1] * g.L[2]);
        c[0] = 2 * (ks % hx) + ((parity + c[1] + c[2] + c[3]) & 1);
        x = c[0] + g.L[0] * row;
    } else {
        x = ks;
        c[0] = x % g.L[0];
        int r = x / g.L[0];
        c[1] = r % g.L[1];
        r /= g.L[1];
        c[2] = r % g.L[2];
        c[3] = r / g.L[2];
    }
    // warp w stages the hops w, w + nw, ...: neighbour site and link
    for (int h = w; h < 8; h += nw) {
        const int mu = h >> 1;
        const bool fwd = (h & 1) == 0;
        int st = 1;
        for (int d = 0; d < mu; ++d) st *= g.L[d];
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3], L = g.L[mu];
        const bool wrap = fwd ? cm == L - 1 : cm == 0;
        const int y = x + (fwd ? st : -st) * (wrap ? 1 - L : 1);
        const bool edge = mu == 3 && g.tap && wrap;
        const int s = edge != (neg != 0) ? -1 : 1, sz = fwd ? s : -s;      // conjugate: the imaginary part's sign
        const int4* u = links + (size_t)mu * 9 * V + (fwd ? x : y);
        sy[h * 32 + lane] = HALF ? y >> 1 : y;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 q = __ldg(u + (size_t)e * V);
            sl[(h * 9 + (fwd ? e : (e % 3) * 3 + e / 3)) * 32 + lane] = make_int4(s * q.x, s * q.y, sz * q.z, sz * q.w);
        }
    }
    if (AHEAD) {
        step_begin();
        if (idle()) return;
    }
    __syncthreads();
    const int S = w & 1;
    const int f = grp * nfc + (w >> 1);
    const bool on = f < nf;                                    // warp-uniform
    ll2 up[3], lo[3];
    int Em = FX_ZERO, e0 = FX_ZERO;
    const int4* fin = in + (size_t)f * ld;
    unsigned shl = 0, shh = 0;
    bool low = false;                                          // CHECK: a component whose terms are too small
    // the diagonal term of spin s in the accumulators' unit (zero without src); CHECK: its magnitudes in dg
    auto diag = [&](int s, ll2 d[3], unsigned dg[3]) {
        const int4* p = src + (size_t)f * ld + fx_at(ks) + s * 96;
        const int sr = max(0, min(Em - e0, 63)), sf = max(0, e0 - Em);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            d[a] = ll2{0, 0};
            if (CHECK) dg[a] = 0;
            if (src) {
                const int4 u = ld_prev<AHEAD>(p + a * 32);
                d[a] = ll2{fx_join(u.x, u.y) >> sr << sf, fx_join(u.z, u.w) >> sr << sf};
                if (CHECK) dg[a] = fx_high(d[a].x) + fx_high(d[a].y);
            }
        }
    };
    if (on) {
        const int* fe = ei + (size_t)f * Vf;
        if (src) e0 = ld_prev<AHEAD>(es + (size_t)f * Vf + ks);
        int eh[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) {
            eh[h] = ld_prev<AHEAD>(fe + sy[h * 32 + lane]) - kshift;
            Em = max(Em, eh[h]);
        }
        // the diagonal term (at most 2^57) has bits to spare: its unit may be up to 2^4 of the accumulators'
        Em = max(Em, e0 - 4);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            shl |= (unsigned)min(Em - eh[h], 63) << (6 * h);
            shh |= (unsigned)min(Em - eh[4 + h], 63) << (6 * h);
        }
        // CHECK: mg[a] sums the magnitudes of upper component a; the shares of the
        // x, y hops also belong to the other warp's lower component (at), and
        // own turns the sum into that of this thread's lower component
        unsigned mg[3], dg[3];
        unsigned *at = sg + (w * 3) * 32 + lane, *own = at + 2 * FX_FIELDS * 3 * 32;
        diag(S, up, mg);
        if (CHECK) {
#pragma unroll
            for (int a = 0; a < 3; ++a) own[a * 32] = mg[a];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) lo[a] = ll2{0, 0};
        if (S == 0) fx_hops<DAG, 0, 0, AHEAD, CHECK>(fin, sy + lane, sl + lane, shl, up, lo, mg);
        else fx_hops<DAG, 1, 0, AHEAD, CHECK>(fin, sy + lane, sl + lane, shl, up, lo, mg);
#pragma unroll
        for (int a = 0; a < 3; ++a) ex[(w * 3 + a) * 32 + lane] = lo[a];
        diag(2 + S, lo, dg);
        if (CHECK) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                at[a * 32] = mg[a] - own[a * 32];
                own[a * 32] = dg[a] - mg[a];
            }
        }
        if (S == 0) fx_hops<DAG, 0, 1, AHEAD, CHECK>(fin, sy + lane, sl + lane, shh, up, lo, mg);
        else fx_hops<DAG, 1, 1, AHEAD, CHECK>(fin, sy + lane, sl + lane, shh, up, lo, mg);
        if (CHECK) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                own[a * 32] += mg[a];                          // without the x, y hops of the other warp
                low |= mg[a] < FX_LOW;
            }
        }
    }
    __syncthreads();
    if (on) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const ll2 q = ex[((w ^ 1) * 3 + a) * 32 + lane];
            lo[a].x += q.x;
            lo[a].y += q.y;
            if (CHECK) {
                low |= sg[((w ^ 1) * 3 + a) * 32 + lane] + sg[((w + 2 * FX_FIELDS) * 3 + a) * 32 + lane] < FX_LOW;
            }
        }
    }
    const bool bad = Em > FX_NAN / 2;
    const bool store = on && k < Vf;
    // (all nine sites zero: so is the result)
    if (CHECK && store && low && Em > FX_ZERO / 2 && __ldcg(flag) == 0) atomicOr(flag, 1);
    if (OUT64) {
        // v 2^Em: the conversion rounds to FP64, the exponent is added to its bits (the result is a normal
        // number: FX_EB_MIN, FX_EB_MAX)
        if (!store) return;
        double2* o = reinterpret_cast<double2*>(outv) + (size_t)f * lo64.fs + (size_t)k * lo64.xs;
        auto out = [&](long long v) -> double {
            const double d = __ll2double_rn(v);
            if (bad) return __longlong_as_double(0x7ff8000000000000ll);
            return v ? __hiloint2double(__double2hiint(d) + Em * (1 << 20), __double2loint(d)) : 0.0;
        };
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int i = S * 3 + a, j = (2 + S) * 3 + a;
            o[(i >> 1) * lo64.cs + (i & 1)] = make_double2(out(up[a].x), out(up[a].y));
            o[(j >> 1) * lo64.cs + (j & 1)] = make_double2(out(lo[a].x), out(lo[a].y));
        }
    } else {
        unsigned long long mag = 0;
        if (!on) up[0] = up[1] = up[2] = lo[0] = lo[1] = lo[2] = ll2{0, 0};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            mag |= (unsigned long long)(up[a].x ^ (up[a].x >> 63)) | (unsigned long long)(up[a].y ^ (up[a].y >> 63));
            mag |= (unsigned long long)(lo[a].x ^ (lo[a].x >> 63)) | (unsigned long long)(lo[a].y ^ (lo[a].y >> 63));
        }
        // bits of the site's largest magnitude, over both warps -> FX_BITS
        int* ez = sy;                                          // the neighbour sites are no longer needed
        ez[w * 32 + lane] = __clzll((long long)mag);
        __syncthreads();
        if (!store) return;
        const int lz = min(ez[w * 32 + lane], ez[(w ^ 1) * 32 + lane]);
        const int sft = lz - (64 - FX_BITS);
        int4* o = reinterpret_cast<int4*>(outv) + (size_t)f * ld + fx_at(k);
        if (S == 0) eo[(size_t)f * Vf + k] = bad ? FX_NAN : (lz < 64 ? Em - sft : FX_ZERO);
        auto limbs = [&](long long v) { return fx_split(sft >= 0 ? v << sft : fx_shift(v, -sft)); };
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int2 ur = limbs(up[a].x), ui = limbs(up[a].y), lr = limbs(lo[a].x), li = limbs(lo[a].y);
            o[(S * 3 + a) * 32] = make_int4(ur.x, ur.y, ui.x, ui.y);
            o[((2 + S) * 3 + a) * 32] = make_int4(lr.x, lr.y, li.x, li.y);
        }
    }
}

// kappa = k 2^-*shift with 1/2 <= |k| < 1 (0 for 0)
double fx_mantissa(double kappa, int* shift) {
    int e = 0;
    const double k = frexp(kappa, &e);
    *shift = kappa == 0.0 ? 0 : -e;
    return k;
}

}  // namespace

bool fx_kappa_fits(double kappa) { return kappa == 0.0 || (fabs(kappa) > 1e-9 && fabs(kappa) < 1e3); }

void launch_fx_links(void* dst, const double2* src, size_t V, double kappa, cudaStream_t st) {
    int ks;
    const long long kfix = -(long long)ldexp(fx_mantissa(kappa, &ks), 63);
    const size_t grid = (V * 36 + 255) / 256;
    fx_pack_links_kernel<<<(unsigned)(grid < 65535 ? grid : 65535), 256, 0, st>>>((int4*)dst, src, V, kfix);
}

void launch_fx_convert(void* out, int* eo, const void* in, const Lay64& li, size_t ld, size_t Vf, const Ctl* ctl,
                       int nf_static, int nf_max, int* flag, Stream st) {
    const int nfg = ctl ? nf_max : nf_static;
    const dim3 grid((unsigned)((Vf + 127) / 128), (unsigned)nfg);
    launch_step(fx_convert_kernel, grid, 128, 0, st, (int4*)out, eo, (const double2*)in, li, ld, (int)Vf, ctl, nf_static, flag,
                st.ahead);
}

void launch_fx_stencil(void* out, int* eo, const void* in, const int* ei, const void* src, const int* es, size_t ld,
                       const void* links, const Geom& g, double kappa, int dag, int half, int parity, const Lay64* lo,
                       int* flag, const Ctl* ctl, int nf_static, int nf_max, Stream st) {
    const int nfg = ctl ? nf_max : nf_static;
    const int nfc = nfg < FX_FIELDS ? nfg : FX_FIELDS;
    const int ngrp = (nfg + nfc - 1) / nfc;
    const size_t Vf = half ? (size_t)g.V / 2 : (size_t)g.V;
    const unsigned grid = (unsigned)((size_t)ngrp * ((Vf + 31) / 32));
    int ks;
    fx_mantissa(kappa, &ks);
    const int neg = src ? 0 : 1;
    const Lay64 l64 = lo ? *lo : Lay64{};
    constexpr int SMEM0 = 8 * 9 * 32 * sizeof(int4) + 2 * FX_FIELDS * 3 * 32 * sizeof(ll2) + 8 * 32 * sizeof(int);
    constexpr int SMEMC = SMEM0 + 2 * 2 * FX_FIELDS * 3 * 32 * sizeof(unsigned);
#define DSBCG_FX2(DAG, O64, HALF, AHEAD, CHECK)                                                                     \
    {                                                                                                              \
        constexpr int SMEM = CHECK ? SMEMC : SMEM0;                                                                \
        static std::atomic<unsigned long long> devs{0};                                                            \
        max_dyn_smem_once(fx_stencil_kernel<DAG, O64, HALF, AHEAD, CHECK>, SMEM, devs);                            \
        launch_step(fx_stencil_kernel<DAG, O64, HALF, AHEAD, CHECK>, grid, 64 * nfc, SMEM, st, out, eo,            \
                    (const int4*)in, ei, (const int4*)src, es, ld, (const int4*)links, g, ks, neg, parity, l64,    \
                    flag, ctl, nf_static, ngrp);                                                                   \
    }
    // (an application that checks its components is never launched ahead)
#define DSBCG_FX(DAG, O64, HALF)                          \
    if (flag) DSBCG_FX2(DAG, O64, HALF, false, true)      \
    else if (st.ahead) DSBCG_FX2(DAG, O64, HALF, true, false) \
    else DSBCG_FX2(DAG, O64, HALF, false, false)
#define DSBCG_FX1(O64, HALF) \
    if (dag) { DSBCG_FX(true, O64, HALF) } else { DSBCG_FX(false, O64, HALF) }
    if (half) {
        if (lo) { DSBCG_FX1(true, true) } else { DSBCG_FX1(false, true) }
    } else {
        if (lo) { DSBCG_FX1(true, false) } else { DSBCG_FX1(false, false) }
    }
#undef DSBCG_FX1
#undef DSBCG_FX
#undef DSBCG_FX2
}

}  // namespace dsbcg
