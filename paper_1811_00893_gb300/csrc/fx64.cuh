// FP64 hopping term by fixed-point arithmetic (link format LF = 3).
//
// GB300 issues two FP64 operations per clock and SM, but 64 32x32+64-bit
// integer multiply-adds (mad.wide) at the cost of any other integer multiply
// (both measured).  In FP64 one site's SU(3) products and sums take 864
// operations and bound the hopping term of 32^3 x 64 at 1.6 ms, seven times
// the time its bytes take.  Here a real product is three mad.wide on 59-bit
// fixed-point operands instead of one FP64 FMA:
//
//   link entry   w = n_w 2^-59, n_w = wh 2^31 + wl (wh signed, 0 <= wl < 2^31),
//                rounded to nearest at set-up: exact for |w| >= 2^-6;
//   half spinor  the 12 reals of a projected neighbour (projected in FP64, as in
//                the FP64 kernel) in units of 2^(e-1023-58), e an exponent of the
//                site that no neighbour so far exceeds: |n_x| < 2^59, cut towards
//                zero, exact for values within 2^-6 of 2^(e-1023);
//   product sum  six products wh xh (units of 2^62) and the twelve cross products
//                wh xl + wl xh (units of 2^31) are summed exactly in 64 bits; the
//                wl xl terms (below 2^-57 of the largest) are dropped; the cross
//                sum is rounded to the nearest unit of 2^62 and added;
//   site sum     24 signed 64-bit sums in units of 2^(e-1023-55).  When a neighbour
//                exceeds e, e is raised past it (one more bit the first time, so
//                that neighbours of like size rarely need another) and the sums
//                are shifted, rounding to nearest.
//
// Errors, in units of the site sum: a hop adds at most 6 for its wl xl terms, 1/2
// for the cross sum, 3/8 for its links' and 1/3 for its neighbour's rounding, a raise
// of e 1/2: 62 in all, 15.5 2^-53 of 2^(e-1023); typically 2.5.  FP64 rounds each of its
// ~16 dependent operations at 2^-53 of the partial sum.  What is small next to
// 2^(e-1023) is computed in FP64 (kFxLeast).
//
// Links that do not fit (fx_check_link in gauge.cu, at set-up: an entry above 1.25, or
// rows or entries too small for multiples of 2^-59) keep plain FP64 for the whole lattice.
//
// Room: link entries have modulus <= 1.25, so |cross sum|
// <= 6 (1.25 + 1) 2^59 < 2^63 and |site sum| <= 8 * 3 * 1.25 * sqrt(2) * 2^56 < 2^62.
// A site whose neighbours hold an infinity or NaN, exceed
// 2^1007 or all lie below 2^-953 goes through fx_site_general, plain FP64.
#pragma once

namespace wl {

static constexpr int kFxMinExp = 70, kFxMaxExp = 2030;  // biased exponents the fixed-point path takes
static constexpr double kFxMaxLink = 1.25;              // largest modulus of a link entry
static constexpr double kFxMinLink = 0.125;             // least modulus of a row's or column's largest (SU(3): 0.57)
// Nonzero entries of modulus below 2^-14 have an error above 2^-45 of themselves.
// One matters where no other link of a site carries the same component, as on
// links near 1: links with such entries are at most one in 1,024 (Haar links: one
// in 10^7; smooth ones of width 0.3: one in 10^6).
static constexpr double kFxTinyLink = 0x1p-14;
static constexpr int kFxTinyShare = 1024;

// n_w as (wh, wl) of one real: the 53-bit significand shifted to units of
// 2^-59, rounded to nearest, ties to even.  Integer operations: with a multiplication
// and a conversion per real on the FP64 pipe, the check's moduli there too and the link
// in local memory, creating a gauge object of 32^3 x 64 in FP64 and FP32 took 6.1 ms, so
// 4.56 (4.42 with FP64 links).
__device__ __forceinline__ void fx_split(double w, int& h, int& l)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(w);
    const int s = 1026 - ((int)(b >> 52) & 0x7ff);  // 3 for 1 <= |w| < 2
    long long n = 0;
    if (s > 0 && s < 64) {  // 2^-60 <= |w| < 8 (links with larger entries are not held so)
        const unsigned long long y = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
        n = (long long)((y + ((1ULL << (s - 1)) - 1) + (y >> s & 1)) >> s);
        if ((long long)b < 0) n = -n;
    }
    h = (int)(n >> 31);
    l = (int)(n & 0x7fffffffLL);
}
__device__ __forceinline__ double fx_join(int h, int l)
{
    return (double)(((long long)h << 31) + l) * 0x1p-59;
}

// a b + c, 32 x 32 + 64 bits, signed: one instruction
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
__device__ __forceinline__ long long fx_mul(int a, int b) { return (long long)a * b; }

// Half a unit of 2^31: the first addend of a cross sum, so that the shift by
// 31 that follows rounds to nearest.  A cut would go downwards, by half a unit on
// average, and move exact values and zeros off theirs; the addend costs no instruction
// (D of 20x18x14x30 takes 71.7 us, 71.3 with the cut).
static constexpr long long kFxHalfUnit = 1LL << 30;

// The site sum: s[(spin * 3 + colour row) * 2 + (0: re, 1: im)]
struct FxSum {
    long long s[24];
    // size of the hops' shares, in units of 2^48: the largest |re| or |im| so far of
    // u0 (low half) and u1 (high half), [x and y hops | z and t hops][colour row]
    unsigned m[2][3];
    int e;     // biased exponent of the units
    bool bad;  // this site needs fx_site_general
};

// A component of the site sum keeps its fixed-point value if some hop's share
// of it reaches 2^-4 of 2^(e-1023) (2^51 units); a component with none is computed
// in FP64 (fx_site_general), whose rounding follows the size of its own terms.  So a
// component's error is below 2^-45 of the sum of its products' moduli, wherever
// those lie below the site's largest.  With neighbours of like size and links that
// mix the colours one component in 10^13 is that small.  Hopping term of
// 24^3 x 48: Gaussian field 138 us (136 without the test), a point source's
// solution 232 us (Haar links) and 294 us (smooth), one spin row 299 us, one colour on
// unit links 770 us, the plain FP64 kernel 524 us.  Half and a quarter of the
// limit: the solutions 210 and 178 us, 172 and 140 us.
static constexpr int kFxLeast = 8;

// The largest of m's halves and |those of a, b|, 16 bits from the top of re and im
__device__ __forceinline__ unsigned fx_size(unsigned m, long long u0, long long u1)
{
    const unsigned p = __byte_perm((unsigned)(u0 >> 32), (unsigned)(u1 >> 32), 0x7632);
    return __vimax3_s16x2(m, p, ~p);
}
// The sizes after the units grew by 2^by
__device__ __forceinline__ unsigned fx_size_shift(unsigned m, int by)
{
    const int k = min(by, 15);
    return (m >> k) & ((0x7fffu >> k) * 0x10001u);
}

__device__ __forceinline__ void fx_clear(FxSum& S)
{
#pragma unroll
    for (int k = 0; k < 24; ++k) S.s[k] = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r) S.m[0][r] = S.m[1][r] = 0;
    S.e = kFxMinExp;
    S.bad = false;
}

// (s[0], s[1]) += i^K (re, im)
template <int K>
__device__ __forceinline__ void fx_add_ik(long long* s, long long re, long long im)
{
    if constexpr (K == 0) {
        s[0] += re;
        s[1] += im;
    } else if constexpr (K == 1) {
        s[0] -= im;
        s[1] += re;
    } else if constexpr (K == 2) {
        s[0] -= re;
        s[1] -= im;
    } else {
        s[0] += im;
        s[1] -= re;
    }
}

// A projected half spinor as fixed point in the units of a site sum:
// reals (h0, h1) x colour x (re, im), n_x = xh 2^31 + xl
struct FxHalf {
    int xh[12], xl[12];
};

// Convert the half spinor (h0, h1), raising Q's exponent first if it exceeds it.
__device__ __forceinline__ void fx_convert(FxSum& Q, FxHalf& X, const cx<double> (&h0)[3], const cx<double> (&h1)[3])
{
    unsigned hw[12], lw[12];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double v[4] = {h0[c].re, h0[c].im, h1[c].re, h1[c].im};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int q = (k >> 1) * 6 + 2 * c + (k & 1);
            hw[q] = (unsigned)__double2hiint(v[k]);
            lw[q] = (unsigned)__double2loint(v[k]);
        }
    }
    // e minus each value's exponent is in bits 20.. of up[]; negative when one exceeds e
    int up[12], any = 0;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        up[q] = (int)((((unsigned)Q.e << 20) | 0xfffffu) - (hw[q] & 0x7fffffffu));
        any |= up[q];
    }
    if (any < 0) {
        unsigned top = 0;
#pragma unroll
        for (int q = 0; q < 12; ++q) top = max(top, hw[q] & 0x7fffffffu);
        int E = (int)(top >> 20) + (Q.e == kFxMinExp ? 1 : 0);
        if (E > kFxMaxExp) {
            Q.bad = true;
            E = kFxMaxExp;  // (the sums are not used any more)
        }
        const int by = min(E - Q.e, 62);
        if (by > 0) {
            const long long half = 1LL << (by - 1);
#pragma unroll
            for (int k = 0; k < 24; ++k) Q.s[k] = (Q.s[k] + half) >> by;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                Q.m[0][r] = fx_size_shift(Q.m[0][r], by);
                Q.m[1][r] = fx_size_shift(Q.m[1][r], by);
            }
        }
#pragma unroll
        for (int q = 0; q < 12; ++q) up[q] += (E - Q.e) << 20;
        Q.e = E;
    }
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        const unsigned mh = (hw[q] & 0xfffffu) | 0x100000u;
        // the 53-bit significand 7 bits up, then down by the exponent difference
        // (zeros and subnormals: by 63, to 0)
        unsigned long long y = ((unsigned long long)__funnelshift_l(lw[q], mh, 7) << 32) | (lw[q] << 7);
        y >>= min((unsigned)up[q] >> 20, 63u);
        const int sg = ((int)hw[q] >> 31) | 1;
        X.xh[q] = (int)(unsigned)(y >> 32) * sg;
        X.xl[q] = (int)((unsigned)y >> 1) * sg;
    }
}

// Add colour row r of one hop in direction mu to the site sum: link row w,
// converted half spinor X.  X holds S (h0, h1) for the projector 1 + S gamma_mu,
// so rows 2 and 3 take it as it is, and rows 0 and 1 are summed with the sign S
// (the sign of the present pass, see fx_sum).
__device__ __forceinline__ void fx_row(FxSum& Q, const FxHalf& X, const int4 (&w)[3], int r, int mu)
{
    long long R[4];  // u0.re, u0.im, u1.re, u1.im
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int* H = X.xh + 6 * j;
        const int* L = X.xl + 6 * j;
        long long A = fx_mul(w[0].x, H[0]), B = fx_mad(w[0].x, L[0], kFxHalfUnit);
        long long C = fx_mul(w[0].x, H[1]), D = fx_mad(w[0].x, L[1], kFxHalfUnit);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (k) {
                A = fx_mad(w[k].x, H[2 * k], A);
                B = fx_mad(w[k].x, L[2 * k], B);
                C = fx_mad(w[k].x, H[2 * k + 1], C);
                D = fx_mad(w[k].x, L[2 * k + 1], D);
            }
            A = fx_mad(-w[k].z, H[2 * k + 1], A);
            B = fx_mad(w[k].y, H[2 * k], B);
            B = fx_mad(-w[k].z, L[2 * k + 1], B);
            B = fx_mad(-w[k].w, H[2 * k + 1], B);
            C = fx_mad(w[k].z, H[2 * k], C);
            D = fx_mad(w[k].y, H[2 * k + 1], D);
            D = fx_mad(w[k].z, L[2 * k], D);
            D = fx_mad(w[k].w, H[2 * k], D);
        }
        R[2 * j] = A + (B >> 31);
        R[2 * j + 1] = C + (D >> 31);
    }
    long long *s0 = Q.s + 2 * r, *s1 = s0 + 6, *s2 = s1 + 6, *s3 = s2 + 6;
    fx_add_ik<0>(s0, R[0], R[1]);
    fx_add_ik<0>(s1, R[2], R[3]);
    if (mu & 2) Q.m[1][r] = fx_size(fx_size(Q.m[1][r], R[0], R[2]), R[1], R[3]);
    else Q.m[0][r] = fx_size(fx_size(Q.m[0][r], R[0], R[2]), R[1], R[3]);
    if (mu & 1) {
        if (mu & 2) {  // rows 2, 3 += (u0, u1)
            fx_add_ik<0>(s2, R[0], R[1]);
            fx_add_ik<0>(s3, R[2], R[3]);
        } else {  // (u1, -u0)
            fx_add_ik<0>(s2, R[2], R[3]);
            fx_add_ik<2>(s3, R[0], R[1]);
        }
    } else if (mu & 2) {  // (-i u0, i u1)
        fx_add_ik<3>(s2, R[0], R[1]);
        fx_add_ik<1>(s3, R[2], R[3]);
    } else {  // -i (u1, u0)
        fx_add_ik<3>(s2, R[2], R[3]);
        fx_add_ik<3>(s3, R[0], R[1]);
    }
}

__device__ __forceinline__ void fx_negate_upper(FxSum& Q)
{
#pragma unroll
    for (int k = 0; k < 12; ++k) Q.s[k] = -Q.s[k];
}

// S times the projected half spinor of (1 + S gamma_mu), S = sg = 1 or -1, from
// the neighbour spinor q (a fused multiply-add by +-1 is the addition or
// subtraction exactly).
__device__ __forceinline__ void fx_project(cx<double> (&h0)[3], cx<double> (&h1)[3], const cx<double> (&q)[12], int mu,
                                           double sg)
{
    // volatile: the compiler otherwise computes parts of several branches' sums
    auto add = [=](cx<double> p, cx<double> x) -> cx<double> {
        cx<double> r;
        asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r.re) : "d"(sg), "d"(p.re), "d"(x.re));
        asm volatile("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r.im) : "d"(sg), "d"(p.im), "d"(x.im));
        return r;
    };
    if (mu & 1) {
        if (mu & 2) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                h0[c] = add(q[c], q[6 + c]);
                h1[c] = add(q[3 + c], q[9 + c]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                h0[c] = add(q[c], -q[9 + c]);
                h1[c] = add(q[3 + c], q[6 + c]);
            }
        }
    } else if (mu & 2) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            h0[c] = add(q[c], mul_i(q[6 + c]));
            h1[c] = add(q[3 + c], -mul_i(q[9 + c]));
        }
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            h0[c] = add(q[c], mul_i(q[9 + c]));
            h1[c] = add(q[3 + c], mul_i(q[6 + c]));
        }
    }
}

// The k-th hop of the site sum: the four forward hops, then the four backward ones
__device__ __forceinline__ int fx_order(int k) { return 2 * (k & 3) + (k >> 2); }

// The site sum over the eight hops, a loop: the eight bodies side by side would
// overflow the instruction cache.  The projector's sign S costs nothing
// (fx_project, fx_row; rows 0 and 1 change sign between the passes), the
// direction a uniform branch where its spin structure enters.  src gives
// hop fx_order(k) its data:
//   half(k, mu, sg, h0, h1)  sg times the projected half spinor
//   link(k, r, w)            row r of the link
template <bool DAG, typename Src>
__device__ __forceinline__ void fx_sum(FxSum& Q, Src& src)
{
    fx_clear(Q);
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const int mu = k & 3;
        const double sg = (k < 4) != DAG ? -1.0 : 1.0;  // forward hops take S = -1; the adjoint flips both
        FxHalf X;
        {
            cx<double> h0[3], h1[3];
            src.half(k, mu, sg, h0, h1);
            fx_convert(Q, X, h0, h1);
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            int4 w[3];
            src.link(k, r, w);
            fx_row(Q, X, w, r, mu);
        }
        if (k == 3 || (DAG && k == 7)) fx_negate_upper(Q);  // (DAG: the last pass had S = -1)
    }
}

// s 2^(e-1023-55) rounded to nearest, ties to even, by integer operations
// (the hardware conversion runs on the FP64 pipe).  |s| < 2^62; the result is
// zero or normal: e - 55 > 0 and |s| 2^(e-1078) < 2^1024 for the exponents accepted.
__device__ __forceinline__ double fx_value(long long s, int e)
{
    const int m = (int)(s >> 63);
    unsigned long long q = (unsigned long long)((s ^ (long long)m) - m);
    const unsigned hi = (unsigned)(q >> 32);
    int up = __clz((int)hi) - 1;  // leading bit to 62
    if (hi == 0) {                // (below 2^-30 of the scale: rare)
        if (q == 0) return 0.0;
        up = 31 + __clz((int)(unsigned)q);
    }
    q <<= up;
    q += 0x1ffu + ((unsigned)(q >> 10) & 1u);
    q >>= 10;  // 53 bits (a carry to 2^53 runs into the exponent)
    // biased exponent of the leading bit: e - 1078 + (62 - up) + 1023, less one for the implicit bit in q
    return __hiloint2double((int)((unsigned)(q >> 32) + ((unsigned)(e + 6 - up) << 20) + ((unsigned)m << 31)), (int)(unsigned)q);
}

// The projected half spinor of hop d from the neighbour spinor q, spin
// structure from hop_code(): (h0, h1) as project<MU, S>() forms it.
template <typename T, bool DAG>
__device__ __forceinline__ void project_code(cx<T> (&h0)[3], cx<T> (&h1)[3], const cx<T> (&q)[12], int d)
{
    const unsigned code = hop_code(d >> 1);
    const int sflip = ((d & 1) ? DAG == false : DAG == true) ? 0 : 2;
    const int a0 = code & 1, k0 = ((code >> 1) + sflip) & 3;
    const int a1 = (code >> 3) & 1, k1 = ((code >> 4) + sflip) & 3;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h0[c] = q[c] + mul_ik(a0 ? q[9 + c] : q[6 + c], k0);
        h1[c] = q[3 + c] + mul_ik(a1 ? q[9 + c] : q[6 + c], k1);
    }
}

// The site sum in plain FP64 arithmetic (the operations of the LF = 0
// kernel), for components that are small next to the site's scale and for sites
// whose neighbours do not share a scale.  half(d, h0, h1)
// gives the projected half spinor of hop d.  A loop, and called rather than
// inlined: it is rare, and must not cost the fixed-point path registers.  Sets
// the components of out whose bit (spin * 3 + colour) is in `which`.
template <bool DAG, typename F>
__device__ __noinline__ void fx_site_general(double (&out)[24], unsigned which, const void* links, long long lVh, long long li, F half)
{
    cx<double> acc[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = {0.0, 0.0};
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
        cx<double> h0[3], h1[3];
        half(d, h0, h1);
        // the colour rows of u0 and u1 that enter components of `which`
        const unsigned two = which >> (d < 4 ? 9 : 6), three = which >> (d < 4 ? 6 : 9);
        unsigned n0 = (which | two) & 7u, n1 = (which >> 3 | three) & 7u;
        bool zero0 = true, zero1 = true;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            zero0 &= h0[c].re == 0.0 & h0[c].im == 0.0;
            zero1 &= h1[c].re == 0.0 & h1[c].im == 0.0;
        }
        if (zero0) n0 = 0;
        if (zero1) n1 = 0;
        const unsigned code = hop_code(d >> 1);
        const int sflip = ((d & 1) ? DAG == false : DAG == true) ? 0 : 2;
        const int b2 = (code >> 6) & 1, k2 = ((code >> 7) + sflip) & 3;
        const int b3 = (code >> 9) & 1, k3 = ((code >> 10) + sflip) & 3;
        const int4* p = (const int4*)links + (long long)d * 9 * lVh + li;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!((n0 | n1) >> a & 1)) continue;
            cx<double> w[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int4 t = p[(3 * a + k) * lVh];
                w[k] = {fx_join(t.x, t.y), fx_join(t.z, t.w)};
            }
            cx<double> u0 = {0.0, 0.0}, u1 = {0.0, 0.0};
            if (n0 >> a & 1) u0 = dot3(w[0], w[1], w[2], h0);
            if (n1 >> a & 1) u1 = dot3(w[0], w[1], w[2], h1);
            acc[a] = acc[a] + u0;
            acc[3 + a] = acc[3 + a] + u1;
            acc[6 + a] = acc[6 + a] + mul_ik(b2 ? u1 : u0, k2);
            acc[9 + a] = acc[9 + a] + mul_ik(b3 ? u1 : u0, k3);
        }
    }
#pragma unroll
    for (int c = 0; c < 12; ++c)
        if (which >> c & 1) {
            out[2 * c] = acc[c].re;
            out[2 * c + 1] = acc[c].im;
        }
}

// acc = the site sum as FP64 (spin rows 2 and 3 take u1, u0 of the x and y hops
// and u0, u1 of the z and t hops)
template <bool DAG, typename F>
__device__ __forceinline__ void fx_finish(cx<double> (&acc)[12], const FxSum& S, const void* links, long long lVh,
                                          long long li, F half)
{
    unsigned low = 0;  // components that need FP64
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const unsigned up = __vmaxs2(S.m[0][r], S.m[1][r]);
        const unsigned down = __vmaxs2(__byte_perm(S.m[0][r], 0, 0x1032), S.m[1][r]);
        low |= ((up & 0xffffu) < kFxLeast ? 1u : 0u) << r | (up < (unsigned)kFxLeast << 16 ? 8u : 0u) << r |
               ((down & 0xffffu) < kFxLeast ? 64u : 0u) << r | (down < (unsigned)kFxLeast << 16 ? 512u : 0u) << r;
    }
    if (S.bad || S.e == kFxMinExp) low = 0xfffu;  // (nothing above 2^-953: zeros, or too small for fixed point)
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = {fx_value(S.s[2 * c], S.e), fx_value(S.s[2 * c + 1], S.e)};
    if (low) {
        double g[24];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            g[2 * c] = acc[c].re;
            g[2 * c + 1] = acc[c].im;
        }
        fx_site_general<DAG>(g, low, links, lVh, li, half);
#pragma unroll
        for (int c = 0; c < 12; ++c) acc[c] = {g[2 * c], g[2 * c + 1]};
    }
}

// The plain-FP64 path's half spinor of hop d from the local neighbour at n
template <bool DAG>
__device__ __forceinline__ void fx_general_local(int d, cx<double> (&h0)[3], cx<double> (&h1)[3], const void* in, long long Vh,
                                                 int n)
{
    cx<double> q[12];
    load_spinor_ro<WL_F64>(q, in, Vh, n);
    project_code<double, DAG>(h0, h1, q, d);
}

// v[d] of an array held in registers
template <typename T>
__device__ __forceinline__ T fx_pick(const T (&v)[8], int d)
{
    T n = v[0];
#pragma unroll
    for (int k = 1; k < 8; ++k) n = d == k ? v[k] : n;
    return n;
}

// Plain loads: links at index li of planes of stride lVh.
struct FxDirect {
    const void* in;
    long long Vh;
    const int (&nb)[8];
    const void* links;
    long long lVh;
    long long li;

    __device__ __forceinline__ void half(int k, int mu, double sg, cx<double> (&h0)[3], cx<double> (&h1)[3])
    {
        cx<double> q[12];
        load_spinor_ro<WL_F64>(q, in, Vh, fx_pick(nb, fx_order(k)));
        fx_project(h0, h1, q, mu, sg);
    }
    __device__ __forceinline__ void link(int k, int r, int4 (&w)[3])
    {
        const int4* p = (const int4*)links + (fx_order(k) * 9 + 3 * r) * lVh + li;
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = p[c * lVh];
    }
};

// acc = H_{p,1-p} in at the output site whose neighbours are nb (hop_site for LF = 3)
template <bool DAG>
__device__ __forceinline__ void fx_site(cx<double> (&acc)[12], const int (&nb)[8], long long Vh, const void* in,
                                        const void* links, long long lVh, int li)
{
    FxSum S;
    FxDirect src{in, Vh, nb, links, lVh, li};
    fx_sum<DAG>(S, src);
    fx_finish<DAG>(acc, S, links, lVh, li, [=](int d, cx<double>(&h0)[3], cx<double>(&h1)[3]) {
        fx_general_local<DAG>(d, h0, h1, in, Vh, fx_pick(nb, d));
    });
}

// Staged loads: each thread copies the next hop's spinor and link into its own
// shared-memory slots with cp.async while it computes on the present one, so
// that no register waits for memory.  Slot q of a thread is
// slot[q * kStride]: 12 spinor planes, the 8 neighbour indices (two slots), then
// 9 link entries.  Two groups are in flight at a time: the next spinor and the
// next link.  A slot is refilled only after __syncwarp() has ordered the reads of it.
struct FxStaged {
    static constexpr int kSlots = 23;
    static constexpr int kNb = 12, kLink = 14;
    static constexpr int kStride = 32;  // slots of a warp: [kSlots][32]
    int4* slot;
    const char* in;
    long long Vh;
    const char* links;  // this site's entry of the first plane
    long long lVh;      // sites between planes

    __device__ __forceinline__ int neighbour(int d) const { return ((const int*)(slot + kNb * kStride))[d < 4 ? d : kStride * 4 - 4 + d]; }
    __device__ __forceinline__ void fetch_spinor(int d)
    {
        const char* p = in + (unsigned)neighbour(d) * 16u;  // (half indices are below 2^27)
        const unsigned a = (unsigned)__cvta_generic_to_shared(slot);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(a + c * (kStride * 16)), "l"(p) : "memory");
            p += Vh * 16;
        }
    }
    __device__ __forceinline__ void fetch_row(int d, int r)
    {
        const char* p = links + (long long)(d * 9 + 3 * r) * (lVh * 16);
        const unsigned a = (unsigned)__cvta_generic_to_shared(slot);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a + (kLink + 3 * r + k) * (kStride * 16)), "l"(p) : "memory");
            p += lVh * 16;
        }
    }
    __device__ __forceinline__ void start(const int (&nb)[8])
    {
        slot[kNb * kStride] = make_int4(nb[0], nb[1], nb[2], nb[3]);
        slot[(kNb + 1) * kStride] = make_int4(nb[4], nb[5], nb[6], nb[7]);
        fetch_spinor(0);
        cp_async_commit();
        fetch_row(0, 0);
        fetch_row(0, 1);
        fetch_row(0, 2);
        cp_async_commit();
    }
    __device__ __forceinline__ void half(int k, int mu, double sg, cx<double> (&h0)[3], cx<double> (&h1)[3])
    {
        cp_async_wait<1>();
        cx<double> q[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const double2 t = *(const double2*)(slot + c * kStride);
            q[c] = {t.x, t.y};
        }
        fx_project(h0, h1, q, mu, sg);
        __syncwarp();
        if (k < 7) fetch_spinor(fx_order(k + 1));
        cp_async_commit();
    }
    __device__ __forceinline__ void link(int k, int r, int4 (&w)[3])
    {
        if (r == 0) cp_async_wait<1>();
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = slot[(kLink + 3 * r + c) * kStride];
        __syncwarp();
        if (k < 7) fetch_row(fx_order(k + 1), r);
        if (r == 2) cp_async_commit();
    }
};

template <bool DAG>
__device__ __forceinline__ void fx_site_staged(cx<double> (&acc)[12], const int (&nb)[8], long long Vh, const char* in,
                                               const char* links, long long lVh, int li, int4* slot)
{
    FxSum S;
    FxStaged src{slot, in, Vh, links + (unsigned)li * 16u, lVh};
    src.start(nb);
    fx_sum<DAG>(S, src);
    cp_async_wait<0>();
    fx_finish<DAG>(acc, S, links, lVh, li, [=](int d, cx<double>(&h0)[3], cx<double>(&h1)[3]) {
        fx_general_local<DAG>(d, h0, h1, in, Vh, src.neighbour(d));
    });
}

// ---------------------------------------------------------------------------
// Small lattices, where a thread per site leaves the SMs with a warp or two and
// the time is one thread's dependent instructions: six threads per site, one
// for each of the rows j = 0, 1 of the half spinors and each colour row r.
// Lanes l and l + 16 of a warp hold j = 0 and 1 of the same site and colour row.
// The sums are fx_sum's, bit for bit: the two threads agree on e at every
// hop, and join their parts of spin rows 2 and 3 before they are shifted.
// ---------------------------------------------------------------------------

// Spin row j in s, this thread's parts of spin rows 3 - j and 2 + j in a and b (re, im)
struct FxPart {
    long long s[2], a[2], b[2];
    int m[2];  // as FxSum's, of this thread's product: x and y hops, z and t hops
    int e;
    bool bad;
};

__device__ __forceinline__ long long fx_partner(long long v) { return __shfl_xor_sync(0xffffffffu, v, 16); }

// fx_convert for one projected row (colour x (re, im)); whole warps call it
__device__ __forceinline__ void fx_convert_row(FxPart& Q, int (&xh)[6], int (&xl)[6], const cx<double> (&h)[3])
{
    unsigned hw[6], lw[6];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        hw[2 * c] = (unsigned)__double2hiint(h[c].re);
        lw[2 * c] = (unsigned)__double2loint(h[c].re);
        hw[2 * c + 1] = (unsigned)__double2hiint(h[c].im);
        lw[2 * c + 1] = (unsigned)__double2loint(h[c].im);
    }
    int up[6], any = 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        up[q] = (int)((((unsigned)Q.e << 20) | 0xfffffu) - (hw[q] & 0x7fffffffu));
        any |= up[q];
    }
    if (__any_sync(0xffffffffu, any < 0)) {
        unsigned top = 0;
#pragma unroll
        for (int q = 0; q < 6; ++q) top = max(top, hw[q] & 0x7fffffffu);
        top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
        int E = (int)(top >> 20);
        if (E > Q.e) {
            E += Q.e == kFxMinExp ? 1 : 0;
            if (E > kFxMaxExp) {
                Q.bad = true;
                E = kFxMaxExp;  // (the sums are not used any more)
            }
        } else {
            E = Q.e;  // another site's
        }
        const int by = min(E - Q.e, 62);
        Q.m[0] >>= min(by, 15);
        Q.m[1] >>= min(by, 15);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            Q.b[k] += fx_partner(Q.a[k]);
            Q.a[k] = 0;
            if (by > 0) {
                const long long half = 1LL << (by - 1);
                Q.s[k] = (Q.s[k] + half) >> by;
                Q.b[k] = (Q.b[k] + half) >> by;
            }
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) up[q] += (E - Q.e) << 20;
        Q.e = E;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const unsigned mh = (hw[q] & 0xfffffu) | 0x100000u;
        unsigned long long y = ((unsigned long long)__funnelshift_l(lw[q], mh, 7) << 32) | (lw[q] << 7);
        y >>= min((unsigned)up[q] >> 20, 63u);
        const int sg = ((int)hw[q] >> 31) | 1;
        xh[q] = (int)(unsigned)(y >> 32) * sg;
        xl[q] = (int)((unsigned)y >> 1) * sg;
    }
}

// The sign that hop direction MU and row j give the neighbour's spin rows 2 and
// 3 next to the projector's S: -1 for (y, 0) and (z, 1)
template <int MU>
__device__ __forceinline__ int fx_minus(int j)
{
    return MU == 1 ? j - 1 : MU == 2 ? -j : 0;
}

// One hop of direction MU: own spin row p of the neighbour, its row q = 3 - j
// (MU = x, y) or 2 + j (z, t), row w of the link; sg as in fx_project.  The
// projected row is S p + c q, c = i (x, z) or 1 (y, t) with the sign m; its
// product enters spin row j, and spin row 3 - j or 2 + j with -i or 1 and m.
template <int MU>
__device__ __forceinline__ void fx_hop_row(FxPart& Q, const cx<double> (&p)[3], const cx<double> (&q)[3], const int4 (&w)[3],
                                           int j, double sg)
{
    const int m = fx_minus<MU>(j);
    auto flip = [=](double v) {  // v, or -v for m = -1
        return __hiloint2double((int)((unsigned)__double2hiint(v) ^ ((unsigned)m & 0x80000000u)), __double2loint(v));
    };
    cx<double> h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cx<double> t = q[c];
        if constexpr (MU == 1 || MU == 2) t = {flip(t.re), flip(t.im)};
        if constexpr (MU == 0 || MU == 2) t = mul_i(t);
        h[c] = {fma(sg, p[c].re, t.re), fma(sg, p[c].im, t.im)};
    }
    int H[6], L[6];
    fx_convert_row(Q, H, L, h);
    long long A = 0, B = kFxHalfUnit, C = 0, D = kFxHalfUnit;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        A = fx_mad(w[k].x, H[2 * k], A);
        A = fx_mad(-w[k].z, H[2 * k + 1], A);
        B = fx_mad(w[k].x, L[2 * k], B);
        B = fx_mad(w[k].y, H[2 * k], B);
        B = fx_mad(-w[k].z, L[2 * k + 1], B);
        B = fx_mad(-w[k].w, H[2 * k + 1], B);
        C = fx_mad(w[k].x, H[2 * k + 1], C);
        C = fx_mad(w[k].z, H[2 * k], C);
        D = fx_mad(w[k].x, L[2 * k + 1], D);
        D = fx_mad(w[k].y, H[2 * k + 1], D);
        D = fx_mad(w[k].z, L[2 * k], D);
        D = fx_mad(w[k].w, H[2 * k], D);
    }
    const long long re = A + (B >> 31), im = C + (D >> 31);
    const int tr = (int)(re >> 48), ti = (int)(im >> 48);
    int& size = Q.m[MU >> 1];
    size = max(max(size, max(tr, ~tr)), max(ti, ~ti));
    Q.s[0] += re;
    Q.s[1] += im;
    const long long mm = m;
    if constexpr (MU == 0) {
        Q.a[0] += im;
        Q.a[1] -= re;
    } else if constexpr (MU == 1) {
        Q.a[0] += (re ^ mm) - mm;
        Q.a[1] += (im ^ mm) - mm;
    } else if constexpr (MU == 2) {
        Q.b[0] += (im ^ mm) - mm;
        Q.b[1] -= (re ^ mm) - mm;
    } else {
        Q.b[0] += re;
        Q.b[1] += im;
    }
}

// Colour row a of spin rows j (up) and 2 + j (down) of the site sum at li, j =
// lane >> 4.  Every load of a hop is issued a hop ahead into registers.  Whole
// warps call it.
template <bool DAG>
__device__ __forceinline__ void fx_site_row(cx<double>& up, cx<double>& down, const int (&nb)[8], long long Vh, const void* in,
                                            const void* links, long long li, int a, int lane)
{
    const int j = lane >> 4;
    FxPart Q;
    Q.s[0] = Q.s[1] = Q.a[0] = Q.a[1] = Q.b[0] = Q.b[1] = 0;
    Q.m[0] = Q.m[1] = 0;
    Q.e = kFxMinExp;
    Q.bad = false;
    const double2* f = (const double2*)in + 3 * j * Vh;
    const int4* l = (const int4*)links + 3 * a * Vh + li;
    cx<double> p[3], q[3];
    int4 w[3];
    auto load = [&](int d, int n) {  // neighbour n through link d
        const long long g = (d < 4 ? 9 - 6 * j : 6) * Vh;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 u = __ldg(f + c * Vh + n), v = __ldg(f + g + c * Vh + n);
            p[c] = {u.x, u.y};
            q[c] = {v.x, v.y};
            w[c] = l[(d * 9 + c) * Vh];
        }
    };
    load(0, nb[0]);
#pragma unroll 1
    for (int fb = 0; fb < 2; ++fb) {
        const double sg = (fb == 0) != DAG ? -1.0 : 1.0;
        auto hop = [&](auto mu) {
            constexpr int MU = decltype(mu)::value;
            cx<double> p0[3], q0[3];
            int4 w0[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                p0[c] = p[c];
                q0[c] = q[c];
                w0[c] = w[c];
            }
            if constexpr (MU < 3) load(2 * MU + 2 + fb, fb ? nb[2 * MU + 3] : nb[2 * MU + 2]);
            else if (fb == 0) load(1, nb[1]);
            fx_hop_row<MU>(Q, p0, q0, w0, j, sg);
        };
        hop(std::integral_constant<int, 0>());
        hop(std::integral_constant<int, 1>());
        hop(std::integral_constant<int, 2>());
        hop(std::integral_constant<int, 3>());
        if (fb == 0 || DAG) {
            Q.s[0] = -Q.s[0];
            Q.s[1] = -Q.s[1];
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) Q.b[k] += fx_partner(Q.a[k]);
    const int other = __shfl_xor_sync(0xffffffffu, Q.m[0], 16);  // the x and y hops' share of spin row 2 + j
    const unsigned above = max(Q.m[0], Q.m[1]) < kFxLeast ? 1u : 0u, below = max(other, Q.m[1]) < kFxLeast ? 64u : 0u;
    const int c = 3 * j + a;
    unsigned low = (above | below) << c;
    if (Q.bad || Q.e == kFxMinExp) low = 65u << c;
    up = {fx_value(Q.s[0], Q.e), fx_value(Q.s[1], Q.e)};
    down = {fx_value(Q.b[0], Q.e), fx_value(Q.b[1], Q.e)};
    if (low) {
        double g[24];
        fx_site_general<DAG>(g, low, links, Vh, li, [=](int d, cx<double>(&h0)[3], cx<double>(&h1)[3]) {
            fx_general_local<DAG>(d, h0, h1, in, Vh, fx_pick(nb, d));
        });
        if (low >> c & 1) up = {g[2 * c], g[2 * c + 1]};
        if (low >> c & 64) down = {g[2 * c + 12], g[2 * c + 13]};
    }
}

}  // namespace wl
