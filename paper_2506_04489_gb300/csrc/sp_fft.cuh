// Register-resident mixed-radix FFT engine used by the solve passes.
//
// A length-N line is transformed by T = N/E threads that each hold E complex values in
// registers.  Stage s (radix R_s, span P_s = R_0 ... R_{s-1}) is the Stockham step
//     for i < N/R, k = i mod P:   u_r = x[i + r N/R] * w^{r k N/(P R)},  u = DFT_R(u),
//                                 y[(i - k) R + k + q P] = u_q,
// with thread t owning the butterflies i = t + T m, m < E/R.  Between stages the
// values go through shared memory once (write, barrier, read).  After the last stage
// thread t holds y[t + T m + q N/R_last]; the inverse transform runs the radices in
// reverse order, so its first stage wants exactly those values: a diagonal multiplier
// between a forward and an inverse transform is applied in registers with no exchange.
// A forward transform whose upper half of inputs is zero (zero padding) has, in its
// first radix-R stage, exactly inputs r < R/2 nonzero in every butterfly; an inverse
// whose upper half of outputs is discarded (crop) needs only outputs q < R/2 of its
// last stage.  Both are pruned at compile time.
#pragma once

#include <type_traits>

#include "sp_common.cuh"
#include "sp_df32.cuh"

// ------------------------------------------------------------------ numeric traits
// (Num<float>, Num<double>: sp_common.cuh)
template <> struct Num<df32> {
    static SP_HD df32 c(double d) { return df_from_double(d); }
};
template <class R> SP_D cpx<R> czero() { return mk(Num<R>::c(0.0), Num<R>::c(0.0)); }

// Twiddle products: the generic forms for float/double; for double-float each part is
// one fused two-product dot (df_dot_sub / df_dot_add).
template <class R> SP_D cpx<R> tw_mul(cpx<R> a, cpx<R> w) { return cmul(a, w); }
template <class R> SP_D cpx<R> tw_mulc(cpx<R> a, cpx<R> w) { return cmulc(a, w); }
template <> SP_D cpx<df32> tw_mul<df32>(cpx<df32> a, cpx<df32> w)
{
    const df32 ar = re_of(a), ai = im_of(a), wr = re_of(w), wi = im_of(w);
    return mk(df_dot_sub(ar, wr, ai, wi), df_dot_add(ar, wi, ai, wr));
}
template <> SP_D cpx<df32> tw_mulc<df32>(cpx<df32> a, cpx<df32> w)
{
    const df32 ar = re_of(a), ai = im_of(a), wr = re_of(w), wi = im_of(w);
    return mk(df_dot_add(ar, wr, ai, wi), df_dot_sub(ai, wr, ar, wi));
}
// a times an exact power of two; a s + b t with real s, t; -a
template <class R> SP_D cpx<R> scale_exact(cpx<R> a, float p) { return scale(a, (R)p); }
template <> SP_D cpx<df32> scale_exact<df32>(cpx<df32> a, float p)
{
    a.rh = __fmul_rn(a.rh, p);
    a.ih = __fmul_rn(a.ih, p);
    a.rl = __fmul_rn(a.rl, p);
    a.il = __fmul_rn(a.il, p);
    return a;
}
template <class R> SP_D cpx<R> dot2(cpx<R> a, R s, cpx<R> b, R t)
{
    return mk(a.re * s + b.re * t, a.im * s + b.im * t);
}
template <> SP_D cpx<df32> dot2<df32>(cpx<df32> a, df32 s, cpx<df32> b, df32 t)
{
    return mk(df_dot_add(re_of(a), s, re_of(b), t), df_dot_add(im_of(a), s, im_of(b), t));
}
template <class R> SP_D cpx<R> neg(cpx<R> a) { return mk(-re_of(a), -im_of(a)); }
// Values written to global memory are renormalised.  Exchanges through shared memory
// between the stages of one transform keep the pair as the arithmetic left it: sums and
// products accept a low part of a few ulps of the high part (their error stays a small
// multiple of 2^-48 of the operands), so renormalising there would only cost FP32 work.
template <class R> SP_D cpx<R> norm(cpx<R> a) { return a; }
template <> SP_D cpx<df32> norm<df32>(cpx<df32> a) { return df_norm_c(a); }

// ------------------------------------------------------------------ plans
template <int... Rs> struct Radices {
    static constexpr int NS = sizeof...(Rs);
    static constexpr int R[sizeof...(Rs)] = {Rs...};
};
// E values a thread, forward radices in order
template <int E_, int... Rs> struct PlanE : Radices<Rs...> {
    static constexpr int E = E_;
};
// Forward radices: powers of two first (the first stage is radix 8 or 16, so zero padding
// prunes it uniformly), then 3s.  E is a multiple of every radix.
template <int N> struct FFTPlan;
template <> struct FFTPlan<64> { static constexpr int NS = 2, E = 8; static constexpr int R[2] = {8, 8}; };
template <> struct FFTPlan<128> : PlanE<8, 8, 4, 4> {};
template <> struct FFTPlan<192> : PlanE<12, 12, 4, 4> {};
template <> struct FFTPlan<256> { static constexpr int NS = 3, E = 8; static constexpr int R[3] = {8, 8, 4}; };
template <> struct FFTPlan<384> : PlanE<12, 12, 4, 4, 2> {};
template <> struct FFTPlan<512> { static constexpr int NS = 3, E = 8; static constexpr int R[3] = {8, 8, 8}; };
template <> struct FFTPlan<1024> { static constexpr int NS = 4, E = 8; static constexpr int R[4] = {8, 8, 8, 2}; };

// The plan a pass of arithmetic type R uses.  At 1024, FP32 and FP64 take a radix-16
// first stage (16 values a thread, three stages: one exchange fewer, 15 % faster at
// 512^3 in FP32); double-float keeps eight values a thread, whose 16-value form holds
// too many registers (measured 6 % slower).
struct Plan1024Radix16 {
    static constexpr int NS = 3, E = 16;
    static constexpr int R[3] = {16, 8, 8};
};
// Lengths with a factor 3 run 12-point first stages on 12 values a thread (x passes, ps a
// point: at 192 12-4-4 against 8-8-3 on 24 values, double-float 15.4 against 21.2, FP64 77
// against 87, FP32 4.7 against 5.1; at 384 12-4-4-2 against 4-4-4-2-3, double-float 19.9
// against 23.8); FP32 takes 8-8-6 on 24 values at 384.  At 128 8-4-4 (11.4 against 11.9 for
// 8-8-2); FP32 16-8.
struct Plan384Radix6 : PlanE<24, 8, 8, 6> {};
struct Plan128Radix16 : PlanE<16, 16, 8> {};
// At 256, FP32 takes two radix-16 stages (16 values a thread, one exchange instead of
// two: 128^3 FP32 solve 12 % faster); the 16-byte types keep 8-8-4.
struct Plan256Radix16 {
    static constexpr int NS = 2, E = 16;
    static constexpr int R[2] = {16, 16};
};
// At 512, FP32 takes radices 32-16 (32 values a thread, one exchange instead of two:
// the x pass 19 % faster, the z passes slower, the 256^3 solve 9 % faster).
struct Plan512Radix32 {
    static constexpr int NS = 2, E = 32;
    static constexpr int R[2] = {32, 16};
};
template <class R, int N> struct PlanOf : FFTPlan<N> {};
template <> struct PlanOf<float, 512> : Plan512Radix32 {};
template <> struct PlanOf<float, 256> : Plan256Radix16 {};
// FP32 line passes at 1024: radices 32-32 (two stages; 3 % faster at 512^3 than 16-8-8,
// which its z passes keep).
struct Plan1024Radix32 {
    static constexpr int NS = 2, E = 32;
    static constexpr int R[2] = {32, 32};
};
template <> struct PlanOf<float, 1024> : Plan1024Radix32 {};
template <> struct PlanOf<double, 1024> : Plan1024Radix16 {};
template <> struct PlanOf<float, 384> : Plan384Radix6 {};
template <> struct PlanOf<float, 128> : Plan128Radix16 {};
// Lengths of the passes on grids whose own padded length has no plan above (sp_embed.cuh).
// First radices of 4, 6, 8, 10, 12, 16 or 20 points, so that the zero half is pruned; the
// radices 6 to 20 are prime-factor products without inner twiddles.  Plans were chosen by
// timing the x pass of an n^3 grid with every order of such radices, E values a thread and
// register caps: 16-byte values want 8 to 12 values a thread (double-float at 200: 82 us
// with 10-10-2 and E = 10, 104 us with 20-10 and E = 20), FP32 wants fewer stages (at 400:
// 20-20 and E = 20, 4.6 ps a point, against 5.8 with 10-10-4).
// Lengths 5 x 2^k and 400 would need 20 values a thread, or a fourth stage, for their factors 5
// to divide E.  Their middle stage instead gives some threads a butterfly fewer (one in five
// idles for a third of the transform), on 8 or 10 values: whole solves, us, double-float 77^3
// (F = 160) 101 / 85, 150^3 (320) 636 / 521, 200^3 (400) 1458 / 1220, 300^3 (640) 7050 / 4447;
// FP64 200^3 6663 / 6210, 310^3 26390 / 24780, but 150^3 2787 / 2909 and 77^3 383 / 401 (its pipe
// is full either way: FP64 keeps the 20-point plans at 160 and 320); FP32 77^3 40 / 36, 300^3
// 1617 / 1281, and at 320 and 400 the z passes only (155^3 22/29 / 21/20, x 72 / 91).
template <> struct FFTPlan<16> : PlanE<4, 4, 4> {};
template <> struct FFTPlan<32> : PlanE<8, 8, 4> {};
template <> struct FFTPlan<48> : PlanE<12, 12, 4> {};
template <> struct FFTPlan<72> : PlanE<12, 12, 6> {};
template <> struct FFTPlan<80> : PlanE<20, 20, 4> {};
template <> struct FFTPlan<96> : PlanE<12, 6, 4, 4> {};
template <> struct FFTPlan<144> : PlanE<12, 12, 12> {};
template <> struct FFTPlan<160> : PlanE<8, 8, 5, 4> {};
template <> struct FFTPlan<200> : PlanE<10, 10, 10, 2> {};
template <> struct FFTPlan<216> : PlanE<6, 6, 6, 6> {};
template <> struct FFTPlan<288> : PlanE<12, 12, 6, 4> {};
template <> struct FFTPlan<320> : PlanE<8, 8, 5, 8> {};
template <> struct FFTPlan<400> : PlanE<10, 10, 4, 10> {};
template <> struct FFTPlan<432> : PlanE<12, 12, 6, 6> {};
template <> struct FFTPlan<576> : PlanE<12, 12, 12, 4> {};
template <> struct FFTPlan<640> : PlanE<8, 8, 10, 8> {};
template <> struct FFTPlan<768> : PlanE<12, 4, 4, 4, 12> {};
template <> struct FFTPlan<864> : PlanE<12, 12, 12, 6> {};
template <> struct FFTPlan<1280> : PlanE<20, 20, 4, 4, 4> {};
template <> struct FFTPlan<1536> : PlanE<12, 12, 4, 4, 4, 2> {};
template <> struct FFTPlan<2048> : PlanE<16, 16, 16, 8> {};
template <> struct PlanOf<float, 96> : PlanE<24, 12, 8> {};
template <> struct PlanOf<float, 200> : PlanE<20, 20, 10> {};
template <> struct PlanOf<float, 400> : PlanE<20, 20, 20> {};
template <> struct PlanOf<float, 320> : PlanE<20, 20, 4, 4> {};
template <> struct PlanOf<double, 160> : PlanE<20, 20, 4, 2> {};
template <> struct PlanOf<double, 320> : PlanE<20, 20, 4, 4> {};
template <> struct PlanOf<float, 768> : PlanE<24, 8, 8, 12> {};

// Plan key of the z passes (contiguous real lines, packed in pairs): the type's own plan,
// except FP32 at 512 and 1024, whose z passes run faster on 8-8-8 and 16-8-8 than on the
// radix-32 plans of its line passes, and at 320 and 400 (above).  Each axis has its own staged
// twiddle table, so the z axis can differ.
template <class R> struct ZKey {};
template <class R, int N> struct PlanOf<ZKey<R>, N> : PlanOf<R, N> {};
template <> struct PlanOf<ZKey<float>, 512> : FFTPlan<512> {};
template <> struct PlanOf<ZKey<float>, 320> : FFTPlan<320> {};
template <> struct PlanOf<ZKey<float>, 400> : FFTPlan<400> {};
template <> struct PlanOf<ZKey<float>, 1024> : Plan1024Radix16 {};

// Alternative radix plans of the line passes, which the autotuner times against the
// built-in plan of the same type and length (LineKey<R, 1>; LineKey<R, 0> is the built-in
// plan PlanOf<R, N>).  Each has its own staged twiddle table in global memory, after the
// built-in plan's.
template <class R, int N> struct AltPlan {
    static constexpr bool exists = false;
};
// FP32: the eight-value plans (two exchanges a transform instead of one, about a third of
// the registers, so twice the resident warps)
template <> struct AltPlan<float, 256> : FFTPlan<256> { static constexpr bool exists = true; };
template <> struct AltPlan<float, 512> : FFTPlan<512> { static constexpr bool exists = true; };
template <> struct AltPlan<float, 1024> : Plan1024Radix16 { static constexpr bool exists = true; };
// double-float: sixteen values a thread at 256 (one exchange a transform instead of two)
template <> struct AltPlan<df32, 256> : Plan256Radix16 { static constexpr bool exists = true; };
template <class R, int V> struct LineKey {};
template <class R, int N> struct PlanOf<LineKey<R, 0>, N> : PlanOf<R, N> {};
template <class R, int N> struct PlanOf<LineKey<R, 1>, N> : AltPlan<R, N> {};
template <class K> struct KeyVariant { static constexpr int v = 0; };
template <class R, int V> struct KeyVariant<LineKey<R, V>> { static constexpr int v = V; };
// radix of stage s of the forward (INV = false) or inverse (reversed) transform
template <class R, int N, bool INV> constexpr int radix_at(int s)
{
    return INV ? PlanOf<R, N>::R[PlanOf<R, N>::NS - 1 - s] : PlanOf<R, N>::R[s];
}
template <class R, int N, bool INV> constexpr int span_at(int s)
{
    int p = 1;
    for (int i = 0; i < s; ++i) p *= radix_at<R, N, INV>(i);
    return p;
}

// ------------------------------------------------------------------ butterflies
// X_q = sum_r u_r exp(S 2 pi i r q / R), in place.
template <int S, class R> SP_D void bf2(cpx<R>* u)
{
    cpx<R> a = u[0], b = u[1];
    u[0] = a + b;
    u[1] = a - b;
}

template <int S, class R> SP_D void bf3(cpx<R>* u)
{
    const R c = Num<R>::c(-0.5);
    const R s = Num<R>::c(0.86602540378443864676372317075293618);  // sin(2 pi / 3)
    cpx<R> a = u[0], t = u[1] + u[2], v = u[1] - u[2];
    cpx<R> m = a + scale(t, c);
    cpx<R> w = mul_si<S>(scale(v, s));
    u[0] = a + t;
    u[1] = m + w;
    u[2] = m - w;
}

template <int S, class R> SP_D void bf4(cpx<R>* u)
{
    cpx<R> a = u[0] + u[2], b = u[0] - u[2];
    cpx<R> c = u[1] + u[3], d = mul_si<S>(u[1] - u[3]);
    u[0] = a + c;
    u[2] = a - c;
    u[1] = b + d;
    u[3] = b - d;
}

// radix 8 as 2 x 4 (even/odd halves, then twiddles exp(S 2 pi i q / 8))
template <int S, class R> SP_D void bf8_tail(cpx<R>* u, cpx<R> e0, cpx<R> e1, cpx<R> e2, cpx<R> e3, cpx<R> o0,
                                             cpx<R> o1, cpx<R> o2, cpx<R> o3)
{
    const R h = Num<R>::c(0.70710678118654752440084436210484904);
    cpx<R> t1 = scale(o1 + mul_si<S>(o1), h);
    cpx<R> t2 = mul_si<S>(o2);
    cpx<R> t3 = scale(mul_si<S>(o3) - o3, h);
    u[0] = e0 + o0;
    u[4] = e0 - o0;
    u[1] = e1 + t1;
    u[5] = e1 - t1;
    u[2] = e2 + t2;
    u[6] = e2 - t2;
    u[3] = e3 + t3;
    u[7] = e3 - t3;
}

template <int S, class R> SP_D void bf8(cpx<R>* u)
{
    cpx<R> a0 = u[0] + u[4], a1 = u[0] - u[4], a2 = u[2] + u[6], a3 = mul_si<S>(u[2] - u[6]);
    cpx<R> b0 = u[1] + u[5], b1 = u[1] - u[5], b2 = u[3] + u[7], b3 = mul_si<S>(u[3] - u[7]);
    bf8_tail<S>(u, a0 + a2, a1 + a3, a0 - a2, a1 - a3, b0 + b2, b1 + b3, b0 - b2, b1 - b3);
}

// radix 8 with u[4..7] = 0
template <int S, class R> SP_D void bf8_half(cpx<R>* u)
{
    cpx<R> a0 = u[0], a2 = u[2], a3 = mul_si<S>(u[2]);
    cpx<R> b0 = u[1], b2 = u[3], b3 = mul_si<S>(u[3]);
    bf8_tail<S>(u, a0 + a2, a0 + a3, a0 - a2, a0 - a3, b0 + b2, b0 + b3, b0 - b2, b0 - b3);
}

// radix 16 as 2 x 8: the DFTs of the even and odd halves, then
// X_q = E_q + w^q O_q, X_{q+8} = E_q - w^q O_q with w = exp(S 2 pi i / 16).
template <int S, class R> SP_D void bf16_tail(cpx<R>* u, cpx<R>* e, cpx<R>* o)
{
    const R h = Num<R>::c(0.70710678118654752440084436210484904);   // cos(pi/4)
    const R c1 = Num<R>::c(0.92387953251128675612818318939678829);  // cos(pi/8)
    const R s1 = Num<R>::c(0.38268343236508977172845998403039887);  // sin(pi/8)
    cpx<R> t[8];
    t[0] = o[0];
    t[1] = tw_mul(o[1], mk(c1, S > 0 ? s1 : -s1));
    t[2] = scale(o[2] + mul_si<S>(o[2]), h);
    t[3] = tw_mul(o[3], mk(s1, S > 0 ? c1 : -c1));
    t[4] = mul_si<S>(o[4]);
    t[5] = tw_mul(o[5], mk(-s1, S > 0 ? c1 : -c1));
    t[6] = scale(mul_si<S>(o[6]) - o[6], h);
    t[7] = tw_mul(o[7], mk(-c1, S > 0 ? s1 : -s1));
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        u[q] = e[q] + t[q];
        u[q + 8] = e[q] - t[q];
    }
}

template <int S, class R> SP_D void bf16(cpx<R>* u)
{
    cpx<R> e[8], o[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        e[j] = u[2 * j];
        o[j] = u[2 * j + 1];
    }
    bf8<S>(e);
    bf8<S>(o);
    bf16_tail<S>(u, e, o);
}

// radix 16 with u[8..15] = 0: both halves have their upper four inputs zero
template <int S, class R> SP_D void bf16_half(cpx<R>* u)
{
    cpx<R> e[8], o[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        e[j] = u[2 * j];
        o[j] = u[2 * j + 1];
    }
    bf8_half<S>(e);
    bf8_half<S>(o);
    bf16_tail<S>(u, e, o);
}

// radix 32 as 2 x 16: X_q = E_q + w^q O_q, X_{q+16} = E_q - w^q O_q, w = exp(S 2 pi i / 32).
template <int S, class R> SP_D void bf32_tail(cpx<R>* u, cpx<R>* e, cpx<R>* o)
{
    // cos and sin of pi m / 16, m = 0..8
    constexpr double C[9] = {1.0, 0.980785280403230449126182236134239037, 0.923879532511286756128183189396788287,
                             0.831469612302545237078788377617905757, 0.707106781186547524400844362104849039,
                             0.555570233019602224742830813948532874, 0.382683432365089771728459984030398867,
                             0.195090322016128267848284868477022241, 0.0};
    constexpr double Sn[9] = {0.0, 0.195090322016128267848284868477022241, 0.382683432365089771728459984030398867,
                              0.555570233019602224742830813948532874, 0.707106781186547524400844362104849039,
                              0.831469612302545237078788377617905757, 0.923879532511286756128183189396788287,
                              0.980785280403230449126182236134239037, 1.0};
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        cpx<R> t;
        if (q == 0) {
            t = o[0];
        } else if (q == 8) {
            t = mul_si<S>(o[8]);
        } else {
            const double c = q < 8 ? C[q] : -C[16 - q];
            const double sn = q < 8 ? Sn[q] : Sn[16 - q];
            t = tw_mul(o[q], mk(Num<R>::c(c), Num<R>::c(S > 0 ? sn : -sn)));
        }
        u[q] = e[q] + t;
        u[q + 16] = e[q] - t;
    }
}

template <int S, class R> SP_D void bf32(cpx<R>* u)
{
    cpx<R> e[16], o[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        e[j] = u[2 * j];
        o[j] = u[2 * j + 1];
    }
    bf16<S>(e);
    bf16<S>(o);
    bf32_tail<S>(u, e, o);
}

// radix 32 with u[16..31] = 0
template <int S, class R> SP_D void bf32_half(cpx<R>* u)
{
    cpx<R> e[16], o[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        e[j] = u[2 * j];
        o[j] = u[2 * j + 1];
    }
    bf16_half<S>(e);
    bf16_half<S>(o);
    bf32_tail<S>(u, e, o);
}

// radix 4 with u[2] = u[3] = 0
template <int S, class R> SP_D void bf4_half(cpx<R>* u)
{
    const cpx<R> a = u[0], b = u[1], d = mul_si<S>(u[1]);
    u[0] = a + b;
    u[1] = a + d;
    u[2] = a - b;
    u[3] = a - d;
}

// radix 5: with t1 = u1 + u4, t2 = u2 + u3, v1 = u1 - u4, v2 = u2 - u3 and s = t1 + t2,
// the cosine sums are (u0 - s/4) +- (t1 - t2) sqrt(5)/4 (cos(2 pi/5) + cos(4 pi/5) = -1/2,
// their difference sqrt(5)/2): one real product instead of four.
template <int S, class R> SP_D void bf5(cpx<R>* u)
{
    const R s5 = Num<R>::c(0.559016994374947424102293417182819059);  // sqrt(5)/4
    const R s1 = Num<R>::c(0.951056516295153572116439333379382143);  // sin(2 pi/5)
    const R s2 = Num<R>::c(0.587785252292473129168705954639072769);  // sin(4 pi/5)
    const cpx<R> t1 = u[1] + u[4], t2 = u[2] + u[3], v1 = u[1] - u[4], v2 = u[2] - u[3];
    const cpx<R> s = t1 + t2, d = scale(t1 - t2, s5);
    const cpx<R> m = u[0] - scale_exact(s, 0.25f);
    const cpx<R> a1 = m + d, a2 = m - d;
    const cpx<R> b1 = mul_si<S>(dot2(v1, s1, v2, s2)), b2 = mul_si<S>(dot2(v1, s2, v2, -s1));
    u[0] = u[0] + s;
    u[1] = a1 + b1;
    u[4] = a1 - b1;
    u[2] = a2 + b2;
    u[3] = a2 - b2;
}

// a times (S i)^m, m mod 4 known at compile time
template <int S, int M, class R> SP_D cpx<R> rot4(cpx<R> a)
{
    if constexpr ((M & 3) == 0) return a;
    else if constexpr ((M & 3) == 1) return mul_si<S>(a);
    else if constexpr ((M & 3) == 2) return neg(a);
    else return mul_si<-S>(a);
}

// DFT of length A = 2 or 4 of which only the half of the inputs starting at cyclic
// position P is nonzero: w[P] (A = 2), w[P] and w[P + 1 mod 4] (A = 4).
template <int S, int A, int P, class R> SP_D void bf_half_at(cpx<R>* w)
{
    if constexpr (A == 2) {
        const cpx<R> a = w[P];
        w[0] = a;
        w[1] = P ? neg(a) : a;
    } else {
        // sum over d = 0, 1 of w[P + d] (S i)^{(P + d) k}
        const cpx<R> a = w[P], b = w[(P + 1) & 3], d = mul_si<S>(b);
        w[0] = a + b;
        w[1] = rot4<S, P>(a + d);
        w[2] = rot4<S, 2 * P>(a - b);
        w[3] = rot4<S, 3 * P>(a - d);
    }
}

// Radix A B with A and B coprime (A = 2 or 4, B = 3 or 5) by the prime-factor map: input
// j = B j1 + A j2 mod A B, output q = B (B^-1 mod A) k1 + A (A^-1 mod B) k2 mod A B, B
// transforms of length A and A of length B with no twiddles between them.  With the upper
// half of the inputs zero (HALF) each length-A transform has A/2 cyclically adjacent
// nonzero inputs.
template <int A, int B> struct Pfa {
    static constexpr int N = A * B;
    static constexpr int inv(int a, int m)
    {
        for (int x = 1; x < m; ++x)
            if (a * x % m == 1) return x;
        return 1;
    }
    static constexpr int in(int j1, int j2) { return (B * j1 + A * j2) % N; }
    static constexpr int out(int k1, int k2) { return (B * inv(B % A, A) * k1 + A * inv(A % B, B) * k2) % N; }
    // first of the cyclically adjacent j1 whose input lies in the lower half
    static constexpr int first(int j2)
    {
        for (int j1 = 0; j1 < A; ++j1)
            if (in(j1, j2) < N / 2 && (A == 2 || in((j1 + A - 1) % A, j2) >= N / 2)) return j1;
        return 0;
    }
};
template <int S, int A, int B, bool HALF, int J2 = 0, class R> SP_D void pfa_rows(cpx<R>* u, cpx<R> (*w)[A])
{
    if constexpr (J2 < B) {
        using F = Pfa<A, B>;
#pragma unroll
        for (int j1 = 0; j1 < A; ++j1) w[J2][j1] = u[F::in(j1, J2)];
        if constexpr (HALF) bf_half_at<S, A, F::first(J2)>(w[J2]);
        else if constexpr (A == 4) bf4<S>(w[J2]);
        else bf2<S>(w[J2]);
        pfa_rows<S, A, B, HALF, J2 + 1>(u, w);
    }
}
template <int S, int A, int B, bool HALF, class R> SP_D void bf_pfa(cpx<R>* u)
{
    using F = Pfa<A, B>;
    cpx<R> w[B][A];
    pfa_rows<S, A, B, HALF>(u, w);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
        cpx<R> x[B];
#pragma unroll
        for (int j2 = 0; j2 < B; ++j2) x[j2] = w[j2][k1];
        if constexpr (B == 3) bf3<S>(x);
        else bf5<S>(x);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) u[F::out(k1, k2)] = x[k2];
    }
}

template <int RAD, int S, bool HALF, class R> SP_D void butterfly(cpx<R>* u)
{
    if constexpr (RAD == 20) {
        bf_pfa<S, 4, 5, HALF>(u);
    } else if constexpr (RAD == 12) {
        bf_pfa<S, 4, 3, HALF>(u);
    } else if constexpr (RAD == 10) {
        bf_pfa<S, 2, 5, HALF>(u);
    } else if constexpr (RAD == 6) {
        bf_pfa<S, 2, 3, HALF>(u);
    } else if constexpr (RAD == 5) {
        static_assert(!HALF, "an odd radix cannot run first: its zero inputs are not half");
        bf5<S>(u);
    } else if constexpr (RAD == 4 && HALF) {
        bf4_half<S>(u);
    } else if constexpr (RAD == 32) {
        if constexpr (HALF) bf32_half<S>(u);
        else bf32<S>(u);
    } else if constexpr (RAD == 16) {
        if constexpr (HALF) bf16_half<S>(u);
        else bf16<S>(u);
    } else if constexpr (RAD == 8) {
        if constexpr (HALF) bf8_half<S>(u);
        else bf8<S>(u);
    } else if constexpr (RAD == 4) {
        bf4<S>(u);
    } else if constexpr (RAD == 3) {
        bf3<S>(u);
    } else {
        bf2<S>(u);
    }
}

// ------------------------------------------------------------------ stages
// Layouts map an element index e of a line to a shared-memory slot, with padding after every
// `per` elements (0: none): lay(e + d) = lay(e) + lay.step(d) for d a multiple of per, and
// lay(j + q) = lay(j) + q * lay.unit where no multiple of per lies in (j, j + q].  With per
// the transform's first radix every later stage's strides are multiples of it: the stage
// loops compute one slot per butterfly and add compile-time offsets for the others.

// Per-stage twiddle tables (in shared memory; for double-float, one copy per plan in
// global memory): stage s (span P > 1, radix RAD) keeps w^{r k N/(P RAD)} at
// [k (RAD + 1) + r], so a butterfly reads RAD - 1 consecutive entries; the extra entry
// per row puts the rows of neighbouring k on different banks.
template <class R, int N, bool INV> constexpr int tw_stage_offset(int s)
{
    int off = 0;
    for (int i = 0; i < s; ++i)
        if (span_at<R, N, INV>(i) > 1) off += span_at<R, N, INV>(i) * (radix_at<R, N, INV>(i) + 1);
    return off;
}
template <class R, int N> constexpr int tw_stage_size()
{
    return tw_stage_offset<R, N, false>(PlanOf<R, N>::NS) + tw_stage_offset<R, N, true>(PlanOf<R, N>::NS);
}
template <class R, int N, bool INV> constexpr int tw_base() { return INV ? tw_stage_offset<R, N, false>(PlanOf<R, N>::NS) : 0; }

// Fill the staged tables of plan key K (all threads of the block; a barrier must follow).
template <class R, int N, bool INV, class K = R, int ST = 0>
SP_D void fill_stage_twiddles(cpx<R>* tws, const cpx<R>* __restrict__ tw, int tid, int nthreads)
{
    if constexpr (ST < PlanOf<K, N>::NS) {
        constexpr int P = span_at<K, N, INV>(ST), RAD = radix_at<K, N, INV>(ST);
        if constexpr (P > 1) {
            constexpr int TWS = N / (P * RAD);
            cpx<R>* dst = tws + tw_base<K, N, INV>() + tw_stage_offset<K, N, INV>(ST);
            for (int j = tid; j < P * RAD; j += nthreads) {
                const int k = j / RAD, r = j % RAD;
                dst[k * (RAD + 1) + r] = tw[r * k * TWS];
            }
        }
        fill_stage_twiddles<R, N, INV, K, ST + 1>(tws, tw, tid, nthreads);
    }
}

// A plan is usable when its radices multiply to N and the first and the last divide E (each
// thread enters and leaves with E values of whole butterflies).  A middle radix may leave
// butterflies over: threads take up to ceil((N / RAD) / T) of them, in the last round only the
// first threads of the line.
template <class K, int N> constexpr bool plan_ok()
{
    int prod = 1;
    for (int i = 0; i < PlanOf<K, N>::NS; ++i) {
        const int r = PlanOf<K, N>::R[i];
        if ((i == 0 || i + 1 == PlanOf<K, N>::NS) && PlanOf<K, N>::E % r != 0) return false;
        prod *= r;
    }
    return prod == N && N % PlanOf<K, N>::E == 0;
}

template <class Lay> constexpr bool steps(int d) { return Lay::per == 0 || d % (Lay::per == 0 ? 1 : Lay::per) == 0; }

template <class R, int N, bool INV, int ST, class K = R> struct Stage {
    static_assert(plan_ok<K, N>(), "radix plan does not fit the stage rules");
    static constexpr int E = PlanOf<K, N>::E;
    static constexpr int T = N / E;
    static constexpr int RAD = radix_at<K, N, INV>(ST);
    static constexpr int P = span_at<K, N, INV>(ST);
    static constexpr int STRIDE = N / RAD;           // butterflies of a line
    static constexpr int NB = (STRIDE + T - 1) / T;  // of a thread, at most
    static constexpr int EL = NB * RAD;              // values a thread holds in this stage
    SP_D static bool has(int m, int t) { return T * (m + 1) <= STRIDE || t + T * m < STRIDE; }

    // inputs of this stage from shared memory: v[m RAD + r] = x[t + T m + r N/RAD]
    template <class Lay> SP_D static void load(cpx<R> (&v)[EL], const cpx<R>* sm, const Lay& lay, int t)
    {
#pragma unroll
        for (int m = 0; m < NB; ++m) {
            if (!has(m, t)) continue;
            if constexpr (steps<Lay>(STRIDE)) {
                const cpx<R>* p0 = sm + lay(t + T * m);
                const int st = lay.step(STRIDE);
#pragma unroll
                for (int r = 0; r < RAD; ++r) v[m * RAD + r] = p0[r * st];
            } else {
#pragma unroll
                for (int r = 0; r < RAD; ++r) v[m * RAD + r] = sm[lay(t + T * m + r * STRIDE)];
            }
        }
    }

    // twiddles and butterflies (S = -1 forward, +1 inverse); HALF: inputs r >= RAD/2 are zero
    template <int S, bool HALF> SP_D static void compute(cpx<R> (&v)[EL], const cpx<R>* tws, int t)
    {
#pragma unroll
        for (int m = 0; m < NB; ++m) {
            if (!has(m, t)) continue;
            if constexpr (P > 1) {
                const int k = (t + T * m) % P;
                const cpx<R>* w = tws + tw_base<K, N, INV>() + tw_stage_offset<K, N, INV>(ST) + k * (RAD + 1);
                if constexpr (std::is_same<R, float>::value && RAD == 8) {
                    // FP32: w^2, w^3, w^5, w^6, w^7 from the loaded w and w^4 (two table reads
                    // instead of seven; a few ulps more twiddle error, far below FP32's bar)
                    cpx<R> ww[8];
                    ww[1] = w[1];
                    ww[4] = w[4];
                    ww[2] = cmul(ww[1], ww[1]);
                    ww[3] = cmul(ww[1], ww[2]);
                    ww[5] = cmul(ww[4], ww[1]);
                    ww[6] = cmul(ww[4], ww[2]);
                    ww[7] = cmul(ww[4], ww[3]);
#pragma unroll
                    for (int r = 1; r < RAD; ++r)
                        v[m * RAD + r] = S < 0 ? tw_mul(v[m * RAD + r], ww[r]) : tw_mulc(v[m * RAD + r], ww[r]);
                } else {
#pragma unroll
                    for (int r = 1; r < RAD; ++r)
                        v[m * RAD + r] = S < 0 ? tw_mul(v[m * RAD + r], w[r]) : tw_mulc(v[m * RAD + r], w[r]);
                }
            }
            butterfly<RAD, S, HALF>(&v[m * RAD]);
        }
    }

    // outputs of this stage to shared memory: y[(i - k) RAD + k + q P] = v[m RAD + q]
    template <class Lay> SP_D static void store(const cpx<R> (&v)[EL], cpx<R>* sm, const Lay& lay, int t)
    {
#pragma unroll
        for (int m = 0; m < NB; ++m) {
            if (!has(m, t)) continue;
            const int i = t + T * m;
            const int k = i % P;
            const int base = (i - k) * RAD + k;
            if constexpr (P > 1 && steps<Lay>(P)) {
                cpx<R>* p0 = sm + lay(base);
                const int st = lay.step(P);
#pragma unroll
                for (int q = 0; q < RAD; ++q) p0[q * st] = v[m * RAD + q];
            } else if constexpr (P == 1 && (Lay::per == 0 || Lay::per % RAD == 0)) {
                cpx<R>* p0 = sm + lay(base);  // base = RAD i: no padding inside the butterfly
                const int st = lay.unit();
#pragma unroll
                for (int q = 0; q < RAD; ++q) p0[q * st] = v[m * RAD + q];
            } else {
#pragma unroll
                for (int q = 0; q < RAD; ++q) sm[lay(base + q * P)] = v[m * RAD + q];
            }
        }
    }
};

// Element index held in register slot j after the last stage of a transform (and the
// input index of slot j for the first stage of the opposite-direction transform).
template <class R, int N, bool INV> SP_D int last_element(int t, int j)
{
    constexpr int E = PlanOf<R, N>::E, T = N / E;
    constexpr int RL = radix_at<R, N, INV>(PlanOf<R, N>::NS - 1);
    return t + T * (j / RL) + (j % RL) * (N / RL);
}
// Element index of register slot j for the first stage of a transform.
template <class R, int N, bool INV> SP_D int first_element(int t, int j)
{
    constexpr int E = PlanOf<R, N>::E, T = N / E;
    constexpr int R0 = radix_at<R, N, INV>(0);
    return t + T * (j / R0) + (j % R0) * (N / R0);
}

template <class R, int N, bool INV, int S, class K, int ST, class Lay>
SP_D cpx<R>* later_stages(cpx<R> (&v)[PlanOf<K, N>::E], cpx<R>* full, cpx<R>* other, const Lay& lay, const cpx<R>* tws, int t);

// Stage ST, whose inputs are in x, and the stages after it, which leave their outputs in v.
template <class R, int N, bool INV, int S, bool HALF, class K, int ST, class Lay, int EL>
SP_D cpx<R>* stage_then(cpx<R> (&x)[EL], cpx<R> (&v)[PlanOf<K, N>::E], cpx<R>* fresh, cpx<R>* other, const Lay& lay,
                        const cpx<R>* tws, int t)
{
    using St = Stage<R, N, INV, ST, K>;
    St::template compute<S, HALF>(x, tws, t);
    if constexpr (ST + 1 < PlanOf<K, N>::NS) {
        St::store(x, fresh, lay, t);
        __syncthreads();
        return later_stages<R, N, INV, S, K, ST + 1>(v, fresh, other, lay, tws, t);
    } else {
        return fresh;
    }
}
// Stage ST, whose inputs are in `full` behind a barrier, and the stages after it.
template <class R, int N, bool INV, int S, class K, int ST, class Lay>
SP_D cpx<R>* later_stages(cpx<R> (&v)[PlanOf<K, N>::E], cpx<R>* full, cpx<R>* other, const Lay& lay, const cpx<R>* tws, int t)
{
    using St = Stage<R, N, INV, ST, K>;
    if constexpr (St::EL == PlanOf<K, N>::E) {
        St::load(v, full, lay, t);
        if (other == full) __syncthreads();
        return stage_then<R, N, INV, S, false, K, ST>(v, v, other, full, lay, tws, t);
    } else {
        cpx<R> x[St::EL];
        St::load(x, full, lay, t);
        if (other == full) __syncthreads();
        return stage_then<R, N, INV, S, false, K, ST>(x, v, other, full, lay, tws, t);
    }
}

// Run stages [0, NS) of one transform.  On entry v holds the stage-0 inputs (slot
// j = element first_element(t, j)); on return it holds the last stage's outputs (slot
// j = element last_element(t, j)).  `fresh` must be safe to write on entry (no reads of
// it pending in the block); exchanges alternate between `fresh` and `other`, one barrier
// each: a buffer is written again only after the barrier that follows every read of it.
// With other == fresh (one buffer) a second barrier follows each read.  Returns the
// buffer that is safe to write after the call.  All threads of the block must call this.
template <class R, int N, bool INV, int S, bool HALF0, class K = R, class Lay>
SP_D cpx<R>* run_stages(cpx<R> (&v)[PlanOf<K, N>::E], cpx<R>* fresh, cpx<R>* other, const Lay& lay, const cpx<R>* tws, int t)
{
    return stage_then<R, N, INV, S, HALF0, K, 0>(v, v, fresh, other, lay, tws, t);
}
