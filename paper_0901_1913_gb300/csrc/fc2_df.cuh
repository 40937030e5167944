// fc2_df.cuh -- double-float ("float-float") arithmetic for the exact sums.
//
// A value is an unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// which carries about 48 significant bits.  The error-free transformations are
// Knuth's two-sum and the fused multiply-add product error (Dekker, Numer.
// Math. 18 (1971) 224; Joldes, Muller & Popescu, ACM TOMS 44 (2017) 48).  The
// float pipes of this part are some sixty times wider than its double pipe,
// so sums that need more than float but less than double precision are
// cheaper this way.  Not part of the public ABI.
#pragma once
#include "fc2_common.cuh"

namespace fc2 {

struct dfl {
    float h, l;
};
struct dfc {
    dfl re, im;
};

// s + e = a + b exactly (any magnitudes)
FC2_D dfl df_two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return dfl{s, (a - (s - bb)) + (b - bb)};
}
// s + e = a + b exactly, for |a| >= |b| (or a == 0)
FC2_D dfl df_fast_sum(float a, float b) {
    const float s = a + b;
    return dfl{s, b - (s - a)};
}
// a * b, relative error ~2^-47
FC2_D dfl df_mul(dfl a, dfl b) {
    const float p = a.h * b.h;
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, e);
    e = fmaf(a.l, b.h, e);
    return df_fast_sum(p, e);
}

// a * b for double-float complex numbers of modulus about one; each component
// is formed as one two-sum of the leading products plus the small terms, so
// its absolute error is ~2^-47 |a| |b|.
FC2_D dfc dfc_mul(const dfc& a, const dfc& b) {
    dfc r;
    {
        const float p1 = a.re.h * b.re.h, p2 = a.im.h * b.im.h;
        const float e1 = fmaf(a.re.h, b.re.h, -p1), e2 = fmaf(a.im.h, b.im.h, -p2);
        const dfl s = df_two_sum(p1, -p2);
        float lo = s.l + (e1 - e2);
        lo = fmaf(a.re.h, b.re.l, lo);
        lo = fmaf(a.re.l, b.re.h, lo);
        lo = fmaf(-a.im.h, b.im.l, lo);
        lo = fmaf(-a.im.l, b.im.h, lo);
        r.re = df_two_sum(s.h, lo);
    }
    {
        const float p1 = a.re.h * b.im.h, p2 = a.im.h * b.re.h;
        const float e1 = fmaf(a.re.h, b.im.h, -p1), e2 = fmaf(a.im.h, b.re.h, -p2);
        const dfl s = df_two_sum(p1, p2);
        float lo = s.l + (e1 + e2);
        lo = fmaf(a.re.h, b.im.l, lo);
        lo = fmaf(a.re.l, b.im.h, lo);
        lo = fmaf(a.im.h, b.re.l, lo);
        lo = fmaf(a.im.l, b.re.h, lo);
        r.im = df_two_sum(s.h, lo);
    }
    return r;
}

// Accumulator acc += w * z (w, z double-float reals); the running sum keeps
// its rounding errors in acc.l.
FC2_D void df_acc_mul(dfl& acc, dfl w, dfl z) {
    const float p = w.h * z.h;
    float e = fmaf(w.h, z.h, -p);
    e = fmaf(w.h, z.l, e);
    e = fmaf(w.l, z.h, e);
    const dfl s = df_two_sum(acc.h, p);
    acc.h = s.h;
    acc.l += s.l + e;
}

FC2_D dfl df_from_double(double v) {
    const float h = (float)v;
    return dfl{h, (float)(v - (double)h)};
}

// z (1 + eps + i s) for a double-float z of modulus about one and a small
// rotation: eps a float of modulus below 2^-27, s a double-float below 1e-4.
// Each component is z's plus one double-float product (leading product, its
// FMA error and the cross terms) and the float eps term, gathered by two-sums:
// absolute error ~2^-47, like dfc_mul, with fewer operations.
FC2_D dfc dfc_rot_small(const dfc& z, float eps, dfl s) {
    dfc r;
    {
        const float p = z.im.h * s.h;  // z.im s
        float e = fmaf(z.im.h, s.h, -p);
        e = fmaf(z.im.h, s.l, e);
        e = fmaf(z.im.l, s.h, e);
        const dfl t = df_two_sum(z.re.h, -p);
        const float lo = fmaf(z.re.h, eps, (t.l + z.re.l) - e);
        r.re = df_two_sum(t.h, lo);
    }
    {
        const float p = z.re.h * s.h;  // z.re s
        float e = fmaf(z.re.h, s.h, -p);
        e = fmaf(z.re.h, s.l, e);
        e = fmaf(z.re.l, s.h, e);
        const dfl t = df_two_sum(z.im.h, p);
        const float lo = fmaf(z.im.h, eps, (t.l + z.im.l) + e);
        r.im = df_two_sum(t.h, lo);
    }
    return r;
}

// e^{2 pi i u 2^-64} for a 64-bit phase u, to ~2^-46: the top 16 bits select
// two table factors e^{2 pi i a / 256} and e^{2 pi i b / 65536} (double-float,
// t1[a] and t2[b]); the remaining 48 bits give theta = 2 pi delta < 1e-4 and
// e^{i theta} = 1 - theta^2/2 + i (theta - theta^3/6) (the next terms are
// below 1e-17).  theta^2/2 < 4.6e-9 lies below half an ulp of 1, so the real
// part is 1 plus a float correction (float theta^2: 3e-16 absolute), and the
// product with the table factors is a small rotation (dfc_rot_small).
FC2_D dfc df_phasor(uint64_t u, const dfc* t1, const dfc* t2) {
    const int a = (int)(u >> 56), b = (int)((u >> 48) & 255u);
    const uint64_t r = u & ((1ull << 48) - 1);
    const float rh = (float)(uint32_t)(r >> 24), rl = (float)(uint32_t)(r & 0xffffffu);
    const dfl d = df_two_sum(rh * 9.094947017729282e-13f, rl * 5.421010862427522e-20f);  // 2^-40, 2^-64
    const dfl th = df_mul(d, dfl{6.28318548202514648f, -1.74845553146951525e-07f});  // 2 pi
    const float eps = -0.5f * th.h * th.h;
    const float t3 = th.h * th.h * th.h * (1.0f / 6.0f);
    const dfl s = df_fast_sum(th.h, th.l - t3);
    return dfc_rot_small(dfc_mul(t1[a], t2[b]), eps, s);
}

// e^{2 pi i u 2^-64} in double from the same split as df_phasor: two table
// factors times 1 - theta^2/2 + i (theta - theta^3/6), theta < 1e-4 (the
// dropped terms are below 4e-18).
FC2_D double2 d_phasor(uint64_t u, const double2* t1, const double2* t2) {
    const double2 A = t1[(int)(u >> 56)], B = t2[(int)((u >> 48) & 255u)];
    const double th = (double)(int64_t)(u & ((1ull << 48) - 1)) * 3.4061215800865545e-19;  // 2 pi 2^-64
    const double th2 = th * th;
    const double c = fma(-0.5, th2, 1.0);
    const double s = fma(th * th2, -1.0 / 6.0, th);
    const double pr = fma(A.x, B.x, -A.y * B.y), pi = fma(A.x, B.y, A.y * B.x);
    return make_double2(fma(pr, c, -pi * s), fma(pr, s, pi * c));
}

// ---------------------------------------------- sums exact in fixed point
// The last precision tier of the exact fix-up keeps the float pipes' speed but
// none of their accumulation error: each harmonic multiple's phasor is
// evaluated directly from its exact integer phase k u (~2^-46, no chains of
// products), the products with the double-float weights are summed
// in double-float over blocks of FX_BLOCK samples, and every block sum enters
// a 64-bit integer accumulator at a fixed scale 2^s -- integer additions are
// exact and associative, so the result does not depend on the order and the
// only errors are the per-term ones (phasor, product, block, and the
// conversion's rounding at 2^-s).
constexpr int FX_BLOCK = 8;

// Scale exponent s for sums of at most nterm terms of modulus <= vmax: the
// scaled terms add up to less than 2^61 in modulus, and so does every partial
// sum of the converted block pieces (each at most its terms' sum plus half a
// unit of rounding), far inside the 64-bit range.  Clamped to the float
// exponent range.
FC2_D int fx_exponent(float vmax, int64_t nterm) {
    const int ev = (vmax > 0.0f) ? ilogbf(vmax) + 1 : 0;  // vmax < 2^ev
    int en = 0;
    while ((1ll << en) < nterm) ++en;
    int s = 61 - ev - en;
    if (s > 126) s = 126;
    if (s < -126) s = -126;
    return s;
}

// Two double-float values side by side.  The packed float instructions do both
// halves in one issue slot at the scalar rate of the pipe, with the same
// rounding as their scalar forms.
struct dfl2 {
    float2 h, l;
};
struct dfc2 {
    dfl2 re, im;
};
FC2_D float2 f2_of(float v) { return make_float2(v, v); }
FC2_D float2 f2_neg(float2 a) { return make_float2(-a.x, -a.y); }
FC2_D float2 f2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
FC2_D float2 f2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
FC2_D float2 f2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
FC2_D float2 f2_sub(float2 a, float2 b) {
    float2 r;
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
        " sub.rn.f32x2 c, a, b;\n mov.b64 {%0, %1}, c;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// a + b exactly (df_two_sum on both halves), and a - b
FC2_D dfl2 df2_two_sum(float2 a, float2 b) {
    const float2 s = f2_add(a, b), bb = f2_sub(s, a);
    return dfl2{s, f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb))};
}
FC2_D dfl2 df2_two_diff(float2 a, float2 b) {
    const float2 s = f2_sub(a, b), bb = f2_sub(s, a);
    return dfl2{s, f2_sub(f2_sub(a, f2_sub(s, bb)), f2_add(b, bb))};
}
// a + b exactly for |a| >= |b| or a = 0 (or equal exponents)
FC2_D dfl2 df2_fast_sum(float2 a, float2 b) {
    const float2 s = f2_add(a, b);
    return dfl2{s, f2_sub(b, f2_sub(s, a))};
}
FC2_D dfc2 dfc2_mul(const dfc2& a, const dfc2& b) {  // dfc_mul on both halves
    dfc2 r;
    {
        const float2 p1 = f2_mul(a.re.h, b.re.h), p2 = f2_mul(a.im.h, b.im.h);
        const float2 e1 = f2_fma(a.re.h, b.re.h, f2_neg(p1));
        const float2 e2 = f2_fma(a.im.h, b.im.h, f2_neg(p2));
        const dfl2 s = df2_two_diff(p1, p2);
        float2 lo = f2_add(s.l, f2_sub(e1, e2));
        lo = f2_fma(a.re.h, b.re.l, lo);
        lo = f2_fma(a.re.l, b.re.h, lo);
        lo = f2_fma(f2_neg(a.im.h), b.im.l, lo);
        lo = f2_fma(f2_neg(a.im.l), b.im.h, lo);
        r.re = df2_two_sum(s.h, lo);
    }
    {
        const float2 p1 = f2_mul(a.re.h, b.im.h), p2 = f2_mul(a.im.h, b.re.h);
        const float2 e1 = f2_fma(a.re.h, b.im.h, f2_neg(p1));
        const float2 e2 = f2_fma(a.im.h, b.re.h, f2_neg(p2));
        const dfl2 s = df2_two_sum(p1, p2);
        float2 lo = f2_add(s.l, f2_add(e1, e2));
        lo = f2_fma(a.re.h, b.im.l, lo);
        lo = f2_fma(a.re.l, b.im.h, lo);
        lo = f2_fma(a.im.h, b.re.l, lo);
        lo = f2_fma(a.im.l, b.re.h, lo);
        r.im = df2_two_sum(s.h, lo);
    }
    return r;
}
FC2_D dfc2 dfc2_pair(const dfc& a, const dfc& b) {
    return dfc2{{make_float2(a.re.h, b.re.h), make_float2(a.re.l, b.re.l)},
                {make_float2(a.im.h, b.im.h), make_float2(a.im.l, b.im.l)}};
}

// e^{2 pi i u 2^-64} of two 64-bit phases, to ~2^-46, as df_phasor: a table
// value z for the top 16 bits of each times the small rotation by the other 48
// (dfc_rot_small).  z comes from one table of 65536 double-float entries
// e^{2 pi i m / 65536} (T16; 1 MB, read through the caches; no product of two
// table values), or is the product of the two 256-entry tables' values
// (df2_table).  In the T16 table a component is 0 or at least sin(2 pi / 65536),
// which the rotation's correction does not exceed, so its leading sum needs
// only the three-operation form; a product of two table values may leave a
// tiny component there.
FC2_D dfc2 df2_table16(uint64_t u1, uint64_t u2, const dfc* __restrict__ t16) {
    return dfc2_pair(t16[(int)(u1 >> 48)], t16[(int)(u2 >> 48)]);
}
FC2_D dfc2 df2_table(uint64_t u1, uint64_t u2, const dfc* t1, const dfc* t2) {
    return dfc2_mul(dfc2_pair(t1[(int)(u1 >> 56)], t1[(int)(u2 >> 56)]),
                    dfc2_pair(t2[(int)((u1 >> 48) & 255u)], t2[(int)((u2 >> 48) & 255u)]));
}
template <bool T16>
FC2_D dfc2 df2_rotate(uint64_t u1, uint64_t u2, const dfc2& z) {
    const uint64_t M48 = (1ull << 48) - 1;
    const uint64_t r1 = u1 & M48, r2 = u2 & M48;
    const float2 rh = make_float2((float)(uint32_t)(r1 >> 24), (float)(uint32_t)(r2 >> 24));
    const float2 rl = make_float2((float)((uint32_t)r1 & 0xffffffu), (float)((uint32_t)r2 & 0xffffffu));
    // the high part is a multiple of 2^-40, the low part below it
    const dfl2 d = df2_fast_sum(f2_mul(rh, f2_of(9.094947017729282e-13f)),    // 2^-40
                                f2_mul(rl, f2_of(5.421010862427522e-20f)));   // 2^-64
    const float2 ch = f2_of(6.28318548202514648f), cl = f2_of(-1.74845553146951525e-07f);  // 2 pi
    const float2 p = f2_mul(d.h, ch);
    float2 e = f2_fma(d.h, ch, f2_neg(p));
    e = f2_fma(d.h, cl, e);
    e = f2_fma(d.l, ch, e);
    const dfl2 th = df2_fast_sum(p, e);
    const float2 eps = f2_mul(f2_mul(f2_of(-0.5f), th.h), th.h);
    const float2 t3 = f2_mul(f2_mul(th.h, th.h), th.h);
    const dfl2 s = df2_fast_sum(th.h, f2_fma(t3, f2_of(-(1.0f / 6.0f)), th.l));
    dfc2 r;
    {
        const float2 q = f2_mul(z.im.h, s.h);  // z.im s
        float2 g = f2_fma(z.im.h, s.h, f2_neg(q));
        g = f2_fma(z.im.h, s.l, g);
        g = f2_fma(z.im.l, s.h, g);
        dfl2 t;
        if constexpr (T16) {
            t.h = f2_sub(z.re.h, q);
            t.l = f2_sub(z.re.l, f2_add(q, f2_sub(t.h, z.re.h)));
        } else {
            t = df2_two_diff(z.re.h, q);
            t.l = f2_add(t.l, z.re.l);
        }
        r.re = df2_two_sum(t.h, f2_fma(z.re.h, eps, f2_sub(t.l, g)));
    }
    {
        const float2 q = f2_mul(z.re.h, s.h);  // z.re s
        float2 g = f2_fma(z.re.h, s.h, f2_neg(q));
        g = f2_fma(z.re.h, s.l, g);
        g = f2_fma(z.re.l, s.h, g);
        dfl2 t = T16 ? df2_fast_sum(z.im.h, q) : df2_two_sum(z.im.h, q);
        r.im = df2_two_sum(t.h, f2_fma(z.im.h, eps, f2_add(f2_add(t.l, z.im.l), g)));
    }
    return r;
}

// acc += w z on both halves (df_acc_mul)
FC2_D void df2_acc_mul(dfl2& acc, const dfl2& w, const dfl2& z) {
    const float2 p = f2_mul(w.h, z.h);
    float2 e = f2_fma(w.h, z.h, f2_neg(p));
    e = f2_fma(w.h, z.l, e);
    e = f2_fma(w.l, z.h, e);
    const dfl2 s = df2_two_sum(acc.h, p);
    acc.h = s.h;
    acc.l = f2_add(acc.l, f2_add(s.l, e));
}

// v rounded to the nearest integer, |v| < 2^61, from two 32-bit conversions: a
// 64-bit conversion runs on the double pipe (64 clocks per warp).  v = hi 2^30
// + rem exactly (hi = 0 or rem has at most 23 bits), |rem| <= 2^29, and hi 2^30
// is even, so rounding rem rounds v.
FC2_D long long fx_round(float v) {
    const float hi = rintf(v * 9.313225746154785e-10f);  // 2^-30
    const float rem = fmaf(-hi, 1073741824.0f, v);
    return ((long long)__float2int_rn(hi) << 30) + (long long)__float2int_rn(rem);
}
FC2_D void fx_flush(long long& acc, float h, float l, float scale) {
    acc += fx_round(h * scale) + fx_round(l * scale);
}

// Fixed-point sums of the samples [i0, i1) over the 2H multiples k by a group
// of NWG warps.  Warp w of the group takes the samples i = i0 + r + lph w +
// stride q (r < lph = 32 / 2H, stride = lph NWG, q = 0, 1, ..), blocks of
// FX_BLOCK consecutive q summed in double-float.  Lane (g lph + r) 2 + half
// holds the multiples k = g + 1 and g + 1 + H of row r side by side in packed
// arithmetic and takes every second block, so phases and weights serve two
// multiples and the weighted data's sums (k <= H) occupy every lane.  The
// group stages its samples' phases u_i = A_i + ju B_i (mod 2^64) and weights in
// shared memory one tile (qt of a block's samples for both halves) ahead, and
// the next sample's table values are fetched a step ahead.  Bound by the float
// pipe (59% active; about 100 warp instructions per sample and multiple, half of
// them packed) together with L1 (74%: the scattered reads of the large table);
// the one-warp form, on shared-memory tables, 46% and 25% in a short launch.
// One lane per multiple with every load, phase and 64-bit conversion of its own
// took 177 instructions and waited on its loads:
//   plan of n = 10^6, H = 8, N = 2^25 (481 bins): 66.3 -> 34.2 ms
//   1024 survey curves, H = 2..6 (30526 entries): 10.0 -> 7.6 ms
// Samples past i1 enter with weight zero, which
// leaves a block's bits unchanged.  Weights as float high parts at [i] and low
// parts at [ntot + i]; sq, sp = 2^s of each kind.
// Lanes of group g return, per multiple m = 0, 1 (k = g + 1 + m H), their
// q[m][re, im] = sum w e^{2 pi i k u_i} 2^s and p[re, im] (k = g + 1, weighted
// data).
struct FxSums {
    long long q[2][2], p[2];
};
template <int NWG>
struct FxStage {
    static constexpr int CAP = 64 * NWG + 2;  // two runs, the second two slots on (banks)
    uint64_t u[2][CAP];
    float4 w[2][CAP];
};
template <bool T16, int NWG>
FC2_D FxSums fx_group_sums(FxStage<NWG>& st, const uint64_t* __restrict__ Aph,
                           const uint64_t* __restrict__ Bph, const float* __restrict__ wq32,
                           const float* __restrict__ wp32, int64_t ntot, uint64_t ju, int H,
                           int64_t i0, int64_t i1, const dfc* __restrict__ t1,
                           const dfc* __restrict__ t2, float sq, float sp) {
    constexpr int NTG = 32 * NWG;
    constexpr int UN = NWG == 1 ? 4 : 8;  // (8 in the one-warp form: 8.3 against 7.6 ms)
    const int lane = threadIdx.x & 31;
    const int tid = NWG == 1 ? lane : (int)threadIdx.x, wg = tid >> 5;
    auto sync = [] {
        if constexpr (NWG == 1) __syncwarp();
        else __syncthreads();
    };
    const int lph = 32 / (2 * H);
    const int qt = lph <= 4 ? 8 : (lph <= 8 ? 4 : 2);  // 2 qt lph <= 64
    const int stride = lph * NWG, run = qt * stride;
    const int unit = lane >> 1, half = lane & 1;
    const int g = unit / lph, r = unit - g * lph;
    const bool act = g < H;
    FxSums out{};
    const uint32_t k1 = act ? g + 1 : 1, kH = H;
    // tiles: block pair, then the sub-runs of its blocks
    const int subs = FX_BLOCK / qt;
    const int64_t pair = 2 * FX_BLOCK * (int64_t)stride;
    const int64_t ntile = (i1 - i0 + pair - 1) / pair * subs;
    int64_t base = i0;  // first sample of the tile to stage
    int sub = 0;
    auto stage = [&](int buf) {
        for (int e = tid; e < 2 * run; e += NTG) {
            const int hf = e >= run ? 1 : 0, x = e - hf * run;
            const int64_t i = base + (int64_t)hf * FX_BLOCK * stride + x;
            uint64_t u = 0;
            float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < i1) {
                u = Aph[i] + ju * Bph[i];
                w = make_float4(wq32[i], wq32[ntot + i], wp32[i], wp32[ntot + i]);
            }
            st.u[buf][e + 2 * hf] = u;
            st.w[buf][e + 2 * hf] = w;
        }
        base += run;
        if (++sub == subs) { sub = 0; base += FX_BLOCK * stride; }
    };
    const float2 zero = f2_of(0.f);
    dfl2 b0{zero, zero}, b1{zero, zero}, b2{zero, zero};
    const int at = act ? r + lph * wg + half * (run + 2) : 0;
    if (ntile > 0) stage(0);
    int done = 0;
    for (int64_t t = 0; t < ntile; ++t) {
        const int buf = (int)(t & 1);
        sync();  // tile t is staged, and the other buffer's readers are done
        if (t + 1 < ntile) stage(buf ^ 1);
        const uint64_t* su = st.u[buf] + at;
        const float4* sw = st.w[buf] + at;
        dfc2 zn;
        uint64_t n1 = su[0] * k1, n2 = n1 + su[0] * kH;
        if constexpr (T16) zn = df2_table16(n1, n2, t1);
#pragma unroll UN
        for (int q = 0; q < qt; ++q) {
            const uint64_t u1 = n1, u2 = n2;
            dfc2 z = zn;
            if (q + 1 < qt) {  // the next sample's table values, a step ahead
                const uint64_t u = su[(q + 1) * stride];
                n1 = u * k1;
                n2 = n1 + u * kH;
                if constexpr (T16) zn = df2_table16(n1, n2, t1);
            }
            if constexpr (!T16) z = df2_table(u1, u2, t1, t2);
            z = df2_rotate<T16>(u1, u2, z);
            const float4 w = sw[q * stride];
            const dfl2 a{f2_of(w.x), f2_of(w.y)}, b{f2_of(w.z), f2_of(w.w)};
            df2_acc_mul(b0, a, z.re);
            df2_acc_mul(b1, a, z.im);
            df2_acc_mul(b2, b, dfl2{make_float2(z.re.h.x, z.im.h.x), make_float2(z.re.l.x, z.im.l.x)});
        }
        if (++done == subs) {
            done = 0;
            fx_flush(out.q[0][0], b0.h.x, b0.l.x, sq);
            fx_flush(out.q[0][1], b1.h.x, b1.l.x, sq);
            fx_flush(out.q[1][0], b0.h.y, b0.l.y, sq);
            fx_flush(out.q[1][1], b1.h.y, b1.l.y, sq);
            fx_flush(out.p[0], b2.h.x, b2.l.x, sp);
            fx_flush(out.p[1], b2.h.y, b2.l.y, sp);
            b0 = b1 = b2 = dfl2{zero, zero};
        }
    }
    sync();  // the stage may be written again
    return out;
}

// Adds the lanes of each group (2 lph consecutive lanes) into its first lane;
// exact integers, any order.
FC2_D void fx_group_sum(FxSums& s, int H) {
    const int lane = threadIdx.x & 31, n = 2 * (32 / (2 * H));
    FxSums t = s;
    for (int o = 1; o < n; ++o) {
        const int src = (lane + o) & 31;
        t.q[0][0] += __shfl_sync(0xffffffffu, s.q[0][0], src);
        t.q[0][1] += __shfl_sync(0xffffffffu, s.q[0][1], src);
        t.q[1][0] += __shfl_sync(0xffffffffu, s.q[1][0], src);
        t.q[1][1] += __shfl_sync(0xffffffffu, s.q[1][1], src);
        t.p[0] += __shfl_sync(0xffffffffu, s.p[0], src);
        t.p[1] += __shfl_sync(0xffffffffu, s.p[1], src);
    }
    s = t;
}

FC2_D float warp_max_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Every lane receives the warp's sum of (hi, lo) float pairs (butterfly of
// error-free two-sums; two-sum is symmetric in its operands, so all lanes end
// with the same bits).
FC2_D float2 warp_allsum_pair(float hi, float lo) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        const dfl t = df_two_sum(hi, h2);
        hi = t.h;
        lo = (lo + l2) + t.l;
    }
    return make_float2(hi, lo);
}

}  // namespace fc2
