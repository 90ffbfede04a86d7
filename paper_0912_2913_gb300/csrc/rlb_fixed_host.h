// rlb_fixed_host.h -- host-side construction of the fixed-point constants
// (included inside namespace rlb by rlb_fixed.cuh).

// a / b as an unevaluated pair of binary64 values
inline void fx_div2(double a, double b, double& hi, double& lo) {
    hi = a / b;
    lo = fma(-hi, b, a) / b;
}
inline FxConst fx_const(int64_t v) {
    const int32_t l = (int32_t)((uint32_t)v >> 1);
    return {(int32_t)(v >> 32), l, (1u << 30) + ((uint32_t)l >> 1)};
}
// (hi + lo) 2^s as a constant for fx_mul; |value| < 2^63
inline FxConst fx_const(double hi, double lo, int s) {
    return fx_const((int64_t)ldexp(hi, s) + (int64_t)llrint(ldexp(lo, s)));
}
// (hi + lo) 2^s times the factor (1 - 2^-54) of the binary64 weights
inline FxConst fx_const_w(double hi, double lo, int s) {
    const int64_t v = (int64_t)ldexp(hi, s) + (int64_t)llrint(ldexp(lo, s));
    return fx_const(v - (v >> 54));
}
// The constants of FxRun.  Those in fixed point exist for the lattice speeds of
// the kernels that use them (outside they would not fit 64 bits; 0 there).
inline bool fx_covers(double c_l) { return c_l >= 1.0 && c_l <= 2.0; }
inline FxRun make_fx_run(double omega, double c_l) {
    FxRun k{};
    k.om4 = 0.25 * omega;
    k.omw = 1.0 - omega;
    k.m3cl2 = -3.0 * c_l * c_l;
    k.three_cl = 3.0 * c_l;
    k.m_max = (float)(0.98 / (c_l * c_l));
    k.q_scale = (float)ldexp(12.0 * c_l / omega, -33);
    if (!(68.0f * k.q_scale < 9e-5f)) k.q_scale = NAN;  // (fx_nonpositive)
    k.c_l = (float)c_l;
    if (!fx_covers(c_l)) return k;
    double qh, ql, th, tl, c2h = c_l * c_l, c2l = fma(c_l, c_l, -c2h);
    fx_div2(omega, 36.0, qh, ql);
    th = qh / c2h;
    tl = (fma(-th, c2h, qh) + (ql - th * c2l)) / c2h;
    k.kE = fx_const_w(th, tl, 65);
    k.kS = fx_const_w(qh, ql, 65);
    fx_div2(omega, 12.0, qh, ql);
    k.kU = fx_const_w(qh, ql, 65);
    // omega (1 - 2 / (3 c_l^2)) = omega - 24 omega / (36 c_l^2)
    const int64_t kE65 = (int64_t)ldexp(th, 65) + (int64_t)llrint(ldexp(tl, 65));
    const int64_t v = (int64_t)ldexp(omega, 62) - 3 * kE65;
    k.k0 = fx_const(v - (v >> 54));
    fx_div2(1.0, 36.0, qh, ql);
    th = qh / c2h;
    tl = (fma(-th, c2h, qh) + (ql - th * c2l)) / c2h;
    k.kE1 = fx_const_w(th, tl, 65);
    // (3 - 2 / c_l^2) / 3 = 1 - 24 / (36 c_l^2)
    const double ph = 24.0 * th, hi = 1.0 - ph;
    k.kE0 = fx_const_w(hi, ((1.0 - hi) - ph) - fma(24.0, th, -ph) - 24.0 * tl, 62);
    fx_div2(5.0, 9.0, qh, ql);
    k.kQ = fx_const(qh, ql, 63);
    fx_div2(1.0, 6.0, qh, ql);
    k.kG = fx_const(qh, ql, 63);
    return k;
}
