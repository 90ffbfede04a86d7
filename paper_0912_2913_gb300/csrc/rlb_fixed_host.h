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
