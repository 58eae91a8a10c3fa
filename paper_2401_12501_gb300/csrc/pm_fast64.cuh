// 1/x and log x in float64 for the kernels that the float64 pipe bounds (two instructions a
// clock and SM on GB300): 3 and 11 instructions of it instead of some 10 and 30 (the integer
// ones of the special cases cost nothing beside them).  Both good to an ulp or two of the result
// (of log 2 for arguments next to 1); zero, infinite and undefined arguments give what 1 / x and
// log x give.
#pragma once

// 1 / x: the hardware's approximation (20 bits) and one cubic Newton step.  Results below the
// normal range are 0, those of subnormal arguments infinite.
__device__ __forceinline__ double pm_rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    // 0, infinite or undefined: an exponent of all zeros or ones, on which the step gives NaN
    const bool special = ((__double2hiint(y) + 0x00100000) & 0x7fe00000) == 0;
    return special ? y : fma(y, fma(e, e, e), y);
}

// c_k = 1 / (1 + (k + 1/2) / 128) and -log c_k, by log v = 2 atanh((v - 1) / (v + 1)) summed
// from the small terms (the compiler evaluates it)
struct PmLogTable {
    double2 t[128];
};
constexpr PmLogTable pm_log_table() {
    PmLogTable T{};
    for (int k = 0; k < 128; ++k) {
        const double c = 1.0 / (1.0 + (k + 0.5) / 128.0);
        const double z = (1.0 - c) / (1.0 + c), z2 = z * z;      // -log c = 2 atanh z
        double s = 0.0;
        for (int j = 25; j >= 0; --j) s = s * z2 + 1.0 / (2 * j + 1);
        T.t[k].x = c;
        T.t[k].y = 2.0 * z * s;
    }
    return T;
}
static __device__ const PmLogTable g_pm_log = pm_log_table();

// log x by the table (Tang, "Table-driven implementation of the logarithm function in IEEE
// floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e m, c the tabulated reciprocal next to
// 1/m, log x = e log 2 - log c + log(1 + t), t = c m - 1, |t| <= 2^-8.  For x >= 0 or undefined;
// -infinity for 0 and subnormal x.
__device__ __forceinline__ double pm_log64(double x) {
    const int hi = __double2hiint(x);
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(x));
    const double2 c = g_pm_log.t[(hi >> 13) & 127];
    // e from the bits of 2^52 + 2^51 + e
    const double ed = __hiloint2double(0x43380000, (hi >> 20) - 1023) -
                      ((hi >> 20) < 1023 ? 6755403736023040.0 : 6755399441055744.0);
    const double t = fma(m, c.x, -1.0);
    double q = fma(t, 1.0 / 7.0, -1.0 / 6.0);
    q = fma(t, q, 0.2);
    q = fma(t, q, -0.25);
    q = fma(t, q, 1.0 / 3.0);
    q = fma(t, q, -0.5);
    const double l = fma(ed, 0.69314718055994530942, c.y) + fma(t * t, q, t);
    if ((unsigned int)hi >= 0x7ff00000u) return x;               // infinite or undefined
    return (unsigned int)hi < 0x00100000u ? __hiloint2double((int)0xfff00000, 0) : l;
}
