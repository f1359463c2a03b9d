// CPU check of the fixed-point primitives (csrc/ivb_fixed.cuh, the file the
// kernels include) with stand-ins for the device intrinsics. The MUFU
// approximations are modelled as the nearest float moved by up to one (rcp) or
// two (rsqrt) units in the last place, their documented error.
// Usage: fixed_check N  ->  key=value counts of wrong results.
#include <cfenv>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#if defined(__x86_64__) || defined(__i386__)
#include <quadmath.h>
typedef __float128 quad;
#define Q_EXP expq
#define Q_LOG logq
#define Q_EXP2 exp2q
#define Q_FLOOR floorq
#else
typedef long double quad;
#define Q_EXP expl
#define Q_LOG logl
#define Q_EXP2 exp2l
#define Q_FLOOR floorl
#endif
#define __device__
#define __forceinline__ inline

static inline long long bits(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline double from_bits(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
static inline int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
static inline float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
static inline int __clz(int a) { return a ? __builtin_clz((unsigned)a) : 32; }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
static int off = 0;   // units the modelled approximation is off by
static inline float moved(float r, int u) { return r > 0.5f && r < 1.0f ? __int_as_float(__float_as_int(r) + u) : r; }
static inline float rcp_approx_f(float x) { return moved((float)(1.0 / (double)x), off); }
static inline float rsqrt_approx_f(float x) { return moved((float)(1.0 / std::sqrt((double)x)), 2 * off); }

#include "../../paper_2507_20769_gb300/csrc/ivb_fixed.cuh"
using namespace ivb;

static uint64_t state = 88172645463325252ULL;
static uint64_t rnd() {   // xorshift64* (Vigna, 2016)
    state ^= state >> 12; state ^= state << 25; state ^= state >> 27;
    return state * 2685821657736338717ULL;
}
static double uniform(double a, double b) { return a + (b - a) * (double)(rnd() >> 11) * 0x1p-53; }
// biased exponent in [e0, e1]; half of the significands powers of two, all ones, or with a run of either
static double pick(int e0, int e1) {
    uint64_t m = rnd() & 0xFFFFFFFFFFFFFULL;
    const uint64_t low = (1ULL << (rnd() % 52)) - 1;
    switch (rnd() & 7) {
    case 0: m = 0; break;
    case 1: m = 0xFFFFFFFFFFFFFULL; break;
    case 2: m &= ~low; break;
    case 3: m |= low; break;
    }
    return from_bits((long long)(((uint64_t)(e0 + (int)(rnd() % (uint64_t)(e1 - e0 + 1))) << 52) | m));
}
static double near_of(double x) { return from_bits(bits(x) + (long long)(rnd() % 5) - 2); }

int main(int argc, char** argv) {
    const long N = argc > 1 ? std::atol(argv[1]) : 100000;
    static fx64 et[kExpTab];
    static LogEntry lt[kLogTab];
    const quad two32 = 4294967296.0;
    for (int j = 0; j < kExpTab; ++j) et[j] = (fx64)(Q_EXP2((quad)j / kExpTab) * two32 * (two32 / 4) + (quad)0.5);
    const quad ln2 = Q_LOG((quad)2);
    for (int j = 0; j < kLogTab; ++j) {
        lt[j].c = (fx32)(((1u << 30) + (kLogTab + j) - 1) / (kLogTab + j));
        const quad v = -Q_LOG((quad)lt[j].c / 1048576) - 1023 * ln2, w = Q_FLOOR(v);
        lt[j].ip = (int)w;
        lt[j].frac = (fx64)((v - w) * two32 * two32);
    }
    long rcp = 0, div = 0, root = 0, exact = 0, ex = 0, lg = 0, wide2 = 0, small = 0;
    for (long i = 0; i < N; ++i) {
        off = (int)(rnd() % 3) - 1;
        const double y = pick(1, 2044), k = (double)(1 + rnd() % 64);
        double x = pick(1, 2046), s = pick(1, 2046);
        switch (i & 7) {
        case 0: x = from_bits((bits(x) & 0xFFFFFFFFFFFFFLL) | ((long long)bexp(y) << 52)); break;
        case 1: x = std::ldexp(y, (int)(rnd() % 40) - 20) * k; break;      // exact quotients
        case 2: x = near_of(y); break;
        case 3: s = pick(800, 1200); s = from_bits(bits(s) & ~0x7FFFFFFLL); s *= s; break;   // squares
        case 4: s = pick(800, 1200); s = from_bits(bits(s) & ~0x7FFFFFFLL); s = near_of(s * s); break;
        case 5: s = from_bits(bits(4.0) - 1 - (long long)(rnd() % 64)); break;
        }
        for (int up = 0; up < 2; ++up) {
            volatile double vx = x, vy = y, vs = s;
            std::fesetround(up ? FE_UPWARD : FE_DOWNWARD);
            volatile double r = 1.0 / vy, q = vx / vy, g = std::sqrt(vs);
            std::fesetround(FE_TONEAREST);
            if (up == 0) {   // round to nearest
                volatile double rn = 1.0 / vy, qn = vx / vy, gn = std::sqrt(vs);
                rcp += from_bits((long long)rcp_near(y)) != rn;
                if (std::isfinite(x) && x > 0 && div_fits(x, y)) div += from_bits((long long)div_near(x, y)) != qn;
                root += from_bits((long long)sqrt_near(s)) != gn;
            }
            rcp += from_bits((long long)rcp_mag(y, up)) != r;
            if (std::isfinite(x) && x > 0 && div_fits(x, y)) {
                div += from_bits((long long)div_mag(x, y, rcp62(sig53(y)), up)) != q;
                exact += up == 0 && std::fma(q, y, -x) == 0.0;
            }
            root += from_bits((long long)sqrt_mag(s, up)) != g;
        }
        double a = 0.0;
        switch (i & 3) {
        case 0: a = uniform(-700, 700); break;
        case 1: a = uniform(-2, 2); break;
        case 2: a = pick(0, 1032) * ((rnd() & 1) ? -1 : 1); break;
        case 3: a = near_of((double)((long)(rnd() % 1000000) - 500000) * 0x1.62e42fefa39efp-10); break;   // near k ln2/512
        }
        if (i == 0) a = 0.0;
        if (exp_fits(a)) {
            const quad t = Q_EXP((quad)a);
            const double d = from_bits((long long)exp_mag(a, et, false)), u = from_bits((long long)exp_mag(a, et, true));
            ex += !(d <= t && t <= u && from_bits(bits(d) + 3) >= t && from_bits(bits(u) - 3) <= t);
            wide2 += from_bits(bits(u) - 2) > d;
            const double e = from_bits((long long)exp_near(a, et));
            const quad half = ((quad)from_bits(bits(e) + 1) - (quad)e) / 2;   // below 0.52 units, above half of them at a power of two
            ex += !(e - half * (quad)1.04 <= t && t <= e + half * (quad)1.04);
        }
        switch (i & 3) {
        case 0: a = pick(1, 2046); break;
        case 1: a = uniform(0.5, 4); break;
        case 2: a = uniform(0.9, 1.1); break;
        case 3: a = near_of((i & 4) ? 1.0 : 1.0 + (double)(rnd() % 1024) / 1024); break;
        }
        const quad t = Q_LOG((quad)a);
        double d, u;
        if (log_val(a, lt, FX_DOWN, &d) != log_val(a, lt, FX_UP, &u)) ++lg;
        else if (!log_val(a, lt, FX_DOWN, &d)) {
            small += 1;
            lg += !(t < 0x1.01p-7 && t > -0x1.01p-7);
        } else {
            const long long st = t < 0 ? -3 : 3;   // three steps toward +inf
            lg += !(d <= t && t <= u && from_bits(bits(d) + st) >= t && from_bits(bits(u) - st) <= t);
            double e;
            if (!log_val(a, lt, FX_NEAR, &e)) {
                lg += !(t < 0x1.01p-3 && t > -0x1.01p-3);
                continue;
            }
            // half a unit, and 12 units of 2^-64
            const quad most = std::fabs(from_bits(bits(e) + 1) - e) / 2 + (quad)0xCp-64, off = t - (quad)e;
            lg += !(off <= most && off >= -most);
        }
    }
    std::printf("rcp=%ld div=%ld sqrt=%ld exp=%ld log=%ld exact=%ld wide=%ld small=%ld\n", rcp, div, root, ex, lg, exact,
                wide2, small);
    return 0;
}
