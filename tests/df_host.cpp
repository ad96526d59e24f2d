// The float-float header compiled for the host: plain IEEE float operations stand
// for the _rn intrinsics (compile with -ffp-contract=off), and the two approximate
// instructions are the exact results off by up to +-2^-22 relative, more than the
// hardware's error, so what holds here holds for any reciprocal that accurate.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

template <typename T, typename F> static T bits_as(F f) {
    static_assert(sizeof(T) == sizeof(F), "same size");
    T t;
    memcpy(&t, &f, sizeof t);
    return t;
}
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static float __fsqrt_rn(float a) { return std::sqrt(a); }
static float __frcp_rn(float a) { return 1.0f / a; }
static float __int_as_float(int i) { return bits_as<float>(i); }
static int __float_as_int(float f) { return bits_as<int>(f); }
static int __double2hiint(double d) { return (int)(bits_as<uint64_t>(d) >> 32); }
static int __double2loint(double d) { return (int)bits_as<uint64_t>(d); }
static double __hiloint2double(int h, int l) { return bits_as<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static float __uint2float_rn(unsigned u) { return (float)u; }
static float __int2float_rn(int i) { return (float)i; }
static int max(int a, int b) { return a > b ? a : b; }
static float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
static float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
static float2 __ffma2_rn(float2 a, float2 b, float2 c) {
    return make_float2(std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y));
}
static float off(double exact, float x) {
    const uint32_t h = bits_as<uint32_t>(x) * 2654435761u;
    return (float)(exact * (1.0 + ((int)(h >> 22) - 512) * 0x1p-31));
}
struct Approx {
    float* y;
    void operator()(const char* text, float x) const {
        *y = strstr(text, "rsqrt") ? off(1.0 / std::sqrt((double)x), x) : off(1.0 / (double)x, x);
    }
};
// asm("op %0, %1;" : "=f"(y) : "f"(x)) of a float x, or of x.hi
#define asm(...) HOST_ASM(__VA_ARGS__)
#define HOST_ASM(...) Approx{&y}(#__VA_ARGS__, host_operand(x))
template <typename T> static float host_operand(const T& x) {
    if constexpr (sizeof(T) == 4) return x;
    else return x.hi;
}
#include "../paper_2305_09163_gb300/csrc/mfc_df.cuh"
#undef asm

using namespace mfc;

static df pair(const float* p) { return {p[0], p[1]}; }
static void put(float* p, df v) { p[0] = v.hi; p[1] = v.lo; }

extern "C" {
void df_host_tf(long long n, const double* x, float* parts) {
    for (long long i = 0; i < n; ++i) {
        const tf t = tf_from_double(x[i]);
        parts[3 * i] = t.hi;
        parts[3 * i + 1] = t.mid;
        parts[3 * i + 2] = t.lo;
    }
}
void df_host_tf_diff(long long n, const double* x, const double* y, float* d) {
    for (long long i = 0; i < n; ++i) put(d + 2 * i, tf_diff(tf_from_double(x[i]), tf_from_double(y[i])));
}
void df_host_split(long long n, const double* x, int nearest, float* d) {
    for (long long i = 0; i < n; ++i) put(d + 2 * i, nearest ? df_from_double_rn(x[i]) : df_from_double(x[i]));
}
// two-operand functions on float-float pairs, by name
int df_host_op(const char* name, long long n, const float* a, const float* b, float* r) {
#define OP(f, expr)                                             \
    if (!strcmp(name, f)) {                                     \
        for (long long i = 0; i < n; ++i) {                     \
            const df x = pair(a + 2 * i), y = pair(b + 2 * i);  \
            (void)y;                                            \
            put(r + 2 * i, expr);                               \
        }                                                       \
        return 0;                                               \
    }
    OP("prod", df_prod(x, y))
    OP("square", df_square(x))
    OP("scale", df_scale(x, y.hi))
    OP("sum", df_sum(x, y))
    OP("quot", df_quot(x, y))
    OP("quot_f", df_quot_f(x.hi, y))
    OP("root", df_root(x))
    OP("norm", df_norm(x))
#undef OP
    return 1;
}
}
