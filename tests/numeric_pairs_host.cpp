// numeric_pairs_host.cpp -- the fixed-point pair products and the three-word accumulators of the
// library's numerics header (rs_numeric.cuh) compiled as host C++, for tests/test_numeric_pairs.py.
// The device intrinsics are given their IEEE-754 meaning on the host, as in numeric_host.cpp.
#include <cmath>
#include <cstdint>
#include <cstring>

#define __device__
#define __forceinline__ inline
static inline uint32_t __float_as_uint(float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; }
static inline float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
static inline double __longlong_as_double(long long x) { double d; std::memcpy(&d, &x, 8); return d; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline long long __float2ll_rz(float a) { return (long long)a; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
template <class T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }   // not called here
static inline unsigned long long atomicAdd(unsigned long long *p, unsigned long long v) {
    const unsigned long long o = *p;
    *p = o + v;
    return o;
}
#include "rs_numeric.cuh"

using namespace rs;

static u96 load96(const uint64_t *p) { return u96{p[0], (uint32_t)p[1]}; }
static void store96(uint64_t *p, u96 v) { p[0] = v.lo; p[1] = v.hi; }
static u192 load192(const uint64_t *p) { return u192{p[0], p[1], p[2]}; }
static void store192(uint64_t *p, u192 v) { p[0] = v.w0; p[1] = v.w1; p[2] = v.w2; }

extern "C" {

int sig_frac(void) { return kSigFrac; }
int term_frac(void) { return kTermFrac; }
int acc_frac(void) { return kAccFrac; }

uint64_t sig(float hi, float lo) { return sig_fixed(df{hi, lo}); }
void pair(uint64_t x, uint64_t y, uint64_t *out) { store96(out, pair_term(x, y)); }
void add96(uint64_t *a, const uint64_t *b) {
    u96 x = load96(a);
    u96_add(x, load96(b));
    store96(a, x);
}
// the sum of the pairs of m factors (x, y) as carry-free words
void limb_sum(const uint64_t *xy, int m, uint64_t *out) {
    uint32_t l[kLimbs] = {};
    for (int i = 0; i < m; ++i)
        for (int j = 0; j < kLimbs; ++j) l[j] += pair_limb(product(xy[2 * i], xy[2 * i + 1]), j);
    store96(out, from_limbs(l[0], l[1], l[2], l[3]));
}
void scaled(uint64_t s, const uint64_t *p, uint64_t *out) { store192(out, scale(s, load96(p))); }
void term192(uint64_t lo, uint64_t hi, uint64_t *out) { store192(out, u192_from_term(((u128)hi << 64) | lo)); }
void add192(uint64_t *a, const uint64_t *b, int neg, int atomic) {
    const u192 v = neg ? u192_neg(load192(b)) : load192(b);
    if (atomic) atomic_add_u192(reinterpret_cast<unsigned long long *>(a), v);
    else store192(a, u192_add(load192(a), v));
}
double to_double(const uint64_t *a) { return u192_to_double(load192(a)); }

}  // extern "C"
