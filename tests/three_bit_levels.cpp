// Host build of the quantizer's device code: a thread's three-bit codes and sums for given coefficients, against Algorithm 1 as it stands (eight
// levels sorted by value and code, midpoints, ">=" descent).  Whole coefficients, ties and coefficients that rounding makes meet are what it is
// about.  (Infinities and NaN, whose sign differs between the machines, are left out: they fail the test for regular tables.)
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>
#include <math.h>
#include <stdio.h>
#include <algorithm>
#include <random>

static inline uint32_t __float_as_uint(float x) { uint32_t u; memcpy(&u, &x, 4); return u; }
static inline float __uint_as_float(uint32_t u) { float x; memcpy(&x, &u, 4); return x; }
static inline int __float_as_int(float x) { int u; memcpy(&u, &x, 4); return u; }
static inline float __int_as_float(int u) { float x; memcpy(&x, &u, 4); return x; }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) { return (uint32_t)((((uint64_t)hi << 32 | lo) << s) >> 32); }
static inline int __popc(uint32_t x) { return __builtin_popcount(x); }
// (named by templates of the header that nothing here instantiates)
static inline uint32_t __byte_perm(uint32_t, uint32_t, uint32_t) { return 0; }
static inline float __fdividef(float a, float b) { return a / b; }
static inline void __syncwarp() {}
static inline void __syncthreads() {}
static inline unsigned __ballot_sync(unsigned, bool) { return 0; }
template <class T> static inline T __shfl_sync(unsigned, T v, int) { return v; }
template <class T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
static inline int __reduce_add_sync(unsigned, int v) { return v; }
static struct { int x; } threadIdx, blockDim;

#include "amq_quantize_device.cuh"

using namespace amq;

template <int EPT>
static void reference(const float (&w)[EPT], const float (&a)[3], uint32_t (&bits)[3], float (&csum)[3])
{
    struct Level { float v; int c; } l[8];
    for (int c = 0; c < 8; ++c) {
        float s = 0;
        for (int i = 0; i < 3; ++i) s += ((c >> (2 - i)) & 1) ? a[i] : -a[i];
        l[c] = {s, c};
    }
    std::stable_sort(l, l + 8, [](const Level& x, const Level& y) { return x.v < y.v; });
    float thr[7];
    for (int p = 0; p < 7; ++p) thr[p] = (l[p].v + l[p + 1].v) * 0.5f;
    for (int i = 0; i < 3; ++i) { bits[i] = 0; csum[i] = 0; }
    for (int j = EPT - 1; j >= 0; --j) {                        // (the device's order of the sums)
        int lo = 0, hi = 7;
        while (lo < hi) { const int m = (lo + hi) / 2; if (w[j] >= thr[m]) lo = m + 1; else hi = m; }
        for (int i = 0; i < 3; ++i) {
            const bool b = (l[lo].c >> (2 - i)) & 1;
            bits[i] |= (uint32_t)b << j;
            csum[i] += b ? w[j] : -w[j];
        }
    }
}

static long different = 0, seen = 0;

template <int EPT>
static void compare(const float (&a)[3], std::mt19937& g)
{
    const uint32_t valid = EPT == 32 ? ~0u : (1u << EPT) - 1;
    std::uniform_real_distribution<float> u(-1, 1);
    const float span = 1.2f * (fabsf(a[0]) + fabsf(a[1]) + fabsf(a[2])) + 1e-30f;
    float w[EPT], abs_w = 0;
    uint32_t positive = 0;
    for (int j = EPT - 1; j >= 0; --j) {
        float v = u(g) * span;
        if (j % 4 == 1) { v = 0; for (int i = 0; i < 3; ++i) v += (g() & 1) ? a[i] : -a[i]; }                   // a level
        if (j % 4 == 2) { v = a[g() % 3]; if (g() & 1) v = -v; if (g() & 1) v = 0.5f * (v + a[g() % 3]); }      // often a midpoint
        if (j % 8 == 3) v = 0;
        w[j] = v + 0.0f;
        abs_w += fabsf(w[j]);
        positive |= (uint32_t)!(__float_as_uint(w[j]) >> 31) << j;
    }
    uint32_t want[3], bits[3];
    float want_sum[3], sum[3], thr[7];
    reference<EPT>(w, a, want, want_sum);
    for (int sums = 0; sums < 2; ++sums) {
        three_bit_codes<EPT>(w, a, positive, abs_w, valid, sums != 0, thr, bits, sum);
        ++seen;
        for (int i = 0; i < 3; ++i)
            if (bits[i] != want[i] || (sums && sum[i] != want_sum[i])) {
                if (++different <= 8)
                    printf("coefficients %.9g %.9g %.9g: plane %d is %x, not %x (sum %.9g, %.9g)\n", a[0], a[1], a[2], i, bits[i], want[i],
                           sums ? sum[i] : 0.0f, want_sum[i]);
                break;
            }
    }
}

static void both(float x, float y, float z, std::mt19937& g)
{
    const float a[3] = {x, y, z};
    compare<8>(a, g);
    compare<32>(a, g);
}

int main()
{
    std::mt19937 g(7);
    std::normal_distribution<float> normal(0, 1);
    std::uniform_real_distribution<float> exponent(-30, 2);
    auto sign = [&](float v) { return g() & 1 ? v : -v; };
    const float few[] = {0.0f, -0.0f, 1, 2, 3, 0.5f, -1, -2, 0.1f, 0.3f, 0.2f, 1e8f, 16777216.0f, 1.0000001f, 0.99999994f, 3e37f, 1e-40f};
    for (float x : few) for (float y : few) for (float z : few) both(x, y, z, g);
    for (int r = 0; r < 100000; ++r) {
        const float x = normal(g), y = normal(g), z = normal(g);
        both(x, y, z, g);
        // two that nearly tie, beside one of any size
        const float big = x * exp2f(-exponent(g)), near = y * (1 + (int)(g() % 5 - 2) * 1.2e-7f);
        float p[3] = {big, y, near};
        std::shuffle(p, p + 3, g);
        both(p[0], p[1], p[2], g);
        // one that is the sum of the others, one far larger than the others
        float s[3] = {sign(y + z), y, z}, t[3] = {sign(16777216.0f * (1 + g() % 4)), y, z};
        std::shuffle(s, s + 3, g);
        std::shuffle(t, t + 3, g);
        both(s[0], s[1], s[2], g);
        both(t[0], t[1], t[2], g);
    }
    printf("%ld of %ld differ\n", different, seen);
    return different != 0;
}
