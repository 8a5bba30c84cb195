// Host check of the 32-bit squares of the distance kernels
// (paper_2203_02527_gb300/csrc/emu64.cuh) under the rule that the kernels use:
// a dimension is narrow when a tile's coordinates lie less than 2^32 units
// apart (they then reach at most 2^33 units: binary32 values beyond have
// no unit that fine).  Against the host's
// own binary64 arithmetic, one rounded subtraction, product and sum per
// dimension.
//   emu64_narrow_check squares <seed> <count> : square_bits_narrow alone, all
//       edges of its range, ties of its rounding and random factors
//   emu64_narrow_check tiles <seed> <tiles>   : whole distances in 1 to 70
//       dimensions, every form
//   emu64_narrow_check bounds <seed> <count>  : within_32_bits just below, at
//       and just above 2^32 units
// Prints "checked bad [narrow dimensions, of them beyond 32 bits]".
#define __host__
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "../../paper_2203_02527_gb300/csrc/emu64.cuh"

using namespace ph0::emu;

static uint32_t fbits(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
static uint64_t dbits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }

static double ref_d2(const float *u, const float *v, int d) {
    volatile double s = 0.0;
    for (int k = 0; k < d; ++k) {
        volatile double t = (double)v[k] - (double)u[k];
        volatile double p = t * t;
        s = s + p;
    }
    return s;
}

static long g_checked = 0, g_bad = 0;
static void want(uint64_t got, uint64_t ref, const char *what) {
    ++g_checked;
    if (got != ref && ++g_bad <= 5) std::fprintf(stderr, "%s: %016llx, not %016llx\n", what, (unsigned long long)got,
                                                 (unsigned long long)ref);
}

static void squares(std::mt19937_64 &rng, long count) {
    auto one = [](uint32_t a, int32_t g) {
        const double t = std::ldexp(double(a), g);
        volatile double p = t * t;
        want(square_bits_narrow(a, g), dbits(p), "square");
    };
    std::vector<uint32_t> edge = {0, 1, 2, 3, 0x7fffffffu, 0x80000000u, 0x80000001u, 0xffffffffu, 0xfffffffeu,
                                  0xb504f333u, 0xb504f334u, 94906265u, 94906266u, 94906267u};  // around sqrt(2^63), sqrt(2^53)
    for (int b = 0; b < 32; ++b)
        for (int o = -2; o <= 2; ++o) edge.push_back((1u << b) + uint32_t(o));
    for (int32_t g = -149; g <= 104; ++g)
        for (uint32_t a : edge) one(a, g);
    for (long i = 0; i < count; ++i) {
        uint32_t a = uint32_t(rng());
        if (i % 4 == 1) a |= 0x80000000u;
        // a square whose bits below the last place are exactly half of it:
        // an odd factor times a power of two
        if (i % 4 == 2) a = (uint32_t(rng()) | 1u) << (rng() % 6);
        if (i % 4 == 3) a >>= rng() % 32;
        one(a, int32_t(rng() % 200) - 120);
    }
}

static void tiles(std::mt19937_64 &rng, long count, long &narrow_dims, long &far_dims) {
    std::uniform_real_distribution<double> U(0.0, 1.0);
    const int P = 12;
    for (long t = 0; t < count; ++t) {
        const int d = 1 + int(t % 70);
        std::vector<float> x(size_t(P) * d);
        for (int k = 0; k < d; ++k) {
            const int kind = int(rng() % 8), up = int(rng() % 24);
            const double off = (rng() & 1 ? -1.0 : 1.0) * std::ldexp(1.0 + U(rng), up);
            for (int p = 0; p < P; ++p) {
                double r;
                switch (kind) {
                    case 0: r = U(rng); break;
                    case 1: r = off + U(rng); break;                               // far from zero, close together
                    case 2: r = off + std::ldexp(std::floor(U(rng) * 4096.0), -up % 12); break;
                    case 3: r = std::floor(U(rng) * 65536.0) * 65536.0 + std::floor(U(rng) * 128.0); break;
                    case 4: r = (rng() & 1 ? -1.0 : 1.0) * U(rng) * 3.0; break;
                    case 5: r = rng() % 3 ? 0.0 : std::ldexp(U(rng), -int(rng() % 9)); break;
                    case 6:  // from 2^23 units, odd, to just above 2^32: beyond 32 bits, differences below 2^32
                        r = std::ldexp((off < 0 ? -1.0 : 1.0) * (p % 2 ? 4294967296.0 + 512.0 * double(rng() % 16000)
                                                                     : 8388609.0 + 2.0 * double(rng() % 4000000)), up - 40);
                        break;
                    default: r = 0.25; break;                                      // all equal
                }
                x[size_t(p) * d + k] = float(r);
            }
        }
        std::vector<int32_t> g(d);
        std::vector<uint32_t> narrow((d + 31) / 32, 0u);
        bool ok = true;
        for (int k = 0; k < d; ++k) {  // as the kernels do
            int32_t lo = 1 << 30, hi = -(1 << 30);
            uint32_t first = ~0u, last = 0;
            for (int p = 0; p < P; ++p) {
                const uint32_t b = fbits(x[size_t(p) * d + k]), o = order_f32(b);
                first = o < first ? o : first;
                last = o > last ? o : last;
                if ((b & 0x7fffffffu) == 0) continue;
                int32_t l, h;
                bit_range_f32(b, l, h);
                lo = l < lo ? l : lo;
                hi = h > hi ? h : hi;
            }
            const bool zero = lo == 1 << 30;
            g[k] = zero ? 0 : lo;
            if (!zero && hi + 1 - lo > 52) ok = false;
            else if (within_32_bits(first, last, g[k])) {
                narrow[k >> 5] |= 1u << (k & 31);
                ++narrow_dims;
                far_dims += !zero && hi + 1 - lo > 32;
            }
        }
        if (!ok) continue;
        std::vector<int64_t> X(size_t(P) * d);
        for (int p = 0; p < P; ++p)
            for (int k = 0; k < d; ++k) X[size_t(p) * d + k] = to_fixed(fbits(x[size_t(p) * d + k]), g[k]);
        for (int i = 0; i < P; ++i)
            for (int j = i + 1; j < P; ++j) {
                const int64_t *xi = &X[size_t(i) * d], *xj = &X[size_t(j) * d];
                const uint64_t ref = dbits(ref_d2(&x[size_t(i) * d], &x[size_t(j) * d], d));
                want(sq_dist_fixed(xi, xj, g.data(), d, 1, 1, narrow.data()), ref, "fixed");
                want(sq_dist_mixed(xi, xj, g.data(), d, 1, 1, narrow.data()), ref, "mixed");
                want(sq_dist_mixed_st<1>(xi, xj, g.data(), d, narrow.data()), ref, "strided");
                switch (d) {
                    case 1: want(sq_dist_mixed_ct<1, 1>(xi, xj, g.data(), narrow[0]), ref, "1"); break;
                    case 5: want(sq_dist_mixed_ct<5, 1>(xi, xj, g.data(), narrow[0]), ref, "5"); break;
                    case 13: want(sq_dist_mixed_ct<13, 1>(xi, xj, g.data(), narrow[0]), ref, "13"); break;
                    case 16: want(sq_dist_mixed_ct<16, 1>(xi, xj, g.data(), narrow[0]), ref, "16"); break;
                    case 31: want(sq_dist_mixed_ct<31, 1>(xi, xj, g.data(), narrow[0]), ref, "31"); break;
                    case 32: want(sq_dist_mixed_ct<32, 1>(xi, xj, g.data(), narrow[0]), ref, "32"); break;
                    default: break;
                }
            }
    }
}

static void bounds(std::mt19937_64 &rng, long count) {
    // two values a unit of 2^g apart from a spread of 2^32 units: lo + 2^32
    // units less one, exactly, plus one, where both fit binary32
    for (long i = 0; i < count; ++i) {
        const int32_t g = int32_t(rng() % 60) - 40;
        const int64_t lo = -(int64_t(rng() % (1u << 24)) << 9);  // 24 bits above 2^9 units
        for (int64_t spread : {(int64_t(1) << 32) - (int64_t(1) << 9), int64_t(1) << 32, (int64_t(1) << 32) + (int64_t(1) << 9)}) {
            const double a = std::ldexp(double(lo), g), b = std::ldexp(double(lo + spread), g);
            if (double(float(a)) != a || double(float(b)) != b) continue;
            const bool got = within_32_bits(order_f32(fbits(float(a))), order_f32(fbits(float(b))), g);
            want(got, spread < (int64_t(1) << 32), "bound");
        }
    }
    want(within_32_bits(~0u, 0, 0), 1, "no values");
    want(within_32_bits(order_f32(fbits(-0.0f)), order_f32(fbits(0.0f)), 0), 1, "zeros");
    want(within_32_bits(order_f32(fbits(-2147483648.0f)), order_f32(fbits(2147483648.0f)), 0), 0, "2^32 across zero");
    want(within_32_bits(order_f32(fbits(-2147483648.0f)), order_f32(fbits(2147483520.0f)), 0), 1, "less across zero");
}

int main(int argc, char **argv) {
    const std::string what = argc > 1 ? argv[1] : "squares";
    std::mt19937_64 rng(argc > 2 ? strtoull(argv[2], 0, 10) : 1);
    const long count = argc > 3 ? atol(argv[3]) : 1000;
    long narrow_dims = 0, far_dims = 0;
    if (what == "squares") squares(rng, count);
    else if (what == "tiles") tiles(rng, count, narrow_dims, far_dims);
    else bounds(rng, count);
    std::printf("%ld %ld %ld %ld\n", g_checked, g_bad, narrow_dims, far_dims);
    return g_bad != 0;
}
