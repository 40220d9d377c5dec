// Host check of the exponents by which time-split calls jump BBS generators of
// any modulus (ci_modarith.cuh): x^e with e = 2^E mod lambda, plus lambda where
// that is below a bound, against E plain squarings in 128-bit arithmetic, for
// units and other x.  Prints "ok" when nothing differs.
#include <cstdint>
#include <cstdio>
#include <random>

#include "ci_modarith.cuh"

using namespace ci::dev;
typedef unsigned __int128 u128;

static uint64_t power(uint64_t x, uint64_t e, uint64_t m) {
    uint64_t r = 1 % m;
    for (x %= m; e; e >>= 1) {
        if (e & 1) r = (uint64_t)((u128)r * x % m);
        x = (uint64_t)((u128)x * x % m);
    }
    return r;
}

static long differs(uint64_t m, uint64_t lam, uint64_t x, int E, uint64_t below) {
    uint64_t want = x % m;
    for (int i = 0; i < E; ++i) want = (uint64_t)((u128)want * want % m);
    const uint64_t e = power(2, (uint64_t)E, lam);
    return power(x, e < below ? e + lam : e, m) != want;
}

int main() {
    std::mt19937_64 g(1112);
    long bad = 0, n = 0;
    const uint32_t p = (1u << 30) + 3, q = (1u << 31) - 1;
    const uint32_t pairs[][2] = {{p, q}, {p, p}, {q, q}, {p, 1500000003u}, {1500000003u, 1500000005u},
                                 {65537, 65537}, {59049, 177147}, {3, 2863311531u}, {255 * 257, 65537 * 3},
                                 {5, 4000000005u}, {46349, 4294967291u / 8 * 2 + 1}};
    for (auto &f : pairs) {
        const uint64_t m = (uint64_t)f[0] * f[1], lam = carmichael(f[0], f[1]);
        for (int k = 0; k < 40; ++k) {
            const uint64_t x = k == 0 ? 0 : k == 1 ? f[0] : k == 2 ? f[1] : k == 3 ? 3 : g() % m;
            for (int E : {6, 7, 64, 352, 1000}) bad += differs(m, lam, x, E, 62), ++n;
        }
    }
    for (int k = 0; k < 300; ++k) {
        const uint32_t a = (uint32_t)(g() >> 33) | 3u, b = (uint32_t)(g() >> 33) | 3u;
        const uint64_t m = (uint64_t)a * b, lam = carmichael(a, b);
        bad += differs(m, lam, g() % m, 352, 62), ++n;
    }
    printf("two factors: %ld of %ld differ\n", bad, n);
    long all = bad;
    bad = n = 0;
    for (uint32_t m = 3; m < (1u << 16); ++m) {  // every modulus a 16-bit generator may have
        const uint64_t lam = carmichael16(m);
        for (uint64_t x : {(uint64_t)0, (uint64_t)2, (uint64_t)3, (uint64_t)15, (uint64_t)(g() % m), (uint64_t)(g() % m)})
            for (int E : {4, 5, 32, 33, 64, 77}) bad += differs(m, lam, x, E, 15), ++n;
    }
    printf("16-bit moduli: %ld of %ld differ\n", bad, n);
    bad += all;
    printf("%s\n", bad ? "FAILED" : "ok");
    return bad != 0;
}
