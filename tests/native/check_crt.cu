// Host check of the residue form of the modular square (ci_crt.cuh) against
// 128-bit arithmetic, over the whole range of factors it accepts: random
// and consecutive odd factors, the ends of (2^30, 2^31), and residues 0, 1,
// p / 2 on both sides, p - 1 and where the quotient is nearly exact.  Prints
// "ok" when nothing differs.
#include <cstdint>
#include <cstdio>
#include <random>

#include "ci_crt.cuh"

using namespace ci::dev;
typedef unsigned __int128 u128;

static uint64_t gcd(uint64_t a, uint64_t b) {
    while (b) {
        const uint64_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

int main() {
    std::mt19937_64 g(11125239);
    long bad = 0, n = 0;
    const uint32_t lo = (1u << 30) + 1, hi = (1u << 31) - 1;

    // CrtPrime::sqr
    for (int k = 0; k < 400000; ++k) {
        uint32_t p;
        if (k < 4000) p = lo + (uint32_t)k;
        else if (k < 8000) p = hi - (uint32_t)(k - 4000);
        else p = lo + (uint32_t)(g() % (hi - lo + 1));
        p |= 1u;
        CrtPrime c;
        c.set(p);
        for (int j = 0; j < 24; ++j) {
            uint32_t r;
            switch (j) {
                case 0: r = 0; break;
                case 1: r = 1; break;
                case 2: r = p - 1; break;
                case 3: r = p - 2; break;
                case 4: r = p / 2; break;
                case 5: r = p / 2 + 1; break;
                default: r = (uint32_t)(g() % p);
            }
            if (j >= 12) {  // r^2 just above or below a multiple of p near the top of the range
                const uint64_t m = (uint64_t)p * (p / 4 - (uint64_t)(g() % 1000));
                uint64_t s = (uint64_t)__builtin_sqrtl((long double)m);
                r = (uint32_t)(s + (g() & 1));
                if (r >= p) r = p - 1;
            }
            bad += c.sqr(r) != (uint32_t)((uint64_t)r * r % p), ++n;
        }
    }
    printf("square modulo a factor: %ld of %ld differ\n", bad, n);
    long all = bad;

    // CrtModulus: acceptance, value, chains of squarings
    bad = n = 0;
    CrtModulus m;
    bad += m.set(1u << 30, hi) || m.set(lo, lo) || m.set(lo, 1u << 31) || m.set(lo + 1, hi) || m.set(3, hi);
    long taken = 0;
    for (int k = 0; k < 60000; ++k) {
        uint32_t a = (k & 1) ? lo + 2 * (uint32_t)(g() % 5000) : lo + (uint32_t)(g() % (hi - lo + 1));
        uint32_t b = (k & 2) ? hi - 2 * (uint32_t)(g() % 5000) : lo + (uint32_t)(g() % (hi - lo + 1));
        a |= 1u;
        b |= 1u;
        if (!m.set(a, b)) continue;  // not coprime, or a composite q without Fermat's inverse
        ++taken;
        bad += gcd(a, b) != 1, ++n;
        const uint32_t p = m.P.p, q = m.Q.p;
        const uint64_t M = (uint64_t)p * q;
        uint64_t x = k % 7 == 0 ? M - 1 : k % 7 == 1 ? 0 : k % 7 == 2 ? (uint64_t)p * (g() % q) : g() % M;
        uint32_t rp = (uint32_t)(x % p), rq = (uint32_t)(x % q);
        bad += m.value(rp, rq) != x, ++n;
        for (int j = 0; j < 40; ++j) {
            x = (uint64_t)((u128)x * x % M);
            rp = m.P.sqr(rp);
            rq = m.Q.sqr(rq);
            bad += m.value(rp, rq) != x, ++n;
            bad += m.low(rp, rq) != (uint32_t)x, ++n;
        }
    }
    printf("square modulo p q: %ld of %ld differ (%ld moduli)\n", bad, n, taken);
    all += bad;

    // Mont31: products, conversions, powers; primality against the 32-bit form
    bad = n = 0;
    const uint32_t edge[] = {3u, 5u, 7u, 61u, 65535u, 1073741827u, 2147483629u, 2147483647u};
    for (int t = 0; t < 60000; ++t) {
        const uint32_t mod = t < 8 ? edge[t] : (uint32_t)((g() >> (33 + g() % 20)) | 3u);
        const Mont31 M(mod);
        for (int k = 0; k < 4; ++k) {
            const uint32_t a = k == 0 ? mod - 1 : (uint32_t)(g() % mod), b = k < 2 ? mod - 1 : (uint32_t)(g() % mod);
            bad += M.from(M.mul(M.to(a), M.to(b))) != (uint32_t)((uint64_t)a * b % mod), ++n;
            const uint64_t w = g() % ((uint64_t)mod << 32);
            bad += M.from(M.to_wide(w)) != w % mod, ++n;
            const uint64_t e = g() >> (g() % 64);
            uint64_t r = 1 % mod, c = a, d = 1 % mod;
            for (uint64_t x = e; x; x >>= 1) {
                if (x & 1) r = r * c % mod;
                c = c * c % mod;
            }
            c = 2 % mod;
            for (uint64_t x = e; x; x >>= 1) {
                if (x & 1) d = d * c % mod;
                c = c * c % mod;
            }
            bad += M.from(M.pow_m(M.to(a), e)) != r, ++n;
            bad += M.from(M.pow2_m(e)) != d, ++n;
        }
        bad += is_prime_u32<true>(mod) != is_prime_u32<false>(mod), ++n;
    }
    printf("31-bit Montgomery: %ld of %ld differ\n", bad, n);
    all += bad;

    // squarings_m and pow2_mod_order over Blum primes and primes = 1 mod 4
    bad = n = 0;
    for (int k = 0; k < 400; ++k) {
        uint32_t p = (k < 20 ? (k < 10 ? lo : hi - 4000u) + 2u * (uint32_t)(g() % 1000) : lo + (uint32_t)(g() % (hi - lo + 1))) | 1u;
        while (!is_prime_u32(p)) p += 2;
        if (p > hi) continue;
        const Mont32 M(p);
        for (int j = 0; j < 60; ++j) {
            const uint64_t e = j < 40 ? 1 + (uint64_t)j : 1 + (g() >> (20 + g() % 40));
            u128 r = 1, b = 2;
            for (uint64_t t = e; t; t >>= 1) {
                if (t & 1) r = r * b % (p - 1);
                b = b * b % (p - 1);
            }
            bad += pow2_mod_order(p, e) != (uint32_t)r, ++n;
            const uint32_t x = (uint32_t)(j % 7 == 0 ? 0 : g() % p);
            uint32_t y = x;
            if (e <= 64) {
                for (uint64_t t = 0; t < e; ++t) y = (uint32_t)((uint64_t)y * y % p);
                bad += M.from(squarings_m(p, M.one, M.to(x), e)) != y, ++n;
            }
        }
    }
    printf("repeated squarings: %ld of %ld differ\n", bad, n);
    all += bad;
    if (all || taken < 1000) return 1;
    printf("ok\n");
    return 0;
}
