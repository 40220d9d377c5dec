// ci_crt.cuh -- x <- x^2 mod M for M = p q with both factors known, p and q in
// [2^30, 2^31), on the residues x mod p and x mod q (Garner's form of the
// Chinese remainder theorem; Knuth, TAOCP 2, 4.3.2).  Host-callable, so that a
// host test checks these exact functions against 128-bit arithmetic.
//
// Why: a 62-bit modular square is bound by the FMA-heavy pipe, where a wide
// multiply holds a warp's slot about twice as long as a narrow one.  In the
// 62-bit Barrett form it is 8 wide and 2 narrow products and their carry
// chains (35 instructions, 17 of them on that pipe).  On 32-bit residues it is
// 2 wide + 1 narrow per factor and 1 wide + 3 narrow to join them, i.e. 5 wide
// and 5 narrow, without carries.
#pragma once

#include <cstdint>

#include "ci_modarith.cuh"

namespace ci {
namespace dev {

__host__ __device__ __forceinline__ uint32_t funnel_r32(uint32_t lo, uint32_t hi, uint32_t s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> s);
#endif
}

__host__ __device__ __forceinline__ uint32_t min32(uint32_t a, uint32_t b) { return a < b ? a : b; }

// r^2 mod p for an odd modulus p in (2^30, 2^31) and r in [0, p), by Barrett
// reduction with one subtraction.  r and p - r have the same square, so the
// smaller of the two is squared: t <= (p - 1)^2 / 4 < 2^60.  With h = t >> 29
// (below 2^31) and mu = floor(2^61 / p), the quotient floor(h mu / 2^32) is
// never above t / p and below it by less than
//   2^29 / p < 1/2   (the low bits of t) +
//   h / 2^32 < 1/2   (the fraction of 2^61 / p) +
//   1                (the last floor),
// so the remainder lies in [0, 2p) and one conditional subtraction gives the
// canonical residue.  Squaring r itself leaves one bit less for the quotient;
// its remainder then needs either a second subtraction, which does not fit 32
// bits, or a rounded mu with a 64-bit correction term added to h mu, which
// measured 8 % slower (38.7 against 35.7 cycles per squaring modulo p q of a
// warp at 32 warps per SM): the two integer additions and minima go to the
// ALU, the correction term to the FMA-heavy pipe that bounds the loop.
struct CrtPrime {
    uint32_t p, np, mu;  // np = -p
    __host__ __device__ __forceinline__ void set(uint32_t mod, uint32_t reciprocal) {
        p = mod;
        np = 0u - mod;
        mu = reciprocal;
    }
    __host__ __device__ __forceinline__ void set(uint32_t mod) { set(mod, (uint32_t)((1ull << 61) / mod)); }
    __host__ __device__ __forceinline__ uint32_t sqr(uint32_t r) const {
        const uint32_t v = min32(r, p - r);
        const uint64_t t = (uint64_t)v * v;
        const uint32_t quo = umulhi32(funnel_r32((uint32_t)t, (uint32_t)(t >> 32), 29), mu);
        return addmin32((uint32_t)t + quo * np, np);
    }
};

// Squaring modulo M = p q on the residues (rp, rq), p < q.  digit() is
// Garner's T = (rq - rp) p^-1 mod q, by Shoup's product with a precomputed
// quotient (beta = p^-1 mod q, beta_s = floor(beta 2^32 / q): the estimate is
// floor(d beta / q) or one less for any 32-bit d), so x = rp + p T.
struct CrtModulus {
    CrtPrime P, Q;
    uint32_t beta, beta_s;

    // False (nothing usable) unless both factors lie in (2^30, 2^31), differ
    // and p is invertible modulo q (Fermat's inverse, verified).
    __host__ __device__ __forceinline__ bool set(uint32_t a, uint32_t b) {
        const uint32_t lo = a < b ? a : b, hi = a < b ? b : a;
        if (lo <= (1u << 30) || hi >= (1u << 31) || lo == hi || !(lo & hi & 1u)) return false;
        const Mont31 Mq(hi);
        const uint32_t pm = Mq.to(lo), inv = Mq.pow_m(pm, hi - 2);
        if (Mq.mul(inv, pm) != Mq.one) return false;
        set_inverse(lo, hi, Mq.from(inv));
        return true;
    }
    // p < q in (2^30, 2^31), inv = p^-1 mod q.
    __host__ __device__ __forceinline__ void set_inverse(uint32_t p, uint32_t q, uint32_t inv) {
        P.set(p);
        Q.set(q);
        beta = inv;
        beta_s = (uint32_t)(((uint64_t)inv << 32) / q);
    }
    __host__ __device__ __forceinline__ uint32_t digit(uint32_t rp, uint32_t rq) const {
        const uint32_t d = rq - rp + Q.p;  // in (0, 2q): rp < p < q
        const uint32_t quo = umulhi32(d, beta_s);
        return addmin32(d * beta + quo * Q.np, Q.np);
    }
    // x = rp + p T in [0, M); its low word alone.
    __host__ __device__ __forceinline__ uint64_t value(uint32_t rp, uint32_t rq) const {
        return rp + (uint64_t)P.p * digit(rp, rq);
    }
    __host__ __device__ __forceinline__ uint32_t low(uint32_t rp, uint32_t rq) const {
        return rp + P.p * digit(rp, rq);
    }
};

// 2^e mod (p - 1) for 2 < p < 2^31, through the odd part of p - 1.
__host__ __device__ __forceinline__ uint32_t pow2_mod_order(uint32_t p, uint64_t e) {
    uint32_t m = p - 1, v = 0;
    while (!(m & 1u)) {
        m >>= 1;
        ++v;
    }
    if (e < v || m == 1) return e < v ? 1u << e : 0u;
    const Mont31 M(m);
    return M.from(M.pow2_m(e - v)) << v;
}

// x^(2^e) mod p for an odd p < 2^31 and an x with x^(p-1) = 1 mod p, from and to
// the Montgomery form of x (`one`: that of 1): the exponent reduced mod p - 1.
// e >= 1.
__host__ __device__ __forceinline__ uint32_t squarings_m(uint32_t p, uint32_t one, uint32_t xm, uint64_t e) {
    return Mont31(p, one).pow_m(xm, pow2_mod_order(p, e));
}

}  // namespace dev
}  // namespace ci
