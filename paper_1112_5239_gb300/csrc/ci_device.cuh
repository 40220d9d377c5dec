// ci_device.cuh -- device building blocks of the chaotic-iterations PRNG for
// sm_103a: seeding, strategy sources (Algorithm 2 XORshift, 32-bit xor128,
// BBS with Barrett reduction), and the per-warp generation loop that runs
// Algorithm 4/5's mixing and the Eq. (Oplus) update with the lanes' state in
// registers.
//
// Mapping of the paper's thread model onto a warp: one lane per stream; a group
// of C <= 32 consecutive lanes mixes within itself, so a warp holds 32 / C
// whole groups and the exchange of last strategies ("shmem[o1]",
// "shmem[o2]") is two register shuffles.  All lanes of the warp execute each
// shuffle before any lane updates its slot, which is the synchronous reading
// of Algorithm 4's unsynchronised shared-memory read/write: iteration i reads
// the partners' strategies of iteration i - 1.
#pragma once

#include <cuda.h>  // CUtensorMap (TMA descriptor type only)

#include <cstdint>
#include <type_traits>

#include "ci_crt.cuh"
#include "ci_internal.h"

namespace ci {
namespace dev {

constexpr uint32_t kFull = 0xffffffffu;

// A bounds check of the CI_CHECKED build, written where every lane of the warp
// is converged: if `cond` fails in any lane, lane 0 records (id, index) in the
// state's status word (the first failure wins) and the whole warp returns from
// the enclosing function, so no lane leaves a warp-collective step early and
// the guarded access is never made.  Compiled out otherwise.
#ifdef CI_CHECKED
#define CI_WARP_CHECK(st, cond, id, index)                                                             \
    do {                                                                                              \
        if (__any_sync(0xffffffffu, !(cond))) {                                                       \
            if ((threadIdx.x & 31) == 0 && (st).check)                                                \
                atomicCAS((st).check, 0ull,                                                           \
                          ((unsigned long long)(id) << 56) | ((unsigned long long)(index) & ((1ull << 56) - 1))); \
            return;                                                                                   \
        }                                                                                             \
    } while (0)
#else
#define CI_WARP_CHECK(st, cond, id, index) ((void)0)
#endif

// ------------------------------------------------------------------ seeding
// splitmix64 (Steele, Lea & Flood 2014) used counter-based: draw k of lane l
// is the (l * 2^32 + k + 1)-th output of the generator started at `seed`.
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t lane_draw(uint64_t seed, uint64_t lane, uint64_t k) {
    return sm64_mix(seed + ((lane << 32) + k + 1ull) * 0x9E3779B97F4A7C15ull);
}

// ------------------------------------------------------- strategy sources
// Each source: load/store of its words for lane l, the pair of combination
// arrays the lane uses, and next() returning the lane's own strategy word.
// kHeavy: next() is long, the output loops are not unrolled; kOneStep: nor
// are four steps written per turn (eleven squarings each would leave the
// instruction cache).

// 32-bit xor128 (Marsaglia), the xor-like the paper uses for Algorithm 4.
struct SrcXor128 {
    static constexpr bool kHeavy = false, kOneStep = false;
    uint32_t a, b, c, d;
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) {
        a = s.u32[F_A * s.P + l];
        b = s.u32[F_B * s.P + l];
        c = s.u32[F_C * s.P + l];
        d = s.u32[F_D * s.P + l];
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const {
        s.u32[F_A * s.P + l] = a;
        s.u32[F_B * s.P + l] = b;
        s.u32[F_C * s.P + l] = c;
        s.u32[F_D * s.P + l] = d;
    }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = 0;
        a2 = 1;
    }
    __device__ __forceinline__ uint32_t next() {
        const uint32_t s = a ^ (a << 11);
        a = b;
        b = c;
        c = d;
        d = d ^ (d >> 19) ^ (s ^ (s >> 8));
        return d;
    }
};

// Algorithm 2: z ^= z << 13; z ^= z >> 17; z ^= z << 5.
struct SrcXorshift32 {
    static constexpr bool kHeavy = false, kOneStep = false;
    uint32_t z;
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) { z = s.u32[F_A * s.P + l]; }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const { s.u32[F_A * s.P + l] = z; }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = 0;
        a2 = 1;
    }
    __device__ __forceinline__ uint32_t next() {
        z ^= z << 13;
        z ^= z >> 17;
        z ^= z << 5;
        return z;
    }
};

// xor64, the 64-bit xorshift of the paper's Sec. 7 measurements; the lane's
// strategy word is the low 32 bits of each step.
struct SrcXor64 {
    static constexpr bool kHeavy = false, kOneStep = false;
    uint64_t z;
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) {
        z = (uint64_t)s.u32[F_A * s.P + l] | ((uint64_t)s.u32[F_B * s.P + l] << 32);
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const {
        s.u32[F_A * s.P + l] = (uint32_t)z;
        s.u32[F_B * s.P + l] = (uint32_t)(z >> 32);
    }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = 0;
        a2 = 1;
    }
    __device__ __forceinline__ uint32_t next() {
        z ^= z << 13;
        z ^= z >> 7;
        z ^= z << 17;
        return (uint32_t)z;
    }
};

// ------------------------------------------------ Barrett arithmetic
// a b mod M for M of bit length n, 2 <= n <= 62, and canonical a, b < M, by
// Barrett reduction (Barrett 1986; base-2 form of Menezes et al., Handbook of
// Applied Cryptography, Alg. 14.42) with one bit more precision on both sides
// of the quotient estimate: X = a b, q1 = floor(X / 2^(n-2)),
// mu = floor(2^(2n+1) / M), q = floor(q1 mu / 2^(n+3)).  Each floor then
// costs less than 1/2 (X < 2^(2n), M >= 2^(n-1)), so q >= floor(X / M) - 1
// and r = X - q M lies in [0, 2M): one subtraction gives the canonical
// residue (the textbook estimate needs two).  q1 < 2^(n+2) and
// mu < 2^(n+2) fit 64 bits; the state stores mu << (61 - n) for n <= 61 and
// mu itself for n = 62, where one shift of the product's high half follows.
// Canonical at every step, so the BBS low bits need no conversion (a
// Montgomery square plus the reduction to canonical form measured 22 % slower
// at full occupancy on sm_103a).
__host__ __device__ __forceinline__ uint64_t mul_hi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

__host__ __device__ __forceinline__ uint32_t bit_length64(uint64_t M) {
#ifdef __CUDA_ARCH__
    return 64u - (uint32_t)__clzll((long long)M);
#else
    return 64u - (uint32_t)__builtin_clzll(M);
#endif
}

// The stored reciprocal floor(2^(2n+1) / M), shifted as described above.
// Scaled by 2^(64-n), it is the quotient of the 128-bit 2^(n+65) = hi 2^64 by
// the normalised divisor d = M 2^(64-n) (top bit set, d > hi), found as two
// 32-bit quotient digits, each estimated from the divisor's top half and
// corrected at most twice (Knuth, TAOCP 2, Alg. 4.3.1D, in the two-digit form
// of Warren's Hacker's Delight).  The only other case, M = 2^61 (d = hi),
// and M < 2 take restoring long division.
__host__ __device__ __forceinline__ uint64_t barrett_mu(uint64_t M) {
    const uint32_t n = bit_length64(M);
    uint64_t q;
    const uint64_t d = n >= 2 ? M << (64 - n) : 0, hi = 1ull << (n + 1);
    if (n >= 2 && hi < d) {
        const uint64_t d1 = d >> 32, d0 = d & 0xFFFFFFFFull;
        uint64_t q1 = hi / d1, r = hi - q1 * d1;  // digit 1 of (hi 2^32) / d
        while ((q1 >> 32) || q1 * d0 > (r << 32)) {
            --q1;
            r += d1;
            if (r >> 32) break;
        }
        const uint64_t u = (hi << 32) - q1 * d;  // partial remainder, below d
        uint64_t q0 = u / d1;                    // digit 0 of (u 2^32) / d
        r = u - q0 * d1;
        while ((q0 >> 32) || q0 * d0 > (r << 32)) {
            --q0;
            r += d1;
            if (r >> 32) break;
        }
        q = (q1 << 32) | q0;
    } else {
        uint64_t rem = 1;
        q = 0;
        for (uint32_t i = 0; i < 2 * n + 1; ++i) {
            rem <<= 1;
            q <<= 1;
            if (rem >= M) {
                rem -= M;
                q |= 1;
            }
        }
    }
    return n <= 61 ? q << (61 - n) : q;
}

// 32 x 32 -> 64-bit product, one mul.wide (a single wide multiply-add on the
// FMA-heavy pipe).
__device__ __forceinline__ uint64_t mul_wide32(uint32_t a, uint32_t b) {
    uint64_t r;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}

struct Barrett62 {
    uint64_t M, mu;      // mu: barrett_mu(M)
    uint32_t s1, s2, t;  // n - 2; 66 - n (at most 63: below n = 4, X < 2^64 and the high half is 0); n == 62
    uint32_t sl;         // n - 34 (limb form, n >= 34)
    uint64_t nM;         // 2^64 - M
    __host__ __device__ __forceinline__ void set(uint64_t mod, uint64_t mu_stored) {
        M = mod;
        mu = mu_stored;
        const uint32_t n = bit_length64(mod);
        s1 = n - 2;
        s2 = 66 - n < 63 ? 66 - n : 63;
        t = n == 62 ? 1u : 0u;
        sl = n >= 34 ? n - 34 : 0u;
        nM = 0ull - mod;
    }
    __host__ __device__ __forceinline__ uint64_t mul(uint64_t a, uint64_t b) const {
        const uint64_t lo = a * b, hi = mul_hi64(a, b);
        const uint64_t q = mul_hi64((hi << s2) | (lo >> s1), mu) >> t;
        const uint64_t r = lo - q * M;
        return r >= M ? r - M : r;
    }
    __host__ __device__ __forceinline__ uint64_t sqr(uint64_t x) const { return mul(x, x); }

    // The same Barrett square on 32-bit limbs, for 34 <= n <= 62 (so the
    // quotient input floor(X / 2^(n-2)) starts in limb 1 or above).
    // Schoolbook products (Knuth, TAOCP 2, Alg. 4.3.1M), each one mul.wide;
    // every carry is an explicit add-with-carry, so the products are the only
    // work on the FMA-heavy pipe, the kernel's limiting pipe.
    //   X = x^2 = x0^2 + 2 x0 x1 2^32 + x1^2 2^64 (x1 < 2^30, so 2 x1 fits);
    //   q1 = X >> (n - 2): two funnel shifts by n - 34 of limbs 1..3;
    //   q = floor(q1 mu / 2^64) >> t: all four partial products, exactly;
    //   r = X - q M mod 2^64 (r < 2M < 2^63), then one conditional
    //   subtraction, decided by the sign of r - M.
    // Equal to mul(x, x) for every canonical x (checked on the host against
    // 128-bit remainders for every n from 34 to 62, and on the GPU).
    __device__ __forceinline__ uint64_t sqr_limb(uint64_t x) const {
        const uint32_t x0 = (uint32_t)x, x1 = (uint32_t)(x >> 32);
        const uint64_t p00 = mul_wide32(x0, x0), d = mul_wide32(x0, x1 + x1), p11 = mul_wide32(x1, x1);
        uint32_t X1, X2, X3;
        asm("add.cc.u32 %0, %3, %4;\n\t"
            "addc.cc.u32 %1, %5, %6;\n\t"
            "addc.u32 %2, %7, 0;"
            : "=r"(X1), "=r"(X2), "=r"(X3)
            : "r"((uint32_t)(p00 >> 32)), "r"((uint32_t)d), "r"((uint32_t)p11), "r"((uint32_t)(d >> 32)),
              "r"((uint32_t)(p11 >> 32)));
        const uint32_t q0 = __funnelshift_r(X1, X2, sl), q1 = __funnelshift_r(X2, X3, sl);
        const uint32_t m0 = (uint32_t)mu, m1 = (uint32_t)(mu >> 32);
        const uint32_t c00 = __umulhi(q0, m0);
        const uint64_t c01 = mul_wide32(q0, m1), c10 = mul_wide32(q1, m0), c11 = mul_wide32(q1, m1);
        uint32_t w2, w3;  // bits 64..127 of q1 mu
        asm("{\n\t.reg .u32 a, b, c, a2;\n\t"
            "add.cc.u32 a, %2, %3;\n\t"
            "addc.cc.u32 b, %4, %5;\n\t"
            "addc.u32 c, %6, 0;\n\t"
            "add.cc.u32 a2, a, %7;\n\t"
            "addc.cc.u32 %0, b, %8;\n\t"
            "addc.u32 %1, c, 0;\n\t}"
            : "=r"(w2), "=r"(w3)
            : "r"(c00), "r"((uint32_t)c01), "r"((uint32_t)(c01 >> 32)), "r"((uint32_t)c11),
              "r"((uint32_t)(c11 >> 32)), "r"((uint32_t)c10), "r"((uint32_t)(c10 >> 32)));
        const uint32_t qa = __funnelshift_r(w2, w3, t), qb = w3 >> t;
        const uint32_t n0 = (uint32_t)nM, n1 = (uint32_t)(nM >> 32);
        uint64_t r = mul_wide32(qa, n0) + (((uint64_t)X1 << 32) | (uint32_t)p00);
        const uint32_t rh = (uint32_t)(r >> 32) + qa * n1 + qb * n0;
        r = ((uint64_t)rh << 32) | (uint32_t)r;
        const uint64_t dm = r - M;
        return (int32_t)(dm >> 32) < 0 ? r : dm;
    }
};

// Blum Blum Shub strategy source (Algorithm 5 generalised to w = 5 bits per
// squaring for 62-bit moduli): 7 chunks of 5 bits, then two shift steps.
struct SrcBbs {
    static constexpr bool kHeavy = true, kOneStep = true;
    Barrett62 B;
    uint64_t y;  // BBS state, canonical in [0, M)
    uint32_t sel;
    bool limb;  // every modulus of the warp has 34..62 bits (all seeded ones): the limb-form square;
                // otherwise (33-bit imported moduli) the generic one
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) {
        y = s.u64[G_Y * s.P + l];
        B.set(s.u64[G_M * s.P + l], s.u64[G_MU * s.P + l]);
        sel = s.u32[F_SEL * s.P + l];
        limb = __all_sync(kFull, bit_length64(B.M) >= 34u);
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const { s.u64[G_Y * s.P + l] = y; }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = (int)(sel & 7u);
        a2 = 8 + (int)((sel >> 8) & 7u);
    }
    // One BBS output: x <- x^2 mod M (its low bits are the secure ones).
    template <bool kLimb>
    __device__ __forceinline__ uint32_t bbs() {
        y = kLimb ? B.sqr_limb(y) : B.sqr(y);
        return (uint32_t)y;
    }
    template <bool kLimb>
    __device__ __forceinline__ uint32_t assemble() {
        uint32_t t = 0;
#pragma unroll
        for (int c = 0; c < 7; ++c) t = (t << 5) | (bbs<kLimb>() & 31u);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint32_t shift = bbs<kLimb>() & 3u;
            t <<= shift;
            t |= bbs<kLimb>() & ((1u << shift) - 1u);  // array_shift = {0, 1, 3, 7}
        }
        return t;
    }
    // `limb` is the same in every lane of the warp, so the branch never diverges.
    __device__ __forceinline__ uint32_t next() { return limb ? assemble<true>() : assemble<false>(); }
};

// The same source on the residues of the two factors (ci_crt.cuh), bound by
// the FMA-heavy pipe as the 62-bit form is, but with 30 instead of 51 cycles
// of it per squaring of a warp: 2^16 x 4096 outputs in 3.10 instead of 5.38
// ms, 300 uneven requests in one launch 4.46 instead of 6.88 ms.  Its constants are computed from
// the state's p and q when a warp's work starts, or read from `crt` (kCrtWords
// fields of P words, written by crt_store) where a call prepares them once for
// many units.  load() is false in every lane unless all lanes of the warp hold
// factors the residue form takes (all seeded ones do; imported moduli may have
// shorter factors, which keep the 62-bit form).
constexpr int kCrtWords = 4;  // mu_p, mu_q, beta (0: not usable), beta_s

// Lane l's residue constants: false (beta stored as 0) where the residue form
// does not apply.
__device__ __forceinline__ bool crt_store(const DevState &s, uint64_t l, uint32_t *crt) {
    CrtModulus C{};
    const bool ok = C.set(s.u32[F_P * s.P + l], s.u32[F_Q * s.P + l]);
    crt[l] = C.P.mu;
    crt[s.P + l] = C.Q.mu;
    crt[2 * s.P + l] = ok ? C.beta : 0u;
    crt[3 * s.P + l] = C.beta_s;
    return ok;
}
__device__ __forceinline__ bool crt_load(const DevState &s, uint64_t l, const uint32_t *crt, CrtModulus &C) {
    const uint32_t a = s.u32[F_P * s.P + l], b = s.u32[F_Q * s.P + l];
    C.P.set(min(a, b), crt[l]);
    C.Q.set(max(a, b), crt[s.P + l]);
    C.beta = crt[2 * s.P + l];
    C.beta_s = crt[3 * s.P + l];
    return C.beta != 0u;
}

struct SrcBbsCrt {
    static constexpr bool kHeavy = true, kOneStep = true;
    CrtModulus C;
    uint32_t rp, rq, sel;
    __device__ __forceinline__ bool load(const DevState &s, uint64_t l, const uint32_t *crt) {
        const bool ok = crt ? crt_load(s, l, crt, C) : C.set(s.u32[F_P * s.P + l], s.u32[F_Q * s.P + l]);
        if (!__all_sync(kFull, ok)) return false;
        const uint64_t y = s.u64[G_Y * s.P + l];
        rp = (uint32_t)(y % C.P.p);
        rq = (uint32_t)(y % C.Q.p);
        sel = s.u32[F_SEL * s.P + l];
        return true;
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const {
        s.u64[G_Y * s.P + l] = C.value(rp, rq);
    }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = (int)(sel & 7u);
        a2 = 8 + (int)((sel >> 8) & 7u);
    }
    // One BBS output: x <- x^2 mod M; the low word of x (its low bits are the secure ones).
    __device__ __forceinline__ uint32_t bbs() {
        rp = C.P.sqr(rp);
        rq = C.Q.sqr(rq);
        return C.low(rp, rq);
    }
    __device__ __forceinline__ uint32_t next() {
        uint32_t t = 0;
#pragma unroll
        for (int c = 0; c < 7; ++c) t = (t << 5) | (bbs() & 31u);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint32_t shift = bbs() & 3u;
            t <<= shift;
            t |= bbs() & ((1u << shift) - 1u);  // array_shift = {0, 1, 3, 7}
        }
        return t;
    }
};

// Shortest unit that takes the residue form when its constants have to be
// computed first (2^16 streams, written: 12 outputs 21.3 us against 23.1 in
// the 62-bit form, 16 outputs 25.2 against 29.2; 8 outputs 18.8 against 17.6).
constexpr uint64_t kCrtMinLength = 12;

// Algorithm 5 as printed: eight BBS generators per lane with moduli below
// 2^16, so x^2 fits 32 bits.  x^2 mod M by Barrett reduction with
// mu = floor(2^32 / M): q = mulhi(x^2, mu) is floor(x^2 / M) or one less, so a
// single conditional subtraction gives the canonical residue, taken as the
// unsigned minimum of r and r - M (r - M wraps above r when r < M), addition
// and minimum in one instruction.  The
// arrays are read from BBS1 and BBS2 when the call starts; at the end of the
// call generator k (state and modulus) is stored in place k + 1.
struct SrcBbs16 {
    static constexpr bool kHeavy = true, kOneStep = false;
    uint32_t y[8], nM[8], mu[8];  // nM = -M
    uint32_t sel1, sel2;
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            y[k] = s.u32[(F_Y16 + k) * s.P + l];
            const uint32_t M = s.u32[(F_M16 + k) * s.P + l];
            nM[k] = 0u - M;
            mu[k] = (uint32_t)((1ull << 32) / M);
        }
        sel1 = y[0] & 7u;
        sel2 = y[1] & 7u;
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            s.u32[(F_Y16 + (k + 1) % 8) * s.P + l] = y[k];
            s.u32[(F_M16 + (k + 1) % 8) * s.P + l] = 0u - nM[k];
        }
    }
    __device__ __forceinline__ void arrays(const DevState &, uint64_t, int &a1, int &a2) const {
        a1 = (int)sel1;
        a2 = 8 + (int)sel2;
    }
    template <int K>
    __device__ __forceinline__ uint32_t bbs() {  // BBS(K+1)
        const uint32_t a = y[K] * y[K];
        y[K] = addmin32(a + __umulhi(a, mu[K]) * nM[K], nM[K]);
        return y[K];
    }
    __device__ __forceinline__ uint32_t next() {
        // Four low bits of BBS1 .. BBS8 into bits 31-28 .. 3-0: each funnel
        // shift moves t down four bits and brings the next generator's low
        // nibble in at the top, so BBS8 enters first and BBS1 last (the eight
        // generators are independent, so the order of their steps is free).
        uint32_t t = bbs<7>() << 28;
        t = __funnelshift_r(t, bbs<6>(), 4);
        t = __funnelshift_r(t, bbs<5>(), 4);
        t = __funnelshift_r(t, bbs<4>(), 4);
        t = __funnelshift_r(t, bbs<3>(), 4);
        t = __funnelshift_r(t, bbs<2>(), 4);
        t = __funnelshift_r(t, bbs<1>(), 4);
        t = __funnelshift_r(t, bbs<0>(), 4);
        uint32_t shift = bbs<2>() & 3u;
        t <<= shift;
        t |= bbs<0>() & ((1u << shift) - 1u);  // array_shift = {0, 1, 3, 7}
        shift = bbs<6>() & 3u;
        t <<= shift;
        t |= bbs<1>() & ((1u << shift) - 1u);
        return t;
    }
};

// ----------------------------------------------------- generation loop
enum Sink { SINK_V4 = 0, SINK_SCALAR = 1, SINK_QC = 2, SINK_DIGEST = 3, SINK_NONE = 4 };  // NONE: the end state alone

// Multiplier of the per-stream output digest D <- D * K + x (mod 2^64),
// an odd 64-bit constant.
constexpr uint64_t kDigestMul = 0xD1342543DE82EF95ull;
// Its powers, for compile-time exponents.
__host__ __device__ constexpr uint64_t digest_power(int e) {
    uint64_t p = 1;
    for (int i = 0; i < e; ++i) p *= kDigestMul;
    return p;
}
// xor128's outputs join the digest sixteen at a time, each times its own power:
// in Horner's form a warp alone waited for the product of every step (16000 x
// 2000: 57 us, 45 so; 2^20 x 1024: 550, 531).  The other xor-likes are faster
// by Horner (xor64 16000 x 2000: 43 us, 58 in blocks).
constexpr int kDigestBlock = 16;

// One lane's stream while a warp advances its group: the strategy source, the
// CI state x, the slot (last strategy) and the two partner lanes.  step() is
// Algorithm 4/5's inner step, t = own ^ slot[o1] ^ slot[o2]; slot = t; x ^= t
// (Eq. Oplus), and returns the output x.
template <class Src>
struct Lane {
    Src src;
    uint32_t x, slot;
    int p1, p2;
    // The source is loaded already.
    __device__ __forceinline__ void load(const DevState &st, uint64_t l) {
        x = st.u32[F_X * st.P + l];
        slot = st.u32[F_SLOT * st.P + l];
        int a1, a2;
        src.arrays(st, l, a1, a2);
        p1 = st.table[a1 * 32 + (threadIdx.x & 31)];
        p2 = st.table[a2 * 32 + (threadIdx.x & 31)];
    }
    __device__ __forceinline__ uint32_t step() {
        const uint32_t own = src.next();
        const uint32_t s1 = __shfl_sync(kFull, slot, p1);
        const uint32_t s2 = __shfl_sync(kFull, slot, p2);
        slot = own ^ s1 ^ s2;
        x ^= slot;
        return x;
    }
    __device__ __forceinline__ void store(const DevState &st, uint64_t l) const {
        src.store(st, l);
        st.u32[F_X * st.P + l] = x;
        st.u32[F_SLOT * st.P + l] = slot;
    }
};

// Quarter-circle test of one output pair in 24-bit fixed point, as a miss:
// a = o0 >> 8, b = o1 >> 8, and the pair misses iff a^2 + b^2 >= 2^48, i.e.
// iff bit 16 of the high word of the (at most 49-bit) sum is set.  The two
// shifts and the bit test are written as high halves of products by 2^24 and
// 2^16, which keep them on the FMA pipe: the fused loop is otherwise bound by
// the integer ALU pipe (xor-like shifts, mixing XORs).  The multipliers sit in
// constant memory so that they stay multiplies.
static __constant__ uint32_t c_qc_mul[2] = {1u << 24, 1u << 16};
__device__ __forceinline__ uint32_t qc_miss(uint32_t o0, uint32_t o1) {
    const uint32_t a = __umulhi(o0, c_qc_mul[0]), b = __umulhi(o1, c_qc_mul[0]);
    const uint64_t s = (uint64_t)a * a + (uint64_t)b * b;
    return __umulhi((uint32_t)(s >> 32), c_qc_mul[1]);
}

// The same test by the high halves of o0^2 and o1^2, for blocks of pairs: with
// h = floor(o0^2 / 2^32) + floor(o1^2 / 2^32) and V = (a^2 + b^2) / 2^16 (miss
// iff V >= 2^32), h - 1024 < V < h + 2, since the low bytes that a and b leave
// out add less than 1024 and the two floors take less than 2.  So h >= 2^32 is
// the answer except for h in [2^32 - 1, 2^32 + 1023], one pair in 5 million;
// `near` keeps the smallest (h + 1) mod 2^32 of a block, at most kQcNear if any
// pair was that close, and the block is then run again by the exact test.  Two
// wide products, a carry and a minimum a pair instead of five wide products and
// an addition: the loop is bound by what its schedulers can dispatch (a cycle
// for a narrow multiply or an addition, two for an ALU operation or a wide
// multiply).  2^20 x 1024 xor128 outputs: 622 us by the exact test (23.3 cycles
// a step), 563 so; 605 with the two halves and 1 added in 64 bits and one
// three-way minimum for two pairs.
constexpr uint32_t kQcNear = 1024;
__device__ __forceinline__ void qc_miss_high(uint32_t o0, uint32_t o1, uint32_t &miss, uint32_t &near) {
    uint32_t h;
    asm("add.cc.u32 %0, %2, %3;\n\t"
        "addc.u32 %1, %1, 0;"
        : "=r"(h), "+r"(miss)
        : "r"(__umulhi(o0, o0)), "r"(__umulhi(o1, o1)));
    near = __viaddmin_u32(h, 1u, near);
}

// Launch-shape choices of the written sinks, picked by the autotuner:
// KT = outputs per stream staged per flush (tile depth: 32 or 64, i.e. 128- or
// 256-byte row segments), CACHE = store policy (0: streaming st.global.cs,
// evict-first; 1: default write-back st.global).
template <int KT_, int CACHE_>
struct TileCfg {
    static constexpr int KT = KT_;
    static constexpr int CH = KT_ / 4;  // 16-byte chunks per tile row
    static constexpr int CACHE = CACHE_;
    static constexpr bool kBrief = false;
};
using TileDefault = TileCfg<32, 0>;
// For warps that run a few tiles in a launch of some 10 us: the loops with the
// least code and staging, since their first fetch costs more than conflicts or a
// longer chain (32 x 8192 digested: 20.5 us, 21.6 with blocks of sixteen; 4096 x
// 2047 written 24.7, 26.7 with the forms of several strides in one kernel).
// PITCH: of written_lines.
template <int PITCH>
struct TileBrief : TileDefault {
    static constexpr bool kBrief = true;
    static constexpr int kPitch = PITCH;
};

// Index of word `col` of row `row` in a warp's 32 x KT staging tile: 16-byte
// chunks XOR-swizzled by row so that both the per-lane 16-byte row writes and
// the per-row reads are free of bank conflicts.
template <int KT>
__device__ __forceinline__ int tile_word(int row, int col) {
    return row * KT + ((((col >> 2) ^ (row & 7))) << 2) + (col & 3);
}

template <int CACHE>
__device__ __forceinline__ void store16(uint32_t *p, const uint4 &v) {
    if (CACHE == 0)
        __stcs(reinterpret_cast<uint4 *>(p), v);
    else
        *reinterpret_cast<uint4 *>(p) = v;
}

// Words [lo, hi) of the 16-byte chunk v at p (aligned): one store when the
// chunk is whole, else word by word.
template <int CACHE>
__device__ __forceinline__ void store_words(uint32_t *p, const uint4 &v, int lo, int hi) {
    if (lo <= 0 && hi >= 4) {
        store16<CACHE>(p, v);
    } else {
        if (lo <= 0 && hi > 0) p[0] = v.x;
        if (lo <= 1 && hi > 1) p[1] = v.y;
        if (lo <= 2 && hi > 2) p[2] = v.z;
        if (lo <= 3 && hi > 3) p[3] = v.w;
    }
}

// Rows of up to kPitch words with nothing between them (ld == n): the group's
// rows are one span of the output, staged at an odd pitch (32 banks a step) and
// stored as that span, 32 consecutive words per warp-wide store.
template <int kPitch, class Step>
__device__ __forceinline__ void written_short(Step step, uint64_t S, uint64_t row0, uint32_t n, uint32_t *out,
                                              uint4 *tile) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t *stage = reinterpret_cast<uint32_t *>(tile);
#pragma unroll 1
    for (uint32_t i = 0; i < n; ++i) stage[lane * kPitch + i] = step();
    __syncwarp();
    const uint32_t rows = S - row0 < 32 ? (uint32_t)(S - row0) : 32u, words = rows * n;
    const uint32_t dr = 32 / n, dc = 32 % n;
    uint32_t *dst = out + row0 * n;
    uint32_t r = lane / n, c = lane % n;
#pragma unroll 4
    for (uint32_t i = lane; i < words; i += 32) {
        dst[i] = stage[r * kPitch + c];
        r += dr;
        c += dc;
        if (c >= n) {
            c -= n;
            ++r;
        }
    }
    __syncwarp();
}

// Written rows of any alignment (out 4-byte aligned, any ld, col0 and n).  Row
// r starts ph_r = 0..31 words after a 128-byte line; its staging row starts at
// that line, so that everything but a row's first and last words leaves as
// whole lines, four rows' per warp-wide store.  (A line, or a 32-byte sector,
// written in two parts 32 steps apart costs its memory write twice: 400 MB in
// rows of 401 took 132 us by 16-byte, 108 by 32-byte boundaries.)  Output j of
// the call stands at word (j + ph_r) mod 64 of the row's two lines, of which one
// is stored after every 32 steps.  `step` makes the lane's next output; kUnroll
// of a tile's 32 steps are unrolled.
// (50001 x 1001 XORshift outputs: the word-wise form this replaces, a row per
// warp-wide store, issued 34 instructions per step of a warp, 20 of them for
// the stores, and took 82 us; now 52.)
// Banks: the lanes of one step write 32 different ones when ld is odd, 16 when
// it is 2 mod 4.  When ld is a multiple of 4 (in a buffer that is not 16-byte
// aligned) the rows' phases are equal mod 4: after up to three steps every row
// stands at a 16-byte word and four steps make one store of it, without
// conflicts at a pitch of 16 or 17 such words (ld / 4 odd or even).  Word by
// word, 2^18 x 256 from the second word of a buffer on took 269 us, and the
// older form 135.
// kPitch: 16-byte words between staging rows, 0 for 16 or 17 by ld; kQuads: ld
// is a multiple of 4.
constexpr int kTileVec = 32 * 17;  // 16-byte words of a warp's staging tile (the aligned 32 x 32 form: 256)
template <int kUnroll, int CACHE, int kPitch, bool kQuads, class Step>
__device__ __forceinline__ void written_lines(Step step, uint64_t S, uint64_t row0, uint64_t n, uint32_t *out,
                                              uint64_t ld, uint64_t col0, uint4 *tile) {
    const int lane = threadIdx.x & 31;
    // words of row r before its first output, up to the line below it
    auto phase = [&](uint64_t r) { return (int)((reinterpret_cast<uintptr_t>(out + r * ld + col0) >> 2) & 31u); };
    const int ph = phase(row0 + lane);  // the row this lane computes
    const int pitch = kPitch ? kPitch : ld % 8 == 0 ? 17 : 16;
    uint4 *mine = tile + lane * pitch;
    uint32_t *w = reinterpret_cast<uint32_t *>(mine) + ph;
    // the rows this lane stores: 4 k + lane / 8, 16-byte word c of their lines
    const int c = lane & 7;
    const uint4 *stored = tile + (lane >> 3) * pitch + c;
    const uint64_t row = row0 + (lane >> 3);
    const bool all_rows = row0 + 32 <= S;
    uint32_t *dst = out + row * ld + col0;  // output `at` of row `row`

    // stores line `half` / 32 of every staging row and goes on to the next
    int64_t at = 0;
    const int64_t len = (int64_t)n;
    int half = 0;
    auto flush = [&]() {
        __syncwarp();
        uint32_t *q = dst;
        const uint4 *from = stored + half / 4;
        if (at > 0 && at + 32 <= len && all_rows) {  // words of the rows only
#pragma unroll(kUnroll > 1 ? 8 : 2)
            for (int k = 0; k < 8; ++k, q += 4 * ld, from += 4 * pitch) {
                uint32_t *line = reinterpret_cast<uint32_t *>(reinterpret_cast<uintptr_t>(q) & ~(uintptr_t)127);
                store16<CACHE>(line + 4 * c, *from);
            }
        } else {
#pragma unroll 1
            for (int k = 0; k < 8; ++k, q += 4 * ld, from += 4 * pitch) {
                const uintptr_t a = reinterpret_cast<uintptr_t>(q);
                const int p = (int)((a >> 2) & 31u);
                uint32_t *line = reinterpret_cast<uint32_t *>(a & ~(uintptr_t)127);
                // words [lo, hi) of this 16-byte word belong to the row
                const int64_t hi = len - at + p - 4 * c;
                if (row + 4 * k < S)
                    store_words<CACHE>(line + 4 * c, *from, at == 0 ? p - 4 * c : 0, hi > 4 ? 4 : (int)hi);
            }
        }
        dst += 32;
        at += 32;
        half ^= 32;
        __syncwarp();
    };
    // word (ph + j + half) mod 64 of the lane's row, ph + j < 64
    auto place = [&](int j) { return j + ph < 32 ? w + half + j : w - half + j; };
    int head = 0;  // outputs up to the first 16-byte word, the same in every lane
    if constexpr (kQuads) {
        head = -ph & 3;
        if (head > len) head = (int)len;
        for (int j = 0; j < head; ++j) w[j] = step();
        const int first = (ph + head) / 4;
        while (at + head + 32 <= len) {
#pragma unroll(kUnroll / 4)
            for (int q = 0; q < 8; ++q) {
                uint4 v;
                v.x = step();
                v.y = step();
                v.z = step();
                v.w = step();
                mine[(first + half / 4 + q) & 15] = v;
            }
            flush();
        }
    } else {
        while (at + 32 <= len) {
            if (kUnroll < 32) {
#pragma unroll(kUnroll)
                for (int j = 0; j < 32; ++j) *place(j) = step();
            } else if (half == 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) w[j] = step();
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) *place(j) = step();
            }
            flush();
        }
    }
    // the rest: up to 31 steps behind the words kept from the last tile (and the
    // head), at most 63 words of a row
    const int rest = (int)(len - at);
    for (int j = head; j < rest; ++j) *place(j) = step();
    if (__any_sync(kFull, rest + ph > 0)) flush();
    if (__any_sync(kFull, rest + ph > 32)) flush();
}

template <int kUnroll, int CACHE, class Step>
__device__ __forceinline__ void written_unaligned(Step step, uint64_t S, uint64_t row0, uint64_t n, uint32_t *out,
                                                  uint64_t ld, uint64_t col0, uint4 *tile) {
    constexpr bool kLong = kUnroll == 1;  // a step takes far longer than its store: the least code and staging
    constexpr int kShort = kLong ? 63 : 65;
    if (n <= kShort && ld == n) {
        written_short<kShort>(step, S, row0, (uint32_t)n, out, tile);
    } else if constexpr (kLong) {
        written_lines<kUnroll, CACHE, 16, false>(step, S, row0, n, out, ld, col0, tile);
    } else {
        if (ld % 4 == 0)
            written_lines<kUnroll, CACHE, 0, true>(step, S, row0, n, out, ld, col0, tile);
        else
            written_lines<kUnroll, CACHE, 16, false>(step, S, row0, n, out, ld, col0, tile);
    }
}
template <class Src>  // of a source's unaligned rows
constexpr int kScalarTile = Src::kHeavy ? 32 * 16 : kTileVec;

// Runs n steps of a loaded lane into the sink; returns the lane's
// quarter-circle hits or the Horner digest of these outputs (0 for the others).
// Written outputs go to out[r * ld + col0 + i], rows r = row0 + lane < S.
template <class Src, int SINK, class TC>
__device__ __forceinline__ uint64_t warp_run(Lane<Src> &s, uint64_t S, uint64_t row0, uint64_t n, uint32_t *out,
                                             uint64_t ld, uint64_t col0, uint4 *tile) {
    constexpr int KT = (SINK == SINK_V4 || SINK == SINK_SCALAR) ? TC::KT : 32;
    constexpr int CH = KT / 4;
    const int lane = threadIdx.x & 31;
    if constexpr (SINK == SINK_SCALAR) {
        auto step = [&]() { return s.step(); };
        if constexpr (TC::kBrief)
            written_lines<32, TC::CACHE, TC::kPitch, false>(step, S, row0, n, out, ld, col0, tile);
        else
            written_unaligned<Src::kHeavy ? 1 : 32, TC::CACHE>(step, S, row0, n, out, ld, col0, tile);
        return 0;
    }
    const uint64_t nfull = n - n % KT;
    uint32_t *tw = reinterpret_cast<uint32_t *>(tile);
    uint64_t hits = 0;

    for (uint64_t i0 = 0; i0 < nfull; i0 += KT) {
        if (SINK == SINK_NONE) {
#pragma unroll(Src::kHeavy ? 1 : 32)
            for (int k = 0; k < 32; ++k) s.step();
        } else if (SINK == SINK_DIGEST) {
            constexpr int kBlock = std::is_same<Src, SrcXor128>::value && !TC::kBrief ? kDigestBlock : 1;
#pragma unroll(Src::kHeavy ? 1 : 32)
            for (int k = 0; k < 32; k += kBlock) {
                uint32_t o[kBlock];
#pragma unroll
                for (int j = 0; j < kBlock; ++j) o[j] = s.step();
                hits *= digest_power(kBlock);
#pragma unroll
                for (int j = 0; j < kBlock; ++j) hits += o[j] * digest_power(kBlock - 1 - j);
            }
        } else if (SINK == SINK_QC) {
            uint32_t m = 0, near = ~0u;
            const Lane<Src> before = s;
            if (!Src::kHeavy) {
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const uint32_t o0 = s.step();
                    const uint32_t o1 = s.step();
                    qc_miss_high(o0, o1, m, near);
                }
            }
            if (Src::kHeavy || __any_sync(kFull, near <= kQcNear)) {
                s = before;
                m = 0;
#pragma unroll 1
                for (int k = 0; k < 16; ++k) {
                    const uint32_t o0 = s.step();
                    const uint32_t o1 = s.step();
                    m += qc_miss(o0, o1);
                }
            }
            hits += 16u - m;
        } else {
            if (Src::kOneStep) {
#pragma unroll 1
                for (int k = 0; k < KT; ++k) tw[tile_word<KT>(lane, k)] = s.step();
            } else {
#pragma unroll(Src::kHeavy ? 1 : CH)
                for (int q = 0; q < CH; ++q) {
                    uint4 v;
                    v.x = s.step();
                    v.y = s.step();
                    v.z = s.step();
                    v.w = s.step();
                    tile[lane * CH + (q ^ (lane & 7))] = v;
                }
            }
            __syncwarp();
            constexpr int RPI = 32 / CH;  // tile rows per warp-wide store
#pragma unroll(Src::kOneStep ? 2 : CH)
            for (int k = 0; k < CH; ++k) {
                const int r = RPI * k + lane / CH, c = lane % CH;
                const uint4 v = tile[r * CH + (c ^ (r & 7))];
                if (row0 + r < S) store16<TC::CACHE>(out + (row0 + r) * ld + col0 + i0 + 4 * c, v);
            }
            __syncwarp();
        }
    }

    const int rem = (int)(n - nfull);
    if (rem) {
        if (SINK == SINK_NONE) {
            for (int k = 0; k < rem; ++k) s.step();
        } else if (SINK == SINK_DIGEST) {
            for (int k = 0; k < rem; ++k) hits = hits * kDigestMul + s.step();
        } else if (SINK == SINK_QC) {
            uint32_t m = 0;
            for (int k = 0; k < rem / 2; ++k) {
                const uint32_t o0 = s.step();
                const uint32_t o1 = s.step();
                m += qc_miss(o0, o1);
            }
            hits += (uint32_t)(rem / 2) - m;
        } else {
            for (int k = 0; k < rem; ++k) tw[tile_word<KT>(lane, k)] = s.step();
            __syncwarp();
            constexpr int RPI = 32 / CH;
#pragma unroll 2
            for (int k = 0; k < CH; ++k) {
                const int r = RPI * k + lane / CH, c = lane % CH;
                if (row0 + r < S)
                    store_words<TC::CACHE>(out + (row0 + r) * ld + col0 + nfull + 4 * c, tile[r * CH + (c ^ (r & 7))],
                                           -4 * c, rem - 4 * c);
            }
            __syncwarp();
        }
    }

    return hits;
}

template <class Src, int SINK, class TC>
__device__ __forceinline__ void warp_loop(Lane<Src> &s, const DevState &st, uint64_t g, uint64_t n, uint32_t *out,
                                          uint64_t ld, uint64_t col0, uint64_t *counts, uint4 *tile) {
    const uint64_t l = g * 32 + (threadIdx.x & 31);
    s.load(st, l);
    const uint64_t hits = warp_run<Src, SINK, TC>(s, st.S, g * 32, n, out, ld, col0, tile);
    s.store(st, l);
    if (SINK == SINK_QC && l < st.S) counts[l] += hits;
    if (SINK == SINK_DIGEST && l < st.S) counts[l] = hits;
}


template <class Src, int SINK, class TC = TileDefault>
__device__ __forceinline__ void warp_task(const DevState &st, uint64_t g, uint64_t n, uint32_t *out,
                                          uint64_t ld, uint64_t col0, uint64_t *counts,
                                          uint4 *tile, const uint32_t *crt = nullptr) {
    CI_WARP_CHECK(st, g < st.P / 32, CHK_GROUP, g);
    if (SINK == SINK_V4 || SINK == SINK_SCALAR) CI_WARP_CHECK(st, col0 + n <= ld, CHK_COLS, col0 + n);
    if (SINK == SINK_V4) CI_WARP_CHECK(st, (col0 | ld) % 4 == 0, CHK_V4_ALIGN, col0);
    const uint64_t l = g * 32 + (threadIdx.x & 31);
    if constexpr (std::is_same<Src, SrcBbs>::value) {
        if (crt || n >= kCrtMinLength) {
            Lane<SrcBbsCrt> c;
            if (c.src.load(st, l, crt)) {  // the same in every lane
                warp_loop<SrcBbsCrt, SINK, TC>(c, st, g, n, out, ld, col0, counts, tile);
                return;
            }
        }
    }
    Lane<Src> s;
    s.src.load(st, l);
    warp_loop<Src, SINK, TC>(s, st, g, n, out, ld, col0, counts, tile);
}

// ------------------------------------------------ TMA bulk tensor stores
// A warp's 32 x 32 staging tile leaves as ONE cp.async.bulk.tensor store: the
// tile's layout (16-byte chunk c of row r at chunk position c ^ (r % 8), tile
// base 1024-byte aligned) is the TMA 128-byte swizzle, so the tensor map uses
// CU_TENSOR_MAP_SWIZZLE_128B over the output [rows][cols] with a 32 x 32 box.
// The store carries an L2 evict-first policy (outputs are streamed out, as the
// 16-byte path's st.global.cs does).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void tma_store_tile(const CUtensorMap *map, const void *smem, int x, int y,
                                               uint64_t policy) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%1, %2}], [%3], %4;"
                 :
                 : "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(s), "l"(policy)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Wait until at most kLeft committed stores still read their shared-memory source.
template <int kLeft>
__device__ __forceinline__ void tma_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kLeft) : "memory");
}
// Make this thread's ordinary shared-memory writes visible to the TMA unit.
__device__ __forceinline__ void fence_smem_to_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Written sink through TMA: per 32-iteration tile, the lanes fill one of
// kTmaTiles 4 KB tiles in turn (refilled only after the store issued from it
// has read it), then lane 0 issues the tile's bulk
// tensor store at (column i0, row 32 g).  The TMA unit clips rows past the
// tensor's row count (streams >= S) and, in a last tile of fewer than 32
// iterations, columns past n.  `tiles` is kTmaTiles x 4 KB, 1024-byte aligned.
// Requires out 16-byte aligned and n % 4 == 0 (checked by the host when it
// builds the tensor map).
// Tiles per warp.  A third one covers the time a store waits behind the others
// of a busy memory: 100000 x 1500 xor64 188 us with two, 162 with three, 156
// with four; 2^20 x 256 xor128 176 / 173 / 175, xor64 189 / 193 / 199 (fewer
// warps beside the tiles).
constexpr int kTmaTiles = 3;
template <class Src>
__device__ __forceinline__ void warp_task_tma(const DevState &st, uint64_t g, uint64_t n, const CUtensorMap *map,
                                              uint4 *tiles) {
    CI_WARP_CHECK(st, g < st.P / 32, CHK_GROUP, g);
    CI_WARP_CHECK(st, n % 4 == 0, CHK_TMA_ALIGN, n);
    const int lane = threadIdx.x & 31;
    const uint64_t l = g * 32 + lane;
    Lane<Src> s;
    s.src.load(st, l);
    s.load(st, l);
    const uint64_t policy = l2_evict_first_policy();
    int k = 0;
    for (uint64_t i0 = 0; i0 < n; i0 += 32, ++k) {
        uint4 *tile = tiles + k % kTmaTiles * 256;
        if (k >= kTmaTiles) {
            if (lane == 0) tma_wait_read<kTmaTiles - 1>();
            __syncwarp();
        }
        auto chunk = [&](int q) {
            uint4 v;
            v.x = s.step();
            v.y = s.step();
            v.z = s.step();
            v.w = s.step();
            tile[lane * 8 + (q ^ (lane & 7))] = v;
        };
        if (n - i0 >= 32) {
#pragma unroll
            for (int q = 0; q < 8; ++q) chunk(q);
        } else {
            const int chunks = (int)(n - i0) / 4;
            for (int q = 0; q < chunks; ++q) chunk(q);
        }
        fence_smem_to_async();
        __syncwarp();
        if (lane == 0) tma_store_tile(map, tile, (int)i0, (int)(g * 32), policy);
    }
    s.store(st, l);
    if (lane == 0) tma_wait_read<0>();  // every store has read its tile before the block exits
    __syncwarp();
}

// Written sink of short rows through one bulk store per warp group: the
// group's 32 rows of n words (ld == n) are one contiguous span of the output,
// staged whole, in order, in `stage` (128 n bytes) and stored by a single
// cp.async.bulk.  Whole lines leave whatever n is, where 128-byte pieces of
// rows that start anywhere cost two partial lines each: 10^6 x 100 written
// 70 us, by TMA tiles 117 (160 before those clipped the last tile).  Requires out 16-byte
// aligned (the span then is); the last group of a ragged state, whose span may
// end anywhere, leaves through ordinary stores.
template <class Src>
__device__ __forceinline__ void warp_task_span(const DevState &st, uint64_t g, uint32_t n, uint32_t *out,
                                               uint32_t *stage) {
    CI_WARP_CHECK(st, g < st.P / 32, CHK_GROUP, g);
    const int lane = threadIdx.x & 31;
    const uint64_t l = g * 32 + lane;
    Lane<Src> s;
    s.src.load(st, l);
    s.load(st, l);
    uint32_t *w = stage + lane * n;
    auto run = [&](auto width) {  // steps `width` words at a time; n is a multiple of it
        constexpr int N = decltype(width)::value;
        auto put = [&](uint32_t *p) {
            uint32_t v[N];
#pragma unroll
            for (int j = 0; j < N; ++j) v[j] = s.step();
            if constexpr (N == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(v[0], v[1], v[2], v[3]);
            if constexpr (N == 2) *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
            if constexpr (N == 1) *p = v[0];
        };
        uint32_t i = 0;
        for (; i + 16 <= n; i += 16)
#pragma unroll
            for (int j = 0; j < 16; j += N) put(w + i + j);
        for (; i < n; i += N) put(w + i);
    };
    if (n % 4 == 0)
        run(std::integral_constant<int, 4>());
    else if (n % 2 == 0)
        run(std::integral_constant<int, 2>());
    else
        run(std::integral_constant<int, 1>());
    uint32_t *dst = out + g * 32 * n;
    if (g * 32 + 32 <= st.S) {
        fence_smem_to_async();
        __syncwarp();
        if (lane == 0) {
            const uint32_t s = (uint32_t)__cvta_generic_to_shared(stage);
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;"
                         :
                         : "l"(dst), "r"(s), "r"(128u * n), "l"(l2_evict_first_policy())
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    } else {
        __syncwarp();
        const uint32_t words = (uint32_t)(st.S - g * 32) * n;
        for (uint32_t i = lane; i < words; i += 32) dst[i] = stage[i];
    }
    s.store(st, l);
    if (lane == 0) tma_wait_read<0>();  // the store has read the stage before the block exits
    __syncwarp();
}

}  // namespace dev
}  // namespace ci
