// ci_bg.cu -- the chaotic Blum-Goldwasser cryptosystem of Sec. 9.2 on the
// device (include/ci_prng.h: ci_bg_encrypt, ci_bg_decrypt).
//
// Per message: x_0 = r^2 mod N, b_i = the w low bits of x_i
// (w = floor(log2 floor(log2 N))), x_{i+1} = x_i^2 mod N.  The keystream is
// Eq. (Oplus) run on the b_i from S^0: k_i = S^0 ^ b_0 ^ ... ^ b_i, and
// chunk i of the ciphertext is c_i = m_i ^ k_i; the ciphertext carries
// y = x_L.  Decryption recovers x_0 from y with the factors p, q = 3 mod 4
// (square roots by the exponent ((p + 1) / 4)^L, joined by Garner's CRT) and
// regenerates the same keystream.
//
// One lane owns one message; a warp owns 32 consecutive messages.  When the
// chunk count is a multiple of 32 and both buffers are 16-byte aligned, each
// lane moves its own 32 chunks per step with two 16-byte loads and stores.
// Otherwise the warp moves its messages' chunks (one byte each,
// message-major) through a warp-private 32 x 32 byte tile in shared memory,
// so global loads and stores are 32-byte rows while each lane walks its own
// row.  The squarings use the Barrett reduction of the BBS strategy source
// (modulus odd, below 2^62), which keeps x_i canonical so its low bits are
// read directly; a warp whose moduli all have at least 34 bits takes its
// limb form.  Decryption knows the factors: a warp whose factors all lie in
// (2^30, 2^31) squares their residues instead (ci_crt.cuh), starting from the
// two square roots, and never forms x_0 (2^18 x 1024: 334 us against 578 in
// the 62-bit form).
#include <cuda_runtime.h>


#include "ci_crt.cuh"
#include "ci_device.cuh"
#include "ci_gen.cuh"
#include "ci_internal.h"
#include "ci_modarith.cuh"
#include "ci_trace.h"

namespace ci {
namespace {

using namespace dev;

// Resident blocks per SM asked of the register allocator: 64 registers, no
// spills (2^18 x 1024: decryption 365 us, 375 with 5 blocks, 379 with 3;
// encryption 437, 447 and 457; blocks in order, gen_grid, took another 23 us
// off each).
constexpr int kBgMinBlocks = 4;

constexpr int kBgWarps = 8;    // warps per block
constexpr int kBgTile = 32;    // chunks per staged row
constexpr int kBgRowPad = 36;  // bytes per staged row: 9 words, so the 32 lanes'
                               // word reads of their own rows hit 32 banks

__device__ __forceinline__ uint32_t bg_w(uint64_t N) {
    const uint32_t lg = 63u - (uint32_t)__clzll((long long)N);  // floor(log2 N), N >= 2
    return lg ? 31u - (uint32_t)__clz((int)lg) : 0u;             // floor(log2 lg)
}

// The keystream of one message: draw() returns b = x_i & mask (x_i canonical)
// and takes x_{i+1} = x_i^2.  One form per way of squaring.
template <bool kLimb>  // 62-bit Barrett; kLimb: every modulus of the warp has 34..62 bits
struct BgBarrett {
    Barrett62 B;
    uint64_t x;
    uint32_t mask, key;
    __device__ __forceinline__ uint32_t draw() {
        const uint32_t b = (uint32_t)x & mask;
        x = kLimb ? B.sqr_limb(x) : B.sqr(x);
        return b;
    }
};
struct BgCrt {  // both factors known, in (2^30, 2^31)
    CrtModulus C;
    uint32_t rp, rq, mask, key;
    __device__ __forceinline__ uint32_t draw() {
        const uint32_t b = C.low(rp, rq) & mask;
        rp = C.P.sqr(rp);
        rq = C.Q.sqr(rq);
        return b;
    }
};

// One chunk: key ^= b, c = m ^ key.
template <class Lane>
__device__ __forceinline__ uint32_t bg_chunk(Lane &s, uint32_t v) {
    s.key ^= s.draw();
    return (v ^ s.key) & 0xFFu;
}
// Four chunks, one per byte of w: the keystream bytes are gathered into one
// word and XORed in once (key < 2^8: S^0 is a byte, the b_i have at most 5
// bits).
template <class Lane>
__device__ __forceinline__ uint32_t bg_word(Lane &s, uint32_t w) {
    uint32_t ks = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        s.key ^= s.draw();
        ks |= s.key << (8 * b);
    }
    return w ^ ks;
}

// Encryption key check: N odd, 3 <= N < 2^62 (the range of Barrett62).
__device__ __forceinline__ bool bg_setup_encrypt(uint64_t N, uint64_t r, Barrett62 &B, uint64_t &x) {
    const bool ok = (N & 1ull) && N >= 3 && N < (1ull << 62);
    if (!ok) N = 3;
    B.set(N, barrett_mu(N));
    x = B.sqr(r % N);  // x_0 = r^2 mod N
    return ok;
}

// ((p + 1) / 4)^L mod (p - 1) for p = 3 mod 4 and L >= 1.  p - 1 = 2 m with m
// odd: the power mod m (Montgomery), and its parity, that of (p + 1) / 4, from
// which the residue mod 2 m follows.
template <bool k31>
__device__ __forceinline__ uint32_t root_exponent(uint32_t p, uint64_t L) {
    const uint32_t m = (p - 1) / 2, h = (uint32_t)(((uint64_t)p + 1) / 4);  // h = (m + 1) / 2 <= m
    if (m == 1) return 1;
    const Mont<k31> M(m);
    const uint32_t e = M.from(M.pow_m(M.to(h), L));
    return ((e ^ h) & 1u) ? e + m : e;
}

// Decryption key check: p != q, both prime, = 3 mod 4, below 2^32, p q < 2^62.
// The residues of x_0, the square root of y taken L times mod p and mod q,
// and p^-1 mod q for joining them (Garner: x_0 = r_p + p ((r_q - r_p) p^-1
// mod q)); p < q on return.  A rejected key becomes a valid dummy pair.
struct BgRoots {
    uint32_t p, q, rp, rq, pinv;
};
template <bool k31>  // k31: every factor of the warp is below 2^31
__device__ __forceinline__ bool bg_setup_decrypt(uint64_t a, uint64_t b, uint64_t y, uint64_t L, BgRoots &s) {
    const uint64_t p = a < b ? a : b, q = a < b ? b : a;
    const bool ok = q < (1ull << 32) && (p & 3ull) == 3 && (q & 3ull) == 3 && p != q && p * q < (1ull << 62) &&
                    is_prime_u32<k31>(p) && is_prime_u32<k31>(q);
    s = BgRoots{(1u << 30) + 3u, (1u << 31) - 1u, 0u, 0u, 1u};
    if (ok) {
        const Mont<k31> Mp((uint32_t)p), Mq((uint32_t)q);
        const uint32_t ep = root_exponent<k31>((uint32_t)p, L), eq = root_exponent<k31>((uint32_t)q, L);
        // y mod N < p q, below p 2^32 and q 2^32: taken to Montgomery form by REDC
        const uint64_t yN = y < p * q ? y : y % (p * q);
        s.p = (uint32_t)p;
        s.q = (uint32_t)q;
        s.rp = Mp.from(Mp.pow_m(Mp.to_wide(yN), ep));
        s.rq = Mq.from(Mq.pow_m(Mq.to_wide(yN), eq));
        s.pinv = Mq.from(Mq.pow_m(Mq.to((uint32_t)p), q - 2));  // Fermat: p^(q-2) = p^-1 mod q
    }
    return ok;
}

// The chunks of one warp's 32 messages (lane = message), after key setup.
template <bool kVec, class Lane>
__device__ __forceinline__ void bg_rows(Lane &s, uint32_t keep, bool live, uint64_t msg, uint64_t m0,
                                        uint32_t rows, uint64_t L, const uint8_t *in, uint8_t *out, uint8_t *tile,
                                        uint8_t *row, uint32_t lane) {
    if constexpr (kVec) {  // L a multiple of 32, rows 16-byte aligned
        if (live) {
            const uint4 *src = reinterpret_cast<const uint4 *>(in + msg * L);
            uint4 *dst = reinterpret_cast<uint4 *>(out + msg * L);
            const uint64_t steps = L / kBgTile;
            for (uint64_t t = 0; t < steps; ++t) {  // each step reads its 32 bytes before writing them
                uint4 a = src[2 * t], b = src[2 * t + 1];
                a.x = bg_word(s, a.x) & keep;
                a.y = bg_word(s, a.y) & keep;
                a.z = bg_word(s, a.z) & keep;
                a.w = bg_word(s, a.w) & keep;
                b.x = bg_word(s, b.x) & keep;
                b.y = bg_word(s, b.y) & keep;
                b.z = bg_word(s, b.z) & keep;
                b.w = bg_word(s, b.w) & keep;
                dst[2 * t] = a;
                dst[2 * t + 1] = b;
            }
        }
    } else {
        for (uint64_t k0 = 0; k0 < L; k0 += kBgTile) {
            const uint32_t width = L - k0 < (uint64_t)kBgTile ? (uint32_t)(L - k0) : (uint32_t)kBgTile;
            __syncwarp();
#pragma unroll 8
            for (uint32_t r = 0; r < rows; ++r)
                if (lane < width) tile[r * kBgRowPad + lane] = in[(m0 + r) * L + k0 + lane];
            __syncwarp();
            if (live) {
                uint32_t *w = reinterpret_cast<uint32_t *>(row);
                if (width == kBgTile) {
#pragma unroll
                    for (int j = 0; j < kBgTile / 4; ++j) w[j] = bg_word(s, w[j]) & keep;
                } else {
                    for (uint32_t j = 0; j < width; ++j) row[j] = (uint8_t)(bg_chunk(s, row[j]) & keep);
                }
            }
            __syncwarp();
#pragma unroll 8
            for (uint32_t r = 0; r < rows; ++r)
                if (lane < width) out[(m0 + r) * L + k0 + lane] = tile[r * kBgRowPad + lane];
        }
    }
}

template <bool kDecrypt, bool kVec>
__global__ void __launch_bounds__(kBgWarps * 32, kBgMinBlocks)
    k_bg(uint64_t n_msgs, uint64_t L, const uint64_t *__restrict__ key_a, const uint64_t *__restrict__ key_b,
         const uint8_t *__restrict__ S0, const uint64_t *__restrict__ y_in, const uint8_t *in, uint8_t *out,
         uint64_t *__restrict__ y_out, uint32_t *__restrict__ n_rejected, uint32_t in_order) {
    __shared__ __align__(16) uint8_t stage[kBgWarps][32 * kBgRowPad];
    const uint32_t lane = threadIdx.x & 31u;
    uint8_t *tile = stage[threadIdx.x >> 5];
    uint8_t *row = tile + lane * kBgRowPad;
    const uint64_t g = warp_group(in_order);  // at most one group a warp (gen_grid)
    if (g < (n_msgs + 31) / 32) {
        const uint64_t m0 = g * 32;
        const uint64_t msg = m0 + lane;
        const bool live = msg < n_msgs;
        const uint32_t rows = n_msgs - m0 < 32 ? (uint32_t)(n_msgs - m0) : 32u;
        uint32_t key = 0, mask = 0;
        Barrett62 B;
        uint64_t x = 0;
        bool ok = false;
        if constexpr (kDecrypt) {
            BgRoots k{(1u << 30) + 3u, (1u << 31) - 1u, 0u, 0u, 1u};  // dead lanes: the dummy pair
            const uint64_t fa = live ? key_a[msg] : 3, fb = live ? key_b[msg] : 3;
            const bool short31 = __all_sync(0xFFFFFFFFu, fa < (1ull << 31) && fb < (1ull << 31));
            if (live)
                ok = short31 ? bg_setup_decrypt<true>(fa, fb, y_in[msg], L, k)
                             : bg_setup_decrypt<false>(fa, fb, y_in[msg], L, k);
            if (live) key = S0[msg];
            if (live && !ok && n_rejected) atomicAdd(n_rejected, 1u);
            const uint32_t keep = ok ? 0xFFFFFFFFu : 0u;  // a rejected key's row is written as zeros
            mask = ok ? (1u << bg_w((uint64_t)k.p * k.q)) - 1u : 0u;
            // the same in every lane: the branches never diverge
            if (__all_sync(0xFFFFFFFFu, k.p > (1u << 30) && k.q < (1u << 31))) {
                BgCrt s;
                s.C.set_inverse(k.p, k.q, k.pinv);
                s.rp = k.rp;
                s.rq = k.rq;
                s.mask = mask;
                s.key = key;
                bg_rows<kVec>(s, keep, live, msg, m0, rows, L, in, out, tile, row, lane);
                return;
            }
            // x_0 by Garner; p < q, so r_p < q
            const Mont32 Mq(k.q);
            const uint32_t diff = k.rq >= k.rp ? k.rq - k.rp : k.rq + (k.q - k.rp);
            x = k.rp + (uint64_t)k.p * Mq.mul(Mq.to(diff), k.pinv);  // < p + p (q - 1) = N
            B.set((uint64_t)k.p * k.q, barrett_mu((uint64_t)k.p * k.q));
        } else {
            B.set(3, barrett_mu(3));
            if (live) {
                ok = bg_setup_encrypt(key_a[msg], key_b[msg], B, x);
                mask = ok ? (1u << bg_w(B.M)) - 1u : 0u;
                key = S0[msg];
                if (!ok && n_rejected) atomicAdd(n_rejected, 1u);
            }
        }
        const uint32_t keep = ok ? 0xFFFFFFFFu : 0u;
        if (__all_sync(0xFFFFFFFFu, !live || B.M >= (1ull << 33))) {
            BgBarrett<true> s{B, x, mask, key};
            bg_rows<kVec>(s, keep, live, msg, m0, rows, L, in, out, tile, row, lane);
            x = s.x;
        } else {
            BgBarrett<false> s{B, x, mask, key};
            bg_rows<kVec>(s, keep, live, msg, m0, rows, L, in, out, tile, row, lane);
            x = s.x;
        }
        if (!kDecrypt && live) y_out[msg] = ok ? x : 0ull;
    }
}

ci_status bg_check(uint64_t n_msgs, uint64_t n_chunks, const void *a, const void *b, const void *S0,
                   const void *y, const void *in, const void *out) {
    if (!a || !b || !S0 || !y) return fail(CI_E_INVAL, "bg: key, S0 and y arrays must be non-null");
    if (n_chunks && (!in || !out)) return fail(CI_E_INVAL, "bg: message and ciphertext must be non-null");
    if (n_chunks > ~0ull / n_msgs) return fail(CI_E_INVAL, "bg: n_msgs * n_chunks overflows");
    return CI_OK;
}

// The per-lane 16-byte path: whole 32-chunk steps and 16-byte aligned rows.
bool bg_vec(uint64_t n_chunks, const void *in, const void *out) {
    return n_chunks % kBgTile == 0 && (reinterpret_cast<uintptr_t>(in) & 15u) == 0 &&
           (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
}

template <bool kDecrypt>
cudaError_t bg_launch(uint64_t n_msgs, uint64_t L, const uint64_t *a, const uint64_t *b, const uint8_t *S0,
                      const uint64_t *y_in, const uint8_t *in, uint8_t *out, uint64_t *y_out, uint32_t *n_rejected,
                      cudaStream_t stream) {
    const bool vec = bg_vec(L, in, out);
    auto kern = vec ? k_bg<kDecrypt, true> : k_bg<kDecrypt, false>;
    static const int per_sm[2] = {resident_blocks_per_sm(k_bg<kDecrypt, false>, kBgWarps * 32, 0),
                                  resident_blocks_per_sm(k_bg<kDecrypt, true>, kBgWarps * 32, 0)};
    // a wave is always spread (22704 x 391 encryption: 51.6 us, 53.3 in one-warp blocks)
    const GenGrid gg = gen_grid((n_msgs + 31) / 32, kBgWarps, (uint64_t)sm_count() * per_sm[vec], 0);
    kern<<<gg.grid, gg.warps * 32, 0, stream>>>(n_msgs, L, a, b, S0, y_in, in, out, y_out, n_rejected, gg.in_order);
    return cudaGetLastError();
}

}  // namespace
}  // namespace ci

extern "C" {

ci_status ci_bg_encrypt(uint64_t n_msgs, uint64_t n_chunks, const uint64_t *N_dev, const uint8_t *S0_dev,
                        const uint64_t *r_dev, const uint8_t *msg_dev, uint8_t *cipher_dev, uint64_t *y_dev,
                        uint32_t *n_rejected_dev, void *cuda_stream) {
    ci::TraceRange trace("bg encrypt");
    using namespace ci;
    if (n_msgs == 0) return CI_OK;
    const ci_status st = bg_check(n_msgs, n_chunks, N_dev, r_dev, S0_dev, y_dev, msg_dev, cipher_dev);
    if (st != CI_OK) return st;
    const cudaError_t e = bg_launch<false>(n_msgs, n_chunks, N_dev, r_dev, S0_dev, nullptr, msg_dev, cipher_dev, y_dev,
                                           n_rejected_dev, (cudaStream_t)cuda_stream);
    return e == cudaSuccess ? CI_OK : cuda_fail(e, "ci_bg_encrypt launch");
}

ci_status ci_bg_decrypt(uint64_t n_msgs, uint64_t n_chunks, const uint64_t *p_dev, const uint64_t *q_dev,
                        const uint8_t *S0_dev, const uint64_t *y_dev, const uint8_t *cipher_dev, uint8_t *msg_dev,
                        uint32_t *n_rejected_dev, void *cuda_stream) {
    ci::TraceRange trace("bg decrypt");
    using namespace ci;
    if (n_msgs == 0 || n_chunks == 0) return CI_OK;
    const ci_status st = bg_check(n_msgs, n_chunks, p_dev, q_dev, S0_dev, y_dev, cipher_dev, msg_dev);
    if (st != CI_OK) return st;
    const cudaError_t e = bg_launch<true>(n_msgs, n_chunks, p_dev, q_dev, S0_dev, y_dev, cipher_dev, msg_dev, nullptr,
                                          n_rejected_dev, (cudaStream_t)cuda_stream);
    return e == cudaSuccess ? CI_OK : cuda_fail(e, "ci_bg_decrypt launch");
}

}  // extern "C"
