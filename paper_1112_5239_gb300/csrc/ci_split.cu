// ci_split.cu -- time-parallel generation of long streams by jump-ahead
// (include/ci_prng.h: ci_generate_split).  Not a construct of the paper: it
// cuts one call of n iterations into K segments of `len` iterations that run
// at the same time, with results identical to the sequential call.
//
// Why it is exact.  Per warp, the own words o(i) of the strategy sources do
// not depend on the mixing state, and the mixing is GF(2)-linear on the
// lanes: with s the vector of the 32 lanes' slots and P the 32 x 32 matrix
// whose row l has ones at the partners o1(l), o2(l) (Algorithm 4/5),
//   s(i) = o(i) ^ P s(i-1),   x(i) = x(i-1) ^ s(i)   (Eq. Oplus),
// so a segment started from (s, x) = (0, 0) gives a particular solution, and
// the true one adds P^j s_a to s and x_a ^ (P + ... + P^j) s_a to x.
//
// Steps of one call (all on the caller's stream):
//   1. k_split_setup: segment states k = 0 .. K-1 are copies of the state
//      with the own generator jumped ahead by k len iterations (GF(2) matrix
//      powers for the xor-likes, for BBS x <- x^(2^(11 k len)) modulo each
//      factor, the exponent mod p - 1 (k_split_constants), each of the eight 16-bit generators by its own squaring count for
//      Algorithm 5 as printed) and (s, x) = (0, 0) for k >= 1;
//   2. written outputs of the BBS sources (62-bit and Algorithm 5 as
//      printed), where generation is the cost, with many warp groups:
//      k_split_run_fix runs every segment from there into its output
//      columns, and as soon as a segment and its predecessor's true end are
//      done, XORs the segment's homogeneous part into its outputs (the
//      mixing step with zero own words: two shuffles per output), which also
//      gives the segment's true end; the fix-ups overlap the other segments'
//      generation;
//   3. the same with few warp groups, where one serial chain of fix-ups per
//      group would outlast the generation: pass 1 (k_split_run) into the
//      output columns, the carry scan of step 4 (true starts only), then
//      k_split_fixup runs all fix-ups at once;
//   4. otherwise (xor-like outputs are cheaper to generate again than to
//      read back, and consumer sinks have no outputs to fix): pass 1
//      (k_split_run) runs segments 0 .. K-2 for their end states alone;
//      k_split_carry, one cluster of blocks per warp group, scans the segments: the true start of segment k is its predecessor's
//      particular end plus (Q s_a, x_a ^ S s_a) with Q = P^len,
//      S = P + ... + P^len (a chunked parallel scan over up to 32 warps);
//      pass 2 (k_split_run) runs every segment from its true start, with the
//      own words k_split_setup jumped to, into the sink;
//   5. the last segment's end state becomes the caller's state, and the
//      per-segment quarter-circle counts or digests are combined.
// A short call of a narrow xor-like state does all of it in one launch
// (k_narrow); single_call chooses among the forms.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "ci_split.h"
#include "ci_device.cuh"
#include "ci_trace.h"

namespace ci {
namespace {

using namespace dev;

// ------------------------------------------------ xor-like jump tables
// Column form of the GF(2)-linear step A of a xor-like with W 32-bit words:
// T[i][j] = A^(2^i) e_j, so v <- A^(2^i) v is the XOR of the columns j at the
// set bits of v.  Built on the device from the sources' own next(); the jumps
// use the XORs of each four columns, N[i][g][b] = XOR of T[i][4 g + k] over
// the set bits k of b, so a level takes 8 W lookups instead of 32 W
// conditional XORs (256 xor128 streams in 64 segments: setup 52 us by columns).
constexpr int kJumpLevels = 64;
__device__ uint32_t g_columns_xor128[kJumpLevels][128][4];
__device__ uint32_t g_columns_xor64[kJumpLevels][64][2];
__device__ uint32_t g_columns_xs32[kJumpLevels][32][1];
__device__ __align__(16) uint32_t g_jump_xor128[kJumpLevels][32][16][4];
__device__ __align__(16) uint32_t g_jump_xor64[kJumpLevels][16][16][2];
__device__ __align__(16) uint32_t g_jump_xs32[kJumpLevels][8][16][1];

template <int W>
__device__ __forceinline__ void step_words(uint32_t (&v)[W]) {
    if (W == 4) {
        SrcXor128 s;
        s.a = v[0];
        s.b = v[1 % W];
        s.c = v[2 % W];
        s.d = v[3 % W];
        s.next();
        v[0] = s.a;
        v[1 % W] = s.b;
        v[2 % W] = s.c;
        v[3 % W] = s.d;
    } else if (W == 2) {
        SrcXor64 s;
        s.z = (uint64_t)v[0] | ((uint64_t)v[1 % W] << 32);
        s.next();
        v[0] = (uint32_t)s.z;
        v[1 % W] = (uint32_t)(s.z >> 32);
    } else {
        SrcXorshift32 s;
        s.z = v[0];
        s.next();
        v[0] = s.z;
    }
}

// One block of 32 W threads; thread j owns column j at every level.
template <int W>
__global__ void k_build_jump(uint32_t (*T)[32 * W][W]) {
    const int j = threadIdx.x;
    uint32_t v[W];
#pragma unroll
    for (int w = 0; w < W; ++w) v[w] = (w == j / 32) ? (1u << (j % 32)) : 0u;
    step_words<W>(v);
#pragma unroll
    for (int w = 0; w < W; ++w) T[0][j][w] = v[w];
    for (int i = 1; i < kJumpLevels; ++i) {
        __syncthreads();
        uint32_t r[W] = {};
        for (int b = 0; b < 32 * W; ++b)
            if ((T[i - 1][j][b / 32] >> (b % 32)) & 1u)
#pragma unroll
                for (int w = 0; w < W; ++w) r[w] ^= T[i - 1][b][w];
#pragma unroll
        for (int w = 0; w < W; ++w) T[i][j][w] = r[w];
    }
}

// Thread (i, g, b) of the nibble tables.
template <int W>
__global__ void __launch_bounds__(256) k_build_nibbles(const uint32_t (*T)[32 * W][W], uint32_t (*N)[8 * W][16][W]) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= kJumpLevels * 8 * W * 16) return;
    const int b = t % 16, g = t / 16 % (8 * W), i = t / (16 * 8 * W);
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint32_t r = 0;
        for (int k = 0; k < 4; ++k)
            if ((b >> k) & 1) r ^= T[i][4 * g + k][w];
        N[i][g][b][w] = r;
    }
}

template <int W>
struct JumpWord {
    using type = uint32_t;
};
template <>
struct JumpWord<2> {
    using type = uint2;
};
template <>
struct JumpWord<4> {
    using type = uint4;
};

template <int W>
__device__ __forceinline__ void jump_words(uint32_t (&v)[W], uint64_t dist, const uint32_t (*N)[8 * W][16][W]) {
    using Word = typename JumpWord<W>::type;
    for (int i = 0; dist; ++i, dist >>= 1) {
        if (!(dist & 1ull)) continue;
        uint32_t r[W] = {};
#pragma unroll
        for (int w = 0; w < W; ++w)
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const Word e = __ldg(reinterpret_cast<const Word *>(N[i][8 * w + g][(v[w] >> (4 * g)) & 15u]));
                if constexpr (W == 1) r[0] ^= e;
                if constexpr (W >= 2) {
                    r[0] ^= e.x;
                    r[1] ^= e.y;
                }
                if constexpr (W == 4) {
                    r[2] ^= e.z;
                    r[3] ^= e.w;
                }
            }
#pragma unroll
        for (int w = 0; w < W; ++w) v[w] = r[w];
    }
}

// Builds one source's tables on `stream`.
template <int W>
cudaError_t build_jump_tables(const void *columns_symbol, const void *jump_symbol, cudaStream_t stream) {
    void *columns = nullptr, *jump = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&columns, columns_symbol);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&jump, jump_symbol);
    if (e != cudaSuccess) return e;
    k_build_jump<W><<<1, 32 * W, 0, stream>>>(static_cast<uint32_t(*)[32 * W][W]>(columns));
    k_build_nibbles<W><<<(kJumpLevels * 8 * W * 16 + 255) / 256, 256, 0, stream>>>(
        static_cast<const uint32_t(*)[32 * W][W]>(columns), static_cast<uint32_t(*)[8 * W][16][W]>(jump));
    return cudaGetLastError();
}

// The tables of one device: built by the first call that jumps, on its stream,
// with `done` recorded behind them.  Calls on other streams wait for the event
// on the device until it has been seen finished; the host never waits.
struct JumpTables {
    cudaEvent_t done = nullptr;
    bool ready = false;
};
std::mutex g_tables_mu;
std::vector<JumpTables> g_tables;  // per device ordinal

// Lets this thread build and query on `stream` while it captures another one
// (a capture in the global mode refuses such calls otherwise).
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The current device's entry, with g_tables_mu held; null without a device.
JumpTables *device_tables() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return nullptr;
    if ((int)g_tables.size() <= dev) g_tables.resize(dev + 1);
    return &g_tables[dev];
}

// Whether the tables are finished, with g_tables_mu held.
bool tables_ready(JumpTables &t) {
    if (t.ready || !t.done) return t.ready;
    RelaxedCapture relaxed;
    t.ready = cudaEventQuery(t.done) == cudaSuccess;
    if (!t.ready) cudaGetLastError();  // "not ready" is no error of the call
    return t.ready;
}

// Work put on `stream` after this finds finished tables.  Not for a capturing
// stream, unless they are ready.
cudaError_t ensure_jump_tables(cudaStream_t stream) {
    std::lock_guard<std::mutex> lk(g_tables_mu);
    JumpTables *t = device_tables();
    if (!t) return cudaErrorInvalidDevice;
    if (tables_ready(*t)) return cudaSuccess;
    if (t->done) return cudaStreamWaitEvent(stream, t->done, 0);
    RelaxedCapture relaxed;
    cudaEvent_t done;
    cudaError_t e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
    if (e != cudaSuccess) return e;
    e = build_jump_tables<4>(g_columns_xor128, g_jump_xor128, stream);
    if (e == cudaSuccess) e = build_jump_tables<2>(g_columns_xor64, g_jump_xor64, stream);
    if (e == cudaSuccess) e = build_jump_tables<1>(g_columns_xs32, g_jump_xs32, stream);
    if (e == cudaSuccess) e = cudaEventRecord(done, stream);
    if (e == cudaSuccess)
        t->done = done;
    else
        cudaEventDestroy(done);
    return e;
}

// ------------------------------------------------ BBS jump
// x <- x^(2^E) mod M with E = 11 * dist squarings, through the exponent
// 2^E mod lambda, plus lambda where that is below 62, with lambda from
// k_split_constants: Carmichael's lambda of M, which holds for every x, or a
// multiple of the order of x.
// a^e mod M for a < M, left to right over 2-bit windows of e: two squarings
// and one product by a^w (by 1 for w = 0) per window, the same work in every
// lane whatever its exponent bits.
__device__ __forceinline__ uint64_t pow_mod(const Barrett62 &B, uint64_t a, uint64_t e) {
    if (e == 0) return 1 % B.M;
    const uint64_t a2 = B.mul(a, a), a3 = B.mul(a2, a), one = 1 % B.M;
    int i = (63 - __clzll((long long)e)) & ~1;  // the window that holds the top bit
    uint32_t w = (uint32_t)(e >> i) & 3u;
    uint64_t r = w == 1u ? a : w == 2u ? a2 : a3;
    for (i -= 2; i >= 0; i -= 2) {
        r = B.mul(r, r);
        r = B.mul(r, r);
        w = (uint32_t)(e >> i) & 3u;
        r = B.mul(r, w == 0u ? one : w == 1u ? a : w == 2u ? a2 : a3);
    }
    return r;
}

__device__ __forceinline__ uint64_t bbs_jump(uint64_t y, uint64_t M, uint64_t mu, uint64_t lam, uint64_t lam_mu,
                                             uint64_t squarings) {
    Barrett62 L;
    L.set(lam, lam_mu);
    // 2^squarings mod lam by square-and-multiply on the exponent's bits
    uint64_t e = pow_mod(L, 2 % lam, squarings);
    if (e < 62) e += lam;
    Barrett62 B;
    B.set(M, mu);
    return pow_mod(B, y, e);
}

// ------------------------------------------------ segment states
struct SegSpace {
    DevState v0;        // view of segment 0 (pointers into the workspace)
    uint64_t stride;    // bytes between segment states
    __device__ __forceinline__ DevState at(uint64_t k) const {
        DevState s = v0;
        const uint64_t off = k * stride;
        s.table = v0.table + off;
        s.u32 = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(v0.u32) + off);
        if (v0.u64) s.u64 = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(v0.u64) + off);
        return s;
    }
};

constexpr int kOwnWords = 4;  // F_A .. F_D (CI_VAR_BBS16: the eight states F_Y16 ..)

// Own words of every segment's start (k >= 1), saved by k_split_setup for the
// regenerate form: field f of segment k, lane l at u32[(f * K + k) * P + l].
struct OwnSave {
    uint32_t *u32;  // `count` fields from `first` (nullptr: not saved)
    uint64_t *u64;  // the BBS state (CI_VAR_BBS)
    int first, count;
};

// Algorithm 5 as printed, run as a segment of one call: the arrays are the
// ones the call chose when it started (stored in the sel field by
// k_split_setup, as sel1 | sel2 << 8), and the generators are not rotated at
// the segment's end (the call rotates them once, when its last segment
// becomes the caller's state).
struct SrcBbs16Seg : SrcBbs16 {
    __device__ __forceinline__ void load(const DevState &s, uint64_t l) {
        SrcBbs16::load(s, l);
        const uint32_t sel = s.u32[F_SEL * s.P + l];
        sel1 = sel & 7u;
        sel2 = (sel >> 8) & 7u;
    }
    __device__ __forceinline__ void store(const DevState &s, uint64_t l) const {
#pragma unroll
        for (int k = 0; k < 8; ++k) s.u32[(F_Y16 + k) * s.P + l] = y[k];
    }
};

// Squarings of generator k (BBS1 .. BBS8) per output of Algorithm 5 as printed:
// one chunk each, then BBS3 and BBS1, BBS7 and BBS2 for the two shift steps.
__constant__ uint32_t c_bbs16_squarings[8] = {2, 2, 2, 1, 1, 1, 2, 1};

// Once per lane, for every segment: the constants of the residue form
// (crt_store) and, in kJumpWords fields behind them, what its jump starts from
// (the Montgomery forms of y mod p, y mod q, 1 mod p and 1 mod q, p < q), or
// lam[l] = lambda and lam[P + l] = barrett_mu(lambda) for bbs_jump.
// An imported state may have factors that are not prime or not distinct, or a
// y that is no unit.  The exponents may be reduced modulo p - 1 and q - 1 if
// y^(p-1) = 1 mod p and y^(q-1) = 1 mod q, which all seeded lanes pass and is
// tested here.  Lanes that fail jump by Carmichael's lambda of their M, factored
// by trial division (some tenths of a millisecond).
// Three threads per lane, in warps of their own: the residue constants, the
// test of p, the test of q, one power each (one thread after the other: 4 us
// more for 32 streams).  A failed test leaves its `one` field 0.
constexpr int kJumpWords = 4;
__global__ void __launch_bounds__(256) k_split_constants(DevState src, uint64_t *lam, uint32_t *crt) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, P = src.P;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < 3 * P; t += stride) {
        const uint64_t l = t % P;
        const int role = (int)(t / P);
        const uint32_t a = src.u32[F_P * P + l], b = src.u32[F_Q * P + l];
        const bool range = min(a, b) > (1u << 30) && max(a, b) < (1u << 31);
        const uint64_t y = src.u64[G_Y * P + l];
        uint64_t v;
        if (role == 0) {
            if (crt_store(src, l, crt)) continue;
            v = 0;
            if (!range) {
                Barrett62 B;
                B.set(src.u64[G_M * P + l], src.u64[G_MU * P + l]);
                v = lcm<uint64_t>(a - 1, b - 1);
                if (pow_mod(B, y, v) != 1) v = 0;
            }
        } else {
            uint32_t *jump = crt + (kCrtWords + role - 1) * P + l;
            jump[2 * P] = 0u;
            if (!range) continue;
            const Mont31 Mf(role == 1 ? min(a, b) : max(a, b));
            const uint32_t yf = Mf.to((uint32_t)(y % Mf.m));
            if (Mf.pow_m(yf, Mf.m - 1) == Mf.one) {
                jump[0] = yf;
                jump[2 * P] = Mf.one;
                continue;
            }
            v = 0;
        }
        if (!v) v = carmichael(a, b);
        lam[l] = v;  // of one lane: the same value, whichever of its threads get here
        lam[P + l] = barrett_mu(v);
    }
}

// The lane's BBS state after `squarings` more squarings.
__device__ __forceinline__ uint64_t bbs_jump_lane(const DevState &src, uint64_t l, uint64_t squarings,
                                                  const uint64_t *lam, const uint32_t *crt) {
    const uint64_t P = src.P;
    CrtModulus C;
    const uint32_t *jump = crt + kCrtWords * P + l;
    // all loaded before the test: one round trip
    const uint32_t yp = jump[0], yq = jump[P], one_p = jump[2 * P], one_q = jump[3 * P];
    if (crt_load(src, l, crt, C) & (one_p != 0u) & (one_q != 0u)) {
        const Mont31 Mp(C.P.p, one_p), Mq(C.Q.p, one_q);
        return C.value(Mp.from(squarings_m(C.P.p, one_p, yp, squarings)),
                       Mq.from(squarings_m(C.Q.p, one_q, yq, squarings)));
    }
    return bbs_jump(src.u64[G_Y * P + l], src.u64[G_M * P + l], src.u64[G_MU * P + l], lam[l], lam[P + l], squarings);
}

// Carmichael's lambda of each 16-bit modulus; lam[k * P + l] for generator k of
// lane l.
__global__ void __launch_bounds__(256) k_split_lambda16(DevState src, uint32_t *lam) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < 8 * src.P; t += stride)
        lam[t] = carmichael16(src.u32[F_M16 * src.P + t]);  // generator t / P of lane t % P
}

// a^e mod m for m < 2^16 (products fit 32 bits).
__device__ __forceinline__ uint32_t pow_mod16(uint32_t a, uint64_t e, uint32_t m) {
    uint32_t r = 1 % m, b = a % m;
    while (e) {
        if (e & 1ull) r = r * b % m;
        b = b * b % m;
        e >>= 1;
    }
    return r;
}

// Thread (k, l): segment k's lane l.  Copies the caller's lane (and the
// partner table), jumps the own generator by k * len iterations and, for
// k >= 1, clears slot and x.
__global__ void __launch_bounds__(256) k_split_setup(DevState src, SegSpace seg, uint32_t K, uint64_t len,
                                                     int variant, int xl, OwnSave own, const uint32_t *lam16,
                                                     const uint64_t *lam64, const uint32_t *crt) {
    const int nf = variant == CI_VAR_BBS16 ? kU32FieldsBbs16 : kU32Fields;
    const uint64_t total = (uint64_t)(K + (variant == CI_VAR_BBS16 ? 1 : 0)) * src.P;  // BBS16: slot K, a copy of the start
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const uint64_t k = t / src.P, l = t % src.P;
        const DevState d = seg.at(k);
        for (uint64_t w = l; w < kTableBytes / 4; w += src.P)
            reinterpret_cast<uint32_t *>(const_cast<uint8_t *>(d.table))[w] =
                reinterpret_cast<const uint32_t *>(src.table)[w];
#pragma unroll
        for (int f = 0; f < kU32FieldsBbs16; ++f)
            if (f < nf) d.u32[f * src.P + l] = src.u32[f * src.P + l];
        if (variant == CI_VAR_BBS)
            for (int f = 0; f < kU64Fields; ++f) d.u64[f * src.P + l] = src.u64[f * src.P + l];
        if (variant == CI_VAR_BBS16)  // the arrays the call chose at its start, for every segment
            d.u32[F_SEL * src.P + l] = (src.u32[F_Y16 * src.P + l] & 7u) | ((src.u32[(F_Y16 + 1) * src.P + l] & 7u) << 8);
        if (k == 0 || k == K) continue;
        d.u32[F_X * src.P + l] = 0;
        d.u32[F_SLOT * src.P + l] = 0;
        const uint64_t dist = k * len;
        if (variant == CI_VAR_BBS16) {
#pragma unroll  // (rolled: 1000 x 65536 74 us instead of 56, and 2^16 BBS streams 95 instead of 84)
            for (int g = 0; g < 8; ++g) {  // x <- x^(2^(c_g dist)) mod M, for any x and M (carmichael16)
                const uint32_t M = src.u32[(F_M16 + g) * src.P + l], lam = lam16[(uint64_t)g * src.P + l];
                uint32_t e = pow_mod16(2, c_bbs16_squarings[g] * dist, lam);
                if (e < 15) e += lam;
                d.u32[(F_Y16 + g) * src.P + l] = pow_mod16(src.u32[(F_Y16 + g) * src.P + l], e, M);
            }
        } else if (variant == CI_VAR_BBS) {
            d.u64[G_Y * src.P + l] = bbs_jump_lane(src, l, 11ull * dist, lam64, crt);
        } else if (xl == CI_XL_XOR128) {
            uint32_t v[4];
            for (int w = 0; w < 4; ++w) v[w] = src.u32[(F_A + w) * src.P + l];
            jump_words<4>(v, dist, g_jump_xor128);
            for (int w = 0; w < 4; ++w) d.u32[(F_A + w) * src.P + l] = v[w];
        } else if (xl == CI_XL_XOR64) {
            uint32_t v[2] = {src.u32[F_A * src.P + l], src.u32[F_B * src.P + l]};
            jump_words<2>(v, dist, g_jump_xor64);
            d.u32[F_A * src.P + l] = v[0];
            d.u32[F_B * src.P + l] = v[1];
        } else {
            uint32_t v[1] = {src.u32[F_A * src.P + l]};
            jump_words<1>(v, dist, g_jump_xs32);
            d.u32[F_A * src.P + l] = v[0];
        }
        if (own.u32) {
            for (int f = 0; f < own.count; ++f)
                own.u32[((uint64_t)f * K + k) * src.P + l] = d.u32[(own.first + f) * src.P + l];
            if (own.u64) own.u64[k * src.P + l] = d.u64[G_Y * src.P + l];
        }
    }
}

// 32 x 32 GF(2) matrices over a warp's lanes, lane l holding row l (bit m of
// row l = entry (l, m)); M v for a vector of words v (one per lane): lane l
// takes the XOR of v_m over the set bits m of row_l(M).  A product A B is A
// applied to the words of B's rows.
//
// (M v, N v) of two matrices and one vector, by the method of four Russians:
// the warp tabulates the 16 XORs of each four consecutive lanes' words in
// shared memory, and every lane looks its eight nibbles per row up (lanes that
// read one group's table hit 16 banks).
struct MatVecScratch {
    uint32_t v[32], tab[8][16];
};
__device__ __forceinline__ uint2 mat_vec2(uint32_t m_row, uint32_t n_row, uint32_t v, MatVecScratch &sc) {
    const int lane = threadIdx.x & 31;
    sc.v[lane] = v;
    __syncwarp();
    const uint4 w = reinterpret_cast<const uint4 *>(sc.v)[lane >> 2];
    const uint32_t h = ((lane & 1) ? w.z : 0u) ^ ((lane & 2) ? w.w : 0u);
    reinterpret_cast<uint4 *>(sc.tab[lane >> 2])[lane & 3] = make_uint4(h, h ^ w.x, h ^ w.y, h ^ w.x ^ w.y);
    __syncwarp();
    uint2 r = make_uint2(0u, 0u);
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        r.x ^= sc.tab[g][(m_row >> (4 * g)) & 15u];
        r.y ^= sc.tab[g][(n_row >> (4 * g)) & 15u];
    }
    return r;
}

// Row of P for a lane with partners p1 and p2.  The bytes of an imported partner
// table are lane numbers modulo 32, as the shuffles of the generation loop take
// them.
__device__ __forceinline__ uint32_t partner_row(int p1, int p2) { return (1u << (p1 & 31)) ^ (1u << (p2 & 31)); }

// Q = P^len and S = P + ... + P^len, len >= 1, by the bits of len from the
// top: (Q, S) for k -> 2k: S <- S ^ S Q, Q <- Q Q; k -> k + 1: Q <- Q P,
// S <- S ^ Q (all are polynomials in P, so they commute).
__device__ __forceinline__ void power_sums(uint32_t prow, uint64_t len, uint32_t &Q, uint32_t &S, MatVecScratch &sc) {
    Q = S = prow;
    for (int b = 62 - __clzll((long long)len); b >= 0; --b) {
        const uint2 sq = mat_vec2(Q, S, Q, sc);
        Q = sq.x;
        S ^= sq.y;
        if ((len >> b) & 1ull) {
            Q = mat_vec2(Q, Q, prow, sc).x;
            S ^= Q;
        }
    }
}

// The carry scan over the segments of one warp group, with a cluster of
// kCarryBlocks blocks, NW = 32 warps together, per group: a step is some 20
// shared-memory operations of a warp, which 32 warps on one SM queued for (60
// us for 1024 segments of one group).  c_j, the true (slot, x) at the start of segment j, obeys
// c_j = e_{j-1} ^ H(c_{j-1}), c_0 = 0 (segment 0 ran from the true state),
// with e_{j-1} the particular end of segment j-1 and H(s, x) = (Q s, x ^ S s).
// Warp w owns steps j in [j0, j1) (m = ceil((K-1) / NW) each):
//   1. local scan from zero: d_j = e_{j-1} ^ H(d_{j-1}), d_{j0-1} = 0, kept in
//      starts[j]; its end goes to shared memory;
//   2. carry-in c_{j0-1}: fold the earlier warps' local ends through H^m,
//      whose pair (Q_m, T_m) follows from (Q, S) by the binary method on m
//      (H^(a+b) = (Q_a Q_b, T_b ^ T_a Q_b));
//   3. c_j = d_j ^ H^(j - j0 + 1)(c_{j0-1}).
// The segments' words are loaded kCarryAhead steps at a time: a step is short
// next to a memory round trip.  (32 streams in 256 segments: 118 us with
// shuffled matrix-vector products, 64-step powers and one load ahead.)
// Fix-up form (`own` == nullptr): c_j goes to starts[j].  Regenerate form:
// c_j and the saved own words of segment j's start go into its state.
constexpr int kCarryBlocks = 8, kCarryWarps = 4, kCarryAhead = 8;
template <class Src>
__global__ void __cluster_dims__(kCarryBlocks, 1, 1) __launch_bounds__(32 * kCarryWarps)
    k_split_carry(SegSpace seg, uint32_t K, uint64_t len, uint2 *starts, OwnSave own) {
    constexpr int NW = kCarryBlocks * kCarryWarps;
    __shared__ uint2 ends[kCarryWarps][32];  // this block's warps' (slot, x)
    __shared__ uint2 all[NW][32];            // every warp's
    __shared__ __align__(16) MatVecScratch scratch[kCarryWarps];
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const uint64_t g = blockIdx.x / kCarryBlocks;
    const int lane = threadIdx.x & 31, bw = threadIdx.x >> 5, w = (int)cluster.block_rank() * kCarryWarps + bw;
    MatVecScratch &sc = scratch[bw];
    const DevState s0 = seg.at(0);
    const uint64_t P = s0.P, l = g * 32 + lane;
    CI_WARP_CHECK(s0, g < P / 32, CHK_GROUP, g);  // the same in the whole cluster: its warps return together
    Src src;
    src.load(s0, l);
    int a1, a2;
    src.arrays(s0, l, a1, a2);
    const uint32_t prow = partner_row(s0.table[a1 * 32 + lane], s0.table[a2 * 32 + lane]);
    uint32_t Q, S;
    power_sums(prow, len, Q, S, sc);
    const uint32_t m = (K - 1 + NW - 1) / NW;
    const uint32_t j0 = 1 + w * m, j1 = min(K, j0 + m);
    // 1. local scan
    uint32_t ds = 0, dx = 0;
    for (uint32_t jb = j0; jb < j1; jb += kCarryAhead) {
        uint32_t es[kCarryAhead], ex[kCarryAhead];
#pragma unroll
        for (int i = 0; i < kCarryAhead; ++i)
            if (jb + i < j1) {
                const DevState d = seg.at(jb + i - 1);
                es[i] = d.u32[F_SLOT * P + l];
                ex[i] = d.u32[F_X * P + l];
            }
#pragma unroll
        for (int i = 0; i < kCarryAhead; ++i)
            if (jb + i < j1) {
                const uint2 hv = mat_vec2(Q, S, ds, sc);
                dx = ex[i] ^ dx ^ hv.y;
                ds = es[i] ^ hv.x;
                starts[(uint64_t)(jb + i) * P + l] = make_uint2(ds, dx);
            }
    }
    ends[bw][lane] = make_uint2(ds, dx);
    // 2. H^m and this warp's carry-in
    uint32_t Qm = Q, Tm = S;
    for (int b = 30 - __clz((int)m); b >= 0; --b) {
        const uint2 sq = mat_vec2(Qm, Tm, Qm, sc);
        Qm = sq.x;
        Tm ^= sq.y;
        if ((m >> b) & 1u) {
            const uint2 up = mat_vec2(Qm, Tm, Q, sc);
            Qm = up.x;
            Tm = S ^ up.y;
        }
    }
    cluster.sync();
    for (int v = bw; v < NW; v += kCarryWarps)
        all[v][lane] = cluster.map_shared_rank(&ends[0][0], v / kCarryWarps)[(v % kCarryWarps) * 32 + lane];
    cluster.sync();  // every warp's ends are here, and no block is read any more
    uint32_t cs = 0, cx = 0;
    for (int v = 0; v < w; ++v) {
        const uint2 hv = mat_vec2(Qm, Tm, cs, sc);
        cx ^= all[v][lane].y ^ hv.y;
        cs = all[v][lane].x ^ hv.x;
    }
    // 3. true starts of this warp's segments
    for (uint32_t jb = j0; jb < j1; jb += kCarryAhead) {
        uint2 dj[kCarryAhead];
#pragma unroll
        for (int i = 0; i < kCarryAhead; ++i)
            if (jb + i < j1) dj[i] = starts[(uint64_t)(jb + i) * P + l];
#pragma unroll
        for (int i = 0; i < kCarryAhead; ++i)
            if (jb + i < j1) {
                const uint32_t j = jb + i;
                const uint2 hv = mat_vec2(Q, S, cs, sc);
                cs = hv.x;
                cx ^= hv.y;
                const uint32_t ts = dj[i].x ^ cs, tx = dj[i].y ^ cx;
                if (!own.u32) {
                    starts[(uint64_t)j * P + l] = make_uint2(ts, tx);
                } else {
                    const DevState d = seg.at(j);
                    d.u32[F_SLOT * P + l] = ts;
                    d.u32[F_X * P + l] = tx;
                    for (int f = 0; f < own.count; ++f)
                        d.u32[(own.first + f) * P + l] = own.u32[((uint64_t)f * K + j) * P + l];
                    if (own.u64) d.u64[G_Y * P + l] = own.u64[(uint64_t)j * P + l];
                }
            }
    }
}

// Written sink: segment k >= 1 wrote its particular outputs (zero start).
// From its true start c = (s_a, x_a), the homogeneous part is h <- P h,
// acc <- acc ^ h per iteration (two shuffles, as in the mixing step with a
// zero own word); output i of the segment gets acc XORed in.  The warp stages
// 32 iterations of its 32 rows in the swizzled tile and updates the outputs
// as 16-byte row segments (V4) or words.  Another warp wrote those outputs,
// so they are read through L2 (ld.global.cg).  Returns H(c) = (h, acc) at the
// segment's end.
// kAhead: the tile's outputs are loaded before its steps, whose 32 serial
// shuffles then hide the round trip (the fix-ups as a kernel of their own; among
// the squaring warps of the one-launch form other warps hide it, and the 32
// registers are not to be had).
template <bool V4, bool kAhead>
__device__ __forceinline__ uint2 fix_segment(uint2 c, int p1, int p2, uint64_t n, uint32_t *base, uint64_t row0,
                                             uint64_t S, uint64_t ld, uint4 *tile) {
    const int lane = threadIdx.x & 31;
    uint32_t *tw = reinterpret_cast<uint32_t *>(tile);
    uint32_t h = c.x, acc = c.y;
    auto step = [&]() {
        h = __shfl_sync(kFull, h, p1) ^ __shfl_sync(kFull, h, p2);
        acc ^= h;
        return acc;
    };
    const uint64_t nfull = n - n % 32;
    for (uint64_t i0 = 0; i0 < nfull; i0 += 32) {
        uint4 ahead[kAhead ? 8 : 1];
        if (V4 && kAhead) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const int r = 4 * kk + lane / 8;
                if (row0 + r < S)
                    ahead[kk] = __ldcg(reinterpret_cast<const uint4 *>(base + (row0 + r) * ld + i0 + 4 * (lane % 8)));
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint4 f;
            f.x = step();
            f.y = step();
            f.z = step();
            f.w = step();
            tile[lane * 8 + (q ^ (lane & 7))] = f;
        }
        __syncwarp();
        if (V4) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const int r = 4 * kk + lane / 8, cc = lane % 8;
                if (row0 + r < S) {
                    uint4 *p = reinterpret_cast<uint4 *>(base + (row0 + r) * ld + i0 + 4 * cc);
                    const uint4 v = tile[r * 8 + (cc ^ (r & 7))];
                    uint4 o = kAhead ? ahead[kk] : __ldcg(p);
                    o.x ^= v.x;
                    o.y ^= v.y;
                    o.z ^= v.z;
                    o.w ^= v.w;
                    store16<0>(reinterpret_cast<uint32_t *>(p), o);
                }
            }
        } else {
            for (int r = 0; r < 32; ++r)
                if (row0 + r < S) {
                    uint32_t *p = base + (row0 + r) * ld + i0 + lane;
                    *p = __ldcg(p) ^ tw[tile_word<32>(r, lane)];
                }
        }
        __syncwarp();
    }
    const int rem = (int)(n - nfull);
    if (rem) {
        for (int kk = 0; kk < rem; ++kk) tw[tile_word<32>(lane, kk)] = step();
        __syncwarp();
        for (int r = 0; r < 32; ++r)
            if (lane < rem && row0 + r < S) {
                uint32_t *p = base + (row0 + r) * ld + nfull + lane;
                *p = __ldcg(p) ^ tw[tile_word<32>(r, lane)];
            }
        __syncwarp();
    }
    return make_uint2(h, acc);
}

// The fix-ups as a kernel of their own, after pass 1 and the carry scan:
// work unit = (segment k >= 1, warp group g), all independent; the last
// segment also corrects its end state.
template <class Src, bool V4>
__global__ void __launch_bounds__(256) k_split_fixup(SegSpace seg, const uint2 *starts, uint32_t K, uint64_t len,
                                                     uint64_t len_last, uint64_t groups, uint32_t *out, uint64_t ld,
                                                     uint64_t col0) {
    __shared__ uint4 tiles[8][256];
    const int lane = threadIdx.x & 31;
    uint4 *tile = tiles[threadIdx.x >> 5];
    const DevState s0 = seg.at(0);
    const uint64_t P = s0.P;
    const uint64_t units = (uint64_t)(K - 1) * groups;
    for (uint64_t u = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < units; u += (uint64_t)gridDim.x * 8) {
        const uint64_t k = 1 + u / groups, g = u % groups, l = g * 32 + lane;
        CI_WARP_CHECK(s0, k < K && g < P / 32, CHK_SEGMENT, k);
        CI_WARP_CHECK(s0, col0 + k * len + (k + 1 == K ? len_last : len) <= ld, CHK_SEG_COLS, k);
        if (V4) CI_WARP_CHECK(s0, ((col0 + k * len) | ld) % 4 == 0, CHK_V4_ALIGN, k);
        Src src;
        src.load(s0, l);
        int a1, a2;
        src.arrays(s0, l, a1, a2);
        const uint2 hk = fix_segment<V4, true>(starts[k * P + l], s0.table[a1 * 32 + lane], s0.table[a2 * 32 + lane],
                                         k + 1 == K ? len_last : len, out + col0 + k * len, g * 32, s0.S, ld, tile);
        if (k + 1 == K) {
            const DevState d = seg.at(K - 1);
            d.u32[F_SLOT * P + l] ^= hk.x;
            d.u32[F_X * P + l] ^= hk.y;
        }
    }
}

// The last segment's state becomes the caller's state (the sel field, which
// generation never changes, stays the caller's).  CI_VAR_BBS16: generator k
// (state and modulus) moves to place k + 1, the call's one rotation.
__global__ void __launch_bounds__(256) k_split_copy_back(DevState dst, DevState last, int variant) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, P = dst.P;
    const int n32 = variant == CI_VAR_BBS16 ? kU32FieldsBbs16 : kU32Fields;
    const uint64_t total = (n32 + (dst.u64 ? kU64Fields : 0)) * P;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const int f = (int)(t / P);
        const uint64_t l = t % P;
        if (f >= n32) {
            dst.u64[(f - n32) * P + l] = last.u64[(f - n32) * P + l];
        } else if (f != F_SEL) {
            const int to = f < F_Y16 ? f : f < F_M16 ? F_Y16 + (f - F_Y16 + 1) % 8 : F_M16 + (f - F_M16 + 1) % 8;
            dst.u32[to * P + l] = last.u32[f * P + l];
        }
    }
}

// Combines per-segment consumer results r[k * P + l] for stream l < S:
// quarter-circle counts are added to out[l]; digests are joined by Horner,
// D = sum_k D_k K^(n - end of segment k), the last segment ending at n.
__global__ void __launch_bounds__(256) k_split_combine(const uint64_t *r, uint64_t *out, uint64_t P, uint64_t S,
                                                       uint32_t K, uint64_t len, uint64_t len_last, int digest) {
    const uint64_t l = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= S) return;
    if (!digest) {
        uint64_t c = 0;
        for (uint32_t k = 0; k < K; ++k) c += r[(uint64_t)k * P + l];
        out[l] += c;
        return;
    }
    auto kpow = [](uint64_t e) {
        uint64_t b = kDigestMul, p = 1;
        while (e) {
            if (e & 1ull) p *= b;
            b *= b;
            e >>= 1;
        }
        return p;
    };
    const uint64_t step = kpow(len);
    uint64_t d = 0, mult = 1;
    for (uint32_t k = K; k-- > 0;) {
        d += r[(uint64_t)k * P + l] * mult;
        mult *= (k == K - 1) ? kpow(len_last) : step;
    }
    out[l] = d;
}

// Consumer results from written rows: the scratch form of a BBS-source
// consumer call, whose outputs were written (and fixed up) into `rows`, row r
// (stride n) holding stream r's n outputs.  Work unit = (row r, chunk
// [b, e) of clen outputs), one warp.  Quarter-circle sink: the chunk's hits
// among its pairs (o_2k, o_2k+1) are added to out[r] (clen and n even).
// Digest sink: the chunk contributes K^(n-e) sum_{b<=i<e} o_i K^(e-1-i), so
// the contributions of all chunks sum to D = sum_i o_i K^(n-1-i); lane j
// takes outputs e-1-j, e-1-j-32, ... with the running power K^j, K^(j+32), ...,
// and out[r] (cleared before) receives the warp's sum.
__device__ __forceinline__ uint64_t digest_pow(uint64_t e) {
    uint64_t b = kDigestMul, p = 1;
    while (e) {
        if (e & 1ull) p *= b;
        b *= b;
        e >>= 1;
    }
    return p;
}

template <bool kDigest>
__global__ void __launch_bounds__(256) k_consume_rows(const uint32_t *rows, uint64_t S, uint64_t n, uint64_t clen,
                                                      uint64_t chunks, uint64_t *out) {
    const int lane = threadIdx.x & 31;
    const uint64_t units = S * chunks;
    for (uint64_t u = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < units; u += (uint64_t)gridDim.x * 8) {
        const uint64_t r = u / chunks, c = u % chunks;
        const uint64_t b = c * clen, e = b + clen < n ? b + clen : n;
        const uint32_t *row = rows + r * n;
        uint64_t v = 0;
        if (kDigest) {
            uint64_t pw = digest_pow((uint64_t)lane);
            const uint64_t step = digest_pow(32);
            for (uint64_t t = (uint64_t)lane; t < e - b; t += 32) {
                v += (uint64_t)row[e - 1 - t] * pw;
                pw *= step;
            }
        } else {
            const uint2 *pairs = reinterpret_cast<const uint2 *>(row + b);
            for (uint64_t k = (uint64_t)lane; k < (e - b) / 2; k += 32) {
                const uint2 o = pairs[k];
                v += 1u - qc_miss(o.x, o.y);
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
        if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long *>(out + r), kDigest ? v * digest_pow(n - e) : v);
    }
}

// ------------------------------------------------ narrow xor-like calls
// A call of few warp groups in one launch: a cluster of up to kNarrowBlocks
// blocks per group, whose up to 32 warps take one time segment of `len`
// iterations each (len a multiple of 32; K segments, the last one shorter).  Bound by latency:
// a warp alone on its scheduler takes 55 cycles a step, so 4096 x 1024 unsplit
// spent 27 us on one chain of 1024 steps per SM, and five launches of the
// general form take 45.  Per warp:
//   1. the own generator jumps to its segment's start;
//   2. pass 1 from a zero mixing state (segment 0: from the true one), for the
//      particular end alone; then H = (Q, S) = (P^len, P + ... + P^len);
//   3. carries: the four ends of a block are folded through H, the
//      blocks' aggregates, exchanged by distributed shared memory, through
//      H^4;
//   4. pass 2 from the true start into the sink.
// All state is read before the first cluster barrier; the last segment's warp
// writes it back after it.
constexpr int kNarrowBlocks = 8, kNarrowWarps = 4;  // most blocks of a cluster; warps of a block

__device__ __forceinline__ void jump_source(SrcXor128 &s, uint64_t dist) {
    uint32_t v[4] = {s.a, s.b, s.c, s.d};
    jump_words<4>(v, dist, g_jump_xor128);
    s.a = v[0];
    s.b = v[1];
    s.c = v[2];
    s.d = v[3];
}
__device__ __forceinline__ void jump_source(SrcXor64 &s, uint64_t dist) {
    uint32_t v[2] = {(uint32_t)s.z, (uint32_t)(s.z >> 32)};
    jump_words<2>(v, dist, g_jump_xor64);
    s.z = (uint64_t)v[0] | ((uint64_t)v[1] << 32);
}
__device__ __forceinline__ void jump_source(SrcXorshift32 &s, uint64_t dist) {
    uint32_t v[1] = {s.z};
    jump_words<1>(v, dist, g_jump_xs32);
    s.z = v[0];
}

template <class Src, int SINK, int PITCH = 16>
__global__ void __launch_bounds__(32 * kNarrowWarps)
    k_narrow(DevState st, uint64_t n, uint64_t len, uint32_t K, uint32_t *out, uint64_t *aux) {
    __shared__ uint4 tiles[kNarrowWarps][SINK == SINK_V4 ? 256 : SINK == SINK_SCALAR ? 32 * PITCH : 1];
    __shared__ __align__(16) MatVecScratch scratch[kNarrowWarps];
    __shared__ uint2 ends[kNarrowWarps][32], aggregate[32], all[kNarrowBlocks][32];
    __shared__ uint64_t results[kNarrowWarps][32];
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int nb = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const uint64_t g = blockIdx.x / nb;
    const int lane = threadIdx.x & 31, bw = threadIdx.x >> 5;
    const uint32_t seg = rank * kNarrowWarps + bw;
    CI_WARP_CHECK(st, g < st.P / 32, CHK_GROUP, g);  // the same in the whole cluster: its warps return together
    CI_WARP_CHECK(st, (uint64_t)(K - 1) * len < n && n <= K * len, CHK_SEG_COLS, K);
    MatVecScratch &sc = scratch[bw];
    const uint64_t l = g * 32 + lane;
    Lane<Src> s;
    s.src.load(st, l);
    s.load(st, l);
    const uint32_t slot0 = s.slot, x0 = s.x;
    if (seg > 0 && seg < K) jump_source(s.src, seg * len);
    const Src start = s.src;
    if (seg > 0) s.slot = s.x = 0;
    if (seg + 1 < K) warp_run<Src, SINK_NONE, TileBrief<PITCH>>(s, 0, 0, len, nullptr, 0, 0, nullptr);
    const uint2 e = make_uint2(s.slot, s.x);
    ends[bw][lane] = e;
    uint32_t Q, S;
    power_sums(partner_row(s.p1, s.p2), len, Q, S, sc);
    __syncthreads();
    // H(c) ^ e for c = (slot, x)
    auto advance = [&](uint32_t q, uint32_t t, uint2 c, uint2 add) {
        const uint2 h = mat_vec2(q, t, c.x, sc);
        return make_uint2(add.x ^ h.x, add.y ^ c.y ^ h.y);
    };
    const uint2 zero = make_uint2(0u, 0u);
    uint2 pre = zero;  // the carry into this warp's segment from the block's earlier ones
    for (int v = 0; v < bw; ++v) pre = v ? advance(Q, S, pre, ends[v][lane]) : ends[0][lane];
    if (bw == kNarrowWarps - 1) aggregate[lane] = advance(Q, S, pre, e);
    uint32_t Q4 = Q, S4 = S;  // H^4
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint2 sq = mat_vec2(Q4, S4, Q4, sc);
        Q4 = sq.x;
        S4 ^= sq.y;
    }
    cluster.sync();
    for (int v = bw; v < nb; v += kNarrowWarps) all[v][lane] = cluster.map_shared_rank(aggregate, v)[lane];
    cluster.sync();  // every aggregate is here, and no block's is read any more
    uint2 c = zero;  // the carry into this block's first segment
    for (int v = 0; v < rank; ++v) c = v ? advance(Q4, S4, c, all[v][lane]) : all[0][lane];
    if (rank)
        for (int i = 0; i < bw; ++i) c = advance(Q, S, c, zero);
    s.src = start;
    s.slot = seg ? pre.x ^ c.x : slot0;
    s.x = seg ? pre.y ^ c.y : x0;
    uint64_t r = 0;
    if (seg < K) {
        const uint64_t from = seg * len, m = seg + 1 == K ? n - from : len;
        r = warp_run<Src, SINK, TileBrief<PITCH>>(s, st.S, g * 32, m, out, n, from, tiles[bw]);
        if (SINK == SINK_DIGEST) r *= digest_pow(n - from - m);
        if (seg + 1 == K) s.store(st, l);
    }
    if (SINK == SINK_QC || SINK == SINK_DIGEST) {
        results[bw][lane] = r;
        cluster.sync();
        if (seg == 0) {
            uint64_t sum = 0;
            for (int v = 0; v < nb * kNarrowWarps; ++v)
                sum += cluster.map_shared_rank(&results[0][0], v / kNarrowWarps)[(v % kNarrowWarps) * 32 + lane];
            if (l < st.S) aux[l] = SINK == SINK_QC ? aux[l] + sum : sum;
        }
        cluster.sync();
    }
}

template <class Src>
cudaError_t launch_narrow_src(const DevState &st, int sink, int blocks, uint64_t n, uint64_t len, uint32_t K,
                              uint32_t *out, uint64_t *aux, cudaStream_t stream) {
    cudaLaunchAttribute cluster;
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim = {(unsigned)blocks, 1, 1};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(st.P / 32) * blocks);
    cfg.blockDim = dim3(32 * kNarrowWarps);
    cfg.stream = stream;
    cfg.attrs = &cluster;
    cfg.numAttrs = 1;
    auto kern = sink == SINK_V4       ? k_narrow<Src, SINK_V4>
                : sink == SINK_SCALAR ? (n % 8 == 0 ? k_narrow<Src, SINK_SCALAR, 17> : k_narrow<Src, SINK_SCALAR>)
                : sink == SINK_QC     ? k_narrow<Src, SINK_QC>
                                      : k_narrow<Src, SINK_DIGEST>;
    return cudaLaunchKernelEx(&cfg, kern, st, n, len, K, out, aux);
}

// ------------------------------------------------ host side
constexpr uint32_t kMaxSegments = kSplitMaxSegments;
constexpr uint64_t kMinSegment = 256;       // iterations per segment (auto choice, BBS)
constexpr uint64_t kMinShortSegment = 64;   // ... while they do not fill the GPU (BBS sources)
constexpr uint64_t kMinXorSplit = 2048;     // iterations of a xor-like call that splits on its own
constexpr uint64_t kMinAutoSegment = 1024;  // ... xor-likes, and when a single call splits on its own
constexpr uint64_t kScratchWords = 1ull << 29;  // scratch outputs of a BBS-source consumer call (2 GiB)
// Written BBS-source outputs take the one-launch fix-up form from this many
// warp groups per SM on: its fix-ups run as one serial chain per group among
// the squaring warps, which keeps pace only with enough groups; below it,
// pass 1, the carry scan and the fix-ups run as three launches.
#ifndef CI_ONE_LAUNCH_GROUPS_PER_SM
#define CI_ONE_LAUNCH_GROUPS_PER_SM 12
#endif
constexpr uint64_t kOneLaunchGroupsPerSm = CI_ONE_LAUNCH_GROUPS_PER_SM;

// One pass over segments [k_begin, k_end): work unit u is segment
// k_begin + u / groups, warp group u % groups, run for its length (len, the
// last segment len_last) by the generator's warp loop into SINK: written
// outputs at column col0 + k len of rows of stride ld; consumer results into
// aux + k P.  Segment 0 is the caller's own state when `zero` < 0, else the
// segment state with that index.
// Instantiated per source and sink, with at most 64 registers (4 blocks of 8
// warps per SM): the all-source batched kernel needs 128, which held the
// BBS segments to 16 resident warps per SM.  BBS segments ask for 3 blocks, 80
// registers: the residue form's constants fit without spills (k_split_run_fix,
// with the fix-ups beside them, spills 8 bytes, 24 for unaligned rows), and its
// two independent chains per lane fill the pipes from 24 warps per SM on
// (2^16 x 4096: 3.28 ms; 3.50 with 4 blocks, 3.95 with 5, 3.39 with 2;
// 5.38 in the 62-bit form with 5).  Segments of Algorithm 5 as printed (eight
// generators per lane, 118 registers in the single-call kernel) ask for 2
// blocks, 128 registers, so that their loop does not spill.
template <class Src>
constexpr int split_min_blocks() {
    return std::is_same<Src, SrcBbs>::value ? 3 : std::is_same<Src, SrcBbs16Seg>::value ? 2 : 4;
}

template <class Src, int SINK>
__global__ void __launch_bounds__(256, split_min_blocks<Src>()) k_split_run(SegSpace seg, DevState caller, int zero, uint32_t k_begin,
                                                   uint32_t k_end, uint32_t K, uint64_t len, uint64_t len_last,
                                                   uint64_t groups, uint32_t *out, uint64_t ld, uint64_t col0,
                                                   uint64_t *aux, const uint32_t *crt) {
    __shared__ uint4 tiles[8][SINK == SINK_SCALAR ? kScalarTile<Src> : 256];
    uint4 *tile = tiles[threadIdx.x >> 5];
    const uint64_t units = (uint64_t)(k_end - k_begin) * groups;
    // warp w of block b starts at unit w * gridDim.x + b: a partial last
    // round of warps is spread over every block (and SM)
    for (uint64_t u = (uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < units; u += (uint64_t)gridDim.x * 8) {
        const uint64_t k = k_begin + u / groups, g = u % groups;
        CI_WARP_CHECK(caller, k < K, CHK_SEGMENT, k);
        const DevState st = k != 0 ? seg.at(k) : zero < 0 ? caller : seg.at((uint64_t)zero);
        const uint64_t n = k + 1 == K ? len_last : len;
        if (SINK == SINK_V4 || SINK == SINK_SCALAR)
            warp_task<Src, SINK>(st, g, n, out, ld, col0 + k * len, nullptr, tile, crt);
        else
            warp_task<Src, SINK>(st, g, n, nullptr, 0, 0, aux + k * caller.P, tile, crt);
    }
}

template <class Src, int SINK>
cudaError_t launch_split_run(const SegSpace &sp, const DevState &caller, int zero, uint32_t kb, uint32_t ke,
                             uint32_t K, uint64_t len, uint64_t len_last, uint32_t *out, uint64_t ld, uint64_t col0,
                             uint64_t *aux, const uint32_t *crt, cudaStream_t stream) {
    static int per_sm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_split_run<Src, SINK>, 256, 0);
        if (per_sm <= 0) per_sm = 1;
    });
    const uint64_t groups = caller.P / 32, units = (uint64_t)(ke - kb) * groups;
    if (units == 0) return cudaSuccess;
    const int blocks = (int)std::min<uint64_t>(units, (uint64_t)sm_count() * per_sm);  // a block per unit at most
    k_split_run<Src, SINK><<<blocks, 256, 0, stream>>>(sp, caller, zero, kb, ke, K, len, len_last, groups, out, ld,
                                                       col0, aux, crt);
    return cudaGetLastError();
}

// Written BBS-source outputs, fix-up form, in one launch.  Work units are the
// pass-1 units (segment k, warp group g), taken from a device counter in
// segment-major order.  Fix-up (g, k), k >= 1, needs two events: pass 1 of
// (g, k) has written its particular outputs and end e_k, and the true start
// c_k of segment k is known.  c_1 is the end of segment 0 (which ran from the
// true state), and c_(k+1) = e_k ^ H(c_k), which fix-up (g, k) produces
// itself by running the homogeneous recurrence through the segment, so the
// carry needs no matrix powers.  Each event adds one to events[k groups + g];
// the warp whose addition makes it two runs the fix-up at once, then goes on
// to the group's next segment while that one's pass 1 is already done.  No
// warp waits for another, and the fix-ups' memory traffic overlaps the other
// warps' squarings.  The last segment's fix-up corrects the call's end state.

// Adds one to the event count *ev once the earlier writes of every lane are
// visible device-wide (the release half of the pattern); true in every lane
// when this addition made the count two, the other event's writes then being
// visible to the warp's L2 reads (the acquire half).
__device__ __forceinline__ bool second_event(uint32_t *ev) {
    __threadfence();
    __syncwarp();
    uint32_t old = 0;
    if ((threadIdx.x & 31) == 0) old = atomicAdd(ev, 1u);
    old = __shfl_sync(kFull, old, 0);
    __threadfence();
    return old == 1u;
}

template <class Src, int SINK>
__global__ void __launch_bounds__(256, split_min_blocks<Src>()) k_split_run_fix(SegSpace seg, uint32_t K, uint64_t len,
                                                       uint64_t len_last, uint64_t groups, uint32_t *out, uint64_t ld,
                                                       uint64_t col0, uint2 *starts, uint32_t *events,
                                                       unsigned long long *next_unit, const uint32_t *crt) {
    __shared__ uint4 tiles[8][SINK == SINK_SCALAR ? kScalarTile<Src> : 256];
    uint4 *tile = tiles[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const DevState s0 = seg.at(0);
    const uint64_t P = s0.P, units = (uint64_t)K * groups;
    for (;;) {
        unsigned long long u = 0;
        if (lane == 0) u = atomicAdd(next_unit, 1ull);
        u = __shfl_sync(kFull, u, 0);
        if (u >= units) return;
        uint64_t k = u / groups;
        const uint64_t g = u % groups, l = g * 32 + lane;
        const DevState st = seg.at(k);
        warp_task<Src, SINK>(st, g, k + 1 == K ? len_last : len, out, ld, col0 + k * len, nullptr, tile, crt);
        if (k == 0) {  // the same threads stored segment 0's end: c_1
            starts[P + l] = make_uint2(st.u32[F_SLOT * P + l], st.u32[F_X * P + l]);
            k = 1;
        }
        int p1 = -1, p2 = -1;
        while (second_event(events + k * groups + g)) {
            CI_WARP_CHECK(s0, k < K && g < P / 32, CHK_SEGMENT, k);
            CI_WARP_CHECK(s0, col0 + k * len + (k + 1 == K ? len_last : len) <= ld, CHK_SEG_COLS, k);
            if (SINK == SINK_V4) CI_WARP_CHECK(s0, ((col0 + k * len) | ld) % 4 == 0, CHK_V4_ALIGN, k);
            if (p1 < 0) {
                Src src;
                src.load(s0, l);
                int a1, a2;
                src.arrays(s0, l, a1, a2);
                p1 = s0.table[a1 * 32 + lane];
                p2 = s0.table[a2 * 32 + lane];
            }
            const uint2 hk = fix_segment<SINK == SINK_V4, false>(__ldcg(starts + k * P + l), p1, p2,
                                                          k + 1 == K ? len_last : len, out + col0 + k * len, g * 32,
                                                          s0.S, ld, tile);
            const DevState d = seg.at(k);
            const uint32_t ts = __ldcg(d.u32 + F_SLOT * P + l) ^ hk.x, tx = __ldcg(d.u32 + F_X * P + l) ^ hk.y;
            if (k + 1 == K) {
                d.u32[F_SLOT * P + l] = ts;
                d.u32[F_X * P + l] = tx;
                break;
            }
            starts[(k + 1) * P + l] = make_uint2(ts, tx);
            ++k;
        }
    }
}

template <class Src, int SINK>
cudaError_t launch_split_run_fix(const SegSpace &sp, uint32_t K, uint64_t len, uint64_t len_last, uint64_t groups,
                                 uint32_t *out, uint64_t ld, uint64_t col0, uint2 *starts, uint32_t *events,
                                 unsigned long long *next_unit, const uint32_t *crt, cudaStream_t stream) {
    static int per_sm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_split_run_fix<Src, SINK>, 256, 0);
        if (per_sm <= 0) per_sm = 1;
    });
    const uint64_t units = (uint64_t)K * groups;
    const int blocks = (int)std::min<uint64_t>((units + 7) / 8, (uint64_t)sm_count() * per_sm);
    k_split_run_fix<Src, SINK><<<blocks, 256, 0, stream>>>(sp, K, len, len_last, groups, out, ld, col0, starts, events,
                                                           next_unit, crt);
    return cudaGetLastError();
}

template <int SINK>
cudaError_t split_run_sink(int variant, int xl, const SegSpace &sp, const DevState &caller, int caller0, uint32_t kb,
                           uint32_t ke, uint32_t K, uint64_t len, uint64_t len_last, uint32_t *out, uint64_t ld,
                           uint64_t col0, uint64_t *aux, const uint32_t *crt, cudaStream_t stream) {
    if (variant == CI_VAR_BBS)
        return launch_split_run<SrcBbs, SINK>(sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0, aux, crt, stream);
    if (variant == CI_VAR_BBS16)
        return launch_split_run<SrcBbs16Seg, SINK>(sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0, aux,
                                                   crt, stream);
    if (xl == CI_XL_XORSHIFT32)
        return launch_split_run<SrcXorshift32, SINK>(sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0, aux,
                                                     crt, stream);
    if (xl == CI_XL_XOR64)
        return launch_split_run<SrcXor64, SINK>(sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0, aux,
                                                crt, stream);
    return launch_split_run<SrcXor128, SINK>(sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0, aux,
                                             crt, stream);
}

constexpr int kSinkNone = -1;  // end states only

// Runs segments [kb, ke) into the caller's sink (CI_SINK_*, or kSinkNone); written outputs
// take 16-byte stores when out, ld and col0 allow it.  Segment 0: the caller's
// state (zero < 0) or segment state `zero`.
cudaError_t split_run(const ci_states_s &h, int sink, const SegSpace &sp, int caller0, uint32_t kb, uint32_t ke,
                      uint32_t K, uint64_t len, uint64_t len_last, uint32_t *out, uint64_t ld, uint64_t col0,
                      uint64_t *aux, const uint32_t *crt, cudaStream_t stream) {
    const DevState caller = h.view();
    if (sink == kSinkNone)
        return split_run_sink<SINK_NONE>(h.variant, h.xl, sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0,
                                         aux, crt, stream);
    if (sink == CI_SINK_QC)
        return split_run_sink<SINK_QC>(h.variant, h.xl, sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0,
                                       aux, crt, stream);
    if (sink == CI_SINK_DIGEST)
        return split_run_sink<SINK_DIGEST>(h.variant, h.xl, sp, caller, caller0, kb, ke, K, len, len_last, out, ld,
                                           col0, aux, crt, stream);
    const bool v4 = (reinterpret_cast<uintptr_t>(out) & 15u) == 0 && ld % 4 == 0 && col0 % 4 == 0 && len % 4 == 0;
    if (v4)
        return split_run_sink<SINK_V4>(h.variant, h.xl, sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0,
                                       aux, crt, stream);
    return split_run_sink<SINK_SCALAR>(h.variant, h.xl, sp, caller, caller0, kb, ke, K, len, len_last, out, ld, col0,
                                       aux, crt, stream);
}

int split_block_count(uint64_t items) {
    return (int)std::max<uint64_t>(1, std::min<uint64_t>((items + 255) / 256, (uint64_t)sm_count() * 8));
}

}  // namespace
}  // namespace ci

namespace ci {

cudaError_t split_prepare(cudaStream_t stream) { return ensure_jump_tables(stream); }

namespace {

// Whether a captured call of h may jump.  A graph can neither build the tables
// nor wait for a build outside it: before they are finished such a call runs
// whole, in one launch, with the same results.
bool jumps_at_hand(const ci_states_s &h) {
    if (h.variant != CI_VAR_XOR) return true;
    std::lock_guard<std::mutex> lk(g_tables_mu);
    JumpTables *t = device_tables();
    return t && tables_ready(*t);
}

// Blocks per cluster of the one-launch form for a call of n iterations; 0: it
// does not apply.  From where its jumps and carries (some 7 us) are repaid up
// to where segments of a thirty-second are longer than the general form's.
// About 8 warps per SM, 16 for long calls.  Measured, xor128 written, unsplit
// or general split against this form: 1000 x 448 14 / 10.5 us, 4096 x 512 15 /
// 12, 4096 x 1024 27 / 16 (19 with 16 warps per SM), 9000 x 600 17 / 19, 9000 x
// 2000 49 / 33, 4096 x 4096 72 / 35 (37 with 8), 32 x 4096 44 / 17, 256 x 16384
// 55 / 35, 256 x 65536 76 / 107, 16000 x 2000 51 / 50.
constexpr uint64_t kNarrowMin = 448, kNarrowWideMin = 1024, kNarrowLong = 2048, kNarrowMax = 16384;
int narrow_blocks(const ci_states_s &h, uint64_t n) {
    const uint64_t groups = h.P / 32, sms = (uint64_t)sm_count();
    if (h.variant != CI_VAR_XOR || groups > 2 * sms || n > kNarrowMax) return 0;
    if (n < (groups > sms ? kNarrowWideMin : kNarrowMin)) return 0;
    const uint64_t warps = (n < kNarrowLong ? 8 : 16) * sms;
    int blocks = kNarrowBlocks;
    while (blocks > 1 && groups * kNarrowWarps * blocks > warps) blocks /= 2;
    return blocks;
}

cudaError_t launch_narrow(const ci_states_s &h, int blocks, uint64_t n, int sink, uint32_t *out, uint64_t *aux,
                          cudaStream_t stream) {
    const cudaError_t e = ensure_jump_tables(stream);
    if (e != cudaSuccess) return e;
    const uint64_t segments = (uint64_t)blocks * kNarrowWarps;
    const uint64_t len = ((n + segments - 1) / segments + 31) / 32 * 32;
    const uint32_t K = (uint32_t)((n + len - 1) / len);
    const int kind = sink == CI_SINK_QC       ? SINK_QC
                     : sink == CI_SINK_DIGEST ? SINK_DIGEST
                     : (reinterpret_cast<uintptr_t>(out) & 15u) == 0 && n % 4 == 0 ? SINK_V4
                                                                                   : SINK_SCALAR;
    const DevState st = h.view();
    if (h.xl == CI_XL_XORSHIFT32) return launch_narrow_src<SrcXorshift32>(st, kind, blocks, n, len, K, out, aux, stream);
    if (h.xl == CI_XL_XOR64) return launch_narrow_src<SrcXor64>(st, kind, blocks, n, len, K, out, aux, stream);
    return launch_narrow_src<SrcXor128>(st, kind, blocks, n, len, K, out, aux, stream);
}

}  // namespace

uint64_t split_segments(const ci_states_s &h, uint64_t n, uint64_t requested) {
    const uint64_t groups = h.P / 32;
    uint64_t K = requested;
    if (K == 0) {  // fill about four waves of resident warps
        const uint64_t target = (uint64_t)sm_count() * 64;
        // cheap xor-like segments: fewer, longer ones (the setup's GF(2) jumps
        // cost more than their generation)
        const uint64_t min_len = h.variant == CI_VAR_XOR ? kMinAutoSegment : kMinSegment;
        K = std::max<uint64_t>(1, target / groups);
        K = std::min<uint64_t>(K, std::max<uint64_t>(1, n / min_len));
    }
    K = std::min<uint64_t>(K, kMaxSegments);
    const uint64_t len = ((n + K - 1) / K + 31) / 32 * 32;  // whole staging tiles, 16-byte column offsets
    return (n + len - 1) / len;
}

namespace {

// Whether a call of n iterations of a BBS state is faster whole than in
// segments, by the times of both forms (ns).  Whole: a chain of 390 per output
// up to a warp per scheduler, then by the warps of the fullest one.  In
// segments: a fixed part and the squarings of all warp groups at the split
// kernels' rate.  Whole / in segments, us, written: 32 x 128 55 / 59, x 256 105 /
// 58; 10^4 x 256 105 / 125, x 512 203 / 154; 30000 x 512 266 / 363, x 2048 1041 /
// 901; 2^16 x 512 463 / 499, x 2048 1829 / 1645; digests (written to scratch and
// reduced) 30000 x 1024 511 / 575, 2^16 x 1024 919 / 991, 2^18 x 1024 2931 / 3499.
bool whole_bbs(uint64_t groups, uint64_t n, bool written) {
    const uint64_t sms = (uint64_t)sm_count();
    const bool one_launch = groups >= kOneLaunchGroupsPerSm * sms;
    const uint64_t w = 1 + 51 * groups / (200 * sms);  // the schedulers fill up 2 % before the count says so
    const uint64_t chain = w == 1 ? 390 : 100 + 210 * w + (!written && !one_launch && w >= 3 ? 150 : 0);
    const uint64_t rate = (written ? (one_launch ? 53 : 59) : (one_launch ? 62 : 71)) * groups / sms;
    const uint64_t fixed = (one_launch ? 180000 : 62000 + 110 * groups) + (written ? 0 : 10000);
    return chain <= rate || n * (chain - rate) < fixed;
}

// Segment count a single call uses for a CI_VAR_BBS state.  Written sink, and
// consumer sinks whose outputs fit the scratch (they are written, fixed up and
// reduced): whole by the rule above, else from the GPU size and the form
// split_launch takes; larger consumer
// calls, which generate twice: > 1 only for states that fill less than about
// two waves.  `captured`: calls too short for segments of
// kMinSegment stay one plain launch (a split allocates its workspace, which a
// graph then has to own).
uint64_t split_auto_bbs(const ci_states_s &h, uint64_t n, int sink, bool captured) {
    if (h.variant != CI_VAR_BBS) return 1;
    const uint64_t groups = h.P / 32, sms = (uint64_t)sm_count();
    uint64_t K;
    // consumer sinks whose outputs fit the scratch are written, fixed up and
    // reduced (split_launch), so they take the written rule
    if (sink == CI_SINK_WRITTEN || h.S <= kScratchWords / n) {
        if (whole_bbs(groups, n, sink == CI_SINK_WRITTEN)) return 1;
        // Measured on 2^9 .. 2^13 warp groups of 2^12 .. 2^15 iterations:
        // about ten waves of resident warps (40 per SM) in the one-launch
        // form, four in the three-launch form; segments of at least 256.
        K = groups >= kOneLaunchGroupsPerSm * sms ? (400 * sms + groups / 2) / groups : 160 * sms / groups;
        K = std::min<uint64_t>(K, n / kMinSegment);
        // ... or shorter, down to 64, while the segments are fewer than the
        // resident warps (24 per SM): 32 streams x 4096 82 us, 103 from 128
        // on, 309 from 256 on; x 65536 149 us, 171 down to 32; 1000 x 16384
        // 295 us, 337 up to 16 warps per SM.
        if (!captured) K = std::max<uint64_t>(K, std::min<uint64_t>(n / kMinShortSegment, 24 * sms / groups));
    } else {
        // Larger consumer calls generate twice (pass 1, then pass 2 from the
        // true starts): only states that fill less than about two waves.
        const uint64_t target = sms * 128;
        if (groups * 2 > target) return 1;
        K = std::min<uint64_t>(target / groups, std::max<uint64_t>(1, n / kMinAutoSegment));
    }
    K = std::min<uint64_t>(K, kMaxSegments);
    if (K <= 1) return 1;
    const uint64_t len = ((n + K - 1) / K + 31) / 32 * 32;
    return (n + len - 1) / len;
}

// ... and for any state; 1: unsplit.
uint64_t split_auto(const ci_states_s &h, uint64_t n, int sink, bool captured) {
    if (h.variant == CI_VAR_BBS) return split_auto_bbs(h, n, sink, captured);
    const uint64_t groups = h.P / 32, sms = (uint64_t)sm_count();
    if (h.variant == CI_VAR_BBS16) {
        // Algorithm 5 as printed: each warp is bound by its own eight chains,
        // so only states of at most one warp group per SM gain from more
        // warps (measured, written: 1 group 39x, 32 groups 7x, 128 groups
        // 2.8x faster; 512 groups slower), with about two waves of the split
        // kernels' 16 resident warps per SM and segments of at least 256, or
        // 64 while they fill less than one wave.  Shorter calls run whole, at
        // 87 ns an output (whole / in segments, us: 32 x 512 49 / 77, x 1024 90 /
        // 80; 1000 x 1024 90 / 94, x 1500 131 / 111; 4864 x 1500 131 / 160, x 2048
        // 176 / 169).
        if (groups > sms || n < 880 + 1140 * groups / sms) return 1;
        uint64_t K = std::min<uint64_t>(sms * 32 / groups, n / kMinSegment);
        if (!captured) K = std::max<uint64_t>(K, std::min<uint64_t>(sms * 16 / groups, n / kMinShortSegment));
        K = std::min<uint64_t>(K, kMaxSegments);
        if (K <= 1) return 1;
        const uint64_t len = ((n + K - 1) / K + 31) / 32 * 32;
        return (n + len - 1) / len;
    }
    // xor-likes: only states with no more warp groups than SMs, and calls long
    // enough to pay for the five launches; about one wave of 16 warps per SM,
    // segments of at least 256.  Measured, unsplit against this rule: 32
    // streams x 1000 27 against 51 us, x 4096 107 against 46, 4096 x 4096 107
    // against 76; 1000 x 65536 127 us, 155 with 64 warps per SM; 256 x 65536
    // 77 us, 96 from 1024 iterations on, 94 from 128 on.
    if (h.variant != CI_VAR_XOR || groups > sms || n < kMinXorSplit) return 1;
    uint64_t K = std::min<uint64_t>(sms * 16 / groups, n / kMinSegment);
    K = std::min<uint64_t>(K, kMaxSegments);
    if (K <= 1) return 1;
    const uint64_t len = ((n + K - 1) / K + 31) / 32 * 32;
    return (n + len - 1) / len;
}

}  // namespace

static ci_status launch_status(cudaError_t e) {
    return e == cudaSuccess ? CI_OK : cuda_fail(e, "generation kernel launch");
}

ci_status single_call(const ci_states_s &h, uint64_t n, int sink, uint32_t *out, uint64_t *aux, cudaStream_t stream) {
    const int blocks = narrow_blocks(h, n);
    uint64_t K = blocks ? 1 : split_auto(h, n, sink, false);
    if (blocks || K > 1) {  // the others run the same captured or not, and are not kept from their launch by the question
        const bool captured = stream_capturing(stream);
        if (captured && !jumps_at_hand(h))
            K = 1;
        else if (blocks)
            return launch_status(launch_narrow(h, blocks, n, sink, out, aux, stream));
        else if (captured)
            K = split_auto(h, n, sink, true);
        if (K > 1) return split_launch(h, n, sink, out, n, 0, aux, K, stream);
    }
    return launch_status(sink == CI_SINK_QC       ? launch_fused_qc(h, n, aux, stream)
                         : sink == CI_SINK_DIGEST ? launch_digest(h, n, aux, stream)
                                                  : launch_generate(h, n, out, stream));
}

ci_status split_launch(const ci_states_s &hs, uint64_t n, int sink, uint32_t *out, uint64_t ld, uint64_t col0,
                       uint64_t *aux, uint64_t K, cudaStream_t stream) {
    TraceRange trace("split");
    const ci_states_s *h = &hs;
    const bool b16 = h->variant == CI_VAR_BBS16, bbs = h->variant == CI_VAR_BBS;
    cudaError_t e;
    if (K <= 1) {  // one segment: the caller's state, straight into the sink
        if (b16) {  // one whole call, with its array choice and rotation
            if (sink == CI_SINK_QC) e = launch_fused_qc(*h, n, aux, stream);
            else if (sink == CI_SINK_DIGEST) e = launch_digest(*h, n, aux, stream);
            else if (ld == n && col0 == 0) e = launch_generate(*h, n, out, stream);
            else return fail(CI_E_INVAL, "unsplit CI_VAR_BBS16 output needs ld == n and col0 == 0");
        } else {
            SegSpace none{};
            e = split_run(*h, sink, none, -1, 0, 1, 1, n, n, out, ld, col0, aux, nullptr, stream);
        }
        return e == cudaSuccess ? CI_OK : cuda_fail(e, "split run");
    }
    // BBS-source consumer sinks: generation is the cost, so the outputs are
    // written (and fixed up) once into a scratch of at most kScratchWords
    // words and reduced into the sink, instead of generating the segments
    // twice; larger calls take the regenerate form below.
    if (sink != CI_SINK_WRITTEN && (bbs || b16) && h->S <= kScratchWords / n) {
        uint32_t *rows = nullptr;
        if ((e = workspace_alloc(reinterpret_cast<void **>(&rows), 4 * h->S * n, stream)) != cudaSuccess)
            return cuda_fail(e, "scratch outputs");
        ci_status st = CI_OK;
        if (sink == CI_SINK_DIGEST && (e = cudaMemsetAsync(aux, 0, 8 * h->S, stream)) != cudaSuccess)
            st = cuda_fail(e, "clearing digests");
        if (st == CI_OK) st = split_launch(*h, n, CI_SINK_WRITTEN, rows, n, 0, nullptr, K, stream);
        if (st == CI_OK) {
            // about four waves of 8-warp blocks; chunks of whole 64-output steps
            const uint64_t target = (uint64_t)sm_count() * 8 * 16;
            uint64_t chunks = std::max<uint64_t>(1, std::min<uint64_t>((target + h->S - 1) / h->S, n / 1024));
            const uint64_t clen = ((n + chunks - 1) / chunks + 63) / 64 * 64;
            chunks = (n + clen - 1) / clen;
            const int blocks = (int)std::min<uint64_t>(h->S * chunks, (uint64_t)sm_count() * 16);
            if (sink == CI_SINK_DIGEST)
                k_consume_rows<true><<<blocks, 256, 0, stream>>>(rows, h->S, n, clen, chunks, aux);
            else
                k_consume_rows<false><<<blocks, 256, 0, stream>>>(rows, h->S, n, clen, chunks, aux);
            if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "consuming scratch outputs");
        }
        cudaFreeAsync(rows, stream);
        return st;
    }
    if (h->variant == CI_VAR_XOR && (e = ensure_jump_tables(stream)) != cudaSuccess) return cuda_fail(e, "jump tables");
    const uint64_t groups = h->P / 32;
    const uint64_t len = ((n + K - 1) / K + 31) / 32 * 32;
    const uint64_t len_last = n - (K - 1) * len;

    const uint64_t stride = (h->bytes + 255) / 256 * 256;
    const uint64_t slots = K + (b16 ? 1 : 0);  // BBS16: slot K keeps the call's start (for pass 2)
    // Written BBS outputs are fixed up in place (generation is the cost);
    // xor-like outputs are cheaper to generate again than to read back.
    const bool written = sink == CI_SINK_WRITTEN;
    const bool fixup = written && (bbs || b16);
    const int own_first = b16 ? (int)F_Y16 : (int)F_A, own_count = b16 ? 8 : kOwnWords;
    const uint64_t res_bytes = 8ull * K * h->P;  // per-segment consumer results
    const uint64_t own_bytes = fixup ? 0 : (4ull * own_count + (bbs ? 8ull : 0ull)) * K * h->P;
    const uint64_t lam_bytes = b16 ? 4ull * 8 * h->P : bbs ? (16ull + 4ull * (kCrtWords + kJumpWords)) * h->P : 0;
    uint8_t *ws = nullptr;
    if ((e = workspace_alloc(reinterpret_cast<void **>(&ws), stride * slots + 2 * res_bytes + own_bytes + lam_bytes,
                             stream)) != cudaSuccess)
        return cuda_fail(e, "workspace");
    uint64_t *res1 = reinterpret_cast<uint64_t *>(ws + stride * slots);
    uint64_t *res3 = res1 + K * h->P;
    uint8_t *after = reinterpret_cast<uint8_t *>(res3 + K * h->P);
    OwnSave own{nullptr, nullptr, own_first, own_count};
    if (!fixup) {
        own.u32 = reinterpret_cast<uint32_t *>(after);
        own.u64 = bbs ? reinterpret_cast<uint64_t *>(own.u32 + (uint64_t)own_count * K * h->P) : nullptr;
    }
    uint32_t *lam16 = b16 ? reinterpret_cast<uint32_t *>(after + own_bytes) : nullptr;
    uint64_t *lam64 = bbs ? reinterpret_cast<uint64_t *>(after + own_bytes) : nullptr;
    uint32_t *crt = bbs ? reinterpret_cast<uint32_t *>(lam64 + 2 * h->P) : nullptr;  // residue-form constants

    // Views over the segment states (the caller's, moved).
    auto segment = [&](uint64_t k) {
        ci_states_s moved = *h;
        moved.dev = ws + k * stride;
        return moved.view();
    };
    SegSpace sp;
    sp.v0 = segment(0);
    sp.stride = stride;
    const DevState src = h->view();

    ci_status st = CI_OK;
    if (b16) k_split_lambda16<<<split_block_count(8 * h->P), 256, 0, stream>>>(src, lam16);
    if (bbs) k_split_constants<<<split_block_count(3 * h->P), 256, 0, stream>>>(src, lam64, crt);
    k_split_setup<<<split_block_count(slots * h->P), 256, 0, stream>>>(src, sp, (uint32_t)K, len, h->variant, h->xl,
                                                                       own, lam16, lam64, crt);
    if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "split setup");

    if (st == CI_OK && fixup && groups >= kOneLaunchGroupsPerSm * (uint64_t)sm_count()) {
        // one launch: pass 1 with the fix-ups folded in; then the final state
        uint2 *starts = reinterpret_cast<uint2 *>(res1);  // true starts (slot, x) of segments 1 .. K-1
        unsigned long long *next_unit = reinterpret_cast<unsigned long long *>(res3);
        uint32_t *events = reinterpret_cast<uint32_t *>(next_unit + 1);  // K * groups counts
        const bool v4 = (reinterpret_cast<uintptr_t>(out) & 15u) == 0 && ld % 4 == 0 && col0 % 4 == 0;
        const uint32_t k32 = (uint32_t)K;
        if ((e = cudaMemsetAsync(res3, 0, 8 + 4 * K * groups, stream)) == cudaSuccess) {
            if (bbs)
                e = v4 ? launch_split_run_fix<SrcBbs, SINK_V4>(sp, k32, len, len_last, groups, out, ld, col0, starts,
                                                               events, next_unit, crt, stream)
                       : launch_split_run_fix<SrcBbs, SINK_SCALAR>(sp, k32, len, len_last, groups, out, ld, col0,
                                                                   starts, events, next_unit, crt, stream);
            else
                e = v4 ? launch_split_run_fix<SrcBbs16Seg, SINK_V4>(sp, k32, len, len_last, groups, out, ld, col0,
                                                                    starts, events, next_unit, crt, stream)
                       : launch_split_run_fix<SrcBbs16Seg, SINK_SCALAR>(sp, k32, len, len_last, groups, out, ld, col0,
                                                                        starts, events, next_unit, crt, stream);
        }
        if (e == cudaSuccess) {
            k_split_copy_back<<<split_block_count(12 * h->P), 256, 0, stream>>>(src, segment(K - 1), h->variant);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) st = cuda_fail(e, "split pass 1 with fix-ups");
        cudaFreeAsync(ws, stream);
        return st;
    }
    // pass 1: particular solutions (fix-up: all segments, into their columns;
    // otherwise segments 0 .. K-2, of which only the end states are needed)
    if (st == CI_OK) {
        e = fixup ? split_run(*h, sink, sp, 0, 0, (uint32_t)K, (uint32_t)K, len, len_last, out, ld, col0, nullptr,
                              crt, stream)
                  : split_run(*h, kSinkNone, sp, 0, 0, (uint32_t)K - 1, (uint32_t)K, len, len_last, nullptr, 0,
                              0, res1, crt, stream);
        if (e != cudaSuccess) st = cuda_fail(e, "split pass 1");
    }
    uint2 *starts = reinterpret_cast<uint2 *>(res1);  // K * P (slot, x) pairs, after pass 1
    if (st == CI_OK) {
        const unsigned blocks = (unsigned)groups * kCarryBlocks, threads = 32u * kCarryWarps;
        if (bbs)
            k_split_carry<SrcBbs><<<blocks, threads, 0, stream>>>(sp, (uint32_t)K, len, starts, own);
        else if (b16)
            k_split_carry<SrcBbs16Seg><<<blocks, threads, 0, stream>>>(sp, (uint32_t)K, len, starts, own);
        else
            k_split_carry<SrcXor128><<<blocks, threads, 0, stream>>>(sp, (uint32_t)K, len, starts, own);
        if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "split carry");
    }
    if (st == CI_OK && fixup) {  // homogeneous parts into segments 1 .. K-1, then the final state
        const bool v4 = (reinterpret_cast<uintptr_t>(out) & 15u) == 0 && ld % 4 == 0 && col0 % 4 == 0;
        const int blocks = (int)std::min<uint64_t>((K - 1) * groups, (uint64_t)sm_count() * 8);  // spread over every SM
        if (bbs)
            v4 ? k_split_fixup<SrcBbs, true><<<blocks, 256, 0, stream>>>(sp, starts, (uint32_t)K, len, len_last,
                                                                          groups, out, ld, col0)
               : k_split_fixup<SrcBbs, false><<<blocks, 256, 0, stream>>>(sp, starts, (uint32_t)K, len, len_last,
                                                                           groups, out, ld, col0);
        else
            v4 ? k_split_fixup<SrcBbs16Seg, true><<<blocks, 256, 0, stream>>>(sp, starts, (uint32_t)K, len, len_last,
                                                                               groups, out, ld, col0)
               : k_split_fixup<SrcBbs16Seg, false><<<blocks, 256, 0, stream>>>(sp, starts, (uint32_t)K, len,
                                                                                len_last, groups, out, ld, col0);
        if ((e = cudaGetLastError()) == cudaSuccess)
            k_split_copy_back<<<split_block_count(12 * h->P), 256, 0, stream>>>(src, segment(K - 1), h->variant);
        if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "split fix-up");
        cudaFreeAsync(ws, stream);
        return st;
    }
    if (st == CI_OK && sink == CI_SINK_QC && (e = cudaMemsetAsync(res3, 0, res_bytes, stream)) != cudaSuccess)
        st = cuda_fail(e, "clearing counts");
    if (st == CI_OK) {  // pass 2: every segment from its true start into the sink
        e = split_run(*h, sink, sp, b16 ? (int)K : -1, 0, (uint32_t)K, (uint32_t)K, len, len_last, out, ld, col0,
                      res3, crt, stream);
        if (e != cudaSuccess) st = cuda_fail(e, "split pass 2");
    }
    if (st == CI_OK) {
        k_split_copy_back<<<split_block_count(12 * h->P), 256, 0, stream>>>(src, segment(K - 1), h->variant);
        if (!written)
            k_split_combine<<<(unsigned)((h->S + 255) / 256), 256, 0, stream>>>(res3, aux, h->P, h->S, (uint32_t)K,
                                                                                len, len_last, sink == CI_SINK_DIGEST);
        if ((e = cudaGetLastError()) != cudaSuccess) st = cuda_fail(e, "split finish");
    }
    cudaFreeAsync(ws, stream);
    return st;
}

}  // namespace ci

extern "C" ci_status ci_generate_split(ci_states h, uint64_t n, int32_t sink, void *out_dev,
                                       uint64_t out_capacity, uint32_t n_segments, void *cuda_stream) {
    using namespace ci;
    if (!valid_handle(h)) return fail(CI_E_STATE, "invalid states handle");
    if (sink != CI_SINK_WRITTEN && sink != CI_SINK_QC && sink != CI_SINK_DIGEST)
        return fail(CI_E_INVAL, "unknown sink");
    if (n == 0) return CI_OK;
    if (!out_dev) return fail(CI_E_INVAL, "output is NULL");
    if (sink == CI_SINK_WRITTEN && (n > ~0ull / h->S || out_capacity < h->S * n))
        return fail(CI_E_INVAL, "out_capacity is smaller than n_streams * n");
    if (sink == CI_SINK_QC && (n & 1ull)) return fail(CI_E_INVAL, "quarter-circle sink needs an even length");
    const cudaStream_t cs = static_cast<cudaStream_t>(cuda_stream);
    const uint64_t K = stream_capturing(cs) && !jumps_at_hand(*h) ? 1 : split_segments(*h, n, n_segments);
    if (K <= 1) {  // unsplit: one launch of the tuned single-call kernel
        const cudaError_t e = sink == CI_SINK_QC       ? launch_fused_qc(*h, n, static_cast<uint64_t *>(out_dev), cs)
                              : sink == CI_SINK_DIGEST ? launch_digest(*h, n, static_cast<uint64_t *>(out_dev), cs)
                                                       : launch_generate(*h, n, static_cast<uint32_t *>(out_dev), cs);
        return check_epilogue(cs, e == cudaSuccess ? CI_OK : cuda_fail(e, "unsplit generation kernel launch"));
    }
    if (sink == CI_SINK_WRITTEN)
        return check_epilogue(cs, split_launch(*h, n, sink, static_cast<uint32_t *>(out_dev), n, 0, nullptr, K, cs));
    return check_epilogue(cs, split_launch(*h, n, sink, nullptr, n, 0, static_cast<uint64_t *>(out_dev), K, cs));
}
