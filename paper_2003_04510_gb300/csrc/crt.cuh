// crt.cuh -- the BigInt CRT as an exact integer matrix product on the tensor
// cores (tcgen05; instructions and operand layout as in tc.cuh, digits and barriers
// as in icrt.cuh).
//
// x mod p for x = sum_k byte_k 2^(8k): with a_k = byte_k - 128 and the constants
// C_k = 2^(8k) mod p centred and cut into eight balanced bytes C_{k,c}, column (p, c)
// is sum_k a_k C_{k,c}, at most 8 W 128^2 < 2^22 for W <= 31 words.  One more
// digit of constants makes the accumulator 2^23 + 2^22 + the sum, whose fp32 word is
// the sum plus a constant; a thread per coefficient adds a prime's eight words at
// their weights (below 2^81) and reduces once.  Constants go into `base`.
//
// A CTA keeps the constants of at most kPrimes primes (256 columns) in shared
// memory and runs over tiles of 128 coefficients: eight warps cut digits, one lane
// issues MMAs, sixteen warps (four per TMEM lane quarter, a quarter of the primes each) reduce
// and store; digits and accumulators are doubled, so the three run side by side.
// Measured against 28-bit multiply-adds on the CUDA cores, N = 2^16, log Q = 1200:
// region 1 (four polynomials, 43 primes) 202 -> 52 us in one launch instead of
// four, region 2 (one, 64 primes) 74 -> 23 us (51 and 21 under ncu: 55 and 46% of the
// issue slots, tensor cores 24 and 21% active).  The reducing warps bound it;
// the folding reduction took 61 to 52 us, eight reducing warps instead of sixteen 68.
#pragma once
#include "he_internal.h"
#include "icrt.cuh"
#include "modarith.cuh"
#include "tc.cuh"

namespace he {
namespace crt {

constexpr int kPrimes = 32;  // per CTA
constexpr int kMaxWords = 19;
constexpr int kEpilogue = 512, kProducers = 256;
constexpr int kThreads = kEpilogue + kProducers + 32;
// A pair of neighbouring columns, (w1 << 8) + w0 in 32 bits: the exponent leaves the
// shifted word, and the pair is kPair plus 256 times one sum plus the other, without
// overflow.
constexpr u64 kPair = (((0x4B400000ull << 8) + 0x4B400000ull) & 0xffffffffull);
static_assert(kPair > 257ull * 31 * 8 * 128 * 128 && kPair + 257ull * 31 * 8 * 128 * 128 < (1ull << 32), "pairs of columns");

struct Prime {
    u64 q, mu, base;
    uint32_t s, delta;  // bitlen(q) - 2; 2^b - q (0 if above 31 bits)
};
// Primes of 55 to 57 bits less than 2^31 below their power of two (a context's
// chains are the primes next below it) reduce the words' sum, below 2^81, by two
// foldings at bit b instead of a Barrett quotient.
inline bool folds(const Prime &p) { return p.s >= 53 && p.s <= 55 && p.delta; }

struct Args {
    const u64 *in[4];            // polys, word-major
    u64 *out;                    // [poly][np][N]
    const unsigned char *image;  // [chunk][cores][8 pc][8 digits] f16
    const Prime *prime;          // [np]
    unsigned *flag;
    int wi, W, np, pc, polys, N;  // input words, the image's words, primes, per chunk
};

struct Shared {
    uint64_t a_full[2], a_free[2], d_full[2], d_free[2], drain;
    uint32_t tmem;
    Prime prime[kPrimes];
};

// K of W words and the constants' digit, in core columns of eight.
__host__ __device__ constexpr int cores(int W) { return (W + 2) / 2 * 2; }
// Primes per chunk, an even number: two of them are a multiple of the MMA's 16 columns.
inline int chunk_primes(int np)
{
    const int nch = (np + kPrimes - 1) / kPrimes;
    return ((np + nch - 1) / nch + 1) & ~1;
}
inline int image_bytes(int W, int pc) { return cores(W) * 8 * pc * 16; }
inline int smem_bytes(int W, int pc) { return image_bytes(W, pc) + 2 * cores(W) * tc::kRows * 16; }

// grid: x over CTAs that share the tiles, y over chunks of primes.
template <bool FOLD>
__global__ void __launch_bounds__(kThreads, 1) k_crt(const Args P)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ Shared S;
    const int warp = threadIdx.x / 32, t = threadIdx.x;
    const int nc = cores(P.W), i0 = blockIdx.y * P.pc, cnt = min(P.pc, P.np - i0);
    const int per_poly = P.N / tc::kRows, tiles = P.polys * per_poly;
    const int cols = 8 * P.pc, bbytes = nc * cols * 16, abytes = nc * tc::kRows * 16;
    unsigned char *B = sm, *A = sm + bbytes;

    if (warp == kThreads / 32 - 1) tc::tmem_alloc(&S.tmem, 512);
    if (t == 0) {
        for (int i = 0; i < 2; i++) {
            icrt::bar_init(&S.a_full[i], kProducers / 2);
            icrt::bar_init(&S.a_free[i], 1);
            icrt::bar_init(&S.d_full[i], 1);
            icrt::bar_init(&S.d_free[i], kEpilogue);
        }
        icrt::bar_init(&S.drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::copy_image(B, P.image + (size_t)blockIdx.y * bbytes, bbytes);
    if (t < cnt) S.prime[t] = P.prime[i0 + t];
    // the constants' digit, 2048, and what pads K
    for (int i = t; i < 2 * (nc - P.W) * tc::kRows; i += kThreads) {
        const int b = i / ((nc - P.W) * tc::kRows), r = i % ((nc - P.W) * tc::kRows);
        reinterpret_cast<uint4 *>(A + b * abytes)[P.W * tc::kRows + r] = make_uint4(r < tc::kRows ? 0x6800u : 0u, 0, 0, 0);
    }
    __pipeline_commit();
    __pipeline_wait_prior(0);
    tc::fence_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tmem;
    bool ok = true;  // a wait that gives up ends its role; the others' give up after it

    if (warp < kEpilogue / 32) {
        // ---- residues ----
        griddep_wait();
        const int row = t & 127, part = (P.pc + 3) / 4, u0 = (warp / 4) * part, u1 = min(cnt, u0 + part);
        int it = 0;
        for (int x = blockIdx.x; x < tiles; x += gridDim.x, it++) {
            const int poly = x / per_poly, buf = it & 1;
            u64 *o = P.out + ((size_t)poly * P.np + i0 + u0) * P.N + (size_t)(x - poly * per_poly) * tc::kRows + row;
            const uint32_t lane = tmem + ((uint32_t)(warp & 3) << 21) + buf * 256;
            if (!(ok = tc::warp_wait(&S.d_full[buf], (it >> 1) & 1))) break;
            tc::fence_after_sync();
            uint32_t c[2][8];
            auto put = [&](const uint32_t *p, int u) {
                const Prime &pr = S.prime[u];
                u64 lo = mad_wide((p[3] << 8) + p[2], 1u << 16, pr.base + ((p[1] << 8) + p[0]));  // below 2^58
                const u64 hi = mad_wide((p[7] << 8) + p[6], 1u << 16, (u64)((p[5] << 8) + p[4]));  // below 2^49
                if (FOLD) {
                    const uint32_t sh = pr.s - 30, mask = (1u << sh) - 1;  // b - 32
                    lo += (u64)((uint32_t)hi & mask) << 32;               // bits below b: below 2^59
                    const uint32_t l1 = (uint32_t)(lo >> 32);
                    u64 y = mad_wide((uint32_t)(hi >> sh) + (l1 >> sh), pr.delta, ((u64)(l1 & mask) << 32) | (uint32_t)lo);
                    const uint32_t y1 = (uint32_t)(y >> 32);  // y below 2^b + 2^57
                    y = mad_wide(y1 >> sh, pr.delta, ((u64)(y1 & mask) << 32) | (uint32_t)y);
                    *o = csub(y, pr.q);
                } else {
                    U128 v;
                    v.lo = lo + (hi << 32);
                    v.hi = (hi >> 32) + (v.lo < lo ? 1ull : 0ull);
                    *o = barrett128(v, pr.q, pr.mu, pr.s);
                }
                o += P.N;
            };
            if (u0 < u1) tc::tmem_ld8(c[0], lane + 8 * u0);
            for (int u = u0; u < u1; u += 2) {
                tc::tmem_wait_ld();
                if (u + 1 < u1) tc::tmem_ld8(c[1], lane + 8 * (u + 1));
                put(c[0], u);
                if (u + 1 < u1) {
                    tc::tmem_wait_ld();
                    if (u + 2 < u1) tc::tmem_ld8(c[0], lane + 8 * (u + 2));
                    put(c[1], u + 1);
                }
            }
            tc::fence_before_sync();
            icrt::bar_arrive(&S.d_free[buf]);
        }
    } else if (warp < (kEpilogue + kProducers) / 32) {
        // ---- digits ----
        griddep_wait();
        // each half of the warps takes every other tile: two tiles' words on their way
        const int row = (t - kEpilogue) & 127, buf = (t - kEpilogue) >> 7, step = 2 * gridDim.x;
        u64 v[kMaxWords];
        auto load = [&](int x) {
            const int poly = x / per_poly;
            const u64 *y = (poly < 2 ? poly ? P.in[1] : P.in[0] : poly == 2 ? P.in[2] : P.in[3]) +
                           (size_t)(x - poly * per_poly) * tc::kRows + row;
#pragma unroll
            for (int k = 0; k < kMaxWords; k++) {
                v[k] = k < P.wi ? *y : 0ull;
                y += P.N;
                asm("" : "+l"(y));
            }
        };
        int x = blockIdx.x + buf * gridDim.x;
        if (x < tiles) load(x);
        for (int it = 0; x < tiles; x += step, it++) {
            if (it && !(ok = tc::bar_wait(&S.a_free[buf], (it - 1) & 1))) break;
            uint4 *a = reinterpret_cast<uint4 *>(A + buf * abytes) + row;
#pragma unroll
            for (int k = 0; k < kMaxWords; k++)
                if (k < P.W) a[k * tc::kRows] = icrt::digits<0xE480E480u>(v[k]);
            tc::fence_smem();
            tc::fence_before_sync();
            icrt::bar_arrive(&S.a_full[buf]);
            if (x + step < tiles) load(x + step);
        }
    } else {
        // ---- MMAs: the warp keeps together and one lane issues ----
        griddep_wait();  // as the roles it waits for: their time alone counts against its limits
        const uint64_t b = tc::smem_desc(tc::smem_u32(B), cols * 16);
        const uint32_t idesc = tc::mma_idesc(cols);
        int it = 0;
        for (int x = blockIdx.x; x < tiles; x += gridDim.x, it++) {
            const int buf = it & 1;
            if (it >= 2 && !(ok = tc::warp_wait(&S.d_free[buf], ((it >> 1) - 1) & 1))) break;
            if (!(ok = tc::warp_wait(&S.a_full[buf], (it >> 1) & 1))) break;
            tc::fence_after_sync();
            if (tc::elect_one()) {
                uint64_t as = tc::smem_desc(tc::smem_u32(A + buf * abytes), tc::kRows * 16), bs = b;
                for (int k = 0; k < nc / 2; k++) {
                    tc::mma_f16(tmem + buf * 256, as, bs, idesc, k > 0);
                    as += 2 * tc::kRows;
                    bs += 2 * cols;
                }
                tc::mma_commit(&S.a_free[buf]);
                tc::mma_commit(&S.d_full[buf]);
            }
        }
        // the last arrivals land before the CTA ends
        for (int k = it > 2 ? it - 2 : 0; k < it && ok; k++)
            ok = tc::warp_wait(&S.a_free[k & 1], (k >> 1) & 1);
        if (!ok) {  // products still under way read the operands: a second wait
            if (tc::elect_one()) tc::mma_commit(&S.drain);
            tc::warp_wait(&S.drain, 0);
        }
    }
    if (!ok) *(volatile unsigned *)P.flag = 1;
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == kThreads / 32 - 1) tc::tmem_free(tmem, 512);
}

}  // namespace crt
}  // namespace he
