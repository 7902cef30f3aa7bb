// icrt.cuh -- the BigInt iCRT as an exact integer matrix product on the
// tensor cores (tcgen05; instructions and operand layout as in tc.cuh).
//
// T = sum_i y_i M_i + NEG_u (mod 2^(64 W)) with M_i = Phat_i mod 2^(64 W) and
// u = round(sum_i y_i / p_i).  In base 2^8, y_i = sum_d a_d 2^(8d) + H (a_d the
// byte less 128 for d < 7, the byte itself, 0 or 1, for d = 7; H collects the
// offsets) and M_i = sum_e m_e 2^(8e) with m_e in [-128, 128): byte column c of T
// is sum_{i,d} a_{i,d} m_{i,c-d}, a matrix product with K = 8 np.  Half the
// primes, at most 32 of them, go to one accumulator and half to another, so a sum
// is at most 32 (7 * 128 * 128 + 128) < 2^22 whatever the primes, and a K step of
// constants makes each accumulator 2^23 + 2^22 + the sum: fp32 is exact and the
// accumulator's word is the sum plus a constant, which is part of NEG_u like H's
// products.  A thread per coefficient adds eight columns' words at their weights to
// a 64-bit word, and carries.
//
// A tile is 128 coefficients: its digits (128 x 8 np, up to 128 KB) stay in shared
// memory while kWords words (80 columns) at a time are formed; their constants
// (8 primes x 80 columns, 10 KB) stream from L2 through a ring of kStages bulk
// copies.  One CTA per SM keeps running over tiles with a role per warp: eight
// warps cut digits (the next tile's residues are in registers by the time its room
// is free), one issues MMAs, one the copies, and four carry the words of one chunk
// while the MMAs of the next one run (two accumulator buffers); a tile's MMAs
// start with its first eight primes' digits.  Measured against 64 x 64-bit products
// on the CUDA cores, N = 2^16, log Q = 1200: region 1 (three products, 43 primes,
// 19 words) 211 -> 55 us, region 2 (two, 64 primes, 38 words) 468 -> 78 us (53 and 76
// under ncu: 33 and 29% of the issue slots, tensor cores 20 and 25% active).  What
// bounds it is shared memory: an MMA reads 4 KB of digits and 2.5 KB of constants
// for 80 columns, beside the copies that bring the constants.
#pragma once
#include "he_internal.h"
#include "modarith.cuh"
#include "tc.cuh"

namespace he {
namespace icrt {

constexpr int kWords = 10;             // words per chunk
constexpr int kCols = 8 * kWords;      // its columns (the N of an MMA)
constexpr int kPiece = kCols * 16;     // bytes of a prime's eight digits against a chunk
constexpr int kStagePrimes = 8;        // primes per copy
constexpr int kStageBytes = kStagePrimes * kPiece;
constexpr int kStages = 6;
constexpr int kMaxNp = 64;
constexpr int kProducers = 256, kEpilogue = 128;
constexpr int kThreads = kEpilogue + kProducers + 64;
constexpr int kLimbs = kMaxNp * tc::kRows / kProducers;  // residues of a tile per producer
constexpr int kUBuf = 4;               // tiles whose u sums are kept
// A word's offset: two accumulators of 2^23 + 2^22 as fp32 words.
constexpr u64 kOff = 2 * (0x4B000000ull + (1ull << 22));

struct Prime {
    uint32_t inv, shift;  // floor(2^(25 + b) / p), b - 32, b = bitlen(p)
};

struct Args {
    const u64 *y;                // [poly][np][N]
    const unsigned char *image;  // [chunk][prime, padded][kCols][8 digits] f16
    const u64 *neg;              // [np + 1][W]
    const Prime *prime;
    u64 *out;                    // [poly][out_stride][N]
    const u64 *d;                // KS: [poly][d_stride][N]
    unsigned *flag;
    int np, W, chunks, polys, out_stride, d_stride, wo, kout, s, N;
};

struct Shared {
    uint64_t a_full[kMaxNp / kStagePrimes], a_free, b_full[kStages], b_free[kStages], d_full[2], d_free[2], drain;
    uint32_t tmem;
    Prime prime[kMaxNp];
    uint32_t usum[kUBuf][2][tc::kRows];
};

__host__ __device__ constexpr int padded(int np) { return (np + kStagePrimes - 1) / kStagePrimes * kStagePrimes; }
// Shared memory: digits, the constant K step of both operands, the ring, the rows NEG_u.
constexpr int kConstA = tc::kRows * 32, kConstB = kCols * 32;
inline int smem_bytes(int np, int W)
{
    return padded(np) * tc::kRows * 16 + kConstA + kConstB + kStages * kStageBytes + (np + 1) * W * (int)sizeof(u64);
}

__device__ __forceinline__ void bar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// Copy `bytes` (multiples of 16, 16-byte aligned) to shared memory; the barrier
// completes its phase with them.
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(tc::smem_u32(bar))
                 : "memory");
}

// The eight digits of y as f16; o7: minus the offsets of the last two, 1024 each and 128
// where the byte is not small.
template <uint32_t o7>
__device__ __forceinline__ uint4 digits(u64 y)
{
    const uint32_t lo = (uint32_t)y, hi = (uint32_t)(y >> 32), e = 0x64646464u;  // f16 1024 + byte
    const uint32_t o = 0xE480E480u;                                               // -1152 twice
    uint4 r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r.x) : "r"(__byte_perm(lo, e, 0x4140)), "r"(o));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r.y) : "r"(__byte_perm(lo, e, 0x4342)), "r"(o));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r.z) : "r"(__byte_perm(hi, e, 0x4140)), "r"(o));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r.w) : "r"(__byte_perm(hi, e, 0x4342)), "r"(o7));
    return r;
}

// KS = false: out[poly] = T mod 2^kout (wo words).  KS = true: out[poly] =
// d[poly] + floor((T + 2^(s-1)) / 2^s) mod 2^kout, the rounding term being part
// of NEG_u.
template <bool KS>
__global__ void __launch_bounds__(kThreads, 1) k_icrt(const Args P)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ Shared S;
    const int warp = threadIdx.x / 32, t = threadIdx.x;
    const int stages = padded(P.np) / kStagePrimes, first = (stages + 1) / 2;  // stages of the first accumulator
    const int per_poly = P.N / tc::kRows, tiles = P.polys * per_poly;
    u64 *NEG = reinterpret_cast<u64 *>(sm + (size_t)padded(P.np) * tc::kRows * 16 + kConstA + kConstB + kStages * kStageBytes);
    unsigned char *A = sm, *CA = A + (size_t)padded(P.np) * tc::kRows * 16, *CB = CA + kConstA, *B = CB + kConstB;

    if (warp == kThreads / 32 - 1) tc::tmem_alloc(&S.tmem, 512);
    if (t == 0) {
        for (int i = 0; i < kMaxNp / kStagePrimes; i++) bar_init(&S.a_full[i], kProducers);
        bar_init(&S.a_free, 1);
        for (int i = 0; i < kStages; i++) {
            bar_init(&S.b_full[i], 1);
            bar_init(&S.b_free[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            bar_init(&S.d_full[i], 2);  // the MMAs, and their thread (which has seen the tile's u sums)
            bar_init(&S.d_free[i], kEpilogue);
        }
        bar_init(&S.drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = t; i < P.np; i += kThreads) S.prime[i] = P.prime[i];
    for (int i = t; i < (P.np + 1) * P.W; i += kThreads) NEG[i] = P.neg[i];
    // digits of the primes that pad np, and the constants' K step: 2048 x 6144
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int i = P.np * tc::kRows + t; i < padded(P.np) * tc::kRows; i += kThreads) reinterpret_cast<uint4 *>(A)[i] = zero;
    for (int i = t; i < 2 * tc::kRows; i += kThreads)
        reinterpret_cast<uint4 *>(CA)[i] = i < tc::kRows ? make_uint4(0x6800u, 0, 0, 0) : zero;
    for (int i = t; i < 2 * kCols; i += kThreads)
        reinterpret_cast<uint4 *>(CB)[i] = i < kCols ? make_uint4(0x6E00u, 0, 0, 0) : zero;
    tc::fence_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tmem;
    bool ok = true;  // a wait that gives up ends its role; the others' give up after it

    if (warp < kEpilogue / 32) {
        // ---- words and carries ----
        griddep_wait();
        const uint32_t lane = tmem + ((uint32_t)warp << 21);
        const int q0 = P.s >> 6, r = P.s & 63, last = P.wo - 1;
        const u64 mask = (P.kout & 63) ? (1ull << (P.kout & 63)) - 1 : ~0ull;
        uint32_t g = 0;  // chunks so far
        int it = 0;
        for (int x = blockIdx.x; x < tiles && ok; x += gridDim.x, it++) {
            const int poly = x / per_poly;
            const size_t n = (size_t)(x - poly * per_poly) * tc::kRows + t;
            u64 *o = P.out + (size_t)poly * P.out_stride * P.N + n;
            const u64 *dp = KS ? P.d + (size_t)poly * P.d_stride * P.N + n : nullptr;
            u64 carry = 0, prev = 0, dc = 0;
            const u64 *neg = nullptr;
            // word w of T
            auto emit = [&](int w, u64 col, u64 dv) {
                if (!KS) {
                    if (w < P.wo) o[(size_t)w * P.N] = w == last ? col & mask : col;
                } else {
                    // output word j = bits [s + 64 j, s + 64 j + 64) of T: words q0 + j and q0 + j + 1
                    const int j = w - q0 - 1;
                    if (j >= 0 && j < P.wo) {
                        const u64 v = r ? (prev >> r) | (col << (64 - r)) : prev;
                        u64 sum = v + dv;
                        const u64 c1 = sum < v ? 1ull : 0ull;
                        sum += dc;
                        dc = c1 + (sum < dc ? 1ull : 0ull);
                        o[(size_t)j * P.N] = j == last ? sum & mask : sum;
                    }
                    prev = col;
                }
            };
            auto dload = [&](int w) {
                const int j = w - q0 - 1;
                return KS && j >= 0 && j < P.wo ? dp[(size_t)j * P.N] : 0ull;
            };
            u64 dv[kWords], dn[kWords];  // the chunk's words of d and the next one's
#pragma unroll
            for (int k = 0; k < kWords; k++) dn[k] = dload(k);
#pragma unroll 1
            for (int ch = 0; ch < P.chunks; ch++, g++) {
                const int buf = g & 1, w0 = ch * kWords;
#pragma unroll
                for (int k = 0; k < kWords; k++) {
                    dv[k] = dn[k];
                    dn[k] = dload(w0 + kWords + k);
                }
                if (!(ok = tc::warp_wait(&S.d_full[buf], (g >> 1) & 1))) break;
                tc::fence_after_sync();
                if (ch == 0) {
                    const uint32_t u = (S.usum[it % kUBuf][0][t] + S.usum[it % kUBuf][1][t] + (1u << 24)) >> 25;
                    neg = NEG + (size_t)u * P.W;
                }
                uint32_t c[2][16];
                auto fetch = [&](uint32_t *p, int k) {
                    tc::tmem_ld8(p, lane + buf * 2 * kCols + 8 * k);
                    tc::tmem_ld8(p + 8, lane + buf * 2 * kCols + kCols + 8 * k);
                };
                fetch(c[0], 0);
#pragma unroll
                for (int k = 0; k < kWords; k++) {
                    tc::tmem_wait_ld();
                    uint32_t *p = c[k & 1];
                    if (k + 1 < kWords) fetch(c[(k + 1) & 1], k + 1);
                    u64 lo = p[0] + p[8], hi = p[4] + p[12];
#pragma unroll
                    for (int b = 1; b < 4; b++) {
                        lo += (u64)(p[b] + p[8 + b]) << (8 * b);
                        hi += (u64)(p[4 + b] + p[12 + b]) << (8 * b);
                    }
                    u64 col = lo + carry;  // both far below 2^63
                    u64 cy = hi >> 32;
                    u64 s = col + (hi << 32);
                    cy += s < col ? 1ull : 0ull;
                    const u64 ng = w0 + k < P.W ? neg[w0 + k] : 0ull;
                    col = s + ng;
                    cy += col < ng ? 1ull : 0ull;
                    carry = cy;
                    if (w0 + k < P.W) emit(w0 + k, col, dv[k]);
                }
                tc::fence_before_sync();
                bar_arrive(&S.d_free[buf]);
            }
            if (KS && ok && P.W <= q0 + P.wo) emit(P.W, 0, dload(P.W));  // bits above T's words are masked
        }
    } else if (warp < (kEpilogue + kProducers) / 32) {
        // ---- digits ----
        griddep_wait();
        const int row = (t - kEpilogue) & 127, half = (t - kEpilogue) >> 7;
        u64 v[kLimbs];
        auto load = [&](int x) {
            const int poly = x / per_poly;
            const u64 *y = P.y + ((size_t)poly * P.np + half) * P.N + (size_t)(x - poly * per_poly) * tc::kRows + row;
#pragma unroll
            for (int k = 0; k < kLimbs; k++) {
                if (2 * k + half < P.np) v[k] = *y;
                y += 2 * (size_t)P.N;
                asm("" : "+l"(y));  // one address, not thirty-two held from tile to tile
            }
        };
        if ((int)blockIdx.x < tiles) load(blockIdx.x);
        int it = 0;
        for (int x = blockIdx.x; x < tiles; x += gridDim.x, it++) {
            if (it && !(ok = tc::bar_wait(&S.a_free, (it - 1) & 1))) break;
            uint32_t f = 0;
#pragma unroll
            for (int k = 0; k < kLimbs; k++) {
                const int i = 2 * k + half;
                if (i < P.np) {
                    const Prime pr = S.prime[i];
                    f += __umulhi((uint32_t)(v[k] >> pr.shift), pr.inv);
                    reinterpret_cast<uint4 *>(A)[i * tc::kRows + row] = digits<0xE400E480u>(v[k]);  // -1024 | -1152
                }
                constexpr int per = kStagePrimes / 2;
                if (k % per == per - 1 && k / per < stages) {  // the stage's primes: its MMAs may start
                    if (k / per == stages - 1) S.usum[it % kUBuf][half][row] = f;
                    tc::fence_smem();
                    tc::fence_before_sync();
                    bar_arrive(&S.a_full[k / per]);
                }
            }
            if (x + (int)gridDim.x < tiles) load(x + gridDim.x);
        }
    } else if (warp == (kEpilogue + kProducers) / 32) {
        // ---- constants ----
        if (t % 32 == 0) {
            uint32_t c = 0;  // copies so far
            for (int x = blockIdx.x; x < tiles && ok; x += gridDim.x)
                for (int k = 0; k < P.chunks * stages; k++, c++) {
                    const int slot = c % kStages;
                    if (c == kStages) griddep_wait();  // as the roles it waits for from here on
                    if (c >= kStages && !(ok = tc::bar_wait(&S.b_free[slot], (c / kStages - 1) & 1))) break;
                    bulk_copy(B + slot * kStageBytes, P.image + (size_t)k * kStageBytes, kStageBytes, &S.b_full[slot]);
                }
            // the copies in flight land before the CTA ends
            for (uint32_t k = c > kStages ? c - kStages : 0; k < c; k++)
                if (!tc::bar_wait(&S.b_full[k % kStages], (k / kStages) & 1)) break;
        }
    } else {
        // ---- MMAs ----
        griddep_wait();  // as the roles it waits for: their time alone counts against its limits
        // the warp keeps together and one lane issues: descriptors stay in
        // uniform registers (issued by a lane of a diverged warp, an MMA took
        // about 115 cycles)
        const uint64_t ca = tc::smem_desc(tc::smem_u32(CA), tc::kRows * 16), cb = tc::smem_desc(tc::smem_u32(CB), kPiece);
        const uint64_t a = tc::smem_desc(tc::smem_u32(A), tc::kRows * 16), b = tc::smem_desc(tc::smem_u32(B), kPiece);
        const uint32_t idesc = tc::mma_idesc(kCols);
        uint32_t slot = 0, turn = 0, g = 0;  // ring slot and its use; chunks so far
        int it = 0;
        for (int x = blockIdx.x; x < tiles && ok; x += gridDim.x, it++) {
            for (int ch = 0; ch < P.chunks && ok; ch++, g++) {
                const int buf = g & 1;
                if (g >= 2 && !(ok = tc::warp_wait(&S.d_free[buf], ((g >> 1) - 1) & 1))) break;
                tc::fence_after_sync();
                const uint32_t d0 = tmem + buf * 2 * kCols;
                if (tc::elect_one()) {
                    tc::mma_f16(d0, ca, cb, idesc, false);
                    tc::mma_f16(d0 + kCols, ca, cb, idesc, false);
                }
                uint64_t as = a;
                for (int st = 0; st < stages; st++) {
                    if (ch == 0 && !(ok = tc::warp_wait(&S.a_full[st], it & 1))) break;
                    if (!(ok = tc::warp_wait(&S.b_full[slot], turn & 1))) break;
                    tc::fence_after_sync();
                    if (tc::elect_one()) {
                        const uint32_t d = st < first ? d0 : d0 + kCols;
                        const uint64_t bs = b + slot * (kStageBytes / 16);
#pragma unroll
                        for (int k = 0; k < kStagePrimes / 2; k++)
                            tc::mma_f16(d, as + 2 * k * tc::kRows, bs + 2 * k * (kPiece / 16), idesc, true);
                        tc::mma_commit(&S.b_free[slot]);
                    }
                    as += kStagePrimes * tc::kRows;
                    if (++slot == kStages) {
                        slot = 0;
                        turn++;
                    }
                }
                if (!ok) break;
                if (tc::elect_one()) {
                    tc::mma_commit(&S.d_full[buf]);
                    bar_arrive(&S.d_full[buf]);
                    if (ch + 1 == P.chunks) tc::mma_commit(&S.a_free);
                }
            }
        }
        // the last arrival lands before the CTA ends
        if (it && ok) ok = tc::warp_wait(&S.a_free, (it - 1) & 1);
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

}  // namespace icrt
}  // namespace he
