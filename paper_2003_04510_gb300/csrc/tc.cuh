// tc.cuh -- exact integer matrix products on the fifth-generation tensor cores
// (tcgen05), for the base conversions.
//
// A conversion is out[e][n] = sum_i y_i[n] c[e][i] mod q_e: a matrix product of
// the constants with the residues, exact as integers.  Operands are cut into
// nine-bit digits, which f16 holds exactly: y_i = sum_d a_d 2^(9d) + H with
// a_d in [-256, 256) (the digit minus an offset; H collects the offsets and
// is a constant of the target), c centred mod q with balanced digits in
// [-256, 256).  Column (e, p) of the product collects every pair of a residue
// digit and a constant digit whose constant is [c 2^(9d)]_q: the constant is
// reduced before it is cut, so an output has six planes p of weight 2^(9p)
// whatever the residue digit's weight, not the eleven of a plain product.
// Every plane is an integer of magnitude at most an offset below 2^22 (the context
// checks the actual constants), and one more digit of the residues' rows, a
// constant times a constant, adds 2^23 plus the offset to it: fp32 accumulation is
// exact, and the low 23 bits of the accumulator's word are the plane plus the
// offset.  Six planes are
// recombined and folded at bit b = bitlen(q) by ten instructions, against 24 to
// 36 wide multiply-adds and a Barrett reduction per output on the CUDA cores.
//
// A team of 256 threads takes tiles of 128 coefficients (the M of one
// tcgen05.mma, one TMEM lane each) against at most 24 targets (N = 6 planes x
// targets <= 144 columns), one after another: it cuts the tile's residues into
// digits in shared memory, one thread issues K / 16 MMAs (K = 24 per four
// limbs), and each thread recombines its coefficient's planes for half the
// targets.  Every step of a tile waits for the one before (loads 1300 cycles,
// MMA 600, TMEM reads 350 each), so an SM runs three teams in one CTA that keeps
// its TMEM columns, and each team loads its next tile's residues behind its
// current one.  (A CTA per tile spent a third of its time on launch, TMEM
// allocation and the constants' copy.)
// Measured, CUDA cores against this: ModUp 32.7 -> 18.5 us at N = 2^16, level 24
// (three digits of eight limbs), 174 -> 63 us at 2^17, level 44, 897 -> 496 us for
// 64 jobs at 2^16; the ModDown conversions of the 64 jobs 748 -> 483 us.  What is
// left is the recombination's integer instructions and, below a tile or two per
// team, the chain of one tile.
#pragma once
#include <cuda_pipeline_primitives.h>

#include "he_internal.h"
#include "modarith.cuh"

namespace he {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- TMEM, MMA and barrier instructions --------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols)  // one whole warp
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t cols)  // the warp that allocated
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}
// D[128 x N] (+)= A B^T: f16 operands in shared memory, fp32 accumulators in TMEM.
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc),
                 "r"((uint32_t)accumulate)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(const uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// One lane of the warp, the same at every call.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory writes of this thread become visible to the tensor core.
__device__ __forceinline__ void fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void bar_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Wait for the phase; false after the limit.
constexpr int kTries = 1 << 18;  // about a second: a try that fails takes 3.8 us
__device__ __forceinline__ bool bar_wait(const uint64_t *bar, uint32_t parity, int tries = kTries)
{
    for (int it = 0; it < tries; it++) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(smem_u32(bar)), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}
// The same for a warp that acts on the answer as one.
__device__ __forceinline__ bool warp_wait(const uint64_t *bar, uint32_t parity)
{
    return __all_sync(~0u, bar_wait(bar, parity));
}
// The wait of a team's thread (team_tiles) for a tile's products, which take a
// microsecond.  Some threads may give up and others not; what must not split does not: a
// thread that gives up marks its CTA (end() reports it) and goes on with its team,
// barriers and whole-warp instructions included.  Its outputs are as wrong as the report
// says.  A team has up to 86 tiles, hence a shorter limit (62 ms).  The code around
// the wait is kept this short because the tiles' chain runs through it: an answer shared
// by the warp or the team, or a report from here, cost up to 10 us of a 78 us launch of
// short tiles.
constexpr int kTeamTries = 1 << 14;
__device__ __forceinline__ void team_wait(const uint64_t *bar, uint32_t parity, uint32_t *lost, int tries = kTeamTries)
{
    const bool ok = bar_wait(bar, parity, tries);
    __syncwarp();
    if (!ok) *(volatile uint32_t *)lost = 1;
}

// Consecutive columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t *r, uint32_t addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t *r, uint32_t addr)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major, no swizzle: 8-row x 16-byte core
// matrices of 128 contiguous bytes; `kstep` bytes between core matrices along
// K, 128 bytes along the rows.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t kstep)
{
    return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)(kstep >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
           (1ull << 46);
}
// Instruction descriptor: f16 x f16 -> f32, both operands K-major, M = 128.
__device__ __forceinline__ constexpr uint32_t mma_idesc(uint32_t n)
{
    return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- operands ------------------------------------------------------------------
constexpr int kRows = 128;                    // coefficients per tile
constexpr int kTeam = 256;                    // threads per team
constexpr int kTargets = 24;                  // most targets of a tile
constexpr int kCols = 6 * kTargets + 16;      // TMEM columns of a team: a tile's planes and one more target's

// K of G groups of four limbs (24 digits each) and the digit that adds the
// planes' offset, padded to the MMA's 16.
__host__ __device__ constexpr int k_pad(int groups) { return (24 * groups + 1 + 15) / 16 * 16; }

// The six digits of y minus their offsets, as three f16 pairs: digits 0..4
// nine bits (offset 256), digit 5 the rest, at most ten bits (offset `top`,
// packed twice with 256 in the low half: off5 = -(1024 + 256) | -(1024 + top)).
__device__ __forceinline__ void digits(u64 y, uint32_t off5, uint32_t &p0, uint32_t &p1, uint32_t &p2)
{
    const uint32_t lo = (uint32_t)y, hi = (uint32_t)(y >> 32);
    const uint32_t a = lo, b = __funnelshift_r(lo, hi, 18), c = hi >> 4;
    const uint32_t kExp = 0x64006400u;  // f16 1024 + digit
    const uint32_t o = 0xE500E500u;     // f16 -1280 twice
    const uint32_t u0 = (a & 0x1ffu) | ((a << 7) & 0x01ff0000u) | kExp;
    const uint32_t u1 = (b & 0x1ffu) | ((b << 7) & 0x01ff0000u) | kExp;
    const uint32_t u2 = (c & 0x1ffu) | ((c << 7) & 0x03ff0000u) | kExp;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(p0) : "r"(u0), "r"(o));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(p1) : "r"(u1), "r"(o));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(p2) : "r"(u2), "r"(off5));
}

// Four limbs of one coefficient -> 24 digits = three 16-byte pieces of its row.
// The operand is stored K-piece major: piece k8 (eight digits) of row r at
// (k8 * kRows + r) * 16 bytes, so a warp's rows are consecutive.
__device__ __forceinline__ void put_group(unsigned char *A, int row, int g, const u64 (&y)[4], uint32_t off5)
{
    uint32_t p[12];
#pragma unroll
    for (int i = 0; i < 4; i++) digits(y[i], off5, p[3 * i], p[3 * i + 1], p[3 * i + 2]);
#pragma unroll
    for (int k = 0; k < 3; k++)
        *reinterpret_cast<uint4 *>(A + ((size_t)(3 * g + k) * kRows + row) * 16) =
            make_uint4(p[4 * k], p[4 * k + 1], p[4 * k + 2], p[4 * k + 3]);
}
template <int G>
__device__ __forceinline__ void put_padding(unsigned char *A, int row)
{
#pragma unroll
    for (int k = 3 * G; k < k_pad(G) / 8; k++)
        *reinterpret_cast<uint4 *>(A + ((size_t)k * kRows + row) * 16) =
            make_uint4(k == 3 * G ? 0x6800u : 0u, 0, 0, 0);  // f16 2048, the offset's digit
}

// Copy a constant image (16-byte multiples) to shared memory, all threads.
__device__ __forceinline__ void copy_image(unsigned char *dst, const unsigned char *src, int bytes)
{
    for (int f = threadIdx.x * 16; f < bytes; f += blockDim.x * 16) __pipeline_memcpy_async(dst + f, src + f, 16);
}

// One thread: all MMAs of a tile with an image of `rows` columns
// (a multiple of 16) into TMEM columns [col, col + rows).
template <int G>
__device__ __forceinline__ void issue(uint32_t tmem, const unsigned char *A, const unsigned char *B, uint32_t rows)
{
    const uint32_t a = smem_u32(A), b = smem_u32(B);
#pragma unroll
    for (int k = 0; k < k_pad(G) / 16; k++)
        mma_f16(tmem, smem_desc(a + 2 * k * kRows * 16, kRows * 16), smem_desc(b + 2 * k * rows * 16, rows * 16),
                mma_idesc(rows), k > 0);
}

// ---- recombination ---------------------------------------------------------------
__device__ __forceinline__ u64 mad_wide_s(int32_t a, int32_t b, u64 c)
{
    u64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// One target as the teams read it: TcTarget with its mask, and where its output
// goes.
struct Row {
    u64 base;
    uint32_t delta, mask;  // 2^b - q, 2^shift - 1
    uint32_t shift, off;   // b - 36, words from the job's first output
    u64 pad;
};
__device__ __forceinline__ Row make_row(const TcTarget &t, uint32_t off)
{
    return Row{t.base, t.delta, (1u << t.shift) - 1, t.shift, off, 0};
}

// The accumulator words of one output's planes -> a value congruent to
// sum_p P_p 2^(9p) plus the target's constant, below 3q.  A plane's word is
// 0x4B000000 + offset + P: shifted left by nine, the exponent leaves the word,
// and a pair s = (w1 << 9) + w0 is P0 + 512 P1 plus a constant, in 32 signed bits
// (the last pair in 32 unsigned ones, w4's exponent taken out to make room for
// larger planes).  s45's part at and above bit b is folded by delta = 2^b - q;
// all constants are part of `base`.
__device__ __forceinline__ u64 recombine(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t w4, uint32_t w5,
                                         const Row &t)
{
    const int32_t s01 = (int32_t)((w1 << 9) + w0), s23 = (int32_t)((w3 << 9) + w2);
    const uint32_t s45 = (w5 << 9) + (w4 - 0x4B000000u);
    u64 v = mad_wide(s45 >> t.shift, t.delta, t.base);
    v = mad_wide_s(s23, 1 << 18, v);
    v = mad_wide_s(s01, 1, v);
    return v + ((u64)((s45 & t.mask) << 4) << 32);
}

// Barriers and TMEM of a CTA of NT teams.
template <int NT>
struct Shared {
    uint64_t bar[NT];
    uint32_t tmem, lost;  // lost: a thread of the CTA has given up a wait
};
template <int NT>
__host__ __device__ constexpr uint32_t alloc_cols() { return NT * kCols <= 256 ? 256 : 512; }

// Every thread: TMEM columns, barriers; the caller copies images and targets
// and then calls ready().
template <int NT>
__device__ __forceinline__ void begin(Shared<NT> &s)
{
    static_assert(NT * kCols <= 512, "TMEM");
    if (threadIdx.x / 32 == 0) tmem_alloc(&s.tmem, alloc_cols<NT>());
    if (threadIdx.x == 32) s.lost = 0;
    if (threadIdx.x >= 32 && threadIdx.x < 32 + NT) bar_init(&s.bar[threadIdx.x - 32]);
}
template <int NT>
__device__ __forceinline__ uint32_t ready(Shared<NT> &s)
{
    __pipeline_commit();
    __pipeline_wait_prior(0);
    fence_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    return s.tmem;
}
template <int NT>
__device__ __forceinline__ void end(Shared<NT> &s, unsigned *flag)
{
    fence_before_sync();
    __syncthreads();
    if (threadIdx.x / 32 == 0) {
        if (s.lost) {
            *(volatile unsigned *)flag = 1;
            // products may be under way: operands and TMEM outlive a second wait, for either phase
            for (int i = 0; i < 2 * NT; i++) bar_wait(&s.bar[i / 2], i & 1, kTeamTries);
        }
        __syncwarp();
        tmem_free(s.tmem, alloc_cols<NT>());
    }
}

// One team's tiles x, x + step, ... < tiles.  A: the team's operand buffer; B, B1:
// images of the targets and (EXTRA) of one more.  J supplies the residues and
// takes the outputs of the thread's coefficient n:
//   load(n, half)    issue the loads of the thread's limb groups (half, half + 2)
//   value(k, i)      limb i of the k-th of them
//   start(n)         the values have been cut; the outputs of n come next
//   extra(P)         planes of the extra target (EXTRA)
//   put(u, v, t)     output of target u
template <int G, bool EXTRA, class J>
__device__ __forceinline__ void team_tiles(J &job, unsigned char *A, const unsigned char *B, const unsigned char *B1,
                                           uint32_t rows, uint32_t tmem, const uint64_t *bar, int team, int x,
                                           int step, int tiles, int cnt, const Row *st, uint32_t off5,
                                           uint32_t *lost)
{
    const int t = threadIdx.x - team * kTeam, row = t & 127, half = t >> 7;
    const uint32_t lane = tmem + (((threadIdx.x / 32) & 3u) << 21);  // warp w reads lanes 32 (w mod 4) + its lane
    const int per = ((cnt + 1) / 2 + 1) & ~1, u0 = half * per, u1 = min(cnt, u0 + per);
    if (half) put_padding<G>(A, row);
    uint32_t phase = 0;
    if (x < tiles) job.load((size_t)x * kRows + row, half);
    for (; x < tiles; x += step) {
#pragma unroll
        for (int k = 0; k < (G + 1) / 2; k++)
            if (2 * k + half < G) {
                u64 v[4];
#pragma unroll
                for (int i = 0; i < 4; i++) v[i] = job.value(k, i);
                put_group(A, row, 2 * k + half, v, off5);
            }
        job.start((size_t)x * kRows + row);
        fence_smem();
        fence_before_sync();  // the team's reads of the tile before, and these writes, precede the MMAs
        asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeam) : "memory");
        if (t == 0) {
            fence_after_sync();
            issue<G>(tmem, A, B, rows);
            if (EXTRA) issue<G>(tmem + rows, A, B1, 16);
            mma_commit(bar);
        }
        if (x + step < tiles) job.load((size_t)(x + step) * kRows + row, half);
        team_wait(bar, phase, lost);
        fence_after_sync();
        phase ^= 1;
        if (EXTRA) {
            uint32_t P[8];
            tmem_ld8(P, lane + rows);
            tmem_wait_ld();
            job.extra(P);
        }
        // two targets a step (planes of target u in columns 6u .. 6u + 5), the
        // next two's planes on their way while these are recombined
        uint32_t P[2][12];
        auto fetch = [&](uint32_t *p, int u) {
            tmem_ld8(p, lane + (uint32_t)(6 * u));
            tmem_ld4(p + 8, lane + (uint32_t)(6 * u + 8));
        };
        auto put2 = [&](const uint32_t *p, int u) {
            const Row &a = st[u], &b = st[u + 1];
            job.put(u, recombine(p[0], p[1], p[2], p[3], p[4], p[5], a), a);
            if (u + 1 < u1) job.put(u + 1, recombine(p[6], p[7], p[8], p[9], p[10], p[11], b), b);
        };
        if (u0 < u1) fetch(P[0], u0);
        for (int u = u0; u < u1; u += 4) {
            tmem_wait_ld();
            if (u + 2 < u1) fetch(P[1], u + 2);
            put2(P[0], u);
            if (u + 2 < u1) {
                tmem_wait_ld();
                if (u + 4 < u1) fetch(P[0], u + 4);
                put2(P[1], u + 2);
            }
        }
    }
}

}  // namespace tc
}  // namespace he
