// ntt.cu -- negacyclic NTT / iNTT of batches of limbs on sm_103a.
//
// The transform is the paper's Algo 3 (Cooley-Tukey, twiddles
// TB_W[m + j] = psi^bitrev(m + j), bit-reversed output) with Algo 4's
// butterfly, and its inverse (Gentleman-Sande with TB_invW, then N^-1).
// GPU mapping (the paper's high-radix idea, Sec. 5.3, rebuilt for 64-bit
// words): the log N stages are split into two passes over memory (one for
// N = 2^12).  A pass works on tiles of TE elements, 2^E of them in each
// thread's registers, and runs its stages as rounds of at most E stages, with
// one exchange through shared memory between two rounds.  The strided pass
// (the first forward one, the last inverse one) reads its first round's
// operands from memory straight into registers and writes its last round's
// results straight back: a row of a tile is NG consecutive words, so both are
// coalesced.  The contiguous pass does the same on the side of its early
// stages; on the other side a thread's 2^R words are consecutive, and one
// trip through shared memory turns them into coalesced accesses.
//
// What bounds it: the multiply pipe and the issue slots.  A butterfly is
// about 13 instructions (mul_tw); everything else a pass issues per butterfly
// is overhead, so rounds are as long as the registers allow (16 elements and
// four stages: 32 butterflies per exchange), indices are compile-time offsets
// from one base per round, and twiddles are read where they are used, from
// L1 (the strided pass's few, shared by every tile; the early stages' of a
// contiguous tile) or L2 (the last round's, one set per thread).
//
// Measured against rounds that went through shared memory three times per
// pass with a modified Shoup product (30 instructions per butterfly): 19
// instructions; one HE Mul + rescale 232 -> 212 us at 2^16 (level 24), 1029 ->
// 952 us at 2^17 (level 44), 100 -> 42 us at 2^12; a 64-job batch's forward
// passes over 2660 limbs run at 1.1 and 0.98 T butterflies/s (0.78 and 0.77
// before).
//
// Butterflies are lazy and carry no correction step: the twiddle product is
// congruent to x w and below a bound the context derives for the prime, and
// values are folded only where the exact range analysis says so (NttMod; at
// 2^16 with 54-bit primes the forward transform never folds, at 2^17 once
// between the passes; the inverse folds the sums of each round's last stage).
// The last pass reduces to [0, q) and, for the inverse, multiplies by N^-1
// times a per-limb constant.
//
// Stage / twiddle indexing.  Global stage sigma (m = 2^sigma) pairs j and
// j + N/2^(sigma+1) and uses twiddle m + floor(j / 2^(logN - sigma)).  A pass
// covering stages [s0, s0 + M) sees element j = G * 2^(logN - s0) + k * C + c
// (k < 2^M the in-group index, c < C the column, G the group's high bits); at
// local stage l the twiddle index is 2^(s0+l) + (G << l) + (k >> (M - l)).
// In the strided pass s0 = 0 and G = 0; the contiguous pass has C = 1.
#include <cstring>
#include <utility>

#include <cuda_pipeline_primitives.h>

#include "he_internal.h"
#include "modarith.cuh"

namespace he {

namespace {

constexpr int kSMs = 152;

__device__ __forceinline__ int padi(int e) { return e + (e >> 4); }

struct NttArgs {
    const u64 *src;  // base of group.src offsets
    u64 *dst;        // base of group.dst offsets
    const NttGroup *groups;
    const DevPrime *primes;
    int logN;
    const int *count;  // optional device-side group count (grids sized for a maximum)
    int pdl;           // programmatic dependent launch: 0 off, 1, 2
    // fused final combine (COMBINE passes only)
    JobRef R;
    const DevLevel *levels;
    const ulonglong2 *pinv;
    // fused key-switch sums (kFuseIp passes only): the evaluation key
    // [dnum][2][EL][N], EL = K + L
    const u64 *evk;
    int EL;
};

// 16-byte read-only load that does not allocate in L1 (twiddles read once).
// The table's lines are kept in L2 (evict-last): every HE Mul rereads them.
__device__ __forceinline__ ulonglong2 ld_tw(const ulonglong2 *p) { return ld2_static(p, l2_policy_keep()); }

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Final stages whose twiddle runs the device table stores transposed: the
// last round of the sixteen-element plan's contiguous pass.
__host__ __device__ constexpr int direct_stages(int logN) { return logN >= 16 ? 4 : 3; }

// The tensor product (Fig. 2 region 1 in RNS form: d0 = b1 b2, d1 = a1 b2 +
// a2 b1, d2 = a1 a2 mod q_i) of the contiguous tile `tile` of limb i, as the
// tile load of an inverse contiguous first pass.  The group's limb k carries
// the job (job[k]) and ci[k] = i | comp << 16 | keep << 18: the product comp
// (0: d0, 1: d1, 2: d2) goes to shared memory for the transform, and with
// keep all three are also stored to the job's workspace (d0, d1 for the final
// additions, d2 in the NTT domain for the inner product's own-digit rows).
// Without keep only the product needed is formed (the rescale limbs of d0,
// d1, whose d2 job stores them).
template <int TE, int NT>
__device__ __forceinline__ void tensor_tile(const NttArgs &P, const NttGroup &G, int k, int tile, const DevPrime &pr,
                                            u64 *b)
{
    const int lg = P.logN;
    const BatchItem it = job_item(P.R, (int)G.job[k]);
    const unsigned spec = G.ci[k];
    const int li = (int)(spec & 0xffffu), comp = (int)((spec >> 16) & 3u);
    const bool keep = ((spec >> 18) & 1u) != 0;
    const int l = it.level;
    const DevLevel &lv = P.levels[l];
    const size_t t0 = (size_t)tile * TE;
    const u64 *c1b = it.ct1 + ((size_t)li << lg) + t0, *c1a = it.ct1 + (((size_t)l + li) << lg) + t0;
    const u64 *c2b = it.ct2 + ((size_t)li << lg) + t0, *c2a = it.ct2 + (((size_t)l + li) << lg) + t0;
    u64 *w0 = it.ws + (((size_t)lv.o_d0 + li) << lg) + t0, *w1 = it.ws + (((size_t)lv.o_d1 + li) << lg) + t0;
    u64 *w2 = it.ws + (((size_t)lv.o_d2 + li) << lg) + t0;
    const u64 pol = l2_policy_stream();  // the ciphertexts are read once
    constexpr int PAIRS = TE / 2 / NT;
    static_assert(PAIRS % 2 == 0, "pairs per thread");
    constexpr int UNROLL = NT >= 256 ? 1 : 2;  // registers: the 256-thread tiles run at 64
#pragma unroll UNROLL
    for (int s = 0; s < PAIRS; s++) {
        const int e = 2 * (threadIdx.x + s * NT);
        const int gi = e;
        u64 x, y;
        if (keep) {
            const ulonglong2 b1 = ld2_hint(c1b + gi, pol), a1 = ld2_hint(c1a + gi, pol), b2 = ld2_hint(c2b + gi, pol),
                             a2 = ld2_hint(c2a + gi, pol);
            U128 sx = mul_wide(a1.x, b2.x), sy = mul_wide(a1.y, b2.y);
            mac(sx, a2.x, b1.x);
            mac(sy, a2.y, b1.y);
            const u64 d0x = mul_mod(b1.x, b2.x, pr.q, pr.mu, pr.s), d0y = mul_mod(b1.y, b2.y, pr.q, pr.mu, pr.s);
            const u64 d1x = barrett128(sx, pr.q, pr.mu, pr.s), d1y = barrett128(sy, pr.q, pr.mu, pr.s);
            const u64 d2x = mul_mod(a1.x, a2.x, pr.q, pr.mu, pr.s), d2y = mul_mod(a1.y, a2.y, pr.q, pr.mu, pr.s);
            *reinterpret_cast<ulonglong2 *>(w0 + gi) = make_ulonglong2(d0x, d0y);
            *reinterpret_cast<ulonglong2 *>(w1 + gi) = make_ulonglong2(d1x, d1y);
            *reinterpret_cast<ulonglong2 *>(w2 + gi) = make_ulonglong2(d2x, d2y);
            x = comp == 0 ? d0x : comp == 1 ? d1x : d2x;
            y = comp == 0 ? d0y : comp == 1 ? d1y : d2y;
        } else if (comp == 1) {
            const ulonglong2 b1 = ld2_hint(c1b + gi, pol), a1 = ld2_hint(c1a + gi, pol), b2 = ld2_hint(c2b + gi, pol),
                             a2 = ld2_hint(c2a + gi, pol);
            U128 sx = mul_wide(a1.x, b2.x), sy = mul_wide(a1.y, b2.y);
            mac(sx, a2.x, b1.x);
            mac(sy, a2.y, b1.y);
            x = barrett128(sx, pr.q, pr.mu, pr.s);
            y = barrett128(sy, pr.q, pr.mu, pr.s);
        } else {
            const u64 *u1 = comp == 0 ? c1b : c1a, *u2 = comp == 0 ? c2b : c2a;
            const ulonglong2 v1 = ld2_hint(u1 + gi, pol), v2 = ld2_hint(u2 + gi, pol);
            x = mul_mod(v1.x, v2.x, pr.q, pr.mu, pr.s);
            y = mul_mod(v1.y, v2.y, pr.q, pr.mu, pr.s);
        }
        b[padi(e)] = x;
        b[padi(e + 1)] = y;
    }
}

// The key-switch sum KS_h[e] = sum_j U_j[e] evk_{j,h}[e] mod q_e (Fig. 2
// region 2, the inner product with the evaluation key in the NTT domain) of
// the contiguous tile `tile` of one special limb (or q_{l-1}), as the tile
// load of the inverse contiguous first pass that takes it out of the NTT
// domain: the group's limb k carries the job (job[k]) and ci[k] = e | h << 16.
// U_j[e] is row e of digit j's ModUp output, or row e - K of d2 for the
// digit's own limbs; the products of up to kIpFuseDigits digits are summed in
// 128 bits and reduced once (below 4 q^2 <= 2^116, within barrett128's bound).  The sums are not stored:
// only this transform reads them.  At most kIpFuseDigits digits.

template <int TE, int NT>
__device__ __forceinline__ void ip_tile(const NttArgs &P, const NttGroup &G, int k, int tile, const DevPrime &pr,
                                        u64 *b)
{
    const int lg = P.logN;
    const BatchItem it = job_item(P.R, (int)G.job[k]);
    const unsigned spec = G.ci[k];
    const int e = (int)(spec & 0xffffu), h = (int)((spec >> 16) & 1u);
    const DevLevel &lv = P.levels[it.level];
    const int beta = lv.beta, E = lv.E, K = lv.E - it.level;
    // per digit: the limb of U_j[e] in the workspace (or of d2's row for the
    // digit's own limbs) and the key's limb, as limb indices
    unsigned uo[kIpFuseDigits], ko[kIpFuseDigits];
#pragma unroll
    for (int j = 0; j < kIpFuseDigits; j++) {
        const int jj = j < beta ? j : 0;
        const int lo = lv.dig_lo[jj], nj = lv.dig_n[jj];
        const bool own = e >= K && e - K >= lo && e - K < lo + nj;
        uo[j] = own ? lv.o_d2 + (unsigned)(e - K) : lv.o_u + (unsigned)(jj * E + e);
        ko[j] = (unsigned)((2 * jj + h) * P.EL + e);
    }
    const u64 *ws = it.ws + (size_t)tile * TE, *kb = P.evk + (size_t)tile * TE;
    const u64 pol = l2_policy_stream();  // U and the key are read once
    constexpr int PAIRS = TE / 2 / NT;
    constexpr int UNROLL = NT >= 256 ? 1 : 2;  // registers: the 256-thread tiles run at 64
#pragma unroll UNROLL
    for (int s = 0; s < PAIRS; s++) {
        const int x = 2 * (threadIdx.x + s * NT);
        ulonglong2 u[kIpFuseDigits], w[kIpFuseDigits];
#pragma unroll
        for (int j = 0; j < kIpFuseDigits; j++)
            if (j < beta) {
                u[j] = ld2_hint(ws + ((size_t)uo[j] << lg) + x, pol);
                w[j] = ld2_hint(kb + ((size_t)ko[j] << lg) + x, pol);
            }
        U128 ax = {0, 0}, ay = {0, 0};
#pragma unroll
        for (int j = 0; j < kIpFuseDigits; j++)
            if (j < beta) {
                mac(ax, u[j].x, w[j].x);
                mac(ay, u[j].y, w[j].y);
            }
        b[padi(x)] = barrett128(ax, pr.q, pr.mu, pr.s);
        b[padi(x + 1)] = barrett128(ay, pr.q, pr.mu, pr.s);
    }
}

// Final combine in place of a forward last pass's store: for limb i of the
// group (ModDown output (h, ci) of job G.job[i]),
// out[h][ci] = (d_h[ci] + KS_h[K+ci] P^-1 - z) q_{l-1}^-1 with z the
// transform in shared memory (thread pairs 2 t, +1 at g2 + k gs2 and shared
// word padi(2 t) + k (2 NT + NT / 8)).  PLAIN: out[h][ci] = d_h[ci] +
// (KS_h[K+ci] - z) P^-1, which was a kernel of its own (a rotation at 2^16, level
// 13: 125.4 -> 123.5 us).
template <int TE, int NT, bool PLAIN>
__device__ __forceinline__ void combine_store(const NttArgs &P, const NttGroup &G, int i, const u64 *sm, size_t g2,
                                              size_t gs2, const DevPrime &pr, u64 nq)
{
    const BatchItem it = job_item(P.R, (int)G.job[i]);
    const int ci = (int)(G.ci[i] & 0x7fffffffu), hh = (int)(G.ci[i] >> 31);
    const ulonglong2 pv = P.pinv[ci], qv = PLAIN ? pv : P.levels[it.level].qinv_last[ci];
    // at least any forward-NTT output: d + KS P^-1 (lazy, < 4q) + Cz - z
    // stays positive and below Cz + 5q < 2^64 (ntt_mod leaves 8q of room),
    // and one Shoup product by q_{l-1}^-1 reduces it
    const u64 Cz = pr.nt.cz;
    u64 *o = it.out + ((((size_t)hh * (PLAIN ? it.level : it.level - 1) + ci)) << P.logN) + g2;
    const u64 *dd = P.dst + ((size_t)G.cd[i] << P.logN) + g2, *kk = P.dst + ((size_t)G.cks[i] << P.logN) + g2;
    const u64 *sp = sm + padi(2 * threadIdx.x);
    // four pairs per step: their d and KS loads are all in flight before the first product
    constexpr int PAIRS = TE / 2 / NT, B4 = PAIRS >= 4 ? 4 : PAIRS;
    static_assert(PAIRS % B4 == 0, "pairs per thread");
    for (int b0 = 0; b0 < PAIRS; b0 += B4) {
        ulonglong2 dv[B4], kv[B4];
#pragma unroll
        for (int k = 0; k < B4; k++) {
            dv[k] = *reinterpret_cast<const ulonglong2 *>(dd + (b0 + k) * gs2);
            kv[k] = *reinterpret_cast<const ulonglong2 *>(kk + (b0 + k) * gs2);
        }
#pragma unroll
        for (int k = 0; k < B4; k++) {
            // KS P^-1 lazily in [0, 4q)
            const u64 *z = sp + (b0 + k) * (2 * NT + NT / 8);
            if (PLAIN) {
                *reinterpret_cast<ulonglong2 *>(o + (b0 + k) * gs2) =
                    make_ulonglong2(add_mod(dv[k].x, shoup_canon(kv[k].x + Cz - z[0], pv.x, pv.y, pr.q, nq), pr.q),
                                    add_mod(dv[k].y, shoup_canon(kv[k].y + Cz - z[1], pv.x, pv.y, pr.q, nq), pr.q));
                continue;
            }
            const u64 x = dv[k].x + shoup_approx_nq(kv[k].x, pv.x, pv.y, nq) + Cz - z[0];
            const u64 y = dv[k].y + shoup_approx_nq(kv[k].y, pv.x, pv.y, nq) + Cz - z[1];
            *reinterpret_cast<ulonglong2 *>(o + (b0 + k) * gs2) =
                make_ulonglong2(shoup_canon(x, qv.x, qv.y, pr.q, nq), shoup_canon(y, qv.x, qv.y, pr.q, nq));
        }
    }
}

// Shared memory -> HBM for limb i of the group (same thread walk as
// combine_store), 16-byte stores, with the forward transform's output
// reduction: from any word to [0, q), one fold and two conditional
// subtractions where the prime allows it.
template <int TE, int NT>
__device__ __forceinline__ void final_store(const NttArgs &P, const NttGroup &G, int i, const u64 *sm, size_t g2,
                                            size_t gs2, const DevPrime &pr)
{
    u64 *dst = P.dst + ((size_t)G.dst[i] << P.logN) + g2;
    const bool fast = (pr.nt.flags & kFastFinal) != 0;
    const u64 *sp = sm + padi(2 * threadIdx.x);
#pragma unroll
    for (int k = 0; k < TE / 2 / NT; k++) {
        u64 x = sp[0], y = sp[1];
        if (fast) {
            x = csub(csub(fold_tw(x, pr.nt), 2 * pr.q), pr.q);
            y = csub(csub(fold_tw(y, pr.nt), 2 * pr.q), pr.q);
        } else {
            x = shoup(x, 1, pr.r64, pr.q);
            y = shoup(y, 1, pr.r64, pr.q);
        }
        *reinterpret_cast<ulonglong2 *>(dst) = make_ulonglong2(x, y);
        dst += gs2;
        sp += 2 * NT + NT / 8;
    }
}

// One pass: stages of rounds R0, R1, R2, R3 (forward order, 0: absent; the
// inverse runs them in reverse) on tiles of TE elements of a ring of 2^LOGN,
// each thread holding 2^E of them (E the longest round).  FUSE: kFuseNone;
// kFuseCombine, the final combine in the store loop of the forward contiguous
// last pass (ModDown + rescale limbs), kFusePlain the same after a plain ModDown; kFuseTensor, the tensor product computed
// in place of the inverse contiguous first pass's tile load (d2 limbs and the
// rescale limbs of d0, d1); kFuseIp, the key-switch sums of Fig. 2 region 2
// computed in place of the tile load of the special limbs' inverse contiguous
// first pass.
enum { kFuseNone = 0, kFuseCombine = 1, kFuseTensor = 2, kFuseIp = 3, kFusePlain = 4 };

template <int LOGN_, bool STRIDED_, int R0, int R1, int R2, int R3, int TE_>
struct Pass {
    static constexpr int LOGN = LOGN_, TE = TE_;
    static constexpr bool STRIDED = STRIDED_;
    static constexpr int LOGM = R0 + R1 + R2 + R3, M = 1 << LOGM, NG = TE / M;
    static constexpr int E = cmax(cmax(R0, R1), cmax(R2, R3)), NT = TE >> E;
    static constexpr int S0 = STRIDED ? 0 : LOGN - LOGM;        // first stage
    static constexpr int ROUNDS = R3 ? 4 : R2 ? 3 : 2;
    static constexpr int RL = R3 ? R3 : R2 ? R2 : R1;           // last round in forward order
    static constexpr int TILES = (1 << LOGN) / TE;              // per limb
    static constexpr int TS = LOGN - direct_stages(LOGN);       // stages from TS on are stored transposed
    static constexpr bool WHOLE = LOGM == LOGN;                 // a single pass
    static constexpr int TWN = STRIDED ? M - 1 : NG * ((1 << (LOGM - RL)) - 1);  // staged twiddles
    static constexpr size_t SMEM = sizeof(ulonglong2) * TWN + sizeof(u64) * (TE + TE / 16);
    static_assert(R0 > 0 && R1 > 0, "at least two rounds");
    static_assert(TE % M == 0 && (STRIDED || S0 + LOGM == LOGN), "tiles of whole groups");
};

// Set `si` (of 2^(E-R)) of this thread in the round of stages [L0, L0 + R):
// element v of the set is in-group index k = (khi << (LOGM - L0)) |
// (v << LO) | klo of group (or column) grp, LO = LOGM - L0 - R.  The lowest
// thread bits walk the words that are consecutive in memory.
template <class P, int L0, int R>
struct RoundSet {
    static constexpr int LO = P::LOGM - L0 - R, SPT = 1 << (P::E - R);
    int grp, khi, klo;
    __device__ __forceinline__ explicit RoundSet(int si)
    {
        const int s = threadIdx.x + si * P::NT;
        if (P::STRIDED) {
            grp = s % P::NG;
            klo = (s / P::NG) & ((1 << LO) - 1);
            khi = (s / P::NG) >> LO;
        } else {
            klo = s & ((1 << LO) - 1);
            khi = (s >> LO) & ((1 << L0) - 1);
            grp = s >> (LO + L0);
        }
    }
    __device__ __forceinline__ int k() const { return (khi << (P::LOGM - L0)) | klo; }
    // tile-linear index of element 0, and the step to element v
    __device__ __forceinline__ int lin() const { return P::STRIDED ? k() * P::NG + grp : grp * P::M + k(); }
    static __device__ __forceinline__ constexpr int step(int v) { return (v << LO) * (P::STRIDED ? P::NG : 1); }
    // word of the limb
    __device__ __forceinline__ size_t word(int tile) const
    {
        return P::STRIDED ? ((size_t)k() << (P::LOGN - P::LOGM)) + (size_t)(tile * P::NG + grp)
                          : (size_t)tile * P::TE + lin();
    }
    static __device__ __forceinline__ constexpr size_t wstep(int v)
    {
        return P::STRIDED ? (size_t)(v << LO) << (P::LOGN - P::LOGM) : (size_t)step(v);
    }
};

// Shared-memory words of a set: one pad word per 16.  Element v's offset has
// no bit in common with element 0's index, so the padding of the sum splits
// into the base's and a compile-time one.
template <class P, int L0, int R>
__device__ __forceinline__ void smem_put(u64 *sm, const u64 (&a)[1 << P::E])
{
    using S = RoundSet<P, L0, R>;
#pragma unroll
    for (int si = 0; si < S::SPT; si++) {
        u64 *b = sm + padi(S(si).lin());
#pragma unroll
        for (int v = 0; v < (1 << R); v++) b[S::step(v) + (S::step(v) >> 4)] = a[(si << R) + v];
    }
}
template <class P, int L0, int R>
__device__ __forceinline__ void smem_get(const u64 *sm, u64 (&a)[1 << P::E])
{
    using S = RoundSet<P, L0, R>;
#pragma unroll
    for (int si = 0; si < S::SPT; si++) {
        const u64 *b = sm + padi(S(si).lin());
#pragma unroll
        for (int v = 0; v < (1 << R); v++) a[(si << R) + v] = b[S::step(v) + (S::step(v) >> 4)];
    }
}
template <class P, int L0, int R>
__device__ __forceinline__ void mem_get(const u64 *src, int tile, u64 (&a)[1 << P::E])
{
    using S = RoundSet<P, L0, R>;
#pragma unroll
    for (int si = 0; si < S::SPT; si++) {
        const u64 *b = src + S(si).word(tile);
#pragma unroll
        for (int v = 0; v < (1 << R); v++) a[(si << R) + v] = b[S::wstep(v)];
    }
}

// Base and step (per j) of the twiddles of local stage l = L0 + lp for the
// sets with T0 = (G << L0) + khi: twiddle j of the stage is entry
// t = (T0 << lp) + j of the run of stage sigma.  The runs of stages
// sigma >= TS are stored transposed (with d = sigma - TS, entry t at
// (t mod 2^d) 2^TS + floor(t / 2^d)), so that a warp whose sets are
// consecutive reads consecutive entries per j.
template <class P, int L0>
__device__ __forceinline__ const ulonglong2 *tw_entry(const ulonglong2 *twg, int T0, int lp, int j)
{
    const int sigma = P::S0 + L0 + lp, d = sigma - P::TS;
    const ulonglong2 *run = twg + ((size_t)1 << sigma);
    if (d <= 0) return run + ((size_t)T0 << lp) + j;
    if (d <= lp) return run + ((size_t)(j & ((1 << d) - 1)) << P::TS) + ((size_t)T0 << (lp - d)) + (j >> d);
    const int e = d - lp;
    return run + ((size_t)(((T0 & ((1 << e) - 1)) << lp) + j) << P::TS) + (T0 >> e);
}

// Staged twiddles (shared memory): the strided pass keeps TB_W[1, M), which
// every tile uses; the contiguous pass the runs of its tile for the stages
// before the last round, stage l of group grp at NG (2^l - 1) + (grp << l).
template <class P>
__device__ __forceinline__ void stage_twiddles(ulonglong2 *tw, const ulonglong2 *twg, int tile)
{
    if constexpr (P::STRIDED) {
        for (int f = threadIdx.x; f < P::TWN; f += P::NT) __pipeline_memcpy_async(&tw[f], &twg[1 + f], 16);
    } else {
#pragma unroll
        for (int l = 0; l < P::LOGM - P::RL; l++)
            for (int f = threadIdx.x; f < (P::NG << l); f += P::NT)
                __pipeline_memcpy_async(&tw[P::NG * ((1 << l) - 1) + f],
                                        tw_entry<P, 0>(twg, 0, l, tile * (P::NG << l) + f), 16);
    }
    __pipeline_commit();
}

// Where a round's twiddles come from: the staged ones, or registers loaded
// ahead (the contiguous pass's last round, whose twiddles one thread uses
// once: entry 2^lp - 1 + j of stage L0 + lp).
template <class P, int L0>
struct TwSmem {
    const ulonglong2 *tw;
    int grp, khi;
    __device__ __forceinline__ ulonglong2 get(int lp, int j) const
    {
        const int l = L0 + lp;
        return P::STRIDED ? tw[(1 << l) - 1 + (khi << lp) + j]
                          : tw[P::NG * ((1 << l) - 1) + (grp << l) + (khi << lp) + j];
    }
};
template <int R>
struct TwRegs {
    ulonglong2 w[(1 << R) - 1];
    __device__ __forceinline__ ulonglong2 get(int lp, int j) const { return w[(1 << lp) - 1 + j]; }
};
// Stages [LP0, LP1) of the last round's twiddles of set si -> registers.
template <class P, int LP0, int LP1>
__device__ __forceinline__ void load_last(TwRegs<P::RL> &t, const ulonglong2 *twg, int tile, int si)
{
    constexpr int L0 = P::LOGM - P::RL;
    const RoundSet<P, L0, P::RL> st(si);
    const int T0 = ((tile * P::NG + st.grp) << L0) + st.khi;
#pragma unroll
    for (int lp = LP0; lp < LP1; lp++)
#pragma unroll
        for (int j = 0; j < (1 << lp); j++) t.w[(1 << lp) - 1 + j] = ld_tw(tw_entry<P, L0>(twg, T0, lp, j));
}

// Stage L0 + LP of a round on one set of the thread's registers.
template <int R, int LP, bool INV, class TW>
__device__ __forceinline__ void stage_regs(u64 *x, const TW &tw, const NttMod &km)
{
    constexpr int H = 1 << (R - 1 - LP);
#pragma unroll
    for (int j = 0; j < (1 << LP); j++) {
        const ulonglong2 w = tw.get(LP, j);
#pragma unroll
        for (int v = 0; v < H; v++) {
            const int i = (j << (R - LP)) + v;
            if (INV) gs_bfly(x[i], x[i + H], w, km);
            else ct_bfly(x[i], x[i + H], w, km);
        }
    }
    if (!INV && R > 2 && LP == 1 && (km.flags & kFwdFoldSecond)) {
#pragma unroll
        for (int v = 0; v < (1 << R); v++) x[v] = fold_tw(x[v], km);
    }
    if (INV && R > 2 && LP == R - 2 && (km.flags & kInvFoldSecond)) {
#pragma unroll
        for (int v = 0; v < (1 << R); v++)
            if (!(v & H)) x[v] = fold_tw(x[v], km);
    }
}

template <int R, bool INV, class TW, int... LP>
__device__ __forceinline__ void stages_regs(std::integer_sequence<int, LP...>, u64 *x, const TW &tw, const NttMod &km)
{
    (stage_regs<R, INV ? R - 1 - LP : LP, INV>(x, tw, km), ...);
}

// All stages of a round on one set.
template <int R, bool INV, class TW>
__device__ __forceinline__ void set_stages(u64 *x, const TW &tw, const NttMod &km)
{
    stages_regs<R, INV>(std::make_integer_sequence<int, R>(), x, tw, km);
    if (!INV && (km.flags & kFwdFoldRound)) {
#pragma unroll
        for (int v = 0; v < (1 << R); v++) x[v] = fold_tw(x[v], km);
    }
    if (INV) {
        // the sums of the last stage; the products only where the prime needs it
#pragma unroll
        for (int v = 0; v < (1 << R) / 2; v++) x[v] = fold_tw(x[v], km);
        if (km.flags & kInvFoldAll) {
#pragma unroll
            for (int v = (1 << R) / 2; v < (1 << R); v++) x[v] = fold_tw(x[v], km);
        }
    }
}

// The stages [L0, L0 + R) on the thread's registers, twiddles staged.
template <class P, int L0, int R, bool INV>
__device__ __forceinline__ void round_regs(u64 (&a)[1 << P::E], const ulonglong2 *tw, const NttMod &km)
{
    using S = RoundSet<P, L0, R>;
#pragma unroll
    for (int si = 0; si < S::SPT; si++) {
        const S st(si);
        const TwSmem<P, L0> t = {tw, st.grp, st.khi};
        set_stages<R, INV>(a + (si << R), t, km);
    }
}

// L2 prefetch of the lines the contiguous pass's last round will read (one
// thread per 128-byte line); issued when a CTA starts, before it waits for the
// previous kernel.
template <class P>
__device__ __forceinline__ void prefetch_last_round(const ulonglong2 *twg, int tile)
{
    constexpr int L0 = P::LOGM - P::RL;
    using S = RoundSet<P, L0, P::RL>;
    constexpr int e = P::S0 + L0 - P::TS;  // consecutive entries: the sets whose floor(T0 / 2^e) differ
#pragma unroll
    for (int si = 0; si < S::SPT; si++) {
        const S st(si);
        const int T0 = ((tile * P::NG + st.grp) << L0) + st.khi;
        if ((T0 >> (e > 0 ? e : 0)) & 7) continue;
#pragma unroll
        for (int lp = 0; lp < P::RL; lp++)
#pragma unroll
            for (int j = 0; j < (1 << lp); j++)
                asm volatile("prefetch.global.L2::evict_last [%0];" ::"l"(tw_entry<P, L0>(twg, T0, lp, j)));
    }
}

// Resident CTAs per SM the register allocation is bounded for.
__host__ __device__ constexpr int ntt_min_blocks(int nt) { return nt >= 512 ? 1 : nt >= 256 ? 4 : nt >= 128 ? 5 : 8; }

template <class P, int R0, int R1, int R2, int R3, bool INV, int FUSE, int MIN = ntt_min_blocks(P::NT)>
__global__ void __launch_bounds__(P::NT, MIN) k_ntt_pass(const NttArgs A)
{
    constexpr bool STRIDED = P::STRIDED, COMBINE = FUSE == kFuseCombine || FUSE == kFusePlain;
    constexpr bool COMPUTED = FUSE == kFuseTensor || FUSE == kFuseIp;  // the tile load computes its words
    constexpr bool FIRST = P::WHOLE || STRIDED != INV, LAST = P::WHOLE || STRIDED == INV;
    static_assert(!COMBINE || (LAST && !INV && !STRIDED), "the combine follows a forward contiguous last pass");
    static_assert(!COMPUTED || (FIRST && INV && !STRIDED), "computed tiles feed an inverse contiguous first pass");
    constexpr int TE = P::TE, NT = P::NT, RL = P::RL, LL = P::LOGM - RL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ulonglong2 *tw = reinterpret_cast<ulonglong2 *>(smem_raw);
    u64 *sm = reinterpret_cast<u64 *>(tw + P::TWN);

    const int gidx = blockIdx.x / P::TILES, tile = blockIdx.x % P::TILES;
    if (A.count && gidx >= *A.count) return idle_exit();
    const NttGroup &G = A.groups[gidx];
    const int nl = (int)G.nl;
    const DevPrime pr = A.primes[G.prime];
    const NttMod &km = pr.nt;
    const u64 nq = 0ull - pr.q;
    const ulonglong2 *twg = INV ? pr.iw : pr.w;
    // the tables are static: staged, and the last round's lines brought to L2,
    // while the previous kernel still runs
    stage_twiddles<P>(tw, twg, tile);
    if (!STRIDED) prefetch_last_round<P>(twg, tile);
    // the limbs come from the previous kernels; the pass that streams the key
    // (kFuseIp) does not launch its successor early, whose waiting CTAs would
    // hold SM slots its last loads need (measured: 2^17 985 against 992 us)
    griddep_wait(A.pdl >= 1 && FUSE != kFuseIp);
    const size_t g2 = (size_t)tile * TE + 2 * threadIdx.x, gs2 = 2 * NT;  // coalesced pairs of a contiguous tile

    using SL = RoundSet<P, LL, RL>;
    for (int i = 0; i < nl; i++) {
        const u64 *src = FIRST ? A.src + ((size_t)G.src[i] << P::LOGN) : A.dst + ((size_t)G.dst[i] << P::LOGN);
        u64 *dst = A.dst + ((size_t)G.dst[i] << P::LOGN);
        u64 a[1 << P::E];
        if constexpr (!INV) {
            mem_get<P, 0, R0>(src, tile, a);
            if (i == 0) __pipeline_wait_prior(0);
            __syncthreads();  // the staged twiddles; the previous limb's words have been read
            round_regs<P, 0, R0, false>(a, tw, km);
            smem_put<P, 0, R0>(sm, a);
            if constexpr (P::ROUNDS > 2) {
                __syncthreads();
                smem_get<P, R0, R1>(sm, a);
                round_regs<P, R0, R1, false>(a, tw, km);
                smem_put<P, R0, R1>(sm, a);  // the words this thread read
            }
            if constexpr (P::ROUNDS > 3) {
                __syncthreads();
                smem_get<P, R0 + R1, R2>(sm, a);
                round_regs<P, R0 + R1, R2, false>(a, tw, km);
                smem_put<P, R0 + R1, R2>(sm, a);
            }
            if constexpr (STRIDED) {
                __syncthreads();
                smem_get<P, LL, RL>(sm, a);
                round_regs<P, LL, RL, false>(a, tw, km);
                const bool mid = (km.flags & kFwdFoldPass) != 0;
#pragma unroll
                for (int si = 0; si < SL::SPT; si++) {
                    u64 *d = dst + SL(si).word(tile);
#pragma unroll
                    for (int v = 0; v < (1 << RL); v++) {
                        u64 x = a[(si << RL) + v];
                        if (mid) x = fold_tw(x, km);
                        d[SL::wstep(v)] = x;
                    }
                }
            } else {
                // the last round's twiddles but its last stage's travel while the
                // words are exchanged, the last stage's during the stages before it
                TwRegs<RL> t;
                load_last<P, 0, RL - 1>(t, twg, tile, 0);
                __syncthreads();
                smem_get<P, LL, RL>(sm, a);
#pragma unroll
                for (int si = 0; si < SL::SPT; si++) {
                    if (si) load_last<P, 0, RL - 1>(t, twg, tile, si);
                    load_last<P, RL - 1, RL>(t, twg, tile, si);
                    set_stages<RL, false>(a + (si << RL), t, km);
                }
                smem_put<P, LL, RL>(sm, a);
                __syncthreads();
                if constexpr (COMBINE) combine_store<TE, NT, FUSE == kFusePlain>(A, G, i, sm, g2, gs2, pr, nq);
                else final_store<TE, NT>(A, G, i, sm, g2, gs2, pr);
            }
        } else {
            if constexpr (STRIDED) {
                mem_get<P, LL, RL>(src, tile, a);
                if (i == 0) __pipeline_wait_prior(0);
                __syncthreads();  // as above
                round_regs<P, LL, RL, true>(a, tw, km);
            } else {
                TwRegs<RL> t;
                if constexpr (!COMPUTED) load_last<P, RL - 1, RL>(t, twg, tile, 0);
                if (i) __syncthreads();  // the previous limb's words have been read
                if constexpr (FUSE == kFuseTensor) {
                    tensor_tile<TE, NT>(A, G, i, tile, pr, sm);
                } else if constexpr (FUSE == kFuseIp) {
                    ip_tile<TE, NT>(A, G, i, tile, pr, sm);
                } else {
                    const u64 *p = src + (size_t)tile * TE + threadIdx.x;
                    u64 *d = sm + padi(threadIdx.x);
#pragma unroll
                    for (int k = 0; k < TE / NT; k++) __pipeline_memcpy_async(d + k * (NT + NT / 16), p + k * NT, 8);
                    __pipeline_commit();
                }
                if constexpr (COMPUTED) load_last<P, RL - 1, RL>(t, twg, tile, 0);
                __pipeline_wait_prior(0);
                __syncthreads();
                smem_get<P, LL, RL>(sm, a);
#pragma unroll
                for (int si = 0; si < SL::SPT; si++) {
                    if (si) load_last<P, RL - 1, RL>(t, twg, tile, si);
                    load_last<P, 0, RL - 1>(t, twg, tile, si);
                    set_stages<RL, true>(a + (si << RL), t, km);
                }
            }
            smem_put<P, LL, RL>(sm, a);
            __syncthreads();
            if constexpr (P::ROUNDS > 3) {
                smem_get<P, R0 + R1, R2>(sm, a);
                round_regs<P, R0 + R1, R2, true>(a, tw, km);
                smem_put<P, R0 + R1, R2>(sm, a);
                __syncthreads();
            }
            if constexpr (P::ROUNDS > 2) {
                smem_get<P, R0, R1>(sm, a);
                round_regs<P, R0, R1, true>(a, tw, km);
                smem_put<P, R0, R1>(sm, a);
                __syncthreads();
            }
            smem_get<P, 0, R0>(sm, a);
            round_regs<P, 0, R0, true>(a, tw, km);
            const u64 sc = G.scale[i], scs = G.scale_sh[i];
            using S = RoundSet<P, 0, R0>;
#pragma unroll
            for (int si = 0; si < S::SPT; si++) {
                u64 *d = dst + S(si).word(tile);
#pragma unroll
                for (int v = 0; v < (1 << R0); v++) {
                    const u64 x = a[(si << R0) + v];
                    d[S::wstep(v)] = LAST ? shoup_canon(x, sc, scs, pr.q, nq) : x;
                }
            }
        }
    }
}

// ngroups == 0 only sets the kernel's shared-memory limit (no launch).
template <class P, int R0, int R1, int R2, int R3, bool INV, int FUSE, int MIN>
cudaError_t launch_pass(const NttArgs &a, int ngroups, cudaStream_t st)
{
    auto kern = k_ntt_pass<P, R0, R1, R2, R3, INV, FUSE, MIN>;
    static bool configured = false;  // once per instantiation
    if (!configured) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::SMEM);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    if (ngroups == 0) return cudaSuccess;
    launch_k(a.pdl != 0, kern, dim3(ngroups * P::TILES), dim3(P::NT), P::SMEM, st, a);
    return cudaGetLastError();
}

// The ring of one tile (2^12, 512 threads) has a second form, of two CTAs per SM at 64
// registers, for more CTAs than SMs: 200 jobs of 8-limb digits (levels 2 to 16) 938 -> 813
// us, 512 jobs of three limbs 818 -> 691 us of kernels.  Up to one CTA per SM the registers
// (116 to 124) are worth more: 32 jobs of the first kind 177 us, 188 at 64 registers.  A
// batch graph's grid is that of a full batch at the highest level (its launches are
// smaller: 16 jobs 110 us, 119 at 64 registers), so it takes that form from two CTAs per SM.
template <int LOGN, bool STRIDED, bool INV, int FUSE, int TE, int R0, int R1, int R2 = 0, int R3 = 0>
cudaError_t run_pass(const NttArgs &a, int ngroups, cudaStream_t st)
{
    using P = Pass<LOGN, STRIDED, R0, R1, R2, R3, TE>;
    constexpr int MIN = ntt_min_blocks(P::NT);
    if constexpr (MIN == 1) {
        if (ngroups == 0) {
            const cudaError_t e = launch_pass<P, R0, R1, R2, R3, INV, FUSE, 2>(a, 0, st);
            if (e != cudaSuccess) return e;
        } else if (ngroups * P::TILES > (a.count ? 2 : 1) * kSMs) {
            return launch_pass<P, R0, R1, R2, R3, INV, FUSE, 2>(a, ngroups, st);
        }
    }
    return launch_pass<P, R0, R1, R2, R3, INV, FUSE, MIN>(a, ngroups, st);
}

// The two passes of each ring size: the strided one covers the first stages
// (forward order), the contiguous one the rest.  N = 2^12 is a single
// contiguous pass.  Rounds of four stages (sixteen elements per thread) where
// the multiply pipe bounds the pass; rounds of at most three (eight elements,
// twice the warps) where memory latency does, in the passes that compute
// their tile from many streams, and for the nine stages of 2^17.
template <bool STRIDED, bool INV, int FUSE>
cudaError_t pass(int logN, const NttArgs &a, int ng, cudaStream_t st)
{
    constexpr bool COMPUTED = FUSE == kFuseTensor || FUSE == kFuseIp;
#define HE_PASS(...) run_pass<__VA_ARGS__>(a, ng, st)
    if constexpr (STRIDED) {
        switch (logN) {
        case 13: return HE_PASS(13, true, INV, FUSE, 2048, 4, 3);
        case 14: return HE_PASS(14, true, INV, FUSE, 2048, 4, 3);
        case 15: return HE_PASS(15, true, INV, FUSE, 2048, 4, 4);
        case 16: return HE_PASS(16, true, INV, FUSE, 2048, 4, 4);
        case 17: return HE_PASS(17, true, INV, FUSE, 2048, 3, 3, 3);
        default: return cudaErrorInvalidValue;
        }
    } else if constexpr (COMPUTED) {
        switch (logN) {
        case 12: return HE_PASS(12, false, INV, FUSE, 4096, 3, 3, 3, 3);
        case 13: return HE_PASS(13, false, INV, FUSE, 2048, 3, 3);
        case 14: return HE_PASS(14, false, INV, FUSE, 2048, 2, 3, 2);
        case 15: return HE_PASS(15, false, INV, FUSE, 2048, 2, 3, 2);
        case 16: return HE_PASS(16, false, INV, FUSE, 2048, 2, 3, 3);
        case 17: return HE_PASS(17, false, INV, FUSE, 2048, 2, 3, 3);
        default: return cudaErrorInvalidValue;
        }
    } else {
        switch (logN) {
        case 12: return HE_PASS(12, false, INV, FUSE, 4096, 3, 3, 3, 3);
        case 13: return HE_PASS(13, false, INV, FUSE, 2048, 3, 3);
        case 14: return HE_PASS(14, false, INV, FUSE, 2048, 4, 3);
        case 15: return HE_PASS(15, false, INV, FUSE, 2048, 4, 3);
        case 16: return HE_PASS(16, false, INV, FUSE, 2048, 4, 4);
        case 17: return HE_PASS(17, false, INV, FUSE, 2048, 4, 4);
        default: return cudaErrorInvalidValue;
        }
    }
#undef HE_PASS
}

// The whole transform; ngroups == 0 configures its kernels.
template <bool INV, int FUSE>
cudaError_t transform(const he_ctx *c, const NttArgs &a, int ng, cudaStream_t st, const char *tag)
{
    static const char *const kMark[4] = {"", "", ".tensor_inv", ".ip_inv"};
    const int lg = c->logN;
    if (lg == 12) {
        const cudaError_t e = pass<false, INV, FUSE>(lg, a, ng, st);
        if (ng) {
            if (FUSE == kFuseTensor || FUSE == kFuseIp) prof_mark(c, st, tag, kMark[FUSE]);
            else prof_mark(c, st, tag, INV ? ".inv" : FUSE == kFuseNone ? ".fwd" : ".fwd_combine");
        }
        return e;
    }
    cudaError_t e = INV ? pass<false, true, INV ? FUSE : kFuseNone>(lg, a, ng, st)
                        : pass<true, false, kFuseNone>(lg, a, ng, st);
    if (e != cudaSuccess) return e;
    if (ng)
        prof_mark(c, st, tag, !INV ? ".fwd_pass1" : FUSE == kFuseTensor ? ".tensor_inv_pass1" : FUSE == kFuseIp ? ".ip_inv_pass1" : ".inv_pass1");
    e = INV ? pass<true, true, kFuseNone>(lg, a, ng, st) : pass<false, false, INV ? kFuseNone : FUSE>(lg, a, ng, st);
    if (ng) prof_mark(c, st, tag, INV ? ".inv_pass2" : FUSE == kFuseNone ? ".fwd_pass2" : ".fwd_pass2_combine");
    return e;
}

NttArgs ntt_args(const he_ctx *c, const u64 *src, u64 *dst, const NttGroup *groups, const int *dev_count)
{
    NttArgs a;
    memset(&a, 0, sizeof(a));
    a.src = src;
    a.dst = dst;
    a.groups = groups;
    a.primes = c->d_primes;
    a.logN = c->logN;
    a.count = dev_count;
    a.pdl = c->pdl;
    return a;
}

}  // namespace

cudaError_t launch_ntt_tensor(const he_ctx *c, u64 *base, const NttGroup *groups, int ngroups, const JobRef &R,
                              cudaStream_t st, const char *tag, const int *dev_count)
{
    if (ngroups < 0) return cudaSuccess;  // ngroups == 0: configure the kernels only
    NttArgs a = ntt_args(c, base, base, groups, dev_count);
    a.R = R;
    a.levels = c->d_levels;
    return transform<true, kFuseTensor>(c, a, ngroups, st, tag);
}

cudaError_t launch_ntt_ip(const he_ctx *c, u64 *base, const NttGroup *groups, int ngroups, const JobRef &R,
                          const u64 *evk, cudaStream_t st, const char *tag, const int *dev_count)
{
    if (ngroups < 0) return cudaSuccess;
    NttArgs a = ntt_args(c, base, base, groups, dev_count);
    a.R = R;
    a.levels = c->d_levels;
    a.evk = evk;
    a.EL = c->K + c->L;
    return transform<true, kFuseIp>(c, a, ngroups, st, tag);
}

cudaError_t launch_ntt_combine(const he_ctx *c, u64 *base, const NttGroup *groups, int ngroups, const JobRef &R,
                               bool plain, cudaStream_t st, const char *tag, const int *dev_count)
{
    if (ngroups < 0) return cudaSuccess;
    NttArgs a = ntt_args(c, base, base, groups, dev_count);
    a.R = R;
    a.levels = c->d_levels;
    a.pinv = c->d_pinv;
    return plain ? transform<false, kFusePlain>(c, a, ngroups, st, tag)
                 : transform<false, kFuseCombine>(c, a, ngroups, st, tag);
}

cudaError_t launch_ntt2(const he_ctx *c, const u64 *src, u64 *dst, const NttGroup *groups, int ngroups, bool inverse,
                        cudaStream_t st, const char *tag, const int *dev_count)
{
    if (ngroups < 0) return cudaSuccess;
    const NttArgs a = ntt_args(c, src, dst, groups, dev_count);
    return inverse ? transform<true, kFuseNone>(c, a, ngroups, st, tag)
                   : transform<false, kFuseNone>(c, a, ngroups, st, tag);
}

int ntt_direct_stages(int logN) { return logN >= 12 && logN <= 17 ? direct_stages(logN) : 0; }

cudaError_t launch_ntt(const he_ctx *c, u64 *base, const NttGroup *groups, int ngroups, bool inverse, cudaStream_t st,
                       const char *tag, const int *dev_count)
{
    return launch_ntt2(c, base, base, groups, ngroups, inverse, st, tag, dev_count);
}

// Set the dynamic shared-memory limit of every NTT pass this ring size uses,
// (done once per context, before any launch or stream capture).
cudaError_t configure_ntt(const he_ctx *c)
{
    JobRef R;
    memset(&R, 0, sizeof(R));
    cudaError_t e = launch_ntt2(c, nullptr, nullptr, nullptr, 0, false, nullptr);
    if (e == cudaSuccess) e = launch_ntt2(c, nullptr, nullptr, nullptr, 0, true, nullptr);
    if (e == cudaSuccess) e = launch_ntt_combine(c, nullptr, nullptr, 0, R, false, nullptr);
    if (e == cudaSuccess) e = launch_ntt_combine(c, nullptr, nullptr, 0, R, true, nullptr);
    if (e == cudaSuccess) e = launch_ntt_tensor(c, nullptr, nullptr, 0, R, nullptr);
    if (e == cudaSuccess) e = launch_ntt_ip(c, nullptr, nullptr, 0, R, nullptr, nullptr, nullptr, nullptr);
    return e;
}

}  // namespace he
