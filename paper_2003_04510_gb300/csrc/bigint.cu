// bigint.cu -- the paper's own (non-RNS) HEAAN HE Mul on sm_103a.
//
// Ciphertext and key coefficients are BigInts modulo powers of two (the
// paper's Table 3: q = 2^logq, Q = 2^logQ, p = 2^logp), stored word-major:
// word w of coefficient n at a[w * N + n], little-endian, ceil(k / 64) words.
// Each polynomial product follows the paper's five steps (Fig. 2, Sec. 4):
//   CRT    BigInt -> residues mod np NTT primes (k_crt, crt.cuh: bytes times
//          2^(8k) mod p_i on the tensor cores, one Barrett reduction -- Algo
//          1's accumulate-then-reduce, without BigInt carries; the evaluation
//          key's, once per key: k_nr_crt, 28-bit chunks times 2^(28k) mod p_i)
//   NTT    the RNS path's k_ntt_pass over the context's primes
//   mul    element-wise (k_nr_tensor: d0 = b1 b2, d1 = a1 b2 + a2 b1,
//          d2 = a1 a2 mod p_i; k_nr_ks_mult: d2 times the evaluation key)
//   iNTT   with N^-1 [Phat_i^-1]_{p_i} folded into its scaling, so its
//          outputs are y_i = [x_i Phat_i^-1]_{p_i}
//   iCRT   (k_icrt, icrt.cuh: Algo 6's matrix form) C = sum_i y_i Phat_i - u P
//          with u = round(sum_i y_i / p_i), which is exact because P exceeds
//          four times the product's magnitude (the fraction is never near
//          1/2); the sums mod 2^(64 W) on the tensor cores, u P taken from a
//          table of (2^(64 W) - u P) rows.
// Region 2 (the evaluation key, coefficients mod Q^2) folds the division by
// Q with rounding and the final addition into its iCRT.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "crt.cuh"
#include "he_internal.h"
#include "host_math.h"
#include "icrt.cuh"
#include "modarith.cuh"

struct he_nr_plan {
    he_ctx *c = nullptr;
    int logQ = 0, logp = 0, np1 = 0, np2 = 0, W1 = 0, W2 = 0;
    int chunks_evk = 0;
    bool crt_folds = false;  // every prime reduces by folding (crt.cuh)
    void *dev = nullptr;  // one allocation: tables and NTT group lists
    const u64 *crt = nullptr;           // [np2][chunks_evk]: 2^(28k) mod p_i, split at bit 28
    const unsigned char *crt1 = nullptr, *crt2 = nullptr;      // CRT constants over np1 and np2 primes (crt.cuh)
    const he::crt::Prime *crt_prime = nullptr;                 // [np2]
    const unsigned char *image1 = nullptr, *image2 = nullptr;  // iCRT constants (icrt.cuh)
    const u64 *neg1 = nullptr, *neg2 = nullptr;
    const he::icrt::Prime *prime = nullptr;                    // [np2]
    const he::NttGroup *gF1 = nullptr, *gI1 = nullptr, *gF2 = nullptr, *gI2 = nullptr, *gFe = nullptr;
    int nF1 = 0, nI1 = 0, nF2 = 0, nI2 = 0, nFe = 0;
};

namespace he {

namespace {

constexpr int kT = 256;     // one coefficient per thread (CRT, products, rescale)
constexpr int kCP = 8;      // primes per CTA in the CRT
constexpr int kMaxNp = icrt::kMaxNp;  // primes of a plan (the context's ciphertext primes)
constexpr int kSMs = 152;
constexpr int kChunkBlock = 40;  // 28-bit chunks accumulated before a reduction

__device__ __forceinline__ ulonglong2 ld2(const u64 *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
__device__ __forceinline__ void st2(u64 *p, u64 x, u64 y) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(x, y); }

// bits [28k, 28k + 28) of the WI-word integer w
template <int WI>
__device__ __forceinline__ uint32_t chunk28(const u64 (&w)[WI], int k)
{
    const int bit = 28 * k, q = bit >> 6, o = bit & 63;
    u64 v = q < WI ? w[q] >> o : 0;
    if (o > 36 && q + 1 < WI) v |= w[q + 1] << (64 - o);
    return (uint32_t)(v & 0xFFFFFFFull);
}

// CRT of `polys` BigInt polynomials (wi <= WI words each, word-major, poly
// stride `stride` words) to residues out[poly][np][N].  grid: x over N / kT,
// y over polys, z over prime groups of kCP.
template <int WI>
__global__ void __launch_bounds__(kT)
k_nr_crt(const u64 *in, int wi, size_t stride, u64 *out, int np,
         const u64 *__restrict__ tab, int tab_stride, const DevPrime *__restrict__ primes, int K, int N)
{
    constexpr int CH = (64 * WI + 27) / 28;
    __shared__ u64 sc[kCP][CH];
    const int i0 = blockIdx.z * kCP, cnt = min(kCP, np - i0);
    for (int t = threadIdx.x; t < kCP * CH; t += kT) {
        const int r = t / CH, k = t % CH;
        sc[r][k] = r < cnt ? tab[(size_t)(i0 + r) * tab_stride + k] : 0;
    }
    const int n = blockIdx.x * kT + threadIdx.x;
    const u64 *src = in + (size_t)blockIdx.y * stride + n;
    griddep_wait();
    u64 w[WI];
#pragma unroll
    for (int q = 0; q < WI; q++) w[q] = q < wi ? src[(size_t)q * N] : 0;
    __syncthreads();
    for (int r = 0; r < cnt; r++) {
        const DevPrime pr = primes[K + i0 + r];
        u64 res = 0;
#pragma unroll
        for (int k0 = 0; k0 < CH; k0 += kChunkBlock) {
            u64 a0 = 0, a1 = 0;  // weights 1 and 2^28: each term below 2^57, 40 terms below 2^63
#pragma unroll
            for (int k = k0; k < min(CH, k0 + kChunkBlock); k++) {
                const uint32_t x = chunk28<WI>(w, k);
                const u64 b = sc[r][k];
                a0 = mad_wide(x, (uint32_t)b, a0);
                a1 = mad_wide(x, (uint32_t)(b >> 32), a1);
            }
            U128 v;
            v.lo = a0 + (a1 << 28);
            v.hi = (a1 >> 36) + (v.lo < a0 ? 1ull : 0ull);
            res = add_mod(res, barrett128(v, pr.q, pr.mu, pr.s), pr.q);
        }
        out[((size_t)blockIdx.y * np + i0 + r) * N + n] = res;
    }
}

// Region 1 products in place: slots [A1 | B1 | A2 | B2][np][N] become
// [D0 | D1 | D2 | -] with d0 = b1 b2, d1 = a1 b2 + a2 b1, d2 = a1 a2 mod p_i.
// grid: x over N / 2 / kT, y over primes.
__global__ void __launch_bounds__(kT)
k_nr_tensor(u64 *r, int np, const DevPrime *__restrict__ primes, int K, int N)
{
    const int i = blockIdx.y;
    const DevPrime pr = primes[K + i];
    const size_t n = 2 * ((size_t)blockIdx.x * kT + threadIdx.x);
    const size_t L = (size_t)np * N, o = (size_t)i * N + n;
    griddep_wait();
    const ulonglong2 a1 = ld2(r + o), b1 = ld2(r + L + o), a2 = ld2(r + 2 * L + o), b2 = ld2(r + 3 * L + o);
    U128 x = mul_wide(a1.x, b2.x), y = mul_wide(a1.y, b2.y);
    mac(x, a2.x, b1.x);
    mac(y, a2.y, b1.y);
    st2(r + o, mul_mod(b1.x, b2.x, pr.q, pr.mu, pr.s), mul_mod(b1.y, b2.y, pr.q, pr.mu, pr.s));
    st2(r + L + o, barrett128(x, pr.q, pr.mu, pr.s), barrett128(y, pr.q, pr.mu, pr.s));
    st2(r + 2 * L + o, mul_mod(a1.x, a2.x, pr.q, pr.mu, pr.s), mul_mod(a1.y, a2.y, pr.q, pr.mu, pr.s));
}

// Region 2 products: r[0] (d2 residues) -> KS_b in place, r[1] = KS_a, with
// the prepared key ek = [b | a][np][N].  grid: x over N / 2 / kT, y over primes.
__global__ void __launch_bounds__(kT)
k_nr_ks_mult(u64 *r, const u64 *ek, int np, const DevPrime *__restrict__ primes, int K,
             int N)
{
    const int i = blockIdx.y;
    const DevPrime pr = primes[K + i];
    const size_t n = 2 * ((size_t)blockIdx.x * kT + threadIdx.x);
    const size_t L = (size_t)np * N, o = (size_t)i * N + n;
    griddep_wait();
    const ulonglong2 d = ld2(r + o), kb = ld2(ek + o), ka = ld2(ek + L + o);
    st2(r + o, mul_mod(d.x, kb.x, pr.q, pr.mu, pr.s), mul_mod(d.y, kb.y, pr.q, pr.mu, pr.s));
    st2(r + L + o, mul_mod(d.x, ka.x, pr.q, pr.mu, pr.s), mul_mod(d.y, ka.y, pr.q, pr.mu, pr.s));
}

// Rescale by 2^s with rounding: out = floor((a + 2^(s-1)) / 2^s) mod 2^kout.
// grid: x over N / kT, y over the two halves.
__global__ void __launch_bounds__(kT)
k_nr_rescale(const u64 *in, int wi, u64 *out, int wo, int kout, int s, int N)
{
    const int n = blockIdx.x * kT + threadIdx.x;
    const u64 *a = in + (size_t)blockIdx.y * wi * N + n;
    u64 *o = out + (size_t)blockIdx.y * wo * N + n;
    griddep_wait();
    const int q0 = s >> 6, r = s & 63;
    // add 2^(s-1) and shift right by s, word by word
    u64 carry = 0, prev = 0;
    for (int w = 0; w <= wi; w++) {
        u64 x = w < wi ? a[(size_t)w * N] : 0;
        const u64 add = (w == ((s - 1) >> 6)) ? (1ull << ((s - 1) & 63)) : 0;
        u64 t = x + add;
        u64 c = t < x ? 1ull : 0ull;
        t += carry;
        c += t < carry ? 1ull : 0ull;
        carry = c;
        const int j = w - q0 - 1;
        if (j >= 0 && j < wo) {
            u64 v = r ? (prev >> r) | (t << (64 - r)) : prev;
            if (j == wo - 1 && (kout & 63)) v &= (1ull << (kout & 63)) - 1;
            o[(size_t)j * N] = v;
        }
        prev = t;
    }
    // the last output word may need the column past the input
    const int j = wi - q0;
    if (j >= 0 && j < wo) {
        u64 v = r ? (prev >> r) | (carry << (64 - r)) : prev;
        if (j == wo - 1 && (kout & 63)) v &= (1ull << (kout & 63)) - 1;
        o[(size_t)j * N] = v;
    }
}

int nwords(int k) { return (k + 63) / 64; }

// ---- host-side multiword helpers for the plan's tables ----------------------
typedef std::vector<u64> MW;
void mw_mul_small(MW &a, u64 v)
{
    unsigned __int128 c = 0;
    for (auto &x : a) {
        c += (unsigned __int128)x * v;
        x = (u64)c;
        c >>= 64;
    }
}
void mw_add(MW &a, const MW &b)
{
    unsigned __int128 c = 0;
    for (size_t i = 0; i < a.size(); i++) {
        c += (unsigned __int128)a[i] + (i < b.size() ? b[i] : 0);
        a[i] = (u64)c;
        c >>= 64;
    }
}
u64 mw_mod(const MW &a, u64 p)
{
    unsigned __int128 r = 0;
    for (size_t i = a.size(); i-- > 0;) r = ((r << 64) | a[i]) % p;
    return (u64)r;
}
u64 powmod(u64 b, u64 e, u64 m)
{
    u64 r = 1 % m;
    b %= m;
    while (e) {
        if (e & 1) r = (u64)((unsigned __int128)r * b % m);
        b = (u64)((unsigned __int128)b * b % m);
        e >>= 1;
    }
    return r;
}
u64 invmod(u64 a, u64 p) { return powmod(a, p - 2, p); }
u64 shoup_c(u64 w, u64 p) { return (u64)(((unsigned __int128)w << 64) / p); }

// Phat_i mod 2^(64 W) for the first np primes, P mod 2^(64 W), Phat_i^-1 mod p_i
void crt_tables(const he_ctx *c, int np, int W, std::vector<u64> &M, std::vector<u64> &P, std::vector<u64> &phinv)
{
    const int len = np + 2;
    M.assign((size_t)np * W, 0);
    P.assign(W, 0);
    phinv.assign(np, 0);
    MW full(len, 0);
    full[0] = 1;
    for (int i = 0; i < np; i++) mw_mul_small(full, c->ext[c->K + i]);
    for (int w = 0; w < W && w < len; w++) P[w] = full[w];
    for (int i = 0; i < np; i++) {
        MW h(len, 0);
        h[0] = 1;
        for (int j = 0; j < np; j++)
            if (j != i) mw_mul_small(h, c->ext[c->K + j]);
        for (int w = 0; w < W && w < len; w++) M[(size_t)i * W + w] = h[w];
        phinv[i] = invmod(mw_mod(h, c->ext[c->K + i]), c->ext[c->K + i]);
    }
}

// (2^(64 W) - u P + add) mod 2^(64 W) for u = 0..np
std::vector<u64> neg_rows(const std::vector<u64> &P, int np, int W, int add_bit)
{
    std::vector<u64> out((size_t)(np + 1) * W, 0);
    for (int u = 0; u <= np; u++) {
        MW uP(W + 1, 0);
        for (int w = 0; w < W; w++) uP[w] = P[w];
        uP[W] = 0;
        mw_mul_small(uP, (u64)u);
        MW v(W, 0);  // 0 - uP mod 2^(64W)
        unsigned __int128 borrow = 0;
        for (int w = 0; w < W; w++) {
            unsigned __int128 t = (unsigned __int128)0 - uP[w] - borrow;
            v[w] = (u64)t;
            borrow = (t >> 64) ? 1 : 0;
        }
        if (add_bit >= 0) {
            MW a(W, 0);
            if (add_bit / 64 < W) a[add_bit / 64] = 1ull << (add_bit & 63);
            mw_add(v, a);
        }
        for (int w = 0; w < W; w++) out[(size_t)u * W + w] = v[w];
    }
    return out;
}

// The evaluation key's CRT.
void launch_crt_evk(const he_nr_plan *pl, const u64 *in, int wi, int polys, u64 *out, int np, cudaStream_t st)
{
    const he_ctx *c = pl->c;
    dim3 g((unsigned)(c->N / kT), (unsigned)polys, (unsigned)((np + kCP - 1) / kCP));
    launch_k(c->pdl, k_nr_crt<2 * crt::kMaxWords>, g, dim3(kT), 0, st, in, wi, (size_t)wi * c->N, out, np, pl->crt,
             pl->chunks_evk, (const DevPrime *)c->d_primes, c->K, c->N);
}

// CRT of polys polynomials of wi <= W1 words over np primes.
cudaError_t launch_crt(const he_nr_plan *pl, const u64 *const *in, int polys, int wi, u64 *out, int np,
                       const unsigned char *image, cudaStream_t st)
{
    const he_ctx *c = pl->c;
    crt::Args P;
    for (int k = 0; k < 4; k++) P.in[k] = in[k < polys ? k : 0];
    P.out = out;
    P.image = image;
    P.prime = pl->crt_prime;
    P.flag = c->d_flag;
    P.wi = wi;
    P.W = pl->W1;
    P.np = np;
    P.pc = crt::chunk_primes(np);
    P.polys = polys;
    P.N = c->N;
    const int nch = (np + P.pc - 1) / P.pc;
    dim3 g((unsigned)std::min(kSMs / nch, polys * (c->N / tc::kRows)), (unsigned)nch);
    launch_k(c->pdl, pl->crt_folds ? crt::k_crt<true> : crt::k_crt<false>, g, dim3(crt::kThreads), (size_t)crt::smem_bytes(P.W, P.pc), st, P);
    return cudaGetLastError();
}

// f16 of the balanced bytes, which the images hold by the hundred thousand.
const uint16_t *byte_halves()
{
    static const std::vector<uint16_t> t = [] {
        std::vector<uint16_t> h(256);
        for (int v = -128; v < 128; v++) h[v + 128] = half_of(v);
        return h;
    }();
    return t.data() + 128;
}

// Images of 2^(8k) mod p_i, k < 8 W, over the first np1 and over all np2 >= np1 primes,
// and each prime's constants.
void crt_images(const he_ctx *c, int np1, int np2, int W, std::vector<uint16_t> &image1, std::vector<uint16_t> &image2,
                std::vector<crt::Prime> &prime)
{
    const uint16_t *half = byte_halves(), offset = half_of(6144);  // times the digits' 2048
    std::vector<uint16_t> *image[2] = {&image1, &image2};
    const int np[2] = {np1, np2};
    int pc[2];
    for (int t = 0; t < 2; t++) {
        pc[t] = crt::chunk_primes(np[t]);
        image[t]->assign((size_t)((np[t] + pc[t] - 1) / pc[t]) * crt::image_bytes(W, pc[t]) / 2, 0);
    }
    prime.resize(np2);
    for (int i = 0; i < np2; i++) {
        const u64 p = c->ext[c->K + i];
        const u64 two8 = shoup_c(256, p);  // 256 < p
        uint16_t *im[2];  // the prime's first row: rows of eight digits, 8 pc rows to a core column
        for (int t = 0; t < 2; t++)
            im[t] = i < np[t] ? image[t]->data() + (size_t)(i / pc[t]) * crt::image_bytes(W, pc[t]) / 2 + (size_t)(i % pc[t]) * 64
                              : nullptr;
        u64 v = 1 % p, sum = 0;  // sum of the bytes' offsets
        for (int k = 0; k < 8 * W; k++) {
            long long x = v > p / 2 ? (long long)v - (long long)p : (long long)v;
            for (int col = 0; col < 8; col++) {
                const int r = (int)((x + 128) & 255) - 128;
                for (int t = 0; t < 2; t++)
                    if (im[t]) im[t][((size_t)(k / 8) * 8 * pc[t] + col) * 8 + k % 8] = half[r];
                x = (x - r) >> 8;  // exact
            }
            sum = hm::add(sum, v, p);
            v = v * 256 - (u64)(((unsigned __int128)v * two8) >> 64) * p;  // Shoup: below 2 p
            v = v >= p ? v - p : v;
        }
        u64 off = 0, w = 1 % p;
        for (int col = 0; col < 8; col++) {
            for (int t = 0; t < 2; t++)
                if (im[t]) im[t][((size_t)W * 8 * pc[t] + col) * 8] = offset;
            if (col % 2 == 0) off = hm::add(off, hm::mul(crt::kPair % p, w, p), p);
            w = hm::mul(w, 256, p);
        }
        prime[i].q = p;
        prime[i].s = (uint32_t)hm::bitlen(p) - 2;
        prime[i].mu = (u64)(((unsigned __int128)1 << (64 + prime[i].s)) / p);
        prime[i].base = hm::sub(hm::mul(sum, 128, p), off, p);
        const u64 delta = (1ull << hm::bitlen(p)) - p;
        prime[i].delta = delta >> 31 ? 0 : (uint32_t)delta;
    }
}

// Constants of an iCRT: the image of M_i = Phat_i mod 2^(64 W) (balanced bytes)
// and the rows NEG_u, to which the products of the digits' offsets and the
// accumulators' offsets are added.
void icrt_tables(const he_ctx *c, int np, int W, int add_bit, std::vector<u64> &phinv, std::vector<uint16_t> &image,
                 std::vector<u64> &neg)
{
    const int chunks = (W + icrt::kWords - 1) / icrt::kWords, npad = icrt::padded(np);
    std::vector<u64> M, P;
    crt_tables(c, np, W, M, P, phinv);
    image.assign((size_t)chunks * npad * icrt::kCols * 8, 0);
    const uint16_t *half = byte_halves();
    std::vector<int> m(8 * W);
    MW fix(W, 0);  // sum_i H M_i - sum_c kOff 2^(8c)
    for (int i = 0; i < np; i++) {
        int carry = 0;
        for (int e = 0; e < 8 * W; e++) {
            int v = (int)((M[(size_t)i * W + e / 8] >> (8 * (e % 8))) & 255) + carry;
            carry = v >= 128;
            m[e] = v - 256 * carry;
        }
        for (int ct = 0; ct < 8 * W; ct++) {
            uint16_t *row = &image[(((size_t)(ct / icrt::kCols) * npad + i) * icrt::kCols + ct % icrt::kCols) * 8];
            for (int d = 0; d < 8 && d <= ct; d++) row[d] = half[m[ct - d]];
        }
        MW h(M.begin() + (size_t)i * W, M.begin() + (size_t)(i + 1) * W);
        mw_mul_small(h, 0x0080808080808080ull);
        mw_add(fix, h);
    }
    MW off(W, 0);
    for (int w = 0; w < W; w++) {
        unsigned __int128 v = 0;
        for (int b = 0; b < 8; b++) v += (unsigned __int128)icrt::kOff << (8 * b);
        MW x(W, 0);
        x[w] = (u64)v;
        if (w + 1 < W) x[w + 1] = (u64)(v >> 64);
        mw_add(off, x);
    }
    for (auto &x : off) x = ~x;  // minus off
    MW one(1, 1);
    mw_add(off, one);
    mw_add(fix, off);
    neg = neg_rows(P, np, W, add_bit);
    for (int u = 0; u <= np; u++) {
        MW row(neg.begin() + (size_t)u * W, neg.begin() + (size_t)(u + 1) * W);
        mw_add(row, fix);
        std::copy(row.begin(), row.end(), neg.begin() + (size_t)u * W);
    }
}

// out[poly] (out_stride words apart): T mod 2^kout, or (d) d[poly] (d_stride words
// apart) plus T / 2^s rounded, mod 2^kout.
cudaError_t launch_icrt(const he_nr_plan *pl, const u64 *y, int np, int W, const unsigned char *image, const u64 *neg,
                        u64 *out, int out_stride, int kout, const u64 *d, int d_stride, int s, int polys, cudaStream_t st)
{
    const he_ctx *c = pl->c;
    icrt::Args P;
    P.y = y;
    P.image = image;
    P.neg = neg;
    P.prime = pl->prime;
    P.out = out;
    P.d = d;
    P.flag = c->d_flag;
    P.np = np;
    P.W = W;
    P.chunks = (W + icrt::kWords - 1) / icrt::kWords;
    P.polys = polys;
    P.out_stride = out_stride;
    P.d_stride = d_stride;
    P.wo = (kout + 63) / 64;
    P.kout = kout;
    P.s = s;
    P.N = c->N;
    dim3 g((unsigned)std::min(kSMs, polys * (c->N / tc::kRows)));
    launch_k(c->pdl, d ? icrt::k_icrt<true> : icrt::k_icrt<false>, g, dim3(icrt::kThreads), (size_t)icrt::smem_bytes(np, W),
             st, P);
    return cudaGetLastError();
}

}  // namespace

}  // namespace he

using namespace he;

namespace {

// Supported: log Q with nwords(logQ) <= 19 and nwords(2 logQ) <= 38, the
// template widths of the kernels below.
constexpr int kW1 = 19, kW2 = 38;

size_t ws_words(const he_nr_plan *pl)
{
    const size_t N = (size_t)pl->c->N;
    return (size_t)4 * pl->np1 * N + (size_t)3 * kW1 * N + (size_t)2 * pl->np2 * N;
}

int dev_try(cudaError_t e) { return e == cudaSuccess ? HE_OK : HE_ECUDA; }

}  // namespace

extern "C" {

int he_nr_plan_create(he_ctx *c, int logQ, int logp, he_nr_plan **out)
{
    if (!c || !c->device || !out) return HE_EINVAL;
    if (logQ < 64 || nwords(logQ) > kW1 || nwords(2 * logQ) > kW2 || logp < 1 || logp >= logQ) return HE_EINVAL;
    // primes: the fewest leading context primes whose product exceeds
    // 2^(2 logQ + logN + 2) (region 1) and 2^(3 logQ + logN + 2) (region 2)
    auto count = [&](double bits) {
        double tot = 0;
        for (int i = 0; i < c->L; i++) {
            tot += std::log2((double)c->ext[c->K + i]);
            if (tot > bits) return i + 1;
        }
        return -1;
    };
    const int np1 = count(2.0 * logQ + c->logN + 2), np2 = count(3.0 * logQ + c->logN + 2);
    if (np1 < 0 || np2 < 0 || np2 > kMaxNp) return HE_EINVAL;
    for (int i = 0; i < np2; i++)
        if (c->ext[c->K + i] >= (1ull << 57) || c->ext[c->K + i] < (1ull << 40)) return HE_EINVAL;
    he_nr_plan *pl = new (std::nothrow) he_nr_plan();
    if (!pl) return HE_ENOMEM;
    pl->c = c;
    pl->logQ = logQ;
    pl->logp = logp;
    pl->np1 = np1;
    pl->np2 = np2;
    pl->W1 = nwords(logQ);
    pl->W2 = nwords(2 * logQ);
    pl->chunks_evk = (64 * kW2 + 27) / 28;
    const int N = c->N, K = c->K;
    // host tables
    std::vector<u64> crt((size_t)np2 * pl->chunks_evk);
    for (int i = 0; i < np2; i++) {
        const u64 p = c->ext[K + i];
        u64 v = 1;
        for (int k = 0; k < pl->chunks_evk; k++, v = hm::mul(v, 1ull << 28, p)) {
            crt[(size_t)i * pl->chunks_evk + k] = (v & 0xFFFFFFFull) | ((v >> 28) << 32);
        }
    }
    std::vector<u64> phinv1, phinv2, neg1, neg2;
    std::vector<uint16_t> image1, image2;
    std::vector<uint16_t> crt1, crt2;
    std::vector<crt::Prime> crt_prime;
    crt_images(c, np1, np2, pl->W1, crt1, crt2, crt_prime);
    pl->crt_folds = true;
    for (const crt::Prime &p : crt_prime) pl->crt_folds = pl->crt_folds && crt::folds(p);
    icrt_tables(c, np1, pl->W1, -1, phinv1, image1, neg1);
    icrt_tables(c, np2, pl->W2, logQ - 1, phinv2, image2, neg2);
    std::vector<icrt::Prime> prime(np2);
    for (int i = 0; i < np2; i++) {
        const u64 p = c->ext[K + i];
        const int b = hm::bitlen(p);
        prime[i].inv = (uint32_t)(((unsigned __int128)1 << (25 + b)) / p);
        prime[i].shift = (uint32_t)(b - 32);
    }
    // NTT job lists (offsets in limbs from the workspace, or from the prepared key)
    const unsigned d_limbs = (unsigned)(3 * kW1);  // the d0, d1, d2 words, in units of N words
    const unsigned r2 = (unsigned)(4 * np1) + d_limbs;
    std::vector<NttJob> F1, I1, F2, I2, Fe;
    auto job = [&](unsigned src, unsigned dst, int i, u64 sc, u64 scs) {
        NttJob j;
        memset(&j, 0, sizeof(j));
        j.src = src;
        j.dst = dst;
        j.prime = (unsigned)(K + i);
        j.scale = sc;
        j.scale_sh = scs;
        return j;
    };
    for (int t = 0; t < 4; t++)
        for (int i = 0; i < np1; i++) F1.push_back(job(t * np1 + i, t * np1 + i, i, 0, 0));
    for (int t = 0; t < 3; t++)
        for (int i = 0; i < np1; i++) {
            const u64 p = c->ext[K + i];
            const u64 sc = (u64)((unsigned __int128)c->ninv[K + i] * phinv1[i] % p);
            I1.push_back(job(t * np1 + i, t * np1 + i, i, sc, shoup_c(sc, p)));
        }
    for (int i = 0; i < np2; i++) F2.push_back(job(r2 + i, r2 + i, i, 0, 0));
    for (int t = 0; t < 2; t++)
        for (int i = 0; i < np2; i++) {
            const u64 p = c->ext[K + i];
            const u64 sc = (u64)((unsigned __int128)c->ninv[K + i] * phinv2[i] % p);
            I2.push_back(job(r2 + t * np2 + i, r2 + t * np2 + i, i, sc, shoup_c(sc, p)));
        }
    for (int t = 0; t < 2; t++)
        for (int i = 0; i < np2; i++) Fe.push_back(job(t * np2 + i, t * np2 + i, i, 0, 0));
    std::vector<NttGroup> gF1 = group_jobs(F1, 1), gI1 = group_jobs(I1, 1), gF2 = group_jobs(F2, 1), gI2 = group_jobs(I2, 1),
                          gFe = group_jobs(Fe, 1);
    // one device allocation for everything
    size_t off = 0;
    auto take = [&](size_t b) {
        size_t o = off;
        off += (b + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_crt = take(crt.size() * 8), o_m1 = take(image1.size() * 2), o_n1 = take(neg1.size() * 8),
                 o_m2 = take(image2.size() * 2), o_n2 = take(neg2.size() * 8),
                 o_p = take(prime.size() * sizeof(icrt::Prime)), o_c1 = take(crt1.size() * 2),
                 o_c2 = take(crt2.size() * 2), o_cp = take(crt_prime.size() * sizeof(crt::Prime)), o_g1 = take(gF1.size() * sizeof(NttGroup)),
                 o_g2 = take(gI1.size() * sizeof(NttGroup)), o_g3 = take(gF2.size() * sizeof(NttGroup)),
                 o_g4 = take(gI2.size() * sizeof(NttGroup)), o_g5 = take(gFe.size() * sizeof(NttGroup));
    // the iCRTs' operands and ring
    if (cudaFuncSetAttribute(crt::k_crt<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             crt::smem_bytes(crt::kMaxWords, crt::kPrimes)) != cudaSuccess ||
        cudaFuncSetAttribute(crt::k_crt<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             crt::smem_bytes(crt::kMaxWords, crt::kPrimes)) != cudaSuccess ||
        cudaFuncSetAttribute(icrt::k_icrt<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             icrt::smem_bytes(kMaxNp, kW2)) != cudaSuccess ||
        cudaFuncSetAttribute(icrt::k_icrt<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             icrt::smem_bytes(kMaxNp, kW2)) != cudaSuccess ||
        cudaMalloc(&pl->dev, off) != cudaSuccess) {
        delete pl;
        return HE_ECUDA;
    }
    std::vector<unsigned char> img(off, 0);
    auto put = [&](size_t o, const void *p, size_t b) { memcpy(img.data() + o, p, b); };
    put(o_crt, crt.data(), crt.size() * 8);
    put(o_m1, image1.data(), image1.size() * 2);
    put(o_n1, neg1.data(), neg1.size() * 8);
    put(o_m2, image2.data(), image2.size() * 2);
    put(o_n2, neg2.data(), neg2.size() * 8);
    put(o_p, prime.data(), prime.size() * sizeof(icrt::Prime));
    put(o_c1, crt1.data(), crt1.size() * 2);
    put(o_c2, crt2.data(), crt2.size() * 2);
    put(o_cp, crt_prime.data(), crt_prime.size() * sizeof(crt::Prime));
    put(o_g1, gF1.data(), gF1.size() * sizeof(NttGroup));
    put(o_g2, gI1.data(), gI1.size() * sizeof(NttGroup));
    put(o_g3, gF2.data(), gF2.size() * sizeof(NttGroup));
    put(o_g4, gI2.data(), gI2.size() * sizeof(NttGroup));
    put(o_g5, gFe.data(), gFe.size() * sizeof(NttGroup));
    if (cudaMemcpy(pl->dev, img.data(), off, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(pl->dev);
        delete pl;
        return HE_ECUDA;
    }
    char *b = (char *)pl->dev;
    pl->crt = (const u64 *)(b + o_crt);
    pl->image1 = (const unsigned char *)(b + o_m1);
    pl->neg1 = (const u64 *)(b + o_n1);
    pl->image2 = (const unsigned char *)(b + o_m2);
    pl->neg2 = (const u64 *)(b + o_n2);
    pl->prime = (const icrt::Prime *)(b + o_p);
    pl->crt1 = (const unsigned char *)(b + o_c1);
    pl->crt2 = (const unsigned char *)(b + o_c2);
    pl->crt_prime = (const crt::Prime *)(b + o_cp);
    pl->gF1 = (const NttGroup *)(b + o_g1);
    pl->gI1 = (const NttGroup *)(b + o_g2);
    pl->gF2 = (const NttGroup *)(b + o_g3);
    pl->gI2 = (const NttGroup *)(b + o_g4);
    pl->gFe = (const NttGroup *)(b + o_g5);
    pl->nF1 = (int)gF1.size();
    pl->nI1 = (int)gI1.size();
    pl->nF2 = (int)gF2.size();
    pl->nI2 = (int)gI2.size();
    pl->nFe = (int)gFe.size();
    (void)N;
    *out = pl;
    return HE_OK;
}

int he_nr_plan_destroy(he_nr_plan *pl)
{
    if (!pl) return HE_EINVAL;
    if (pl->dev) cudaFree(pl->dev);
    delete pl;
    return HE_OK;
}

int he_nr_plan_info(const he_nr_plan *pl, int *np1, int *np2)
{
    if (!pl) return HE_EINVAL;
    if (np1) *np1 = pl->np1;
    if (np2) *np2 = pl->np2;
    return HE_OK;
}

size_t he_nr_workspace_bytes(const he_nr_plan *pl) { return pl ? ws_words(pl) * sizeof(u64) : 0; }

size_t he_nr_evk_bytes(const he_nr_plan *pl) { return pl ? (size_t)2 * pl->np2 * pl->c->N * sizeof(u64) : 0; }

int he_nr_evk_prepare(he_nr_plan *pl, const uint64_t *evk, uint64_t *prep, void *stream)
{
    if (!pl || !evk || !prep) return HE_EINVAL;
    if (int w = device_waits(pl->c)) return w;
    cudaStream_t st = (cudaStream_t)stream;
    launch_crt_evk(pl, evk, nwords(2 * pl->logQ), 2, prep, pl->np2, st);
    if (cudaGetLastError() != cudaSuccess) return HE_ECUDA;
    return dev_try(launch_ntt(pl->c, prep, pl->gFe, pl->nFe, false, st, "nr_evk"));
}

int he_nr_mul(he_nr_plan *pl, const uint64_t *ct1, const uint64_t *ct2, const uint64_t *prep, int logq,
              uint64_t *out, void *ws, size_t ws_bytes, void *stream)
{
    if (!pl || !ct1 || !ct2 || !prep || !out || !ws) return HE_EINVAL;
    if (logq < pl->logp + 1 || logq > pl->logQ) return HE_ELEVEL;
    if (ws_bytes < ws_words(pl) * sizeof(u64)) return HE_ENOMEM;
    if (int w = device_waits(pl->c)) return w;
    const he_ctx *c = pl->c;
    he_ctx *cm = pl->c;
    const size_t N = (size_t)c->N;
    const int wq = nwords(logq), np1 = pl->np1, np2 = pl->np2;
    cudaStream_t st = (cudaStream_t)stream;
    u64 *w = (u64 *)ws;
    u64 *R1 = w, *D = w + (size_t)4 * np1 * N, *R2 = D + (size_t)3 * kW1 * N;
    prof_mark(c, st, "");
    // region 1: CRT of a1, b1, a2, b2 (ct = [b | a], word-major)
    const u64 *in1[4] = {ct1 + (size_t)wq * N, ct1, ct2 + (size_t)wq * N, ct2};
    if (launch_crt(pl, in1, 4, wq, R1, np1, pl->crt1, st) != cudaSuccess) return HE_ECUDA;
    prof_mark(c, st, "nr_crt1");
    if (launch_ntt(cm, w, pl->gF1, pl->nF1, false, st, "nr_ntt1") != cudaSuccess) return HE_ECUDA;
    launch_k(c->pdl, k_nr_tensor, dim3((unsigned)(N / 2 / kT), (unsigned)np1), dim3(kT), 0, st, R1, np1,
             (const DevPrime *)c->d_primes, c->K, c->N);
    if (cudaGetLastError() != cudaSuccess) return HE_ECUDA;
    prof_mark(c, st, "nr_tensor");
    if (launch_ntt(cm, w, pl->gI1, pl->nI1, true, st, "nr_intt1") != cudaSuccess) return HE_ECUDA;
    // d0, d1, d2 mod q (word-major, wq words each, stride kW1 words)
    if (launch_icrt(pl, R1, np1, pl->W1, pl->image1, pl->neg1, D, kW1, logq, nullptr, 0, 0, 3, st) != cudaSuccess)
        return HE_ECUDA;
    prof_mark(c, st, "nr_icrt1");
    // region 2: CRT of d2, NTT, products with the prepared key, iNTT, iCRT + shift + add
    const u64 *d2 = D + (size_t)2 * kW1 * N;
    if (launch_crt(pl, &d2, 1, wq, R2, np2, pl->crt2, st) != cudaSuccess) return HE_ECUDA;
    prof_mark(c, st, "nr_crt2");
    if (launch_ntt(cm, w, pl->gF2, pl->nF2, false, st, "nr_ntt2") != cudaSuccess) return HE_ECUDA;
    launch_k(c->pdl, k_nr_ks_mult, dim3((unsigned)(N / 2 / kT), (unsigned)np2), dim3(kT), 0, st, R2, prep, np2,
             (const DevPrime *)c->d_primes, c->K, c->N);
    if (cudaGetLastError() != cudaSuccess) return HE_ECUDA;
    prof_mark(c, st, "nr_ks_mult");
    if (launch_ntt(cm, w, pl->gI2, pl->nI2, true, st, "nr_intt2") != cudaSuccess) return HE_ECUDA;
    // out[h] = d_h + round(KS_h / Q) mod q; the d's sit kW1 words apart, out wq words apart
    if (launch_icrt(pl, R2, np2, pl->W2, pl->image2, pl->neg2, out, wq, logq, D, kW1, pl->logQ, 2, st) != cudaSuccess)
        return HE_ECUDA;
    prof_mark(c, st, "nr_icrt2");
    return HE_OK;
}

int he_nr_rescale(he_nr_plan *pl, const uint64_t *ct, int logq, uint64_t *out, void *stream)
{
    if (!pl || !ct || !out) return HE_EINVAL;
    if (logq <= pl->logp || logq > pl->logQ) return HE_ELEVEL;
    if (int w = device_waits(pl->c)) return w;
    const he_ctx *c = pl->c;
    const int wi = nwords(logq), wo = nwords(logq - pl->logp);
    launch_k(c->pdl, k_nr_rescale, dim3((unsigned)(c->N / kT), 2u), dim3(kT), 0, (cudaStream_t)stream, ct, wi, out,
             wo, logq - pl->logp, pl->logp, c->N);
    return dev_try(cudaGetLastError());
}

}  // extern "C"
