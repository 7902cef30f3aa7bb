// host_params.cpp -- context construction: primes, roots, twiddle tables,
// base-conversion constants, per-level workspace layouts and NTT job lists,
// and the upload of every device table into one arena.
//
// Parameter rules (the paper is silent on the RNS choices):
//   * q_0 > q_1 > ... : the L largest primes below 2^q_bits with q = 1 mod 2N
//   * p_0 > p_1 > ... : the K largest primes below 2^p_bits with p = 1 mod 2N
//                       that are not ciphertext primes
//   * psi             : the smallest primitive 2N-th root of unity mod each prime
//   * digits          : I_j = {j*alpha, ..., min((j+1)*alpha, l) - 1}
// Twiddles follow Algo 3's table TB_W[m + j] = psi^bitrev(m + j) and the iNTT's
// TB_invW; every constant carries its Shoup companion (Algo 2).
#include <algorithm>
#include <cstring>

#include "he_internal.h"
#include "host_math.h"

namespace he {

using namespace hm;

static std::vector<u64> find_primes(int logN, int bits, int count, const std::vector<u64> &skip)
{
    std::vector<u64> out;
    const u64 step = 2ull << logN;
    u64 top = (1ull << bits) - 1;
    u64 c = top - (top - 1) % step;  // largest c <= top with c = 1 mod 2N
    while ((int)out.size() < count && c > step) {
        if (std::find(skip.begin(), skip.end(), c) == skip.end() && is_prime(c)) out.push_back(c);
        c -= step;
    }
    return out;
}

// Smallest primitive 2N-th root: take a generator g of Z_q^*, psi0 = g^((q-1)/2N);
// the primitive 2N-th roots are psi0^k for odd k.
static u64 smallest_psi(u64 q, int logN)
{
    const u64 twoN = 2ull << logN;
    std::vector<u64> f = prime_factors(q - 1);
    u64 g = 2;
    for (;; g++) {
        bool gen = true;
        for (u64 p : f)
            if (pw(g, (q - 1) / p, q) == 1) { gen = false; break; }
        if (gen) break;
    }
    u64 psi0 = pw(g, (q - 1) / twoN, q);
    u64 sq = mul(psi0, psi0, q), best = psi0, cur = psi0;
    for (u64 k = 1; k < twoN / 2; k++) {
        cur = mul(cur, sq, q);
        best = std::min(best, cur);
    }
    return best;
}

static ulonglong2 pair(u64 v, u64 m) { return make_ulonglong2(v, shoup(v, m)); }

// a twiddle as the kernels' mul_tw takes it: w and w 2^32 mod q, split at bit s.
// wsh = floor(w 2^64 / q): its high half is floor(w 2^32 / q), and no 128-bit
// division is needed (tables of two words per ring element and prime: 2^17, 56 primes
// 820 ms a context with divisions, 567 without)
static ulonglong2 split_tw(u64 w, u64 wsh, u64 q, unsigned s)
{
    const u64 w2 = (w << 32) - (wsh >> 32) * q, m = ((u64)1 << s) - 1;
    return make_ulonglong2((w & m) | ((w >> s) << 32), (w2 & m) | ((w2 >> s) << 32));
}

// base-conversion constant stored split at bit 28 for the kernels' lazy MACs
static u64 split28(u64 b) { return (b & 0xFFFFFFFull) | ((b >> 28) << 32); }

// Groups of one prime next to each other: their CTAs run at the same time and read that
// prime's twiddle runs from L2 instead of each from DRAM.  Every group's place follows
// from the counts, so none is moved (a batch's thousands of groups are formed at every
// call; sorting them took a tenth of it).
std::vector<NttGroup> group_jobs(const std::vector<NttJob> &jobs, int cap)
{
    cap = std::max(1, std::min(cap, kGroupMax));
    std::vector<size_t> n, at;  // per prime: its limbs, its first group
    for (const NttJob &j : jobs) {
        if (j.prime >= n.size()) n.resize(j.prime + 1, 0);
        n[j.prime]++;
    }
    size_t groups = 0;
    for (size_t &k : n) {
        at.push_back(groups);
        groups += (k + cap - 1) / cap;
        k = 0;
    }
    std::vector<NttGroup> out(groups);  // zeros
    for (const NttJob &j : jobs) {
        const size_t k = n[j.prime]++;
        NttGroup &G = out[at[j.prime] + k / cap];
        G.prime = j.prime;
        G.src[G.nl] = j.src;
        G.dst[G.nl] = j.dst;
        G.scale[G.nl] = j.scale;
        G.scale_sh[G.nl] = j.scale_sh;
        G.job[G.nl] = j.job;
        G.ci[G.nl] = j.ci;
        G.cd[G.nl] = j.cd;
        G.cks[G.nl] = j.cks;
        G.nl++;
    }
    return out;
}

namespace {

// Upper bound of mul_tw's result for any x <= X (modarith.cuh): A, Bl 2^s and
// Bh c with x1 <= X / 2^32, w < q.
u128 tw_bound(u128 X, u64 q, int s, u64 c)
{
    const u128 xs = ((u128)0xffffffffu) + (X >> 32);  // x0 + x1
    const u128 a = xs * (((u64)1 << s) - 1), b = xs * ((q - 1) >> s);
    return a + ((u128)0xffffffffu << s) + (b >> 32) * c;
}

// Largest multiple-of-q ceiling: the smallest multiple of q that is >= x.
u128 ceil_mul(u128 x, u64 q) { return (x + q - 1) / q * q; }

// Forward growth from inputs up to x over `stages` stages (each adds at most
// cf); the final bound, with cf the ceiling of the largest product met.
u128 fwd_growth(u128 x, int stages, u64 q, int s, u64 c, u128 *cf)
{
    u128 f = ceil_mul(tw_bound(x, q, s, c), q);
    for (int it = 0; it < 64; it++) {
        const u128 last = x + (u128)(stages - 1) * f;  // the last stage's inputs
        if (last >> 64) return last;
        const u128 g = ceil_mul(tw_bound(last, q, s, c), q);
        if (g == f) break;
        f = g;
    }
    *cf = std::max(*cf, f);
    return x + (u128)stages * f;
}

// One inverse round of four stages (the longest) from inputs up to x; the
// bound of its outputs, 0 if a value could reach 2^64 (or the offset ci would
// not cover a stage's inputs).
u128 inv_round(u128 x, u64 q, int s, u64 c, u128 folded, uint32_t flags, u128 *ci)
{
    const u128 lim = (u128)1 << 64;
    u128 m = x, prod = 0;
    for (int st = 1; st <= 4; st++) {
        const u128 off = ceil_mul(m, q);
        *ci = std::max(*ci, off);
        if (m + *ci >= lim || 2 * m >= lim) return 0;
        prod = tw_bound(m + *ci, q, s, c);
        u128 sum = 2 * m;
        if (st == 4 || (st == 2 && (flags & kInvFoldSecond))) sum = std::min(sum, folded);
        if (st == 4 && (flags & kInvFoldAll)) prod = std::min(prod, folded);
        m = std::max(sum, prod);
    }
    return m;
}

}  // namespace

bool ntt_mod(u64 q, int logN, NttMod *out)
{
    const int s = std::max(0, bitlen(q) - 31);
    const u64 c = (u64)(((u128)1 << (32 + s)) % q);
    if (c >> 32) return false;
    const u128 lim = ((u128)1 << 64) - 8 * (u128)q;  // the combine adds up to 5q (ntt.cu)
    const u128 folded = ((u128)1 << (32 + s)) + ((u128)c << (32 - s));
    memset(out, 0, sizeof(*out));
    out->c = (uint32_t)c;
    out->s = (uint32_t)s;
    out->p2 = 1u << s;
    if (folded <= 3 * (u128)q) out->flags |= kFastFinal;
    // forward: inputs below 4q; passes of at most ten stages (twelve at 2^12)
    // and rounds of at most four
    const u128 in = 4 * (u128)q;
    const int pass = std::min(logN, 10);
    u128 cf = 0, end = fwd_growth(in, logN, q, s, c, &cf);
    if (end >= lim) {
        out->flags |= kFwdFoldPass;
        cf = 0;
        end = std::max(fwd_growth(in, pass, q, s, c, &cf), fwd_growth(std::max(folded, in), pass, q, s, c, &cf));
        if (end >= lim || logN == 12) {
            out->flags |= kFwdFoldRound;
            cf = 0;
            end = fwd_growth(std::max(folded, in), 4, q, s, c, &cf);
            if (end >= lim) {
                out->flags |= kFwdFoldSecond;
                cf = 0;
                end = fwd_growth(std::max(folded, in), 2, q, s, c, &cf);
            }
        }
        if (end >= lim) return false;
    }
    out->cf = (u64)cf;
    out->cz = (u64)ceil_mul(end, q);
    // inverse: canonical inputs, then each round's outputs
    static const uint32_t modes[3] = {0, kInvFoldAll, kInvFoldAll | kInvFoldSecond};
    for (uint32_t mode : modes) {
        u128 m = q, ci = 0;
        bool ok = true;
        for (int it = 0;; it++) {  // to a fixed point of the round's bound and the offset
            const u128 ci0 = ci, r = inv_round(m, q, s, c, folded, mode, &ci);
            if (!r || it == 64) ok = false;
            if (!ok || (r <= m && ci == ci0)) break;
            m = std::max(m, r);
        }
        if (ok) {
            out->flags |= mode;
            out->ci = (u64)ci;
            return true;
        }
    }
    return false;
}

static WsLayout layout_for(int l, int K, int alpha)
{
    int beta = (l + alpha - 1) / alpha;
    int E = K + l;
    WsLayout w;
    w.d0 = 0;
    w.d1 = (size_t)l;
    w.d2 = 2 * (size_t)l;
    w.y = 3 * (size_t)l;
    w.u = 4 * (size_t)l;
    w.ks = w.u + (size_t)beta * E;
    w.ys = w.ks + 2 * (size_t)E;
    w.r = w.ys + 2 * (size_t)K;
    w.z = w.r + 4;
    w.total = w.z + 2 * (size_t)l;
    return w;
}

// Images and targets of the tensor-core conversions (tc.cuh); false where the
// context's primes or sizes do not allow them, and the CUDA-core kernels run.  The
// line is where the six planes are exact: primes of at most 55 bits fill six digits
// (a 56-bit target's last plane passes its 22 bits), targets of 52 or more fold in
// one step, and some 14 limbs' worth of digits stay below the planes' offsets, for
// the constants at hand (tc_image counts).  Inside it this form is the faster one at
// every size measured: one HE Mul + rescale 212 -> 198 us at 2^16 (level 24), 952 ->
// 804 at 2^17 (level 44), 71.9 -> 69.8 at 2^15 (level 9).
static bool build_tc(he_ctx *c)
{
    const int K = c->K, L = c->L;
    const std::vector<u64> ps(c->ext.begin(), c->ext.begin() + K), qs(c->ext.begin() + K, c->ext.end());
    for (u64 x : c->ext)  // every prime is a source and a target of some conversion
        if (!tc_source_ok(x) || bitlen(x) < 52) return false;
    auto round8 = [](int v) { return (v + 7) & ~7; };
    auto k_pad = [](int g) { return (24 * g + 1 + 15) / 16 * 16; };  // tc::k_pad
    auto rows = [](int tp) { return (6 * tp + 15) / 16 * 16; };
    // [prod_{i2 != i} m[i2]]_t over m[lo, hi), for every i
    auto hats = [&](const std::vector<u64> &m, int lo, int hi, u64 t) {
        std::vector<u64> h(hi - lo, 1);
        u64 below = 1, above = 1;
        for (int i = 0; i < hi - lo; i++) {
            h[i] = below;
            below = mul(below, m[lo + i] % t, t);
        }
        for (int i = hi - lo - 1; i >= 0; i--) {
            h[i] = mul(h[i], above, t);
            above = mul(above, m[lo + i] % t, t);
        }
        return h;
    };
    c->up_off5 = tc_off5(qs);
    c->dn_off5 = tc_off5(ps);
    // ModDown: chunks of at most 24 targets (tc::kTargets)
    const int kd = k_pad(tc_groups(K));
    c->dn_nch = (L + 23) / 24;
    c->dn_tc = (L + c->dn_nch - 1) / c->dn_nch;
    c->dn_tp = round8(c->dn_tc);
    c->dn_bytes = rows(c->dn_tp) * kd * 2;
    c->dn_last_bytes = 16 * kd * 2;
    c->dn_smem = 3 * 128 * kd * 2 + c->dn_bytes + c->dn_last_bytes;  // three teams
    c->tc_PB.assign((size_t)c->dn_nch * c->dn_bytes, 0);
    c->tc_PBP.assign((size_t)c->dn_nch * c->dn_bytes, 0);
    c->tc_last.assign((size_t)L * c->dn_last_bytes, 0);
    c->tc_PB_t.resize((size_t)c->dn_nch * c->dn_tp);
    c->tc_PBP_t.resize((size_t)c->dn_nch * c->dn_tp);
    std::vector<u64> pb((size_t)L * K), pbp((size_t)L * K);
    for (int i = 0; i < L; i++) {
        const std::vector<u64> h = hats(ps, 0, K, qs[i]);
        for (int k = 0; k < K; k++) {
            pb[(size_t)i * K + k] = h[k];
            pbp[(size_t)i * K + k] = mul(h[k], c->pinv[i].x, qs[i]);
        }
    }
    auto slice = [&](const std::vector<u64> &m, int i0, int n) {
        return std::vector<u64>(m.begin() + (size_t)i0 * K, m.begin() + (size_t)(i0 + n) * K);
    };
    for (int ch = 0; ch < c->dn_nch; ch++) {
        const int i0 = ch * c->dn_tc, n = std::min(c->dn_tc, L - i0);
        const std::vector<u64> t(qs.begin() + i0, qs.begin() + i0 + n);
        if (!tc_image(slice(pb, i0, n), t, n, ps, c->dn_tp, &c->tc_PB[(size_t)ch * c->dn_bytes],
                      &c->tc_PB_t[(size_t)ch * c->dn_tp]) ||
            !tc_image(slice(pbp, i0, n), t, n, ps, c->dn_tp, &c->tc_PBP[(size_t)ch * c->dn_bytes],
                      &c->tc_PBP_t[(size_t)ch * c->dn_tp]))
            return false;
    }
    for (int i = 0; i < L; i++) {
        TcTarget t1;
        if (!tc_image(slice(pbp, i, 1), {qs[i]}, 1, ps, 1, &c->tc_last[(size_t)i * c->dn_last_bytes], &t1)) return false;
    }
    // per level: ModUp images of every digit, and the one-division ModDown's
    const int ku = k_pad(tc_groups(c->alpha));
    for (int l = 1; l <= L; l++) {
        HostLevel &H = c->host_levels[l];
        const int beta = (l + c->alpha - 1) / c->alpha, El = K + l;
        const int nlast = l - (beta - 1) * c->alpha, tmax = El - nlast;  // the last digit has the most targets
        H.up_nch = (tmax + 23) / 24;
        H.up_tc = (tmax + H.up_nch - 1) / H.up_nch;
        H.up_tp = round8(H.up_tc);
        H.up_bytes = rows(H.up_tp) * ku * 2;
        c->up_smem = std::max(c->up_smem, 3 * 128 * ku * 2 + H.up_bytes);  // three teams
        H.tc_up.assign((size_t)beta * H.up_nch * H.up_bytes, 0);
        H.tc_up_t.resize((size_t)beta * H.up_nch * H.up_tp);
        for (int j = 0; j < beta; j++) {
            const int lo = j * c->alpha, hi = std::min((j + 1) * c->alpha, l), nj = hi - lo;
            std::vector<u64> src(c->alpha, qs[lo]);  // every digit runs with alpha limbs; unused ones have no constant
            for (int i = lo; i < hi; i++) src[i - lo] = qs[i];
            for (int ch = 0; ch < H.up_nch; ch++) {
                std::vector<u64> cst, t;
                for (int u = ch * H.up_tc; u < std::min((ch + 1) * H.up_tc, El - nj); u++) {
                    const int e = u < K + lo ? u : u + nj;
                    t.push_back(c->ext[e]);
                    const std::vector<u64> h = hats(qs, lo, hi, c->ext[e]);
                    cst.insert(cst.end(), h.begin(), h.end());
                    cst.resize(cst.size() + c->alpha - nj, 0);
                }
                const size_t at = (size_t)j * H.up_nch + ch;
                if (!tc_image(cst, t, (int)t.size(), src, H.up_tp, &H.tc_up[at * H.up_bytes], &H.tc_up_t[at * H.up_tp]))
                    return false;
            }
        }
        H.tc_pq.assign((size_t)c->dn_nch * c->dn_bytes, 0);
        H.tc_pq_t.resize((size_t)c->dn_nch * c->dn_tp);
        const u64 ql = qs[l - 1];
        for (int ch = 0; ch < c->dn_nch; ch++) {
            std::vector<u64> cst, t;
            for (int i = ch * c->dn_tc; i < std::min((ch + 1) * c->dn_tc, l - 1); i++) {
                t.push_back(qs[i]);
                for (int k = 0; k < K; k++) cst.push_back(mul(pbp[(size_t)i * K + k], ql % qs[i], qs[i]));
            }
            if (!tc_image(cst, t, (int)t.size(), ps, c->dn_tp, &H.tc_pq[(size_t)ch * c->dn_bytes],
                          &H.tc_pq_t[(size_t)ch * c->dn_tp]))
                return false;
        }
    }
    return true;
}

int build_context(he_ctx *c, const he_params *p, bool device)
{
    // q_bits, p_bits <= 57 keep every base-conversion accumulator (at most 16
    // products of a residue and a constant) below barrett128's 2^(b+61) bound.
    if (p->logN < 12 || p->logN > 17 || p->L < 1 || p->L > kMaxL || p->K < 1 || p->K > kMaxK ||
        p->alpha < 1 || p->alpha > 16 || p->q_bits < 30 || p->q_bits > 57 || p->p_bits < 30 ||
        p->p_bits > 57 || p->h < 1 || p->h > (1 << p->logN) || !(p->sigma > 0))
        return HE_EINVAL;
    c->prm = *p;
    c->logN = p->logN;
    c->N = 1 << p->logN;
    c->L = p->L;
    c->K = p->K;
    c->alpha = p->alpha;
    c->dnum = (p->L + p->alpha - 1) / p->alpha;
    c->E = p->K + p->L;
    c->device = device;
    if (c->dnum > kMaxDigits) return HE_EINVAL;
    auto pad_width = [](int v) { return v <= 2 ? v : v <= 4 ? 4 : v <= 8 ? 8 : v <= 12 ? 12 : 16; };
    c->AP = pad_width(p->alpha);
    c->KP = pad_width(p->K);

    std::vector<u64> q = find_primes(p->logN, p->q_bits, p->L, {});
    if ((int)q.size() != p->L) return HE_EINVAL;
    std::vector<u64> sp = find_primes(p->logN, p->p_bits, p->K, q);
    if ((int)sp.size() != p->K) return HE_EINVAL;
    c->ext = sp;
    c->ext.insert(c->ext.end(), q.begin(), q.end());
    const int N = c->N, K = c->K, L = c->L, E = c->E, logN = c->logN;
    c->nt.resize(E);
    for (int e = 0; e < E; e++)
        if (!ntt_mod(c->ext[e], logN, &c->nt[e])) return HE_EINVAL;

    // the ciphertext primes descend, so a rescale residue r < q_{l-1} is
    // already reduced mod every q_i with i < l-1.

    c->psi.resize(E);
    c->w.assign(E, {});
    c->wsh.assign(E, {});
    c->iw.assign(E, {});
    c->iwsh.assign(E, {});
    c->ninv.resize(E);
    c->ninv_sh.resize(E);
    for (int e = 0; e < E; e++) {
        u64 m = c->ext[e];
        u64 psi = smallest_psi(m, logN);
        c->psi[e] = psi;
        u64 ipsi = inv(psi, m);
        std::vector<u64> pow_f(N), pow_i(N);
        pow_f[0] = pow_i[0] = 1;
        for (int k = 1; k < N; k++) {
            pow_f[k] = mul(pow_f[k - 1], psi, m);
            pow_i[k] = mul(pow_i[k - 1], ipsi, m);
        }
        auto &W = c->w[e], &Ws = c->wsh[e], &IW = c->iw[e], &IWs = c->iwsh[e];
        W.resize(N); Ws.resize(N); IW.resize(N); IWs.resize(N);
        for (int k = 0; k < N; k++) {
            u64 br = bitrev((u64)k, logN);
            W[k] = pow_f[br];
            Ws[k] = shoup(W[k], m);
            IW[k] = pow_i[br];
            IWs[k] = shoup(IW[k], m);
        }
        c->ninv[e] = inv((u64)N % m, m);
        c->ninv_sh[e] = shoup(c->ninv[e], m);
    }

    // ModDown constants
    c->PB.assign((size_t)L * c->KP, 0);
    c->PBP.assign((size_t)L * c->KP, 0);
    c->pinv.resize(L);
    c->phat_inv.resize(K);
    for (int k = 0; k < K; k++) {
        u64 pk = c->ext[k], v = 1;
        for (int k2 = 0; k2 < K; k2++)
            if (k2 != k) v = mul(v, c->ext[k2] % pk, pk);
        c->phat_inv[k] = pair(inv(v, pk), pk);
    }
    for (int i = 0; i < L; i++) {
        u64 qi = c->ext[K + i], P = 1;
        for (int k = 0; k < K; k++) {
            u64 v = 1;
            for (int k2 = 0; k2 < K; k2++)
                if (k2 != k) v = mul(v, c->ext[k2] % qi, qi);
            c->PB[(size_t)i * c->KP + k] = split28(v);
            P = mul(P, c->ext[k] % qi, qi);
        }
        c->pinv[i] = pair(inv(P, qi), qi);
        for (int k = 0; k < K; k++) {
            u64 v = 1;
            for (int k2 = 0; k2 < K; k2++)
                if (k2 != k) v = mul(v, c->ext[k2] % qi, qi);
            c->PBP[(size_t)i * c->KP + k] = split28(mul(v, c->pinv[i].x, qi));
        }
    }

    // per level
    c->host_levels.assign(L + 1, HostLevel());
    for (int l = 1; l <= L; l++) {
        HostLevel &H = c->host_levels[l];
        const int beta = (l + c->alpha - 1) / c->alpha, El = K + l;
        const int A = c->AP;
        H.ws = layout_for(l, K, c->alpha);
        const WsLayout &W = H.ws;
        // ModUp tables and the iNTT scale N^-1 * Qhat_{j,i}^-1
        H.modupB.assign((size_t)beta * El * A, 0);
        for (int j = 0; j < beta; j++) {
            int lo = j * c->alpha, hi = std::min((j + 1) * c->alpha, l);
            for (int i = lo; i < hi; i++) {
                u64 qi = c->ext[K + i], qh = 1;
                for (int i2 = lo; i2 < hi; i2++)
                    if (i2 != i) qh = mul(qh, c->ext[K + i2] % qi, qi);
                u64 sc = mul(c->ninv[K + i], inv(qh, qi), qi);
                // tensor fields (the fused first pass): limb i, product d2, keep d0..d2
                H.intt1.push_back(NttJob{(unsigned)(W.d2 + i), (unsigned)(W.y + i), (unsigned)(K + i), 0, sc,
                                         shoup(sc, qi), 0, (unsigned)i | (2u << 16) | (1u << 18), 0, 0});
            }
            for (int e = 0; e < El; e++) {
                bool own = e >= K && (e - K) >= lo && (e - K) < hi;
                if (own) continue;
                u64 t = c->ext[e];
                for (int i = lo; i < hi; i++) {
                    u64 v = 1;
                    for (int i2 = lo; i2 < hi; i2++)
                        if (i2 != i) v = mul(v, c->ext[K + i2] % t, t);
                    H.modupB[((size_t)j * El + e) * A + (i - lo)] = split28(v);
                }
                H.ntt_up.push_back(NttJob{(unsigned)(W.u + (size_t)j * El + e), (unsigned)(W.u + (size_t)j * El + e),
                                          (unsigned)e, 0, 0, 0});
            }
        }
        const u64 ql = c->ext[K + l - 1];
        H.intt1f = H.intt1;
        for (int h = 0; h < 2; h++)
            H.intt1f.push_back(NttJob{(unsigned)((h ? W.d1 : W.d0) + l - 1), (unsigned)(W.r + h), (unsigned)(K + l - 1),
                                      0, c->ninv[K + l - 1], c->ninv_sh[K + l - 1], 0,
                                      (unsigned)(l - 1) | ((unsigned)h << 16), 0, 0});
        for (int h = 0; h < 2; h++)
            for (int k = 0; k < K; k++) {
                u64 pk = c->ext[k];
                u64 sc = mul(c->ninv[k], c->phat_inv[k].x, pk);
                // ci: the key-switch row and half (the first pass that computes the sums itself)
                H.intt2.push_back(NttJob{(unsigned)(W.ks + (size_t)h * El + k), (unsigned)(W.ys + (size_t)h * K + k),
                                         (unsigned)k, 0, sc, shoup(sc, pk), 0, (unsigned)k | ((unsigned)h << 16), 0, 0});
            }
        H.intt2f = H.intt2;
        for (int h = 0; h < 2; h++)
            H.intt2f.push_back(NttJob{(unsigned)(W.ks + (size_t)h * El + K + l - 1), (unsigned)(W.r + 2 + h),
                                      (unsigned)(K + l - 1), 0, c->ninv[K + l - 1], c->ninv_sh[K + l - 1], 0,
                                      (unsigned)(K + l - 1) | ((unsigned)h << 16), 0, 0});
        // one division by M = P q_{l-1}: y_k = x_k [Mhat_k^-1]_{p_k}, Mhat_k = Phat_k q_{l-1};
        // the conversion constants [Mhat_k P^-1]_{q_i} = [Phat_k P^-1 q_{l-1}]_{q_i}
        for (int h = 0; h < 2; h++)
            for (int k = 0; k < K; k++) {
                u64 pk = c->ext[k];
                u64 sc = mul(mul(c->ninv[k], c->phat_inv[k].x, pk), inv(ql % pk, pk), pk);
                H.intt2pq.push_back(NttJob{(unsigned)(W.ks + (size_t)h * El + k),
                                           (unsigned)(W.ys + (size_t)h * K + k), (unsigned)k, 0, sc, shoup(sc, pk), 0,
                                           (unsigned)k | ((unsigned)h << 16), 0, 0});
            }
        for (int h = 0; h < 2; h++) H.intt2pq.push_back(H.intt2f[(size_t)2 * K + h]);
        H.pbpq.assign((size_t)std::max(l - 1, 1) * c->KP, 0);
        for (int i = 0; i + 1 < l; i++) {
            u64 qi = c->ext[K + i];
            for (int k = 0; k < K; k++) {
                u64 v = 1;
                for (int k2 = 0; k2 < K; k2++)
                    if (k2 != k) v = mul(v, c->ext[k2] % qi, qi);
                H.pbpq[(size_t)i * c->KP + k] = split28(mul(mul(v, c->pinv[i].x, qi), ql % qi, qi));
            }
        }
        for (int h = 0; h < 2; h++)
            for (int i = 0; i < l; i++)
                H.ntt_conv.push_back(NttJob{(unsigned)(W.z + (size_t)h * l + i), (unsigned)(W.z + (size_t)h * l + i),
                                            (unsigned)(K + i), 0, 0, 0, 0, ((unsigned)h << 31) | (unsigned)i,
                                            (unsigned)((h ? W.d1 : W.d0) + i), (unsigned)(W.ks + (size_t)h * El + K + i)});
        for (int h = 0; h < 2; h++)
            for (int i = 0; i + 1 < l; i++)
                H.ntt_z.push_back(NttJob{(unsigned)(W.z + (size_t)h * (l - 1) + i),
                                         (unsigned)(W.z + (size_t)h * (l - 1) + i), (unsigned)(K + i), 0, 0, 0, 0,
                                         ((unsigned)h << 31) | (unsigned)i, (unsigned)((h ? W.d1 : W.d0) + i),
                                         (unsigned)(W.ks + (size_t)h * El + K + i)});
        // rescale on its own: src offsets are relative to the input ciphertext
        for (int h = 0; h < 2; h++)
            H.rs_intt.push_back(NttJob{(unsigned)((size_t)h * l + l - 1), (unsigned)(W.r + h), (unsigned)(K + l - 1), 0,
                                       c->ninv[K + l - 1], c->ninv_sh[K + l - 1]});
        for (int h = 0; h < 2; h++)
            for (int i = 0; i + 1 < l; i++)
                H.rs_ntt.push_back(NttJob{(unsigned)(W.r + h), (unsigned)(W.z + (size_t)h * (l - 1) + i), (unsigned)(K + i),
                                          0, 0, 0});
        H.qinv_last.resize(l > 1 ? l - 1 : 1);
        for (int i = 0; i + 1 < l; i++) {
            u64 qi = c->ext[K + i];
            u64 qinv = inv(ql % qi, qi);
            H.qinv_last[i] = pair(qinv, qi);
        }
    }
    if (!device) return HE_OK;
    c->tc = build_tc(c);
    if (cudaHostAlloc((void **)&c->flag, sizeof(unsigned), cudaHostAllocMapped) != cudaSuccess) return HE_ECUDA;
    *c->flag = 0;
    if (cudaHostGetDevicePointer((void **)&c->d_flag, c->flag, 0) != cudaSuccess) return HE_ECUDA;

    // ---- device arena -------------------------------------------------------
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_primes = take(sizeof(DevPrime) * E);
    std::vector<size_t> o_w(E), o_iw(E);
    for (int e = 0; e < E; e++) {
        o_w[e] = take(sizeof(ulonglong2) * N);
        o_iw[e] = take(sizeof(ulonglong2) * N);
    }
    const size_t o_PB = take(sizeof(u64) * c->PB.size());
    const size_t o_PBP = take(sizeof(u64) * c->PBP.size());
    const size_t o_tPB = take(c->tc_PB.size()), o_tPBP = take(c->tc_PBP.size()), o_tlast = take(c->tc_last.size()),
                 o_tPBt = take(sizeof(TcTarget) * c->tc_PB_t.size()),
                 o_tPBPt = take(sizeof(TcTarget) * c->tc_PBP_t.size());
    const size_t o_pinv = take(sizeof(ulonglong2) * L);
    const size_t o_levels = take(sizeof(DevLevel) * (L + 1));
    // per level: the NTT lists of one job, one limb per group (a group's limbs
    // run one after another in their CTAs: a single job's lists are too short
    // to give up CTAs for it; at N = 2^16, level 24, 211 us against 236 with
    // two limbs per group and 264 with four)
    constexpr int NL = 10;  // job lists per level
    struct LvlOff { size_t modupB, qinv, pbpq, tc[4], j[NL]; };
    std::vector<LvlOff> lo(L + 1);
    std::vector<std::vector<std::vector<NttGroup>>> gl(L + 1, std::vector<std::vector<NttGroup>>(NL));
    for (int l = 1; l <= L; l++) {
        HostLevel &H = c->host_levels[l];
        lo[l].modupB = take(sizeof(u64) * H.modupB.size());
        lo[l].qinv = take(sizeof(ulonglong2) * H.qinv_last.size());
        lo[l].pbpq = take(sizeof(u64) * H.pbpq.size());
        lo[l].tc[0] = take(H.tc_up.size());
        lo[l].tc[1] = take(sizeof(TcTarget) * H.tc_up_t.size());
        lo[l].tc[2] = take(H.tc_pq.size());
        lo[l].tc[3] = take(sizeof(TcTarget) * H.tc_pq_t.size());
        const std::vector<NttJob> *lists[NL] = {&H.intt1, &H.intt1f, &H.ntt_up, &H.intt2, &H.intt2f,
                                                &H.ntt_conv, &H.ntt_z, &H.rs_intt, &H.rs_ntt, &H.intt2pq};
        for (int t = 0; t < NL; t++) {
            gl[l][t] = group_jobs(*lists[t], 1);
            lo[l].j[t] = take(sizeof(NttGroup) * std::max<size_t>(1, gl[l][t].size()));
        }
    }
    c->arena_bytes = off;
    if (cudaGetDevice(&c->device_id) != cudaSuccess) return HE_ECUDA;
    if (cudaMalloc(&c->arena, off) != cudaSuccess) return HE_ECUDA;
    std::vector<unsigned char> img(off, 0);
    char *base = (char *)c->arena;
    std::vector<DevPrime> dp(E);
    const int direct = ntt_direct_stages(logN);
    if (direct <= 0) return HE_EINVAL;
    const int sd = logN - direct;  // first stage with transposed runs
    for (int e = 0; e < E; e++) {
        u64 m = c->ext[e];
        int b = bitlen(m);
        dp[e].q = m;
        dp[e].r64 = (u64)((((u128)1) << 64) / m);
        dp[e].s = (unsigned)(b - 2);
        dp[e].mu = (u64)(((u128)1 << (64 + b - 2)) / m);
        dp[e].pad = 0;
        dp[e].nt = c->nt[e];
        dp[e].w = (const ulonglong2 *)(base + o_w[e]);
        dp[e].iw = (const ulonglong2 *)(base + o_iw[e]);
        ulonglong2 *W = (ulonglong2 *)(img.data() + o_w[e]);
        ulonglong2 *IW = (ulonglong2 *)(img.data() + o_iw[e]);
        for (int k = 0; k < 1 << sd; k++) {
            W[k] = split_tw(c->w[e][k], c->wsh[e][k], m, dp[e].nt.s);
            IW[k] = split_tw(c->iw[e][k], c->iwsh[e][k], m, dp[e].nt.s);
        }
        // The last `direct` stages' runs are stored transposed (the NTT's
        // contiguous pass reads them one entry per thread): stage m = 2^sigma,
        // lp = sigma - sd, entry m + T 2^lp + j moves to m + j 2^sd + T.
        for (int sigma = sd; sigma < logN; sigma++) {
            const int lp = sigma - sd;
            const size_t run = (size_t)1 << sigma;
            for (size_t T = 0; T < ((size_t)1 << sd); T++)
                for (size_t j = 0; j < ((size_t)1 << lp); j++) {
                    const size_t from = run + (T << lp) + j, to = run + (j << sd) + T;
                    W[to] = split_tw(c->w[e][from], c->wsh[e][from], m, dp[e].nt.s);
                    IW[to] = split_tw(c->iw[e][from], c->iwsh[e][from], m, dp[e].nt.s);
                }
        }
    }
    memcpy(img.data() + o_primes, dp.data(), sizeof(DevPrime) * E);
    memcpy(img.data() + o_PB, c->PB.data(), sizeof(u64) * c->PB.size());
    memcpy(img.data() + o_PBP, c->PBP.data(), sizeof(u64) * c->PBP.size());
    memcpy(img.data() + o_pinv, c->pinv.data(), sizeof(ulonglong2) * L);
    if (c->tc) {
        memcpy(img.data() + o_tPB, c->tc_PB.data(), c->tc_PB.size());
        memcpy(img.data() + o_tPBP, c->tc_PBP.data(), c->tc_PBP.size());
        memcpy(img.data() + o_tlast, c->tc_last.data(), c->tc_last.size());
        memcpy(img.data() + o_tPBt, c->tc_PB_t.data(), sizeof(TcTarget) * c->tc_PB_t.size());
        memcpy(img.data() + o_tPBPt, c->tc_PBP_t.data(), sizeof(TcTarget) * c->tc_PBP_t.size());
    }
    c->dev_levels.assign(L + 1, DevLevel());
    c->jobs.assign(L + 1, LevelJobs());
    for (int l = 1; l <= L; l++) {
        HostLevel &H = c->host_levels[l];
        DevLevel &D = c->dev_levels[l];
        memset(&D, 0, sizeof(D));
        D.l = l;
        D.beta = (l + c->alpha - 1) / c->alpha;
        D.E = K + l;
        D.A = c->AP;
        const WsLayout &Wl = H.ws;
        D.o_d0 = (unsigned)Wl.d0; D.o_d1 = (unsigned)Wl.d1; D.o_d2 = (unsigned)Wl.d2; D.o_y = (unsigned)Wl.y;
        D.o_u = (unsigned)Wl.u; D.o_ks = (unsigned)Wl.ks; D.o_ys = (unsigned)Wl.ys; D.o_r = (unsigned)Wl.r;
        D.o_z = (unsigned)Wl.z; D.o_total = (unsigned)Wl.total;
        for (int j = 0; j < D.beta; j++) {
            D.dig_lo[j] = j * c->alpha;
            D.dig_n[j] = std::min((j + 1) * c->alpha, l) - j * c->alpha;
        }
        memcpy(img.data() + lo[l].modupB, H.modupB.data(), sizeof(u64) * H.modupB.size());
        memcpy(img.data() + lo[l].qinv, H.qinv_last.data(), sizeof(ulonglong2) * H.qinv_last.size());
        memcpy(img.data() + lo[l].pbpq, H.pbpq.data(), sizeof(u64) * H.pbpq.size());
        D.modupB = (const u64 *)(base + lo[l].modupB);
        D.qinv_last = (const ulonglong2 *)(base + lo[l].qinv);
        D.pbpq = (const u64 *)(base + lo[l].pbpq);
        if (c->tc) {
            memcpy(img.data() + lo[l].tc[0], H.tc_up.data(), H.tc_up.size());
            memcpy(img.data() + lo[l].tc[1], H.tc_up_t.data(), sizeof(TcTarget) * H.tc_up_t.size());
            memcpy(img.data() + lo[l].tc[2], H.tc_pq.data(), H.tc_pq.size());
            memcpy(img.data() + lo[l].tc[3], H.tc_pq_t.data(), sizeof(TcTarget) * H.tc_pq_t.size());
            D.tc_up = (const unsigned char *)(base + lo[l].tc[0]);
            D.tc_up_t = (const TcTarget *)(base + lo[l].tc[1]);
            D.tc_pq = (const unsigned char *)(base + lo[l].tc[2]);
            D.tc_pq_t = (const TcTarget *)(base + lo[l].tc[3]);
            D.up_nch = H.up_nch;
            D.up_tc = H.up_tc;
            D.up_tp = H.up_tp;
            D.up_bytes = H.up_bytes;
        }
        const NttGroup *dptr[NL];
        int cnt[NL];
        for (int t = 0; t < NL; t++) {
            const std::vector<NttGroup> &G = gl[l][t];
            if (!G.empty()) memcpy(img.data() + lo[l].j[t], G.data(), sizeof(NttGroup) * G.size());
            dptr[t] = (const NttGroup *)(base + lo[l].j[t]);
            cnt[t] = (int)G.size();
        }
        LevelJobs &J = c->jobs[l];
        J.intt1 = dptr[0];    J.n_intt1 = cnt[0];
        J.intt1f = dptr[1];   J.n_intt1f = cnt[1];
        J.ntt_up = dptr[2];   J.n_ntt_up = cnt[2];
        J.intt2 = dptr[3];    J.n_intt2 = cnt[3];
        J.intt2f = dptr[4];   J.n_intt2f = cnt[4];
        J.ntt_conv = dptr[5]; J.n_ntt_conv = cnt[5];
        J.ntt_z = dptr[6];    J.n_ntt_z = cnt[6];
        J.rs_intt = dptr[7];  J.n_rs_intt = cnt[7];
        J.rs_ntt = dptr[8];   J.n_rs_ntt = cnt[8];
        J.intt2pq = dptr[9];  J.n_intt2pq = cnt[9];
    }
    memcpy(img.data() + o_levels, c->dev_levels.data(), sizeof(DevLevel) * (L + 1));
    if (cudaMemcpy(c->arena, img.data(), off, cudaMemcpyHostToDevice) != cudaSuccess) return HE_ECUDA;
    c->d_primes = (DevPrime *)(base + o_primes);
    c->d_PB = (const u64 *)(base + o_PB);
    c->d_PBP = (const u64 *)(base + o_PBP);
    c->d_tc_PB = (const unsigned char *)(base + o_tPB);
    c->d_tc_PBP = (const unsigned char *)(base + o_tPBP);
    c->d_tc_last = (const unsigned char *)(base + o_tlast);
    c->d_tc_PB_t = (const TcTarget *)(base + o_tPBt);
    c->d_tc_PBP_t = (const TcTarget *)(base + o_tPBPt);
    c->d_pinv = (const ulonglong2 *)(base + o_pinv);
    c->d_levels = (DevLevel *)(base + o_levels);
    if (configure_ntt(c) != cudaSuccess) return HE_ECUDA;
    if (c->tc && configure_conversions(c) != cudaSuccess) return HE_ECUDA;
    return HE_OK;
}

}  // namespace he
