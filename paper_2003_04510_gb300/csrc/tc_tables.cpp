// tc_tables.cpp -- constant images of the tensor-core base conversions (tc.cuh).
#include <algorithm>
#include <cstring>

#include "he_internal.h"
#include "host_math.h"

namespace he {

using namespace hm;

namespace {

// Offsets of the planes (tc.cuh), multiples of 8192, so that (2^23 + offset) /
// 2048 has eleven significant bits, and the largest magnitudes they allow.
// Planes 0 to 4: a pair is P0 + 512 P1 + 513 kTcOff + 0x4B000000, in 32 signed
// bits.  The last one, whose digits are larger for 55-bit targets: 512 (P5 +
// kTcOffTop) + P4 + kTcOff, in 32 unsigned bits.
constexpr int kTcOff = 603 * 8192, kTcMass = 3200000, kTcOffTop = 510 * 8192;
constexpr long long kTcPair = 513ll * kTcOff + 0x4B000000ll - (1ll << 32);
static_assert(kTcPair < 0 && kTcMass <= kTcOff && kTcOff + kTcMass < (1 << 23) && kTcPair - 513ll * kTcMass > -(1ll << 31) &&
                  kTcPair + 513ll * kTcMass < (1ll << 31),
              "pairs of planes");
static_assert(2 * kTcOffTop < (1 << 23) && 512ll * 2 * kTcOffTop + (1 << 23) < (1ll << 32), "the last pair");

}  // namespace

uint16_t half_of(int v)
{
    if (v == 0) return 0;
    const uint16_t sign = v < 0 ? 0x8000 : 0;
    const unsigned m = (unsigned)(v < 0 ? -v : v);
    int e = 0;
    while ((m >> e) > 1) e++;
    return (uint16_t)(sign | ((e + 15) << 10) | ((e <= 10 ? m << (10 - e) : m >> (e - 10)) & 0x3ff));
}

int tc_groups(int nsrc) { return (nsrc + 3) / 4; }

bool tc_source_ok(u64 p) { const int b = bitlen(p); return b > 45 && b <= 55; }

uint32_t tc_off5(const std::vector<u64> &src)
{
    int b = 46;
    for (u64 p : src) b = std::max(b, bitlen(p));
    return ((uint32_t)half_of(-(1024 + (1 << (b - 46)))) << 16) | half_of(-1280);
}

// Image and target constants of out[t] = sum_i y_i c[t][i] mod q[t] for
// targets t < T (room for tp >= T of them; row 6t + p of the image is plane p
// of target t, a column of the product; rows = 6 tp rounded up to 16) and sources i < nsrc < 2^b each, b the longest
// source modulus.  false if a target or a plane is out of range.
bool tc_image(const std::vector<u64> &c, const std::vector<u64> &q, int T, const std::vector<u64> &src, int tp,
              unsigned char *image, TcTarget *targets)
{
    const int nsrc = (int)src.size(), G = tc_groups(nsrc), kp = (24 * G + 1 + 15) / 16 * 16;
    const int rows = (6 * tp + 15) / 16 * 16;
    int sb = 46;
    for (u64 p : src) {
        if (!tc_source_ok(p)) return false;
        sb = std::max(sb, bitlen(p));
    }
    const int top = 1 << (sb - 46);  // offset of a residue's last digit (of sb - 45 bits)
    std::vector<uint16_t> img((size_t)rows * kp, 0);
    auto at = [&](int row, int k) -> uint16_t & { return img[((size_t)(k / 8) * rows + row) * 8 + k % 8]; };
    u64 H = (u64)top << 45;
    for (int d = 0; d < 5; d++) H += 256ull << (9 * d);
    static const std::vector<uint16_t> halves = [] {  // the digits' f16, which the images hold by the hundred thousand
        std::vector<uint16_t> h(4097);
        for (int v = -2048; v <= 2048; v++) h[v + 2048] = half_of(v);
        return h;
    }();
    for (int t = 0; t < T; t++) {
        const u64 m = q[t];
        const int b = bitlen(m);
        if (b < 52 || b > 55) return false;
        const u64 two9 = shoup(512, m);
        u64 base = 0;
        std::vector<long> mass(6, 0);  // per plane: the largest magnitude its sum can reach
        for (int i = 0; i < nsrc; i++) {
            base = add(base, mul(H % m, c[(size_t)t * nsrc + i], m), m);
            u64 cd = c[(size_t)t * nsrc + i];  // [c 2^(9d)]_m
            for (int d = 0; d < 6; d++) {
                long long v = cd > m / 2 ? (long long)cd - (long long)m : (long long)cd;
                for (int p = 0; p < 6; p++) {
                    long long r = v;
                    if (p < 5) r = ((v + 256) & 511) - 256;
                    v = (v - r) / 512;
                    if (r < -2048 || r > 2048) return false;
                    at(6 * t + p, 24 * (i / 4) + 6 * (i % 4) + d) = halves[(int)r + 2048];
                    mass[p] += (long)(r < 0 ? -r : r) * (d < 5 ? 256 : top);
                }
                cd = cd * 512 - (u64)(((u128)cd * two9) >> 64) * m;  // Shoup: below 2 m
                cd = cd >= m ? cd - m : cd;
            }
        }
        for (int p = 0; p < 6; p++) {
            const int off = p < 5 ? kTcOff : kTcOffTop;
            if (mass[p] > (p < 5 ? kTcMass : kTcOffTop)) return false;
            at(6 * t + p, 24 * G) = half_of(((1 << 23) + off) / 2048);  // times the rows' 2048
        }
        // the pairs' constants at weights 1, 2^18 and 2^36
        const u64 low = sub(0, (u64)-kTcPair % m, m), high = 512ull * kTcOffTop + kTcOff;
        base = sub(base, add(mul(low, ((1ull << 18) + 1) % m, m), mul(high % m, (1ull << 36) % m, m), m), m);
        if (base < (1ull << 50)) base += m;  // the pairs are signed: their sum is above -2^50
        targets[t].base = base;
        targets[t].delta = (uint32_t)((1ull << b) - m);
        targets[t].shift = (uint32_t)(b - 36);
        if ((((1ull << b) - m) >> 31) != 0) return false;
    }
    for (int t = T; t < tp; t++) targets[t] = TcTarget{0, 0, 1};
    memcpy(image, img.data(), img.size() * 2);
    return true;
}

}  // namespace he
