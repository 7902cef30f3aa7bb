// ntt_mod.h -- per-prime constants of the NTT's twiddle product and the range
// bounds they are valid for (shared by the kernels and the context builder).
#pragma once
#include <cstdint>

typedef uint64_t u64;

namespace he {

// What a pass does against growth beyond 64 bits.  Forward: nothing, fold when
// the first pass stores, fold after every round, or also after a round's
// second stage.  Inverse: the sums of a
// round's last stage are always folded; optionally every output of a round,
// and the sums after a round's second stage.
enum NttFlags : uint32_t {
    kFwdFoldPass = 1,
    kFwdFoldRound = 2,
    kInvFoldAll = 4,
    kInvFoldSecond = 8,
    kFwdFoldSecond = 32,
    kFastFinal = 16  // fold_tw of any word is below 3q
};

struct NttMod {
    u64 cf;           // multiple of q, at least any forward twiddle product
    u64 ci;           // multiple of q, at least any inverse stage input
    u64 cz;           // multiple of q, at least any forward output
    uint32_t c;       // 2^(32+s) mod q
    uint32_t s;       // split position of the twiddles: max(0, bitlen(q) - 31)
    uint32_t p2;      // 2^s
    uint32_t flags;
};

// The constants of one prime at one ring size, from exact worst-case ranges;
// false if some range could not be kept below 2^64 (never for primes as the
// contexts choose them: tests/test_gpu_ntt_ranges.py).
bool ntt_mod(u64 q, int logN, NttMod *out);

}  // namespace he

using he::NttMod;
