// full_fix_plan.h -- how the FP64 full estimate's tensor-core recursion
// (full_fix_tc.cu) is cut into CTAs and launches, by sizes and the number of SMs
// alone, and the scratch that it takes.  Host code, no CUDA.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#include "special_fix.h"

namespace vk {

constexpr int kXP = 128;                              // lattice points per tile = MMA M
constexpr int kXB = 32;                               // panel width = MMA N
constexpr int kXK = 16;                               // history chunk (variables) = MMA K
constexpr int kXDig = 8;                              // digits
constexpr uint32_t kRowGroup = kXDig * 256;           // 8 rows: eight 256-byte digit matrices
constexpr uint32_t kXChunkA = (kXP / 8) * kRowGroup;  // 32,768
constexpr uint32_t kXChunkB = (kXB / 8) * kRowGroup;  // 8,192
constexpr int kFullP = 64;                            // lattice points per CTA of the integer form (full.cu)

struct FullFixPlan {
    int halves;         // tiles of 128 points a CTA (1 or 2)
    int64_t per_shift;  // CTAs a shift
    int64_t ctas;       // CTAs in all
    int64_t launch;     // CTAs a launch: the launches share one history buffer
    size_t tables;      // bytes of the rows' digits
    size_t history;     // bytes of a launch's history
};

// What the integer form holds in their place: its rows and its history.
inline size_t full_integer_bytes(int64_t D, int64_t N, int S) {
    const size_t points = (size_t)((N + kFullP - 1) / kFullP) * kFullP * S;
    return sizeof(fix::Digits) * (size_t)D * ((size_t)D + points);
}

// Halves: one CTA fits an SM, and a round of two-tile CTAs takes 1.23 (D = 64),
// 1.42 (256), 1.64 (512), 1.78 (1,021) or 1.90 (2,500) times a round of one-tile CTAs: two
// pay where they take nearly half the rounds.  N S = 24,000 (two rounds or one): D = 64
// 0.129 -> 0.084 ms, 256 0.54 -> 0.39, 512 1.25 -> 1.03, 1,021 3.48 -> 3.13; N S = 65,536
// (four or two): 2,500 32.4 -> 30.9.
// Launches: the history takes 16 bytes a y value, twice the integer form's.  So a launch
// takes whole rounds, up to four, as long as rows and history stay within what the
// integer form holds, and one round at least (0.62 MB a variable): D = 2,500, N S =
// 65,536 1.6 GB in two launches, 31.1 ms (2.6 GB in one, 30.9); D = 600, N S = 262,144 9.33
// against 9.30.
inline FullFixPlan full_fix_plan(int64_t D, int64_t N, int S, int sms) {
    auto ctas = [&](int64_t points) { return (N + points - 1) / points * S; };
    auto rounds = [&](int64_t n) { return (n + sms - 1) / sms; };
    const int64_t panels = (D + kXB - 1) / kXB, chunks = 2 * panels;
    FullFixPlan p;
    p.halves = N > kXP && 10 * rounds(ctas(kXP)) >= 19 * rounds(ctas(2 * kXP)) ? 2 : 1;
    p.ctas = ctas((int64_t)p.halves * kXP);
    p.per_shift = p.ctas / S;
    p.tables = (size_t)panels * chunks * kXChunkB;
    const size_t cta = (size_t)p.halves * chunks * kXChunkA, room = full_integer_bytes(D, N, S);
    const size_t fit = room > p.tables ? (room - p.tables) / (cta * sms) : 0;
    p.launch = std::min<int64_t>(p.ctas, sms * (int64_t)std::clamp<size_t>(fit, 1, 4));
    p.history = cta * p.launch;
    return p;
}

}  // namespace vk
