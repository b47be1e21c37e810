// launch_shape.h -- how many CTAs a single-source CSR search launches.  Host
// arithmetic only, apart from the CUDA sources so that it can be checked alone.
#pragma once

namespace bfsrt {

// Graphs of up to so many vertices launch one CTA per SM unless told otherwise: their
// levels are the chain of their reads and barriers, not work to spread, and the launch
// halves the arrivals of a barrier.  By vertices alone, because edges do not move the
// line in a direction-optimizing search: one CTA per SM is 1 to 10 % faster at 2^10,
// 2^12, 2^14, 2^16 and 2^18 vertices with 4, 16, 64 and 256 edges each (R-MAT; 2^18 with
// 16: 77.8 and 82.6 us, with 256: 73.6 and 74.9) and on Erdos-Renyi graphs of 2 to 600
// edges a vertex (60 K vertices with 600: 57 and 63 us); R-MAT 20 is even at 107 / 108.
// Searches that stay bottom-up, or draw their directions, gain 2 to 6 % up to 2^14
// vertices and are undecided at 2^18 (R-MAT of 256 edges 1362 and 1316 us, Erdos-Renyi
// of 100 1265 and 1319).  One that stays top-down reads every edge with scattered
// claims, and has those to spread (R-MAT 17: 140 us with one CTA per SM, 134 with two).
constexpr long long kSmallN = 1LL << 18;
constexpr int kModeTdOnly = 1;   // BFS_MODE_TD_ONLY

inline bool one_cta_by_default(long long n, int mode) { return n <= kSmallN && mode != kModeTdOnly; }

// CTAs of the launch: options.ctas_per_sm per SM, or as many as fit (`resident`) by default
inline int search_grid(long long n, int mode, int ctas_per_sm, int sms, int resident) {
    const int per_sm = ctas_per_sm > 0 ? ctas_per_sm : one_cta_by_default(n, mode) ? 1 : 0;
    return per_sm > 0 && (long long)per_sm * sms < resident ? per_sm * sms : resident;
}

// The two settings of options.ctas_per_sm that the autotuner times (direction-optimizing
// searches): one CTA per SM, and as many as fit -- 0 where the default means that.
inline void tuner_ctas(long long n, int mode, int sms, int resident, int (&out)[2]) {
    out[0] = 1;
    out[1] = one_cta_by_default(n, mode) ? (resident + sms - 1) / sms : 0;
}

}  // namespace bfsrt
