// How many CTAs share an event's scoring in the prefill kernel (akv_event_prefill.cuh), by the shape of the call. Plain C++, so
// that it can also be compiled for the host by itself.
#pragma once

namespace akv {

constexpr int kSplitStageRows = 64;   // rows of a stage of the kernel's ring
constexpr int kSplitStages = 8;       // a CTA's share is a multiple of so many stages (rotations are taken afresh there)

// The longest share, in stages, when `split` CTAs take an event's stages.
inline int split_share(int stages, int split) { return ((stages + split - 1) / split + kSplitStages - 1) / kSplitStages * kSplitStages; }

// Two CTAs fit an SM, so up to as many events as SMs leave half of the places empty. Where every CTA of a cluster has an SM to itself
// (148 SMs: 33 clusters of four, 74 of two) a split costs some 2 us at the start and the rounding of the shares, and pays from 1024
// rows on by four, from 2048 by two. Where CTAs share an SM they score at half the rate, or nearly, when every row takes its own
// rotation (positions that are not spaced like those a stage before, which the host does not know): then four pay up to two per SM and
// 3072 rows, and two only where the longest share is hardly more than half of the event, and where that half is known (ragged:
// candidate counts, which only the device knows). Measured, us per call by 1 / 2 / 4 CTAs per event:
//   regular positions, lambda 0.5 (mean of six batches): 37 events of 1100 rows 62 / 62 / 57, 56 of 4096 93 / 77 / 70, 66 of 4096 91 / 76 /
//     71, 74 of 2113 73 / 68 / 72, of 4096 91 / 74 / 77, 112 of 2048 73 / 67, of 2113 74 / 71, of 3072 83 / 73, of 3136 84 / 78, 148 of 2113
//     76 / 76, of 3072 84 / 78, of 4096 94 / 85
//   the same, lambda 1: 112 of 2048 80 / 77, of 2113 82 / 84, of 3072 90 / 84, of 3136 93 / 93, 148 of 2048 82 / 82, of 2113 84 / 88, of
//     3072 91 / 89, of 3136 93 / 93
//   the same, lambda 0: 33 of 1100 29 / 30 / 25, 37 of 1100 29 / 31 / 31, of 1536 33 / 31 / 33, 66 of 4096 58 / 44 / 41, 74 of 2049 40 / 38 /
//     49, of 4096 59 / 45 / 55, 90 of 2048 39 / 41, 112 of 2113 42 / 48, of 3008 50 / 48, of 3136 52 / 57, of 4096 60 / 58, 148 of 2113 44 / 49,
//     of 3008 51 / 49, of 3136 54 / 58
//   irregular positions, lambda 0.5: 37 of 1100 79 / 79 / 66, 56 of 4096 147 / 107 / 95, 74 of 4096 157 / 116 / 121, 112 of 2113 102 / 117,
//     of 2048 101 / 93, of 3072 125 / 118, of 3136 126 / 140, of 3904 142 / 143, 148 of 2048 101 / 101, of 3072 125 / 125, of 4096 147 / 145
//   the same, lambda 1 (the one kind of call that the last line of the rule makes slower): 112 of 2048 109 / 109, of 3008 131 / 134, of
//     3904 151 / 158, 148 of 2048 110 / 112, of 3008 132 / 134
//   the same, lambda 0: 37 of 2113 70 / 61 / 70, 74 of 2113 70 / 62 / 82, 112 of 2113 72 / 94, of 3072 95 / 95, of 4096 120 / 119
//   300 candidates of 4096 rows, lambda 0: 28 events 19 / 21 / 21, 74 20 / 23 / 31, 112 21 / 27; lambda 0.5: 74 51 / 52 / 53, 148 52 / 55
// With more events than SMs it never pays: 160 events of 2048 rows 76 / 121, of 5000 121 / 156; 210 of 4096 107 / 142.
inline int prefill_split(long long events, int N, int sms, bool topk, bool ragged) {
    const int stages = (N + kSplitStageRows - 1) / kSplitStageRows;
    if (events * 9 <= sms * 2ll) return stages >= 16 ? 4 : 1;                  // an SM for each of four
    if (events * 4 <= sms) return stages >= (topk ? 24 : 16) ? 4 : 1;
    if (events * 9 <= sms * 4ll && stages >= 48) return 4;                     // two on every SM
    if (events * 2 <= sms) return stages >= 32 ? 2 : 1;                        // an SM for each of two
    if (events > sms || ragged || stages < (topk ? 44 : 32)) return 1;
    return split_share(stages, 2) * 33 <= stages * 17 ? 2 : 1;
}

// How many of a call's events, the last ones, are left to a launch of their own: those beyond the full waves of two per SM, where
// sharing their scoring shortens the call, at most half as many as SMs, for candidates known to be many. It does for top-k, whose selection is
// short: with a penalty such an event is mostly selection, and the places that fall free early have it half done by the time that the last full
// wave ends. Measured, us per call in one
// launch / two, 296 events and 8, 37, 65, 74 more, lambda 0: 2113 rows 83 / 87, 93 / 100, 85 / 93, 85 / 93, 3072 rows 102 / 97, 114 / 110,
// 103 / 102, 104 / 102, 4096 rows 124 / 108, 138 / 126, 127 / 118, 127 / 118, 5000 rows 146 / 126, 160 / 147, 148 / 136, 148 / 134, 896 events
// of 4096 rows 260 / 243; lambda 0.5: 304 events of 1100 rows 114 / 139, of 4096 179 / 181, 896 of 4096 359 / 372.
inline long long prefill_tail(long long events, int N, int sms, bool topk, bool ragged) {
    const long long places = 2ll * sms, rest = events % places;
    if (!topk || ragged || events < places || rest * 2 > sms || (N + kSplitStageRows - 1) / kSplitStageRows < 48) return 0;
    return prefill_split(rest, N, sms, topk, ragged) > 1 ? rest : 0;
}
// How many CTAs share such an event: four or two, as long as each has an SM. (Four each up to 65 events, as in a call of their own, take no less,
// and in two and three streams with such a call each 296 + 64 events of 3072 rows 195 and 282 us instead of 174 and 264, of 4096 223 and 320 instead of
// 209 and 311; in one launch 166 and 247, 202 and 302.)
inline int prefill_tail_split(long long tail, int sms) { return tail * 4 <= sms ? 4 : 2; }

}  // namespace akv
