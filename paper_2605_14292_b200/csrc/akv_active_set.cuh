// Which candidates make up an active set: the search for the key that bounds it. Plain C++ beside the counting, which the
// caller does (one warp, or a whole CTA), so that the search also runs on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define AKV_HD __host__ __device__ __forceinline__
#else
#define AKV_HD inline
#endif

namespace akv {

AKV_HD int highest_bit(uint32_t x) {   // of a non-zero word
#ifdef __CUDA_ARCH__
    return 31 - __clz((int)x);
#else
    return 31 - __builtin_clz(x);
#endif
}

// The set: every key above `key`, at most `cap` of them, and, where that leaves places and more keys equal `key` than fit,
// `ties` of those (the lowest slots), so that it has `cap` rows. No row left out has a larger key than `key`.
struct ActiveBound {
    uint32_t key;
    int ties;
};

// For keys of which more than `cap` reach `low`, the pool's threshold, and at most `cap` exceed kb | 0x3FFF (kb: the
// picks-th largest key with its 14 low bits open). The common leading bits of the two are the bound's own; the others come
// two a round from three counts, count3(v1, v2, v3, c1, c2, c3): c = the number of keys >= v. The search ends
//   - at any round that leaves `enough` to `cap` keys above the bound;
//   - after fourteen bits if `least` are: that places it to 1e-3 of the value as a rule, a row or two short of `cap`;
//   - else at the last bit. Fourteen bits from the sign bit on are a bucket of 3 % of the value: with scores close together
//     all of them may lie in one, and a bound at its end would leave the set empty or nearly so. The bound is then the
//     (cap + 1)-th largest key itself.
template <class Count3>
AKV_HD ActiveBound active_bound(uint32_t low, uint32_t kb, int cap, int enough, int least, Count3 count3) {
    const int top = highest_bit(((kb | 0x3FFFu) ^ low) | 2u) | 1;   // an odd bit number
    const int last = top > 13 ? top - 13 : 0;
    uint32_t v = top == 31 ? 0u : low & ~((2u << top) - 1u);
    int above = 0, c1, c2, c3;   // above: keys from v + step on (of the keys beyond the first range none are counted)
    for (int lo = top - 1;; lo -= 2) {
        const uint32_t v1 = v | (1u << lo), v2 = v | (2u << lo), v3 = v | (3u << lo);
        count3(v1, v2, v3, c1, c2, c3);
        if (c3 > cap) v = v3;
        else if (c2 > cap) { v = v2; above = c3; }
        else if (c1 > cap) { v = v1; above = c2; }
        else above = c1;
        if (above >= (lo > last ? enough : least)) return ActiveBound{v | ((1u << lo) - 1u), 0};
        if (lo == 0) break;
    }
    count3(v + 1u, v + 1u, v + 1u, above, c2, c3);
    return ActiveBound{v, cap - above};
}

}  // namespace akv
