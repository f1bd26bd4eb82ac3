// shape_rule.h -- transform shapes by batch size, for degrees where none is
// set. Host code without CUDA types, so that it can be tested by itself.
#pragma once
#include <stdint.h>

#include <algorithm>

namespace he {

// Batches of at most this many words are small: one 512-thread CTA an SM of
// the 8-word shapes covers them.
inline uint64_t small_batch_words(uint32_t sms) { return (uint64_t)sms * 4096; }

// 2^16 in 2^12-word blocks takes clusters of 16 CTAs, more than the portable 8:
// the caller asks the GPU whether it can place one (`wide` below). Where it
// cannot, the degree's default, in clusters of 8, is taken.
constexpr int kWideLogB = 12;

// Shape of a batch of `items` limbs when none is set for the degree (0, 0: the
// default, 16 words a thread). Small batches take 8 words a thread, in one CTA
// up to 2^12 and in 2^12-word blocks above: twice the threads on the batch, and
// half the chain of butterflies in each, which is what a launch costs that does
// not fill the GPU. Above the limit the 16-word shapes' fewer exchanges win.
// Measured against the default, forward / inverse, us:
//   2^10: 76 limbs 6.4 / 5.8 -> 4.5 / 4.6, 608 7.9 / 7.3 -> 6.5 / 6.2
//   2^12: 19 limbs 8.4 / 8.5 -> 7.1 / 6.9, 152 8.7 / 8.9 -> 7.1 / 7.2; equal at
//     256, 5 % slower at 512
//   2^13: 76 limbs 10.1 / 10.4 -> 9.0 / 8.9; up to 19 limbs four 2^11-word blocks
//     of 16-word threads, 9.9 / 10.3 -> 8.7 / 8.5
//   2^14: 33 limbs 10.8 / 10.1 -> 8.9 / 9.0; 2^15: 14 limbs 11.4 / 11.2 -> 9.7 / 9.5.
//     Clusters of four and eight do not reach every SM: with more than 3/4 of
//     the words (38 and 16 limbs) a second CTA lands on some, 13.7 / 14.4
//     against 11.5 / 11.3. The inverse of up to 8 limbs of 2^14 is 2 % faster
//     in the default (8.25 against 8.41; 9 to 12 limbs 1 to 2 %, 16
//     limbs 9.43 against 8.47).
//   2^16: 2^12-word blocks in clusters of 16 at every size (one limb 17.3 -> 12.2,
//     128 limbs 117 / 109 -> 101 / 102).
inline void auto_shape(int log_n, uint32_t items, bool inv, uint32_t sms, bool wide, int *lb, int *le)
{
    const uint64_t words = (uint64_t)items << log_n, small = small_batch_words(sms);
    if (log_n == 16) {
        if (wide) *lb = kWideLogB, *le = 4;
    } else if (log_n == 13 && (uint64_t)items * 8 <= sms) {
        *lb = 11, *le = 4;
    } else if (log_n >= 14 ? words <= small / 4 * 3 && !(log_n == 14 && inv && items <= 8) : words <= small) {
        *lb = std::min(log_n, 12), *le = 3;
    }
}

// The same for the fused product. Three transforms in a row: at 2^13 the four
// 2^11-word blocks hold out longer, as long as each CTA has an SM of its own.
// Clusters of four do not reach every SM: against one pair of 8-word-thread
// blocks, us, 27 limbs 20.5 / 21.9, 36 20.7 / 22.0, but 38 23.9 / 22.0 and 57
// 24.5 / 22.1 (of 152 SMs; 37 like 38).
inline void product_shape(int log_n, uint32_t items, uint32_t sms, bool wide, int *lb, int *le)
{
    if (log_n == 13 && (uint64_t)items * 4 + 8 <= sms)
        *lb = 11, *le = 4;
    else
        auto_shape(log_n, items, false, sms, wide, lb, le);
}

}  // namespace he
