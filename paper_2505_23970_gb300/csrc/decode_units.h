// How decode at head_dim 128 numbers its work with 32-bit ints (host arithmetic).
#pragma once
#include <cstdint>
#include <initializer_list>

namespace gc {

// What a pair (request, kv head) costs beyond its keys, counted as keys in front of
// it: its look-ups and merge take a CTA about as long as 256 keys.  Shares of equal
// keys alone left the CTAs of the short contexts running when the others were done,
// SMs busy 75 % of the time on 64 multi-turn contexts over 8-bit pages (146 us; with
// 128, 256, 384 keys 131, 123, 124); one context of 9000 keys 19.1 us, now 16.2.
constexpr int kPairKeys = 256;

// Keys per unit as a shift, and the units in front of each pair's keys.
struct DecodeUnits {
  int shift, lead;
};

// For `pairs` pairs of at most `cap` keys, `margin` being what the kernel adds to
// the count.  Units of 16 keys where a 32-bit count can hold all of the block
// tables' capacity, of 128 keys otherwise, then with the allowance if it fits too.
inline DecodeUnits decode_units(int64_t pairs, int64_t cap, int64_t margin) {
  const int64_t per_pair = (INT32_MAX - margin) / pairs;  // units it may have
  for (const int shift : {4, 7}) {
    const int lead = kPairKeys >> shift;
    if (((cap - 1) >> shift) + 1 + lead <= per_pair) return {shift, lead};
  }
  return {7, 0};
}

}  // namespace gc
