// sort_digits.h -- how the radix sort shares a key's bits over its passes. Plain C++: the host test of the shares
// compiles it alone.
#pragma once
#include <stdint.h>

struct SortDigit {
  int shift, bits;  // the pass sorts by bits shift .. shift + bits - 1 of the key
  uint32_t mask;    // of the digit, for every kernel of the pass: one that took more bits than were counted would find
                    // no counts for its digits, and write past the end
  int ballots;      // the scatter's instantiation, 4 to 8: bits, but 4 for fewer
};

inline int sort_passes(int key_bits) { return (key_bits + 7) / 8; }

// Pass p of the key's bits in equal shares of at most 8, the larger ones first.
inline SortDigit sort_digit(int key_bits, int p) {
  const int passes = sort_passes(key_bits);
  SortDigit d = {0, 0, 0u, 0};
  for (int q = 0; q <= p; q++) {
    d.shift += d.bits;
    d.bits = (key_bits - d.shift + passes - q - 1) / (passes - q);
  }
  d.mask = (1u << d.bits) - 1u;
  d.ballots = d.bits < 4 ? 4 : d.bits;
  return d;
}
