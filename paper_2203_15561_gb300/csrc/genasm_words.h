// Which words of a packed sequence a window's bases lie in. Plain C++, for the
// kernels and for the host test of its bounds.
#pragma once

#include <cstdint>

namespace ga {

// The bases from `pos` on of a sequence of `len` bases, `most` of them at most,
// begin at bit `o` of an aligned 32-bit word (o < 32): the first bit past the
// last of them (`o` itself if there are none).
constexpr uint32_t bases_end(uint32_t o, uint32_t len, uint32_t pos, uint32_t most) {
  const uint32_t left = len > pos ? len - pos : 0u;
  return o + 2u * (left < most ? left : most);
}

// Whether word k on from there holds one of them. (Not even word 0 does where the
// sequence ends before `pos`: what an empty sequence's offset points at need not
// be memory.)
constexpr bool holds_base(uint32_t k, uint32_t o, uint32_t end) { return (k ? 32u * k : o) < end; }

}  // namespace ga
