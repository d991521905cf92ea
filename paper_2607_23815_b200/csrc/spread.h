// How the blocks of an append, a warp per token, are laid over the SMs (plain C++: the rules are tested without a GPU).
#pragma once

#include <stdint.h>

namespace kvattn {

// Tokens of a block of the prologue that builds the plan beside the append: one block takes the plan, the others share the tokens,
// up to 32 (the block's warps) each.
inline int prologue_tokens(int total_new, int sms) {
  const int64_t others = sms > 1 ? sms - 1 : 1, n = ((int64_t)total_new + others - 1) / others;
  return n < 32 ? (int)n : 32;
}

}  // namespace kvattn
