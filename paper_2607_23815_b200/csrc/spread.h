// How the blocks of an append, a warp per token, are laid over the SMs (plain C++: the rules are tested without a GPU).
#pragma once

#include <stdint.h>

#include <atomic>

namespace kvattn {

// Whether what `set` does once per device is done; where it is not, callers go the way that does without.
template <int N, typename Set>
bool once_per_device(std::atomic<bool> (&done)[N], int device, Set set) {
  if (device < 0 || device >= N) return false;
  if (done[device].load(std::memory_order_acquire)) return true;
  if (!set()) return false;
  done[device].store(true, std::memory_order_release);
  return true;
}

// Dynamic shared memory of a block that lets `n` of them onto an SM and no more (228 KB, of which every block takes one more).
constexpr int spread_smem(int n) { return 228 * 1024 / (n + 1) / 128 * 128; }

struct AppendSpread {
  int blocks, warps;  // blocks == 0: the tokens are not spread
  int smem;           // of a block of kv_append
  int smem_front;     // of a block in front of the attention kernel of the same call
};

// An append's blocks of at most eight warps, a token each.  They are launched early and wait for the kernel in front, and the SMs that
// one leaves free, or frees first, would take all of them, as many as fit: the rows of a hundred tokens then go through three or four
// SMs.  So up to 24 tokens per SM a block asks for so much shared memory, which it does not use, that one, two or three of them are
// on an SM, and has no more warps than it takes to hold an SM's share of the tokens in that many.  (Eight warps in each of two or
// three blocks would hold 16 tokens on half of the SMs where every SM's share is 9.)  Whole calls, us (32/8 heads of 128 where not
// stated): 1 sequence of 37 tokens appended and extended 16.0 -> 14.4; 4 layers of 9 sequences, 500 tokens each, 171 -> 159 (165 with
// 40 KB a block, which lets five of them onto an SM); 2 extends beside 23 decodes 34.1 -> 26.7; 39 beside 49, 8/8 heads, 54.0 -> 43.5.
// An append and a decode of 9 sequences, not spread / eight warps / as many as it takes: 1184 tokens (one block of eight per SM) 13.2 /
// 11.1, 1185 13.2 / 11.8 / 11.3, 1260 13.2 / 11.8 / 11.4, 1500 13.2 / 11.8 / 11.5, 2000 13.6 / 12.2 / 12.0, 2369 13.8 / 13.0 / 12.7, 2800
// 13.9 / 13.3 / 13.1, 3552 14.6 / 14.0.  The same tokens through bulk copies into shared memory, a block's warps storing them from
// there, were slower (the first four calls: 15.1, 161, 28.6, 49.3).
//
// Waiting blocks with an SM to themselves keep other streams' blocks off it.  So a second such call has to find room beside the first:
// where one block per SM would fill more than half of the device, two are let onto one.  Rows of 4 KB of K and V and more, of more than
// a token per SM, keep their SMs in kv_append (held): one stream gains more by it than two lose.  Us for a call, one block per SM /
// two, not spread in brackets: 1000 tokens and a decode of 9 sequences behind them 11.0 / 11.6 (13.1); 39 extends beside 49 decodes,
// 8/8 heads, 44.0 / 47.7 (54.1); two streams of 148 tokens in three sequences 5.18 / 3.95 (4.14), of 592 4.69 / 4.30 (4.64), of 1184
// 5.73 / 5.16 (5.34).  In front of attention the gain is smaller and a CTA of the other stream wants a whole SM, so there only those
// rows ask for shared memory at all, and two blocks share an SM: 7 sequences of 32 tokens 16.4 either way, on two streams 28.9 /
// 25.2 (25.1); 9 of 58 27.9 either way, without shared memory 30.2 (31.2).
// Rows of less than 2 KB: no second block per SM.  22 sequences of 64 tokens, 16/2 heads, appended and extended 32.1 with two,
// 25.6 as not spread (27.7); 148 decode tokens of one head on two streams 10.3 with one per SM, 6.7 with two (7.7).
// Rows of more than 4 KB: no third block (append_kernel<8> has registers for two): 32 heads, 3552 tokens and a decode, 39.3 with the
// third, 38.9 without (38.9).
inline AppendSpread append_spread(int total_new, int chunks, int sms) {
  const bool held = chunks >= 128 && total_new > sms;  // (chunks: 16-byte pieces of a token's K, as many of its V)
  const int64_t per_sm = ((int64_t)total_new + sms - 1) / sms, k = (per_sm + 7) / 8;  // tokens and blocks of an SM
  if (k > (chunks < 64 ? 1 : chunks <= 128 ? 3 : 2)) return {0, 0, 0, 0};
  const int64_t warps = (per_sm + k - 1) / k, blocks = (total_new + warps - 1) / warps;
  const int shared = spread_smem(k == 1 && 2 * blocks > sms ? 2 : (int)k);
  return {(int)blocks, (int)warps, held ? spread_smem((int)k) : shared, held ? shared : 0};
}

// Tokens of a block of the prologue that builds the plan beside the append: one block takes the plan, the others share the tokens,
// up to 32 (the block's warps) each.
inline int prologue_tokens(int total_new, int sms) {
  const int64_t others = sms > 1 ? sms - 1 : 1, n = ((int64_t)total_new + others - 1) / others;
  return n < 32 ? (int)n : 32;
}

}  // namespace kvattn
