// Which kernel replays a prompt: the block kernel (tensor cores, one CTA per SM) or the CUDA-core kernels. Plain C++.
#pragma once

namespace he {

// Smallest max_budget of the block kernel. It has one CTA per SM and pays a block's settling (5200 to 11 000 cycles, with 8-bit codes
// up to 130 000) whatever the budget; the CUDA-core kernels scan every slot at every step, several units per SM. us with CUDA cores / block kernel:
//   up to one unit per SM the block kernel is ahead from the smallest budgets where the register kernel exists (64 slots, G = 4,
//   b = 32, N = 2 C: 38 / 31) and from 128 slots where it does not (G = 8, b = 64: 66 / 53); codes of 8 bits are not split off there, though on
//   some keys the register kernel is ahead (N = 2 C, block kernel on independent, drifting, clustered keys): G = 1, 4 units 64 slots 35 / 32, 37,
//   47, 128 slots 50 / 41, 45, 70, 384 slots 115 / 68, 89, 181, 128 units 128 slots clustered 78 / 75, 384 slots 169 / 222; G = 4, 4 units 64 slots
//   38 / 41, 44, 45, 200 slots 76 / 86, 96, 120, 384 slots 129 / 128, 145, 213, 32 and 128 units behind on clustered keys alone;
//   with more units they cross between 256 and 512 slots, sooner or later with the keys (320 units, b = 32, G = 4, N = 2.5 C: 411 / 418
//   at 512 slots on clustered keys, 410 / 316 on drifting ones), sooner with two words and G = 4 (N = 3 C: 250 / 253 at 160 slots,
//   336 / 302 at 224).
// Codes of few bits have few distinct distances, so that steps keep meeting in the same slots and a block needs more passes, most on
// clustered keys and least on independent ones. The lines lie where the product of the three ratios (clustered, drifting, independent
// keys) turns; 320 units, N = 2.5 C, CUDA cores / block kernel on the three kinds:
//   b = 8, G = 1    2556 slots 2580 / 5919, 3213, 1689    4096 slots 4460 / 9881, 5382, 2873: still ahead there, and not measured beyond
//   b = 8, G = 4    2556 slots 3800 / 7354, 5350, 5655    4096 slots 7360 / 12 369, 8725, 9278
//   b = 8, G = 2    2556 slots 9036 / 10 701, 8648, 9447  3072 slots 12 630 / 12 810, 10 539, 11 364
//   b = 5, G = 3    2556 slots 9135 / 13 215, 10 217, 7644  3072 slots 12 764 / 16 320, 12 292, 9276
//   b = 12, G = 1   1024 slots 632 / 1279, 656, 544       1536 slots 1280 / 2545, 957, 677
//   b = 16, G = 1   768 slots 523 / 742, 448, 407         1024 slots 632 / 976, 571, 524       1536 slots 1281 / 1849, 731, 614
// (a thread of the register kernel holds four slots up to 1024 and eight beyond, which doubles its time there).
// The block kernel's time goes with the rounds of units on the SMs, the others' less so: up to two units per SM codes of 13 to 16
// distances are ahead from the smaller tables on (1024 slots, b = 16, G = 1: 160 units 503 / 682, 368, 339, 296 units 550 / 830, 436, 395,
// 448 units 771 / 1208, 738, 682, 592 units 823 / 1530, 831, 763; 512 slots: 160 units 284 / 357, 215, 195, 592 units 486 / 826, 492, 443),
// those of 12 are level (160 units 503 / 863, 432, 351, 296 units 551 / 1045, 497, 413) and stay with the line.
inline int block_replay_min_budget(int words, int group_size, int hash_bits, long long units, int sms) {
  const bool has_reg = group_size == 1 || group_size == 4;  // group sizes with a register kernel
  const int distances = group_size * hash_bits;
  if (units <= sms) return has_reg ? 1 : 128;
  if (hash_bits <= 8 && distances <= 32) return has_reg ? 4096 : 2560;
  if (distances <= 16 && (distances <= 12 || units > 2LL * sms)) return 1025;
  return words == 2 && group_size == 4 ? 256 : 384;
}

}  // namespace he
