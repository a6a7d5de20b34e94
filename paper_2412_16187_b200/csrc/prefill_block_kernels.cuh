// he_prefill_compress, phase 2: the sequential replay of Algorithm 1 over the prompt ("Prompt Encoding Stage" of Section
// 3), a block of up to 128 evicting steps at a time.
//
// Distances as a contraction. With codes read as +-1 vectors s, the group distance of slot j at step t is
//   D(j, t) = sum_g popc(h_j xor h(q_{t,g})) = (G K - <s_j, u_t>) / 2,   u_t = sum_g s(q_{t,g})  (entries in -G..G),
// so the distances of a block of steps to every slot are one [steps x K] * [K x slots] product of small integers. The
// operands are 8-bit (e5m2 holds 2^n u for |u| <= 8, e4m3 every whole number up to 16), accumulation is fp32 over whole
// numbers below 2^24, so the result is exact in any order. For even G the parity of D is the same for every slot of a
// step, so the RANK D >> 1 orders the slots (D itself for odd G). Operands A = -alpha u, B = +-2 with 2 alpha = 32 (even G) or 64
// (odd G) and five more columns (a constant and the parity of the step, two digits of the index, 2^23) make the accumulator
// 2^23 + 128 * rank + 128 - slot in tile: the largest of a 128-slot tile is the arg-max key of Eq. 6 over the tile (largest
// distance, lowest slot on ties). Slots past the budget and protected first tokens have zeros in B and come to 2^23 alone, below
// everything else. At 2^23 the last mantissa bit is worth one, so an accumulator's low 16 bits ARE that key (rank <= 448: below
// 2^16), and the readers take them from tensor memory two to a register (tcgen05.ld.pack::16b) and compare two at a time: 36
// instructions a tile and thread for 68 on the fp32 values, and half the registers.
//
// What is sequential, and how it is settled side by side. Step r's victim depends on the victims s[0..r-1] of the block:
// a base slot (the table as the block found it) may be taken already, and the keys of earlier steps are candidates
// themselves. Written as s[r] = F_r(s[0..r-1]), any vector s with s = F(s) is the sequential result (by induction on r),
// so the block iterates s <- F(s), all steps at once, from s[r] = best base slot, until nothing changes. After k passes
// at least the first k entries are final; on the workloads' keys 2 to 4 passes settle a block, because few steps
// depend on one another. A step is EASY when its best base slot is not taken by an earlier step and no earlier key can
// reach its rank; easy steps cost nothing. The others ("hard", 5-40 %) are evaluated by a warp each: best new
// entry still resident, best base slot (a taken one makes its tile be scanned again with popcounts).
//
// Where passes do not converge quickly, the window that is evaluated at a time shrinks to a dozen steps. Where they do not converge
// at all (queries that keep preferring the same slots, near-constant ones, say, let a pass settle one step and make every evaluation
// scan tile after tile), the block is finished by a walk: one step after the other, all settling warps scanning the table for each
// (rb_walk). us per call with passes alone / with the walk, and what one warp resolving step by step took before the passes: constant
// queries, 32 units of 2048 slots, 2048 steps, 8110 / 890 (1980); 512 units of 2304, two words, 43 700 / 6830 (13 600); 8 of 9830,
// 4070 steps, 20 000 / 4330 (10 500); 128 of 192, 960 steps, 1860 / 460 (380 on CUDA cores); queries with a tenth of their
// variation, the first two 7310 / 1150 (1920) and 11 900 / 7250 (6780). Independent queries, where the test for it costs 0 to 1.4 %,
// take 150 (420), 1210 (2310), 260 (1320) and 214 (380).
//
// Few units: a cluster of up to 8 CTAs shares one unit. Tiles are dealt round-robin over its CTAs; each CTA keeps the
// whole packed code table (at most 48 KB at 32 bits), copies its tiles' maxima to the others through distributed shared
// memory, and all of them settle the block redundantly: one exchange per block.
//
// One CTA per SM, 18 warps of at most 96 registers:
//   warps 0-11   tile phase: groups of four read accumulators from tensor memory, one step per thread, a group a tile: three groups, or two
//                for two-word codes, whose warps 8-11 expand with the next four
//   warps 12-15  tile phase: expand packed codes into +-2 operand tiles (K-major, 128-byte swizzle), teams of two warps a tile, two slots
//                per thread; then they prepare the next block beside everything else: its operand A and the distances between its own
//                keys and queries, none of which depend on this block's outcome
//   warps 16-17  issue tcgen05.mma (M = 128 steps, N = 128 slots, K = 32) for the even and the odd tiles. The loop is warp-uniform, its counters
//                come out of a reduction so that they sit in uniform registers, and one elected lane issues
//   afterwards   warps 0-11 settle the block's steps
// A tile's tensor time is 64 cycles a K step (128 with one word, 192 with two), its read 64 and its maxima 72; what a tile costs instead is the
// latency of the hand-overs around them: 100 cycles for a wait on a completed mbarrier and 170 from an arrival to the waiter, 260 from
// the last MMA to its commit. So every tile has an accumulator of its own (pairs of tiles, with two groups and two accumulator pairs, took
// 630 cycles a pair), a freed accumulator and a written operand tile meet the issuing warp in ONE named barrier (45 cycles; two mbarriers
// 120), and no warp handles more than every second tile. A tile now takes 235 cycles with one word at 9830 slots. In a program of the tile
// phase alone: three groups 201, two 246, one 393 (in this kernel a single issuing warp is the bound, at 290 to 430 cycles a tile); two words
// 271 with three groups and 285 with two; with mbarriers instead 235 to 290. Here two words take two groups, so that eight warps expand:
// replay of 512 units of 512 to 4096 slots 835 -> 810 us (840 with three groups and four expanding warps); of 256 units of 9830 slots, one word, 5630 ->
// 4800 us (5400 with two groups).
// Every wait on an mbarrier is bounded; a CTA that gives up raises a flag that turns its later waits into no-ops, but it
// still walks the same blocks and cluster barriers as its peers (their copies into its shared memory must find it), then
// releases tensor memory and raises the device error counter. The tiles' named barriers count arrivals and have no limit of their
// own, and what keeps the arrivals of one tile apart from those of four tiles on are the mbarriers: once roles run on without them a
// barrier's phases may pass without its issuing warp, which would then wait for arrivals that nobody owes. So a warp that is not needed
// elsewhere sees the issuing warps out of every turn, and arrives for them where the flag is up (rb_see_out).
#pragma once
#include <cuda_fp16.h>

#include "hash_tc_kernels.cuh"
#include "prefill_kernels.cuh"

namespace he {

constexpr int kRbResWarps = 12;          // warps that settle a block
constexpr int kRbResThreads = 32 * kRbResWarps;
constexpr int kRbAuxWarp = kRbResWarps;  // the four warps that prepare the next block
constexpr int kRbAuxThreads = 128;
constexpr int kRbMmaWarp = 16;           // the two warps that issue products
constexpr int kRbThreads = 32 * (kRbMmaWarp + 2);
// Groups of four warps that read accumulators; the warps from there to kRbMmaWarp expand.
__host__ __device__ constexpr int rb_read_groups(int words) { return words == 2 ? 2 : 3; }
constexpr int kRbAccs = 4;               // accumulators, and tiles of operand B in shared memory
constexpr int kRbDoneBars = 2 * kRbAccs; // mbarriers that say a product is complete
constexpr int kRbTileBar = 8;            // named barriers kRbTileBar .. + 3: one for each accumulator
constexpr int kRbRows = 128;             // steps per block at most = MMA M
constexpr int kRbTile = 128;             // slots per tile = MMA N
constexpr int kRbKeyShift = 14;
constexpr int kRbIdxMask = (1 << kRbKeyShift) - 1;
constexpr int kRbMaxSlots = 12288;
constexpr int kRbMaxCluster = 8;
constexpr int kRbWidePasses = 6;         // passes over the whole block before the window shrinks
// The walk through a block takes over from the passes where hardly a step of the window is easy and as many passes at this one's cost
// would have cost twice the walk through the steps that are final: at the second pass where more than half of the block is left,
// later where less is (a few steps are soon settled by passes, and one slow pass is often chance). On independent queries 5 to 90 %
// of the steps are hard, most with few distinct distances, and passes win: with three quarters as the line, 4792 slots at b = 8 took
// 6190 us for 4960. On repeating queries 97 % are. Cycles, fitted to 8 units of 192 to 6144 slots: a pass (an evaluation scans a tile
// or two), and a step of the walk with `slots` slots for each thread (group sizes without a form of their own scan all eight places
// of a group).
__device__ __forceinline__ int rb_pass_cost(int hard) { return 1000 + (hard + kRbResWarps - 1) / kRbResWarps * 1400; }
__host__ __device__ constexpr int rb_walk_cost(int words, int gt, bool prot, int slots) {
  return (prot ? 550 : 400) + slots * ((gt == 4 ? 55 : (gt == 1 ? 35 : 215)) * words + (prot ? 20 : 0));
}
constexpr int kRbAtom = 128 * 128;       // 128 operand rows x one 128-byte swizzle atom
constexpr int kRbDnPitch = 136;          // 16-bit entries between rows of the new-entry table
constexpr int kRbDnPitchHalf = 68;       // ... when blocks have at most 64 steps
constexpr int kRbStaticSmem = 512;       // bytes kept back for the kernel's static arrays
// Eras of the owner table of words: the passes of a unit go from the first one down, 256 apart, and start again at a block that finds
// the last one behind it (a block uses a hundred or two, so none reaches the walk's mark of zero). The bounds-checking build starts over
// every few blocks, so that its tests pass there.
#ifdef HE_BOUNDS_CHECK
constexpr uint32_t kRbFirstEra = 0x22800u;
#else
constexpr uint32_t kRbFirstEra = 0xFFFFFE00u;
#endif
constexpr uint32_t kRbLastEra = 0x20000u;

// Byte offsets of the kernel's dynamic shared memory (after rounding its base up to 1024 bytes). Tile maxima: per CTA of the
// cluster one block of keys, a row for each step, an odd number of words apart (a warp stores a column, a lane per
// step), then the best key of each step over each reader group's tiles.
struct RbLayout {
  uint32_t a, bidx, b, codes, own, mx, mx_pitch, mx_block, top_at, dn, dn_buf, rn, nr, sv, sn, list, par, qraw, kraw, rec, total;
};
__host__ __device__ inline RbLayout rb_layout(int words, int slots, int G, int ncta, int abuf, int rows_max, bool wide) {
  RbLayout L;
  const uint32_t nt = (uint32_t)slots / kRbTile, ntl = (nt + ncta - 1) / ncta;
  uint32_t o = 0;
  auto take = [&](uint32_t bytes) {
    const uint32_t at = o;
    o += (bytes + 15u) & ~15u;
    return at;
  };
  // a 128-byte atom row holds two tiles' 64-bit rows or four tiles' 32-bit rows, and both buffers of a 32-bit operand A
  L.a = take(words == 2 ? (uint32_t)abuf * kRbAtom : kRbAtom);
  L.bidx = take(kRbAtom);  // index columns: four variants side by side
  L.b = take((uint32_t)kRbAccs / (words == 2 ? 2 : 4) * kRbAtom);
  L.codes = take((uint32_t)slots * words * 4u);
  L.own = take((uint32_t)slots * (wide ? 4u : 1u));
  L.mx_pitch = ntl | 1u;  // words
  // (one more row takes the threads without a step; whole 16-byte units, as the copies between CTAs want)
  L.top_at = (L.mx_pitch * (rows_max < kRbRows ? rows_max + 1 : rows_max) + 3u) & ~3u;
  L.mx_block = L.top_at + (uint32_t)rb_read_groups(words) * rows_max;
  L.mx = take(L.mx_block * ncta * 4u);
  L.dn_buf = rows_max == kRbRows ? kRbRows / 2 * kRbDnPitch : rows_max * kRbDnPitchHalf;  // entries
  L.dn = take(2u * L.dn_buf * 2u);
  L.rn = take(kRbRows * 4u);
  L.nr = take(2u * kRbRows * 4u);
  L.sv = take(kRbRows * 2u);
  L.sn = take(kRbRows * 4u);
  L.list = take(kRbRows);
  L.par = take(2u * kRbRows * 4u);
  L.qraw = take(2u * kRbRows * G * words * 4u);  // this block's codes and the next block's
  L.kraw = take(2u * kRbRows * words * 4u);
  L.rec = take(kRbRows * 4u);
  L.total = o + 1024u;
  return L;
}

struct RbArgs {
  ReplayArgs r;
  int ncta;       // CTAs per unit (cluster size, a power of two)
  int scheduled;  // units are claimed from r.sched; 0: unit = cluster index
  int abuf;       // operand A buffers (2: the next block's is built during the tile phase)
  int rows_max;   // steps per block at most: 128, or 64 (kRbHalf)
  RbLayout L;     // computed by the host: kernel parameters cost no registers
};

// Steps per block. A block of R steps against C slots meets about R / (2 C) taken slots per step, and the passes it needs
// grow with them, so smaller tables use shorter blocks (1024 slots, b = 16: 42 000 cycles to settle 128 steps at once,
// 2 x 14 000 in two blocks). Codes with few distinct distances (distances = G b of them) take the same slots more often:
// 32 steps instead of 64 at 192 slots, 128 units, N = 6 C: 554 -> 440 us with 8 distances, 172 -> 184 with 128.
__host__ __device__ inline int rb_block_rows(int C, int distances) { return C >= 1536 ? 128 : (C >= (distances <= 16 ? 256 : 144) ? 64 : 32); }

__device__ __forceinline__ void rb_mma_f8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}

// e4m3 bit pattern of a small non-negative integer with at most four significant bits (exact), e5m2 of an integer with at
// most three (e5m2 is the high half of f16).
__device__ __forceinline__ uint32_t rb_e4m3(int v) {
  if (v <= 0) return 0u;
  const int p = 31 - __clz(v);
  const uint32_t mant = p >= 3 ? ((uint32_t)v >> (p - 3)) & 7u : ((uint32_t)v << (3 - p)) & 7u;
  return ((uint32_t)(p + 7) << 3) | mant;
}
__device__ __forceinline__ uint32_t rb_e5m2(int v) { return (uint32_t)__half_as_ushort(__int2half_rn(v)) >> 8; }

// Byte offset of 16-byte chunk `chunk` (0..7) of row `row` inside one swizzle atom.
__device__ __forceinline__ uint32_t rb_swz(int row, int chunk) {
  return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((chunk ^ (row & 7)) << 4));
}

// The low halves of 64 accumulator columns, two to a register.
__device__ __forceinline__ void rb_ld64_low(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}

// tcgen05.wait::ld that the loaded registers pass through, so that nothing uses them ahead of it.
__device__ __forceinline__ void rb_wait_ld(uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]),
        "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]),
        "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), "+r"(v[24]),
        "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
      :
      : "memory");
}
// Pairwise maximum of 64 registers: a tree of three-input maxima, four levels deep.
__device__ __forceinline__ uint32_t rb_max64(const uint32_t (&a)[32], const uint32_t (&b)[32]) {
  uint32_t t[21], u[7];
#pragma unroll
  for (int k = 0; k < 10; ++k) {
    t[k] = __vimax3_u16x2(a[3 * k], a[3 * k + 1], a[3 * k + 2]);
    t[10 + k] = __vimax3_u16x2(b[3 * k], b[3 * k + 1], b[3 * k + 2]);
  }
  t[20] = __vimax3_u16x2(a[30], a[31], b[30]);
#pragma unroll
  for (int k = 0; k < 7; ++k) u[k] = __vimax3_u16x2(t[3 * k], t[3 * k + 1], t[3 * k + 2]);
  return __vimax3_u16x2(__vimax3_u16x2(u[0], u[1], u[2]), __vimax3_u16x2(u[3], u[4], u[5]), __vmaxu2(u[6], b[31]));
}

// Columns of a code word in operand order: output word m (four bytes) holds bits m, m + 8, m + 16, m + 24, in both
// operands, so that one shift and one logic operation expand four bits. Set: +2 (e4m3 0x40), clear: -2 (0xC0).
__device__ __forceinline__ uint32_t rb_expand4(uint32_t h, int m) { return lop3<0x6A>(h << (7 - m), 0x80808080u, 0xC0C0C0C0u); }

// The ranks of a block's own keys at its steps: step r only needs those of the r steps before it, so steps 64 + k and 63 - k
// share a row (64 + k entries from its start, 63 - k from the next multiple of four). Blocks of 64 have a row each.
__device__ __forceinline__ int rb_dn_at(int r, int rows_max) {
  if (rows_max < kRbRows) return r * kRbDnPitchHalf;
  return r >= 64 ? (r - 64) * kRbDnPitch : (63 - r) * kRbDnPitch + ((127 - r + 3) & ~3);
}

__device__ __forceinline__ uint32_t rb_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t rb_mapa(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void rb_st_remote(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Copy to a peer's shared memory that counts its bytes on the peer's mbarrier. (Stores by the reading warps, fenced by a
// releasing arrive, took about 2000 cycles a block with four CTAs; asynchronous 4-byte stores 10 000 with eight.)
__device__ __forceinline__ void rb_copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void rb_arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// mbar_wait_warp with its loop left rolled: unrolled by the compiler, each of this kernel's waits was 5 KB of code, half of the kernel's 143 KB
// (128 units of 1024 slots, b = 16, windows, the kernel otherwise as it was: 1290 -> 1230 us).
__device__ __forceinline__ bool rb_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (__builtin_expect(__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)), 1)) return true;
  bool ok = false, on = true;
#pragma unroll 1
  for (uint32_t i = 0; i < kTcSpinLimit && on; ++i) {
    ok = mbar_try_wait(bar, parity);
    on = !ok && *abort_flag == 0;
  }
  if (!ok) *abort_flag = 1;
  return __all_sync(0xFFFFFFFFu, ok);
}
// Bounded wait for copies and arrivals of other CTAs of the cluster.
__device__ __forceinline__ bool rb_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
#pragma unroll 1
  for (uint32_t i = 0; i < kTcSpinLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (*abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void rb_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int ID, int THREADS>
__device__ __forceinline__ void rb_bar() {
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}
// An accumulator's named barrier (`acc` 0 .. 3): four warps that have read it, two that have written the operand tile of the same number,
// and the issuing warp, which waits.
constexpr int kRbTileBarThreads = 128 + 64 + 32;
__device__ __forceinline__ void rb_tile_arrive(int acc) { asm volatile("bar.arrive %0, %1;" ::"r"(kRbTileBar + acc), "n"(kRbTileBarThreads) : "memory"); }
__device__ __forceinline__ void rb_tile_sync(int acc) { asm volatile("bar.sync %0, %1;" ::"r"(kRbTileBar + acc), "n"(kRbTileBarThreads) : "memory"); }

// Until both issuing warps have come through the turn (`turns`: the last one of each): once the abort flag is up nobody else waits at the tiles'
// barriers, and an arrival at each lets an issuing warp on after seven rounds at the latest. The limit is several times that of the
// waits after which other roles raise the flag (seconds); what is still out there then is given up on as a wait is.
__device__ __noinline__ void rb_see_out(volatile int* turns, int turn, volatile int* abort_flag) {
#pragma unroll 1
  for (uint32_t i = 0; i < 8u * kTcSpinLimit && __any_sync(0xFFFFFFFFu, turns[0] < turn || turns[1] < turn); ++i) {
    if (i == 7u * kTcSpinLimit) *abort_flag = 1;
    if (__any_sync(0xFFFFFFFFu, *abort_flag != 0)) {
#pragma unroll 1
      for (int x = 0; x < kRbAccs; ++x) rb_tile_arrive(x);
    } else {
      __nanosleep(100);
    }
    __syncwarp();
  }
}

// The loops of the tile phase, and the preparation of the next block. Functions of their own, so that their registers and their code
// don't change with what the settling around them needs: inlined, a change of the settling moved a tile by 4 % either way. Replay when they became
// functions, us inlined / as functions: 256 units of 9830 slots 4970 / 4600, 512 of 512 to 4096, two words, 810 / 763, 128 of 1024 with windows
// 1228 / 1182, 8 of 9830 1155 / 1140. (Today 4600, 761, 1138 and 1115: the first with an owner table of words; where code falls still moves it by 1 to 2 %.) (The evaluation of a hard step as a function: 1182 -> 1328, its caller's registers go to the stack.)
// `bars`: the products' mbarriers (product n's is n mod 8, its phase n / 8).
__device__ __forceinline__ uint32_t rb_done_bar(uint32_t bars, int n) { return bars + 8u * (uint32_t)(n & (kRbDoneBars - 1)); }
__device__ __forceinline__ uint32_t rb_done_phase(int n) { return (uint32_t)(n >> 3) & 1u; }

// One group's tiles i = grp, grp + GROUPS, ...: the best key of each into mrow[i]. taddr: this warp's lanes of the first accumulator; ct: 127 - tile of
// the unit goes above the index within the tile (lower tiles first), cstep less from tile to tile. Returns the best of all.
template <int GROUPS>
__device__ __noinline__ int rb_read_tiles(uint32_t bars, volatile int* abort_flag, int it, int grp, int ntl, uint32_t taddr, uint32_t mrow, int ct, int cstep) {
  int top = -1;
#pragma unroll 1
  for (int i = grp; i < ntl; i += GROUPS) {
    const int n = it + i, acc = n & 3;
    rb_wait(rb_done_bar(bars, n), rb_done_phase(n), abort_flag);
    tc_fence_after();
    uint32_t v0[32], v1[32];
    rb_ld64_low(taddr + (uint32_t)(acc * kRbTile), v0);
    rb_ld64_low(taddr + (uint32_t)(acc * kRbTile) + 64, v1);
    rb_wait_ld(v0);
    rb_wait_ld(v1);
    tc_fence_before();  // the accumulator goes back
    rb_tile_arrive(acc);
    const uint32_t m = rb_max64(v0, v1);
    // the tile's best key, 2^14 rank + index; negative: no slot of the tile may win
    const int k16 = (int)max(m & 0xFFFFu, m >> 16) - 1, key = ((k16 & ~127) << 7) + (k16 & 127) + ct;
    ct -= cstep;
    top = max(top, key);
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(mrow + 4u * (uint32_t)i), "r"(key) : "memory");
  }
  return top;
}

__device__ __forceinline__ void rb_st_chunk(uint32_t at, uint32_t v0, uint32_t v1, uint32_t v2, uint32_t v3) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v0), "r"(v1), "r"(v2), "r"(v3) : "memory");
}
// A slot's or a key's code as a row of an operand tile whose first chunk is at `at` (a multiple of the row's chunks, so chunk c is at `at` xor c).
template <int WORDS>
__device__ __forceinline__ void rb_expand_row(const uint32_t (&h)[WORDS], uint32_t at) {
#pragma unroll
  for (int c = 0; c < 2 * WORDS; ++c) {
    const uint32_t hw = h[c >> 1];
    const int m = (c & 1) * 4;
    rb_st_chunk(at ^ (uint32_t)(c << 4), rb_expand4(hw, m), rb_expand4(hw, m + 1), rb_expand4(hw, m + 2), rb_expand4(hw, m + 3));
  }
}
template <int WORDS>
__device__ __forceinline__ void rb_clear_row(uint32_t at) {
#pragma unroll
  for (int c = 0; c < 2 * WORDS; ++c) rb_st_chunk(at ^ (uint32_t)(c << 4), 0u, 0u, 0u, 0u);
}

// One team's tiles i, i + TEAMS, ...: rows x and x + 64 (8 KB further on) of the tile by a thread. src: the thread's first code of the CTA's tile 0, step:
// bytes from tile to tile; at, at_next: where its row is in this tile and the next. Slots below S and from C on may not win and get zeros: j is the
// thread's first slot of tile 0, jstep slots from tile to tile.
template <int WORDS, int TEAMS>
__device__ __noinline__ void rb_expand_tiles(uint32_t bars, volatile int* abort_flag, int it, int i, int ntl, uint32_t src, uint32_t step, uint32_t at, uint32_t at_next, int j,
                                             int jstep, int S, int C) {
  uint32_t h0[WORDS], h1[WORDS];
  auto fetch = [&](int t) {
    const uint32_t from = src + step * (uint32_t)t;
    if (WORDS == 2) {
      asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(h0[0]), "=r"(h0[WORDS - 1]) : "r"(from));
      asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(h1[0]), "=r"(h1[WORDS - 1]) : "r"(from + 64u * 4u * WORDS));
    } else {
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(h0[0]) : "r"(from));
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(h1[0]) : "r"(from + 64u * 4u));
    }
  };
  if (i < ntl) fetch(i);
#pragma unroll 1
  for (; i < ntl; i += TEAMS) {
    const int n = it + i;
    rb_wait(rb_done_bar(bars, n - 4), rb_done_phase(n - 4), abort_flag);  // product n - 4 is done with the operand tile
    rb_expand_row<WORDS>(h0, at);
    rb_expand_row<WORDS>(h1, at + 8192u);
    const int j0 = j + jstep * i;
    if (__any_sync(0xFFFFFFFFu, j0 < S || j0 + 64 >= C)) {  // some slots of the tile may not win
      if (j0 < S || j0 >= C) rb_clear_row<WORDS>(at);
      if (j0 + 64 < S || j0 + 64 >= C) rb_clear_row<WORDS>(at + 8192u);
      __syncwarp();
    }
    fence_proxy_async();
    rb_tile_arrive(n & 3);
    if (i + TEAMS < ntl) fetch(i + TEAMS);
    const uint32_t t = at;
    at = at_next, at_next = t;
  }
}

// Rank of one slot's code at a step from the packed words. GT = 4 uses the bit-plane form, which yields (D - pc) / 2 with pc
// the bits set in the exclusive or of the step's query codes (`parity_bits`, worked out with operand A).
template <int WORDS, int GT>
struct RbRank {
  static constexpr int kQ = (GT > 0 ? GT : kMaxGroup) * WORDS;
  uint32_t q[kQ];
  Planes4 p[WORDS];
  int add, G;
  __device__ __forceinline__ void fetch(const uint32_t* src, int G_, int parity_bits) {
    G = G_;
    add = parity_bits;
    if (GT * WORDS % 4 == 0 && GT > 0) {
#pragma unroll
      for (int i = 0; i < kQ; i += 4) *reinterpret_cast<uint4*>(q + i) = *reinterpret_cast<const uint4*>(src + i);
    } else {
#pragma unroll
      for (int i = 0; i < kQ; ++i) q[i] = (GT > 0 || i < G * WORDS) ? src[i] : 0u;
    }
  }
  __device__ __forceinline__ void prepare() {
    if (GT == 4) {
#pragma unroll
      for (int w = 0; w < WORDS; ++w) {
        uint32_t parity;
        p[w] = make_planes4(q[w], q[WORDS + w], q[(2 * WORDS + w) % kQ], q[(3 * WORDS + w) % kQ], &parity);
      }
    }
  }
  __device__ __forceinline__ void load(const uint32_t* src, int G_, int parity_bits) {
    fetch(src, G_, parity_bits);
    prepare();
  }
  __device__ __forceinline__ int dist(const uint32_t (&h)[WORDS]) const {
    if (GT == 4) return 2 * half_distance4<WORDS>(h, p) + add;
    int d = 0;
#pragma unroll
    for (int g = 0; g < (GT > 0 ? GT : kMaxGroup); ++g)
      if (GT > 0 || g < G) {
#pragma unroll
        for (int w = 0; w < WORDS; ++w) d += __popc(h[w] ^ q[g * WORDS + w]);
      }
    return d;
  }
  __device__ __forceinline__ int rank(const uint32_t (&h)[WORDS]) const {
    if (GT == 4) return half_distance4<WORDS>(h, p) + (add >> 1);
    if (GT == 1) return dist(h);
    return (G & 1) ? dist(h) : dist(h) >> 1;
  }
};

// The walk through the steps fin .. rows - 1 of a block by the settling warps (file comment), every step on the table that the one
// before it left. Every thread scans its slots (tid, tid + 384, ...), and a slot is rewritten by the thread that scans it, so that a
// step needs one barrier: 400 cycles, and 35 (G = 1) or 55 (G = 4) more for each slot of a thread and word. The owner table (no claims
// before and after) marks the slots of recent tokens meanwhile. Steps from writes_end on leave the table as it is; pos is null where
// another CTA of the cluster writes the positions. Not inlined: inside the block loop it cost independent queries 2 % (64 ragged
// prompts), and itself gains 6 %.
extern __shared__ unsigned char rb_smem_raw[];
template <int WORDS, int GT, bool PROT>
__device__ __noinline__ void rb_walk(const RbLayout& L, bool wide, int base, int cur, int32_t* pos, int t0, int fin, int rows, int writes_end, int C, int G,
                                     int S, int Rn) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, GW = G * WORDS;
  unsigned char* smem = rb_smem_raw + base;  // (not passed as pointers, so that the accesses stay shared-memory accesses)
  uint32_t* codes = reinterpret_cast<uint32_t*>(smem + L.codes);
  auto recent = [&](int slot) { return wide ? reinterpret_cast<const uint32_t*>(smem + L.own)[slot] == 0u : smem[L.own + slot] == 0; };
  auto mark = [&](int slot, uint32_t v) {
    if (wide) reinterpret_cast<uint32_t*>(smem + L.own)[slot] = v;
    else smem[L.own + slot] = (uint8_t)v;
  };
  uint16_t* SV = reinterpret_cast<uint16_t*>(smem + L.sv);
  int32_t* SN = reinterpret_cast<int32_t*>(smem + L.sn);
  const int32_t* REC = reinterpret_cast<const int32_t*>(smem + L.rec);
  const int32_t* par = reinterpret_cast<const int32_t*>(smem + L.par) + cur * kRbRows;
  const uint32_t* qb = reinterpret_cast<const uint32_t*>(smem + L.qraw) + cur * kRbRows * GW;
  const uint32_t* kb = reinterpret_cast<const uint32_t*>(smem + L.kraw) + cur * kRbRows * WORDS;
  auto newest = [&](int r, int m) { return r >= m ? (int)SV[r - m] : REC[m - r - 1]; };  // slot of the m-th newest token at step r
  rb_bar<2, kRbResThreads>();
  if (PROT && Rn > 0) {
    if (tid < Rn) mark(newest(fin, tid + 1), 0u);
    rb_bar<2, kRbResThreads>();
  }
  const int mine = tid < C ? (C - tid + kRbResThreads - 1) / kRbResThreads : 0;  // slots of this thread
  RbRank<WORDS, GT> rk;
  rk.load(qb + fin * GW, G, par[fin]);
  int last = PROT && Rn == 1 ? newest(fin, 1) : 0;  // slot of the step before
#pragma unroll 1
  for (int r = fin; r < rows; ++r) {
    // what the rewrite and the next step want and this step's outcome does not decide
    RbRank<WORDS, GT> next;
    const int rn = min(r + 1, rows - 1);
    next.fetch(qb + rn * GW, G, par[rn]);
    uint32_t kc[WORDS];
#pragma unroll
    for (int w = 0; w < WORDS; ++w) kc[w] = kb[r * WORDS + w];
    const int out = PROT && Rn > 1 ? newest(r, Rn) : last;  // its token is recent no longer
    int best = -1, kx = kRbIdxMask - tid;
    const uint32_t* cp = codes + tid * WORDS;
    int slot = tid;
#pragma unroll 4
    for (int i = 0; i < mine; ++i) {
      uint32_t h[WORDS];
      if (WORDS == 2) {
        const uint2 h2 = *reinterpret_cast<const uint2*>(cp);
        h[0] = h2.x, h[WORDS - 1] = h2.y;
      } else {
        h[0] = *cp;
      }
      int key = (rk.rank(h) << kRbKeyShift) + kx;
      if (PROT) key = kx <= kRbIdxMask - S && !recent(slot) ? key : -1;
      best = max(best, key);
      cp += kRbResThreads * WORDS;
      slot += kRbResThreads;
      kx -= kRbResThreads;
    }
    int32_t* wbest = SN + (r & 1) * 16;
    const int wb = __reduce_max_sync(0xFFFFFFFFu, best);
    if (lane == 0) wbest[warp] = wb;
    rb_bar<2, kRbResThreads>();
    const int wtop = lane < kRbResWarps ? wbest[lane] : -1;
    rk = next;
    rk.prepare();
    const int top = __reduce_max_sync(0xFFFFFFFFu, wtop);
    last = min(kRbIdxMask - (top & kRbIdxMask), C - 1);
    if (tid == 0) SV[r] = (uint16_t)last;
    if (best == top && HE_IN_RANGE(last, C)) {  // (keys differ between slots)
      if (r < writes_end) {
#pragma unroll
        for (int w = 0; w < WORDS; ++w) codes[last * WORDS + w] = kc[w];
        if (pos != nullptr) pos[last] = t0 + r;
      }
      if (PROT && Rn > 0) mark(last, 0u);
    }
    if (PROT && Rn > 0 && out % kRbResThreads == tid) mark(out, ~0u);
  }
  rb_bar<2, kRbResThreads>();
  if (PROT && tid < Rn) mark(newest(rows, tid + 1), ~0u);
}

// First chunk of row x of operand tile sx, as an offset into operand B.
template <int WORDS>
__device__ __forceinline__ uint32_t rb_row_at(int x, int sx) {
  const int c0 = WORDS == 2 ? 4 * (sx & 1) : 2 * sx;
  return (uint32_t)((WORDS == 2 ? sx >> 1 : 0) * kRbAtom + (x >> 3) * 1024 + (x & 7) * 128 + ((c0 ^ (x & 7)) << 4));
}

// Scaling of the operands (file comment): data columns' sum + off - 64 parity (even G) = 128 * rank.
__device__ __forceinline__ int rb_alpha(int G) { return (G & 1) == 0 ? 16 : 32; }
template <int WORDS>
__device__ __forceinline__ int rb_off(int G) {
  return 2 * rb_alpha(G) * G * 32 * WORDS;
}

// An issuing warp's products of a turn, the even (odd = 0) or the odd ones: the block's tiles with operand A at `a`, then, if there is a next block,
// its own keys (product it + ntl, no index columns) with operand A at `a_next`. bidx, b: index columns and operand tiles. first, last: the
// tiles that take the index-column variants (-1: none). adone: mbarrier to tell when the tiles are multiplied (0: nobody asks).
template <int WORDS>
__device__ __noinline__ void rb_issue_tiles(uint32_t bars, int it_, int ntl_, int odd, uint32_t tmem_, uint32_t a_, uint32_t a_next_, uint32_t bidx_, uint32_t b_, int first,
                                            int last, uint32_t adone, bool next) {
  // (a reduction's result sits in a uniform register: the loop's counters and the descriptors then stay in those)
  auto uniform = [](uint32_t v) { return __reduce_max_sync(0xFFFFFFFFu, v); };
  const int it = (int)uniform((uint32_t)it_), ntl = (int)uniform((uint32_t)ntl_), first_i = (int)uniform((uint32_t)(first + 1)) - 1, last_i = (int)uniform((uint32_t)(last + 1)) - 1;
  const uint32_t tmem = uniform(tmem_);
  const uint64_t ad = umma_desc_k128(uniform(a_)), ad_next = umma_desc_k128(uniform(a_next_)), xd = umma_desc_k128(uniform(bidx_)), bd0 = umma_desc_k128(uniform(b_));
  // instruction descriptor: fp32 accumulate, e5m2 x e4m3, both operands K-major, N = 128, M = 128
  const uint32_t idesc = (1u << 4) | (1u << 7) | ((uint32_t)(kRbTile >> 3) << 17) | ((uint32_t)(kRbRows >> 4) << 24);
  auto issue = [&](int n, uint64_t a, bool index, uint64_t x) {
    const int acc = n & 3;
    const uint64_t bd = bd0 + (uint64_t)((WORDS == 2 ? (acc >> 1) * kRbAtom + (acc & 1) * 64 : acc * 32) >> 4);
    rb_tile_sync(acc);
    tc_fence_after();
    if (tc_elect()) {
      const uint32_t d = tmem + (uint32_t)(acc * kRbTile);
#pragma unroll
      for (int w = 0; w < WORDS; ++w) rb_mma_f8(d, a + (uint64_t)(2 * w), bd + (uint64_t)(2 * w), idesc, w > 0);
      if (index) rb_mma_f8(d, a + (uint64_t)(2 * WORDS), x, idesc, true);
      tc_commit(rb_done_bar(bars, n));
    }
    __syncwarp();
  };
#pragma unroll 1
  for (int i = (it ^ odd) & 1; i < ntl; i += 2) issue(it + i, ad, true, xd + (uint64_t)((i == first_i ? 2 : 0) + (i == last_i ? 4 : 0)));
  if (adone != 0u && tc_elect()) tc_commit(adone);
  __syncwarp();
  if (next && ((it + ntl) & 1) == odd) issue(it + ntl, ad_next, false, 0);
}

// Warps 12-15 prepare a block in buffer `buf`: operand A from the queries' codes, then the ranks of its own keys at its steps (product n).
template <int WORDS, int GT, bool PROT, int RM>
__device__ __noinline__ void rb_prepare(const RbLayout& L, int base, int buf, int nrows, int n, int G_, int Rn, int abuf, uint32_t bars, volatile int* abort_flag,
                                        uint32_t tmem_base) {
  const int tid = threadIdx.x, warp = tid >> 5, first = tid & (kRbAuxThreads - 1);
  const int G = GT > 0 ? GT : G_, GW = G * WORDS;
  unsigned char* smem = rb_smem_raw + base;
  const uint32_t* kraw = reinterpret_cast<const uint32_t*>(smem + L.kraw);
  int32_t* PAR = reinterpret_cast<int32_t*>(smem + L.par);
  int32_t* NR = reinterpret_cast<int32_t*>(smem + L.nr);
  uint16_t* Dn = reinterpret_cast<uint16_t*>(smem + L.dn);
  const bool even = (G & 1) == 0;
  const int alpha = rb_alpha(G), off = rb_off<WORDS>(G);
  // the e5m2 codes of -alpha (2 c - G) for c = 0..7 set bits among the group's queries, as two words of a byte table; c = 8 (G = 8 only) is
  // patched where it occurs
  uint32_t lut_lo = 0u, lut_hi = 0u;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    lut_lo |= rb_e5m2(-alpha * (2 * c - G)) << (8 * c);
    lut_hi |= (c + 4 <= G ? rb_e5m2(-alpha * (2 * (c + 4) - G)) : 0u) << (8 * c);
  }
  // operand A, row r = step r of the block: -alpha u_t, then the five further columns; one thread per (row, word)
  const uint32_t* qd = reinterpret_cast<const uint32_t*>(smem + L.qraw) + buf * kRbRows * GW;
  unsigned char* ad = smem + L.a + (WORDS == 2 && abuf > 1 ? buf * kRbAtom : 0);
  const int c0 = WORDS == 1 && abuf > 1 ? 4 * buf : 0;
#pragma unroll 1
  for (int item = first; item < kRbRows * WORDS; item += kRbAuxThreads) {
    const int r = item & (kRbRows - 1), w = item >> 7;
    const bool valid = r < nrows;
    uint32_t cnt[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) cnt[m] = 0u;
    if (valid)
      for (int g = 0; g < G; ++g) {
        const uint32_t x = qd[r * GW + g * WORDS + w];
#pragma unroll
        for (int m = 0; m < 8; ++m) cnt[m] += (x >> m) & 0x01010101u;  // set bits among the queries, one counter per byte
      }
    uint32_t v[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const uint32_t t = cnt[m] | (cnt[m] >> 4);
      v[m] = __byte_perm(lut_lo, lut_hi, __byte_perm(t, 0u, 0x4420));
      // eight of eight: -128 = 0xD8 (selector 8 made the lookup give 0 there)
      if (GT == 0) v[m] |= (cnt[m] & 0x08080808u) * 0x1Bu;
      if (!valid) v[m] = 0u;
    }
    *reinterpret_cast<uint4*>(ad + rb_swz(r, c0 + 2 * w)) = make_uint4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<uint4*>(ad + rb_swz(r, c0 + 2 * w + 1)) = make_uint4(v[4], v[5], v[6], v[7]);
    if (w == 0) {
      int pc = 0;
      if (even && valid) {
#pragma unroll
        for (int v2 = 0; v2 < WORDS; ++v2) {
          uint32_t x = 0u;
          for (int g = 0; g < G; ++g) x ^= qd[r * GW + g * WORDS + v2];
          pc += __popc(x);
        }
      }
      PAR[buf * kRbRows + r] = pc;
      *reinterpret_cast<uint4*>(ad + rb_swz(r, c0 + 2 * WORDS)) =
          valid ? make_uint4(0x4Cu | (0x3Cu << 8) | (0x78u << 16) | (rb_e5m2(off) << 24), (pc & 1) ? 0xD4u : 0u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(ad + rb_swz(r, c0 + 2 * WORDS + 1)) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  // The ranks: one more tile, without index columns. Also each step's largest rank of any key that enters before it (and is no longer recent):
  // no new entry can beat that.
  const int x = tid & 127, acc = n & 3;
  rb_wait(rb_done_bar(bars, n - 4), rb_done_phase(n - 4), abort_flag);
  uint32_t h[WORDS];
#pragma unroll
  for (int w = 0; w < WORDS; ++w) h[w] = kraw[(buf * kRbRows + x) * WORDS + w];
  rb_expand_row<WORDS>(h, smem_u32(smem + L.b) + rb_row_at<WORDS>(x, acc));
  fence_proxy_async();
  rb_bar<3, kRbAuxThreads>();
  if (warp < kRbAuxWarp + 2) rb_tile_arrive(acc);
  rb_wait(rb_done_bar(bars, n), rb_done_phase(n), abort_flag);
  tc_fence_after();
  // Conversions by an fp32 addition (the integer conversions run at a sixteenth of its rate): 2^22 + rank has 2 * rank
  // in its low bits, which is what is kept.
  const int r = x, last = PROT ? r - Rn : r;  // entries below `last` are candidates
  const float magic = (float)(off - ((PAR[buf * kRbRows + r] & 1) << 6)) * (1.f / 128.f) + 4194304.f;
  const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(acc * kRbTile);
  uint16_t* dst = Dn + buf * L.dn_buf + rb_dn_at(r, RM);
  float dmax = -1e9f;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    uint32_t v[32];
    tc_ld32(taddr + c * 32, v);
    tc_wait_ld();
    if (c == 3) {
      tc_fence_before();
      rb_tile_arrive(acc);
    }
    if (c > (warp & 3)) continue;  // no step of this warp comes after those keys
    const int lc = last - c * 32;
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (k < lc) dmax = fmaxf(dmax, __uint_as_float(v[k]));
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      uint32_t pk[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float y0 = fmaf(__uint_as_float(v[4 * k + 2 * e]), 1.f / 128.f, magic);
        const float y1 = fmaf(__uint_as_float(v[4 * k + 2 * e + 1]), 1.f / 128.f, magic);
        pk[e] = __byte_perm(__float_as_uint(y0), __float_as_uint(y1), 0x5410);
      }
      if (c * 32 + 4 * k < r && r < RM) *reinterpret_cast<uint2*>(dst + c * 32 + 4 * k) = make_uint2(pk[0], pk[1]);
    }
  }
  NR[buf * kRbRows + r] = last > 0 ? (int)(__float_as_uint(fmaf(dmax, 1.f / 128.f, magic)) & 0xFFFFu) >> 1 : -1;
}

// PROT: protected windows (Section 4 setup). The first n_sink tokens never leave slots 0 .. n_sink-1, so those slots are
// masked like slots past the budget. A recent token that is already in the table is recognised by the list of the newest
// slots, one of this block's own keys by its step. Needs every budget > n_sink + n_recent (so that some slot is always
// eligible), n_sink <= 128 (one tile) and n_recent < 128.
// FORM: kRbHalf has blocks of at most 64 steps, where the largest two-word tables leave no room for the tables of more; kRbWide an
// owner table of a word per slot instead of a byte (claims below).
enum : int { kRbFull = 0, kRbHalf = 1, kRbWide = 2 };
template <int WORDS, int GT, bool PROT, int FORM>
__global__ void __launch_bounds__(kRbThreads, 1) prefill_replay_block_kernel(const __grid_constant__ RbArgs ar) {
  constexpr int NT = kRbThreads;
  constexpr int kGroups = rb_read_groups(WORDS), kExpWarp = 4 * kGroups, kTeams = (kRbMmaWarp - kExpWarp) / 2;
  constexpr bool HALF = FORM == kRbHalf, wide = FORM == kRbWide;
  constexpr int RM = HALF ? kRbRows / 2 : kRbRows;
  __shared__ __align__(8) unsigned long long bars[kRbDoneBars + 5];
  __shared__ uint32_t tmem_base_s;
  __shared__ volatile int abort_flag;
  __shared__ volatile int s_turns[2];            // the issuing warps' last turns
  __shared__ int s_unit[2];
  __shared__ int s_change[2];                    // by pass parity: first step that changed
  __shared__ uint32_t s_hard[2];                 // by pass parity: stale steps to evaluate, others << 16
  static_assert(sizeof(bars) + sizeof(tmem_base_s) + sizeof(abort_flag) + sizeof(s_turns) + sizeof(s_unit) + sizeof(s_change) + sizeof(s_hard) <= kRbStaticSmem,
                "the host sizes the dynamic shared memory beside these");

  griddep_launch_dependents();
  const ReplayArgs& a = ar.r;
  const he_config& cfg = a.cfg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = GT > 0 ? GT : cfg.group_size;
  const int GW = G * WORDS;
  const long long Cmax = cfg.max_budget;
  const bool write_scores = (cfg.flags & HE_FLAG_WRITE_SCORES) != 0;
  const int ncta = ar.ncta, lg_ncta = 31 - __clz(ncta), abuf = ar.abuf;
  const int rank = ncta > 1 ? (int)rb_cluster_rank() : 0;
  // rounded up to 1024 bytes by an offset from the array itself: the accesses stay shared-memory accesses
  unsigned char* smem = rb_smem_raw + ((1024u - (smem_u32(rb_smem_raw) & 1023u)) & 1023u);
  const RbLayout& L = ar.L;
  unsigned char* As = smem + L.a;
  unsigned char* Bx = smem + L.bidx;
  unsigned char* Bs = smem + L.b;
  uint32_t* codes = reinterpret_cast<uint32_t*>(smem + L.codes);
  uint8_t* own = smem + L.own;
  uint32_t* own32 = reinterpret_cast<uint32_t*>(own);  // wide
  int32_t* Mx = reinterpret_cast<int32_t*>(smem + L.mx);
  const int top_at = HALF ? L.top_at : RM * L.mx_pitch;  // where a CTA's block of Mx holds its groups' best keys
  uint16_t* Dn = reinterpret_cast<uint16_t*>(smem + L.dn);
  int32_t* RN = reinterpret_cast<int32_t*>(smem + L.rn);    // per step: best base key
  int32_t* NR = reinterpret_cast<int32_t*>(smem + L.nr);    // per step: largest rank of any earlier key of the block, two buffers
  uint16_t* SV = reinterpret_cast<uint16_t*>(smem + L.sv);  // per step: the slot it writes, as far as known
  int32_t* SN = reinterpret_cast<int32_t*>(smem + L.sn);    // what the evaluation of a hard step gave
  uint8_t* LIST = smem + L.list;                            // the pass's hard steps: step | stale << 7
  int32_t* PAR = reinterpret_cast<int32_t*>(smem + L.par);  // per step: bits set in the xor of its query codes, two buffers
  uint32_t* qraw = reinterpret_cast<uint32_t*>(smem + L.qraw);
  uint32_t* kraw = reinterpret_cast<uint32_t*>(smem + L.kraw);
  int32_t* REC = reinterpret_cast<int32_t*>(smem + L.rec);  // PROT: slot of the m-th newest token before the block at [m - 1]
  const int a_step = WORDS == 2 ? kRbAtom : 64;             // bytes between the two buffers of operand A

  const uint32_t bar0 = smem_u32(bars);
  // bar0 ..: product n mod 8 is complete, its accumulator may be read and its operand tile rewritten
  const uint32_t peer_bar = bar0 + 8u * kRbDoneBars;           // peers' copies of their tiles' maxima have arrived
  const uint32_t used_bar = bar0 + 8u * (kRbDoneBars + 1);     // peers: they are done with this CTA's maxima
  const uint32_t adone_bar = bar0 + 8u * (kRbDoneBars + 2);    // one operand A buffer: the block's tiles are multiplied
  const uint32_t drain_bar = bar0 + 8u * (kRbDoneBars + 3);    // abort path
  const uint32_t tops_bar = bar0 + 8u * (kRbDoneBars + 4);     // peers' copies of their best keys have arrived
  if (tid == 0) {
    abort_flag = 0;
    s_turns[0] = s_turns[1] = -1;
    mbar_init(drain_bar, 2);
    mbar_init(adone_bar, 2);
    for (int i = 0; i < kRbDoneBars; ++i) mbar_init(rb_done_bar(bar0, i), 1);
    mbar_init(peer_bar, 1);
    mbar_init(tops_bar, 1);
    mbar_init(used_bar, ncta > 1 ? ncta - 1 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kRbMmaWarp) {  // four accumulators of 128 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(kRbAccs * kRbTile)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (!wide)
#pragma unroll 1
    for (int i = tid; i < a.smem_slots / 4; i += NT) own32[i] = 0xFFFFFFFFu;
  griddep_wait();  // everything above overlaps the hashing kernel's tail
  tc_fence_before();
  __syncthreads();
  if (ncta > 1) rb_cluster_sync();  // every CTA of the cluster runs before anyone copies into it
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  // Tiles so far; every role counts the same sequence. Tile n lives in operand tile and accumulator n mod 4; warp 16 + (n mod 2) issues its
  // product, so that the even and the odd products each complete in order. A wait for product n may only be begun once product n - 8
  // is known to be complete (the barrier's phases alternate): readers have read product n - 6 before it or come from a block's start, where
  // everything is complete, and expanding warps have waited for products of the same parity.
  int it = 0;
  int blk = 0, turn = 0;  // blocks settled and turns of the block loop so far
  if (warp < 4)
    for (int x = 0; x < kRbAccs; ++x) rb_tile_arrive(x);  // nothing is in the accumulators

  // (the unit number is double-buffered: a peer may still be reading the one before)
#pragma unroll 1
  for (int nunit = 0;; ++nunit) {
    if (ar.scheduled) {
      if (rank == 0 && warp == 0) {
        const int u = claim_unit(a.sched, lane);
        if (lane < ncta) {
          if (ncta > 1) rb_st_remote(rb_mapa(smem_u32(&s_unit[nunit & 1]), (uint32_t)lane), (uint32_t)u);
          else s_unit[nunit & 1] = u;
        }
      }
      __syncthreads();
      if (ncta > 1) rb_cluster_sync();
    } else {
      if (nunit > 0) break;
      if (tid == 0) s_unit[0] = (int)blockIdx.x >> lg_ncta;
      __syncthreads();
    }
    const long long unit = s_unit[nunit & 1];
    if (unit < 0) break;
    const int s = (int)(unit / cfg.n_kv_heads);
    const int C = clamp_budget(a.ca.budget[s], (int)Cmax);
    const int N = clamp_len(a.prompt_len[s], a.Nmax, C);
    const int fill0 = N < C ? N : C;
    const uint32_t* kc_u = a.kcodes + unit * a.Nmax * WORDS;
    const uint32_t* qc_u = a.qcodes + unit * a.Nmax * G * WORDS;
    float* sc = a.ca.scores + unit * Cmax;
    int32_t* pos_g = a.ca.pos + unit * Cmax;
    const int S = PROT ? cfg.n_sink : 0, Rn = PROT ? cfg.n_recent : 0;
    const int nbase = (C + kRbTile - 1) / kRbTile;
    const int ntl_unit = nbase > rank ? (nbase - rank + ncta - 1) >> lg_ncta : 0;  // this CTA's tiles: rank, rank + ncta, ...
    const int R = min(rb_block_rows(C, G * cfg.hash_bits), RM);
    // the first C tokens fill the cache in order; everything beyond `fill` is reset
    for (int j = tid; j < nbase * kRbTile; j += NT) {
#pragma unroll
      for (int w = 0; w < WORDS; ++w) codes[j * WORDS + w] = j < fill0 ? __ldg(kc_u + (long long)j * WORDS + w) : 0u;
    }
    for (int j = rank * NT + tid; j < (int)Cmax; j += ncta * NT) pos_g[j] = j < fill0 ? j : -1;
    if (wide)
      for (int j = tid; j < nbase * kRbTile; j += NT) own32[j] = 0xFFFFFFFFu;
    uint32_t era = kRbFirstEra;  // wide: claims of the current pass are era | step, of earlier ones larger
    if (PROT && tid < Rn) REC[tid] = C - 1 - tid;  // (the first C tokens sit in slot = position)
    // Further columns of operand B (columns of A: 16, 1, 2^15, off, -64 parity): digits of 128 - x, 256, 1, 1; rows that may not win
    // have 256 alone. Variant bit 0: the tile holds the protected first tokens, bit 1: the budget ends inside the tile.
    if (tid < 4 * kRbTile) {
      const int x = tid & 127, v = tid >> 7;
      const bool bad = ((v & 1) && x < S) || ((v & 2) && x >= C - (nbase - 1) * kRbTile);
      const uint32_t one = rb_e4m3(1), top = rb_e4m3(256) << 16;
      *reinterpret_cast<uint4*>(Bx + rb_swz(x, 2 * v)) =
          bad ? make_uint4(top, 0u, 0u, 0u) : make_uint4(rb_e4m3((128 - x) >> 4) | (rb_e4m3((128 - x) & 15) << 8) | top | (one << 24), one, 0u, 0u);
      *reinterpret_cast<uint4*>(Bx + rb_swz(x, 2 * v + 1)) = make_uint4(0u, 0u, 0u, 0u);
    }
    // The block's query and key codes into buffer `buf` (rows past the prompt keep what was there: nothing reads them).
    auto stage_codes = [&](int buf, int tb, int nrows, int first, int nthreads) {
      uint32_t* qd = qraw + buf * kRbRows * GW;
      uint32_t* kd = kraw + buf * kRbRows * WORDS;
      const uint32_t* qs = qc_u + (long long)tb * GW;
      const uint32_t* ks = kc_u + (long long)tb * WORDS;
#pragma unroll 1
      for (int i = first; i < nrows * GW; i += nthreads)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(qd + i)), "l"(qs + i) : "memory");
#pragma unroll 1
      for (int i = first; i < nrows * WORDS; i += nthreads)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(kd + i)), "l"(ks + i) : "memory");
      cp_async_commit();
    };
    fence_proxy_async();
    __syncthreads();
    // A turn works on the block of steps t0 .. tn - 1 and prepares the next one; a unit's first turn has no steps yet.
    int cur = 0, rows = 0;
#pragma unroll 1
    for (int t0 = C; t0 < N;) {
      const int tn = t0 + rows, ntl = rows > 0 ? ntl_unit : 0;
      const uint32_t* qb = qraw + cur * kRbRows * GW;
      const uint32_t* kb_codes = kraw + cur * kRbRows * WORDS;
      // ---------------------------------------------------------------- tile phase
      // this CTA's base tiles 0 .. ntl - 1 (tile i of the CTA is tile i * ncta + rank of the unit)
      if (warp < kExpWarp) {
        const int r = tid & 127, grp = warp >> 2;  // this thread's step = its tensor-memory lane; tiles grp, grp + kGroups, ...
        int32_t* mrow = Mx + rank * L.mx_block + min(r, RM) * L.mx_pitch;
        const int ct = (127 - ((grp << lg_ncta) + rank)) * 128;  // 127 - tile goes above the index within the tile (lower tiles first)
        const int cstep = (128 * kGroups) << lg_ncta;
        const uint32_t taddr0 = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        if (ncta > 1 && blk > 0 && rows > 0) rb_wait_cluster(used_bar, (blk - 1) & 1, &abort_flag);  // peers still read the block before
        const int top = rb_read_tiles<kGroups>(bar0, &abort_flag, it, grp, ntl, taddr0, smem_u32(mrow), ct, cstep);
        if (rows > 0 && r < RM) Mx[rank * L.mx_block + top_at + grp * RM + r] = top;  // this group's best key of the step
        if (ncta > 1) fence_proxy_async();
      } else if (warp < kRbMmaWarp) {
        if (ncta > 1 && rows > 0 && tid == 32 * kRbAuxWarp) {
          mbar_arrive_expect_tx(tops_bar, (uint32_t)(kGroups * RM * (ncta - 1)) * 4u);
          mbar_arrive_expect_tx(peer_bar, 4u * (uint32_t)(top_at * (ncta - 1)));
        }
        const int aux = tid - 32 * kRbAuxWarp, nrows = min(N - tn, R);
        if (tn < N && warp >= kRbAuxWarp) stage_codes(cur ^ 1, tn, nrows, aux, kRbAuxThreads);  // the next block's codes arrive meanwhile
        // teams of two warps write the operand tiles in turn
        const int x = tid & 63, i = (((warp - kExpWarp) >> 1) - it) & (kTeams - 1), j = rank * kRbTile + x;
        rb_expand_tiles<WORDS, kTeams>(bar0, &abort_flag, it, i, ntl, smem_u32(codes + j * WORDS), (uint32_t)(kRbTile * WORDS * 4) << lg_ncta, smem_u32(Bs) + rb_row_at<WORDS>(x, (it + i) & 3),
                                       smem_u32(Bs) + rb_row_at<WORDS>(x, (it + i + kTeams) & 3), j, kRbTile << lg_ncta, S, C);
        if (tn < N && warp >= kRbAuxWarp) {  // the next block: operand A, its own keys' ranks
          cp_async_wait_all();
          if (abuf == 1) rb_wait(adone_bar, turn & 1, &abort_flag);  // a single operand A is free after the block's last tile
          rb_bar<3, kRbAuxThreads>();
          rb_prepare<WORDS, GT, PROT, RM>(L, (int)(smem - rb_smem_raw), cur ^ 1, nrows, it + ntl, G, Rn, abuf, bar0, &abort_flag, tmem_base);
        }
        if (warp == kRbAuxWarp) rb_see_out(s_turns, turn, &abort_flag);
      } else {
        // index-column variants: the unit's first tile (protected first tokens) and its last (the budget ends in it)
        const int first_i = S > 0 && rank == 0 ? 0 : -1, last_i = ((nbase - 1 - rank) & (ncta - 1)) == 0 ? ntl - 1 : -1;
        const uint32_t a_at = smem_u32(As);
        if (__builtin_expect(!__any_sync(0xFFFFFFFFu, abort_flag != 0), 1))
          rb_issue_tiles<WORDS>(bar0, it, ntl, warp - kRbMmaWarp, tmem_base, a_at + (abuf > 1 ? cur * a_step : 0), a_at + (abuf > 1 ? (cur ^ 1) * a_step : 0), smem_u32(Bx),
                                smem_u32(Bs), first_i, last_i, abuf == 1 ? adone_bar : 0u, tn < N);
        s_turns[warp - kRbMmaWarp] = turn;
      }
      it += ntl + (tn < N ? 1 : 0);
      if (warp < kRbResWarps && rows > 0) {
        rb_bar<2, kRbResThreads>();  // the reader groups see each other's results
        if (tid < ncta - 1) {        // ... and every peer gets this CTA's block
          const uint32_t peer = (uint32_t)((rank + 1 + tid) & (ncta - 1)), la = smem_u32(Mx + rank * L.mx_block);
          // the best keys, which the settling starts from, then the tiles' (1 KB each against 6 KB at 9830 slots and 8 CTAs)
          const uint32_t tops = la + 4u * (uint32_t)top_at;
          rb_copy_to_peer(rb_mapa(tops, peer), tops, (uint32_t)(kGroups * RM) * 4u, rb_mapa(tops_bar, peer));
          rb_copy_to_peer(rb_mapa(la, peer), la, 4u * (uint32_t)top_at, rb_mapa(peer_bar, peer));
        }
        __syncwarp();
      }
      // ---------------------------------------------------------------- settle the block's steps
      // Owner table: the first step that claims a slot in this pass. Wide: the smallest of era | step, by an atomic minimum; eras
      // descend from pass to pass, so that older claims count as none and nothing is ever cleared: (own32 - era) < r says that a
      // step before r claims the slot. Narrow: own[slot] = step | pass parity << 7, (own ^ tag) < r says so (0xFF: nobody), and
      // claims of the pass before are taken back.
      if (warp < kRbResWarps && rows > 0) {
        tc_fence_before();
        const int r = tid;  // warps 0-3: this thread's step
        era -= 256u;
        if (wide && __builtin_expect(era < kRbLastEra, 0)) {  // (16 million passes on)
#pragma unroll 1
          for (int j = tid; j < nbase * kRbTile; j += kRbResThreads) own32[j] = 0xFFFFFFFFu;
          era = kRbFirstEra;
          rb_bar<2, kRbResThreads>();
        }
        const bool mine = tid < rows;
        int top_slot = 0, sv = 0, prev = 0;  // warps 0-3: best base slot, slot that the step writes (now, a pass ago)
        bool forced = false, flagged = false;  // ... the best base slot holds a recent token; or a new entry may win
        if (warp < 4) {
          if (ncta > 1) rb_wait_cluster(tops_bar, blk & 1, &abort_flag);
          int top = -1;
#pragma unroll 1
          for (int c = 0; c < ncta; ++c)
#pragma unroll
            for (int g = 0; g < kGroups; ++g) top = max(top, Mx[c * L.mx_block + top_at + g * RM + (r < RM ? r : 0)]);
          top_slot = max(0, min(kRbIdxMask - (top & kRbIdxMask), C - 1));
          sv = prev = top_slot;
          if (PROT && 32 * warp < Rn)  // REC[m] entered m + 1 steps before the block: recent while r + m < Rn
            for (int m = 0; m < Rn; m += 4) {
              const int4 q = *reinterpret_cast<const int4*>(REC + m);
              const int left = Rn - r - m;
              forced |= (left > 0 && q.x == top_slot) | (left > 1 && q.y == top_slot) | (left > 2 && q.z == top_slot) | (left > 3 && q.w == top_slot);
            }
          flagged = forced || NR[cur * kRbRows + r] >= (top >> kRbKeyShift);
          RN[r] = top;
          if (tid < 2) s_change[tid] = kRbRows, s_hard[tid] = 0u;
        }
        int fb = 0;                    // steps below are final
#pragma unroll 1
        for (int pass = 0;; ++pass) {  // every pass but the last of a window makes at least one more step final
          const int wend = min(fb + (pass < kRbWidePasses ? kRbRows : kRbResWarps), rows);
          const uint32_t tag = (uint32_t)(pass & 1) << 7;
          const int par = pass & 1;
          bool is_hard = false;
          if (warp < 4) {
            SV[r] = mine ? (uint16_t)sv : (uint16_t)0xFFFFu;
            bool stale;
            if (wide) {
              if (mine) atomicMin(&own32[sv], era | (uint32_t)r);
              rb_bar<1, kRbRows>();
              stale = own32[top_slot] - era < (uint32_t)r;
            } else {
              // Earlier warps store after later ones, so that a slot goes to its first warp; among that warp's lanes any may win,
              // the earlier ones store again.
#pragma unroll
              for (int k = 3; k >= 0; --k) {
                if (warp == k && mine) own[sv] = (uint8_t)((uint32_t)r | tag);
                rb_bar<1, kRbRows>();
              }
#pragma unroll 1
              for (;;) {
                const uint32_t o = own[sv] ^ tag;
                const bool again = mine && (int)(o >> 5) == warp && o > (uint32_t)r;
                if (!__any_sync(0xFFFFFFFFu, again)) break;
                if (again) own[sv] = (uint8_t)((uint32_t)r | tag);
                __syncwarp();
              }
              rb_bar<1, kRbRows>();
              const uint32_t o_top = own[top_slot];
              if (prev != sv && (own[prev] ^ (tag ^ 0x80u)) < 128u) own[prev] = 0xFFu;  // claimed a pass ago, by nobody now
              stale = (o_top ^ tag) < (uint32_t)r;
            }
            // hard steps of the window
            is_hard = r >= fb && r < wend && (flagged || stale);
            const uint32_t hm = __ballot_sync(0xFFFFFFFFu, is_hard);
            const bool scan = is_hard && (stale || forced);
            const uint32_t sm = __ballot_sync(0xFFFFFFFFu, scan), fm = hm & ~sm, lt = (1u << lane) - 1u;
            uint32_t at = 0u;
            if (lane == 0 && hm != 0u) at = atomicAdd(&s_hard[par], (uint32_t)(__popc(sm) | __popc(fm) << 16));
            at = __shfl_sync(0xFFFFFFFFu, at, 0);
            // the stale steps from the list's start on, the others from its end
            if (is_hard) LIST[scan ? (at & 0xFFFFu) + __popc(sm & lt) : kRbRows - 1 - (at >> 16) - __popc(fm & lt)] = (uint8_t)((uint32_t)r | (scan ? 0x80u : 0u));
            if (!is_hard && r >= fb && r < wend && sv != top_slot) atomicMin(&s_change[par], r);
            if (ncta > 1 && pass == 0) rb_wait_cluster(peer_bar, blk & 1, &abort_flag);  // the peers' tile maxima
          }
          rb_bar<2, kRbResThreads>();
          if (tid == 0) s_change[par ^ 1] = kRbRows, s_hard[par ^ 1] = 0u;
          // The stale steps first, then the others, dealt to and fro over the warps: an evaluation with a scan takes twice as long as one without
          // (900 to 1400 cycles, 450 to 680), so that a warp with a second one has two short ones. 128 units of 1024 slots, windows: 1243 -> 1225 us
          // of replay; dealing to 18 warps instead gained nothing, as the longest evaluation counts. One list, filled from both ends by an atomic
          // addition a warp. The addition costs a pass 110 cycles (one layer of 32 units: 560 a pass for 450), 0.9 % of a block of the longest tables, which
          // have five hard steps a pass and gain nothing; what else there is costs more. Four lists looked through at every evaluation: the same call
          // 1404 us for 1359, b = 8 2 to 4 %; the ballots as words, an entry found in them by lane: 250 cycles a pass, but 490 more in its
          // evaluations, 1424 us; places from the warps' counts behind one more barrier: 1377; four lists without an order: 1427, while 256 units of 9830
          // slots take 6181 for 6208 and b = 8 stays where it is.
          const int ns = (int)(s_hard[par] & 0xFFFFu), n3 = ns + (int)(s_hard[par] >> 16);
          if (__builtin_expect(32 * n3 > 31 * (wend - fb), 0)) {
            const int walk = rb_walk_cost(WORDS, GT, PROT, (C + kRbResThreads - 1) / kRbResThreads);
            if (pass * rb_pass_cost(n3) > 2 * fb * walk && 2 * pass * (rows - fb) > rows) break;  // the rest is walked
          }
#pragma unroll 1
          for (int e0 = warp, fro = kRbResWarps - 1 - 2 * warp; e0 < n3; e0 += kRbResWarps + fro, fro = -fro) {
            const int entry = LIST[e0 < ns ? e0 : kRbRows - 1 - (e0 - ns)];
            const int r2 = entry & 127;
            const uint2 dd = *reinterpret_cast<const uint2*>(Dn + cur * L.dn_buf + rb_dn_at(r2, RM) + (4 * lane < r2 ? 4 * lane : 0));
            const uint2 s4 = *reinterpret_cast<const uint2*>(SV + 4 * lane);
            int kb = RN[r2];
            const int sv2 = SV[r2];
            // best new entry: written by an earlier step and no longer recent (whether a later step has overwritten it is
            // looked at below, if it matters)
            const int elim = (PROT ? r2 - Rn : r2) - 4 * lane;
            auto ekey = [&](int e, uint32_t d2, uint32_t slot) {
              return e < elim ? (int)((d2 << (kRbKeyShift - 1)) + (kRbIdxMask - slot)) : -1;
            };
            int k0 = ekey(0, dd.x & 0xFFFFu, s4.x & 0xFFFFu), k1 = ekey(1, dd.x >> 16, s4.x >> 16);
            int k2 = ekey(2, dd.y & 0xFFFFu, s4.y & 0xFFFFu), k3 = ekey(3, dd.y >> 16, s4.y >> 16);
            int kn = __reduce_max_sync(0xFFFFFFFFu, max(max(k0, k1), max(k2, k3)));
            // Both candidates are upper bounds until looked at; the larger one is, until it holds. A base slot may be taken
            // (or recent): its tile is scanned again for this step and its live slots replace the tile's maximum. A new
            // entry may have been overwritten: it leaves the race. Each round takes a tile or an entry out.
            bool exact = (entry & 0x80) == 0;  // kb is a live slot's key
            bool loaded = false;
            int mt[4];  // lane l: tiles l, l + 32, ...
            RbRank<WORDS, GT> rk;
            int live = -1;  // best live slot of the tiles scanned so far, this lane's share
#pragma unroll 1
            for (int round = 0; round <= nbase + kRbRows; ++round) {
              if (kn > kb) {
                const uint32_t slot = (uint32_t)(kRbIdxMask - (kn & kRbIdxMask));
                const bool e0s = (s4.x & 0xFFFFu) == slot, e1s = (s4.x >> 16) == slot, e2s = (s4.y & 0xFFFFu) == slot, e3s = (s4.y >> 16) == slot;
                const int before = r2 - 4 * lane;  // entries of this lane below it were written before step r2
                int l = -1, kl = -1;
                if (e0s && 0 < before) l = 0, kl = k0;
                if (e1s && 1 < before) l = 1, kl = k1;
                if (e2s && 2 < before) l = 2, kl = k2;
                if (e3s && 3 < before) l = 3, kl = k3;
                const int newest = __reduce_max_sync(0xFFFFFFFFu, l < 0 ? -1 : 4 * lane + l);
                if (__any_sync(0xFFFFFFFFu, l >= 0 && 4 * lane + l == newest && kl == kn)) break;
                // the slot holds a later entry with another rank, or one that is still recent
                if (e0s && 4 * lane != newest) k0 = -1;
                if (e1s && 4 * lane + 1 != newest) k1 = -1;
                if (e2s && 4 * lane + 2 != newest) k2 = -1;
                if (e3s && 4 * lane + 3 != newest) k3 = -1;
                kn = __reduce_max_sync(0xFFFFFFFFu, max(max(k0, k1), max(k2, k3)));
                continue;
              }
              if (exact || kb < 0) break;
              const int sb = min(kRbIdxMask - (kb & kRbIdxMask), C - 1);
              if (loaded) {  // (the first time it is known to be taken, or recent)
                bool bad = wide ? own32[sb] - era < (uint32_t)r2 : (own[sb] ^ tag) < (uint32_t)r2;
                if (PROT && r2 < Rn && !bad) {  // REC[m - 1] entered m steps before the block: recent while r2 + m <= Rn
                  bool hit = false;
#pragma unroll 1
                  for (int m0 = 0; m0 < Rn - r2; m0 += 32) hit |= m0 + lane < Rn - r2 && REC[m0 + lane] == sb;
                  bad = __any_sync(0xFFFFFFFFu, hit);
                }
                if (!bad) break;
              }
              if (!loaded) {
                loaded = true;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const int T = lane + 32 * i;
                  mt[i] = T < nbase ? Mx[(T & (ncta - 1)) * L.mx_block + r2 * L.mx_pitch + (T >> lg_ncta)] : -1;
                }
                rk.load(qb + r2 * GW, G, PAR[cur * kRbRows + r2]);
              }
              const int cb = sb >> 7, j0 = cb * kRbTile + 4 * lane;
              uint32_t hw[4 * WORDS];
#pragma unroll
              for (int i = 0; i < WORDS; ++i) *reinterpret_cast<uint4*>(hw + 4 * i) = *reinterpret_cast<const uint4*>(codes + j0 * WORDS + 4 * i);
              uint32_t ok4;  // bit 7 of a byte: nobody claims the slot before r2
              if (wide) {
                const uint4 o = *reinterpret_cast<const uint4*>(own32 + j0);
                ok4 = (o.x - era < (uint32_t)r2 ? 0u : 0x80u) | (o.y - era < (uint32_t)r2 ? 0u : 0x8000u) |
                      (o.z - era < (uint32_t)r2 ? 0u : 0x800000u) | (o.w - era < (uint32_t)r2 ? 0u : 0x80000000u);
              } else {  // (unclaimed bytes have bit 7 set, claims are below 128)
                const uint32_t o4 = *reinterpret_cast<const uint32_t*>(own + j0) ^ (tag * 0x01010101u);
                ok4 = (((o4 | 0x80808080u) - (uint32_t)r2 * 0x01010101u) | o4);
              }
              if (PROT && r2 < Rn)  // recent tokens in this tile
#pragma unroll 1
                for (int m0 = 0; m0 < Rn - r2; m0 += 32) {
                  const int q = m0 + lane < Rn - r2 ? REC[m0 + lane] : -1;
#pragma unroll 1
                  for (uint32_t in = __ballot_sync(0xFFFFFFFFu, q >> 7 == cb); in != 0u; in &= in - 1u) {
                    const int at = __shfl_sync(0xFFFFFFFFu, q, __ffs(in) - 1) - j0;
                    if (at >= 0 && at < 4) ok4 &= ~(0x80u << (8 * at));
                  }
                }
              const int hi = C - j0, lo = PROT ? S - j0 : 0;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                uint32_t h[WORDS];
#pragma unroll
                for (int w = 0; w < WORDS; ++w) h[w] = hw[e * WORDS + w];
                const int key = (rk.rank(h) << kRbKeyShift) + (kRbIdxMask - (j0 + e));
                const bool ok = (ok4 & (0x80u << (8 * e))) != 0u && e < hi && (!PROT || e >= lo);
                live = max(live, ok ? key : -1);
              }
              int km = -1;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                if (cb == lane + 32 * i) mt[i] = -1;
                km = max(km, mt[i]);
              }
              kb = __reduce_max_sync(0xFFFFFFFFu, max(live, km));
            }
            const int slot = min(kRbIdxMask - (max(max(kb, kn), 0) & kRbIdxMask), C - 1);
            if (lane == 0) {
              SN[r2] = slot;
              if (slot != sv2) atomicMin(&s_change[par], r2);
            }
          }
          rb_bar<2, kRbResThreads>();
          const int ch = s_change[par];
          era -= 256u;
          prev = sv;
          if (ch < kRbRows) {
            fb = ch + 1;
            if (warp < 4 && r < wend && r >= ch) sv = is_hard ? SN[r] : top_slot;
          } else {
            fb = wend;
            if (fb >= rows) break;
          }
        }
        const int fin = fb;  // the passes have settled the steps below: as a rule all of the block's
        if (ncta > 1 && warp == 4 && lane < ncta - 1) rb_arrive_remote(rb_mapa(used_bar, (uint32_t)((rank + 1 + lane) & (ncta - 1))));
        // ------------------------------------------------------------ Algorithm 1 lines 2-5 on the table
        const bool scoring = write_scores && tn == N;
        auto apply = [&](int slot) {
          if (!HE_IN_RANGE(slot, C)) return;
#pragma unroll
          for (int w = 0; w < WORDS; ++w) codes[slot * WORDS + w] = kb_codes[r * WORDS + w];
          if (rank == 0) pos_g[slot] = t0 + r;
        };
        // last writers: the steps claim again, later ones over earlier ones (the prompt's last step waits until its scores
        // are taken)
        era -= 256u;
        if (warp < 4) {
          const bool in = tid < fin && !(scoring && r == rows - 1);
          if (wide) {
            const uint32_t claim = era | (uint32_t)(kRbRows - 1 - r);
            if (in) atomicMin(&own32[sv], claim);
            rb_bar<1, kRbRows>();
            if (in && own32[sv] == claim) apply(sv);
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (warp == k && in) own[sv] = (uint8_t)r;
              rb_bar<1, kRbRows>();
            }
#pragma unroll 1
            for (;;) {
              const int o = own[sv];
              const bool again = in && (o >> 5) == warp && o < r;
              if (!__any_sync(0xFFFFFFFFu, again)) break;
              if (again) own[sv] = (uint8_t)r;
              __syncwarp();
            }
            rb_bar<1, kRbRows>();
            if (in && own[sv] == (uint8_t)r) apply(sv);
            rb_bar<1, kRbRows>();
            if (mine) own[sv] = 0xFFu;
          }
        }
        if (__builtin_expect(fin < rows, 0)) {
          rb_walk<WORDS, GT, PROT>(L, wide, (int)(smem - rb_smem_raw), cur, rank == 0 ? pos_g : nullptr, t0, fin, rows, scoring ? rows - 1 : rows, C, G, S, Rn);
          if (mine) sv = SV[r];
        }
        int keep = 0;
        if (PROT && tid < Rn) keep = tid < rows ? 0 : REC[tid - rows];
        if (scoring) {  // Eq. 5 for every slot as the prompt's last step sees the table
          rb_bar<2, kRbResThreads>();
          RbRank<WORDS, GT> rk;
          rk.load(qb + (rows - 1) * GW, G, PAR[cur * kRbRows + rows - 1]);
#pragma unroll 1
          for (int j = rank * kRbResThreads + tid; j < C; j += ncta * kRbResThreads) {
            uint32_t h[WORDS];
#pragma unroll
            for (int w = 0; w < WORDS; ++w) h[w] = codes[j * WORDS + w];
            sc[j] = -(float)rk.dist(h);
          }
          rb_bar<2, kRbResThreads>();
          if (tid == rows - 1) apply(sv);
        }
        if (PROT && Rn > 0) {  // the newest tokens before the next block
          rb_bar<2, kRbResThreads>();
          if (tid < Rn) REC[tid] = tid < rows ? (int)SV[rows - 1 - tid] : keep;
        }
      }
      blk += rows > 0 ? 1 : 0;
      ++turn;
      cur ^= 1;
      t0 = tn;
      rows = min(N - tn, R);
      __syncthreads();
      tc_fence_after();
    }
    // final state of the unit; everything beyond `fill` is reset
    const bool scored = write_scores && N > C;
    for (int j = rank * NT + tid; j < (int)Cmax; j += ncta * NT) {
      const bool valid = j < fill0;
      uint32_t cw[WORDS];
#pragma unroll
      for (int w = 0; w < WORDS; ++w) cw[w] = valid ? codes[j * WORDS + w] : 0u;
      store_slot_code<WORDS>(cfg, a.ca.codes, unit * Cmax + j, cw);
      if (!(valid && scored)) sc[j] = 0.f;
    }
    if (rank == 0 && tid == 0) {
      a.ca.fill[unit] = fill0;
      a.ca.next_pos[unit] = N;
    }
    __syncthreads();  // the tables and s_unit are reused by the next unit
  }

  // The readers' last arrivals still stand in the tile barriers: their phases are completed, unless the CTA gave up (every wait that
  // could raise the flag lies before the last barrier of the block loop).
  const bool gave_up = __any_sync(0xFFFFFFFFu, abort_flag != 0);  // one answer for the warp: the election below wants all its lanes
  if (!gave_up && (warp == kRbAuxWarp || warp == kRbAuxWarp + 1))
    for (int x = 0; x < kRbAccs; ++x) rb_tile_arrive(x);
  // A CTA that gave up must not free tensor memory under an MMA that is still writing it (the operands are written by
  // this CTA's own threads, so no copy from outside is ever in flight): one more commit tracks everything that the issuing
  // warp has issued, and its completion is awaited (bounded) first.
  if (warp == kRbMmaWarp || warp == kRbMmaWarp + 1) {
    for (int x = warp - kRbMmaWarp; x < kRbAccs && !gave_up; x += 2) rb_tile_sync(x);
    if (gave_up && tc_elect()) {
      tc_commit(drain_bar);
      mbar_drain(drain_bar, 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kRbMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kRbAccs * kRbTile) : "memory");
  }
  if (tid == 0 && abort_flag) atomicAdd(&g_tc_error, 1);
  if (ncta > 1) rb_cluster_sync();  // no CTA leaves while a peer may still copy into its shared memory
}

}  // namespace he
