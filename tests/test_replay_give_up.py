"""The block replay's way out when a wait is given up: the roles of its tile phase, taken from the kernel's source and run as host threads (a
thread a warp, one lane of it), with named barriers that count arrivals as the hardware's do and products that stop completing at some
point, or an abort flag that another wait raises. Every role has to get through its turns, nothing is issued in a turn that begins with the
flag up, and without it every phase of a tile's barrier is made of one tile's arrivals."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_16187_b200", "csrc")
ROLES = ("rb_wait_polled", "rb_wait", "rb_see_out", "rb_done_bar", "rb_done_phase", "rb_read_tiles", "rb_expand_tiles", "rb_issue_tiles", "rb_prepare")

HARNESS = r"""
#include <atomic>
#include <barrier>
#include <chrono>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <random>
#include <thread>
#include <vector>
struct int2 { int x, y; };
int2 make_int2(int x, int y) { return {x, y}; }
struct uint2 { uint32_t x, y; };
struct uint4 { uint32_t x, y, z, w; };
uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }
#define __device__
#define __noinline__
#define __forceinline__ inline
#define __any_sync(m, x) ((x) != 0)
#define __all_sync(m, x) ((x) != 0)
#define __syncwarp() jitter()
#define __reduce_max_sync(m, x) (x)
constexpr uint32_t kTcSpinLimit = LIMIT;
constexpr int kRbAuxWarp = 12, kRbAuxThreads = 128, kRbMmaWarp = 16, kRbWarps = 18, kRbAccs = 4, kRbDoneBars = 8, kRbTile = 128, kRbRows = 128, kRbAtom = 128 * 128;
thread_local struct { int x; } threadIdx;
thread_local std::minstd_rand rng;
void jitter() { if (rng() % 4 == 0) std::this_thread::yield(); if (rng() % 64 == 0) std::this_thread::sleep_for(std::chrono::microseconds(rng() % 60)); }
std::atomic<bool> mixed{false};

// ---- named barriers of the tiles: 7 warps to a phase; `from` says for which tile an arrival is meant (a reader's arrival frees tile n + 4)
struct Named { std::mutex m; int count = 0; long phase = 0; } named[4];
thread_local std::vector<int> next_tile;  // what this warp arrives for, per accumulator
void arrive_for(int acc, int tile, bool wait) {
  jitter();
  long mine;
  {
    std::lock_guard<std::mutex> l(named[acc].m);
    mine = named[acc].phase;
    if (tile != 4 * mine + acc) mixed = true;
    if (++named[acc].count == 7) named[acc].count = 0, ++named[acc].phase;
  }
  while (wait) {
    { std::lock_guard<std::mutex> l(named[acc].m); if (named[acc].phase != mine) break; }
    jitter();
  }
}
// ---- mbarriers of the products: phases completed so far; a stuck product and all that its warp issues later never complete
std::atomic<long> done[kRbDoneBars];
std::atomic<bool> stuck[2];
int stuck_at, flag_at;
std::mutex late_m; std::vector<std::thread> late;
thread_local int turn_it; thread_local int reading;  // (arrivals that follow a read are for the tile four on)
bool mbar_try_wait(uint32_t bar, uint32_t parity) { jitter(); return (uint32_t)(done[bar / 8].load() & 1) != (parity & 1); }
volatile int abort_flag, turns[2] = {-1, -1};
void __nanosleep(int) { jitter(); }
std::atomic<int> issued_off{0}, products{0};
thread_local bool saw_flag;
void tc_commit(uint32_t bar) {
  if (bar >= 8u * kRbDoneBars) return;
  ++products;
  const int n = next_tile[0];
  if (n == flag_at) abort_flag = 1;  // as if some other wait had run out
  if (n == stuck_at) stuck[n & 1] = true;
  if (!stuck[n & 1]) ++done[bar / 8];
}
void rb_mma_f8(uint32_t, uint64_t, uint64_t, uint32_t, bool) { if (saw_flag) ++issued_off; }
uint64_t umma_desc_k128(uint32_t) { return 0; }
bool tc_elect() { return true; }
void tc_fence_after() {} void tc_fence_before() {} void fence_proxy_async() {} void tc_ld32(uint32_t, uint32_t*) {} void tc_wait_ld() {}
void rb_ld64_low(uint32_t, uint32_t (&v)[32]) { memset(v, 0, sizeof(v)); }
void rb_wait_ld(uint32_t (&)[32]) {}
uint32_t rb_max64(const uint32_t (&)[32], const uint32_t (&)[32]) { return 1; }
uint32_t smem_u32(const void*) { return 0; }
template <int W> void rb_expand_row(const uint32_t (&)[W], uint32_t) {}
template <int W> void rb_clear_row(uint32_t) {}
template <int W> uint32_t rb_row_at(int, int) { return 0; }
template <int W> int rb_off(int) { return 0; }
int rb_alpha(int) { return 1; } int rb_dn_at(int, int) { return 0; } uint32_t rb_e5m2(int) { return 0; } uint32_t rb_swz(int, int) { return 0; }
uint32_t __byte_perm(uint32_t, uint32_t, uint32_t) { return 0; } int __popc(uint32_t x) { return __builtin_popcount(x); }
float __uint_as_float(uint32_t) { return 0.f; } uint32_t __float_as_uint(float) { return 0; }
int max(int a, int b) { return a > b ? a : b; } uint32_t max(uint32_t a, uint32_t b) { return a > b ? a : b; }
using std::fmaxf; using std::fmaf;
struct RbLayout { uint32_t a = 0, kraw = 0, par = 0, nr = 0, dn = 0, dn_buf = 0, qraw = 0, b = 0; };
alignas(16) unsigned char rb_smem_raw_[18][1 << 16];
thread_local int self;
#define rb_smem_raw rb_smem_raw_[self]
std::barrier<> aux_bar(4), all_bar(kRbWarps);
template <int ID, int THREADS> void rb_bar() { static_assert(ID == 3, ""); aux_bar.arrive_and_wait(); }
// a warp arrives for its tiles in the order of its loop; the reader of tile n frees its accumulator for n + 4
thread_local std::vector<int> queue; thread_local size_t at_q;
void rb_tile_arrive(int acc) { arrive_for(acc, at_q < queue.size() ? queue[at_q++] : -1, false); }
void rb_tile_sync(int acc) { const int n = queue[at_q++]; next_tile.assign(1, n); arrive_for(acc, n, true); }
#define asm
#define volatile(...)
ROLES
#undef asm
#undef volatile

template <int WORDS> void warp_main(int warp, const std::vector<int>& tiles, unsigned seed) {
  constexpr int kGroups = WORDS == 2 ? 2 : 3, kExpWarp = 4 * kGroups, kTeams = (kRbMmaWarp - kExpWarp) / 2;
  self = warp; threadIdx.x = 32 * warp; rng.seed(seed * 1000 + warp + 1);
  RbLayout L;
  auto go = [&](std::vector<int> q) { queue = q; at_q = 0; };
  int it = 0;
  if (warp < 4) { go({0, 1, 2, 3}); for (int x = 0; x < 4; ++x) rb_tile_arrive(x); }
  all_bar.arrive_and_wait();
  for (size_t turn = 0; turn < tiles.size(); ++turn) {
    const int ntl = tiles[turn]; const bool next = turn + 1 < tiles.size();
    std::vector<int> q;
    saw_flag = abort_flag != 0;
    if (warp < kExpWarp) {
      for (int i = warp >> 2; i < ntl; i += kGroups) q.push_back(it + i + 4);
      go(q);
      rb_read_tiles<kGroups>(0, &abort_flag, it, warp >> 2, ntl, 0, 0, 0, 0);
    } else if (warp < kRbMmaWarp) {
      const int i0 = (((warp - kExpWarp) >> 1) - it) & (kTeams - 1);
      for (int i = i0; i < ntl; i += kTeams) q.push_back(it + i);
      if (next && warp >= kRbAuxWarp) { if (warp < kRbAuxWarp + 2) q.push_back(it + ntl); q.push_back(it + ntl + 4); }
      go(q);
      rb_expand_tiles<WORDS, kTeams>(0, &abort_flag, it, i0, ntl, 0, 0, 0, 0, 0, 0, 0, 0);
      if (next && warp >= kRbAuxWarp) { rb_bar<3, 128>(); rb_prepare<WORDS, 4, false, 128>(L, 0, 0, 0, it + ntl, 4, 0, 2, 0, &abort_flag, 0); }
      if (at_q != queue.size()) mixed = true;
      if (warp == kRbAuxWarp) rb_see_out(turns, (int)turn, &abort_flag);
    } else {
      const int odd = warp - kRbMmaWarp;
      for (int i = (it ^ odd) & 1; i < ntl; i += 2) q.push_back(it + i);
      if (next && ((it + ntl) & 1) == odd) q.push_back(it + ntl);
      go(q);
      if (saw_flag) at_q = q.size();
      else rb_issue_tiles<WORDS>(0, it, ntl, odd, 0, 0, 0, 0, 0, -1, -1, 8u * kRbDoneBars, next);
      turns[odd] = (int)turn;
    }
    if (warp < kExpWarp && at_q != queue.size()) mixed = true;
    it += ntl + (next ? 1 : 0);
    all_bar.arrive_and_wait();
  }
  auto last = [&](int x) { return it + ((x - it) & 3); };  // what stands in the barriers at the end
  if (abort_flag) return;
  if (warp == kRbAuxWarp || warp == kRbAuxWarp + 1) { go({last(0), last(1), last(2), last(3)}); for (int x = 0; x < 4; ++x) rb_tile_arrive(x); }
  if (warp >= kRbMmaWarp) for (int x = warp - kRbMmaWarp; x < 4; x += 2) { go({last(x)}); rb_tile_sync(x); }
  all_bar.arrive_and_wait();
}
int main(int argc, char** argv) {
  const int code_words = atoi(argv[1]); const unsigned seed = atoi(argv[2]); stuck_at = atoi(argv[3]); flag_at = atoi(argv[4]);
  std::vector<int> tiles = {0};
  for (int i = 5; i < argc; ++i) tiles.push_back(atoi(argv[i]));
  std::thread watch([] { std::this_thread::sleep_for(std::chrono::seconds(20)); printf("stuck\n"); fflush(stdout); _Exit(3); });
  watch.detach();
  std::vector<std::thread> t;
  for (int w = 0; w < kRbWarps; ++w) t.emplace_back([=, &tiles] { code_words == 2 ? warp_main<2>(w, tiles, seed) : warp_main<1>(w, tiles, seed); });
  for (auto& x : t) x.join();
  printf("%s flag %d issued_off %d products %d\n", mixed && !abort_flag ? "mixed" : "whole", (int)abort_flag, issued_off.load(), products.load());
  fflush(stdout);
  _Exit((mixed && !abort_flag) || issued_off ? 4 : 0);
}
"""


def functions(source, names):
    """The definitions of `names`, in the source's order, each with its template line."""
    found = []
    for name in names:
        m = re.search(r"^(?:template <[^\n]*>\n)?(?:__host__ )?__device__[^\n;]*\b%s\(" % name, source, re.M)
        if m is None:
            continue
        end = source.index("\n}\n", m.start()) + 3 if "}" not in source[m.start():].split("\n")[0] else source.index("\n", m.start()) + 1
        found.append((m.start(), source[m.start():end]))
    return "\n".join(text for _, text in sorted(found))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    with open(os.path.join(CSRC, "prefill_block_kernels.cuh")) as f:
        source = f.read()
    roles = functions(source, ROLES)
    roles = roles.replace("#pragma unroll", "// #pragma unroll")
    assert all(f"{name}(" in roles for name in ("rb_wait", "rb_see_out", "rb_read_tiles", "rb_expand_tiles", "rb_issue_tiles", "rb_prepare"))
    at = tmp_path_factory.mktemp("give_up")
    text = HARNESS.replace("ROLES\n", roles + "\n")
    (at / "t.cpp").write_text(text)
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-DLIMIT=4000", "-o", at / "t", at / "t.cpp"], check=True)
    return at / "t"


@pytest.mark.parametrize("words", [1, 2])
@pytest.mark.parametrize("stuck, flag", [(-1, -1), (0, -1), (21, -1), (34, -1), (-1, 17), (-1, 40)])
def test_every_role_gets_through(program, words, stuck, flag):
    for seed in range(3):
        args = [str(x) for x in (words, seed, stuck, flag, 16, 1, 40, 7, 2, 16)]
        r = subprocess.run([program] + args, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0 and r.stdout.startswith("whole"), (args, r.stdout, r.stderr)
        assert f"flag {int(stuck >= 0 or flag >= 0)}" in r.stdout
        if stuck < 0 and flag < 0:
            assert "products 88" in r.stdout  # 82 tiles and the six blocks' own keys
