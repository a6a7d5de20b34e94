// he_attend: Eq. 1 over the compressed cache (Algorithm 1 line 6), the step that follows the eviction:
//   out[g] = sum_j softmax_j(q_g . K_j / sqrt(d)) V_j   over the valid slots of the query head's KV unit.
// All G query heads of a group are served together, so K and V are read once for the group. Each warp walks its
// own slots with an online softmax (running maximum, running sum, unnormalised output) and the partial results are
// merged through shared memory at the end. HBM-bound by design: 2 * C * d * e bytes per unit.
//
//   attend_bf16_kernel<D, NW>  bf16, d = 64 or 128, G <= 8: 32 slots at a time from rings of TMA tiles, Q K^T and P V as warp-level
//                          m16n8k16 MMAs (bf16 products are exact, fp32 accumulation, P as hi + lo bf16); a cluster of up
//                          to 16 CTAs shares a unit when there are few units.
//   attend_generic_kernel  any supported dtype / d, and where no tensor map can be encoded: one slot at a time, dot products by
//                          warp shuffles.
#pragma once
#include <cuda.h>  // CUtensorMap (types only; the encoder is fetched through the runtime)

#include "common.cuh"

namespace he {

struct AttendArgs {
  he_config cfg;
  he_cache ca;
  const void* q;  // [B, Hkv*G, d]
  float* out;     // [B, Hkv*G, d] fp32
};

constexpr int kAttendThreads = 256;
constexpr int kAttendWarps = kAttendThreads / 32;
constexpr float kLog2e = 1.4426950408889634f;

// Merge of the per-warp partial results (m = running max in log2 units, l = running sum, o = unnormalised output).
// part_ml: [warps][G][2], part_o: [warps][G][d]. Every thread writes some of the G * d outputs.
template <int NW>
__device__ __forceinline__ void attend_merge(const float* part_ml, const float* part_o, int G, int d, float* out_unit) {
  for (int idx = threadIdx.x; idx < G * d; idx += 32 * NW) {
    const int g = idx / d, c = idx % d;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) M = fmaxf(M, part_ml[(w * G + g) * 2]);
    float L = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float m = part_ml[(w * G + g) * 2];
      const float f = m == -INFINITY ? 0.f : exp2f(m - M);
      L += part_ml[(w * G + g) * 2 + 1] * f;
      O += part_o[(w * G + g) * d + c] * f;
    }
    out_unit[idx] = L > 0.f ? O / L : 0.f;
  }
}

// A cluster of S CTAs on one unit: CTA r > 0 folds its warps and sends the result (G maxima, G sums, G * d outputs) to CTA 0 as
// asynchronous remote stores that count on CTA 0's mbarrier; CTA 0 folds its own into place 0 of `gather`, waits and
// combines. One way across the cluster, no barrier at the end. (Two cluster barriers around remote reads cost 4 us a call
// with 8 CTAs, as much as the streaming of 5 MB per cluster.) The wait is bounded; on a time-out the unit's output is
// undefined and the device error counter is raised.
__device__ __forceinline__ uint32_t attend_mapa(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
constexpr uint32_t kAttendSpinLimit = 1u << 22;
template <int NW>
__device__ __forceinline__ void attend_merge_cluster(const float* part_ml, const float* part_o, float* gather, uint32_t bar, int G,
                                                     int d, int S, int rank, float* out_unit) {
  const int per = G * (d + 2);  // floats of one CTA's result: [G] maxima, [G] sums, [G][d] outputs
  for (int idx = threadIdx.x; idx < G * d; idx += 32 * NW) {
    const int g = idx / d, c = idx % d;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) M = fmaxf(M, part_ml[(w * G + g) * 2]);
    float L = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float m = part_ml[(w * G + g) * 2];
      const float f = m == -INFINITY ? 0.f : exp2f(m - M);
      L += part_ml[(w * G + g) * 2 + 1] * f;
      O += part_o[(w * G + g) * d + c] * f;
    }
    if (rank == 0) {
      if (c == 0) gather[g] = M, gather[G + g] = L;
      gather[2 * G + idx] = O;
    } else {
      const uint32_t dst = attend_mapa((uint32_t)__cvta_generic_to_shared(gather + rank * per), 0u), rb = attend_mapa(bar, 0u);
      auto send = [&](int at, float v) {
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst + 4u * at), "r"(__float_as_uint(v)), "r"(rb)
                     : "memory");
      };
      if (c == 0) send(g, M), send(G + g, L);
      send(2 * G + idx, O);
    }
  }
  if (rank != 0) return;
  bool ok = false;
  for (uint32_t i = 0; i < kAttendSpinLimit && !ok; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar)
        : "memory");
    ok = done != 0;
  }
  if (!ok && threadIdx.x == 0) atomicAdd(&g_tc_error, 1);
  __syncthreads();
  for (int idx = threadIdx.x; idx < G * d; idx += 32 * NW) {
    const int g = idx / d;
    float M = -INFINITY;
#pragma unroll 4
    for (int r = 0; r < S; ++r) M = fmaxf(M, gather[r * per + g]);
    float L = 0.f, O = 0.f;
#pragma unroll 4
    for (int r = 0; r < S; ++r) {
      const float m = gather[r * per + g];
      const float f = m == -INFINITY ? 0.f : exp2f(m - M);
      L += gather[r * per + G + g] * f;
      O += gather[r * per + 2 * G + idx] * f;
    }
    out_unit[idx] = L > 0.f ? O / L : 0.f;
  }
}

// ------------------------------------------------------------------------------------------------ bf16, d = 64 or 128
//
// A warp takes 32 slots at a time. Scores: S[head][slot] = Q K^T as m16n8k16 MMAs with M = query heads (rows 0..7
// used), N = 8 slots, K = 16 channels. A dot product does not depend on the order of its terms, so the 16 "logical"
// channels of MMA step s are chosen to suit 16-byte reads: lane (gid, tig) reads chunks 2 tig and 2 tig + 1 (8 channels each) of
// every 64 channels of row gid; the c-th of them feeds steps 2c (first two registers) and 2c+1 (last two); the
// query fragment is loaded the same way, so both operands agree on the permutation.
// Output: O[head][channel] += P V with M = heads, K = 16 slots, N = 8 channels. The score tile's accumulator layout
// is already the A-fragment layout of P (head gid, slots 2tig, 2tig+1 [+8]). P is split into two bf16 terms
// (p = hi + lo + O(2^-18 p)): hi in rows 0..7, lo in rows 8..15 of the same MMA, summed at the end, so that the
// rows a group of <= 8 heads leaves empty carry the low-order term. The B fragment wants pairs of slots per
// channel: lane (gid, tig) holds slots 2tig, 2tig+1, 2tig+8, 2tig+9 and chunks gid, gid+8 of each, and a byte
// permute pairs the two slots' values of one channel. Output tile t = 8h + e of lane column n is channel
// (n + 8h) * 8 + e.

__device__ __forceinline__ void mma_bf16_m16n8k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                  uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// (hi, lo) bf16 pairs of two fp32 values: hi = round-to-nearest bf16, lo = bf16 of the exact remainder.
// The first value goes to the low half (the lower k index of the fragment).
__device__ __forceinline__ void split_pair(float x, float y, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(hi) : "f"(y), "f"(x));
  const float xr = x - __uint_as_float(hi << 16), yr = y - __uint_as_float(hi & 0xFFFF0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(lo) : "f"(yr), "f"(xr));
}

__device__ __forceinline__ uint4 ldg_stream16(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// K and V rows travel through shared memory as TMA tile copies, a warp's 32-slot groups as a ring of items K0, V0, K1, V1, ...
// that only this warp asks for and reads (an mbarrier per ring buffer, no block barrier). What bounds the call is bytes in
// flight: HBM's latency under load times its bandwidth is about 8 MB, 55 KB per SM, and registers alone hold half of it
// next to the accumulators; the rings keep 128 KB in flight. Calls with few units are bound by what one SM pulls: 16-byte
// cp.async copies into the same rings reached 28 bytes a cycle. The 128-byte swizzle puts chunk c of row r at c ^ (r & 7), and
// the fragment reads below are chosen to meet every bank once: a K read takes the even or the odd chunks of two
// neighbouring rows, a V read two neighbouring chunks of rows r, r + 2, r + 4, r + 6.
//
// Eight warps per SM: NW = 8 is one CTA per SM, for grids that do not fill the SMs twice; NW = 4 two, so that one streams while
// the other starts or merges.
//
// Grid (Hkv * S, B) in clusters of S CTAs along x: the S CTAs of a cluster share one unit's slots (32-slot groups
// dealt round-robin over the S * NW warps), each merges its own warps, and the cluster merges the S partial results
// through distributed shared memory, so a call with few units still fills the GPU without any scratch in HBM.
// Launched with the programmatic-serialization attribute: set-up overlaps the tail of the stream's previous kernel (usually
// the decode step), everything the caller or that kernel wrote is read after the wait.
// Dynamic shared memory: the warps' rings, reused by part_ml [warps][G][2], part_o [warps][G][d]; then, with S > 1, the S CTAs'
// partial results (CTA 0's are used), which may arrive while the rings are still in use.
constexpr int kAttendGroup = 32;  // slots per item
template <int D, int NW>
struct AttendRing {
  static constexpr int kBufs = 3 * (128 / D);  // items in a warp's ring: one being read, the others in flight
  static constexpr int kItemBytes = kAttendGroup * D * 2;
  static constexpr int kBytes = NW * kBufs * kItemBytes;  // 24 KB per warp
};

template <int D, int NW>
__global__ void __launch_bounds__(32 * NW, 8 / NW) attend_bf16_kernel(const AttendArgs a, const int S, const __grid_constant__ CUtensorMap kmap,
                                                                     const __grid_constant__ CUtensorMap vmap) {
  using Ring = AttendRing<D, NW>;
  extern __shared__ __align__(16) unsigned char attend_smem_raw[];
  __shared__ __align__(8) unsigned long long merge_bar, ring_bar[NW][Ring::kBufs];
  constexpr int d = D, CPR = D / 8;        // 16-byte chunks per row
  constexpr int NC = D / 32, NH = D / 64;  // chunks of a K row per lane, of a V row per lane
  constexpr int NBUF = Ring::kBufs, GRP = kAttendGroup;
  const he_config& cfg = a.cfg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const int rank = blockIdx.x % S;
  const int unit = blockIdx.y * cfg.n_kv_heads + blockIdx.x / S;
  const int G = cfg.group_size;
  // rounded up to 1024 bytes (the swizzle's period) by an offset from the array itself
  float* asm_ = reinterpret_cast<float*>(attend_smem_raw + ((1024u - ((uint32_t)__cvta_generic_to_shared(attend_smem_raw) & 1023u)) & 1023u));
  float* part_ml = asm_;
  float* part_o = part_ml + NW * G * 2;
  float* gather = asm_ + Ring::kBytes / 4;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&merge_bar);
  unsigned char* ring = reinterpret_cast<unsigned char*>(asm_) + warp * NBUF * Ring::kItemBytes;
  auto full = [&](int b) { return (uint32_t)__cvta_generic_to_shared(&ring_bar[warp][b]); };

  griddep_launch_dependents();
  if (lane == 0) {
#pragma unroll
    for (int b = 0; b < NBUF; ++b) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full(b)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (S > 1) {
    if (rank == 0 && tid == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)((S - 1) * G * (d + 2) * 4)) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // waited for before the first remote store
  }
  const int stride = GRP * NW * S, first = GRP * (warp * S + rank);
  // Where the grid is one wave, each warp's first rows are asked into L2 while the stream's previous kernel (usually the decode step,
  // which moves little) runs: a prefetch returns no data, so it cannot see a stale row. (fill is a hint here: read again below, past
  // L1.) 8 units of 9830 slots behind a decode step: 14.9 us for both without, 14.1 with one group per warp, 14.2 with two, 15.0
  // with three, which the copy engine has not worked off when the wait returns.
  if (NW == 8 && lane == 0) {
    const int rows = min(min(__ldcg(a.ca.fill + unit), cfg.max_budget) - first, GRP);
    const size_t at = ((size_t)unit * cfg.max_budget + first) * D * 2;
    if (rows > 0) {
      l2_prefetch_bulk(static_cast<const char*>(a.ca.k_cache) + at, (uint32_t)rows * D * 2);
      l2_prefetch_bulk(static_cast<const char*>(a.ca.v_cache) + at, (uint32_t)rows * D * 2);
    }
  }
  griddep_wait();
  const int fill = __ldcg(a.ca.fill + unit);
  const int items = first < fill ? 2 * ((fill - first + stride - 1) / stride) : 0;
  const int row_base = unit * cfg.max_budget;
  // Item t (K rows of group t / 2, or its V rows) into buffer b.
  auto issue = [&](int t, int b) {
    if (t < items && lane == 0) {
      const int row = row_base + first + (t >> 1) * stride;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + b * Ring::kItemBytes);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(b)), "r"((uint32_t)Ring::kItemBytes) : "memory");
#pragma unroll
      for (int h = 0; h < NH; ++h)
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst + h * GRP * 128),
            "l"(reinterpret_cast<uint64_t>((t & 1) ? &vmap : &kmap)), "r"(h * 64), "r"(row), "r"(full(b))
            : "memory");
    }
  };
#pragma unroll
  for (int t = 0; t < NBUF - 1; ++t) issue(t, t);

  uint32_t qf[2 * NC][2];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    uint4 t = make_uint4(0u, 0u, 0u, 0u);
    if (gid < G) t = static_cast<const uint4*>(a.q)[((size_t)unit * G + gid) * CPR + 2 * tig + (c & 1) + 8 * (c >> 1)];
    qf[2 * c][0] = t.x, qf[2 * c][1] = t.y, qf[2 * c + 1][0] = t.z, qf[2 * c + 1][1] = t.w;
  }
  const float scale = rsqrtf((float)d) * kLog2e;
  float m = -INFINITY, l = 0.f;
  float o[8 * NH][4];
#pragma unroll
  for (int t = 0; t < 8 * NH; ++t) o[t][0] = o[t][1] = o[t][2] = o[t][3] = 0.f;
  int buf = 0;
  uint32_t phase = 0;
  bool ok = true;
  // the next item has landed; its predecessor's buffer, read by the whole warp, takes the item NBUF - 1 ahead
  auto step = [&](int t) -> const uint4* {
    bool got = false;
    for (uint32_t i = 0; ok && i < kAttendSpinLimit && !got; ++i) {
      uint32_t done;
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(done)
          : "r"(full(buf)), "r"(phase)
          : "memory");
      got = done != 0;
    }
    ok = __all_sync(0xFFFFFFFFu, got);
    if (ok) issue(t + NBUF - 1, buf == 0 ? NBUF - 1 : buf - 1);
    const uint4* p = reinterpret_cast<const uint4*>(ring + buf * Ring::kItemBytes);
    if (++buf == NBUF) buf = 0, phase ^= 1u;
    return p;
  };
  for (int t = 0; t < items && ok; t += 2) {
    const int g0 = first + (t >> 1) * stride;
    // scores of slots g0 + 8 i + (0..7): two accumulators each (the chunks' two halves), so no chain is longer than NC
    float sa[4][4], sb[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) sa[i][e] = sb[i][e] = 0.f;
    {
      const uint4* kr = step(t) + gid * 8;
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // (row 8 i + gid of the half of the channels that holds chunk c)
          const uint4 kv = kr[(c >> 1) * GRP * 8 + i * 64 + ((2 * tig + (c & 1)) ^ gid)];
          mma_bf16_m16n8k16(sa[i], qf[2 * c][0], 0u, qf[2 * c][1], 0u, kv.x, kv.y);
          mma_bf16_m16n8k16(sb[i], qf[2 * c + 1][0], 0u, qf[2 * c + 1][1], 0u, kv.z, kv.w);
        }
    }
    // This lane: head gid, slots g0 + 8 i + 2 tig, + 1.
    float x[8];
    float gm = -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        x[2 * i + e] = g0 + 8 * i + 2 * tig + e < fill ? (sa[i][e] + sb[i][e]) * scale : -INFINITY;
        gm = fmaxf(gm, x[2 * i + e]);
      }
    gm = fmaxf(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, 1));
    gm = fmaxf(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, 2));  // finite: slot g0 is valid
    const float mn = fmaxf(m, gm);
    const float corr = exp2f(m - mn);
    float p[8], ps = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = exp2f(x[k] - mn);
#pragma unroll
    for (int k = 0; k < 8; k += 2) ps += p[k] + p[k + 1];
    l = l * corr + ps;
    m = mn;
    uint32_t w[4][2];  // hi and lo halves of the weights of slots 8 i + 2 tig, + 1
#pragma unroll
    for (int i = 0; i < 4; ++i) split_pair(p[2 * i], p[2 * i + 1], w[i][0], w[i][1]);
    if (__any_sync(0xFFFFFFFFu, corr != 1.f)) {
#pragma unroll
      for (int t2 = 0; t2 < 8 * NH; ++t2) o[t2][0] *= corr, o[t2][1] *= corr, o[t2][2] *= corr, o[t2][3] *= corr;
    }
    const uint4* vr = step(t + 1);
    if (g0 + GRP > fill) {  // rows past the fill level (weighted by zero) hold anything: make them finite
      for (int i = lane; i < GRP * CPR; i += 32)
        if (g0 + ((i >> 3) & (GRP - 1)) >= fill) const_cast<uint4*>(vr)[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf)  // 16 slots per MMA
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        uint4 vb[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int row = 16 * hf + 2 * tig + (s & 1) + 8 * (s >> 1);
          vb[s] = vr[h * GRP * 8 + row * 8 + (gid ^ (row & 7))];
        }
        const uint32_t w0[4] = {vb[0].x, vb[0].y, vb[0].z, vb[0].w};
        const uint32_t w1[4] = {vb[1].x, vb[1].y, vb[1].z, vb[1].w};
        const uint32_t w2[4] = {vb[2].x, vb[2].y, vb[2].z, vb[2].w};
        const uint32_t w3[4] = {vb[3].x, vb[3].y, vb[3].z, vb[3].w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t sel = (e & 1) ? 0x7632u : 0x5410u;
          const uint32_t b0 = __byte_perm(w0[e >> 1], w1[e >> 1], sel);
          const uint32_t b1 = __byte_perm(w2[e >> 1], w3[e >> 1], sel);
          mma_bf16_m16n8k16(o[8 * h + e], w[2 * hf][0], w[2 * hf][1], w[2 * hf + 1][0], w[2 * hf + 1][1], b0, b1);
        }
      }
  }
  if (!ok) {  // gave up on a copy: count it, and let what is in flight land (bounded) before the rings are reused
    if (lane == 0) {
      atomicAdd(&g_tc_error, 1);
      for (int b = 0; b < NBUF; ++b)
        for (uint32_t i = 0; i < kAttendSpinLimit; ++i) {
          uint32_t done;
          asm volatile(
              "{\n\t.reg .pred p;\n\t"
              "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
              "selp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(done)
              : "r"(full(b)), "r"(b < buf ? phase : phase ^ 1u)
              : "memory");
          if (done) break;
        }
    }
    __syncwarp();
  }
  __syncthreads();  // the rings give way to the partial results
  // Per-warp partial result. l is summed over the quad (m and corr were equal across it).
  l += __shfl_xor_sync(0xFFFFFFFFu, l, 1);
  l += __shfl_xor_sync(0xFFFFFFFFu, l, 2);
  if (gid < G) {
    if (tig == 0) part_ml[(warp * G + gid) * 2] = m, part_ml[(warp * G + gid) * 2 + 1] = l;
#pragma unroll
    for (int t = 0; t < 8 * NH; ++t) {
      const int h = t >> 3, e = t & 7;
      part_o[(warp * G + gid) * d + (2 * tig + 8 * h) * 8 + e] = o[t][0] + o[t][2];
      part_o[(warp * G + gid) * d + (2 * tig + 1 + 8 * h) * 8 + e] = o[t][1] + o[t][3];
    }
  }
  __syncthreads();
  if (S == 1) {
    attend_merge<NW>(part_ml, part_o, G, d, a.out + (size_t)unit * G * d);
    return;
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  attend_merge_cluster<NW>(part_ml, part_o, gather, bar, G, d, S, rank, a.out + (size_t)unit * G * d);
}

// ------------------------------------------------------------------------------------------------ generic

__global__ void __launch_bounds__(kAttendThreads) attend_generic_kernel(const AttendArgs a) {
  extern __shared__ __align__(16) float asm_[];  // q as fp32 [G][d], then part_ml [warps][G][2], part_o [warps][G][d]
  const he_config& cfg = a.cfg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = blockIdx.y * cfg.n_kv_heads + blockIdx.x;
  const int d = cfg.head_dim, G = cfg.group_size, es = esize_of(cfg.dtype);
  const int fill = a.ca.fill[unit];
  float* qs = asm_;
  float* part_ml = qs + G * d;
  float* part_o = part_ml + kAttendWarps * G * 2;
  const int cpr = d * es / 16;
  for (int idx = tid; idx < G * cpr; idx += kAttendThreads)
    stage_chunk(qs + (idx / cpr) * d, static_cast<const char*>(a.q) + ((size_t)unit * G + idx / cpr) * d * es, idx % cpr, cfg.dtype);
  __syncthreads();
  const float scale = rsqrtf((float)d) * kLog2e;
  const char* Kb = static_cast<const char*>(a.ca.k_cache) + (size_t)unit * cfg.max_budget * d * es;
  const char* Vb = static_cast<const char*>(a.ca.v_cache) + (size_t)unit * cfg.max_budget * d * es;
  const int per = d / 32 + (d % 32 ? 1 : 0);  // channels per lane (<= 8): c = lane + 32 * i
  float m[kMaxGroup], l[kMaxGroup], o[kMaxGroup][kMaxDim / 32];
#pragma unroll
  for (int g = 0; g < kMaxGroup; ++g) {
    m[g] = -INFINITY;
    l[g] = 0.f;
#pragma unroll
    for (int i = 0; i < kMaxDim / 32; ++i) o[g][i] = 0.f;
  }
  auto elem = [&](const char* row, int c) -> float {
    return cfg.dtype == HE_DTYPE_BF16 ? bf16_bits_to_f32(reinterpret_cast<const uint16_t*>(row)[c])
                                      : reinterpret_cast<const float*>(row)[c];
  };
  for (int j = warp; j < fill; j += kAttendWarps) {
    const char* kr = Kb + (size_t)j * d * es;
    const char* vr = Vb + (size_t)j * d * es;
    float kv[kMaxDim / 32], vv[kMaxDim / 32];
#pragma unroll
    for (int i = 0; i < kMaxDim / 32; ++i) {
      const int c = lane + 32 * i;
      kv[i] = (i < per && c < d) ? elem(kr, c) : 0.f;
      vv[i] = (i < per && c < d) ? elem(vr, c) : 0.f;
    }
#pragma unroll
    for (int g = 0; g < kMaxGroup; ++g) {
      if (g < G) {
        float dot = 0.f;
#pragma unroll
        for (int i = 0; i < kMaxDim / 32; ++i) {
          const int c = lane + 32 * i;
          if (i < per && c < d) dot = fmaf(qs[g * d + c], kv[i], dot);
        }
        for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, off);
        const float sc = dot * scale;
        const float mn = fmaxf(m[g], sc);
        const float corr = exp2f(m[g] - mn), p = exp2f(sc - mn);  // exp2f(-inf) = 0 on the first slot
        l[g] = l[g] * corr + p;
#pragma unroll
        for (int i = 0; i < kMaxDim / 32; ++i) o[g][i] = o[g][i] * corr + p * vv[i];
        m[g] = mn;
      }
    }
  }
#pragma unroll
  for (int g = 0; g < kMaxGroup; ++g) {
    if (g < G) {
      if (lane == 0) {
        part_ml[(warp * G + g) * 2] = m[g];
        part_ml[(warp * G + g) * 2 + 1] = l[g];
      }
#pragma unroll
      for (int i = 0; i < kMaxDim / 32; ++i) {
        const int c = lane + 32 * i;
        if (i < per && c < d) part_o[(warp * G + g) * d + c] = o[g][i];
      }
    }
  }
  __syncthreads();
  attend_merge<kAttendWarps>(part_ml, part_o, G, d, a.out + (size_t)unit * G * d);
}

// ------------------------------------------------------------------------------------------------ attention loss
//
// he_attention_loss (Section 4.6 / Appendix B): 1 - the attention mass of the cached tokens, for each query head, under
// softmax(q . k_p / sqrt(d)) over ALL n = next_pos tokens seen so far. The dropped mass is summed directly (a token
// is dropped when no valid slot holds its position: a bitmap in shared memory), so a small loss is not the
// difference of two numbers close to one. One CTA per unit, a warp per token, online maximum as in he_attend.
struct LossArgs {
  he_config cfg;
  he_cache ca;
  const void* q;       // [B, Hkv*G, d]
  const void* k_full;  // strided [B, Hkv, n, d]
  long long s0, s1, s2;
  float* out;          // [B, Hkv*G]
};

__global__ void __launch_bounds__(kAttendThreads) attention_loss_kernel(const LossArgs a) {
  extern __shared__ __align__(16) float lsm_[];  // q as fp32 [G][d], partials [warps][G][3], bitmap of cached positions
  const he_config& cfg = a.cfg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long unit = (long long)blockIdx.y * cfg.n_kv_heads + blockIdx.x;
  const int d = cfg.head_dim, G = cfg.group_size, es = esize_of(cfg.dtype);
  const int n = a.ca.next_pos[unit], fill = a.ca.fill[unit];
  float* qs = lsm_;
  float* part = qs + G * d;
  uint32_t* kept = reinterpret_cast<uint32_t*>(part + kAttendWarps * G * 3);
  const int cpr = d * es / 16;
  for (int idx = tid; idx < G * cpr; idx += kAttendThreads)
    stage_chunk(qs + (idx / cpr) * d, static_cast<const char*>(a.q) + (unit * G + idx / cpr) * d * es, idx % cpr, cfg.dtype);
  for (int i = tid; i < (n + 31) / 32; i += kAttendThreads) kept[i] = 0u;
  __syncthreads();
  for (int j = tid; j < fill; j += kAttendThreads) {
    const int p = a.ca.pos[unit * cfg.max_budget + j];
    if (p >= 0 && p < n) atomicOr(&kept[p >> 5], 1u << (p & 31));
  }
  __syncthreads();
  const float scale = rsqrtf((float)d) * kLog2e;
  const char* Kb = static_cast<const char*>(a.k_full) + ((long long)blockIdx.y * a.s0 + (long long)blockIdx.x * a.s1) * es;
  float m[kMaxGroup], lall[kMaxGroup], ldrop[kMaxGroup];
#pragma unroll
  for (int g = 0; g < kMaxGroup; ++g) m[g] = -INFINITY, lall[g] = 0.f, ldrop[g] = 0.f;
  const int per = (d + 31) / 32;
  for (int p = warp; p < n; p += kAttendWarps) {
    const char* kr = Kb + (long long)p * a.s2 * es;
    float kv[kMaxDim / 32];
#pragma unroll
    for (int i = 0; i < kMaxDim / 32; ++i) {
      const int c = lane + 32 * i;
      kv[i] = (i < per && c < d) ? (cfg.dtype == HE_DTYPE_BF16 ? bf16_bits_to_f32(reinterpret_cast<const uint16_t*>(kr)[c])
                                                                : reinterpret_cast<const float*>(kr)[c])
                                 : 0.f;
    }
    const bool dropped = ((kept[p >> 5] >> (p & 31)) & 1u) == 0u;
#pragma unroll
    for (int g = 0; g < kMaxGroup; ++g) {
      if (g < G) {
        float dot = 0.f;
#pragma unroll
        for (int i = 0; i < kMaxDim / 32; ++i) {
          const int c = lane + 32 * i;
          if (i < per && c < d) dot = fmaf(qs[g * d + c], kv[i], dot);
        }
        for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, off);
        const float sc = dot * scale;
        const float mn = fmaxf(m[g], sc);
        const float corr = exp2f(m[g] - mn), w = exp2f(sc - mn);
        lall[g] = lall[g] * corr + w;
        ldrop[g] = ldrop[g] * corr + (dropped ? w : 0.f);
        m[g] = mn;
      }
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int g = 0; g < kMaxGroup; ++g)
      if (g < G) {
        part[(warp * G + g) * 3] = m[g];
        part[(warp * G + g) * 3 + 1] = lall[g];
        part[(warp * G + g) * 3 + 2] = ldrop[g];
      }
  }
  __syncthreads();
  if (tid < G) {
    float M = -INFINITY;
    for (int w = 0; w < kAttendWarps; ++w) M = fmaxf(M, part[(w * G + tid) * 3]);
    float A = 0.f, D = 0.f;
    for (int w = 0; w < kAttendWarps; ++w) {
      const float mw = part[(w * G + tid) * 3];
      const float f = mw == -INFINITY ? 0.f : exp2f(mw - M);
      A += part[(w * G + tid) * 3 + 1] * f;
      D += part[(w * G + tid) * 3 + 2] * f;
    }
    a.out[unit * G + tid] = A > 0.f ? D / A : 0.f;
  }
}

// The same for bf16 keys with d = 128 and G <= 8: scores of 16 tokens at a time as warp-level MMAs fed straight from
// 16-byte global loads (the fragment scheme of attend_bf16_kernel), next group's rows requested before the current
// group's arithmetic. Dynamic shared memory: partials [warps][G][3] floats, then the bitmap of cached positions.
__global__ void __launch_bounds__(kAttendThreads) attention_loss_bf16_kernel(const LossArgs a) {
  extern __shared__ __align__(16) float lsm_[];
  constexpr int d = 128;
  const he_config& cfg = a.cfg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
  const long long unit = (long long)blockIdx.y * cfg.n_kv_heads + blockIdx.x;
  const int G = cfg.group_size;
  const int n = a.ca.next_pos[unit], fill = a.ca.fill[unit];
  float* part = lsm_;
  uint32_t* kept = reinterpret_cast<uint32_t*>(part + kAttendWarps * G * 3);
  for (int i = tid; i < (n + 31) / 32; i += kAttendThreads) kept[i] = 0u;
  __syncthreads();
  for (int j = tid; j < fill; j += kAttendThreads) {
    const int p = a.ca.pos[unit * cfg.max_budget + j];
    if (p >= 0 && p < n) atomicOr(&kept[p >> 5], 1u << (p & 31));
  }
  __syncthreads();
  uint32_t qf[8][2];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint4 t = make_uint4(0u, 0u, 0u, 0u);
    if (gid < G) t = static_cast<const uint4*>(a.q)[(unit * G + gid) * (d / 8) + tig + 4 * c];
    qf[2 * c][0] = t.x, qf[2 * c][1] = t.y, qf[2 * c + 1][0] = t.z, qf[2 * c + 1][1] = t.w;
  }
  const float scale = rsqrtf((float)d) * kLog2e;
  const char* Kb = static_cast<const char*>(a.k_full) + ((long long)blockIdx.y * a.s0 + (long long)blockIdx.x * a.s1) * 2;
  const int last = n - 1;
  auto load_k = [&](int g0, uint4 (&kb)[2][4]) {  // rows past the end repeat the last row and are weighted by zero
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const uint4* row = reinterpret_cast<const uint4*>(Kb + (long long)min(g0 + gid + 8 * r, last) * a.s2 * 2);
#pragma unroll
      for (int c = 0; c < 4; ++c) kb[r][c] = ldg_stream16(row + tig + 4 * c);
    }
  };
  float m = -INFINITY, lall = 0.f, ldrop = 0.f;
  uint4 kc[2][4], kn[2][4];
  const int stride = 16 * kAttendWarps;
  int g0 = 16 * warp;
  if (g0 < n) load_k(g0, kc);
  for (; g0 < n; g0 += stride) {
    const bool more = g0 + stride < n;
    if (more) load_k(g0 + stride, kn);
    float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      mma_bf16_m16n8k16(s0, qf[2 * c][0], 0u, qf[2 * c][1], 0u, kc[0][c].x, kc[0][c].y);
      mma_bf16_m16n8k16(s1, qf[2 * c][0], 0u, qf[2 * c][1], 0u, kc[1][c].x, kc[1][c].y);
      mma_bf16_m16n8k16(s0, qf[2 * c + 1][0], 0u, qf[2 * c + 1][1], 0u, kc[0][c].z, kc[0][c].w);
      mma_bf16_m16n8k16(s1, qf[2 * c + 1][0], 0u, qf[2 * c + 1][1], 0u, kc[1][c].z, kc[1][c].w);
    }
    // this lane: head gid, tokens g0 + 2tig, + 1, + 8, + 9
    const int j = g0 + 2 * tig;
    const int tok[4] = {j, j + 1, j + 8, j + 9};
    const float sc[4] = {s0[0], s0[1], s1[0], s1[1]};
    float x[4];
    bool dropped[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      x[e] = tok[e] < n ? sc[e] * scale : -INFINITY;
      dropped[e] = tok[e] < n && ((kept[tok[e] >> 5] >> (tok[e] & 31)) & 1u) == 0u;
    }
    float gm = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
    gm = fmaxf(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, 1));
    gm = fmaxf(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, 2));  // finite: token g0 exists
    const float mn = fmaxf(m, gm);
    const float corr = exp2f(m - mn);
    float wa = 0.f, wd = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float w = exp2f(x[e] - mn);
      wa += w;
      wd += dropped[e] ? w : 0.f;
    }
    lall = lall * corr + wa;
    ldrop = ldrop * corr + wd;
    m = mn;
    if (more) {
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) kc[r][c] = kn[r][c];
    }
  }
  lall += __shfl_xor_sync(0xFFFFFFFFu, lall, 1);
  lall += __shfl_xor_sync(0xFFFFFFFFu, lall, 2);
  ldrop += __shfl_xor_sync(0xFFFFFFFFu, ldrop, 1);
  ldrop += __shfl_xor_sync(0xFFFFFFFFu, ldrop, 2);
  if (gid < G && tig == 0) {
    part[(warp * G + gid) * 3] = m;
    part[(warp * G + gid) * 3 + 1] = lall;
    part[(warp * G + gid) * 3 + 2] = ldrop;
  }
  __syncthreads();
  if (tid < G) {
    float M = -INFINITY;
    for (int w = 0; w < kAttendWarps; ++w) M = fmaxf(M, part[(w * G + tid) * 3]);
    float A = 0.f, D = 0.f;
    for (int w = 0; w < kAttendWarps; ++w) {
      const float mw = part[(w * G + tid) * 3];
      const float f = mw == -INFINITY ? 0.f : exp2f(mw - M);
      A += part[(w * G + tid) * 3 + 1] * f;
      D += part[(w * G + tid) * 3 + 2] * f;
    }
    a.out[unit * G + tid] = A > 0.f ? D / A : 0.f;
  }
}

}  // namespace he
