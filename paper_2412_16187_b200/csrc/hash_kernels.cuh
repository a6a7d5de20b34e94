// he_hash_keys and phase 1 of he_prefill_compress: Eq. 2 on many rows with CUDA-core fp32 FMAs.
// A CTA stages W (zero-padded to 32 or 64 columns) and a tile of 128 rows in shared memory as fp32; a warp owns 32 rows, a lane
// a block of 8 rows x 4 bits of every code word (16 shared-memory reads for 256 FMAs with two words). fp32 rows and a dense W are
// staged with cp.async, all of it in flight at once: staged through registers, a few loads at a time, the tile's latency
// bound the kernel (39 000 cycles per tile where its FMAs need 8200).
#pragma once
#include "common.cuh"

namespace he {

constexpr int kHashThreads = 128;
constexpr int kHashRows = 128;  // rows per CTA
constexpr int kHashRpw = 32;    // rows per warp
constexpr int kHashRpl = 8;     // rows per lane
constexpr int kHashPad = 4;     // floats between staged rows: neighbouring rows start on other banks

struct HashJob {
  const void* x;
  const float* W;
  uint32_t* out;
  int mode;  // 0: flat rows; 1: prompt keys; 2: prompt queries
  int dtype, d, b;
  long long rows, row_stride;  // mode 0
  const void* x2;              // mode 0, tensor-core kernel only: a second range of rows2 rows with the same stride, hashed by
  long long rows2;             //   the same launch; its codes follow the first range's in `out`
  long long s0, s1, s2;        // modes 1, 2: element strides (batch, head, token)
  int heads, G, Hkv;           // heads = heads per sequence of this tensor
  long long Nmax;
  const int32_t* prompt_len;
  const int32_t* budget;
  int q_all;            // mode 2: hash the queries of every prompt token, not only of those that evict
  const void* w_image;  // optional: the tensor-core kernel's shared-memory image of W's three bf16 terms (build_w_image_kernel)
};

// Segments below `segs` are job1's, the others job2's (a prompt's key rows and query rows in one launch).
template <int WORDS>
__global__ void __launch_bounds__(kHashThreads) hash_rows_kernel(const __grid_constant__ HashJob job1, const __grid_constant__ HashJob job2, int segs) {
  griddep_launch_dependents();
  const bool first_job = (int)blockIdx.y < segs;
  const HashJob& job = first_job ? job1 : job2;
  extern __shared__ __align__(16) float hsm[];
  constexpr int BP = 32 * WORDS;
  const int d = job.d, b = job.b, es = esize_of(job.dtype);
  float* Ws = hsm;            // [d][BP]
  float* xs = hsm + d * BP;   // [kHashRows][d + kHashPad]
  const int xp = d + kHashPad;

  // which rows does this CTA hash, and where do the codes go
  const char* base;
  long long stride, r_begin, r_end, out_base, out_stride;
  if (job.mode == 0) {
    base = static_cast<const char*>(job.x);
    stride = job.row_stride;
    r_begin = 0;
    r_end = job.rows;
    out_base = 0;
    out_stride = WORDS;
  } else {
    const int seg = first_job ? blockIdx.y : blockIdx.y - segs;
    const int s = seg / job.heads, hh = seg % job.heads;
    const long long C = max(job.budget[s], 0);
    const long long N = clamp_len(job.prompt_len[s], job.Nmax, (int)min(C, 1LL));
    base = static_cast<const char*>(job.x) + (s * job.s0 + hh * job.s1) * es;
    stride = job.s2;
    r_end = N;
    if (job.mode == 1) {
      r_begin = 0;
      out_base = ((long long)s * job.Hkv + hh) * job.Nmax * WORDS;
      out_stride = WORDS;
    } else {
      r_begin = job.q_all ? 0 : (C < N ? C : N);  // queries of appended tokens are never read by Algorithm 1
      const long long unit = (long long)s * job.Hkv + hh / job.G;
      out_base = (unit * job.Nmax * job.G + hh % job.G) * WORDS;
      out_stride = (long long)job.G * WORDS;
    }
  }
  const long long row0 = r_begin + (long long)blockIdx.x * kHashRows;
  if (row0 >= r_end) return;
  const int nrows = (int)((r_end - row0) < kHashRows ? (r_end - row0) : kHashRows);

  if (b == BP && (reinterpret_cast<uintptr_t>(job.W) & 15u) == 0) {
    for (int idx = threadIdx.x; idx < d * BP / 4; idx += kHashThreads) cp_async16(Ws + 4 * idx, job.W + 4 * idx);
  } else {
#pragma unroll 8
    for (int idx = threadIdx.x; idx < d * BP; idx += kHashThreads) {
      const int c = idx / BP, i = idx % BP;
      Ws[idx] = i < b ? __ldg(job.W + (long long)c * b + i) : 0.f;
    }
  }
  const int cpr = d * es / 16;  // 16-byte chunks per row
#pragma unroll 4
  for (int idx = threadIdx.x; idx < kHashRows * cpr; idx += kHashThreads) {
    const int r = idx / cpr, ch = idx - r * cpr;
    // rows past the end repeat the last one; their codes are not stored
    const char* src = base + (row0 + min(r, nrows - 1)) * stride * es;
    if (job.dtype == HE_DTYPE_F32) cp_async16(xs + r * xp + ch * 4, src + ch * 16);
    else stage_chunk(xs + r * xp, src, ch, HE_DTYPE_BF16);
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();

  // lane (rg, bg): rows rg, rg + 4, ... of the warp's 32, bits 4 bg .. 4 bg + 3 of every code word
  constexpr int BPL = 4 * WORDS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, bg = lane & 7, rg = lane >> 3;
  const float* xw = xs + (warp * kHashRpw + rg) * xp;
  const float* ww = Ws + bg * 4;
  float tot[kHashRpl][BPL];
#pragma unroll
  for (int r = 0; r < kHashRpl; ++r)
#pragma unroll
    for (int k = 0; k < BPL; ++k) tot[r][k] = 0.f;

  for (int c0 = 0; c0 < d; c0 += kChunk) {
    float acc[kHashRpl][BPL];
#pragma unroll
    for (int r = 0; r < kHashRpl; ++r)
#pragma unroll
      for (int k = 0; k < BPL; ++k) acc[r][k] = 0.f;
    const int cend = (d - c0) < kChunk ? (d - c0) : kChunk;
#pragma unroll 1
    for (int cc = 0; cc < cend; cc += 4) {
      float4 xv[kHashRpl];
#pragma unroll
      for (int r = 0; r < kHashRpl; ++r) xv[r] = *reinterpret_cast<const float4*>(xw + r * 4 * xp + c0 + cc);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float wv[BPL];
#pragma unroll
        for (int w = 0; w < WORDS; ++w) {
          const float4 w4 = *reinterpret_cast<const float4*>(ww + (c0 + cc + c) * BP + 32 * w);
          wv[4 * w] = w4.x, wv[4 * w + 1] = w4.y, wv[4 * w + 2] = w4.z, wv[4 * w + 3] = w4.w;
        }
#pragma unroll
        for (int r = 0; r < kHashRpl; ++r) {
          const float x = c == 0 ? xv[r].x : (c == 1 ? xv[r].y : (c == 2 ? xv[r].z : xv[r].w));
#pragma unroll
          for (int k = 0; k < BPL; ++k) acc[r][k] = fmaf(x, wv[k], acc[r][k]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kHashRpl; ++r)
#pragma unroll
      for (int k = 0; k < BPL; ++k) tot[r][k] += acc[r][k];
  }

  // a lane's four bits of a word, then the eight lanes of the row together
#pragma unroll
  for (int r = 0; r < kHashRpl; ++r) {
    const int row = warp * kHashRpw + r * 4 + rg;
#pragma unroll
    for (int w = 0; w < WORDS; ++w) {
      uint32_t word = 0u;
#pragma unroll
      for (int k = 0; k < 4; ++k) word |= (tot[r][4 * w + k] >= 0.f ? 1u : 0u) << k;
      word <<= 4 * bg;
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 1);
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 2);
      word |= __shfl_xor_sync(0xFFFFFFFFu, word, 4);
      if (bg == 0 && row < nrows) job.out[out_base + (row0 + row) * out_stride + w] = word & word_mask(b, w);
    }
  }
}

}  // namespace he
