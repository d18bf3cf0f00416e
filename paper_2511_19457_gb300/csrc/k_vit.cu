// Vision-transformer operators (the attention-based models of Sec. 6, Table 2:
// ViT-B16): layer normalisation, multi-head self-attention, the token sequence
// of a patch embedding, and token selection.  The token-wise linear layers of
// a transformer are 1x1 convolutions over [N, 1, T, C] and run on the
// threshold-dispatched GEMM path; these kernels are the rest.  Layer norm (rows
// of up to 1024 values) and attention emit their outputs' Eq. 1 statistics; the
// others' are measured by the stats kernel afterwards.
#include "sparoa_kernels.h"

namespace sparoa {

namespace {

constexpr int kVitThreads = 256;

// ---------------------------------------------------------------------------
// Layer normalisation: one warp per row of C values (C % 8 == 0), fp32: the
// mean, then the mean square of the deviations.
//
// Rows of up to 1024 values (ln_rows_kernel): a warp takes a run of consecutive
// rows; the row is held in registers (one pass over memory, the next row's
// loads in flight while this one is reduced) and so are the lane's gamma and
// beta, and the output's occupancy is emitted on the way: row bitmap words whole
// (one word per row), block-column masks ORed over the run's rows of a 128-row
// block, column counts in 16-bit register halves, added up in shared memory once
// per CTA.  [6304, 768]: 4.7 us, with occupancy and its clear 10.3 us (14.1 us and
// 9.5 us more for a clear and a statistics pass before: gamma and beta were
// re-read, value by value, for every row).  Rows of up to 256 values run two CTAs
// an SM ([87511, 64] 22 us, one CTA 36).  Longer rows than 1024 (layernorm_kernel)
// are re-read for each of the three steps, four loads in flight ([5091, 1312] 19 us;
// loads one at a time 32).
constexpr int kLnRegChunks = 4;     // 8-value chunks per lane held in registers
constexpr int kLnThreads = 512;     // at most: one CTA per SM, whose column counts reach global memory once
constexpr int kLnFlushRows = 16384;  // rows after which 16-bit counters are flushed

__device__ __forceinline__ void ln_store(__nv_bfloat16* __restrict__ yr, const float* __restrict__ gb, int C,
                                         int c, float (&f)[8], float mean, float rstd) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float v = (f[k] - mean) * rstd;
    if (gb) v = fmaf(v, gb[c * 8 + k], gb[C + c * 8 + k]);
    f[k] = v;
  }
  *reinterpret_cast<uint4*>(yr + c * 8) = pack8(f);
}

template <int NCH>
__global__ void __launch_bounds__(kLnThreads, NCH == 1 ? 2 : 1)
    ln_rows_kernel(const __nv_bfloat16* __restrict__ x, int64_t R, int C, const float* __restrict__ gb, int gb_vec,
                   float eps, __nv_bfloat16* __restrict__ y, OccDev o_param, int emit) {
  const OccDev o = o_param;
  __shared__ uint32_t s_cnt[NCH * 256];  // column 8 (32 i + lane) + k at (8 i + k) * 32 + lane
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
  const int64_t w = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int64_t r0 = w * R / warps, r1 = (w + 1) * R / warps;
  const int chunks = C / 8;
  const float inv_c = 1.f / (float)C;
  if (emit) {
    for (int c = threadIdx.x; c < NCH * 256; c += blockDim.x) s_cnt[c] = 0u;
    __syncthreads();  // a warp adds its counts as soon as its own rows are done
  }
  pdl_wait();
  pdl_trigger();
  uint4 u[NCH];
  auto load = [&](int64_t r) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const int c = lane + 32 * i;
      u[i] = c < chunks ? *reinterpret_cast<const uint4*>(x + r * C + c * 8) : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if (r0 < r1) load(r0);
  float gam[NCH][8], bet[NCH][8];
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = lane + 32 * i;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      gam[i][k] = 1.f;
      bet[i][k] = 0.f;
    }
    if (gb && c < chunks) {
      if (gb_vec) {
#pragma unroll
        for (int k = 0; k < 8; k += 4) {
          const float4 g4 = *reinterpret_cast<const float4*>(gb + c * 8 + k);
          const float4 b4 = *reinterpret_cast<const float4*>(gb + C + c * 8 + k);
          gam[i][k] = g4.x; gam[i][k + 1] = g4.y; gam[i][k + 2] = g4.z; gam[i][k + 3] = g4.w;
          bet[i][k] = b4.x; bet[i][k + 1] = b4.y; bet[i][k + 2] = b4.z; bet[i][k + 3] = b4.w;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          gam[i][k] = gb[c * 8 + k];
          bet[i][k] = gb[C + c * 8 + k];
        }
      }
    }
  }
  uint32_t cnt[NCH][4];  // non-zeros per column, 16-bit halves
  uint32_t blk[NCH];     // this lane's 8 columns of the current 128-row block
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    cnt[i][0] = cnt[i][1] = cnt[i][2] = cnt[i][3] = 0u;
    blk[i] = 0u;
  }
  auto flush_cnt = [&]() {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (cnt[i][k] & 0xFFFFu) atomicAdd(&s_cnt[(i * 8 + 2 * k) * 32 + lane], cnt[i][k] & 0xFFFFu);
        if (cnt[i][k] >> 16) atomicAdd(&s_cnt[(i * 8 + 2 * k + 1) * 32 + lane], cnt[i][k] >> 16);
        cnt[i][k] = 0u;
      }
    }
  };
  auto flush_blk = [&](int64_t b) {  // four lanes' masks are one 32-column word
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      uint32_t m = blk[i] << (8 * (lane & 3));
      m |= __shfl_xor_sync(0xffffffffu, m, 1);
      m |= __shfl_xor_sync(0xffffffffu, m, 2);
      if ((lane & 3) == 0 && m) atomicOr(&o.blk_mask[b * o.C32 + ((lane + 32 * i) >> 2)], m);
      blk[i] = 0u;
    }
  };
  int since = 0;
  for (int64_t r = r0; r < r1; ++r) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      float f[8];
      unpack8(u[i], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) s += f[k];
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    const float mean = s * inv_c;
    float q = 0.f;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      if (lane + 32 * i < chunks) {
        float f[8];
        unpack8(u[i], f);
#pragma unroll
        for (int k = 0; k < 8; ++k) q = fmaf(f[k] - mean, f[k] - mean, q);
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) q += __shfl_xor_sync(0xffffffffu, q, d);
    const float rstd = rsqrtf(q * inv_c + eps);
    unsigned long long rowbits = 0ull;
    uint4 v[NCH];
#pragma unroll
    for (int i = 0; i < NCH; ++i) v[i] = u[i];
    if (r + 1 < r1) load(r + 1);
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const int c = lane + 32 * i;
      uint32_t m8 = 0u;
      if (c < chunks) {
        float f[8];
        unpack8(v[i], f);
#pragma unroll
        for (int k = 0; k < 8; ++k) f[k] = fmaf((f[k] - mean) * rstd, gam[i][k], bet[i][k]);
        const uint4 out = pack8(f);
        *reinterpret_cast<uint4*>(y + r * C + c * 8) = out;
        if (emit) {
          const uint32_t n0 = nz_pairs(out.x), n1 = nz_pairs(out.y), n2 = nz_pairs(out.z), n3 = nz_pairs(out.w);
          cnt[i][0] += n0;
          cnt[i][1] += n1;
          cnt[i][2] += n2;
          cnt[i][3] += n3;
          const uint32_t t = n0 | (n1 << 2) | (n2 << 4) | (n3 << 6);  // even columns low, odd ones 16 up
          m8 = (t | (t >> 15)) & 0xFFu;
          blk[i] |= m8;
        }
      }
      if (emit) {
        // eight lanes' 64 columns are one bit of the row's word
        const uint32_t any = __ballot_sync(0xffffffffu, m8 != 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if ((any >> (8 * k)) & 0xFFu) rowbits |= 1ull << (4 * i + k);
      }
    }
    if (emit) {
      if (lane == 0) o.row_bm[r] = rowbits;  // (C <= 1024: one word per row)
      if (((r + 1) & 127) == 0 || r + 1 == r1) flush_blk(r >> 7);
      if (++since == kLnFlushRows) {
        flush_cnt();
        since = 0;
      }
    }
  }
  if (!emit) return;
  flush_cnt();
  __syncthreads();
  unsigned long long total = 0ull;
  for (int c0 = 0; c0 < C; c0 += blockDim.x) {  // (whole warps: a warp's 32 columns are half a tile)
    const int c = c0 + threadIdx.x;
    const uint32_t n = c < C ? s_cnt[((c >> 8) * 8 + (c & 7)) * 32 + ((c >> 3) & 31)] : 0u;
    if (n) atomicAdd(&o.col_nnz[c], n);
    const uint32_t sum = __reduce_add_sync(0xffffffffu, n);
    total += sum;
    if (lane == 0 && sum) atomicAdd(&o.tile_nnz[c >> 6], sum);
  }
  if (lane == 0 && total) atomicAdd(o.nnz, total);
}

__global__ void __launch_bounds__(kVitThreads) layernorm_kernel(const __nv_bfloat16* __restrict__ x,
                                                                int64_t R, int C,
                                                                const float* __restrict__ gb, float eps,
                                                                __nv_bfloat16* __restrict__ y) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kVitThreads / 32);
  const int chunks = C / 8;
  const float inv_c = 1.f / (float)C;
  for (int64_t r = (int64_t)blockIdx.x * (kVitThreads / 32) + (threadIdx.x >> 5); r < R; r += warps) {
    const __nv_bfloat16* xr = x + r * C;
    __nv_bfloat16* yr = y + r * C;
    uint4 u[4];
    auto load4 = [&](int c) {  // chunks c, c + 32, ...: four loads in flight, to the row's end
#pragma unroll
      for (int i = 0; i < 4; ++i)
        u[i] = c + 32 * i < chunks ? *reinterpret_cast<const uint4*>(xr + (c + 32 * i) * 8) : make_uint4(0u, 0u, 0u, 0u);
    };
    float s = 0.f;
    for (int c = lane; c < chunks; c += 128) {
      load4(c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float f[8];
        unpack8(u[i], f);
#pragma unroll
        for (int k = 0; k < 8; ++k) s += f[k];
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float mean = s * inv_c;
    float q = 0.f;
    for (int c = lane; c < chunks; c += 128) {
      load4(c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (c + 32 * i >= chunks) break;
        float f[8];
        unpack8(u[i], f);
#pragma unroll
        for (int k = 0; k < 8; ++k) q = fmaf(f[k] - mean, f[k] - mean, q);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    const float rstd = rsqrtf(q * inv_c + eps);
    for (int c = lane; c < chunks; c += 128) {
      load4(c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (c + 32 * i >= chunks) break;
        float f[8];
        unpack8(u[i], f);
        ln_store(yr, gb, C, c + 32 * i, f, mean, rstd);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Multi-head self-attention on the tensor cores (mma.sync m16n8k16, bf16 in,
// fp32 accumulate), flash-attention style.  Input rows (one per token) hold
// q | k | v, each heads x HD values.  A CTA of up to 7 warps takes some of the
// 16-query tiles of one (image, head) (attention_split): the head's K and V rows
// are copied once into shared memory by cp.async (row pitch HD + 8 elements, so
// the 8 rows of a fragment load fall in distinct banks; rows past T up to the next
// multiple of 16 zero-filled), then the warps take the tiles in turn, at most five
// each.  A warp walks the keys in blocks of 32: S = Q K^T
// (Q fragments in registers, K fragments by ldmatrix), an online softmax per
// query row (running maximum and sum, rescaling the output), and O += P V with P
// taken straight from the S accumulators (their layout is the A-operand layout
// of the next MMA) and the V fragments read by ldmatrix.trans from the row-major
// V.  Key tiles wholly at or past T are not computed.  O / sum is stored as bf16,
// and the output's occupancy is emitted from one non-zero bit per value: row
// bits by votes, block-column masks by warp OR, column counts by a transposition
// of the warp's 32 x 32 bits.
//
// Bound by latency: 14 warps an SM against chains of MMAs, shuffles and
// exponentials.  So a whole block of keys has no branches (the ones around each 8
// keys kept the MMAs of different keys from overlapping) and the first queries
// are loaded beside K and V.  Blocks of 32 keys rather than 64 fit 128 registers.
// (64-key blocks, with branches, occupancy by 64-bit masks and 16 counters a lane:
// [32,197,12x64] with occupancy 39 us, now 28; [8,512,12x64] 76 us, now 42.)
constexpr int kAttnWarps = 7;
constexpr int kAttnThreads = 32 * kAttnWarps;  // at most
constexpr int kAttnMaxT = 512;
constexpr int kAttnKB = 32;        // keys per block

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                               uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8x8 b16 matrices, transposed on the way: lanes 8i..8i+7 address the
// rows of matrix i, register i receives its fragment
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                              uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}

// the same without the transposition, and two matrices
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int HD>
__global__ void __launch_bounds__(kAttnThreads, 2)
    attention_kernel(const __nv_bfloat16* __restrict__ qkv, int T, int heads, __nv_bfloat16* __restrict__ y,
                     OccDev o_param, int emit) {
  const OccDev occ = o_param;
  __shared__ uint32_t s_cnt[HD];
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int KP = HD + 8;  // row pitch of K and V (elements)
  const int T16 = (T + 15) & ~15;
  __nv_bfloat16* sK = reinterpret_cast<__nv_bfloat16*>(smem);  // [T16][KP]
  __nv_bfloat16* sV = sK + (size_t)T16 * KP;                     // [T16][KP]
  const int n = blockIdx.x / heads, h = blockIdx.x - (blockIdx.x / heads) * heads;
  const int D = heads * HD, row3 = 3 * D;
  const __nv_bfloat16* base = qkv + (int64_t)n * T * row3;
  for (int c = threadIdx.x; c < HD; c += blockDim.x) s_cnt[c] = 0u;
  pdl_wait();
  pdl_trigger();
  // K and V rows of the head: 16-byte copies, all in flight at once; a thread
  // takes the same chunk of every (threads / chunks)-th row
  {
    const int c = (int)threadIdx.x % (HD / 8), step = (int)blockDim.x / (HD / 8);
    for (int t = (int)threadIdx.x / (HD / 8); t < T16; t += step) {
      const bool live = t < T;
      const __nv_bfloat16* src = base + (int64_t)(live ? t : 0) * row3 + h * HD + c * 8;
      cp_async_16(smem_u32(sK + t * KP + c * 8), src + D, live ? 16u : 0u);
      cp_async_16(smem_u32(sV + t * KP + c * 8), src + 2 * D, live ? 16u : 0u);
    }
  }
  cp_async_commit();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tq = lane & 3;
  const int qtn = (T + 15) >> 4;  // 16-query tiles
  const int per = (qtn + (int)gridDim.y - 1) / (int)gridDim.y;
  const int qt0 = (int)blockIdx.y * per + warp, qt_end = min(qtn, ((int)blockIdx.y + 1) * per);
  // Q fragments (A operand, rows g and g + 8, HD / 16 k-steps), zero past T
  uint32_t qa[HD / 16][4];
  auto load_q = [&](int q0) {
    const int r0 = q0 + g, r1 = q0 + g + 8;
    const __nv_bfloat16* p0 = base + (int64_t)(r0 < T ? r0 : 0) * row3 + h * HD;
    const __nv_bfloat16* p1 = base + (int64_t)(r1 < T ? r1 : 0) * row3 + h * HD;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) {
      const int c = kk * 16 + 2 * tq;
      qa[kk][0] = r0 < T ? *reinterpret_cast<const uint32_t*>(p0 + c) : 0u;
      qa[kk][1] = r1 < T ? *reinterpret_cast<const uint32_t*>(p1 + c) : 0u;
      qa[kk][2] = r0 < T ? *reinterpret_cast<const uint32_t*>(p0 + c + 8) : 0u;
      qa[kk][3] = r1 < T ? *reinterpret_cast<const uint32_t*>(p1 + c + 8) : 0u;
    }
  };
  if (qt0 < qt_end) load_q(qt0 * 16);  // the first tile's queries arrive beside K and V
  cp_async_wait<0>();
  __syncthreads();
  const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;  // 1/sqrt(HD) * log2(e)
  // ldmatrix.trans lane address within a (16 keys x 16 dimensions) V block:
  // matrices (keys 0-7, dims 0-7), (keys 8-15, dims 0-7), (keys 0-7, dims
  // 8-15), (keys 8-15, dims 8-15) -> b0, b1 of one 8-dimension n-tile, then
  // b0, b1 of the next
  const uint32_t v_lane = smem_u32(sV) + (uint32_t)(((lane & 15) * KP + (lane >> 4) * 8) * 2);
  // K fragments of 8 keys: matrices (dims 0-7, 8-15) of one k-step, then of the next
  const uint32_t k_lane = smem_u32(sK) + (uint32_t)(((lane & 7) * KP + (lane >> 3) * 8) * 2);
  uint32_t cnt = 0u;  // byte i: non-zeros of column 8 (lane & 7) + 2 i + (lane >> 4) in the rows of half (lane >> 3) & 1
  for (int qt = qt0; qt < qt_end; qt += (int)blockDim.x / 32) {
    const int q0 = qt * 16;
    if (qt != qt0) load_q(q0);
    float o[HD / 8][4];
#pragma unroll
    for (int j = 0; j < HD / 8; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
    float m0 = -3.0e38f, m1 = -3.0e38f, l0 = 0.f, l1 = 0.f;  // rows g, g + 8
    // one block of keys; all of its keys are below T if FULL, so that nothing in it
    // branches and the MMAs of independent key tiles overlap
    auto block = [&](auto full, int kb) {
      constexpr bool FULL = decltype(full)::value;
      // S = Q K^T, n-tiles of 8 keys
      float s[kAttnKB / 8][4];
#pragma unroll
      for (int nt = 0; nt < kAttnKB / 8; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
      constexpr int G = FULL ? 4 : 1;  // n-tiles at a time
#pragma unroll
      for (int n0 = 0; n0 < kAttnKB / 8; n0 += G) {
        if (FULL || kb + n0 * 8 < T) {  // uniform across the warp
          const uint32_t ka = k_lane + (uint32_t)((kb + n0 * 8) * KP * 2);
          if constexpr (HD >= 32) {
#pragma unroll
            for (int kk = 0; kk < HD / 16; kk += 2) {
              uint32_t b[G][4];
#pragma unroll
              for (int i = 0; i < G; ++i)
                ldsm_x4(ka + (uint32_t)(i * 8 * KP * 2 + kk * 32), b[i][0], b[i][1], b[i][2], b[i][3]);
#pragma unroll
              for (int i = 0; i < G; ++i) mma_bf16_16816(s[n0 + i], qa[kk], b[i][0], b[i][1]);
#pragma unroll
              for (int i = 0; i < G; ++i) mma_bf16_16816(s[n0 + i], qa[kk + 1], b[i][2], b[i][3]);
            }
          } else {
#pragma unroll
            for (int i = 0; i < G; ++i) {
              uint32_t b0, b1;
              ldsm_x2(ka + (uint32_t)(i * 8 * KP * 2), b0, b1);
              mma_bf16_16816(s[n0 + i], qa[0], b0, b1);
            }
          }
        }
      }
      // keys past T do not take part
      if (!FULL) {
#pragma unroll
        for (int nt = 0; nt < kAttnKB / 8; ++nt) {
          const int key = kb + nt * 8 + 2 * tq;
          if (key >= T) s[nt][0] = s[nt][2] = -3.0e38f;
          if (key + 1 >= T) s[nt][1] = s[nt][3] = -3.0e38f;
        }
      }
      // online softmax: block maxima of rows g and g + 8 over the 4 lanes of a quad
      float bm0 = -3.0e38f, bm1 = -3.0e38f;
#pragma unroll
      for (int nt = 0; nt < kAttnKB / 8; ++nt) {
        bm0 = fmaxf(bm0, fmaxf(s[nt][0], s[nt][1]));
        bm1 = fmaxf(bm1, fmaxf(s[nt][2], s[nt][3]));
      }
      bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 1));
      bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 1));
      bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 2));
      bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 2));
      const float nm0 = fmaxf(m0, bm0), nm1 = fmaxf(m1, bm1);
      const float c0 = exp2f((m0 - nm0) * sl2), c1 = exp2f((m1 - nm1) * sl2);
      m0 = nm0;
      m1 = nm1;
      // exponents (s - max) sl2, the difference first: it is exact for scores near
      // the maximum, whatever their size (s sl2 - max sl2 in one FMA rounds its
      // offset at the size of the maximum: other blocks' weights 3 % off at scores
      // of 4e6; it is 1 to 2 % faster)
      const f2_t sc2 = f2(sl2, sl2), n02 = f2(-nm0, -nm0), n12 = f2(-nm1, -nm1);
      float rs0 = 0.f, rs1 = 0.f;
      uint32_t pa[kAttnKB / 16][4];  // P as A fragments of the P V MMAs
#pragma unroll
      for (int nt = 0; nt < kAttnKB / 8; ++nt) {
        float p0 = 0.f, p1 = 0.f, p2 = 0.f, p3 = 0.f;
        if (FULL || kb + nt * 8 < T) {  // uniform across the warp
          f2_split(fmul2(fadd2(f2(s[nt][0], s[nt][1]), n02), sc2), p0, p1);
          f2_split(fmul2(fadd2(f2(s[nt][2], s[nt][3]), n12), sc2), p2, p3);
          p0 = exp2f(p0);
          p1 = exp2f(p1);
          p2 = exp2f(p2);
          p3 = exp2f(p3);
        }
        rs0 += p0 + p1;
        rs1 += p2 + p3;
        pa[nt >> 1][(nt & 1) * 2 + 0] = pack_bf16x2(p0, p1);
        pa[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16x2(p2, p3);
      }
      l0 = l0 * c0 + rs0;
      l1 = l1 * c1 + rs1;
#pragma unroll
      for (int j = 0; j < HD / 8; ++j) {
        o[j][0] *= c0;
        o[j][1] *= c0;
        o[j][2] *= c1;
        o[j][3] *= c1;
      }
      // O += P V: k-steps of 16 keys (those starting before T), two 8-dimension
      // n-tiles per ldmatrix
#pragma unroll
      for (int kk = 0; kk < kAttnKB / 16; ++kk) {
        if (FULL || kb + kk * 16 < T) {  // uniform across the warp
          const uint32_t va = v_lane + (uint32_t)((kb + kk * 16) * KP * 2);
#pragma unroll
          for (int j = 0; j < HD / 8; j += 2) {
            uint32_t b0, b1, b2, b3;
            ldsm_x4_trans(va + (uint32_t)(j * 8 * 2), b0, b1, b2, b3);
            mma_bf16_16816(o[j], pa[kk], b0, b1);
            mma_bf16_16816(o[j + 1], pa[kk], b2, b3);
          }
        }
      }
    };
    int kb = 0;
    for (; kb + kAttnKB <= T; kb += kAttnKB) block(BoolConst<true>{}, kb);
    if (kb < T) block(BoolConst<false>{}, kb);
    // row sums over the quad, then O / sum
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
    l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    const float i0 = 1.f / l0, i1 = 1.f / l1;
    const int r0 = q0 + g, r1 = q0 + g + 8;
    const int64_t g0 = (int64_t)n * T + r0, g1 = (int64_t)n * T + r1;  // output rows
    // which of this lane's values are non-zero: bit j column 8 j + 2 tq, bit 16 + j
    // the one after it, of rows r0 and r1
    uint32_t nz0 = 0u, nz1 = 0u;
    const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < HD / 8; ++j) {
      const int c = h * HD + j * 8 + 2 * tq;
      const __nv_bfloat162 w0 = __floats2bfloat162_rn(o[j][0] * i0, o[j][1] * i0);
      const __nv_bfloat162 w1 = __floats2bfloat162_rn(o[j][2] * i1, o[j][3] * i1);
      if (r0 < T) *reinterpret_cast<__nv_bfloat162*>(y + g0 * D + c) = w0;
      if (r1 < T) *reinterpret_cast<__nv_bfloat162*>(y + g1 * D + c) = w1;
      nz0 |= __hneu2_mask(w0, zero2) & (0x00010001u << j);
      nz1 |= __hneu2_mask(w1, zero2) & (0x00010001u << j);
    }
    if (emit) {
      if (r0 >= T) nz0 = 0u;
      if (r1 >= T) nz1 = 0u;
      // row bits: a quad holds a row's HD columns
      const uint32_t any0 = __ballot_sync(0xffffffffu, nz0 != 0u), any1 = __ballot_sync(0xffffffffu, nz1 != 0u);
      const int tile = (h * HD) >> 6;
      const unsigned long long bit = 1ull << (tile & 63);
      if (tq == 0 && ((any0 >> (4 * g)) & 15u)) atomicOr(&occ.row_bm[g0 * occ.W64 + (tile >> 6)], bit);
      if (tq == 0 && ((any1 >> (4 * g)) & 15u)) atomicOr(&occ.row_bm[g1 * occ.W64 + (tile >> 6)], bit);
      // block-column words (HD columns from h HD on) of the one or two 128-row
      // blocks that the tile's rows lie in
      auto mask_out = [&](uint32_t v, int64_t b) {
        // four bits to the low bits of four bytes: (x * (1 + 2^7 + 2^14 + 2^21)) & 0x01010101
        auto spread = [](uint32_t x) { return ((x & 15u) * 0x00204081u) & 0x01010101u; };
        const int c = h * HD, sh = c & 31;  // (HD = 64: sh = 0)
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (spread(v) | (spread(v >> 16) << 1)) << (2 * tq)) << sh;
        if (lane == 0 && lo) atomicOr(&occ.blk_mask[b * occ.C32 + (c >> 5)], lo);
        if constexpr (HD > 32) {
          const uint32_t hi = __reduce_or_sync(0xffffffffu, (spread(v >> 4) | (spread(v >> 20) << 1)) << (2 * tq));
          if (lane == 0 && hi) atomicOr(&occ.blk_mask[b * occ.C32 + (c >> 5) + 1], hi);
        }
      };
      const int64_t b0 = ((int64_t)n * T + q0) >> 7;
      const bool in0 = (g0 >> 7) == b0, in1 = (g1 >> 7) == b0;
      mask_out((in0 ? nz0 : 0u) | (in1 ? nz1 : 0u), b0);
      if ((((int64_t)n * T + q0 + 15) >> 7) != b0) mask_out((in0 ? 0u : nz0) | (in1 ? 0u : nz1), b0 + 1);
      // column counts: rows r1's bits beside r0's, transposed over the warp
      const uint32_t x = warp_transpose32(nz0 | (nz1 << 8));
#pragma unroll
      for (int i = 0; i < 4; ++i) cnt += (uint32_t)__popc(x & (0x11111111u << i)) << (8 * i);
    }
  }
  if (!emit) return;
  cnt += __shfl_xor_sync(0xffffffffu, cnt, 8);  // (at most 5 tiles of 16 rows: bytes do not overflow)
  if ((lane & 8) == 0 && (lane & 7) < HD / 8) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t v = (cnt >> (8 * i)) & 0xFFu;
      if (v) atomicAdd(&s_cnt[8 * (lane & 7) + 2 * i + (lane >> 4)], v);
    }
  }
  __syncthreads();
  for (int c0 = warp * 32; c0 < HD; c0 += blockDim.x) {  // (HD columns: whole warps, or half of one)
    const int c = c0 + lane;
    const uint32_t v = c < HD ? s_cnt[c] : 0u;
    if (v) atomicAdd(&occ.col_nnz[h * HD + c], v);
    const uint32_t sum = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0 && sum) {
      atomicAdd(&occ.tile_nnz[(h * HD) >> 6], sum);
      atomicAdd(occ.nnz, (unsigned long long)sum);
    }
  }
}

// ---------------------------------------------------------------------------
// Token sequence: row 0 the class token, rows 1..P the patch vectors, each
// plus its position embedding (fp32 [1 + P][D]); 8 values per thread.
__global__ void __launch_bounds__(kVitThreads) tokens_kernel(const __nv_bfloat16* __restrict__ x, int N,
                                                             int P, int D,
                                                             const __nv_bfloat16* __restrict__ cls,
                                                             const float* __restrict__ pos,
                                                             __nv_bfloat16* __restrict__ y) {
  pdl_wait();
  pdl_trigger();
  const int cpr = D / 8;
  const int64_t total = (int64_t)N * (P + 1) * cpr;
  for (int64_t i = (int64_t)blockIdx.x * kVitThreads + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * kVitThreads) {
    const int c = (int)(i % cpr);
    const int64_t rt = i / cpr;
    const int t = (int)(rt % (P + 1));
    const int n = (int)(rt / (P + 1));
    const __nv_bfloat16* src = t == 0 ? cls + c * 8 : x + ((int64_t)n * P + (t - 1)) * D + c * 8;
    float f[8];
    unpack8(*reinterpret_cast<const uint4*>(src), f);
    const float* pp = pos + (int64_t)t * D + c * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k) f[k] += pp[k];
    *reinterpret_cast<uint4*>(y + rt * D + c * 8) = pack8(f);
  }
}

// Token `index` of every image: [N, T, D] -> [N, D].
__global__ void __launch_bounds__(kVitThreads) select_kernel(const __nv_bfloat16* __restrict__ x, int N, int T,
                                                             int D, int index, __nv_bfloat16* __restrict__ y) {
  pdl_wait();
  pdl_trigger();
  const int cpr = D / 8;
  const int64_t total = (int64_t)N * cpr;
  for (int64_t i = (int64_t)blockIdx.x * kVitThreads + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * kVitThreads) {
    const int c = (int)(i % cpr);
    const int n = (int)(i / cpr);
    *reinterpret_cast<uint4*>(y + (int64_t)n * D + c * 8) =
        *reinterpret_cast<const uint4*>(x + ((int64_t)n * T + index) * D + c * 8);
  }
}

unsigned grid_for(int64_t work, int per_cta) {
  const int64_t b = (work + per_cta - 1) / per_cta;
  const int64_t cap = 8LL * device_sm_count();
  return (unsigned)(b < 1 ? 1 : (b < cap ? b : cap));
}

}  // namespace

size_t attention_smem(int T, int hd) {
  const size_t T16 = (size_t)(T + 15) / 16 * 16;
  return 2 * 2 * T16 * (size_t)(hd + 8);  // K and V, bf16
}

namespace {

// Warps of a CTA and CTAs of a head, for `pairs` (image, head) pairs.
//   - Pairs that fill the SMs twice: one CTA a head, which stages its K and V
//     once, a tile per warp up to 7, then over at most 5 warps (7 beyond 15
//     tiles).  With CTAs of 7 warps and a tile per warp throughout the warps
//     without a tile, and a second copy of K and V, cost more than the fuller
//     SMs gave.  Where one CTA a head leaves the last round mostly empty (some
//     hundred pairs of more than 15 tiles, two CTAs an SM), a tile per warp.
//   - Fewer pairs: a tile per warp, and up to a CTA per SM, of two tiles or more;
//     three a head while two an SM hold them; as many as two an SM hold where each
//     keeps four tiles (48 pairs, T = 384 16.1 -> 12, 96 pairs 23 -> 19.6 us).  Warps
//     without a tile stage.
// Times with occupancy, us: CTAs of 7 warps with a tile per warp / this rule:
//   pairs, dimension  T = 16       64         128        197        257       512
//   12, 64           3.4 / 3.5  4.0 / 3.9  4.9 / 4.8  7.3 / 6.0  8.3 / 6.9  12 / 9.7
//   384, 64          5.7 / 4.4  7.8 / 6.5   17 / 13    30 / 28    42 / 42  145 / 138
//   1536, 64          14 / 7.0   24 / 20    54 / 40    89 / 87   147 / 137
//   1536, 32          13 / 5.4   18 / 14    42 / 28    67 / 61   107 / 97  267 / 254
void attention_split(int64_t pairs, int T, size_t smem, int* warps, int* qsplit) {
  const int64_t sms = device_sm_count();
  const int tiles = (T + 15) / 16;
  auto up = [](int a, int b) { return (a + b - 1) / b; };
  const bool two = smem <= 110 * 1024;  // CTAs that fit an SM
  int q = up(tiles, kAttnWarps);
  if (pairs >= 2 * sms) {
    if (tiles <= 15 || pairs >= 8 * sms || !two) q = 1;
    const int per = up(tiles, q), wmax = per > kAttnWarps && per <= 15 ? 5 : kAttnWarps;
    *warps = up(per, up(per, wmax));
  } else {
    const int64_t fill = sms / pairs;
    if (fill > q) q = (int)(fill < up(tiles, 2) ? fill : up(tiles, 2));
    if (q < 3 && tiles >= 8 && 3 * pairs <= 2 * sms) q = 3;
    const int64_t even = two ? 2 * sms / pairs : 0;  // CTAs of a head that fill the SMs twice
    if (even >= 3 && 4 * even <= tiles) q = (int)even;
    const int per = up(tiles, q);
    q = up(tiles, per);
    *warps = per > kAttnWarps ? up(per, 2) : kAttnWarps;
  }
  *qsplit = q;
}

template <int HD>
cudaError_t launch_attention_hd(const __nv_bfloat16* qkv, int N, int T, int heads, __nv_bfloat16* y,
                                const OccDev& o, int emit, cudaStream_t s) {
  const size_t smem = attention_smem(T, HD);
  if (smem > 40 * 1024) {
    cudaError_t e = smem_optin(reinterpret_cast<const void*>(attention_kernel<HD>), smem);
    if (e != cudaSuccess) return e;
  }
  int warps, qsplit;
  attention_split((int64_t)N * heads, T, smem, &warps, &qsplit);
  return launch_kernel(attention_kernel<HD>, dim3((unsigned)(N * heads), (unsigned)qsplit), dim3(32u * warps), smem, s,
                       qkv, T, heads, y, o, emit);
}

}  // namespace

cudaError_t launch_attention(const __nv_bfloat16* qkv, int N, int T, int heads, int hd, __nv_bfloat16* y,
                             const OccDev& o, int emit, cudaStream_t s) {
  if (N <= 0 || T <= 0) return cudaSuccess;
  if (T > kAttnMaxT || heads <= 0) return cudaErrorInvalidValue;
  switch (hd) {
    case 16: return launch_attention_hd<16>(qkv, N, T, heads, y, o, emit, s);
    case 32: return launch_attention_hd<32>(qkv, N, T, heads, y, o, emit, s);
    case 64: return launch_attention_hd<64>(qkv, N, T, heads, y, o, emit, s);
    default: return cudaErrorInvalidValue;
  }
}

bool layernorm_emits(int C) { return C <= 8 * 32 * kLnRegChunks; }

cudaError_t launch_layernorm(const __nv_bfloat16* x, int64_t R, int C, const float* gb, float eps,
                             __nv_bfloat16* y, const OccDev& o, int emit, cudaStream_t s) {
  if (R <= 0) return cudaSuccess;
  if (C % 8) return cudaErrorInvalidValue;
  if (!layernorm_emits(C)) {
    if (emit) return cudaErrorInvalidValue;
    return launch_kernel(layernorm_kernel, dim3(grid_for(R, kVitThreads / 32)), dim3(kVitThreads), 0, s, x, R, C, gb,
                         eps, y);
  }
  // a warp per row up to the resident warps, then runs of rows; 16 warps a CTA
  // once they fill the SMs (fewer CTAs add their column counts up in global memory)
  const int threads = R >= 8 * (int64_t)device_sm_count() ? kLnThreads : 256;
  const int64_t ctas = (R + threads / 32 - 1) / (threads / 32);
  const int64_t cap = (int64_t)device_sm_count() * (C <= 256 ? 2 : 1);
  const dim3 grid((unsigned)(ctas < cap ? ctas : cap));
  const int vec = (reinterpret_cast<uintptr_t>(gb) & 15u) == 0;  // (C % 8 == 0: beta's rows too)
  switch ((C + 255) / 256) {
    case 1: return launch_kernel(ln_rows_kernel<1>, grid, dim3((unsigned)threads), 0, s, x, R, C, gb, vec, eps, y, o, emit);
    case 2: return launch_kernel(ln_rows_kernel<2>, grid, dim3((unsigned)threads), 0, s, x, R, C, gb, vec, eps, y, o, emit);
    case 3: return launch_kernel(ln_rows_kernel<3>, grid, dim3((unsigned)threads), 0, s, x, R, C, gb, vec, eps, y, o, emit);
    default: return launch_kernel(ln_rows_kernel<4>, grid, dim3((unsigned)threads), 0, s, x, R, C, gb, vec, eps, y, o, emit);
  }
}

cudaError_t launch_tokens(const __nv_bfloat16* x, int N, int P, int D, const __nv_bfloat16* cls,
                          const float* pos, __nv_bfloat16* y, cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  if (D % 8) return cudaErrorInvalidValue;
  return launch_kernel(tokens_kernel, dim3(grid_for((int64_t)N * (P + 1) * (D / 8), kVitThreads)),
                       dim3(kVitThreads), 0, s, x, N, P, D, cls, pos, y);
}

cudaError_t launch_select(const __nv_bfloat16* x, int N, int T, int D, int index, __nv_bfloat16* y,
                          cudaStream_t s) {
  if (N <= 0) return cudaSuccess;
  if (D % 8 || index < 0 || index >= T) return cudaErrorInvalidValue;
  return launch_kernel(select_kernel, dim3(grid_for((int64_t)N * (D / 8), kVitThreads)), dim3(kVitThreads), 0,
                       s, x, N, T, D, index, y);
}

}  // namespace sparoa
