// Depthwise 3x3 convolution, pad 1, stride S in {1, 2} (every depthwise layer
// of MobileNetV2), with folded batch norm, activation, optional residual and
// the output's occupancy (Eq. 1 count and bitmaps, Sec. 3.1).
//
// Work: an item is a 32-channel slice of a strip of 4 PX output columns over a
// run of output rows, and belongs to one warp; warps share nothing but the
// weights, so there is no block barrier between the prologue and the end.  Lane
// l computes channels 4 (l % 8) .. + 3 of PX adjacent pixels (PX (l / 8) ..)
// and marches down the rows: each input value is read from shared memory and
// widened once, and added to the up to three output rows it belongs to, whose
// accumulators and the 36 weights stay in registers.  Channels go in pairs
// through packed fp32x2 FMAs, in the order kernel row, then kernel column.
//
// Input rows reach shared memory as 4-D TMA boxes {32 channels, IW, 3 rows (stride 2: 2), 1}
// (coordinates outside the image read zeros, which is the padding) through a
// ring of boxes per warp that runs on across items.
//
// Bound by instruction issue and latency (FMAs are under a third), so the rows
// come three to a box (one wait and one request for them), pointers advance by
// constants and a value is widened once.  [32, 56, 56, 144] stride 1 without / with
// occupancy 18.5 / 25.8 us, [32, 112, 112, 96] stride 2 17.6 / 23.1 us; CTAs of
// 64-channel windows of 8 x 16 pixels, which read and widened every value three
// times, re-read the weights every step and met at two barriers a step, took
// 28.7 / 40.2 and 23.6 / 29.8 us.
//
// Occupancy: a warp's slice is one 32-channel word of the 128-row block masks,
// which gather in registers until the rows leave the block; row bits are ORed over
// a pixel's lanes; column counts are 16-bit halves per lane, summed per item into
// shared memory and once per CTA into global memory.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "sparoa_kernels.h"

namespace sparoa {

PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder();  // k_igemm.cu

namespace {

// Pixels a lane and warps a CTA (one CTA per SM): 12 warps leave 168 registers a
// thread, 16 leave 128.  Stride 1, [32, 56, 56, C], without / with occupancy:
// C = 128  2 pixels, 12 warps 13.8 / 19.5 us; 16 warps 16.8 / 22.7; 4 pixels,
// 12 warps 15.8 / 21.1; C = 144  18.5 / 25.8; 17.9 / 25.0; 20.4 / 26.9 (12 fill
// the last round of warps less).  Stride 2, [32, 112, 112, 96]: 16 warps 18.1 /
// 23.0, 12 warps 18.5 / 24.1.
template <int S>
struct Dw3Split {
  static constexpr int PX = 2, kWarps = S == 1 ? 12 : 16;
};
constexpr int kMaxRun = 2048;                // rows of an item: its 16-bit column counts cannot overflow
constexpr int kMinStages = 3, kMaxStages = 6;
constexpr size_t kMaxSmem = 200 * 1024;

template <int S>
struct Dw3Shape {
  static constexpr int PX = Dw3Split<S>::PX;
  static constexpr int kWarps = Dw3Split<S>::kWarps;
  static constexpr int kThreads = kWarps * 32;
  static constexpr int TW = 4 * PX;            // output columns of an item
  static constexpr int IW = (TW - 1) * S + 3;  // input columns
  static constexpr int NCOL = (PX - 1) * S + 3;  // input columns of a lane's pixels
  static constexpr int RB = S == 1 ? 3 : 1;    // output rows a box completes, once the first ones are in
  static constexpr int IH = S == 1 ? 3 : 2;    // input rows of a box
  static constexpr int kStageBytes = IH * IW * 64;
  // boxes of an item of `rows` output rows
  static constexpr __host__ __device__ int boxes(int rows) { return S == 1 ? (rows + 4) / 3 : rows + 1; }
  static_assert(kStageBytes % 128 == 0, "TMA destinations");
};

struct Dw3Geo {
  int Cp;       // channels rounded up to 64
  int slices;   // 32-channel slices
  int tiles_w;  // strips of an output row
  int run, runs;  // output rows of an item (the last run of an image may be shorter), runs of an image
  int stages;   // ring of a warp
  uint32_t items;  // below 2^31: 2^38 bf16 values of input are at most 2^30 strips of a row
  int w_off, aff_off, cnt_off;  // shared-memory carve (bytes); the rings come first
};

// a bf16 pair widened to fp32 (exact)
__device__ __forceinline__ f2_t widen(uint32_t w) {
  return f2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}

struct Item {
  int n, r0, rows, tx, ct;
};

__device__ __forceinline__ Item decode_item(uint32_t i, const Dw3Geo& G, int Ho) {
  Item q;
  const uint32_t r = i / (uint32_t)G.slices, r2 = r / (uint32_t)G.tiles_w;
  q.ct = (int)(i - r * G.slices);
  q.tx = (int)(r - r2 * G.tiles_w);
  q.n = (int)(r2 / (uint32_t)G.runs);
  q.r0 = (int)(r2 - (uint32_t)q.n * G.runs) * G.run;
  q.rows = min(G.run, Ho - q.r0);
  return q;
}

template <int S, int ACT, bool RES>
__global__ void __launch_bounds__(Dw3Shape<S>::kThreads, 1)
    dw3_kernel(const __grid_constant__ CUtensorMap tmX, const DwArgs a, const Dw3Geo G) {
  using Sh = Dw3Shape<S>;
  constexpr int PX = Sh::PX, NCOL = Sh::NCOL, kWarps = Sh::kWarps, kThreads = Sh::kThreads;
  extern __shared__ uint8_t dsm_raw[];
  uint8_t* dsm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm_raw) + 127) & ~uintptr_t(127));
  float* s_w = reinterpret_cast<float*>(dsm + G.w_off);        // [9][Cp] weights
  float* s_sc = reinterpret_cast<float*>(dsm + G.aff_off);     // [Cp] affine scale
  float* s_sh = s_sc + G.Cp;                                   // [Cp] affine shift
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(dsm + G.cnt_off);  // [Cp] column counts
  __shared__ __align__(8) unsigned long long s_bar[kWarps * kMaxStages];
  __shared__ int s_abort;

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cg = lane & 7, st = lane >> 3;
  const OccDev o = a.out_occ;
  const bool emit = a.emit != 0;
  const long long wlim = a.wait_limit > 0 ? a.wait_limit : kWaitLimitCycles;
  const uint32_t bar0 = smem_u32(&s_bar[warp * kMaxStages]);
  const uint32_t ring = smem_u32(dsm) + (uint32_t)(warp * G.stages * Sh::kStageBytes);

  if (lane == 0) {
    for (int b = 0; b < G.stages; ++b) mbar_init(bar0 + 8 * b, 1u);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) {
    s_abort = 0;
    prefetch_tmap(&tmX);
  }
  for (int c = threadIdx.x; c < G.Cp; c += kThreads) s_cnt[c] = 0u;
  __syncwarp();
  pdl_wait();
  pdl_trigger();
  if (a.path_out && blockIdx.x == 0 && threadIdx.x == 0) *a.path_out = 3;

  // the boxes of this warp's items in order: item first, first + stride, ...;
  // an item's boxes start at input row S r0 - 1
  const uint32_t stride = gridDim.x * kWarps;
  uint32_t cur = warp * gridDim.x + blockIdx.x;
  uint32_t pit = cur;
  int px, py, pc, pn, pleft, pslot = 0;  // the next box's corner, and the boxes left of its item
  auto start_item = [&]() {
    const Item q = decode_item(pit, G, a.Ho);
    pc = q.ct * 32;
    px = q.tx * Sh::TW * S - 1;
    py = q.r0 * S - 1;
    pn = q.n;
    pleft = Sh::boxes(q.rows);
  };
  start_item();
  uint32_t issued = 0, consumed = 0;
  auto issue_next = [&]() {  // converged: one more box, if there is one
    if (pit >= G.items) return;
    if (elect_one()) {
      const uint32_t bar = bar0 + 8 * pslot;
      mbar_arrive_expect_tx(bar, (uint32_t)Sh::kStageBytes);
      tma_load_4d(ring + (uint32_t)(pslot * Sh::kStageBytes), &tmX, bar, pc, px, py, pn);
    }
    __syncwarp();
    ++issued;
    if (++pslot == G.stages) pslot = 0;
    py += Sh::IH;
    if (--pleft == 0) {
      pit += stride;
      if (pit < G.items) start_item();
    }
  };
  for (int b = 0; b < G.stages; ++b) issue_next();
  // weights and affine of every channel, fp32 (zero / identity past C)
  for (int i = threadIdx.x; i < 9 * G.Cp; i += kThreads) {
    const int t = i / G.Cp, c = i - t * G.Cp;
    s_w[i] = c < a.C ? __bfloat162float(a.w[c * 9 + t]) : 0.f;
  }
  for (int c = threadIdx.x; c < G.Cp; c += kThreads) {
    float sc = 1.f, sh = 0.f;
    if (c < a.C) epi_affine(a.ep, a.C, c, sc, sh);
    s_sc[c] = sc;
    s_sh[c] = sh;
  }
  __syncthreads();

  bool aborted = false;
  int slot = 0;
  uint32_t phase = 0u;
  for (; cur < G.items && !aborted; cur += stride) {
    const Item it = decode_item(cur, G, a.Ho);
    const int c0 = it.ct * 32 + cg * 4;
    const bool cvalid = c0 < a.C;
    const int tile_w = min(Sh::TW, a.Wo - it.tx * Sh::TW);  // live columns of the strip
    f2_t w[9][2];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&s_w[k * G.Cp + c0]);
      w[k][0] = v.x;
      w[k][1] = v.y;
    }
    uint32_t lm[PX];  // low bit of each half where this lane has a live pixel
#pragma unroll
    for (int j = 0; j < PX; ++j) lm[j] = cvalid && st * PX + j < tile_w ? 0x00010001u : 0u;
    // the strip's first pixel in the next output row, and this lane's values there
    uint32_t mt = (uint32_t)(it.n * a.Ho + it.r0) * (uint32_t)a.Wo + (uint32_t)(it.tx * Sh::TW);
    __nv_bfloat16* yp = a.y + ((int64_t)(mt + (uint32_t)(st * PX)) * a.C + c0);
    uint32_t cnt[2] = {0u, 0u};   // column counts, 16-bit halves (channels 2 p, 2 p + 1)
    uint32_t bacc[2] = {0u, 0u};  // non-zero pairs so far in block cur_blk
    uint32_t cur_blk = mt >> 7;
    uint32_t flags = 0u;          // bit PX k + j: pixel j of the box's output row k has a non-zero here
    auto flush_blk = [&]() {
      uint32_t m4 = ((bacc[0] & 1u) | ((bacc[0] >> 15) & 2u) | ((bacc[1] & 1u) << 2) | ((bacc[1] >> 13) & 8u))
                    << (4 * cg);
      m4 = __reduce_or_sync(0xffffffffu, m4);
      if (lane == 0 && m4) atomicOr(&o.blk_mask[(int64_t)cur_blk * o.C32 + it.ct], m4);
    };
    // the next output row, finished; k: its place in the box
    auto epilogue = [&](f2_t (&acc)[PX][2], int k) {
      const ulonglong2 sc = *reinterpret_cast<const ulonglong2*>(&s_sc[c0]);
      const ulonglong2 sh = *reinterpret_cast<const ulonglong2*>(&s_sh[c0]);
      const f2_t sc2[2] = {sc.x, sc.y}, sh2[2] = {sh.x, sh.y};
      uint32_t z[PX][2];
      const __nv_bfloat162 zero2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < PX; ++j) {
        uint2 res = make_uint2(0u, 0u);
        if (RES && lm[j]) res = *reinterpret_cast<const uint2*>(a.ep.residual + (yp - a.y) + j * a.C);
        const uint32_t rw[2] = {res.x, res.y};
        uint32_t pk[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          float lo, hi;
          f2_split(ffma2(acc[j][p], sc2[p], sh2[p]), lo, hi);
          if (RES) {
            lo += __uint_as_float(rw[p] << 16);
            hi += __uint_as_float(rw[p] & 0xFFFF0000u);
          }
          pk[p] = act_pack2<ACT>(lo, hi);
        }
        if (lm[j]) *reinterpret_cast<uint2*>(yp + j * a.C) = make_uint2(pk[0], pk[1]);
#pragma unroll
        for (int p = 0; p < 2; ++p)
          z[j][p] = __hneu2_mask(*reinterpret_cast<const __nv_bfloat162*>(&pk[p]), zero2) & lm[j];
      }
      if (emit) {
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          cnt[0] += z[j][0];
          cnt[1] += z[j][1];
          if (z[j][0] | z[j][1]) flags |= 1u << (PX * k + j);
        }
        const uint32_t bf = mt >> 7, bl = (mt + (uint32_t)(tile_w - 1)) >> 7;
        if (bf != cur_blk) {
          flush_blk();
          bacc[0] = bacc[1] = 0u;
          cur_blk = bf;
        }
        if (bl == bf) {
#pragma unroll
          for (int j = 0; j < PX; ++j) {
            bacc[0] |= z[j][0];
            bacc[1] |= z[j][1];
          }
        } else {
          uint32_t h[2] = {0u, 0u};
#pragma unroll
          for (int j = 0; j < PX; ++j) {
            const bool hi = ((mt + (uint32_t)(st * PX + j)) >> 7) != bf;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              if (hi) h[p] |= z[j][p];
              else bacc[p] |= z[j][p];
            }
          }
          flush_blk();
          cur_blk = bl;
          bacc[0] = h[0];
          bacc[1] = h[1];
        }
      }
      mt += (uint32_t)a.Wo;
      yp += (int64_t)a.Wo * a.C;
    };
    // row bits of a box's output rows, which end before row mt / Wo: the 8 lanes of
    // a pixel's slice OR their flags and take a pixel each
    auto flush_rows = [&](int k_end) {
      uint32_t f = flags;
      flags = 0u;
      f |= __shfl_xor_sync(0xffffffffu, f, 1);
      f |= __shfl_xor_sync(0xffffffffu, f, 2);
      f |= __shfl_xor_sync(0xffffffffu, f, 4);
#pragma unroll
      for (int i = cg; i < PX * Sh::RB; i += 8) {
        const int k = i / PX, j = i % PX;
        const uint32_t m = mt - (uint32_t)((k_end - k) * a.Wo) + (uint32_t)(st * PX + j);
        if ((f >> i) & 1u)
          atomicOr(&o.row_bm[(int64_t)m * o.W64 + (it.ct >> 7)], 1ull << ((it.ct >> 1) & 63));
      }
    };
    auto wait_box = [&]() {
      aborted = !mbar_wait_warp(bar0 + 8 * slot, phase, a.err, &s_abort, kErrTimeoutFull, wlim);
      return dsm + (warp * G.stages + slot) * Sh::kStageBytes + st * PX * S * 64 + cg * 8;
    };
    auto release_box = [&]() {  // every lane has read the box: the next one may land there
      __syncwarp();
      ++consumed;
      if (++slot == G.stages) {
        slot = 0;
        phase ^= 1u;
      }
      issue_next();
    };
    const int nbox = Sh::boxes(it.rows);
    if constexpr (S == 1) {
      f2_t acc[3][PX][2];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < PX; ++j) acc[i][j][0] = acc[i][j][1] = 0ull;
      // input row t (from r0 - 1): kernel row 2 of output row t - 2, 1 of t - 1, 0 of t
      auto row = [&](f2_t (&A)[PX][2], f2_t (&B)[PX][2], f2_t (&C)[PX][2], const uint2 (&raw)[NCOL]) {
#pragma unroll
        for (int q = 0; q < NCOL; ++q) {
          const f2_t in[2] = {widen(raw[q].x), widen(raw[q].y)};
#pragma unroll
          for (int j = 0; j < PX; ++j) {
            const int kc = q - j;
            if (kc >= 0 && kc < 3) {
#pragma unroll
              for (int p = 0; p < 2; ++p) {
                A[j][p] = ffma2(in[p], w[6 + kc][p], A[j][p]);
                B[j][p] = ffma2(in[p], w[3 + kc][p], B[j][p]);
                C[j][p] = ffma2(in[p], w[kc][p], kc == 0 ? f2_t(0) : C[j][p]);
              }
            }
          }
        }
      };
      for (int b = 0; b < nbox; ++b) {
        const uint8_t* src = wait_box();
        if (aborted) break;
        uint2 raw[3][NCOL];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int q = 0; q < NCOL; ++q) raw[k][q] = *reinterpret_cast<const uint2*>(src + (k * Sh::IW + q) * 64);
        release_box();
        const int left = it.rows - (3 * b - 2);  // output rows from the first this box completes
        row(acc[1], acc[2], acc[0], raw[0]);
        if (b > 0) epilogue(acc[1], 0);
        row(acc[2], acc[0], acc[1], raw[1]);
        if (b > 0 && left > 1) epilogue(acc[2], 1);
        row(acc[0], acc[1], acc[2], raw[2]);
        if (left > 2) epilogue(acc[0], 2);
        if (emit) flush_rows(min(left, 3));
      }
    } else {
      f2_t acc[PX][2];
#pragma unroll
      for (int j = 0; j < PX; ++j) acc[j][0] = acc[j][1] = 0ull;
      // box t: input rows 2 t - 1 (kernel row 2 of output row t - 1, 0 of t) and 2 t (1 of t)
      for (int t = 0; t < nbox; ++t) {
        const uint8_t* src = wait_box();
        if (aborted) break;
        uint2 raw[NCOL], raw1[NCOL];
#pragma unroll
        for (int q = 0; q < NCOL; ++q) raw[q] = *reinterpret_cast<const uint2*>(src + q * 64);
#pragma unroll
        for (int q = 0; q < NCOL; ++q) raw1[q] = *reinterpret_cast<const uint2*>(src + (Sh::IW + q) * 64);
        release_box();
        f2_t nxt[PX][2];
#pragma unroll
        for (int q = 0; q < NCOL; ++q) {
          const f2_t in[2] = {widen(raw[q].x), widen(raw[q].y)};
#pragma unroll
          for (int j = 0; j < PX; ++j) {
            const int kc = q - 2 * j;
            if (kc >= 0 && kc < 3) {
#pragma unroll
              for (int p = 0; p < 2; ++p) {
                acc[j][p] = ffma2(in[p], w[6 + kc][p], acc[j][p]);
                nxt[j][p] = ffma2(in[p], w[kc][p], kc == 0 ? f2_t(0) : nxt[j][p]);
              }
            }
          }
        }
        if (t >= 1) epilogue(acc, 0);
        if (t >= 1 && emit) flush_rows(1);
#pragma unroll
        for (int q = 0; q < NCOL; ++q) {
          const f2_t in[2] = {widen(raw1[q].x), widen(raw1[q].y)};
#pragma unroll
          for (int j = 0; j < PX; ++j) {
            const int kc = q - 2 * j;
            if (kc >= 0 && kc < 3) {
#pragma unroll
              for (int p = 0; p < 2; ++p) nxt[j][p] = ffma2(in[p], w[3 + kc][p], nxt[j][p]);
            }
          }
        }
#pragma unroll
        for (int j = 0; j < PX; ++j) {
          acc[j][0] = nxt[j][0];
          acc[j][1] = nxt[j][1];
        }
      }
    }
    if (emit) {
      flush_blk();
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        cnt[p] += __shfl_xor_sync(0xffffffffu, cnt[p], 8);  // the 4 strips
        cnt[p] += __shfl_xor_sync(0xffffffffu, cnt[p], 16);
        if (st == 0 && cvalid) {
          atomicAdd(&s_cnt[c0 + 2 * p], cnt[p] & 0xFFFFu);
          atomicAdd(&s_cnt[c0 + 2 * p + 1], cnt[p] >> 16);
        }
      }
    }
  }
  if (aborted && lane == 0) {
    // a bounded wait ran out: the boxes still in flight land before the shared
    // memory is released (each wait bounded again)
    for (; consumed < issued; ++consumed)
      mbar_drain(bar0 + 8 * (consumed % (uint32_t)G.stages), (consumed / (uint32_t)G.stages) & 1u, wlim);
  }
  __syncwarp();
  __syncthreads();
  if (!emit) return;
  for (int k = warp; k < G.Cp / 64; k += kWarps) {
    uint32_t sum = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = k * 64 + h * 32 + lane;
      const uint32_t v = s_cnt[c];
      if (v) atomicAdd(&o.col_nnz[c], v);
      sum += v;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0 && sum) {
      atomicAdd(&o.tile_nnz[k], sum);
      atomicAdd(o.nnz, (unsigned long long)sum);
    }
  }
}

template <int S, int ACT, bool RES>
cudaError_t launch_one(const CUtensorMap& tm, const DwArgs& a, const Dw3Geo& g, unsigned grid, size_t smem,
                       cudaStream_t s) {
  const void* fn = reinterpret_cast<const void*>(dw3_kernel<S, ACT, RES>);
  cudaError_t e = smem_optin(fn, smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(dw3_kernel<S, ACT, RES>, dim3(grid), dim3(Dw3Shape<S>::kThreads), smem, s, tm, a, g);
}

template <int S, int ACT>
cudaError_t launch_act(const CUtensorMap& tm, const DwArgs& a, const Dw3Geo& g, unsigned grid, size_t smem,
                       cudaStream_t s) {
  return a.ep.residual ? launch_one<S, ACT, true>(tm, a, g, grid, smem, s)
                       : launch_one<S, ACT, false>(tm, a, g, grid, smem, s);
}

size_t smem_bytes(int ring_bytes, int C) {
  return 128 + (size_t)ring_bytes + sizeof(uint32_t) * 12 * (size_t)((C + 63) / 64 * 64);
}

template <int S>
cudaError_t launch_shape(const DwArgs& a, cudaStream_t s) {
  using Sh = Dw3Shape<S>;
  Dw3Geo g;
  g.Cp = (a.C + 63) / 64 * 64;
  g.slices = (a.C + 31) / 32;
  g.tiles_w = (a.Wo + Sh::TW - 1) / Sh::TW;
  g.stages = kMaxStages;
  while (g.stages > kMinStages && smem_bytes(Sh::kWarps * Sh::kStageBytes * g.stages, a.C) > kMaxSmem) --g.stages;
  // rows of an item: the fewest rounds of all warps, each round costing its rows
  // and about three more (halo rows, the first box, the counts)
  const long long base = (long long)a.N * g.tiles_w * g.slices;
  const long long all = (long long)device_sm_count() * Sh::kWarps;
  double best = 0.;
  g.run = 0;
  for (int c = (a.Ho + kMaxRun - 1) / kMaxRun;;) {
    const int run = (a.Ho + c - 1) / c, runs = (a.Ho + run - 1) / run;
    const double cost = (double)((base * runs + all - 1) / all) * (S == 1 ? 3 * Sh::boxes(run) + 1 : run + 3);
    if (g.run == 0 || cost < best) {
      best = cost;
      g.run = run;
      g.runs = runs;
    }
    if (base * runs > 8 * all || run == 1) break;
    c = (a.Ho + run - 2) / (run - 1);  // the fewest runs that are shorter
  }
  if (base * g.runs >= (1ll << 31)) return cudaErrorInvalidValue;
  g.items = (uint32_t)(base * g.runs);
  g.w_off = Sh::kWarps * g.stages * Sh::kStageBytes;
  g.aff_off = g.w_off + (int)sizeof(float) * 9 * g.Cp;
  g.cnt_off = g.aff_off + (int)sizeof(float) * 2 * g.Cp;
  const size_t smem = smem_bytes(Sh::kWarps * Sh::kStageBytes * g.stages, a.C);
  const unsigned grid = g.items < (uint32_t)device_sm_count() ? g.items : (uint32_t)device_sm_count();

  auto enc = tmap_encoder();
  if (!enc) return cudaErrorInvalidValue;
  CUtensorMap tm;
  cuuint64_t dims[4] = {(cuuint64_t)a.C, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.N};
  cuuint64_t strides[3] = {(cuuint64_t)a.C * 2, (cuuint64_t)a.W * a.C * 2, (cuuint64_t)a.H * a.W * a.C * 2};
  cuuint32_t box[4] = {32, (cuuint32_t)Sh::IW, (cuuint32_t)Sh::IH, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  if (enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>((const void*)a.x), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  switch (a.ep.act) {
    case 0: return launch_act<S, 0>(tm, a, g, grid, smem, s);
    case 1: return launch_act<S, 1>(tm, a, g, grid, smem, s);
    case 2: return launch_act<S, 2>(tm, a, g, grid, smem, s);
    default: return launch_act<S, 3>(tm, a, g, grid, smem, s);
  }
}

}  // namespace

bool dw3_supported(const DwArgs& a) {
  if (!(a.kh == 3 && a.kw == 3 && a.pad == 1 && (a.stride == 1 || a.stride == 2) && a.C % 8 == 0)) return false;
  if ((reinterpret_cast<uintptr_t>(a.x) & 15u) != 0) return false;  // TMA: 16-byte aligned base
  if (a.ep.act < 0 || a.ep.act > 3) return false;
  const int box = a.stride == 1 ? Dw3Shape<1>::kWarps * Dw3Shape<1>::kStageBytes
                                : Dw3Shape<2>::kWarps * Dw3Shape<2>::kStageBytes;
  return smem_bytes(kMinStages * box, a.C) <= kMaxSmem;
}

cudaError_t launch_dw3(const DwArgs& a, cudaStream_t s) {
  return a.stride == 1 ? launch_shape<1>(a, s) : launch_shape<2>(a, s);
}

}  // namespace sparoa
