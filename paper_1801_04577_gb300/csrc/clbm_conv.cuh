// Convolutions of the warm-start network on operands that need no gather.
//
// The gathering GEMM (clbm_tc.cuh) builds an im2col tile for every 64 values
// of K: each FP32 activation is fetched nine times, one 4-byte load at a time,
// rounded to BF16 and stored to shared memory, and that bounds it (tensor pipe
// 1-3 % busy).  Here the pass that produces a tensor also writes it as the
// next pass's operand: rounded to BF16, eight channels (16 bytes) together,
// every image with a border of zeros,
//
//   element (sample n, channel c, y, x) at [c / 8][n Pn + (y + 1) Wp + x + 1][c % 8],
//   Wp = W + 2, Pn = (H + 2) Wp rounded up to 16 positions.
//
// A run of positions of one channel group is contiguous, so a tile arrives by
// one bulk copy per channel group, and in shared memory the same tile serves
// all nine taps: the tap (dy, dx) is the tile read dy Wp + dx positions later,
// a different start address in the matrix descriptor (no swizzle, rows 16
// bytes apart).  Border positions are computed and dropped: 6 % of the rows
// at 64^2, 13 % at 32^2.
//
// The products are summed in the order of the gathering GEMM (K tap-major, 16
// at a time, the same split ranges), so results are the same bit for bit.
// What is kept in BF16 is only what every reader rounds to BF16 first; what is
// read in FP32 (skip connections, gradients that are summed) is also stored in
// FP32.
#pragma once

#include "clbm_tc.cuh"

namespace conv {

using bf16 = __nv_bfloat16;

// An operand tensor: `base` points at position 0 of channel group 0 (a guard
// of zeros lies before it and after the last position), groups are pst
// positions apart.
struct Op {
  bf16* base;
  long long pst;
  int C;     // channels
  int H, W;  // image (square)
  __host__ __device__ int Wp() const { return W + 2; }
  __host__ __device__ int Pn() const { return ((H + 2) * (W + 2) + 15) / 16 * 16; }
};

__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(tc::pack_bf16(v[0], v[1]), tc::pack_bf16(v[2], v[3]), tc::pack_bf16(v[4], v[5]),
                    tc::pack_bf16(v[6], v[7]));
}
__device__ __forceinline__ uint4* op_at(const Op& o, int group, long long pos) {
  return reinterpret_cast<uint4*>(o.base) + group * o.pst + pos;
}
__device__ __forceinline__ void unpack8(uint4 u, float* v) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[2 * k] = __uint_as_float(w[k] << 16);
    v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
  }
}

// What becomes of eight output channels n0 .. n0 + 7 of one position.
struct Epilogue {
  const float* bias = nullptr;  // added, or nullptr
  int relu = 0;
  Op mask{};          // ReLU backward: zero where this activation is not positive (base nullptr: none)
  int mask_group = 0;
  Op op{};            // operand copy of the result (base nullptr: none), from channel group op_group
  int op_group = 0;
  float* f32 = nullptr;  // FP32 NCHW copy (nullptr: none): cs channels, from channel coff
  int cs = 0, coff = 0;
  int H = 0, W = 0, N = 0, channels = 0;  // image, samples, valid output channels

  // image coordinates of position pos; false on a border
  __device__ __forceinline__ bool locate(int pos, int& n, int& p) const {
    const int Wp = W + 2, Pn = ((H + 2) * Wp + 15) / 16 * 16;
    n = pos / Pn;
    const int r = pos - n * Pn, yy = r / Wp, xx = r - yy * Wp;
    p = (yy - 1) * W + xx - 1;
    return n < N && yy >= 1 && yy <= H && xx >= 1 && xx <= W;
  }
  // `b`: the bias of channels n0 .. n0 + 7 (read where bias is set)
  __device__ __forceinline__ void apply(int pos, int n, int p, int n0, float (&v)[8], const float* b) const {
    if (bias) {
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] += n0 + k < channels ? b[k] : 0.0f;
    }
    if (relu) {
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = v[k] > 0.0f ? v[k] : 0.0f;
    }
    if (mask.base) {
      float a[8];
      unpack8(*op_at(mask, mask_group + n0 / 8, pos), a);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (!(a[k] > 0.0f)) v[k] = 0.0f;
    }
    if (op.base) *op_at(op, op_group + n0 / 8, pos) = pack8(v);
    if (f32) {
      float* o = f32 + ((long long)n * cs + coff + n0) * H * W + p;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (n0 + k < channels) o[(long long)k * H * W] = v[k];
    }
  }
};

struct ConvArgs {
  Op a;              // input operand, channel groups [0, a.C / 8)
  const bf16* w;     // packed weights: [N tile][slice][bn x 64], chunk order of pair_swapped
  int taps, bn, slices;
  int kper, ranges;  // slices per range of K, ranges
  int mt;            // 128-position tiles of a block
  int stages;
  Epilogue epi;
  int* err;
};

// Programmatic dependent launch: a kernel of the chain may start while its
// predecessor runs; pdl_wait() returns when the predecessor's writes are
// visible, pdl_go() lets the successor start.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr int kMaxBn = 64;         // columns of a tile: a thread keeps its row's sums in registers
// threads of a block: four epilogue warps; copies and MMAs are issued by two of them, or by two more
// warps where sums of several ranges are formed while the MMAs go on
__host__ __device__ constexpr int conv_threads(bool ranges) { return ranges ? 192 : 128; }

constexpr int kMaxMt = 4;
// positions of a block's input: its mt tiles and the rows above and below
__host__ __device__ constexpr int conv_run(int taps, int Wp, int mt) {
  return mt * tc::kBM + (taps == 9 ? 2 * Wp + 2 : 0);
}
// pairs of K chunks (the MMAs), rounded up to whole slices
__host__ __device__ constexpr int conv_pairs(int C, int taps) { return (taps * C / 8 + 7) / 8 * 4; }
__host__ __device__ constexpr int conv_smem(int C, int taps, int Wp, int bn, int stages, int mt) {
  return stages * bn * 128 + (C / 8) * conv_run(taps, Wp, mt) * 16 + conv_pairs(C, taps) * 8 +  // B, A, descriptors,
         (2 * stages + 5) * 8 + 8 + bn * 4 + 64;                                                // barriers, slot, bias
}

// K chunk (eight channels of one tap) u = tap * groups + group; an MMA takes a
// pair of chunks (u, u + 1), u even, whose descriptors must lie at increasing
// addresses: the pair is swapped where it crosses a tap (the second chunk then
// starts before the first), and an odd last chunk is paired with the one
// before it, whose weights are zero there.
__host__ __device__ __forceinline__ bool pair_swapped(int u, int groups, int total) {
  return groups > 1 ? u % groups == groups - 1 : u + 1 == total && u > 0;
}

// Implicit GEMM D[position][channel] of mt 128-position tiles (blockIdx.x) and
// bn channels (blockIdx.y).  The tiles of a block share its input (of one tile
// alone, two thirds is halo at 128^2) and its weights.  The matrix descriptors are made beforehand by all
// threads: one thread that divided by the number of channel groups for every
// MMA took 20 us a tile.
//
// RANGES: K is summed in ranges, each into an accumulator of its own (two, in
// turn), and the ranges' sums are added in order in registers: the order of a
// split-K GEMM whose partial sums are added by a second kernel, without that
// kernel (94 us for the 384 -> 128 convolution at 16^2).  One range needs
// neither the registers nor the extra warps (three blocks per multiprocessor
// instead of seven doubled its time).
// Launch with conv_smem() bytes of dynamic shared memory.
template <bool RANGES>
__global__ void __launch_bounds__(conv_threads(RANGES), RANGES ? 1 : 8) conv_kernel(const __grid_constant__ ConvArgs a) {
  constexpr int kConvThreads = conv_threads(RANGES);
  constexpr int kCopyWarp = RANGES ? 4 : 0, kMmaWarp = RANGES ? 5 : 1;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int groups = a.a.C / 8, Wp = a.a.W + 2;
  const int run = conv_run(a.taps, Wp, RANGES ? 1 : a.mt), total = a.taps * groups;
  uint8_t* B = smem;
  uint8_t* A = smem + a.stages * a.bn * 128;
  uint64_t* desc = reinterpret_cast<uint64_t*>(A + groups * run * 16);
  uint64_t* bar_a = desc + conv_pairs(a.a.C, a.taps);
  uint64_t* bar_b = bar_a + 1;         // [stages] weights have arrived
  uint64_t* bar_m = bar_b + a.stages;  // [stages] MMAs that read the stage are done
  uint64_t* bar_d = bar_m + a.stages;  // [2] a range is complete in its accumulator
  uint64_t* bar_f = bar_d + 2;         // [2] ... and has been read
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar_f + 2);
  float* bias = reinterpret_cast<float*>(slot + 2);  // [bn]
  const int mt = RANGES ? 1 : a.mt;
  const int m0 = blockIdx.x * mt * tc::kBM, n0 = blockIdx.y * a.bn;
  const uint32_t ncols = tc::tmem_cols(RANGES ? 2 * a.bn : mt * a.bn);

  if (warp == 0) tc::tmem_alloc(slot, ncols);
  if (tid == 32) {
    tc::mbar_init(bar_a, 1);
    for (int k = 0; k < 2; ++k) {
      tc::mbar_init(&bar_d[k], 1);
      tc::mbar_init(&bar_f[k], tc::kBM);
    }
    for (int s = 0; s < a.stages; ++s) {
      tc::mbar_init(&bar_b[s], 1);
      tc::mbar_init(&bar_m[s], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // addresses of chunk c (tap t, group g): group run, t / 3 rows and t % 3 columns later
  auto at = [&](int c) {
    const int t = c / groups, g = c - t * groups;
    return (uint32_t)((g * run + (a.taps == 9 ? (t / 3) * Wp + t % 3 : 0)) * 16);
  };
  const int pairs = (total + 1) / 2;
  for (int j = tid; j < pairs; j += kConvThreads) {
    const int u = 2 * j;
    const bool swap = pair_swapped(u, groups, total);
    const uint32_t lo = swap ? (u + 1 < total ? at(u + 1) : at(u - 1)) : at(u);
    const uint32_t hi = swap ? at(u) : (u + 1 < total ? at(u + 1) : at(u));
    desc[j] = tc::smem_desc(tc::smem_u32(A) + lo, hi - lo, 128);
  }
  if (a.epi.bias)
    for (int k = tid; k < a.bn; k += kConvThreads) bias[k] = n0 + k < a.epi.channels ? a.epi.bias[n0 + k] : 0.0f;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  pdl_go();
  const uint32_t tmem = *slot;
  bool failed = false;
  float sum[RANGES ? kMaxBn : 1];

  if (warp == kCopyWarp) {
    const bf16* w = a.w + (long long)blockIdx.y * a.slices * a.bn * 64;
    auto weights = [&](int i) {
      const int s = i % a.stages;
      tc::mbar_expect_tx(&bar_b[s], (uint32_t)(a.bn * 128));
      tc::bulk_load(B + s * a.bn * 128, w + (long long)i * a.bn * 64, (uint32_t)(a.bn * 128), &bar_b[s]);
    };
    const int first = min(a.stages, a.slices);
    if (lane == 0) {  // the weights are older than the predecessor, the input is its result
      tc::mbar_expect_tx(bar_a, (uint32_t)(groups * run * 16));
      for (int i = 0; i < first; ++i) weights(i);
    }
    pdl_wait();
    __syncwarp();
    for (int g = lane; g < groups; g += 32)
      tc::bulk_load(A + g * run * 16, op_at(a.a, g, (long long)m0 - (a.taps == 9 ? Wp + 1 : 0)), (uint32_t)(run * 16),
                    bar_a);
    if (lane == 0) {
      int i = first;
      for (; i < a.slices; ++i) {
        if (!tc::mbar_wait(&bar_m[i % a.stages], (uint32_t)((i / a.stages - 1) & 1))) {
          failed = true;
          break;
        }
        weights(i);
      }
      if (failed) {  // the copies in flight end before the block does (bounded)
        tc::mbar_wait(bar_a, 0);
        for (int k = max(0, i - a.stages); k < i; ++k)
          tc::mbar_wait(&bar_b[k % a.stages], (uint32_t)((k / a.stages) & 1));
      }
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_bf16_f32(tc::kBM, a.bn);
      pdl_wait();  // the waits' limit counts from when the input can come
      failed = !tc::mbar_wait(bar_a, 0);
      int i = 0;
      for (int z = 0; z < (RANGES ? a.ranges : 1) && !failed; ++z) {
        const uint32_t acc = tmem + (z & 1) * a.bn;
        if (z >= 2) {
          failed = !tc::mbar_wait(&bar_f[z & 1], (uint32_t)((z / 2 - 1) & 1));
          tc::fence_after();
        }
        const int s1 = min(a.slices, (z + 1) * a.kper), s0 = i;
        for (; i < s1 && !failed; ++i) {
          const int s = i % a.stages;
          if (!tc::mbar_wait(&bar_b[s], (uint32_t)((i / a.stages) & 1))) {
            failed = true;
            break;
          }
          tc::fence_after();
          const uint64_t bdesc = tc::smem_desc(tc::smem_u32(B) + s * a.bn * 128, 128, 1024);
          const int m = min(4, pairs - 4 * i);
#pragma unroll 1
          for (int u = 0; u < mt; ++u)  // tile u lies 128 positions further (in units of 16 bytes)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j < m)
                tc::mma_bf16(acc + u * a.bn, desc[4 * i + j] + u * tc::kBM, bdesc + j * 16, idesc,
                             (i > s0 || j > 0) ? 1u : 0u);
          tc::mma_commit(&bar_m[s]);
        }
        tc::mma_commit(&bar_d[z & 1]);
      }
      // after a failure the other warps still wait for every range: let them time out on their own
    }
  }
  if constexpr (RANGES) {
    if (warp < 4) {
      pdl_wait();
#pragma unroll
      for (int c = 0; c < kMaxBn; ++c) sum[c] = 0.0f;
      for (int z = 0; z < a.ranges; ++z) {
        if (!tc::mbar_wait(&bar_d[z & 1], (uint32_t)((z / 2) & 1))) {
          failed = true;
          break;
        }
        tc::fence_after();
#pragma unroll
        for (int c0 = 0; c0 < kMaxBn; c0 += 16) {
          if (c0 >= a.bn) break;
          float v[16];
          tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((z & 1) * a.bn + c0), v);
#pragma unroll
          for (int k = 0; k < 16; ++k) sum[c0 + k] += v[k];
        }
        tc::fence_before();
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&bar_f[z & 1])) : "memory");
      }
    }
  } else {
    __syncwarp();
    pdl_wait();
    if (!tc::mbar_wait(&bar_d[0], 0)) failed = true;
  }
  if (__syncthreads_or(failed)) {
    if (tid == 0) atomicExch(a.err, 1);
  } else if (warp < 4) {
    tc::fence_after();
#pragma unroll 1
    for (int u = 0; u < mt; ++u) {
      const int pos = m0 + u * tc::kBM + tid;
      int n, p;
      const bool inside = a.epi.locate(pos, n, p);
#pragma unroll
      for (int c0 = 0; c0 < kMaxBn; c0 += 16) {
        if (c0 >= a.bn) break;
        float v[16];
        if constexpr (RANGES) {
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = sum[c0 + k];
        } else {
          tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(u * a.bn + c0), v);
        }
        if (!inside) continue;
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
          if (n0 + c0 + h >= a.epi.channels) break;
          float x[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) x[k] = v[h + k];
          a.epi.apply(pos, n, p, n0 + c0 + h, x, bias + c0 + h);
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---------------------------------------------------------------------------
// Weight gradient: D[o][tap, c] = sum over positions of g[o][pos] x[c][pos + tap].
// Both operands are the tensors as stored, positions along K (channels
// contiguous: the MN-major layout), g's zero border removes what the padded
// positions would add.  A block takes one range of positions (blockIdx.x), one
// set of columns (blockIdx.y: taps [t0, t0 + nt) of channel groups
// [g0, g0 + ng)) and 128 output channels (blockIdx.z); its partial sums go to
// part[range][tap C + c][o].
// ---------------------------------------------------------------------------
constexpr int kKP = 128;  // positions per stage
constexpr int kThreads = 128;

struct DwArgs {
  Op x, g;
  int taps, tap_set, tap_sets, group_set;  // taps and channel groups per block (columns <= 512)
  int K, kper;                             // positions, positions per range (a multiple of kKP)
  int stages;
  int ci, co;                              // rows of part that are stored: channels of x and g
  float* part;
  int* err;
};

__host__ __device__ constexpr int dw_run(int taps, int Wp) { return kKP + (taps == 9 ? 2 * Wp + 2 : 0); }
// stage: the channel groups of g (at most 16), then those of x; the 16 row groups that an MMA reads
// stay inside the stages (rows beyond g's channels are dropped)
__host__ __device__ constexpr int dw_stage(int gg, int gx, int taps, int Wp) {
  return gg * kKP * 16 + (gx + 1) * dw_run(taps, Wp) * 16;
}
__host__ __device__ constexpr int dw_smem(int gg, int gx, int taps, int Wp, int stages) {
  return stages * dw_stage(gg, gx, taps, Wp) + 16 * kKP * 16 + 256;
}
// columns of one tap: a multiple of 16 (M = 128)
__host__ __device__ constexpr int dw_cols(int groups) { return (groups + 1) / 2 * 16; }

__global__ void __launch_bounds__(kThreads) dw_kernel(const __grid_constant__ DwArgs a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Wp = a.x.W + 2, run = dw_run(a.taps, Wp);
  const int t0 = (blockIdx.y % a.tap_sets) * a.tap_set, nt = min(a.tap_set, a.taps - t0);
  const int g0 = (blockIdx.y / a.tap_sets) * a.group_set, ng = min(a.group_set, a.x.C / 8 - g0);
  const int o0 = blockIdx.z * 128, no = min(16, a.g.C / 8 - o0 / 8);
  const int cols = dw_cols(ng);
  const int k_lo = blockIdx.x * a.kper, k_hi = min(a.K, k_lo + a.kper);
  const int nk = (k_hi - k_lo + kKP - 1) / kKP;
  const int sbytes = dw_stage(min(16, a.g.C / 8), a.group_set, a.taps, Wp);
  uint64_t* bar_l = reinterpret_cast<uint64_t*>(smem + a.stages * sbytes + 16 * kKP * 16);
  uint64_t* bar_m = bar_l + a.stages;
  uint64_t* bar_d = bar_m + a.stages;
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar_d + 1);
  uint32_t ncols = 32;
  while (ncols < (uint32_t)(a.tap_set * dw_cols(a.group_set))) ncols *= 2;

  if (warp == 0) tc::tmem_alloc(slot, ncols);
  if (tid == 0) {
    tc::mbar_init(bar_d, 1);
    for (int s = 0; s < a.stages; ++s) {
      tc::mbar_init(&bar_l[s], 1);
      tc::mbar_init(&bar_m[s], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *slot;
  bool failed = false;
  int issued = 0;  // slices whose copies were started (warp 0)

  if (warp == 0) {
    for (int i = 0; i < nk; ++i) {
      const int s = i % a.stages;
      if (i >= a.stages && !tc::mbar_wait(&bar_m[s], (uint32_t)((i / a.stages - 1) & 1))) failed = true;
      if (__any_sync(0xffffffffu, failed)) {
        failed = true;
        break;
      }
      const int k0 = k_lo + i * kKP, kn = min(kKP, k_hi - k0);
      const int xn = kn + (a.taps == 9 ? 2 * Wp + 2 : 0);
      uint8_t* G = smem + s * sbytes;
      uint8_t* X = G + min(16, a.g.C / 8) * kKP * 16;
      if (lane == 0) tc::mbar_expect_tx(&bar_l[s], (uint32_t)((no * kn + ng * xn) * 16));
      __syncwarp();
      for (int g = lane; g < no + ng; g += 32) {
        if (g < no)
          tc::bulk_load(G + g * kKP * 16, op_at(a.g, o0 / 8 + g, k0), (uint32_t)(kn * 16), &bar_l[s]);
        else
          tc::bulk_load(X + (g - no) * run * 16, op_at(a.x, g0 + g - no, (long long)k0 - (a.taps == 9 ? Wp + 1 : 0)),
                        (uint32_t)(xn * 16), &bar_l[s]);
      }
      issued = i + 1;
    }
  } else if (tid == 32) {
    // both operands MN-major (bits 15, 16)
    const uint32_t idesc = tc::idesc_bf16_f32(128, cols) | (1u << 15) | (1u << 16);
    for (int i = 0; i < nk; ++i) {
      const int s = i % a.stages;
      if (!tc::mbar_wait(&bar_l[s], (uint32_t)((i / a.stages) & 1))) {
        failed = true;
        break;
      }
      tc::fence_after();
      const int kn = min(kKP, k_hi - (k_lo + i * kKP));
      const uint32_t G = tc::smem_u32(smem + s * sbytes), X = G + min(16, a.g.C / 8) * kKP * 16;
      const uint64_t gdesc = tc::smem_desc(G, 128, kKP * 16), xdesc = tc::smem_desc(X, 128, run * 16);
      for (int t = 0; t < nt; ++t) {
        const int tap = t0 + t, shift = a.taps == 9 ? (tap / 3) * Wp + tap % 3 : 0;
#pragma unroll 4
        for (int j = 0; j < kn / 16; ++j)  // start addresses in units of 16 bytes, one position each
          tc::mma_bf16(tmem + t * cols, gdesc + j * 16, xdesc + j * 16 + shift, idesc, (i > 0 || j > 0) ? 1u : 0u);
      }
      tc::mma_commit(&bar_m[s]);
    }
    tc::mma_commit(bar_d);
  }
  const bool done = tc::mbar_wait(bar_d, 0);
  if (__syncthreads_or(failed || !done)) {
    if (tid == 0) {  // the copies in flight end before the block does (bounded)
      atomicExch(a.err, 1);
      for (int i = max(0, issued - a.stages); i < issued; ++i)
        tc::mbar_wait(&bar_l[i % a.stages], (uint32_t)((i / a.stages) & 1));
    }
  } else {
    tc::fence_after();
    const int o = o0 + warp * 32 + lane;
    for (int t = 0; t < nt; ++t)
      for (int c0 = 0; c0 < cols; c0 += 16) {
        float v[16];
        tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(t * cols + c0), v);
        if (o >= a.co) continue;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int c = g0 * 8 + c0 + k;
          if (c0 + k < ng * 8 && c < a.ci)
            a.part[(((long long)blockIdx.x * a.taps + t0 + t) * a.ci + c) * a.co + o] = nk > 0 ? v[k] : 0.0f;
        }
      }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// dW[o][c][tap] = sum over ranges of part[range][tap ci + c][o], in a fixed
// order (as sum_splits_kernel).
__global__ void dw_sum_kernel(const float* __restrict__ part, int splits, int taps, int ci, int co,
                              float* __restrict__ out) {
  __shared__ float sh[32][33];
  const int R = blockDim.y, r = threadIdx.y, l = threadIdx.x;
  const long long n = (long long)taps * ci * co;
  for (long long i0 = (long long)blockIdx.x * 32; i0 < n; i0 += (long long)gridDim.x * 32) {
    const long long i = i0 + l;
    float s = 0.0f;
    if (i < n)
      for (int k = r; k < splits; k += R) s += part[(long long)k * n + i];
    sh[r][l] = s;
    __syncthreads();
    for (int o = R / 2; o > 0; o >>= 1) {
      if (r < o) sh[r][l] += sh[r + o][l];
      __syncthreads();
    }
    if (r == 0 && i < n) {
      const int o = (int)(i % co), tc_ = (int)(i / co), c = tc_ % ci, t = tc_ / ci;
      out[((long long)o * ci + c) * taps + t] = sh[0][l];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Element-wise passes in operand layout: one thread per position of the
// smaller image and eight channels (blockIdx.y = channel group).  All of the
// chain are launched as programmatic dependents (all of the forward pass's
// launches without their work 127 of 411 us at 128^2).
// ---------------------------------------------------------------------------

// FP32 NCHW (cs channels, C <= 8 of them from coff) -> one channel group, zero beyond C
__global__ void to_op_kernel(const float* __restrict__ x, int C, int N, Op o) {
  const int hw = o.H * o.W;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N * hw; i += gridDim.x * blockDim.x) {
    const int n = i / hw, p = i - n * hw, y = p / o.W, xx = p - y * o.W;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k < C ? x[((long long)n * C + k) * hw + p] : 0.0f;
    *op_at(o, 0, (long long)n * o.Pn() + (y + 1) * o.Wp() + xx + 1) = pack8(v);
  }
}

// 2x2 average of an FP32 NCHW view into the operand of the next level
__global__ void pool_op_kernel(const float* __restrict__ in, int cs, int coff, int N, Op o) {
  pdl_go();
  pdl_wait();
  const int W2 = o.W * 2, hw2 = 4 * o.H * o.W, hw = o.H * o.W, g = blockIdx.y;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N * hw; i += gridDim.x * blockDim.x) {
    const int n = i / hw, p = i - n * hw, y = p / o.W, x = p - y * o.W;
    const float* q = in + ((long long)n * cs + coff + 8 * g) * hw2 + 2 * y * W2 + 2 * x;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 a = *reinterpret_cast<const float2*>(q + (long long)k * hw2);
      const float2 b = *reinterpret_cast<const float2*>(q + (long long)k * hw2 + W2);
      v[k] = 0.25f * ((a.x + a.y) + (b.x + b.y));
    }
    *op_at(o, g, (long long)n * o.Pn() + (y + 1) * o.Wp() + x + 1) = pack8(v);
  }
}

// nearest 2x upsampling of an operand into channel groups [0, in.C / 8) of another
__global__ void up_op_kernel(Op in, int N, Op o) {
  pdl_go();
  pdl_wait();
  const int hw = in.H * in.W, g = blockIdx.y;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N * hw; i += gridDim.x * blockDim.x) {
    const int n = i / hw, p = i - n * hw, y = p / in.W, x = p - y * in.W;
    const uint4 v = *op_at(in, g, (long long)n * in.Pn() + (y + 1) * in.Wp() + x + 1);
    uint4* d = op_at(o, g, (long long)n * o.Pn() + (2 * y + 1) * o.Wp() + 2 * x + 1);
    d[0] = v;
    d[1] = v;
    d[o.Wp()] = v;
    d[o.Wp() + 1] = v;
  }
}

// Gradient of the upsampling: the sum of four values of an FP32 NCHW view (in), then the epilogue
// (ReLU backward, operand and FP32 copies)
__global__ void up_back_op_kernel(const float* __restrict__ in, int cs, int coff, Epilogue e) {
  pdl_go();
  pdl_wait();
  const int W2 = e.W * 2, hw2 = 4 * e.H * e.W, hw = e.H * e.W, g = blockIdx.y;
  const int Wp = e.W + 2, Pn = ((e.H + 2) * Wp + 15) / 16 * 16;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < e.N * hw; i += gridDim.x * blockDim.x) {
    const int n = i / hw, p = i - n * hw, y = p / e.W, x = p - y * e.W;
    const float* q = in + ((long long)n * cs + coff + 8 * g) * hw2 + 2 * y * W2 + 2 * x;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 a = *reinterpret_cast<const float2*>(q + (long long)k * hw2);
      const float2 b = *reinterpret_cast<const float2*>(q + (long long)k * hw2 + W2);
      v[k] = (a.x + a.y) + (b.x + b.y);
    }
    e.apply(n * Pn + (y + 1) * Wp + x + 1, n, p, 8 * g, v, nullptr);
  }
}

// Gradient of the pooling added to the gradient already there (FP32 NCHW views), then the epilogue
// of the larger image
__global__ void pool_back_op_kernel(const float* __restrict__ in, int cs, int coff, const float* __restrict__ pooled,
                                    int pcs, Epilogue e) {
  pdl_go();
  pdl_wait();
  const int hw = e.H * e.W, Wo = e.W / 2, ho = (e.H / 2) * Wo, g = blockIdx.y;
  const int Wp = e.W + 2, Pn = ((e.H + 2) * Wp + 15) / 16 * 16;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < e.N * hw; i += gridDim.x * blockDim.x) {
    const int n = i / hw, p = i - n * hw, y = p / e.W, x = p - y * e.W;
    const float* s = in + ((long long)n * cs + coff + 8 * g) * hw + p;
    const float* q = pooled + ((long long)n * pcs + 8 * g) * ho + (y >> 1) * Wo + (x >> 1);
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = s[(long long)k * hw] + 0.25f * q[(long long)k * ho];
    e.apply(n * Pn + (y + 1) * Wp + x + 1, n, p, 8 * g, v, nullptr);
  }
}

}  // namespace conv
