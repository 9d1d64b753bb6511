// Depthwise 7 x 7 convolution (unit stride, no dilation, C % 32 == 0) on the warp-level tensor-core
// instruction mma.m16n8k16 (bf16 operands, fp32 accumulation).
//
// One channel's filter row is a band matrix: eight neighbouring outputs of a row are the product of the
// sixteen image pixels under them (fourteen count) and a 16 x 8 matrix holding the seven taps on its
// diagonals.  With sixteen such windows as the rows of A, one instruction does one filter row of 128 outputs
// of one channel (7 of its 16 columns of K are taps: 2.3 multiply-adds issued per useful one), and seven of
// them, one per filter row, reuse the same A fragment for the seven output rows the image row contributes
// to.  tcgen05.mma has no use here: every channel is a matrix product of its own, with N = 8.
//
// Rounding, before the one to bf16: rms error in units of 2^-24 times the sum of the products' magnitudes, on normal /
// widely spread / positive data, against fp64: a chain of 49 fp32 FMAs .163 / .744 / .801, all rows through one
// accumulator .235 / 1.230 / 1.435 (the last with a mean of -1.23: what an MMA drops, it drops towards zero), rows three
// to seven added in fp32 as here .156 / .617 / .730, rows two to seven .147 / .535 / .687.  The additions take 8 % of the
// kernel's time (128 x 56 x 56 x 96: 55.8 -> 60.5 us, all rows added 63.5; 14 x 14 x 384 28.1 -> 29.9).
//
// What bounds it and why: on fp32 FMA pipes the 1.9 G multiply-adds of a 128 x 56 x 56 x 96 tensor take at
// least 52 us, twice what moving the tensor takes (23 us); as band matrices they are 2.3 M instructions, 16 us
// at the 8.4 cycles per scheduler that one takes.  What is left is bringing channels that are neighbours in
// memory into one fragment per channel, which goes through shared memory.
//
// A block of 24 warps (one per SM, persistent) works on 32 channels and 16 windows (numbered over images and
// blocks of eight columns, so any map width fills them) and walks down the image rows:
//   4 warps bring pieces of 8 pixels x 32 channels in by TMA (zero outside the image, 8 rows ahead: at one row
//     ahead the kernel was bound by the latency of its loads) and write each row transposed, channel by
//     channel, to shared memory, where a window is two 16-byte rows of ldmatrix that neighbouring windows share;
//   16 warps of two channels each keep the band matrices (28 registers) and the accumulators of the seven
//     output rows in flight (56) and write each finished row to shared memory;
//   4 warps store finished rows, 64 bytes per pixel.
// The roles meet at mbarriers only.  A warp that gives up on one (after kDw7Polls polls) ends its part, the others run
// into their own limits, and the block computes its outputs again from the image alone.
// Measured on that tensor (us): the fp32 kernel with tiles of outputs per thread 122; without roles and one row of
// loads ahead 72 under ncu, with one set of helper warps 65, as here 61 before the additions above and the votes on
// the waits (1.5).  Now 61.8 between other launches, 128 x 28 x 28 x 192 44.5 (65 in fp32), 14 x 14 x 384 30.4 (36), 7 x 7 x
// 768 22.9 (25).
//
// Zero entries of the band matrix meet pixels outside an output's window.  An infinity or NaN among those
// would turn the output into a NaN, so a block that meets a non-finite accumulator looks at its outputs again at
// the end and computes every NaN among them from the pixels of its own window alone (recompute_output).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "launch.cuh"
#include "layout.cuh"
#include "sm100_ptx.cuh"
#include "ssconv.h"

namespace ssconv {

constexpr int kDw7K = 7;
constexpr int kDw7MainWarps = 16;                   // two channels each
constexpr int kDw7HelperWarps = 4;                  // bring image rows in; as many more carry finished rows out
constexpr int kDw7Threads = 32 * (kDw7MainWarps + 2 * kDw7HelperWarps);
// Registers per thread: 80 at launch (the launch bound's limit), then 96 for the multiplying warps and 48 for the
// helpers, together what the launch allotted.
constexpr int kDw7LaunchRegs = 80, kDw7MainRegs = 96, kDw7HelperRegs = 48;
static_assert(kDw7MainWarps * kDw7MainRegs + 2 * kDw7HelperWarps * kDw7HelperRegs <=
                  (kDw7MainWarps + 2 * kDw7HelperWarps) * kDw7LaunchRegs,
              "a register split above the launch's total never ends");
constexpr uint32_t kDw7Polls = 1u << 20;            // of a barrier, before a warp gives up on it
constexpr int kDw7Channels = 32;                    // per block
constexpr int kDw7Windows = 16;                     // per block: the rows of the MMA
constexpr int kDw7Slots = 2 * kDw7Windows;          // most 8-pixel pieces of a row they touch
constexpr int kDw7ChannelWords = kDw7Slots * 4;     // a channel's staged row, in 32-bit words
// eight words between channels 8 apart: the four lanes that hold a pixel's channels write to different banks
constexpr int kDw7StageWords = kDw7Channels * kDw7ChannelWords + 3 * 8;
constexpr int kDw7OutWords = kDw7Windows * 8 * 17 + 4;
// An MMA aligns its products to the accumulator it adds them to and drops what falls below, so a long chain through
// the accumulator loses more than fp32 additions do.  Filter rows past this one are therefore multiplied by
// themselves and added in fp32, rounded to nearest.
constexpr int kDw7ChainedRows = 2;
constexpr int kDw7RunRows = 8;                      // (see launch_depthwise7)
constexpr int kDw7StageBufs = 3, kDw7OutBufs = 2;
constexpr int kDw7StageBytes = 4 * kDw7StageWords, kDw7OutBytes = 4 * kDw7OutWords;
// image rows as TMA brings them in: kDw7RawRows rows of every 8-pixel piece per copy, 64 bytes per pixel
// (64-byte swizzle), kDw7RawBufs copies of each piece in flight
constexpr int kDw7RawRows = 2, kDw7RawBufs = 4;
constexpr int kDw7RawSlotBytes = kDw7RawRows * 8 * 64;
constexpr int kDw7RawBytes = kDw7Slots * kDw7RawSlotBytes;
// (alignment,) raw rows, staged and finished rows, barriers (full and empty per buffer; raw: one per helper warp
// and buffer), table, bias, flags
constexpr int kDw7SmemBytes = 1024 + kDw7RawBufs * kDw7RawBytes + kDw7StageBufs * kDw7StageBytes + kDw7OutBufs * kDw7OutBytes +
                              8 * (2 * (kDw7StageBufs + kDw7OutBufs) + kDw7HelperWarps * kDw7RawBufs) +
                              4 * (kDw7Windows * 8 + kDw7Channels + 2);

// A finished row in shared memory: pixel col of window w at this word, 16 words of channel pairs.  17 words per
// pixel and one more per four windows: a warp's fragment (8 windows x 4 columns) writes to 32 banks, and two
// windows two apart are read from 32.
__device__ __forceinline__ int dw7_out_word(int w, int col) { return w * (8 * 17) + (w >> 2) + col * 17; }

struct Dw7Params {
  const uint32_t* x;
  const uint32_t* w;
  const float* bias;
  uint32_t* y;
  int N, H, W, C, Ho, Wo, pad;
  long long y_row;          // bytes per output row
  int nblk;                 // windows per output row
  int groups;               // groups of 16 windows (of N nblk)
  int parts;                // thread blocks per unit (a group's 32 channels), each with one run of its rows; or 0:
  int work_quot, work_rem;  // output rows per thread block (of groups * C / 32 * Ho): quotient and remainder
  uint32_t polls;           // kDw7Polls, or fewer in the self-test (0: every wait gives up)
  uint32_t flags;
};

// Polls a phase of an mbarrier at most `polls` times (0: not at all).  Every lane has an answer of its own; the roles go on
// in lock step (ldmatrix, mma, shuffles) and so only branch on what __all_sync makes of it.
__device__ __forceinline__ bool dw7_poll(uint32_t bar, uint32_t parity, uint32_t polls) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 n;\n\t"
      "mov.u32 n, %3;\n\t"
      "setp.ne.u32 p, 0, 0;\n"
      "SPIN:\n\t"
      "setp.eq.u32 q, n, 0;\n\t"
      "@q bra DONE;\n\t"
      "sub.u32 n, n, 1;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@!p bra SPIN;\n"
      "DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(polls)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void lds128(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr)
               : "memory");
}
template <bool FIRST>  // FIRST: d = a b instead of d += a b
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if (FIRST)
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
  else
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// d += r, each sum rounded to nearest, two at a time.
__device__ __forceinline__ void add4(float (&d)[4], const float (&r)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e += 2)
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t}"
        : "+f"(d[e]), "+f"(d[e + 1])
        : "f"(r[e]), "f"(r[e + 1]));
}

// One output of channel pair c2 from its own window's pixels only.
template <bool RELU>
__device__ __forceinline__ uint32_t recompute_output(const Dw7Params& p, int n, int ho, int wo, int c2) {
  const int C2 = p.C >> 1;
  float lo = 0.0f, hi = 0.0f;
  if (p.flags & SSCONV_FLAG_BIAS) {
    lo = p.bias[2 * c2];
    hi = p.bias[2 * c2 + 1];
  }
  for (int kh = 0; kh < kDw7K; ++kh) {
    const int h = ho - p.pad + kh;
    if (h < 0 || h >= p.H) continue;
    for (int kw = 0; kw < kDw7K; ++kw) {
      const int col = wo - p.pad + kw;
      const uint32_t v = (col >= 0 && col < p.W) ? p.x[(((long long)n * p.H + h) * p.W + col) * C2 + c2] : 0u;
      const uint32_t tap = p.w[(kh * kDw7K + kw) * C2 + c2];
      lo = fmaf(bf16_lo(v), bf16_lo(tap), lo);
      hi = fmaf(bf16_hi(v), bf16_hi(tap), hi);
    }
  }
  return RELU ? pack_bf16x2<false>(fmaxf(lo, 0.0f), fmaxf(hi, 0.0f)) : pack_bf16x2<false>(lo, hi);
}

// Consecutive output rows of one group of windows and 32 channels, from row `pos` of the block's range on.
struct Dw7Segment {
  int z, win0, n_first, b_first, h0, S, rows, row0, row1;
  __device__ __forceinline__ Dw7Segment(const Dw7Params& p, int& pos, int end) {
    const int unit = pos / p.Ho;
    h0 = pos - unit * p.Ho;
    S = min(p.Ho - h0, end - pos);
    pos += S;
    z = unit / p.groups;
    win0 = (unit - z * p.groups) * kDw7Windows;
    n_first = win0 / p.nblk;
    b_first = win0 - n_first * p.nblk;
    rows = S + kDw7K - 1;
    // rows [row0, row1) of the segment's are inside the image
    row0 = max(0, p.pad - h0);
    row1 = min(rows, p.H + p.pad - h0);
  }
};

template <bool RELU>
__global__ void __launch_bounds__(kDw7Threads, 1)
depthwise7_mma_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ Dw7Params p) {
  extern __shared__ uint8_t dw_smem_raw[];
  uint8_t* const raw = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dw_smem_raw) + 1023) & ~uintptr_t(1023));
  uint32_t* const stage_words = reinterpret_cast<uint32_t*>(raw + kDw7RawBufs * kDw7RawBytes);
  uint32_t* const out_words = stage_words + kDw7StageBufs * kDw7StageWords;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(out_words + kDw7OutBufs * kDw7OutWords);
  uint64_t* const raw_bars = bars + 2 * (kDw7StageBufs + kDw7OutBufs);
  uint32_t* const out_at = reinterpret_cast<uint32_t*>(raw_bars + kDw7HelperWarps * kDw7RawBufs);  // [column][window]
  float* const bias_s = reinterpret_cast<float*>(out_at + kDw7Windows * 8);
  volatile int* const again = reinterpret_cast<int*>(bias_s + kDw7Channels);  // set: look for NaNs
  volatile int* const failed = again + 1;                                     // set: a wait ran out, compute everything again
  const uint32_t stage0 = smem_u32(stage_words), out0 = smem_u32(out_words);
  // barriers: image row staged, image row read, finished row written, finished row stored
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kDw7StageBufs;
  const uint32_t ofull0 = empty0 + 8 * kDw7StageBufs, oempty0 = ofull0 + 8 * kDw7OutBufs;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);       // (uniform over the warp, and known to be)
  if (tid == 0) {
    *again = *failed = 0;
    for (int b = 0; b < kDw7StageBufs; ++b) {
      mbar_init(bars + b, kDw7HelperWarps);
      mbar_init(bars + kDw7StageBufs + b, kDw7MainWarps);
    }
    for (int b = 0; b < kDw7OutBufs; ++b) {
      mbar_init(bars + 2 * kDw7StageBufs + b, kDw7MainWarps);
      mbar_init(bars + 2 * kDw7StageBufs + kDw7OutBufs + b, kDw7HelperWarps);
    }
    for (int b = 0; b < kDw7HelperWarps * kDw7RawBufs; ++b) mbar_init(raw_bars + b, 1);
    mbar_fence_init();
    prefetch_tensormap(&tm_x);
  }
  const int blk = (int)blockIdx.x;
  int pos, end;
  if (p.parts != 0) {
    const int unit = blk / p.parts, part = blk - unit * p.parts;
    pos = unit * p.Ho + part * p.Ho / p.parts;
    end = unit * p.Ho + (part + 1) * p.Ho / p.parts;
  } else {
    pos = blk * p.work_quot + min(blk, p.work_rem);
    end = pos + p.work_quot + (blk < p.work_rem ? 1 : 0);
  }
  grid_launch_dependents();
  grid_dependency_wait();  // (loads below it are plain ones: read-only loads could be moved above it)
  __syncthreads();

  // Every role walks the block's segments; three block barriers per segment: tables written, outputs stored, done.
  // Buffers in use and the parity of their barriers are carried on over segments.
  uint32_t sbuf = 0, sphase = 0, obuf = 0, ophase = 0;
  bool ok = true;
  if (warp < kDw7MainWarps) {
    // ------------------------------------------------------------------ multiplications and epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kDw7MainRegs));
    const int g = lane >> 2, t = lane & 3;                      // fragment row and column group
    while (pos < end) {
      const Dw7Segment sg(p, pos, end);
      if (tid < kDw7Windows * 8) {  // where outputs go, in units of 64 bytes (a block's channels of a pixel); ~0: outside
        const int win = sg.win0 + (tid & 15), n = win / p.nblk, wo = 8 * (win - n * p.nblk) + (tid >> 4);
        out_at[tid] = (n < p.N && wo < p.Wo)
                          ? (uint32_t)((((long long)n * p.Ho + sg.h0) * p.Wo + wo) * (p.C / kDw7Channels) + sg.z)
                          : ~0u;
      }
      if (tid < kDw7Channels) bias_s[tid] = (p.flags & SSCONV_FLAG_BIAS) ? p.bias[sg.z * kDw7Channels + tid] : 0.0f;
      // the two channels' band matrices: B[k][n] = tap k - n of the filter row, n = g
      uint32_t band[2][kDw7K][2];
      {
        const int C2 = p.C >> 1;
        const uint32_t* w = p.w + sg.z * (kDw7Channels / 2) + warp;
#pragma unroll
        for (int kh = 0; kh < kDw7K; ++kh) {
          uint32_t v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int kw = 2 * t + (e & 1) + 8 * (e >> 1) - g;
            v[e] = (kw >= 0 && kw < kDw7K) ? w[(kh * kDw7K + kw) * C2] : 0u;
          }
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            band[0][kh][half] = __byte_perm(v[2 * half], v[2 * half + 1], 0x5410);
            band[1][kh][half] = __byte_perm(v[2 * half], v[2 * half + 1], 0x7632);
          }
        }
      }
      // ldmatrix address: matrices 0, 1 = windows 0-7, 8-15 on their first 8 pixels, 2, 3 on the next 8
      const int lw = lane & 15;
      const int lslot = lw + (sg.win0 + lw) / p.nblk - sg.n_first + (lane >> 4);
      const uint32_t a_addr = stage0 + 4u * ((2 * warp) * kDw7ChannelWords + (warp >> 2) * 8 + 4 * lslot);
      const uint32_t out_dst = out0 + 4u * (dw7_out_word(g, 2 * t) + warp);
      const uint32_t bias_at = smem_u32(bias_s) + 8u * warp;
      __syncthreads();
      float acc[2][kDw7K][4];
#pragma unroll
      for (int o = 0; o < kDw7K; ++o)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[0][o][e] = acc[1][o][e] = 0.0f;
      const int rows = sg.rows, row0 = sg.row0, row1 = sg.row1;
      for (int r0 = 0; r0 < rows && ok; r0 += kDw7K) {
#pragma unroll
        for (int ph = 0; ph < kDw7K; ++ph) {  // (unrolled: the accumulator of output row o is o mod 7)
          const int r = r0 + ph;
          if (r >= rows || !ok) break;
          bool got = true;
          // Image row r under filter row kh is output row r - kh.  (Rows before the segment's first are dropped
          // below, rows past its last never leave the accumulators.)
          if (r >= row0 && r < row1) {
            got = dw7_poll(full0 + 8u * sbuf, sphase, p.polls);  // (if it gives up: every output is computed again below)
            uint32_t a[2][4];
            ldmatrix_x4(a_addr + sbuf * kDw7StageBytes, a[0]);
            ldmatrix_x4(a_addr + sbuf * kDw7StageBytes + 4u * kDw7ChannelWords, a[1]);
            if (lane == 0) mbar_arrive_a(empty0 + 8u * sbuf);
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
              // (the row's oldest output first: the epilogue below waits for it)
#pragma unroll
              for (int kh = kDw7K - 1; kh > 0; --kh) {
                float(&d)[4] = acc[ch][(ph - kh + kDw7K) % kDw7K];
                if (kh <= kDw7ChainedRows) {
                  mma_bf16_16816<false>(d, a[ch], band[ch][kh][0], band[ch][kh][1]);
                } else {
                  float row[4];
                  mma_bf16_16816<true>(row, a[ch], band[ch][kh][0], band[ch][kh][1]);
                  add4(d, row);
                }
              }
              mma_bf16_16816<true>(acc[ch][ph], a[ch], band[ch][0][0], band[ch][0][1]);
            }
            if (++sbuf == kDw7StageBufs) {
              sbuf = 0;
              sphase ^= 1u;
            }
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[0][ph][e] = acc[1][ph][e] = 0.0f;
          }
          if (r >= kDw7K - 1) {  // the output row this image row completes
            float(&d0)[4] = acc[0][(ph + 1) % kDw7K];
            float(&d1)[4] = acc[1][(ph + 1) % kDw7K];
            const float bias0 = __uint_as_float(lds32(bias_at)), bias1 = __uint_as_float(lds32(bias_at + 4u));
            got = dw7_poll(oempty0 + 8u * obuf, ophase ^ 1u, p.polls) && got;
            const uint32_t o = out_dst + obuf * kDw7OutBytes;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              d0[e] += bias0;
              d1[e] += bias1;
              sts32(o + 4u * ((e >> 1) * (8 * 8 * 17 + 2) + (e & 1) * 17), pack_bf16x2<RELU>(d0[e], d1[e]));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive_a(ofull0 + 8u * obuf);
            if (++obuf == kDw7OutBufs) {
              obuf = 0;
              ophase ^= 1u;
            }
            // a NaN among the eight makes their sum one (a sum that is infinite only costs the second look)
            const float sum = ((d0[0] + d0[1]) + (d0[2] + d0[3])) + ((d1[0] + d1[1]) + (d1[2] + d1[3]));
            if (!(fabsf(sum) <= 3.0e38f)) *again = 1;
          }
          ok = __all_sync(0xFFFFFFFFu, got);
        }
      }
      if (!ok) *failed = 1;
      __syncthreads();  // (also: this block's stores are visible to all its threads)
      if (*again != 0 || *failed != 0) {
        for (int i = tid; i < sg.S * kDw7Windows * 8 * (kDw7Channels / 2); i += 32 * kDw7MainWarps) {
          const int word = i & 15, at_col = (i >> 4) & 7, w = (i >> 7) & 15, o = i >> 11;
          const uint32_t at = out_at[at_col * 16 + w];
          if (at == ~0u) continue;
          uint32_t* const dst = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(p.y + word) + 64ull * at + o * p.y_row);
          const uint32_t v = *dst;
          if (*failed == 0 && (v & 0x7FFFu) <= 0x7F80u && (v & 0x7FFF0000u) <= 0x7F800000u) continue;  // neither is a NaN
          const int win = sg.win0 + w, n = win / p.nblk;
          *dst = recompute_output<RELU>(p, n, sg.h0 + o, 8 * (win - n * p.nblk) + at_col, sg.z * (kDw7Channels / 2) + word);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kDw7MainWarps) : "memory");
        if (tid == 0) *again = 0;
      }
      __syncthreads();  // (the next segment writes the table)
    }
  } else if (warp < kDw7MainWarps + kDw7HelperWarps) {
    // ------------------------------------------------------------------ image rows in
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kDw7HelperRegs));
    const int ht = tid - 32 * kDw7MainWarps, hw = warp - kDw7MainWarps;
    uint32_t rbuf = 0, rphase = 0;
    uint32_t in_flight = 0;                                     // copies issued and not used up
    while (pos < end) {
      const Dw7Segment sg(p, pos, end);
      // A warp brings in pieces 2 hw, 2 hw + 1, 2 hw + 8, ... of the rows by itself: lane l < 8 copies piece
      // 2 hw + l % 2 + 8 (l / 2), zero outside the image, kDw7RawRows rows at a time.
      const int slots = kDw7Windows + 1 + (sg.win0 + kDw7Windows - 1) / p.nblk - sg.n_first;  // (pieces in use)
      const int my_slot = 2 * hw + (lane & 1) + 8 * (lane >> 1);
      const bool my_copy = lane < 8 && my_slot < slots;
      const uint32_t copies = __popc(__ballot_sync(0xffffffffu, my_copy));  // (at least two: slots >= 17)
      const int my_piece = my_slot + sg.b_first;                // an image has nblk + 1 pieces per row
      const int my_n = sg.n_first + my_piece / (p.nblk + 1), my_col = 8 * (my_piece % (p.nblk + 1)) - p.pad;
      const uint32_t raw0 = smem_u32(raw), raw_bar0 = smem_u32(raw_bars) + 8u * kDw7RawBufs * hw;
      int row_next = sg.row0;                                   // first row of the next copy
      uint32_t cbuf = rbuf;
      auto copy_rows = [&]() {  // (all lanes; the buffer's last rows have been read)
        if (row_next >= sg.row1 || !ok) return;
        const uint32_t bar = raw_bar0 + 8u * cbuf;
        if (lane == 0) mbar_expect_tx_a(bar, copies * kDw7RawSlotBytes);
        __syncwarp();
        if (my_copy)
          tma_load_4d_a(raw0 + cbuf * kDw7RawBytes + my_slot * kDw7RawSlotBytes, &tm_x, bar, sg.z * kDw7Channels, my_col,
                        sg.h0 - p.pad + row_next, my_n);
        row_next += kDw7RawRows;
        ++in_flight;
        cbuf = (cbuf + 1 == kDw7RawBufs) ? 0u : cbuf + 1;
      };
      for (int k = 0; k < kDw7RawBufs; ++k) copy_rows();
      // staging: pixels 2 q, 2 q + 1 of pieces s0 + 8 k, channels [8 cc, 8 cc + 8).  Lanes of odd q read the
      // second pixel first (eight lanes then read 128 bytes on different banks).
      const int cc = ht & 3, q = (ht >> 2) & 3, s0 = ht >> 4;
      const uint32_t raw_src = raw0 + s0 * kDw7RawSlotBytes + (2 * q) * 64 + 16 * (cc ^ q);
      const uint32_t first = (q & 1) ? 64u : 0u;
      const uint32_t sel_lo = (q & 1) ? 0x1054u : 0x5410u, sel_hi = (q & 1) ? 0x3276u : 0x7632u;
      const uint32_t st_dst = stage0 + 4u * (8 * cc * kDw7ChannelWords + 8 * cc + 4 * s0 + q);
      __syncthreads();
      for (int r = sg.row0; r < sg.row1 && ok; ++r) {
        const int sub = (r - sg.row0) % kDw7RawRows;
        bool got = sub != 0 || dw7_poll(raw_bar0 + 8u * rbuf, rphase, p.polls);
        got = dw7_poll(empty0 + 8u * sbuf, sphase ^ 1u, p.polls) && got;
        ok = __all_sync(0xFFFFFFFFu, got);
        if (!ok) break;
        const uint32_t src = raw_src + rbuf * kDw7RawBytes + sub * 512u;
#pragma unroll
        for (int k2 = 0; k2 < 4; k2 += 2) {
          if (8 * k2 >= slots) break;
          uint32_t a[2][4], b[2][4];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            lds128(src + 8u * (k2 + k) * kDw7RawSlotBytes + first, a[k]);
            lds128(src + 8u * (k2 + k) * kDw7RawSlotBytes + (64u - first), b[k]);
          }
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (8 * (k2 + k) >= slots) break;
            const uint32_t d = st_dst + sbuf * kDw7StageBytes + 4u * 32 * (k2 + k);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              sts32(d + 4u * (2 * i) * kDw7ChannelWords, __byte_perm(a[k][i], b[k][i], sel_lo));
              sts32(d + 4u * (2 * i + 1) * kDw7ChannelWords, __byte_perm(a[k][i], b[k][i], sel_hi));
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_a(full0 + 8u * sbuf);
        if (++sbuf == kDw7StageBufs) {
          sbuf = 0;
          sphase ^= 1u;
        }
        if (sub == kDw7RawRows - 1 || r + 1 == sg.row1) {  // the copy is used up
          --in_flight;
          copy_rows();
          if (++rbuf == kDw7RawBufs) {
            rbuf = 0;
            rphase ^= 1u;
          }
        }
      }
      if (!ok) {
        // Copies that are under way land before the block goes on (it may be at its end): no more are issued, and
        // each of these is waited for, with the full limit, in the order of their buffers.
        for (; in_flight != 0; --in_flight) {
          dw7_poll(raw_bar0 + 8u * rbuf, rphase, kDw7Polls);
          if (++rbuf == kDw7RawBufs) {
            rbuf = 0;
            rphase ^= 1u;
          }
        }
        *failed = 1;
      }
      __syncthreads();
      __syncthreads();
    }
  } else {
    // ------------------------------------------------------------------ finished rows out
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kDw7HelperRegs));
    const int hw = warp - kDw7MainWarps - kDw7HelperWarps;
    // a warp stores the words of columns hw, hw + 4 of windows w2, w2 + 4, ... and w2 + 1, w2 + 5, ...
    const int w2 = 2 * (lane >> 4);
    const uint32_t out_src = out0 + 4u * (dw7_out_word(w2, hw) + (lane & 15));
    const uint32_t out_tab = smem_u32(out_at) + 4u * (hw * 16 + w2);
    while (pos < end) {
      const Dw7Segment sg(p, pos, end);
      char* y_row = reinterpret_cast<char*>(p.y + (lane & 15));
      __syncthreads();
      for (int o = 0; o < sg.S && ok; ++o) {
        ok = __all_sync(0xFFFFFFFFu, dw7_poll(ofull0 + 8u * obuf, ophase, p.polls));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t to[8], w[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {  // windows w2 + 4 (k / 2) + k % 2
            to[k] = lds32(out_tab + 4u * (64 * c + 4 * (k >> 1) + (k & 1)));
            w[k] = lds32(out_src + obuf * kDw7OutBytes + 4u * (4 * c * 17 + (k >> 1) * (4 * 8 * 17 + 1) + (k & 1) * 8 * 17));
          }
          if (c == 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive_a(oempty0 + 8u * obuf);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (to[k] != ~0u) *reinterpret_cast<uint32_t*>(y_row + 64ull * to[k]) = w[k];
        }
        y_row += p.y_row;
        if (++obuf == kDw7OutBufs) {
          obuf = 0;
          ophase ^= 1u;
        }
      }
      if (!ok) *failed = 1;
      __syncthreads();
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------------------
// Small maps
// ---------------------------------------------------------------------------------------
// A few images' maps give the kernel above one short run of rows per block: 9 us of start-up (six image rows before the first
// output row, rows handed from role to role), whatever the map holds.  Here a block of 128 threads makes 4 x 8 outputs of 32
// channels: all it needs, 10 x 14 pixels and the filter, is loaded at once (one latency), and a thread then computes four
// neighbouring outputs of one pair of channels from shared memory with fp32 multiply-adds, a filter row at a time (each row a
// chain of its own, added to the sum: rms error in the units above .109 / .469 / .448).  Bound by that one latency and 196
// multiply-adds per thread while the blocks are resident at once; every pixel is loaded 4.4 times, so larger maps are not
// for it.  us between other launches, tensor-core kernel / this one: 3 x 56 x 56 x 96 9.3 / 5.8, 3 x 28 x 28 x 192 8.8 / 4.5,
// 3 x 14 x 14 x 384 8.8 / 3.2, 3 x 7 x 7 x 768 8.1 / 2.6; with 64 threads of eight outputs each 5.6, 4.5, 3.4, 3.3.
constexpr int kDwSmallH = 4, kDwSmallW = 8, kDwSmallRun = 4;
constexpr int kDwSmallThreads = 16 * kDwSmallH * (kDwSmallW / kDwSmallRun);
constexpr int kDwSmallRows = kDwSmallH + kDw7K - 1, kDwSmallCols = kDwSmallW + kDw7K - 1;
constexpr int kDwSmallPixel = 20;  // words from pixel to pixel: the two runs of a warp, four pixels apart, read different banks
constexpr int kDwSmallSharedBytes = 4 * kDwSmallRows * kDwSmallCols * kDwSmallPixel + 8 * kDw7K * kDw7K * 16;
template <bool RELU>
__global__ void __launch_bounds__(kDwSmallThreads) depthwise7_small_kernel(const Dw7Params p, int tiles_h, int tiles_w) {
  __shared__ __align__(16) uint32_t px[kDwSmallRows * kDwSmallCols * kDwSmallPixel];
  __shared__ float2 w_s[kDw7K * kDw7K][16];
  grid_launch_dependents();
  const int t = threadIdx.x, C8 = p.C >> 3;
  int tile = blockIdx.x;
  const int tw = tile % tiles_w;
  tile /= tiles_w;
  const int th = tile % tiles_h;
  const int n = tile / tiles_h;
  const int h0 = th * kDwSmallH, w0 = tw * kDwSmallW;
  const int c8 = blockIdx.y * (kDw7Channels / 8);
  const uint4* x4 = reinterpret_cast<const uint4*>(p.x) + c8;
  const uint4* w4 = reinterpret_cast<const uint4*>(p.w) + c8;
  grid_dependency_wait();
  constexpr int kVecs = kDwSmallRows * kDwSmallCols * 4, kLoads = (kVecs + kDwSmallThreads - 1) / kDwSmallThreads;
  constexpr int kWVecs = kDw7K * kDw7K * 4, kWLoads = (kWVecs + kDwSmallThreads - 1) / kDwSmallThreads;
  uint4 v[kLoads], wv[kWLoads];
#pragma unroll
  for (int j = 0; j < kLoads; ++j) {
    const int i = t + j * kDwSmallThreads, pixel = i >> 2;
    const int r = pixel / kDwSmallCols, h = h0 - p.pad + r, col = w0 - p.pad + pixel - r * kDwSmallCols;
    v[j] = make_uint4(0u, 0u, 0u, 0u);
    if (i < kVecs && h >= 0 && h < p.H && col >= 0 && col < p.W)
      v[j] = x4[(((long long)n * p.H + h) * p.W + col) * C8 + (i & 3)];
  }
#pragma unroll
  for (int j = 0; j < kWLoads; ++j) {
    const int i = t + j * kDwSmallThreads;
    wv[j] = i < kWVecs ? w4[(long long)(i >> 2) * C8 + (i & 3)] : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int j = 0; j < kLoads; ++j) {
    const int i = t + j * kDwSmallThreads;
    if (i < kVecs) *reinterpret_cast<uint4*>(px + (i >> 2) * kDwSmallPixel + 4 * (i & 3)) = v[j];
  }
#pragma unroll
  for (int j = 0; j < kWLoads; ++j) {
    const int i = t + j * kDwSmallThreads;
    if (i < kWVecs) {
      float2* dst = &w_s[i >> 2][4 * (i & 3)];
      dst[0] = make_float2(bf16_lo(wv[j].x), bf16_hi(wv[j].x));
      dst[1] = make_float2(bf16_lo(wv[j].y), bf16_hi(wv[j].y));
      dst[2] = make_float2(bf16_lo(wv[j].z), bf16_hi(wv[j].z));
      dst[3] = make_float2(bf16_lo(wv[j].w), bf16_hi(wv[j].w));
    }
  }
  __syncthreads();
  const int sub = t & 15, run = (t >> 4) & 1, o = t >> 5;
  const int ho = h0 + o, wo0 = w0 + run * kDwSmallRun, c2 = blockIdx.y * 16 + sub;
  if (ho >= p.Ho || wo0 >= p.Wo) return;
  float2 acc[kDwSmallRun];
  {
    float2 b = make_float2(0.0f, 0.0f);
    if (p.flags & SSCONV_FLAG_BIAS) b = make_float2(p.bias[2 * c2], p.bias[2 * c2 + 1]);
#pragma unroll
    for (int k = 0; k < kDwSmallRun; ++k) acc[k] = b;
  }
#pragma unroll 1
  for (int kh = 0; kh < kDw7K; ++kh) {
    const int h = ho - p.pad + kh;
    if (h < 0 || h >= p.H) continue;
    const uint32_t* row = px + ((o + kh) * kDwSmallCols + run * kDwSmallRun) * kDwSmallPixel + sub;
    float2 xv[kDwSmallRun + kDw7K - 1], part[kDwSmallRun];
#pragma unroll
    for (int col = 0; col < kDwSmallRun + kDw7K - 1; ++col) {
      const uint32_t u = row[col * kDwSmallPixel];
      xv[col] = make_float2(bf16_lo(u), bf16_hi(u));
    }
#pragma unroll
    for (int kw = 0; kw < kDw7K; ++kw) {
      const float2 wk = w_s[kh * kDw7K + kw][sub];
#pragma unroll
      for (int k = 0; k < kDwSmallRun; ++k)
        part[k] = kw == 0 ? __fmul2_rn(xv[k], wk) : __ffma2_rn(xv[k + kw], wk, part[k]);
    }
#pragma unroll
    for (int k = 0; k < kDwSmallRun; ++k) acc[k] = __fadd2_rn(acc[k], part[k]);
  }
  uint32_t* out = p.y + (((long long)n * p.Ho + ho) * p.Wo + wo0) * (p.C >> 1) + c2;
#pragma unroll
  for (int k = 0; k < kDwSmallRun; ++k)
    if (wo0 + k < p.Wo)
      out[(long long)k * (p.C >> 1)] =
          RELU ? pack_bf16x2<false>(fmaxf(acc[k].x, 0.0f), fmaxf(acc[k].y, 0.0f)) : pack_bf16x2<false>(acc[k].x, acc[k].y);
}

static int g_tune_mma = -1;    // ssconv_tune: -1 automatic, 0 neither of the two kernels here
static int g_tune_small = -1;  // -1 automatic, 0 never the small maps' kernel
int32_t set_depthwise_tuning(int32_t option, int32_t value) {
  if (value != -1 && value != 0) return SSCONV_ERR_BAD_DESC;
  (option == SSCONV_TUNE_DEPTHWISE_SMALL ? g_tune_small : g_tune_mma) = value;
  return SSCONV_OK;
}

// Layers for this kernel; for the others the caller goes on to the fp32 kernels.  Maps of a few pixels are among the others:
// their windows are mostly empty, and this kernel's start-up is longer than what the fp32 kernel takes for all of it.
// Up to 64 pixels the line is the number of blocks: from about half the SMs on, the copies of empty windows are slow.  us,
// this kernel / the fp32 tiles: 1 x 3 x 3 x 768 7.0 / 5.6, 60 x 2 x 2 x 768 6.5 / 5.5; 84 blocks 1 x 7 x 7 x 384 10.2 / 8.8, 96
// blocks 4 x 4 x 4 x 768 8.1 / 7.0, 144 blocks 1 x 7 x 7 x 768 11.3 / 8.8.  Beyond the lines: 72 blocks 1 x 6 x 6 x 384 8.0 / 9.4, 60
// blocks 1 x 5 x 5 x 384 7.8 / 8.5, 98 pixels 2 x 7 x 7 x 768 8.0 / 8.8, 8 x 4 x 4 x 768 7.0 / 7.0, 32 x 4 x 4 x 768 7.3 / 9.2.
static bool depthwise7_applies(int N, int H, int W, int C, int Ho, int Wo, int KH, int KW, int stride, int dil) {
  if (KH != kDw7K || KW != kDw7K || stride != 1 || dil != 1 || C % kDw7Channels != 0 || g_tune_mma == 0) return false;
  if (Ho <= 3 && Wo <= 8) return false;
  if ((long long)N * Ho * Wo <= 64 && (long long)Ho * (C / kDw7Channels) > 72) return false;
  return (long long)N * Ho * Wo * (C / kDw7Channels) < 0xFFFFFFFFll && (long long)H * W * C < (1ll << 38) &&
         (long long)N * ((Wo + 7) / 8) * (C / kDw7Channels) * Ho < 0x7FFFFFF0ll / 2;
}

// The kernel's SM count on the current device, after it has been made ready there; 0 in *sms: not to be run, because this
// build of it was given another number of registers than its split between the roles counts on (a debug build, another
// compiler).
static cudaError_t depthwise7_ready(bool relu, int* sms) {
  const auto kernel = relu ? depthwise7_mma_kernel<true> : depthwise7_mma_kernel<false>;
  static std::atomic<int> known[64][2];  // SM count + 1 per device and form, 0: not looked at yet
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool keep = dev >= 0 && dev < 64;
  const int k = keep ? known[dev][relu].load(std::memory_order_relaxed) : 0;
  if (k != 0) {
    *sms = k - 1;
    return cudaSuccess;
  }
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  *sms = 0;
  if (fa.numRegs == kDw7LaunchRegs) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDw7SmemBytes);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  if (keep) known[dev][relu].store(*sms + 1, std::memory_order_relaxed);
  return cudaSuccess;
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Blocks of depthwise7_small_kernel for a map, and the most per SM that it is used for.  us on 148 SMs, tensor-core kernel /
// small: 1152 blocks 12 x 14 x 14 x 384 9.7 / 6.9, 1536 blocks 32 x 7 x 7 x 768 8.5 / 8.3, 1764 blocks 6 x 56 x 56 x 96 10.0 /
// 10.1, 2304 blocks 24 x 14 x 14 x 384 10.5 / 11.7.
constexpr int kDwSmallMaxBlocksPerSm = 10;
static long long depthwise7_small_blocks(int N, int C, int Ho, int Wo) {
  return (long long)N * ((Ho + kDwSmallH - 1) / kDwSmallH) * ((Wo + kDwSmallW - 1) / kDwSmallW) * (C / kDw7Channels);
}
// A grid that starts while the one before it drains puts its blocks where that one leaves first, as many as fit: up to a
// dozen on some SMs and none on others.  So much shared memory per block that an even share of the blocks fits on an SM
// spreads them.  us without it and with: 3 x 56 x 56 x 96 7.9 / 5.8, 3 x 28 x 28 x 192 6.8 / 4.5, 3 x 14 x 14 x 384 4.4 / 3.2.
constexpr int kSmSharedBytes = 228 * 1024, kMaxBlockSharedBytes = 232448, kBlockReservedBytes = 1024;
static cudaError_t launch_depthwise7_small(const Dw7Params& p, cudaStream_t st) {
  const int tiles_h = (p.Ho + kDwSmallH - 1) / kDwSmallH, tiles_w = (p.Wo + kDwSmallW - 1) / kDwSmallW;
  const dim3 grid((unsigned)(p.N * tiles_h * tiles_w), (unsigned)(p.C / kDw7Channels));
  const bool relu = (p.flags & SSCONV_FLAG_RELU) != 0;
  const auto kernel = relu ? depthwise7_small_kernel<true> : depthwise7_small_kernel<false>;
  static std::atomic<int> known[64][2];  // per device and form: SM count, once the kernel may take all shared memory
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int sms = dev >= 0 && dev < 64 ? known[dev][relu].load(std::memory_order_relaxed) : 0;
  if (sms == 0) {
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBlockSharedBytes - kDwSmallSharedBytes);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) known[dev][relu].store(sms, std::memory_order_relaxed);
  }
  const long long blocks = (long long)grid.x * grid.y;
  const int per_sm = (int)((blocks + sms - 1) / sms);
  int extra = kSmSharedBytes / per_sm - kBlockReservedBytes - kDwSmallSharedBytes;
  if (extra > kMaxBlockSharedBytes - kDwSmallSharedBytes) extra = kMaxBlockSharedBytes - kDwSmallSharedBytes;
  count_launch();
  return launch_dependent_smem(kernel, grid, kDwSmallThreads, extra > 0 ? (size_t)(extra & ~127) : 0, st, p, tiles_h, tiles_w);
}

static cudaError_t launch_depthwise7_on(int sms, const void* x, const void* w, const float* bias, void* y, int N, int H, int W,
                                        int C, int Ho, int Wo, int pad, uint32_t flags, uint32_t polls, cudaStream_t st) {
  Dw7Params p;
  p.x = static_cast<const uint32_t*>(x);
  p.w = static_cast<const uint32_t*>(w);
  p.bias = bias;
  p.y = static_cast<uint32_t*>(y);
  p.N = N;
  p.H = H;
  p.W = W;
  p.C = C;
  p.Ho = Ho;
  p.Wo = Wo;
  p.pad = pad;
  p.y_row = 2ll * Wo * C;
  p.nblk = (Wo + 7) / 8;
  p.groups = (N * p.nblk + kDw7Windows - 1) / kDw7Windows;
  p.polls = polls;
  p.flags = flags;
  const auto kernel = (flags & SSCONV_FLAG_RELU) ? depthwise7_mma_kernel<true> : depthwise7_mma_kernel<false>;
  // Output rows are dealt out evenly, a block walking a contiguous range of (32 channels, group of windows, row) that may
  // cross from one unit into the next; or, where there are no more units than SMs, every unit is cut into the same
  // number of runs and a block has one of them.  A run starts with six image rows for its first output row and with
  // filling the pipeline, together worth about kDw7RunRows output rows, so that two short runs in a block cost more than
  // a longer one.  us, dealt out evenly -> in runs: 3 x 7 x 7 x 768 12.5 -> 7.9, 12 x 14 x 14 x 384 13.3 -> 9.6,
  // 24 x 28 x 28 x 192 15.5 -> 12.8, 96 x 14 x 14 x 384 21.2 -> 15.9; 64 x 56 x 56 x 96 stays with even ranges (35.3; 57 %
  // of the SMs would have a run).
  const int units = p.groups * (C / kDw7Channels);
  const long long work = (long long)units * Ho;
  const int even = (int)(work < sms ? work : sms);
  p.work_quot = (int)(work / even);
  p.work_rem = (int)(work % even);
  p.parts = 0;
  if (units <= sms) {
    const int rows = p.work_quot + (p.work_rem != 0 ? 1 : 0);
    const int runs = (rows == 1 || (p.work_rem == 0 && Ho % rows == 0)) ? 1 : (rows - 2) / Ho + 2;  // at most, of a block
    const int parts = sms / units < Ho ? sms / units : Ho;
    if ((Ho + parts - 1) / parts + kDw7RunRows < rows + runs * kDw7RunRows) p.parts = parts;
  }
  const int blocks = p.parts != 0 ? units * p.parts : even;
  CUtensorMap tm_x;
  {
    static EncodeFn encode = nullptr;  // (every thread finds the same function)
    if (encode == nullptr) {
      void* f = nullptr;
      cudaDriverEntryPointQueryResult q;
      const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q);
      if (e != cudaSuccess) return e;
      if (q != cudaDriverEntryPointSuccess || f == nullptr) return cudaErrorNotSupported;
      encode = reinterpret_cast<EncodeFn>(f);
    }
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    const cuuint64_t strides[3] = {2ull * C, 2ull * C * W, 2ull * C * W * H};
    const cuuint32_t box[4] = {kDw7Channels, 8, kDw7RawRows, 1}, estr[4] = {1, 1, 1, 1};
    if (encode(&tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kDw7Threads);
  cfg.dynamicSmemBytes = kDw7SmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, tm_x, p);
}

// False: not a layer for this kernel, nothing has been launched.  polls: of a barrier, -1 = kDw7Polls.
bool launch_depthwise7(const void* x, const void* w, const float* bias, void* y, int N, int H, int W, int C, int Ho, int Wo,
                       int KH, int KW, int stride, int pad, int dil, uint32_t flags, int32_t polls, cudaStream_t st,
                       cudaError_t* result) {
  if (polls < 0 && KH == kDw7K && KW == kDw7K && stride == 1 && dil == 1 && C % kDw7Channels == 0 && g_tune_mma != 0 &&
      g_tune_small != 0 && depthwise7_small_blocks(N, C, Ho, Wo) <= kDwSmallMaxBlocksPerSm * device_sms()) {
    Dw7Params p{};
    p.x = static_cast<const uint32_t*>(x);
    p.w = static_cast<const uint32_t*>(w);
    p.bias = bias;
    p.y = static_cast<uint32_t*>(y);
    p.N = N;
    p.H = H;
    p.W = W;
    p.C = C;
    p.Ho = Ho;
    p.Wo = Wo;
    p.pad = pad;
    p.flags = flags;
    *result = launch_depthwise7_small(p, st);
    return true;
  }
  if (!depthwise7_applies(N, H, W, C, Ho, Wo, KH, KW, stride, dil)) return false;
  const bool relu = (flags & SSCONV_FLAG_RELU) != 0;
  int sms = 0;
  *result = depthwise7_ready(relu, &sms);
  if (*result != cudaSuccess) return true;
  if (sms == 0) return false;
  *result = launch_depthwise7_on(sms, x, w, bias, y, N, H, W, C, Ho, Wo, pad, flags, polls < 0 ? kDw7Polls : (uint32_t)polls,
                                 st);
  return true;
}

}  // namespace ssconv
