// Block FFT of B complex points (complex64 or complex128) held by one thread block: B/16 threads, 16 points per
// thread, decimation in time through shared memory in place: a radix-16 stage on registers, a
// radix-RM stage (RM = 2, 4 or 8) when log2(B) is not a multiple of 4, then radix-16 stages
// (B = 128: no more).
//
// Locations l hold the input in digit-reversed order.  Stage with radix R and S = product of the
// earlier radices works on the points l = hi S R + t S + lo (lo < S):
//   a[t] = w^(t lo) x[l(t)],  w = exp(sign 2 pi i / (S R)),  x[l(t)] = DFT_R(a)[t],
// and leaves the result in natural order after the last stage.  A butterfly writes the
// locations it read, so a stage needs no barrier between its reads and its writes: one barrier
// per exchange (an autosort form needs two), and the warps of a block overlap their loads,
// butterflies and stores inside a stage.  Measured against the autosort form, with the magnitudes
// of the window peaks in a region of their own (os_tail.cuh), on one GB300: 256 neighbours at
// n = 2^20 in two buckets 1690 -> 1637 us, the 32768-point two-phase tails of 96 long kernels at
// n = 2^23 10.2 -> 9.7 ms with the rest of that call, matched filters 1.5%.  A barrier of only the
// 256 threads that exchange data between the middle stages was slower (1694 us): the drifted
// warps spread one block's loads over its neighbour phases.
//
// Input: before the call, thread `tid` holds v[t] = x[tid + t B/16] for t < 16.
// Output: after it, thread `tid` holds v[t] = X[tid + t B/16].
// Shared memory: location l is stored at l + PAD (l / (B/16)), B + 16 PAD values.  The 16 lanes of
// the first stage's writes are B/16 locations apart; PAD keeps them 16 bytes apart modulo the
// banks (PAD = 2 for complex64, written two at a time, 1 for complex128), so that eight lanes of
// 128-bit stores fill a wavefront.  The later stages touch runs of 16 locations.
//
// Twiddles come from per-stage tables laid out in thread order: the stage with radix R and S has
// a table of R S entries, entry t S + k = exp(-2 pi i t k / (R S)), so the loads of a warp are
// contiguous.  In FP32 a radix-16 stage reads the rows t = 1 and 4 and forms the other powers by
// complex products; in FP64, whose pipe is the scarce one, it reads every row.  The tables of the stages after the first follow each other; a block size B needs
// block_table_size<B>() entries (built on the host by block_fft_tables).
#pragma once

#include "cplx.cuh"

namespace rf {

// The powers w[t], 0 < t < R (R = 4, 8 or 16), of which table entry t * stride is w^t: the
// entries t = 1 and (R >= 8) 4 are loaded and the others formed by complex products (w^2 = w w,
// w^8 = w^4 w^4, at most three products deep: a few ulp), which keeps 13 of the 15 table loads of
// a radix-16 stage off the load/store pipe, the scarcer one in the block transforms (loading all
// 15 made the 2^23-sample step 12% slower, loading 4 was 2% slower).
template <int R, typename V>
__device__ __forceinline__ void stage_twiddles(V (&w)[R], const V* __restrict__ tw, int stride) {
  static_assert(R == 2 || R == 4 || R == 8 || R == 16, "radix");
  if constexpr (sizeof(V) == sizeof(double2)) {
#pragma unroll
    for (int t = 1; t < R; ++t) w[t] = __ldg(tw + t * stride);
    return;
  }
  w[1] = __ldg(tw + stride);
  if constexpr (R >= 4) {
    w[2] = cmul(w[1], w[1]);
    w[3] = cmul(w[2], w[1]);
  }
  if constexpr (R >= 8) {
    w[4] = __ldg(tw + 4 * stride);
    w[5] = cmul(w[4], w[1]);
    w[6] = cmul(w[4], w[2]);
    w[7] = cmul(w[4], w[3]);
  }
  if constexpr (R == 16) {
    w[8] = cmul(w[4], w[4]);
#pragma unroll
    for (int t = 9; t < 16; ++t) w[t] = cmul(w[8], w[t - 8]);
  }
}

template <int R, int SIGN, typename V>
__device__ __forceinline__ void apply_twiddles(V* a, const V (&w)[R]) {
#pragma unroll
  for (int t = 1; t < R; ++t) a[t] = tw_apply<SIGN>(a[t], w[t]);
}

template <int B, int PAD = 2>
struct BlockFFTShape {
  static constexpr int LOGB = (B == 128) ? 7 : (B == 256) ? 8 : (B == 512) ? 9 : (B == 1024) ? 10 : (B == 2048) ? 11 : (B == 4096) ? 12
                            : (B == 8192) ? 13 : (B == 16384) ? 14 : -1;
  static_assert(LOGB > 0, "block size");
  static constexpr int NT = B / 16;
  static constexpr int RM = 1 << (LOGB % 4);           // radix of the second stage (1: none)
  static constexpr int MID16 = LOGB >= 8 ? LOGB / 4 - 2 : 0;  // radix-16 stages between it and the last (0 or 1)
  static constexpr bool LAST16 = LOGB >= 8;            // the last stage is radix 16 (else the second one is)
  static constexpr int SMEM = B + 16 * PAD;            // shared-memory values
  static constexpr int NTP = NT + PAD;                 // padded stride of NT locations
};

// Entries of the stage twiddle tables of block size B.
template <int B>
__host__ __device__ constexpr int block_table_size() {
  using S = BlockFFTShape<B>;
  return (S::RM > 1 ? 16 * S::RM : 0) + (S::MID16 ? 256 * S::RM : 0) + (S::LAST16 ? B : 0);
}

// tw: the stage tables of B.  SIGN: -1 forward, +1 inverse (unnormalised).  tid: the
// thread's index within the transform (0 .. B/16 - 1); several transforms of B <= 4096 points
// can share a thread block, each with its own shared-memory region (16-byte aligned), as long as
// every thread of the block calls block_fft (it synchronises the whole block).  The region may be
// rewritten by the caller only after a barrier: the last stage reads it without one after it.
template <int B, int SIGN, typename V>
__device__ __forceinline__ void block_fft(V (&v)[16], V* sm, const V* __restrict__ tw, int tid) {
  constexpr int PAD = sizeof(V) == sizeof(double2) ? 1 : 2;
  using S = BlockFFTShape<B, PAD>;
  constexpr int NT = S::NT, RM = S::RM, NTP = S::NTP;
  // First stage: no twiddles.  The thread's bins t B/16 + tid sit at locations base + t, with the
  // digits of tid (t2 of RM, t3 of 16 when there is a middle radix-16 stage, t4 of 16) reversed.
  dft<16, SIGN>(v);
  {
    constexpr int N3 = S::MID16 ? 16 : 1;
    const int rest = tid / 16;
    V* o = S::LAST16 ? sm + 16 * (rest / N3) + 16 * RM * (rest % N3) + NTP * (tid % 16) : sm + (16 + PAD) * tid;
    if constexpr (PAD == 1) {
#pragma unroll
      for (int t = 0; t < 16; ++t) o[t] = v[t];
    } else {
#pragma unroll
      for (int t = 0; t < 16; t += 2)
        *reinterpret_cast<float4*>(o + t) = make_float4(v[t].x, v[t].y, v[t + 1].x, v[t + 1].y);
    }
  }
  __syncthreads();
  if constexpr (!S::LAST16) {
    // B = 128: 16 points, then the radix-8 stage, whose butterflies lo = tid + q NT leave
    // X[lo + 16 t] = X[tid + (q + 2 t) NT]
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int lo = tid + q * NT;
      V a[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) a[t] = sm[lo + t * (16 + PAD)];  // padded per 16 locations
      V w[8];
      stage_twiddles<8>(w, tw + lo, 16);
      apply_twiddles<8, SIGN>(a, w);
      dft<8, SIGN>(a);
#pragma unroll
      for (int t = 0; t < 8; ++t) v[q + 2 * t] = a[t];
    }
    return;
  }
  if constexpr (RM > 1 && S::LAST16) {
    // second stage, S = 16: butterflies tid + q NT, q < 16 / RM; all have lo = tid mod 16
    const int lo = tid % 16;
    V w[RM];
    stage_twiddles<RM>(w, tw + lo, 16);
    const int l0 = (tid / 16) * 16 * RM + lo;
    V* p = sm + l0 + PAD * (l0 / NT);
#pragma unroll
    for (int q = 0; q < 16 / RM; ++q) {
      V a[RM];
      V* pq = p + q * RM * NTP;
#pragma unroll
      for (int t = 0; t < RM; ++t) a[t] = pq[16 * t];
      apply_twiddles<RM, SIGN>(a, w);
      dft<RM, SIGN>(a);
#pragma unroll
      for (int t = 0; t < RM; ++t) pq[16 * t] = a[t];
    }
    tw += 16 * RM;
    __syncthreads();
  }
  if constexpr (S::MID16) {
    // middle radix-16 stage, S = 16 RM: group hi of NT = 16 S locations
    constexpr int ST = 16 * RM;
    const int lo = tid % ST;
    V* p = sm + (tid / ST) * NTP + lo;
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = p[t * ST];
    {
      V w[16];
      stage_twiddles<16>(w, tw + lo, ST);
      apply_twiddles<16, SIGN>(v, w);
    }
    dft<16, SIGN>(v);
#pragma unroll
    for (int t = 0; t < 16; ++t) p[t * ST] = v[t];
    tw += 16 * ST;
    __syncthreads();
  }
  // last stage, S = NT: butterfly lo = tid
  if constexpr (S::LAST16) {
    const V* p = sm + tid;
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = p[t * NTP];
    V w[16];
    stage_twiddles<16>(w, tw + tid, NT);
    apply_twiddles<16, SIGN>(v, w);
    dft<16, SIGN>(v);
  }
}

// One transform per thread block (tid = threadIdx.x).
template <int B, int SIGN, typename V>
__device__ __forceinline__ void block_fft(V (&v)[16], V* sm, const V* __restrict__ tw) {
  block_fft<B, SIGN>(v, sm, tw, (int)threadIdx.x);
}

}  // namespace rf
