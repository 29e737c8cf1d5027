// Four-step FFT of n = N1 N2 points in two passes through HBM, FP32 and FP64 (the matched filter of
// Eq. 2: the data transform and the per-template inverse transforms).
//
// With the input index j = N2 a + b (a < N1, b < N2) and the output index k = k1 + N1 k2,
//   X[k1 + N1 k2] = sum_b w_N2^(b k2) [ w_n^(b k1) sum_a x[N2 a + b] w_N1^(a k1) ],
// w_m = exp(sign 2 pi i / m).  Pass 1 transforms the N2 columns (N1 points each, stride N2),
// multiplies by w_n^(b k1) and stores the result in the same layout; pass 2 transforms the
// N1 rows (N2 contiguous points) and stores X[k1 + N1 k2] (natural order, a transposed store).
//
// Both passes run the shared-memory block FFT (blockfft.cuh) on several lines per thread
// block: pass 1 on G adjacent columns, whose lanes interleave so that every load and store of
// a warp covers runs of G consecutive elements; pass 2 on R adjacent rows, staged through
// shared memory for the transposed store (runs of R elements).  Lines of a tile start 128 / G bytes
// apart modulo the 128 bytes of the banks, which keeps the accesses of every stage conflict free.
//
// FP32: the twiddle w_n^m (m = b k1 < n) is the product of two table entries: w_n^(m mod 2^s) and
// w_n^(2^s floor(m / 2^s)), with 2^s = 2^ceil(log2(n) / 2); the tables (about 2 sqrt(n)
// entries) stay in cache.  FP64 reads w_n^m from the context's n-entry table: products would
// cost the FP64 pipe, which has two lanes per SM, more than the gathers cost.
//
// Modes of pass 1: real input (the data transform) and the one-sided product X[k] F[k] for
// k <= n/2, zero above (the matched-filter integrand, formed on load).
//
// FP32 grids of at most 16384 points fit one thread block: block_mf forms the spectrum of the data,
// the product with a filter and the inverse transform in one launch, a block (or, from 2^14 to 2^16
// points and for few references, a cluster of blocks) per reference.
#include <cstdint>
#include <type_traits>

#include "blockfft.cuh"
#include "rf_internal.h"

namespace rf {

namespace {

// FP64 lines of up to 1024 points: four points per thread, radix-4 stages in place (with one radix-2
// stage when log2(L) is odd), the same digit-reversed scheme as blockfft.cuh.  The FP64 pipe gives
// each of an SM's four partitions half a lane, so a warp alone on a partition takes 64 clocks per
// FP64 instruction and a pass wants a warp on every partition: with 16 points per thread the 128 warps
// of a 2^16-point pass took 16 to 25 us, whatever the tile.  A radix-4 stage costs 28 FP64 instructions for
// four points and two levels, 3.5 per point and level; radix 16 costs 3.7.
// Thread tid holds x[tid + t L/4] before and X[tid + t L/4] after; w: exp(-2 pi i m / 4096).
// Shared memory: L + L/8 values.
constexpr int kRoots64 = 4096;
__device__ __forceinline__ int quad_pad(int l) { return l + (l >> 3); }

template <int L, int SIGN>
__device__ __forceinline__ void quad_fft(double2 (&v)[4], double2* sm, const double2* __restrict__ w, int tid) {
  constexpr int NT = L / 4;
  constexpr int LOG = L == 128 ? 7 : L == 256 ? 8 : L == 512 ? 9 : 10;
  static_assert(L <= 1024 && (1 << LOG) == L, "line length");
  constexpr int RM = 1 << (LOG & 1);
  dft<4, SIGN>(v);
  {
    // location of digit t: 4 r + t, r = the digits of tid (RM first, then fours) reversed
    int rest = tid, r = 0, place = 1;
    if (RM > 1) {
      r = rest / (NT / RM);
      rest %= NT / RM;
      place = RM;
    }
#pragma unroll
    for (int m = NT / RM / 4; m >= 1; m /= 4) {
      r += place * (rest / m);
      rest %= m;
      place *= 4;
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) sm[quad_pad(4 * r + t)] = v[t];
  }
  __syncthreads();
  int S = 4;
  if constexpr (RM > 1) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int b = tid + q * NT, lo = b & 3, l = (b >> 2) * 8 + lo;
      double2 a[2] = {sm[quad_pad(l)], sm[quad_pad(l + 4)]};
      a[1] = tw_apply<SIGN>(a[1], __ldg(w + lo * (kRoots64 / 8)));
      dft<2, SIGN>(a);
      sm[quad_pad(l)] = a[0];
      sm[quad_pad(l + 4)] = a[1];
    }
    __syncthreads();
    S = 8;
  }
#pragma unroll
  for (; S < L; S *= 4) {
    const int lo = tid & (S - 1), l = (tid - lo) * 4 + lo;
    const int step = kRoots64 / (4 * S);
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = sm[quad_pad(l + t * S)];
#pragma unroll
    for (int t = 1; t < 4; ++t) v[t] = tw_apply<SIGN>(v[t], __ldg(w + t * lo * step));
    dft<4, SIGN>(v);
    if (4 * S < L) {
#pragma unroll
      for (int t = 0; t < 4; ++t) sm[quad_pad(l + t * S)] = v[t];
      __syncthreads();
    }
  }
}

// Points per thread and the transform of a line.
template <typename V, int L>
constexpr int f4_points() {
  return sizeof(V) == 16 && L <= 1024 ? 4 : 16;
}

template <int L, int SIGN, typename V, int N>
__device__ __forceinline__ void line_fft(V (&v)[N], V* sm, const V* __restrict__ tw, int tid) {
  if constexpr (N == 4) quad_fft<L, SIGN>(v, sm, tw, tid);
  else block_fft<L, SIGN>(v, sm, tw, tid);
}

constexpr int kF4Real = 0;
constexpr int kF4Product = 1;

// Values of one line's shared-memory region in a tile of G lines.
template <typename V, int L, int G>
__host__ __device__ constexpr int f4_line() {
  return (f4_points<V, L>() == 4 ? L + L / 8 : BlockFFTShape<L, 16 / (int)sizeof(V)>::SMEM) +
         128 / (int)sizeof(V) / G;
}

template <typename V, int L, int G>
constexpr size_t f4_smem() {
  return sizeof(V) * (size_t)G * (size_t)f4_line<V, L, G>();
}

extern __shared__ __align__(16) unsigned char f4_raw[];

// Pass 1: columns col0 .. col0 + G - 1 of batch row blockIdx.y; L = N1.
template <typename V, int L, int G, int MODE, int SIGN>
__global__ void __launch_bounds__(G * L / f4_points<V, L>()) k_fft4_cols(const void* __restrict__ in, const V* __restrict__ F,
                                                          int64_t fstride, V* __restrict__ out, int n2log,
                                                          const V* __restrict__ twb, const V* __restrict__ tw4,
                                                          int lo_bits) {
  using T = typename real_of<V>::type;
  constexpr int NP = f4_points<V, L>();
  constexpr int NT = L / NP;
  V* f4_sm = reinterpret_cast<V*>(f4_raw);
  const int c = (int)threadIdx.x % G;
  const int ltid = (int)threadIdx.x / G;
  const int64_t N2 = (int64_t)1 << n2log;
  const int64_t n = N2 * L;
  const int64_t col = (int64_t)blockIdx.x * G + c;
  const int64_t boff = (int64_t)blockIdx.y * n;
  // element (a = ltid + t NT, col) sits at j0 + t NT N2
  const int64_t j0 = (int64_t)ltid * N2 + col;
  const int64_t tstep = (int64_t)NT * N2;
  V v[NP];
  if constexpr (MODE == kF4Real) {
    const T* p = static_cast<const T*>(in) + boff + j0;
#pragma unroll
    for (int t = 0; t < NP; ++t) v[t] = cmake<V>(p[t * tstep], (T)0);
  } else {
    // X is one spectrum shared by the batch; F holds one filter of n/2 + 1 values per row.
    // Rows a > N1/2 lie above n/2 (zero); row N1/2 holds only column 0.
    const V* px = static_cast<const V*>(in) + j0;
    const V* pf = F + (int64_t)blockIdx.y * fstride + j0;
    const int64_t lim = n / 2 - j0;
#pragma unroll
    for (int t = 0; t < NP; ++t)
      v[t] = t * tstep <= lim ? cmul(px[t * tstep], pf[t * tstep]) : cmake<V>((T)0, (T)0);
  }
  line_fft<L, SIGN>(v, f4_sm + c * f4_line<V, L, G>(), twb, ltid);
  // v[u] holds the column's bin k1 = ltid + NT u, u < NP, which goes to row k1: o + NT u N2.
  V* o = out + boff + j0;
  if constexpr (sizeof(T) == 8) {
    const V* w = tw4 + col * ltid;
    const int64_t step = col * NT;
#pragma unroll
    for (int u = 0; u < NP; ++u) o[(int64_t)(u * NT) * N2] = tw_apply<SIGN>(v[u], __ldg(w + u * step));
    return;
  } else {
  // Twiddle w_n^(col k1) = w_n^(col ltid) e^u with e = w_n^(col NT): e, e^2, e^4 and e^8 come
  // from the tables (a product of two entries each, m = col NT 2^i < n), e^3, e^5 .. e^7 by at
  // most two more products, and e^(u + 8) = e^u e^8 (a few ulp in all).
  const unsigned lomask = (1u << lo_bits) - 1u;
  const float2* thi = tw4 + (1u << lo_bits);
  const auto table = [&](unsigned m) { return cmul(__ldg(tw4 + (m & lomask)), __ldg(thi + (m >> lo_bits))); };
  const unsigned cu = (unsigned)col;  // col k1 < n <= 2^24
  const float2 b0 = table(cu * (unsigned)ltid);
  const float2 e1 = table(cu * NT), e2 = table(cu * 2u * NT), e4 = table(cu * 4u * NT), e8 = table(cu * 8u * NT);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    float2 eu;
    if (u == 0) eu = make_float2(1.f, 0.f);
    else if (u == 1) eu = e1;
    else if (u == 2) eu = e2;
    else if (u == 3) eu = cmul(e2, e1);
    else if (u == 4) eu = e4;
    else if (u == 5) eu = cmul(e4, e1);
    else if (u == 6) eu = cmul(e4, e2);
    else eu = cmul(e4, cmul(e2, e1));
    const float2 w = u == 0 ? b0 : cmul(b0, eu);
    const float2 w8 = cmul(w, e8);
    o[(int64_t)(u * NT) * N2] = tw_apply<SIGN>(v[u], w);
    o[(int64_t)((u + 8) * NT) * N2] = tw_apply<SIGN>(v[u + 8], w8);
  }
  }
}

// Pass 2: rows row0 .. row0 + R - 1 of batch row blockIdx.y; L = N2.  Output k1 + N1 k2.
template <typename V, int L, int R, int SIGN>
__global__ void __launch_bounds__(R * L / f4_points<V, L>()) k_fft4_rows(const V* __restrict__ in, V* __restrict__ out, int n1log,
                                                          const V* __restrict__ twb) {
  constexpr int NP = f4_points<V, L>();
  constexpr int NT = L / NP;
  constexpr int SL = f4_line<V, L, R>();
  V* f4_sm = reinterpret_cast<V*>(f4_raw);
  const int g = (int)threadIdx.x / NT;
  const int ltid = (int)threadIdx.x % NT;
  const int64_t N1 = (int64_t)1 << n1log;
  const int64_t n = N1 * L;
  const int64_t row0 = (int64_t)blockIdx.x * R;
  const V* src = in + (int64_t)blockIdx.y * n + (row0 + g) * L;
  V v[NP];
#pragma unroll
  for (int t = 0; t < NP; ++t) v[t] = src[ltid + t * NT];
  V* sm = f4_sm + g * SL;
  line_fft<L, SIGN>(v, sm, twb, ltid);
  __syncthreads();  // the last stage has read its inputs from shared memory
#pragma unroll
  for (int t = 0; t < NP; ++t) sm[ltid + t * NT] = v[t];
  __syncthreads();
  V* dst = out + (int64_t)blockIdx.y * n + row0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int f = (int)threadIdx.x + i * (R * NT);
    const int gg = f % R;
    const int k2 = f / R;
    dst[gg + (int64_t)k2 * N1] = f4_sm[gg * SL + k2];
  }
}

// One reference per block: spectrum of the data, product with the filter, inverse transform, all
// in registers and shared memory.
template <int B>
__global__ void __launch_bounds__(B / 16) k_block_mf(const float* __restrict__ x, const float2* __restrict__ F,
                                                     int64_t fstride, float2* __restrict__ out,
                                                     const float2* __restrict__ twb) {
  constexpr int NT = B / 16;
  float2* sm = reinterpret_cast<float2*>(f4_raw);
  const int tid = threadIdx.x;
  F += blockIdx.x * fstride + tid;
  out += (int64_t)blockIdx.x * B + tid;
  float2 v[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) v[t] = make_float2(__ldg(x + tid + t * NT), 0.f);
  block_fft<B, -1>(v, sm, twb, tid);
  // bins tid + t NT: those below n/2 are t < 8, n/2 itself is t = 8 of thread 0
#pragma unroll
  for (int t = 0; t < 8; ++t) v[t] = cmul(v[t], __ldg(F + t * NT));
  v[8] = tid == 0 ? cmul(v[8], __ldg(F + 8 * NT)) : make_float2(0.f, 0.f);
#pragma unroll
  for (int t = 9; t < 16; ++t) v[t] = make_float2(0.f, 0.f);
  __syncthreads();  // the forward transform's last stage has read shared memory
  block_fft<B, +1>(v, sm, twb, tid);
#pragma unroll
  for (int t = 0; t < 16; ++t) out[t * NT] = v[t];
}

// A whole matched filter on a cluster of eight blocks, one cluster per reference: the four-step data
// transform, the product and the four-step inverse, with the two exchanges between columns and rows
// through distributed shared memory.  n = N1 N2; block r of the cluster owns the columns and the
// output rows [r GC, r GC + GC) of N1 points and the spectrum's rows [r GR, r GR + GR) of N2 points.  The
// spectrum comes out as X[k1 + N1 k2] in the block that owns k1, which is a column of the inverse
// transform (input index N1 a + b with b = k1, a = k2), so the product and the inverse's columns need
// no exchange.  A single block takes 16 us for 2^14 samples (two 16384-point transforms in a row on
// one SM), the four launches of the two-pass form about as long.
constexpr int kClusterBlocks = 8;

// Line l of a tile starts at 16-byte offsets 2 l modulo the banks; rows of an exchange buffer of
// L points are one value apart.
template <int L> constexpr int cl_line() { return BlockFFTShape<L>::SMEM / 16 * 16 + 2; }
template <int L> constexpr int cl_row() { return L + 1; }
template <int N1, int N2> constexpr size_t cl_smem() {
  const int gc = N2 / kClusterBlocks, gr = N1 / kClusterBlocks;
  const int work = gc * cl_line<N1>() > gr * cl_line<N2>() ? gc * cl_line<N1>() : gr * cl_line<N2>();
  return sizeof(float2) * (size_t)(work + gr * cl_row<N2>() + gc * cl_row<N1>());
}

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}
// v to the value at `p` of this block's shared memory, in block `rank` of the cluster
__device__ __forceinline__ void st_cluster(float2* p, int rank, float2 v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

template <int N1, int N2>
__global__ void __cluster_dims__(kClusterBlocks, 1, 1) __launch_bounds__(N1 * N2 / 16 / kClusterBlocks)
    k_cluster_mf(const float* __restrict__ x, const float2* __restrict__ F, int64_t fstride,
                 float2* __restrict__ out, const float2* __restrict__ tb1, const float2* __restrict__ tb2,
                 const float2* __restrict__ tw) {
  constexpr int N = N1 * N2, GC = N2 / kClusterBlocks, GR = N1 / kClusterBlocks;
  constexpr int NT1 = N1 / 16, NT2 = N2 / 16;
  constexpr int WORK = GC * cl_line<N1>() > GR * cl_line<N2>() ? GC * cl_line<N1>() : GR * cl_line<N2>();
  float2* work = reinterpret_cast<float2*>(f4_raw);
  float2* rows = work + WORK;               // GR rows of N2 points (the spectrum's)
  float2* outs = rows + GR * cl_row<N2>();  // GC rows of N1 points (the output's)
  const int rank = (int)(blockIdx.x % kClusterBlocks);
  const int64_t ref = blockIdx.x / kClusterBlocks;
  const int c = (int)threadIdx.x % GC, lc = (int)threadIdx.x / GC;  // column or output row, index in its line
  const int g = (int)threadIdx.x % GR, lr = (int)threadIdx.x / GR;  // spectrum row, index in its line
  // A block's shared memory may be accessed by its peers only once it is known to have started: every
  // block arrives here and waits just before its first store into the others, so that the loads and the
  // first transform hide the barrier.
  cluster_arrive();
  float2 v[16];
  {
    // data columns b of N1 points, to rows k1
    const int b = rank * GC + c;
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = make_float2(__ldg(x + (int64_t)N2 * (lc + t * NT1) + b), 0.f);
    block_fft<N1, -1>(v, work + c * cl_line<N1>(), tb1, lc);
    cluster_wait();
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int k1 = lc + t * NT1;
      st_cluster(rows + (k1 % GR) * cl_row<N2>() + b, k1 / GR, cmul(v[t], __ldg(tw + b * k1)));
    }
  }
  cluster_barrier();
  {
    // spectrum rows k1, the product, and the inverse's columns k1
    const int k1 = rank * GR + g;
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = rows[g * cl_row<N2>() + lr + t * NT2];
    block_fft<N2, -1>(v, work + g * cl_line<N2>(), tb2, lr);
    const float2* f = F + ref * fstride + k1;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int k = k1 + N1 * (lr + t * NT2);
      v[t] = k <= N / 2 ? cmul(v[t], __ldg(f + (k - k1))) : make_float2(0.f, 0.f);
    }
    __syncthreads();  // the forward transform's last stage has read `work`
    block_fft<N2, +1>(v, work + g * cl_line<N2>(), tb2, lr);
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const int q = lr + t * NT2;  // output row
      st_cluster(outs + (q % GC) * cl_row<N1>() + k1, q / GC, cmulc(v[t], __ldg(tw + k1 * q)));
    }
  }
  cluster_barrier();  // also: `work` has been read by the whole block
  {
#pragma unroll
    for (int t = 0; t < 16; ++t) v[t] = outs[c * cl_row<N1>() + lc + t * NT1];
    block_fft<N1, +1>(v, work + c * cl_line<N1>(), tb1, lc);
    float2* o = out + ref * N + rank * GC + c;
#pragma unroll
    for (int t = 0; t < 16; ++t) o[(int64_t)N2 * (lc + t * NT1)] = v[t];
  }
}

constexpr int kF4MinLog = 15;    // FP32: below, one block does it (block_mf)
constexpr int kF4MinLog64 = 14;  // N1, N2 >= 128
constexpr int kF4MaxLog = 24;    // N1, N2 <= 4096
// FP64: beyond these the radix-16 passes of fft.cu, which waste less of the FP64 pipe once a launch fills
// it, are faster.  Data transform, four-step against radix: 363 / 416 us at 2^21, 767 / 672 at 2^22; inverse
// of one reference 39 / about 80 us at 2^18 (each of 100: 32 / 30), 83 / 76 at 2^19, 175 / 157 at 2^20.
constexpr int kF4MaxForward64 = 21;
constexpr int kF4MaxInverse64 = 18;

// Tile widths: G columns of N1 points, R rows of N2 points.  FP32: lines of 512 and 1024 points in
// tiles of 8 columns, longer ones in tiles of 4, so that two blocks share an SM up to 2048 points
// (8 columns of 2048 points, one block per SM: 640 us against 624 for 6 references of 2^23 samples); shorter
// lines, of small transforms, in tiles of 4 for more blocks.  FP64: at most 1024 threads.
template <typename V, int L> constexpr int f4_cols_g() {
  return sizeof(V) == 8 ? (L == 512 || L == 1024 ? 8 : 4) : (L <= 256 ? 2 : 4);
}
template <typename V, int L> constexpr int f4_rows_r() { return sizeof(V) == 16 && L <= 256 ? 2 : 4; }

template <typename V, int L>
const V* line_tables(const rf_ctx* c) {
  constexpr int LOGB = BlockFFTShape<L>::LOGB;
  if constexpr (sizeof(V) == 8) return c->twb32.as<float2>() + c->twb_off[LOGB];
  else return c->twb64.as<double2>() + c->twb64_off[f4_points<V, L>() == 4 ? 0 : LOGB];
}

template <typename V, int L, int MODE, int SIGN>
void launch_cols(const void* in, const V* F, int64_t fstride, V* out, int n2log, int batch, const rf_ctx* c,
                 cudaStream_t s) {
  constexpr int G = f4_cols_g<V, L>();
  const auto fn = k_fft4_cols<V, L, G, MODE, SIGN>;
  constexpr size_t smem = f4_smem<V, L, G>();
  RF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const V* tw;
  if constexpr (sizeof(V) == 8) tw = c->tw4.as<float2>();
  else tw = c->tw64.as<double2>();
  dim3 grid((unsigned)(((int64_t)1 << n2log) / G), (unsigned)batch);
  fn<<<grid, G * L / f4_points<V, L>(), smem, s>>>(in, F, fstride, out, n2log, line_tables<V, L>(c), tw,
                                     c->tw4_lo_bits);
  RF_LAUNCHED();
}

template <typename V, int L, int SIGN>
void launch_rows(const V* in, V* out, int n1log, int batch, const rf_ctx* c, cudaStream_t s) {
  constexpr int R = f4_rows_r<V, L>();
  const auto fn = k_fft4_rows<V, L, R, SIGN>;
  constexpr size_t smem = f4_smem<V, L, R>();
  RF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  dim3 grid((unsigned)(((int64_t)1 << n1log) / R), (unsigned)batch);
  fn<<<grid, R * L / f4_points<V, L>(), smem, s>>>(in, out, n1log, line_tables<V, L>(c));
  RF_LAUNCHED();
}

int ilog2(int64_t n) {
  int b = 0;
  while (((int64_t)1 << b) < n) ++b;
  return b;
}

template <typename F>
void dispatch_line(int log, F&& f) {
  switch (log) {
    case 7: f(std::integral_constant<int, 128>{}); break;
    case 8: f(std::integral_constant<int, 256>{}); break;
    case 9: f(std::integral_constant<int, 512>{}); break;
    case 10: f(std::integral_constant<int, 1024>{}); break;
    case 11: f(std::integral_constant<int, 2048>{}); break;
    default: f(std::integral_constant<int, 4096>{}); break;
  }
}

// N1 = 2^floor(log2(n) / 2) points per column, N2 = n / N1 per row
void split(int64_t n, int& n1log, int& n2log) {
  const int b = ilog2(n);
  n1log = b / 2;
  n2log = b - n1log;
}

// The two passes: columns from `in` (and F) into tmp, rows from tmp into out.
template <typename V, int MODE, int SIGN>
void two_passes(const rf_ctx* c, const void* in, const V* F, int64_t fstride, V* out, V* tmp, int batch,
                cudaStream_t s) {
  constexpr bool f64 = sizeof(V) == 16;
  RF_REQUIRE(SIGN < 0 ? fft4_forward_supported(c->n, f64) : fft4_inverse_supported(c->n, f64),
             "fft4: n=%lld is not supported", (long long)c->n);
  RF_REQUIRE(sizeof(V) == 16 || c->tw4.p != nullptr, "fft4: twiddle tables missing");
  RF_REQUIRE(batch >= 1 && batch <= 65535, "fft4: batch %d out of range", batch);
  RF_REQUIRE(in != out && in != tmp && out != tmp, "fft4: buffers must be distinct");
  int n1log, n2log;
  split(c->n, n1log, n2log);
  constexpr int longest = 1 << (((f64 ? (SIGN < 0 ? kF4MaxForward64 : kF4MaxInverse64) : kF4MaxLog) + 1) / 2);
  dispatch_line(n1log, [&](auto l) {
    if constexpr (decltype(l)::value <= longest)
      launch_cols<V, decltype(l)::value, MODE, SIGN>(in, F, fstride, tmp, n2log, batch, c, s);
  });
  dispatch_line(n2log, [&](auto l) {
    if constexpr (decltype(l)::value <= longest)
      launch_rows<V, decltype(l)::value, SIGN>(tmp, out, n1log, batch, c, s);
  });
}

}  // namespace

namespace {
bool in_logs(int64_t n, int lo, int hi) { return n >= (int64_t)1 << lo && n <= (int64_t)1 << hi && (n & (n - 1)) == 0; }
}  // namespace
bool fft4_forward_supported(int64_t n, bool f64) {
  return in_logs(n, f64 ? kF4MinLog64 : kF4MinLog, f64 ? kF4MaxForward64 : kF4MaxLog);
}
bool fft4_inverse_supported(int64_t n, bool f64) {
  return in_logs(n, f64 ? kF4MinLog64 : kF4MinLog, f64 ? kF4MaxInverse64 : kF4MaxLog);
}

int fft4_lo_bits(int64_t n) { return (ilog2(n) + 1) / 2; }

void fft4_forward_real(const rf_ctx* c, const float* x, float2* out, float2* tmp, cudaStream_t s) {
  two_passes<float2, kF4Real, -1>(c, x, nullptr, 0, out, tmp, 1, s);
}

void fft4_forward_real(const rf_ctx* c, const double* x, double2* out, double2* tmp, cudaStream_t s) {
  two_passes<double2, kF4Real, -1>(c, x, nullptr, 0, out, tmp, 1, s);
}

void fft4_inverse_product(const rf_ctx* c, const float2* X, const float2* F, int64_t fstride, float2* out,
                          float2* tmp, int batch, cudaStream_t s) {
  RF_REQUIRE(fstride >= c->n / 2 + 1, "fft4: filter stride %lld below n/2 + 1", (long long)fstride);
  two_passes<float2, kF4Product, +1>(c, X, F, fstride, out, tmp, batch, s);
}

void fft4_inverse_product(const rf_ctx* c, const double2* X, const double2* F, int64_t fstride, double2* out,
                          double2* tmp, int batch, cudaStream_t s) {
  RF_REQUIRE(fstride >= c->n / 2 + 1, "fft4: filter stride %lld below n/2 + 1", (long long)fstride);
  two_passes<double2, kF4Product, +1>(c, X, F, fstride, out, tmp, batch, s);
}

// One launch per call: up to 2^14 samples always, 2^14 .. 2^16 on clusters while all of them run at
// once (each forms the data's spectrum anew; beyond that the two-pass form, which forms it once, and
// for 2^14 samples one block per reference keep more of the GPU on useful work).
bool cluster_mf(const rf_ctx* c, int nref) {
  return c->n >= 16384 && c->n <= 65536 && (int64_t)nref * kClusterBlocks <= c->nsm;
}
bool block_mf_supported(const rf_ctx* c, int nref) {
  return c->g.dtype == RF_F32 && ((c->n >= 512 && c->n <= 16384) || cluster_mf(c, nref));
}

void block_mf(const rf_ctx* c, const float* x, const float2* F, int64_t fstride, float2* out, int nref,
              cudaStream_t s) {
  auto run = [&](auto bc) {
    constexpr int B = decltype(bc)::value;
    constexpr size_t smem = sizeof(float2) * BlockFFTShape<B>::SMEM;
    RF_CUDA(cudaFuncSetAttribute(k_block_mf<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_block_mf<B><<<(unsigned)nref, B / 16, smem, s>>>(x, F, fstride, out,
                                                       line_tables<float2, B>(c));
    RF_LAUNCHED();
  };
  auto cluster = [&](auto n1, auto n2) {
    constexpr int N1 = decltype(n1)::value, N2 = decltype(n2)::value;
    auto fn = k_cluster_mf<N1, N2>;
    RF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cl_smem<N1, N2>()));
    fn<<<(unsigned)(nref * kClusterBlocks), N1 * N2 / 16 / kClusterBlocks, cl_smem<N1, N2>(), s>>>(
        x, F, fstride, out, line_tables<float2, N1>(c), line_tables<float2, N2>(c), c->tw32.as<float2>());
    RF_LAUNCHED();
  };
  using I128 = std::integral_constant<int, 128>;
  using I256 = std::integral_constant<int, 256>;
  if (cluster_mf(c, nref)) {
    if (c->n == 16384) cluster(I128{}, I128{});
    else if (c->n == 32768) cluster(I128{}, I256{});
    else cluster(I256{}, I256{});
    return;
  }
  switch (ilog2(c->n)) {
    case 9: run(std::integral_constant<int, 512>{}); break;
    case 10: run(std::integral_constant<int, 1024>{}); break;
    case 11: run(std::integral_constant<int, 2048>{}); break;
    case 12: run(std::integral_constant<int, 4096>{}); break;
    case 13: run(std::integral_constant<int, 8192>{}); break;
    default: run(std::integral_constant<int, 16384>{}); break;
  }
}

}  // namespace rf
