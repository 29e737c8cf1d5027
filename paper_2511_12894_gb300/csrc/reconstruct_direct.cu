// Direct reconstruction on CUDA cores (Eq. 8, circular discrete form):
//   z_j[i] = sum_{l < L_j} c_j[l] z_ref[(i - m0_j - l) mod n]
// and the fused per-window peak (max |z_j|^2 and its first index).
//
// A block owns a range of outputs of one neighbour and walks it in tiles of
// NT*E samples; taps are consumed in chunks of LC.  Per tap chunk the block
// stages the z_ref strip the tile needs in shared memory (padded one slot per
// E entries so that the per-thread stride of E is bank-conflict free).  Each
// thread owns E consecutive outputs and keeps the E strip values it needs in
// registers, sliding them by one sample per tap: one shared load and one
// broadcast tap load per E complex multiply-adds.  Real-form kernels (real taps T = R) take
// complex x real products: two multiply-adds per tap and output instead of four.
#include <cfloat>
#include <cstddef>
#include <cstdint>
#include <type_traits>

#include "cplx.cuh"
#include "rf_internal.h"

namespace rf {

namespace {

template <typename R>
struct Best {
  R v;
  long long i;
};

template <typename R>
__device__ __forceinline__ bool better(R v, long long i, R bv, long long bi) {
  return v > bv || (v == bv && i < bi);
}

// Block-wide (value, index) maximum with lowest-index ties.  All threads get the result.
template <typename R, int NT>
__device__ Best<R> block_best(R v, long long i) {
  __shared__ R sv[NT / 32];
  __shared__ long long si[NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const R ov = __shfl_down_sync(0xffffffffu, v, o);
    const long long oi = __shfl_down_sync(0xffffffffu, i, o);
    if (better(ov, oi, v, i)) {
      v = ov;
      i = oi;
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sv[w] = v;
    si[w] = i;
  }
  __syncthreads();
  Best<R> b{sv[0], si[0]};
  for (int q = 1; q < NT / 32; ++q)
    if (better(sv[q], si[q], b.v, b.i)) b = Best<R>{sv[q], si[q]};
  __syncthreads();
  return b;
}

template <typename V, typename T, int E, int NT, int LC, bool WINMAX>
__global__ void __launch_bounds__(NT) k_direct(const V* __restrict__ z_ref, int64_t n, const T* __restrict__ taps,
                                               const int64_t* __restrict__ off, const int* __restrict__ len,
                                               const int* __restrict__ lag0, int64_t range, V* __restrict__ z_out,
                                               int64_t W, int64_t nw, float* __restrict__ max_out,
                                               int* __restrict__ arg_out) {
  using R = typename real_of<V>::type;
  constexpr bool REAL = std::is_same<T, R>::value;
  constexpr int TILE = NT * E;
  constexpr int SPAN = TILE + LC;               // strip entries (last one unused)
  constexpr int PAD = SPAN + SPAN / E + 1;       // padded strip size
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* strip = reinterpret_cast<V*>(smem_raw);
  T* tp = reinterpret_cast<T*>(strip + PAD);
  R* mag = reinterpret_cast<R*>(tp + LC);
  Best<R>* run = reinterpret_cast<Best<R>*>(mag + TILE);  // running best per window of the range

  const int j = blockIdx.y;
  const int L = len[j];
  const int64_t m0 = lag0[j];
  const T* c = taps + off[j];
  const int64_t mask = n - 1;
  const int64_t r0 = (int64_t)blockIdx.x * range;
  const int64_t r1 = min(n, r0 + range);
  const int tid = threadIdx.x;
  const int64_t w_first = WINMAX ? r0 / W : 0;
  const int64_t w_last = WINMAX ? (r1 - 1) / W : 0;
  if (WINMAX) {
    for (int64_t w = w_first + tid; w <= w_last; w += NT) run[w - w_first] = Best<R>{(R)-1, 0};
  }

  for (int64_t c0 = r0; c0 < r1; c0 += TILE) {
    V acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = cmake<V>((R)0, (R)0);
    for (int l0 = 0; l0 < L; l0 += LC) {
      const int lc = min(LC, L - l0);
      __syncthreads();
      // strip[p] = z_ref[(c0 - m0 - l0 - LC + 1 + p) mod n]
      const int64_t base = c0 - m0 - l0 - LC + 1;
      for (int p = tid; p < SPAN - 1; p += NT) strip[p + p / E] = z_ref[(base + p) & mask];
      for (int r = tid; r < LC; r += NT) {
        if constexpr (REAL) tp[r] = (r < lc) ? c[l0 + r] : (R)0;
        else tp[r] = (r < lc) ? c[l0 + r] : cmake<V>((R)0, (R)0);
      }
      __syncthreads();
      const int p0 = tid * E + LC - 1;
      V win[E], part[E];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        win[e] = strip[(p0 + e) + (p0 + e) / E];
        part[e] = cmake<V>((R)0, (R)0);
      }
#pragma unroll 2
      for (int r = 0; r < LC; ++r) {
        const T cr = tp[r];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if constexpr (REAL) {
            part[e].x = fma(cr, win[e].x, part[e].x);
            part[e].y = fma(cr, win[e].y, part[e].y);
          } else {
            part[e].x = fma(cr.x, win[e].x, part[e].x);
            part[e].x = fma(-cr.y, win[e].y, part[e].x);
            part[e].y = fma(cr.x, win[e].y, part[e].y);
            part[e].y = fma(cr.y, win[e].x, part[e].y);
          }
        }
#pragma unroll
        for (int e = E - 1; e > 0; --e) win[e] = win[e - 1];
        if (r + 1 < LC) {
          const int q = p0 - r - 1;
          win[0] = strip[q + q / E];
        }
      }
      // two-level summation: per-chunk partial sums keep the FP32 rounding error
      // growth at about sqrt(LC) + sqrt(L / LC) instead of sqrt(L)
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] = cadd(acc[e], part[e]);
    }
    const int64_t cend = min(r1, c0 + TILE);
    if (!WINMAX) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int64_t i = c0 + tid * E + e;
        if (i < cend) z_out[(int64_t)j * n + i] = acc[e];
      }
    } else {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; ++e) mag[tid * E + e] = acc[e].x * acc[e].x + acc[e].y * acc[e].y;
      __syncthreads();
      for (int64_t w = c0 / W; w <= (cend - 1) / W; ++w) {
        const int64_t lo = max(c0, w * W), hi = min(cend, (w + 1) * W);
        R bv = (R)-1;
        long long bi = 0;
        for (int64_t i = lo + tid; i < hi; i += NT) {
          const R v = mag[i - c0];
          if (v > bv) {
            bv = v;
            bi = i;
          }
        }
        const Best<R> b = block_best<R, NT>(bv, bi);
        if (tid == 0) {
          Best<R>& rb = run[w - w_first];
          if (b.v > rb.v) rb = b;  // earlier tiles hold the earlier indices
        }
      }
    }
  }
  if (WINMAX) {
    __syncthreads();
    for (int64_t w = w_first + tid; w <= w_last; w += NT) {
      const Best<R> b = run[w - w_first];
      max_out[(int64_t)j * nw + w] = (float)b.v;
      arg_out[(int64_t)j * nw + w] = (int)b.i;
    }
  }
}

template <typename V, typename T, int E, int NT, int LC, bool WINMAX>
void launch_direct(rf_ctx* c, const rf_kernels* kern, const V* z_ref, V* z_out, int64_t W, float* max_out,
                   int32_t* arg_out, cudaStream_t s) {
  using R = typename real_of<V>::type;
  constexpr int TILE = NT * E;
  constexpr int SPAN = TILE + LC;
  constexpr int PAD = SPAN + SPAN / E + 1;
  const int64_t n = c->n;
  int64_t range, nw = 0, wpc = 0;
  if (WINMAX) {
    nw = (n + W - 1) / W;
    wpc = std::max<int64_t>(1, (TILE + W - 1) / W);  // whole windows per block, at least one tile of work
    range = wpc * W;
  } else {
    range = TILE;
  }
  const int64_t nblk = (n + range - 1) / range;
  const size_t smem = sizeof(V) * PAD + sizeof(T) * LC + sizeof(R) * TILE + sizeof(Best<R>) * (size_t)(wpc + 2) + 16;
  constexpr size_t smem_cap = 200 * 1024;
  RF_REQUIRE(smem <= smem_cap, "direct reconstruct: window of %lld samples needs too much shared memory",
             (long long)W);
  auto kfn = k_direct<V, T, E, NT, LC, WINMAX>;
  // a process-wide attribute of the function: set to the cap that bounds every launch, so that a
  // context on another host thread never lowers it under this launch
  RF_CUDA(cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cap));
  int64_t done = 0;
  while (done < kern->k) {
    const int cnt = (int)std::min<int64_t>(65535, kern->k - done);
    dim3 grid((unsigned)nblk, (unsigned)cnt);
    kfn<<<grid, NT, smem, s>>>(z_ref, n, static_cast<const T*>(kern->taps.p), kern->off_d.as<int64_t>() + done,
                               kern->len_d.as<int>() + done, kern->lag0_d.as<int>() + done, range,
                               z_out ? z_out + done * n : nullptr, W, nw, max_out ? max_out + done * nw : nullptr,
                               arg_out ? arg_out + done * nw : nullptr);
    RF_LAUNCHED();
    done += cnt;
  }
}

// Window peaks of series already in memory.  |z|^2 is compared as an integer (non-negative floating-point
// numbers order as their bits; -1: none, NaN never counts): the FP64 pipe, two lanes per SM, has the
// magnitudes to form, and comparisons on it as well (a block of 512 threads, each going through the
// warps' results) made FP64 windows of 1024 samples take 186 us for 4 series of 2^20, 2893 for 64 (256
// threads: 73 and 1097; now 23 and 247, 4.35 TB/s).
template <typename V> struct PeakKey { using type = int; };
template <> struct PeakKey<double2> { using type = long long; };
__device__ __forceinline__ int peak_key(float2 a) { return __float_as_int(a.x * a.x + a.y * a.y); }
__device__ __forceinline__ long long peak_key(double2 a) { return __double_as_longlong(a.x * a.x + a.y * a.y); }
template <typename K>
__device__ __forceinline__ float peak_value(K k) {
  if constexpr (sizeof(K) == 4) return k < 0 ? -1.f : __int_as_float(k);
  else return k < 0 ? -1.f : (float)__longlong_as_double(k);
}
template <typename K>
struct Peak {
  K k;
  int i;
};
template <typename K>
__device__ __forceinline__ void peak_take(Peak<K>& b, K k, int i) {  // samples in increasing order
  constexpr K inf = sizeof(K) == 4 ? (K)0x7f800000 : (K)0x7ff0000000000000ll;
  if (k > b.k && k <= inf) b = Peak<K>{k, i};
}
template <typename K>
__device__ __forceinline__ void peak_join(Peak<K>& b, Peak<K> o) {
  if (o.k > b.k || (o.k == b.k && o.i < b.i)) b = o;
}
template <typename K>
__device__ __forceinline__ Peak<K> peak_warp(Peak<K> b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    peak_join(b, Peak<K>{__shfl_xor_sync(0xffffffffu, b.k, o), __shfl_xor_sync(0xffffffffu, b.i, o)});
  return b;
}

// The peak of samples [lo, hi) of a row by threads tid < NT, 16-byte loads, four in flight each; every thread
// meets its samples in increasing order.
template <typename V, int NT, typename K>
__device__ __forceinline__ void peak_scan(Peak<K>& b, const V* __restrict__ zr, int lo, int hi, int tid) {
  if constexpr (sizeof(V) == 16) {
    int i = lo + tid;
    for (; i + 3 * NT < hi; i += 4 * NT) {
      V a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = __ldg(zr + i + u * NT);
#pragma unroll
      for (int u = 0; u < 4; ++u) peak_take(b, peak_key(a[u]), i + u * NT);
    }
    for (; i < hi; i += NT) peak_take(b, peak_key(zr[i]), i);
  } else {
    // rows start 16-byte aligned (n even): pairs [2p, 2p + 1] inside [lo, hi), and up to one sample at each end
    const int p0 = (lo + 1) / 2, p1 = hi / 2;
    if (tid == 0 && (lo & 1) && lo < hi) peak_take(b, peak_key(zr[lo]), lo);
    const float4* z4 = reinterpret_cast<const float4*>(zr);
    auto pair = [&](float4 q, int p) {
      peak_take(b, peak_key(make_float2(q.x, q.y)), 2 * p);
      peak_take(b, peak_key(make_float2(q.z, q.w)), 2 * p + 1);
    };
    int p = p0 + tid;
    for (; p + 3 * NT < p1; p += 4 * NT) {
      float4 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = __ldg(z4 + p + u * NT);
#pragma unroll
      for (int u = 0; u < 4; ++u) pair(a[u], p + u * NT);
    }
    for (; p < p1; p += NT) pair(__ldg(z4 + p), p);
    if (tid == 0 && (hi & 1) && hi - 1 >= 2 * p0 && lo < hi) peak_take(b, peak_key(zr[hi - 1]), hi - 1);
  }
}

// Windows that a warp takes.  Up to 2048 samples it costs no more than a block (64 series of 2^20 in
// FP32: 77.5 us at 1024, 79 at 2048); at 4096 too few loads are in flight (87.8 against 77.8; 16 series of
// 2^16 in FP64 23.2 against 17.7).
constexpr int64_t kShortWindow = 1024;

// Short windows: a warp each.  (A block each spent its time on starting and reducing: 16-sample windows of
// 4 series of 2^20 took 550 us in FP32, 10262 in FP64; now 42 and 54.)
template <typename V>
__global__ void __launch_bounds__(256) k_winmax_short(const V* __restrict__ z, int64_t n, int W, int nw,
                                                      float* __restrict__ max_out, int* __restrict__ arg_out) {
  using K = typename PeakKey<V>::type;
  const int w = blockIdx.x * 8 + (int)(threadIdx.x >> 5);
  const int64_t row = blockIdx.y;
  if (w >= nw) return;
  const int lane = threadIdx.x & 31;
  const int lo = w * W, hi = min((int)n, lo + W);
  Peak<K> b{-1, 0};
  peak_scan<V, 32>(b, z + row * n, lo, hi, lane);
  b = peak_warp(b);
  if (lane == 0) {
    max_out[row * nw + w] = peak_value(b.k);
    arg_out[row * nw + w] = b.i;
  }
}

// Longer windows: CS blocks per (window, series), one cluster.  Block c
// reads the c-th part of the window and the cluster's first block takes the
// best of the parts through distributed shared memory, so no workspace is needed (calls on
// several streams stay independent).  Bound by HBM.  One block per window left most SMs idle when
// windows are long: 6 series of 2^23 samples in 2^20-sample windows took 464 us on 48 blocks of
// 256 threads (24 series of 2^20 in 2^17-sample windows: 65 us).
template <typename V, int NT>
__global__ void __launch_bounds__(NT) k_winmax_series(const V* __restrict__ z, int64_t n, int64_t W, int nw,
                                                      int CS, float* __restrict__ max_out,
                                                      int* __restrict__ arg_out) {
  using K = typename PeakKey<V>::type;
  constexpr int E = 16 / (int)sizeof(V);  // samples per 16-byte load
  const int w = (int)(blockIdx.x / (unsigned)CS);
  const int part = (int)(blockIdx.x % (unsigned)CS);
  const int64_t row = blockIdx.y;
  const int wlo = (int)(w * W), whi = (int)min(n, wlo + W);
  const int per = ((whi - wlo + CS - 1) / CS + E - 1) / E * E;
  const int lo = min(whi, wlo + part * per), hi = min(whi, lo + per);
  Peak<K> b{-1, 0};
  peak_scan<V, NT>(b, z + row * n, lo, hi, (int)threadIdx.x);
  __shared__ Peak<K> wb[NT / 32];
  __shared__ Peak<K> best;
  b = peak_warp(b);
  if ((threadIdx.x & 31) == 0) wb[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x < 32) {
    b = threadIdx.x < NT / 32 ? wb[threadIdx.x] : Peak<K>{-1, 0x7fffffff};
    b = peak_warp(b);
  }
  if (CS > 1) {
    if (threadIdx.x == 0) best = b;
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (part == 0 && threadIdx.x == 0) {
      const uint32_t own = (uint32_t)__cvta_generic_to_shared(&best);
      for (int c = 1; c < CS; ++c) {
        uint32_t at;
        Peak<K> o;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(own), "r"(c));
        if constexpr (sizeof(K) == 8)
          asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(o.k) : "r"(at) : "memory");
        else
          asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(o.k) : "r"(at) : "memory");
        asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(o.i) : "r"(at + (uint32_t)offsetof(Peak<K>, i)) : "memory");
        peak_join(b, o);
      }
    }
    // the other blocks' shared memory stays until it has been read
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (part == 0 && threadIdx.x == 0) {
    max_out[row * nw + w] = peak_value(b.k);
    arg_out[row * nw + w] = b.i;
  }
}

template <typename V, int NT>
void launch_winmax_series(rf_ctx* c, const void* z, int32_t count, int64_t W, int64_t nw, float* max_out,
                          int32_t* argmax_out, cudaStream_t s) {
  // Blocks per window (clusters of at most 8): doubled while the launch has fewer than four
  // blocks per SM and a part keeps 4096 samples (a shorter part's loads no longer cover its
  // start-up).
  int CS = 1;
  while (CS < 8 && nw * count * CS < 4LL * c->nsm && W / (2 * CS) >= 4096) CS *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(nw * CS), (unsigned)count);
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)CS;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = CS > 1 ? 1 : 0;
  RF_CUDA(cudaLaunchKernelEx(&cfg, k_winmax_series<V, NT>, static_cast<const V*>(z), c->n, W, (int)nw, CS, max_out,
                             (int*)argmax_out));
  RF_LAUNCHED();
}

template <typename V>
void winmax_rows(rf_ctx* c, const void* z, int32_t count, int64_t W, int64_t nw, float* max_out, int32_t* argmax_out,
                 cudaStream_t s) {
  if (W <= kShortWindow) {
    k_winmax_short<V><<<dim3((unsigned)((nw + 7) / 8), (unsigned)count), 256, 0, s>>>(
        static_cast<const V*>(z), c->n, (int)W, (int)nw, max_out, (int*)argmax_out);
    RF_LAUNCHED();
  } else if (W >= 8192) {  // enough samples for 512 threads with four 16-byte loads each in flight
    launch_winmax_series<V, 512>(c, z, count, W, nw, max_out, argmax_out, s);
  } else {
    launch_winmax_series<V, 256>(c, z, count, W, nw, max_out, argmax_out, s);
  }
}

}  // namespace

void reconstruct_direct(rf_ctx* c, const void* z_ref, const rf_kernels* kern, void* z_out, int64_t W,
                        float* max_out, int32_t* argmax_out, cudaStream_t s) {
  if (kern->k == 0) return;
  const bool win = max_out != nullptr;
  auto run = [&](auto vtag, auto ttag, auto etag) {
    using V = decltype(vtag);
    using T = decltype(ttag);
    constexpr int E = decltype(etag)::value;
    auto zr = static_cast<const V*>(z_ref);
    auto zo = static_cast<V*>(z_out);
    if (win) launch_direct<V, T, E, 256, 256, true>(c, kern, zr, nullptr, W, max_out, argmax_out, s);
    else launch_direct<V, T, E, 256, 256, false>(c, kern, zr, zo, W, nullptr, nullptr, s);
  };
  using E4 = std::integral_constant<int, 4>;
  using E8 = std::integral_constant<int, 8>;
  if (c->g.dtype == RF_F64) {
    if (kern->real) run(double2{}, double{}, E4{});
    else run(double2{}, double2{}, E4{});
  } else {
    if (kern->real) run(float2{}, float{}, E8{});
    else run(float2{}, float2{}, E8{});
  }
}

void winmax_series(rf_ctx* c, const void* z, int32_t count, int64_t W, float* max_out, int32_t* argmax_out,
                   cudaStream_t s) {
  const int64_t n = c->n;
  const int64_t nw = (n + W - 1) / W;
  RF_REQUIRE(nw <= 0x7fffffff && count <= 65535, "winmax: too many windows or series");
  if (c->g.dtype == RF_F64) winmax_rows<double2>(c, z, count, W, nw, max_out, argmax_out, s);
  else winmax_rows<float2>(c, z, count, W, nw, max_out, argmax_out, s);
}

}  // namespace rf
