// FP64 reconstruction by overlap-save (the block form of Eq. 7), the choice of RF_ALGO_AUTO on
// RF_F64 grids where it is modelled cheaper than the direct sum.
//
// The identities are those of reconstruct_os.cu: block size B, partitions of Lp = B / Q taps,
// hop H = B - Lp, segment spectra Zs[q] of z_ref at every multiple of Lp, and
//   y = IFFT_B( sum_p Zs[(s (Q - 1) - p - 1) mod NQ] C[p] ),  w[s H + t - Lp] = y[t], Lp <= t < B,
// here in FP64 throughout.  Bound by the FP64 pipe (about 1.6 multiply-adds per clock and SM,
// measured): a block costs about 3.4 log2(B) + 4 P + 5 FP64 instructions per point, the direct sum
// 4 L per output.  16 neighbours of 930 taps at n = 2^16 with window peaks: 7157 us by the direct
// sum, 155 us here (the first call, which prepares the spectra, 398 us).
//
// A transform mixes all samples of its block: one that is not finite would reach every output of the
// block, and the rounding of a loud stretch the quiet ones beside it, where the direct sum keeps both to the
// kernel's own samples.  Each segment therefore leaves the magnitudes of its loudest sample and of its quietest
// run of 32 samples, and a block whose segments span more than 2^10 between the two, or come near the
// end of the FP64 range, forms its outputs as direct sums instead: 2^10 roundings are the 1e-12 that FP64
// results are held to, and series of a matched filter stay within 2^5.
//
// Window peaks compare |z|^2 in FP64.  A block leaves the best of each of its pieces (its run of
// outputs cut at window boundaries and at the wrap to sample 0) in a list, and a second kernel
// takes the best piece of every window; a larger value wins, then the smaller index, and NaN never
// does, as in the direct form.
//
// The workspace of a call (segment spectra, pieces) is allocated in stream order from a pool of
// the context, so that calls on several streams stay independent.
#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>

#include "blockfft.cuh"
#include "rf_internal.h"

namespace rf {

namespace {

constexpr int kB64[3] = {1024, 2048, 4096};  // block sizes; the largest gives 256 threads of 16 points
constexpr size_t kWork64Max = (size_t)8 << 30;

struct Piece {
  long long key;  // bits of |z|^2 (non-negative doubles order as integers), -1: none
  long long i;    // its first sample index
};

__device__ __forceinline__ void piece_take(Piece& b, long long key, long long i) {
  if (key > b.key || (key == b.key && i < b.i)) b = Piece{key, i};
}

__device__ __forceinline__ Piece warp_piece(Piece b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long k = __shfl_xor_sync(0xffffffffu, b.key, o);
    const long long i = __shfl_xor_sync(0xffffffffu, b.i, o);
    piece_take(b, k, i);
  }
  return b;
}

// Most pieces of a run of H outputs: the window boundaries inside it and the wrap.
__host__ __device__ constexpr int64_t piece_slots(int64_t H, int64_t W) { return (H - 1) / W + 3; }

// High words of the magnitudes max(|x|, |y|) of a segment: its largest, and the smallest of the
// largest of runs of 32 samples (NaN is above infinity).
struct Range64 {
  unsigned hi, lo;
};
// Whether a block of these segments is left to the direct sum.
__device__ __forceinline__ bool too_wide(Range64 r) {
  constexpr unsigned top = (1023u + 960u) << 20;  // 2^960: no sum of a block or product overflows below it
  return r.hi >= top || (r.hi >> 20) > (r.lo >> 20) + 10u;
}

// Segment spectra: block q transforms z_ref[(q Lp + t) mod n], t < B.
template <int B>
__global__ void __launch_bounds__(B / 16) k_os64_segments(const double2* __restrict__ z_ref, int64_t n, int Lp,
                                                          const double2* __restrict__ tw, double2* __restrict__ Zs,
                                                          Range64* __restrict__ ranges) {
  constexpr int NT = B / 16;
  extern __shared__ __align__(16) double2 sm64[];
  __shared__ Range64 wr[NT / 32];
  const int64_t q = blockIdx.x;
  const int tid = threadIdx.x;
  double2 v[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) v[t] = z_ref[(q * Lp + tid + t * NT) & (n - 1)];
  Range64 r{0u, ~0u};
#pragma unroll
  for (int t = 0; t < 16; ++t) {  // a warp's samples of one t are a run of 32
    const unsigned h = __reduce_max_sync(0xffffffffu, max((unsigned)__double2hiint(v[t].x) & 0x7fffffffu,
                                                          (unsigned)__double2hiint(v[t].y) & 0x7fffffffu));
    r.hi = max(r.hi, h);
    r.lo = min(r.lo, h);
  }
  if ((tid & 31) == 0) wr[tid >> 5] = r;
  block_fft<B, -1>(v, sm64, tw);  // its barriers come between that and this
  if (tid == 0) {
    for (int w = 1; w < NT / 32; ++w) {
      r.hi = max(r.hi, wr[w].hi);
      r.lo = min(r.lo, wr[w].lo);
    }
    ranges[q] = r;
  }
#pragma unroll
  for (int t = 0; t < 16; ++t) Zs[q * B + tid + t * NT] = v[t];
}

// Partition spectra FFT_B(taps) / B: block g is partition rows[g].y of kernel rows[g].x.
template <int B>
__global__ void __launch_bounds__(B / 16) k_os64_partitions(const void* __restrict__ taps, int real,
                                                            const int64_t* __restrict__ off,
                                                            const int* __restrict__ len,
                                                            const int2* __restrict__ rows, int Lp,
                                                            const double2* __restrict__ tw, double2* __restrict__ C) {
  constexpr int NT = B / 16;
  extern __shared__ __align__(16) double2 sm64[];
  const int64_t g = blockIdx.x;
  const int j = rows[g].x;
  const int64_t l0 = (int64_t)rows[g].y * Lp;
  const int tid = threadIdx.x;
  double2 v[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    const int u = tid + t * NT;
    const int64_t l = l0 + u;
    v[t] = make_double2(0.0, 0.0);
    if (u < Lp && l < len[j]) {
      if (real) v[t].x = static_cast<const double*>(taps)[off[j] + l];
      else v[t] = static_cast<const double2*>(taps)[off[j] + l];
    }
  }
  block_fft<B, -1>(v, sm64, tw);
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    const double sc = 1.0 / B;  // a power of two: exact
    C[g * B + tid + t * NT] = make_double2(v[t].x * sc, v[t].y * sc);
  }
}

// The kernels and the series themselves, for blocks formed as direct sums.
struct Direct64 {
  const double2* z;
  const void* taps;  // double2, or double (real)
  const int64_t* off;
  const int* len;
  int real;
};

// sum_l c_j[l] z[(o - l) mod n], in partial sums of 128 terms
__device__ __noinline__ double2 direct64(const Direct64& d, int j, int64_t o, int64_t mask) {
  const int L = d.len[j];
  const double* cr = static_cast<const double*>(d.taps) + d.off[j] * (d.real ? 1 : 2);
  double2 sum = make_double2(0.0, 0.0);
  for (int l0 = 0; l0 < L; l0 += 128) {
    double2 p = make_double2(0.0, 0.0);
    const int l1 = min(L, l0 + 128);
    for (int l = l0; l < l1; ++l) {
      const double2 z = __ldg(d.z + ((o - l) & mask));
      if (d.real) {
        const double c = __ldg(cr + l);
        p.x = fma(c, z.x, p.x);
        p.y = fma(c, z.y, p.y);
      } else {
        const double a = __ldg(cr + 2 * (int64_t)l), b = __ldg(cr + 2 * (int64_t)l + 1);
        p.x = fma(a, z.x, fma(-b, z.y, p.x));
        p.y = fma(a, z.y, fma(b, z.x, p.y));
      }
    }
    sum.x += p.x;
    sum.y += p.y;
  }
  return sum;
}

// Output block blockIdx.x of neighbour j0 + blockIdx.y: the partition products, the inverse
// transform, then the series row or the pieces of the window peaks.
template <int B, int Q, bool WINMAX>
__global__ void __launch_bounds__(B / 16, 8192 / B) k_os64(const double2* __restrict__ Zs,
                                                           const double2* __restrict__ spec,
                                                           const int64_t* __restrict__ spec_off,
                                                           const int* __restrict__ parts,
                                                           const int* __restrict__ lag0, int j0,
                                                           const Range64* __restrict__ ranges, Direct64 dir,
                                                           const double2* __restrict__ tw, int64_t n, int NQ,
                                                           double2* __restrict__ z_out, Piece* __restrict__ pieces,
                                                           int64_t W, int64_t slots) {
  constexpr int NT = B / 16, LP = B / Q, H = B - LP;
  extern __shared__ __align__(16) double2 sm64[];
  const int s = blockIdx.x;
  const int j = j0 + blockIdx.y;
  const int tid = threadIdx.x;
  const double2* C = spec + spec_off[j] + tid;
  const int P = parts[j];
  double2 v[16];
#pragma unroll
  for (int t = 0; t < 16; ++t) v[t] = make_double2(0.0, 0.0);
  int sp = s * (Q - 1) - 1;
  Range64 range{0u, ~0u};
  for (int p = 0; p < P; ++p, --sp) {
    const Range64 r = ranges[sp & (NQ - 1)];
    range.hi = max(range.hi, r.hi);
    range.lo = min(range.lo, r.lo);
    const double2* z = Zs + (int64_t)(sp & (NQ - 1)) * B + tid;  // NQ a power of two
    const double2* c = C + (int64_t)p * B;
#pragma unroll
    for (int t = 0; t < 16; ++t) {
      const double2 a = __ldcg(z + t * NT), b = __ldcg(c + t * NT);
      v[t].x = fma(a.x, b.x, fma(-a.y, b.y, v[t].x));
      v[t].y = fma(a.x, b.y, fma(a.y, b.x, v[t].y));
    }
  }
  block_fft<B, +1>(v, sm64, tw);
  const int64_t mask = n - 1;
  const int64_t o0 = (int64_t)s * H;  // pre-relabel index of block position LP
  const int64_t base = (o0 + lag0[j]) & mask;
  const int cnt = (int)min((int64_t)H, n - o0);
  if (too_wide(range)) {
#pragma unroll 1
    for (int t = 16 / Q; t < 16; ++t) {
      const int e = tid + t * NT - LP;
      const double2 y = e < cnt ? direct64(dir, j, o0 + e, mask) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 16 / Q; u < 16; ++u)
        if (u == t) v[u] = y;  // registers indexed at compile time
    }
  }
  if constexpr (!WINMAX) {
#pragma unroll
    for (int t = 16 / Q; t < 16; ++t) {
      const int e = tid + t * NT - LP;
      if (e < cnt) z_out[(int64_t)j * n + ((base + e) & mask)] = v[t];
    }
  } else {
    // |y|^2 as integer keys in their own region (NaN: -1)
    long long* key = reinterpret_cast<long long*>(sm64 + BlockFFTShape<B, 1>::SMEM);
#pragma unroll
    for (int t = 16 / Q; t < 16; ++t) {
      const long long k = __double_as_longlong(v[t].x * v[t].x + v[t].y * v[t].y);
      key[tid + t * NT - LP] = k > 0x7ff0000000000000ll ? -1ll : k;
    }
    __syncthreads();
    // pieces q < pre lie before the wrap to sample 0 (windows w0 + q), the others after it
    const int64_t w0 = base / W, end = min(n, base + cnt), rem = base + cnt - end;
    const int pre = (int)((end - 1) / W - w0 + 1), all = pre + (int)((rem + W - 1) / W);
    Piece* out = pieces + ((int64_t)j * gridDim.x + s) * slots;
    auto bounds = [&](int q, int& lo, int& hi) {
      if (q < pre) {
        lo = (int)(max(base, (w0 + q) * W) - base);
        hi = (int)(min(end, (w0 + q + 1) * W) - base);
      } else {
        lo = (int)(n - base + (q - pre) * W);
        hi = (int)(n - base + min(rem, (int64_t)(q - pre + 1) * W));
      }
    };
    auto scan = [&](int lo, int hi, int first, int step) {
      Piece b{-1, 0};
      for (int e = lo + first; e < hi; e += step) {
        const long long k = key[e];
        if (k > b.key) b = Piece{k, (base + e) & mask};
      }
      return b;
    };
    constexpr int NW = NT / 32;
    const int warp = tid >> 5, lane = tid & 31;
    if (all >= NW) {  // a warp per piece
      for (int q = warp; q < all; q += NW) {
        int lo, hi;
        bounds(q, lo, hi);
        const Piece b = warp_piece(scan(lo, hi, lane, 32));
        if (lane == 0) out[q] = b;
      }
    } else {  // all warps on each piece
      __shared__ Piece wb[2][NW];
      for (int q = 0; q < all; ++q) {
        int lo, hi;
        bounds(q, lo, hi);
        const Piece b = warp_piece(scan(lo, hi, tid, NT));
        if (lane == 0) wb[q & 1][warp] = b;
        __syncthreads();
        if (tid == 0) {
          Piece r = wb[q & 1][0];
          for (int u = 1; u < NW; ++u) piece_take(r, wb[q & 1][u].key, wb[q & 1][u].i);
          out[q] = r;
        }
      }
    }
  }
}

// The best piece of window w of row blockIdx.y, a warp each: the blocks whose pre-relabel range
// meets the window's, in one or (across the wrap of the pre-relabel index) two runs.
__global__ void __launch_bounds__(128) k_os64_peaks(const Piece* __restrict__ pieces, const int* __restrict__ lag0,
                                                    int j0, int64_t n, int NB, int H, int64_t W, int64_t nw,
                                                    int64_t slots, float* __restrict__ max_out,
                                                    int* __restrict__ arg_out) {
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= nw) return;
  const int j = j0 + blockIdx.y;
  const int64_t mask = n - 1, m0 = lag0[j];
  const int64_t lo = w * W, len = min(n, lo + W) - lo;
  const int64_t a = (lo - m0) & mask, e1 = min(n, a + len), e2 = a + len - e1;
  Piece b{-1, 0};
  auto block = [&](int64_t s) {
    const int64_t base = (s * H + m0) & mask;
    const int64_t cnt = min((int64_t)H, n - s * H);
    const int64_t w0 = base / W, end = min(n, base + cnt), rem = base + cnt - end;
    const Piece* p = pieces + ((int64_t)j * NB + s) * slots;
    if (w >= w0 && max(lo, base) < min(end, lo + W)) piece_take(b, p[w - w0].key, p[w - w0].i);
    if (lo < rem) {
      const int64_t q = (end - 1) / W - w0 + 1 + w;
      piece_take(b, p[q].key, p[q].i);
    }
  };
  for (int64_t s = a / H + lane; s <= (e1 - 1) / H; s += 32) block(s);
  if (e2 > 0)
    for (int64_t s = lane; s <= (e2 - 1) / H; s += 32) block(s);
  b = warp_piece(b);
  if (lane == 0) {
    max_out[(int64_t)j * nw + w] = b.key < 0 ? -1.f : (float)__longlong_as_double(b.key);
    arg_out[(int64_t)j * nw + w] = b.key < 0 ? 0 : (int)b.i;
  }
}

template <typename F>
void dispatch64(int B, int Q, F&& f) {
  auto q = [&](auto bc) {
    if (Q == 2) f(bc, std::integral_constant<int, 2>{});
    else f(bc, std::integral_constant<int, 4>{});
  };
  switch (B) {
    case 1024: q(std::integral_constant<int, 1024>{}); break;
    case 2048: q(std::integral_constant<int, 2048>{}); break;
    default: q(std::integral_constant<int, 4096>{}); break;
  }
}

template <int B>
constexpr size_t smem64(int H) {
  return sizeof(double2) * BlockFFTShape<B, 1>::SMEM + sizeof(long long) * (size_t)H;
}

int table64(int B) { return B == 1024 ? 10 : (B == 2048 ? 11 : 12); }

// Cheapest (B, Q) for the kernel lengths by modelled SM cycles, or B = 0 for the direct sum.  The
// FP64 pipe runs 1.6 instructions per clock; blocks are spread whole over the SMs, the direct
// sum's 1024-output tiles evenly, but none takes less than its longest; 6000 cycles stand for the
// two extra launches.
void choose64(const rf_ctx* c, const rf_kernels* k, int* B_out, int* Q_out) {
  const double rate = 1.6;
  const int64_t total = k->offset[k->k];
  double best = std::max(4.0 * (double)total * (double)c->n / c->nsm,
                         4.0 * (double)k->max_len * (double)std::min<int64_t>(1024, c->n)) / rate;
  *B_out = 0;
  *Q_out = 0;
  for (const int B : kB64) {
    if (B > c->n) continue;
    for (int Q = 2; Q <= 4; Q *= 2) {
      const int Lp = B / Q, H = B - Lp;
      const int64_t NB = (c->n + H - 1) / H, NQ = c->n / Lp;
      double P = 0.0;
      for (const int L : k->len) P += std::max(1, (L + Lp - 1) / Lp);
      P /= k->k;
      const double fft = 3.4 * std::log2((double)B);
      const double blk = B * (fft + 4.0 * P + 5.0) / rate, seg = B * fft / rate;
      const double cost = std::ceil((double)NB * k->k / c->nsm) * blk + std::ceil((double)NQ / c->nsm) * seg + 6000.0;
      if (cost < best) {
        best = cost;
        *B_out = B;
        *Q_out = Q;
      }
    }
  }
}

// Prepares the partition spectra (allocates, synchronises).
void prepare64(rf_ctx* c, rf_kernels* kern, int B, int Q, cudaStream_t s) {
  const int k = kern->k, Lp = B / Q;
  std::vector<int> parts(k);
  std::vector<int64_t> off(k);
  std::vector<int2> rows;
  for (int j = 0; j < k; ++j) {
    parts[j] = std::max(1, (kern->len[j] + Lp - 1) / Lp);
    off[j] = (int64_t)rows.size() * B;
    for (int p = 0; p < parts[j]; ++p) rows.push_back(make_int2(j, p));
  }
  kern->os64_spec.ensure(sizeof(double2) * rows.size() * (size_t)B);
  kern->os64_off_d.ensure(sizeof(int64_t) * k);
  kern->os64_parts_d.ensure(sizeof(int) * k);
  DevBuf rd;
  rd.ensure(sizeof(int2) * rows.size());
  RF_CUDA(cudaMemcpyAsync(kern->os64_off_d.p, off.data(), sizeof(int64_t) * k, cudaMemcpyHostToDevice, s));
  RF_CUDA(cudaMemcpyAsync(kern->os64_parts_d.p, parts.data(), sizeof(int) * k, cudaMemcpyHostToDevice, s));
  RF_CUDA(cudaMemcpyAsync(rd.p, rows.data(), sizeof(int2) * rows.size(), cudaMemcpyHostToDevice, s));
  dispatch64(B, Q, [&](auto bc, auto) {
    constexpr int BB = decltype(bc)::value;
    auto fn = k_os64_partitions<BB>;
    RF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64<BB>(0)));
    fn<<<(unsigned)rows.size(), BB / 16, smem64<BB>(0), s>>>(
        kern->taps.p, kern->real ? 1 : 0, kern->off_d.as<int64_t>(), kern->len_d.as<int>(), rd.as<int2>(), Lp,
        c->twb64.as<double2>() + c->twb64_off[table64(BB)], kern->os64_spec.as<double2>());
    RF_LAUNCHED();
  });
  RF_CUDA(cudaStreamSynchronize(s));  // the host vectors and the row list go out of scope
  kern->os64_B = B;
  kern->os64_Q = Q;
}

bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
    (void)cudaGetLastError();
    return true;
  }
  return st != cudaStreamCaptureStatusNone;
}

// Allocations of this thread while another thread captures a stream: the capture neither forbids
// them nor records them.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { (void)cudaThreadExchangeStreamCaptureMode(&mode); }
};

}  // namespace

void os64_create(rf_ctx* c) {
  std::vector<double2> tw;
  auto tables = [&](auto bc, int slot) {
    constexpr int B = decltype(bc)::value;
    using S = BlockFFTShape<B, 1>;
    c->twb64_off[slot] = (int64_t)tw.size();
    int st = 16;
    auto stage = [&](int radix) {
      const std::vector<double2>& w = block_twiddles();
      const size_t step = (size_t)(kBlockTwiddles / ((int64_t)radix * st));
      for (int t = 0; t < radix; ++t)
        for (int k = 0; k < st; ++k) tw.push_back(w[(size_t)t * k * step]);
      st *= radix;
    };
    if (S::RM > 1) stage(S::RM);
    if (S::MID16) stage(16);
    if (S::LAST16) stage(16);
  };
  // slot 0: the 4096th roots of unity, for the lines of four points per thread (fft4.cu)
  for (int m = 0; m < 4096; ++m) tw.push_back(block_twiddles()[(size_t)m * (kBlockTwiddles / 4096)]);
  tables(std::integral_constant<int, 1024>{}, 10);
  tables(std::integral_constant<int, 2048>{}, 11);
  tables(std::integral_constant<int, 4096>{}, 12);
  c->twb64.ensure(sizeof(double2) * tw.size());
  RF_CUDA(cudaMemcpy(c->twb64.p, tw.data(), sizeof(double2) * tw.size(), cudaMemcpyHostToDevice));
}

// Prepares a kernel set where the transform form is modelled cheaper.  os64_B is settled (-1: the direct
// sum) by the model and the bound on the spectra alone; a set that met a shortage of memory or a stream
// under capture stays open, and the next call tries again.
bool os64_prepare(rf_ctx* c, rf_kernels* kern, cudaStream_t s) {
  if (!c->pool || kern->k == 0) return false;
  RelaxedCapture relaxed;
  std::lock_guard<std::mutex> lock(kern->os64_mu);
  if (kern->os64_B) return kern->os64_B > 0;
  int B, Q;
  choose64(c, kern, &B, &Q);
  if (B) {
    int64_t rows = 0;
    for (const int L : kern->len) rows += std::max(1, (L + B / Q - 1) / (B / Q));
    if (rows > INT_MAX / 2 || sizeof(double2) * (size_t)rows * B > kWork64Max) B = 0;
  }
  if (!B) {
    kern->os64_B = -1;
    return false;
  }
  if (capturing(s)) return false;
  try {
    prepare64(c, kern, B, Q, s);
  } catch (const Fail& e) {
    if (e.st != RF_ENOMEM) throw;
    clear_error();
    kern->os64_spec.release();
    return false;
  }
  return true;
}

// False where the direct sum should run instead: the set is not prepared or memory for the call is short.
bool reconstruct_os64(rf_ctx* c, const void* z_ref, rf_kernels* kern, void* z_out, int64_t W, float* max_out,
                      int32_t* argmax_out, cudaStream_t s) {
  if (!os64_prepare(c, kern, s)) return false;
  RelaxedCapture relaxed;
  const int B = kern->os64_B, Q = kern->os64_Q;  // they no longer change
  const bool win = max_out != nullptr;
  const int64_t n = c->n;
  const int Lp = B / Q, H = B - Lp;
  const int NQ = (int)(n / Lp), NB = (int)((n + H - 1) / H);
  const int64_t nw = win ? (n + W - 1) / W : 0, slots = win ? piece_slots(H, W) : 0;
  const size_t zs_bytes = sizeof(double2) * (size_t)NQ * B;
  const size_t range_bytes = (sizeof(Range64) * (size_t)NQ + 15) & ~(size_t)15;
  const size_t need = zs_bytes + range_bytes + sizeof(Piece) * (size_t)kern->k * NB * (size_t)slots;
  if (need > kWork64Max) return false;
  StreamBuf work(c, need, s);
  if (!work.p) return false;
  double2* Zs = static_cast<double2*>(work.p);
  Range64* ranges = reinterpret_cast<Range64*>(static_cast<char*>(work.p) + zs_bytes);
  Piece* pieces = reinterpret_cast<Piece*>(static_cast<char*>(work.p) + zs_bytes + range_bytes);
  const Direct64 dir{static_cast<const double2*>(z_ref), kern->taps.p, kern->off_d.as<int64_t>(),
                     kern->len_d.as<int>(), kern->real ? 1 : 0};
  const double2* tw = c->twb64.as<double2>() + c->twb64_off[table64(B)];
  dispatch64(B, Q, [&](auto bc, auto qc) {
    constexpr int BB = decltype(bc)::value, QQ = decltype(qc)::value;
    auto seg = k_os64_segments<BB>;
    RF_CUDA(cudaFuncSetAttribute(seg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem64<BB>(0)));
    seg<<<NQ, BB / 16, smem64<BB>(0), s>>>(static_cast<const double2*>(z_ref), n, Lp, tw, Zs, ranges);
    RF_LAUNCHED();
    auto run = [&](auto fn, size_t smem) {
      RF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      for (int j0 = 0; j0 < kern->k; j0 += 65535) {
        const int cnt = std::min(65535, kern->k - j0);
        fn<<<dim3((unsigned)NB, (unsigned)cnt), BB / 16, smem, s>>>(
            Zs, kern->os64_spec.as<double2>(), kern->os64_off_d.as<int64_t>(), kern->os64_parts_d.as<int>(),
            kern->lag0_d.as<int>(), j0, ranges, dir, tw, n, NQ, static_cast<double2*>(z_out), pieces, W, slots);
        RF_LAUNCHED();
      }
    };
    if (win) run(k_os64<BB, QQ, true>, smem64<BB>(H));
    else run(k_os64<BB, QQ, false>, smem64<BB>(0));
  });
  if (win)
    for (int j0 = 0; j0 < kern->k; j0 += 65535) {
      const int cnt = std::min(65535, kern->k - j0);
      k_os64_peaks<<<dim3((unsigned)((nw + 3) / 4), (unsigned)cnt), 128, 0, s>>>(
          pieces, kern->lag0_d.as<int>(), j0, n, NB, H, W, nw, slots, max_out, (int*)argmax_out);
      RF_LAUNCHED();
    }
  return true;
}

}  // namespace rf
