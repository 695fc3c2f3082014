// FP64 / FP32 fitting net (1600 -> 240 -> 240 -> 240 -> 1, forward and data gradient) with digit
// products on the tensor cores (digits.cuh): eight kernels for all centre types.
//
// A GEMM C = A B works on the atoms of one type (rows) and one weight matrix, whose digits are stored as
// m16n8k16 B fragments (built once per weight upload, 16.0 MB a type in FP64, resident in L2).  A is read
// in FP64 / FP32 and cut into digits on the way: lane (g, t) of a warp loads four consecutive k of rows
// g and g + 8, which are its A fragment when k = 16 s + 4 t + {0, 1, 2, 3} stands at the fragment's columns
// 2t, 2t + 1, 2t + 8, 2t + 9.  Rows of A and columns of B carry a power of two of their own, from their largest element
// (the activations too: with their bounds, 1 and 2, nets of small activations lost bits).
//
// Eight warps a CTA share a tile of 16 (8 / WK) rows: WK warps split K (their sums meet in shared
// memory), so that a box of a few hundred atoms, where 16-row tiles times column blocks do not fill
// 152 SMs, is not one long serial chain of K; with many atoms WK = 1 and the warps read the same
// fragments through L1.
#include <cmath>

#include "digits.cuh"
#include "tc_common.cuh"

namespace dpg {
namespace {

using dig::Fmt;

constexpr int kMats = 6;  // W1, W2, W3 (forward), W3^T, W2^T, W1^T (backward)
struct Mat {
  int K, N;
};
__host__ __device__ __forceinline__ Mat mat_of(int q) {
  return q == 0 ? Mat{kKD, kF} : q == 5 ? Mat{kF, kKD} : Mat{kF, kF};
}
// fragment sets (n-tile, k step) before matrix q of a type
__host__ __device__ __forceinline__ int mat_off(int q) {
  constexpr int big = (kKD / 16) * (kF / 8), small = (kF / 16) * (kF / 8);
  return q == 0 ? 0 : big + (q - 1) * small;
}
// Scales of a type's matrices, one an output column: the dropped digit products count against the largest weight of a
// column (one for the whole matrix let a weight of 16,384 beside 0.03 put FP32 energies 7e-4 off).
constexpr int kScales = 5 * kF + kKD;
__host__ __device__ __forceinline__ int scale_off(int q) { return q * kF; }
constexpr int kTypeFrags = 2 * (kKD / 16) * (kF / 8) + 4 * (kF / 16) * (kF / 8);

// n-tiles of a warp.  FP32: three, so that two CTAs of 128 registers a thread fit an SM; six in one CTA reuse the
// A digits twice as often but leave a warp's latency open (six GEMMs, 32,000 rows: 2.46 -> 1.97 ms, 6,912:
// 0.71 -> 0.50, 2,331: 0.33 -> 0.23, 192: 0.089 -> 0.070; five spill: 2.04, 0.54, 0.35, 0.091).  FP64's three
// take 228 to 244 registers.
constexpr int kNTiles = 3;
// k steps whose digit products stay below 2^24 in the accumulators: 7 x 128 x 2^14, 2 x 80 x 2^16
template <class T> struct Flush { static constexpr int v = sizeof(T) == 8 ? 8 : 5; };
constexpr int kWarps = 8;

enum EpiMode { EPI_TANH = 0, EPI_RES_TANH = 1, EPI_BWD = 2, EPI_NONE = 3 };

template <class T>
struct GemmArgs {
  int ntypes, mat, mode;
  const int* type_off;
  const int* type_count;
  const uint4* frag;       // [type][kTypeFrags][Q][32]
  const int* wscale;       // [type][kScales]: a column's |w| 2^sw within the digits' range
  const T* A;              // [rows][K]
  const unsigned* rowmax;  // [rows] top bits of each row's largest |a|
  T* C;                    // [rows][N]
  const T* bias;           // theta: bias of type 0 (types bias_stride apart)
  long stride;             // parameters of a fitting block
  const T* res;            // [rows][N] or, with res_vec, [N] of type 0
  int res_vec;
  const T* aux_in;
  T* aux_out;
  unsigned* outmax;        // row maxima of C, or null
};

// Top bits of |v|: the high word of a double, a float's bits; ordered as unsigned integers.
__device__ __forceinline__ unsigned top_bits(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned top_bits(float v) { return (unsigned)__float_as_int(v) & 0x7fffffffu; }
// Exponent e with |v| < 2^e for all v with these top bits; not finite: a large one.
__device__ __forceinline__ int exp_of(unsigned b, double) { return max((int)(b >> 20) - 1022, -800); }
__device__ __forceinline__ int exp_of(unsigned b, float) {  // with the margin the full digit range needs
  return max((int)((b + 0x10000u) >> 23) - 126, -110);
}
template <class T> struct RowBits { static constexpr int v = sizeof(T) == 8 ? 54 : 26; };

// v 2^(54 - e) rounded, as integers do it (|v| < 2^e): the conversion instruction would take the FP64 pipe.
__device__ __forceinline__ unsigned long long fix_digits(double v, int e) {
  const int hi = __double2hiint(v);
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 33) |
                               ((unsigned long long)(unsigned)__double2loint(v) << 1);  // mantissa x 2
  const int r = min(max(1022 + e - ex, 0), 62);  // (m >> r): v 2^(54 - e) = m 2^(ex - 1076 + 54 - e)
  const long long q = (long long)((m + ((1ull << r) >> 1)) >> r);
  return dig::biased(hi < 0 ? -q : q);
}
__device__ __forceinline__ float fix_digits(float v, int e) {  // below 256
  return v * __int_as_float((127 + min(8 - e, 127)) << 23);
}
__device__ __forceinline__ void split2(unsigned long long u0, unsigned long long u1, uint32_t* out) { dig::split2(u0, u1, out); }
__device__ __forceinline__ void split2(float u0, float u1, uint32_t* out) { dig::split2f(u0, u1, out); }

__device__ __forceinline__ void load4(const double* p, double* v) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void load4(const float* p, float* v) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}

__device__ __forceinline__ double gtanh(double x) { return tanh(x); }
__device__ __forceinline__ float gtanh(float x) { return tanhf(x); }

// Running sums of a warp's outputs over flushes: joined integers (FP64, exact) or floats.
template <class T> struct Sum;
template <> struct Sum<double> {
  long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(const float (*acc)[4], int e) {
    const dig::Pair64 p = dig::join(acc, e);
    hi += p.hi;
    lo += p.lo;
  }
  __device__ __forceinline__ double value() const { return fma((double)hi, 4294967296.0, (double)lo); }
};
template <> struct Sum<float> {
  float s = 0.f;
  __device__ __forceinline__ void add(const float (*acc)[4], int e) { s += dig::join_f(acc, e); }
  __device__ __forceinline__ float value() const { return s; }
};
// The unit of a product is that of its row (|a| < 2^e) times that of its column (|w| 2^sw within the digits' range):
// 2^(40 - (54 - e) - sw) in FP64 (exponents added: the FP64 pipe is scarce), 2^(36 - (26 - e) - sw) in FP32 (two normal
// numbers multiplied).  A row that is not finite: NaN.
template <class T> struct Units;
template <> struct Units<double> {
  using V = int;
  static constexpr int kBad = 1 << 20;
  __device__ static __forceinline__ V row(int e) { return e > 1024 ? kBad : e - 34; }
  __device__ static __forceinline__ V col(int sw) { return 20 - sw; }
  __device__ static __forceinline__ double both(V r, V c) {
    return r == kBad ? __longlong_as_double(0x7ff8000000000000ll) : dig::pow2d(min(max(r + c, -1022), 1023));
  }
};
template <> struct Units<float> {
  using V = float;
  __device__ static __forceinline__ V row(int e) {
    return e > 128 ? __int_as_float(0x7fc00000) : __int_as_float((127 + e - 8) << 23);
  }
  __device__ static __forceinline__ V col(int sw) { return __int_as_float((127 + 18 - sw) << 23); }
  __device__ static __forceinline__ float both(V r, V c) { return r * c; }
};

// The fragments run through shared memory in stages of KS k steps by cp.async, ST stages deep: one pipeline for
// the warps that share a part of K (they multiply the same fragments).  Loads straight
// into registers left each k step waiting for L2 (32,000 FP32 rows: 3.04 ms for the six GEMMs).
template <class T, int WK> struct Pipe {
  static constexpr int KS = (WK == 1 && sizeof(T) == 4) ? 2 : 1;
  static constexpr int ST = WK == 1 ? 4 : 3;
  static constexpr int kWords = KS * kNTiles * dig::Frag<T>::Q * 32;  // uint4 of a stage
  static constexpr size_t kPipe = (size_t)WK * ST * kWords * 16;
  static constexpr size_t kPart = WK == 1 ? 0 : sizeof(T) * kWarps * kNTiles * 4 * 32;  // the partial sums reuse it
  static constexpr size_t kBytes = kPipe > kPart ? kPipe : kPart;
};

template <class T, int WK>
__global__ void __launch_bounds__(32 * kWarps, sizeof(T) == 8 ? 1 : 2) k_dig_gemm(GemmArgs<T> g) {
  constexpr int ND = Fmt<T>::ND, NO = Fmt<T>::NO, Q = dig::Frag<T>::Q, NT = kNTiles, MW = kWarps / WK;
  using P = Pipe<T, WK>;
  extern __shared__ __align__(16) uint4 sm[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, kw = w % WK, mw = w / WK;
  const int tq = lane & 3, gr = lane >> 2;
  // the CTA's type and rows
  int ty = 0, blk = blockIdx.x;
  for (; ty < g.ntypes; ++ty) {
    const int b = (g.type_count[ty] + 16 * MW - 1) / (16 * MW);
    if (blk < b) break;
    blk -= b;
  }
  if (ty == g.ntypes) return;
  const int rows = g.type_count[ty], r0 = (blk * MW + mw) * 16;
  const size_t base = (size_t)g.type_off[ty];
  const Mat mt = mat_of(g.mat);
  const int ntile0 = blockIdx.y * NT, ntiles = mt.N / 8, ksteps = mt.K / 16;
  const uint4* fr = g.frag + ((size_t)ty * kTypeFrags + mat_off(g.mat)) * Q * 32;
  const int* ws = g.wscale + ty * kScales + scale_off(g.mat);
  int ea[2];
  const T* ap[2];
  bool ok[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int row = r0 + gr + 8 * r;
    ok[r] = row < rows;
    const size_t gi = base + (ok[r] ? row : 0);
    ap[r] = g.A + gi * mt.K + 4 * tq;
    ea[r] = exp_of(g.rowmax[gi], T(0));
  }
  Sum<T> sum[NT][4];
  {
    float acc[NT][NO][4];
#pragma unroll
    for (int n = 0; n < NT; ++n) dig::zero_acc<T>(acc[n]);
    const int k0 = ksteps * kw / WK, k1 = ksteps * (kw + 1) / WK;
    const int nst = (k1 - k0 + P::KS - 1) / P::KS;
    uint4* pipe = sm + kw * P::ST * P::kWords;
    auto issue = [&](int st) {
      if (st < nst) {
        uint4* dst = pipe + (st % P::ST) * P::kWords;
        for (int q = 32 * mw + lane; q < P::kWords; q += 32 * MW) {
          const int ln = q % (Q * 32), f = q / (Q * 32), n = f % NT, s = k0 + st * P::KS + f / NT;
          if (s < k1 && ntile0 + n < ntiles) tc::cp_async16(dst + q, fr + ((size_t)(ntile0 + n) * ksteps + s) * Q * 32 + ln);
        }
      }
      tc::cp_async_commit();
    };
    T v[P::KS][2][4];
    auto load_a = [&](int st) {
#pragma unroll
      for (int k = 0; k < P::KS; ++k) {
        const int s = k0 + st * P::KS + k;
#pragma unroll
        for (int r = 0; r < 2; ++r)
          if (ok[r] && s < k1) load4(ap[r] + 16 * s, v[k][r]);
      }
    };
#pragma unroll
    for (int k = 0; k < P::KS; ++k)
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[k][r][q] = T(0);
    for (int st = 0; st < P::ST - 1; ++st) issue(st);
    load_a(0);
    int left = Flush<T>::v;
    for (int st = 0; st < nst; ++st) {
      tc::cp_async_wait_group<P::ST - 2>();
      // the stage has landed, and everyone is done with the one refilled next
      if (MW == 1) __syncwarp();
      else asm volatile("bar.sync %0, %1;" ::"r"(kw + 1), "n"(32 * MW) : "memory");
      issue(st + P::ST - 1);
      uint4 a[P::KS][ND];
#pragma unroll
      for (int k = 0; k < P::KS; ++k) {
        uint32_t x[ND], y[ND], z[ND], u[ND];
        split2(fix_digits(v[k][0][0], ea[0]), fix_digits(v[k][0][1], ea[0]), x);
        split2(fix_digits(v[k][1][0], ea[1]), fix_digits(v[k][1][1], ea[1]), y);
        split2(fix_digits(v[k][0][2], ea[0]), fix_digits(v[k][0][3], ea[0]), z);
        split2(fix_digits(v[k][1][2], ea[1]), fix_digits(v[k][1][3], ea[1]), u);
#pragma unroll
        for (int i = 0; i < ND; ++i) a[k][i] = make_uint4(x[i], y[i], z[i], u[i]);
      }
      if (st + 1 < nst) load_a(st + 1);
      const uint4* buf = pipe + (st % P::ST) * P::kWords + lane;
#pragma unroll
      for (int k = 0; k < P::KS; ++k) {
        const int s = k0 + st * P::KS + k;
        if (s >= k1) break;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if (ntile0 + n < ntiles) {
            uint4 b[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) b[q] = buf[((k * NT + n) * Q + q) * 32];
            dig::block16<T>(acc[n], a[k], b);
          }
        }
        if (--left == 0 || s + 1 == k1) {
#pragma unroll
          for (int n = 0; n < NT; ++n) {
#pragma unroll
            for (int e = 0; e < 4; ++e) sum[n][e].add(acc[n], e);
            dig::zero_acc<T>(acc[n]);
          }
          left = Flush<T>::v;
        }
      }
    }
    tc::cp_async_wait_group<0>();
  }
  T(*part)[NT * 4][32] = reinterpret_cast<T(*)[NT * 4][32]>(sm);  // [warp]
  if (WK > 1) {
    __syncthreads();  // every pipeline is drained
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) part[w][4 * n + e][lane] = sum[n][e].value();
    __syncthreads();
  }
  if (r0 >= rows) return;
  using U = Units<T>;
  const typename U::V ru[2] = {U::row(ea[0]), U::row(ea[1])};
  typename U::V cu[NT][2];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int c = 0; c < 2; ++c)
      cu[n][c] = ntile0 + n < ntiles ? U::col(ws[8 * (ntile0 + n) + 2 * tq + c]) : typename U::V(0);
  const T* bias = g.bias + (long)ty * g.stride;
  const T* resv = g.res + (g.res_vec ? (long)ty * g.stride : 0);
#pragma unroll
  for (int q = 0; q < NT * 4; ++q) {
    if (WK > 1 && q % WK != kw) continue;
    const int n = q >> 2, e = q & 3, r = e >> 1;
    T v;
    if (WK > 1) {
      v = T(0);
#pragma unroll
      for (int k = 0; k < WK; ++k) v += part[mw * WK + k][q][lane];
    } else {
      v = sum[n][e].value();
    }
    const int col = 8 * (ntile0 + n) + 2 * tq + (e & 1);
    const bool in = ok[r] && ntile0 + n < ntiles;
    T out = T(0);
    if (in) {
      v *= U::both(ru[r], cu[n][e & 1]);
      const size_t o = (base + r0 + gr + 8 * r) * mt.N + col;
      if (g.mode == EPI_TANH) {
        out = gtanh(v + bias[col]);
      } else if (g.mode == EPI_RES_TANH) {
        const T t = gtanh(v + bias[col]);
        g.aux_out[o] = t;
        out = g.res[o] + t;
      } else if (g.mode == EPI_BWD) {
        const T h = v + (g.res_vec ? resv[col] : g.res[o]);
        const T f = g.aux_in[o];
        if (g.aux_out) g.aux_out[o] = h;
        out = h * (T(1) - f * f);
      } else {
        out = v;
      }
      g.C[o] = out;
    }
    if (g.outmax) {
      unsigned m = in ? top_bits(out) : 0u;
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      if (in && tq == 0) atomicMax(g.outmax + base + r0 + gr + 8 * r, m);
    }
  }
}

// Row maxima of D (the descriptor), one warp a row.
template <class T>
__global__ void k_dig_rowmax(int N, const T* __restrict__ D, unsigned* out) {
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= N) return;
  unsigned m = 0;
  for (int q = 4 * lane; q < kKD; q += 128) {
    T v[4];
    load4(D + (size_t)row * kKD + q, v);
#pragma unroll
    for (int k = 0; k < 4; ++k) m = max(m, top_bits(v[k]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) out[row] = m;
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// E_i = H3 . w4 + b4 + e_bias[t];  dZ3 = w4 * (1 - T3^2) written over H3, with its row maximum.
template <class T>
__global__ void k_dig_head(int N, const int* __restrict__ itype, T* H3, const T* __restrict__ T3,
                           const T* __restrict__ fit, const T* __restrict__ ebias, double* e_atom, unsigned* outmax) {
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= N) return;
  const int ty = itype[row];
  const T* P = fit + (size_t)ty * kFitParams;
  const size_t r = (size_t)row;
  T e = T(0);
  unsigned m = 0;
  for (int n = lane; n < kF; n += 32) {
    const T h = H3[r * kF + n], t = T3[r * kF + n], w = P[kFw4 + n];
    e += h * w;
    const T dz = w * (T(1) - t * t);
    H3[r * kF + n] = dz;
    m = max(m, top_bits(dz));
  }
  e = warp_sum<T>(e);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    e_atom[r] = (double)e + (double)P[kFb4] + (double)ebias[ty];
    outmax[r] = m;
  }
}

// ------------------------------------------------------------------ weights
// Element (k, n) of matrix q: W[k][n], or W[n][k] for a transpose.
template <class T>
__device__ __forceinline__ T weight(const T* W, int q, const Mat& mt, int k, int n) {
  return q < 3 ? W[(size_t)k * mt.N + n] : W[(size_t)n * mt.K + k];
}
__device__ __forceinline__ long mat_base(int q) { return q == 0 || q == 5 ? kFW1 : q == 1 || q == 4 ? kFW2 : kFW3; }

__device__ __forceinline__ double from_top(unsigned b, double) { return __hiloint2double((int)b, 0); }
__device__ __forceinline__ float from_top(unsigned b, float) { return __int_as_float((int)b); }

// Scale exponent of every output column, one warp each: its largest |w|.  wide: set if a column has a weight above
// kSpread times the rms of its other nonzero ones, or one that is not finite.
template <class T>
__global__ void __launch_bounds__(256) k_dig_fit_scale(const T* __restrict__ fit, int* wscale, int* wide) {
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), ty = blockIdx.y, lane = threadIdx.x & 31;
  if (c >= kScales) return;
  const int q = min(c / kF, kMats - 1), n = c - scale_off(q);
  const Mat mt = mat_of(q);
  const T* W = fit + (size_t)ty * kFitParams + mat_base(q);
  unsigned m = 0;
  for (int k = lane; k < mt.K; k += 32) m = max(m, top_bits(weight(W, q, mt, k, n)));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  // squares of the weights relative to the largest (within 2^-20 in FP64, whose low word `top_bits` leaves out)
  const T inv = T(1) / from_top(m, T(0));
  float sum = 0.f;
  int num = 0, tops = 0;
  for (int k = lane; k < mt.K; k += 32) {
    const T v = weight(W, q, mt, k, n);
    const bool t = top_bits(v) == m;
    const float x = t ? 0.f : (float)(v * inv);
    sum = fmaf(x, x, sum);
    num += v != T(0);
    tops += t;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    num += __shfl_xor_sync(0xffffffffu, num, o);
    tops += __shfl_xor_sync(0xffffffffu, tops, o);
  }
  if (lane == 0) {
    const int e = max(exp_of(m, T(0)), sizeof(T) == 8 ? -200 : -100);
    wscale[ty * kScales + c] = RowBits<T>::v - e;
    const bool even = m == 0 || num <= 1 || (float)(num - 1) <= dig::kSpread * dig::kSpread * (sum + (float)(tops - 1));
    if (!even || e > (sizeof(T) == 8 ? 1024 : 128)) *wide = 1;
  }
}

// B fragments: one warp per fragment set (n-tile, k step) of a type; rows k = 16 s + 4 t + {0..3}.
template <class T>
__global__ void __launch_bounds__(256) k_dig_fit_weights(const T* __restrict__ fit, const int* __restrict__ wscale,
                                                        uint4* frag) {
  constexpr int Q = dig::Frag<T>::Q;
  const int f = blockIdx.x * 8 + (threadIdx.x >> 5), ty = blockIdx.y, lane = threadIdx.x & 31;
  if (f >= kTypeFrags) return;
  int q = 0;
  while (q + 1 < kMats && f >= mat_off(q + 1)) ++q;
  const Mat mt = mat_of(q);
  const int ks = mt.K / 16, idx = f - mat_off(q), nt = idx / ks, s = idx % ks;
  const int col = 8 * nt + (lane >> 2), k0 = 16 * s + 4 * (lane & 3);
  const T* W = fit + (size_t)ty * kFitParams + mat_base(q);
  const int e = RowBits<T>::v - wscale[ty * kScales + scale_off(q) + col];
  decltype(fix_digits(T(0), 0)) u[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) u[k] = fix_digits(weight(W, q, mt, k0 + k, col), e);
  uint32_t lo[2 * Q], hi[2 * Q];
  lo[2 * Q - 1] = hi[2 * Q - 1] = 0u;
  split2(u[0], u[1], lo);
  split2(u[2], u[3], hi);
  uint4* dst = frag + ((size_t)ty * kTypeFrags + f) * Q * 32 + lane;
#pragma unroll
  for (int p = 0; p < Q; ++p) dst[p * 32] = make_uint4(lo[2 * p], hi[2 * p], lo[2 * p + 1], hi[2 * p + 1]);
}

// A model's scales and the flag of a wide column stand before its fragments.
size_t scale_bytes(int ntypes) { return (sizeof(int) * ((size_t)kScales * ntypes + 1) + 255) / 256 * 256; }

template <class T>
const T* theta_of(const Model* m) {
  return sizeof(T) == 8 ? reinterpret_cast<const T*>(m->w64) : reinterpret_cast<const T*>(m->w32);
}

template <class T>
dp_status upload(Model* m) {
  const T* fit = theta_of<T>(m) + (size_t)m->ntypes * m->ntypes * kEmbParams;
  int* ws = static_cast<int*>(m->dig_fit);
  uint4* fr = reinterpret_cast<uint4*>(static_cast<unsigned char*>(m->dig_fit) + scale_bytes(m->ntypes));
  int* wide = ws + (size_t)kScales * m->ntypes;
  DP_CUDA_TRY(m, cudaMemset(wide, 0, sizeof(int)));
  k_dig_fit_scale<T><<<dim3(cdiv(kScales, 8), m->ntypes), 256>>>(fit, ws, wide);
  int h = 0;
  DP_CUDA_TRY(m, cudaMemcpy(&h, wide, sizeof(int), cudaMemcpyDeviceToHost));
  m->dig_fit_ok = h == 0;
  m->launches += 1;
  if (m->dig_fit_ok) {
    k_dig_fit_weights<T><<<dim3(cdiv(kTypeFrags, 8), m->ntypes), 256>>>(fit, ws, fr);
    m->launches += 1;
  }
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

template <class T, int WK>
dp_status gemm(Model* m, int N, const GemmArgs<T>& g) {
  const int mt = 16 * (kWarps / WK);
  DP_CUDA_TRY(m, ensure_smem(reinterpret_cast<const void*>(k_dig_gemm<T, WK>), Pipe<T, WK>::kBytes));
  const dim3 grid(cdiv(N, mt) + m->ntypes, cdiv(mat_of(g.mat).N / 8, kNTiles));
  k_dig_gemm<T, WK><<<grid, 32 * kWarps, Pipe<T, WK>::kBytes, m->stream>>>(g);
  m->launches += 1;
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

template <class T>
dp_status run(Model* m, int N) {
  const T* theta = theta_of<T>(m);
  const size_t emb = (size_t)m->ntypes * m->ntypes * kEmbParams;
  const T* fit = theta + emb;
  const T* ebias = fit + (size_t)m->ntypes * kFitParams;
  T* act[5];
  for (int q = 0; q < 5; ++q) act[q] = static_cast<T*>(m->act[q]);
  unsigned* mx = static_cast<unsigned*>(m->dig_max);
  const size_t R = (size_t)m->max_atoms;
  DP_CUDA_TRY(m, cudaMemsetAsync(mx + 2 * R, 0, 4 * 4 * R, m->stream));
  k_dig_rowmax<T><<<cdiv(N, 8), 256, 0, m->stream>>>(N, static_cast<const T*>(m->Dm), mx);
  m->launches += 1;
  GemmArgs<T> g{};
  g.ntypes = m->ntypes; g.type_off = m->type_off; g.type_count = m->type_count;
  g.wscale = static_cast<const int*>(m->dig_fit);
  g.frag = reinterpret_cast<const uint4*>(static_cast<unsigned char*>(m->dig_fit) + scale_bytes(m->ntypes));
  g.stride = kFitParams;
  // rows times column blocks against the SMs decide how far K is split inside a CTA: the least splitting
  // (most reuse of the fragments) that still gives four CTAs an SM
  auto go = [&](const GemmArgs<T>& a) {
    const long blocks = cdiv(mat_of(a.mat).N / 8, kNTiles), want = 4l * num_sms();
    if (cdiv(N, 128) * blocks >= want) return gemm<T, 1>(m, N, a);
    if (cdiv(N, 64) * blocks >= want) return gemm<T, 2>(m, N, a);
    if (cdiv(N, 32) * blocks >= want) return gemm<T, 4>(m, N, a);
    return gemm<T, 8>(m, N, a);
  };
#define DP_GO(a)                      \
  do {                                \
    const dp_status s_ = go(a);       \
    if (s_ != DP_OK) return s_;       \
  } while (0)
  // F1: H1 = tanh(D W1 + b1)
  g.mat = 0; g.A = static_cast<const T*>(m->Dm); g.rowmax = mx; g.C = act[0]; g.bias = fit + kFb1; g.mode = EPI_TANH;
  g.outmax = mx + 4 * R;
  DP_GO(g);
  // F2: T2 = tanh(H1 W2 + b2), H2 = H1 + T2
  g.mat = 1; g.A = act[0]; g.rowmax = mx + 4 * R; g.C = act[2]; g.bias = fit + kFb2; g.res = act[0];
  g.aux_out = act[1]; g.mode = EPI_RES_TANH; g.outmax = mx + 5 * R;
  DP_GO(g);
  // F3: T3 = tanh(H2 W3 + b3), H3 = H2 + T3
  g.mat = 2; g.A = act[2]; g.rowmax = mx + 5 * R; g.C = act[4]; g.bias = fit + kFb3; g.res = act[2]; g.aux_out = act[3];
  g.outmax = nullptr;
  DP_GO(g);
  k_dig_head<T><<<cdiv(N, 8), 256, 0, m->stream>>>(N, m->itype, act[4], act[3], fit, ebias, m->e_atom, mx + R);
  m->launches += 1;
  // B3: dH2 = w4 + dZ3 W3^T ; dZ2 = dH2 (1 - T2^2)  (dH2 -> act[3], dZ2 -> act[2])
  g.mat = 3; g.A = act[4]; g.rowmax = mx + R; g.C = act[2]; g.res = fit + kFw4; g.res_vec = 1; g.aux_in = act[1];
  g.aux_out = act[3]; g.mode = EPI_BWD; g.outmax = mx + 2 * R;
  DP_GO(g);
  // B2: dH1 = dH2 + dZ2 W2^T ; dZ1 = dH1 (1 - H1^2)  (dZ1 -> act[1])
  g.mat = 4; g.A = act[2]; g.rowmax = mx + 2 * R; g.C = act[1]; g.res = act[3]; g.res_vec = 0; g.aux_in = act[0];
  g.aux_out = nullptr; g.outmax = mx + 3 * R;
  DP_GO(g);
  // B1: dD = dZ1 W1^T
  g.mat = 5; g.A = act[1]; g.rowmax = mx + 3 * R; g.C = static_cast<T*>(m->dD); g.mode = EPI_NONE; g.outmax = nullptr;
  DP_GO(g);
#undef DP_GO
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

}  // namespace

size_t dig_fit_bytes(int ntypes, bool fp64) {
  return scale_bytes(ntypes) + (size_t)ntypes * kTypeFrags * 512 * (fp64 ? dig::Frag<double>::Q : dig::Frag<float>::Q);
}
dp_status dig_fit_upload(Model* m) { return m->prec == DP_FP64 ? upload<double>(m) : upload<float>(m); }
dp_status launch_dig_fitting(Model* m, int N) { return m->prec == DP_FP64 ? run<double>(m, N) : run<float>(m, N); }

}  // namespace dpg
