// FP64 / FP32 embedding net, T = R_hat^T G and the embedding backward with every matrix product as
// digit products on the tensor cores (digits.cuh).
//
// One warp works on a tile of 16 neighbour rows of one (atom, neighbour type) segment.  The m16n8
// accumulator fragment of one layer is, register for register, the A fragment of the next (lane
// (g, t) = (lane / 4, lane % 4) holds rows g and g + 8 and the units of its slots), so activations
// never leave their lane; the units are numbered so that the two units that share a residual (k and
// k + 25 of layer 2, m and m + 50 of layer 3) are the two columns of one lane:
//   layer 1   slot p (0..6)          unit k = 4 p + t                      (28 slots for 25 units)
//   layer 2   n-tile p, column 2t+e  unit m = 4 p + t + 25 e               (7 n-tiles)
//   layer 3   n-tile j, column 2t+e  unit q = m(j, t) + 50 e               (13 n-tiles)
//             m(j, t) = 4 (j / 2) + t + 25 (j % 2) for j < 12; m(12, 0) = 24, m(12, 1) = 49
// Weight fragments are built once per weight upload in this order (k_dig_weights), one 16-byte load
// per lane and two digits, and are read through L1 / L2 (262 KB a pair in FP64, 100 KB in FP32).
// Scales: weights by the output column, FP32 activations and all gradients by the row, FP64 activations by
// their range; nets that these do not suit take the plain kernels (layer_scale, activations_large).
//
// What bounds it: FP64 keeps layer-1 sums, T, dE/dT products and the environment rows on the FP64
// pipe (64 clocks a warp instruction); tanh and the activations are fixed-point integers.
#include <cmath>
#include <cstring>

#include "digits.cuh"

namespace dpg {
namespace {

using dig::Fmt;

// ------------------------------------------------------------------ layout of one pair's weights
constexpr int kS1 = 7;                      // layer-1 slots
constexpr int kT2 = 7, kK2 = 2;             // layer 2: n-tiles, k steps
constexpr int kT3 = 13, kK3 = 4;            // layer 3 (the last k step has 8 columns)
constexpr int kT3T = 7, kK3T = 7;           // dz3 W3^T (the last k step has 8 columns)
constexpr int kT2T = 4, kK2T = 4;           // dz2 W2^T (likewise)
constexpr int kF2 = 0, kF3 = kF2 + kT2 * kK2, kF3T = kF3 + kT3 * kK3, kF2T = kF3T + kT3T * kK3T,
              kFrags = kF2T + kT2T * kK2T;  // fragment sets of a pair

// uint4 words of a fragment set: FP64 four 16-byte loads a lane (digits 2q, 2q + 1; the eighth is zero); FP32
// a 16-byte load (digits 0, 1) and an 8-byte one (digit 2).
template <class T> struct SetWords { static constexpr int v = sizeof(T) == 8 ? 128 : 48; };

__host__ __device__ __forceinline__ int unit2(int p, int t, int e) { return 4 * p + t < kN1 ? 4 * p + t + kN1 * e : -1; }
__host__ __device__ __forceinline__ int unit3m(int j, int t) {
  if (j < 12) return 4 * (j >> 1) + t + kN1 * (j & 1);
  return t == 0 ? 24 : t == 1 ? 49 : -1;
}

// Scales of a pair, one for every output of a product (a column of W, a row of W for the transposes): its weights
// times 2^sw fill half (FP64) or 255/256 (FP32) of the digits' range.  The dropped digit products count against
// the largest weight of a column, so a scale for the whole matrix let one large weight take the bits of every other
// column (largest weight 30,000 beside 0.1: G 1.2e-3 off in FP32, 6e-14 in FP64; with these 6e-8 and 2e-16).
// FP64: z of an output is a fixed-point number with zs fraction bits, the upper four orders shifted left by s, the
// lower four right by 32 - s.
struct PairScale {
  int sw2[kN2], zs2[kN2], s2[kN2], sw3[kN3], zs3[kN3], s3[kN3];
  int swt3[kN2], swt2[kN1];  // rows of W3, W2
};

// Constants of one output: bias and scale.
template <class T> struct Out;
template <> struct __align__(16) Out<double> {
  long long b;  // fixed point, zs bits
  int zs, s;
};
template <> struct __align__(8) Out<float> {
  float b, c;   // z = c (sum of orders) + b
};
// Bias and layer-1 constants of a pair, and the factors of the transposed products.
template <class T>
struct __align__(16) PairSmall {
  T w1[4 * kS1], b1[4 * kS1];       // [slot][t]
  Out<T> o2[8 * kT2], o3[8 * kT3];  // [n-tile][2 t + e]
  T c3t[8 * kT3T], c2t[4 * kS1];    // [n-tile][2 t + e], [slot][t]: unit of dz3 W3^T, dz2 W2^T
};

template <class T>
struct DigArgs {
  int N, ntypes, S, sp;        // sp: tasks an atom's tiles are dealt to
  int sel_off[kMaxTypes + 1];
  T rc, rs, winv;
  int switch_kind;
  const T* stat;
  const uint4* frag;           // [pair][kFrags][SetWords]
  const PairSmall<T>* small;   // [pair]
  const dig::TanhTab* tab;     // FP64
  const int* itype;
  const int* nl_j;
  const void* nl_d;
  const int* nl_count;
  T* Tm;                       // [N][4][100]
  const T* dT;                 // [N][100][4], 1/S included
  const T* dTmax;              // [N][4] max |dT| per component
  double* force;
  double* vir_atom;
};

template <class T>
__device__ __forceinline__ void pair_vec(const void* nl_d, size_t e, T* d);
template <>
__device__ __forceinline__ void pair_vec<float>(const void* nl_d, size_t e, float* d) {
  const float4 v = static_cast<const float4*>(nl_d)[e];
  d[0] = v.x; d[1] = v.y; d[2] = v.z;
}
template <>
__device__ __forceinline__ void pair_vec<double>(const void* nl_d, size_t e, double* d) {
  const dvec4 v = static_cast<const dvec4*>(nl_d)[e];
  d[0] = v.x; d[1] = v.y; d[2] = v.z;
}

// Environment row: R_hat and what the backward needs of it (1/r, switch and its derivative).
template <class T>
struct Env {
  T d[3], R[4], rinv, sw, dsw;
};
template <class T>
__device__ __forceinline__ void env_row(const DigArgs<T>& a, int ti, Env<T>& v) {
  const T r = sqrt(v.d[0] * v.d[0] + v.d[1] * v.d[1] + v.d[2] * v.d[2]);
  v.rinv = T(1) / r;
  if (r < a.rs) {
    v.sw = T(1); v.dsw = T(0);
  } else if (r >= a.rc) {
    v.sw = T(0); v.dsw = T(0);
  } else {
    const T u = (r - a.rs) * a.winv;
    if (a.switch_kind == 1) {
      const T pi = T(3.14159265358979323846);
      v.sw = T(0.5) * cos(pi * u) + T(0.5);
      v.dsw = T(-0.5) * pi * sin(pi * u) * a.winv;
    } else {
      const T u2 = u * u;
      v.sw = u2 * u * (T(-6) * u2 + T(15) * u - T(10)) + T(1);
      v.dsw = T(-30) * u2 * (u - T(1)) * (u - T(1)) * a.winv;
    }
  }
  const T s = v.sw * v.rinv, q = s * v.rinv;
  v.R[0] = s; v.R[1] = q * v.d[0]; v.R[2] = q * v.d[1]; v.R[3] = q * v.d[2];
#pragma unroll
  for (int c = 0; c < 4; ++c) v.R[c] = (v.R[c] - a.stat[ti * 4 + c]) * a.stat[(a.ntypes + ti) * 4 + c];
}

// Exponent e with |v| <= 2^e (v finite), from the bits; zero and tiny values give the lower limit.
__device__ __forceinline__ int exp_above(double v) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  return max(e - 1022, -800);
}
__device__ __forceinline__ int exp_above(float v) {
  const int e = (__float_as_int(v) >> 23) & 0xff;
  return max(e - 126, -80);
}
__device__ __forceinline__ double pow2t(int e, double) { return dig::pow2d(e); }
__device__ __forceinline__ float pow2t(int e, float) { return __int_as_float((127 + min(max(e, -126), 127)) << 23); }
// 1 / c of a power of two c
__device__ __forceinline__ float unit_inv(float c) { return __int_as_float((254 << 23) - __float_as_int(c)); }

// ------------------------------------------------------------------ activations of either type
// FP64: fixed point with 54 fraction bits; FP32: floats.
__device__ __forceinline__ long long act1(double x, double w, double b, const dig::TanhTab* tab) {
  return dig::tanh_fixed(__double2ll_rn(fma(x, w, b) * 72057594037927936.0), 56, tab);  // saturates beyond 128
}
__device__ __forceinline__ float act1(float x, float w, float b, const dig::TanhTab*) { return tanhf(fmaf(x, w, b)); }

// tanh of element e's output; u: the unit of the row's digits (FP32).
__device__ __forceinline__ long long act(const float (*acc)[4], int e, const Out<double>& o, double, const dig::TanhTab* tab) {
  const dig::Pair64 p = dig::join(acc, e);
  const int r = 32 - o.s;
  const long long z = (p.hi << o.s) + ((p.lo + ((1ll << r) >> 1)) >> r) + o.b;
  return dig::tanh_fixed(z, o.zs, tab);
}
__device__ __forceinline__ float act(const float (*acc)[4], int e, const Out<float>& o, float u, const dig::TanhTab*) {
  return tanhf(fmaf(dig::join_f(acc, e), o.c * u, o.b));
}

// The biased digits of activations: h1 (|h1| <= 1) and h2 (|h2| <= 2); FP32: the value times f, below 256.
__device__ __forceinline__ unsigned long long dig_h1(long long h, double) { return dig::biased(h); }
__device__ __forceinline__ unsigned long long dig_h2(long long h, double) { return dig::biased((h + 1) >> 1); }
__device__ __forceinline__ float dig_h1(float h, float f) { return h * f; }
__device__ __forceinline__ float dig_h2(float h, float f) { return h * f; }
__device__ __forceinline__ unsigned long long dig_of(double v) { return dig::biased(__double2ll_rn(v)); }
__device__ __forceinline__ float dig_of(float v) { return v; }

template <class T> struct DigWord;
template <> struct DigWord<double> { using U = unsigned long long; };
template <> struct DigWord<float> { using U = float; };
__device__ __forceinline__ void split2(unsigned long long u0, unsigned long long u1, uint32_t* out) { dig::split2(u0, u1, out); }
__device__ __forceinline__ void split2(float u0, float u1, uint32_t* out) { dig::split2f(u0, u1, out); }

// A fragment of one k step (all digits) from the lane's four slots of rows g (u[0]) and g + 8 (u[1]); only the
// first two slots unless `full`.
template <class T>
__device__ __forceinline__ void get_a(uint4* a, const typename DigWord<T>::U (*u)[4], bool full) {
  constexpr int ND = Fmt<T>::ND;
  uint32_t x[ND], y[ND], z[ND], w[ND];
  split2(u[0][0], u[0][1], x);
  split2(u[1][0], u[1][1], y);
  if (full) {
    split2(u[0][2], u[0][3], z);
    split2(u[1][2], u[1][3], w);
  }
#pragma unroll
  for (int i = 0; i < ND; ++i) a[i] = make_uint4(x[i], y[i], full ? z[i] : 0u, full ? w[i] : 0u);
}

// The lane's B fragments of one set.
template <class T>
__device__ __forceinline__ void load_b(uint4* b, const uint4* __restrict__ set, int lane) {
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = __ldg(set + q * 32 + lane);
  } else {
    b[0] = __ldg(set + lane);
    const uint2 c = __ldg(reinterpret_cast<const uint2*>(set + 32) + lane);
    b[1] = make_uint4(c.x, c.y, 0u, 0u);
  }
}

// Where a tile's A operand lives.  FP32 (kRegs): digits in registers, since reading A again for every n-tile
// made those kernels bound by shared-memory bandwidth.  FP64 forward (kDigits): digits in the warp's
// shared memory, 112 bytes a lane and k step.  FP64 backward (kWords): the slots' 56-bit digit words, 64
// bytes, cut into digits on every use, so that six warps fit an SM instead of four (8.66 -> 7.30 ms for 4,000 Cu
// atoms, 7.55 with a scale for every column; the forward, which has its eight warps anyway, would lose: 2.73 -> 3.10 ms).
enum Store { kRegs, kDigits, kWords };

// acc = A (KS k steps) times the fragments of one n-tile; with TAIL the last step has 8 columns.
template <class T, int KS, bool TAIL, Store ST>
__device__ __forceinline__ void product(float (*acc)[4], const uint4* A, const uint4* __restrict__ fr, int lane) {
  constexpr int ND = Fmt<T>::ND, Q = dig::Frag<T>::Q;
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const bool tail = TAIL && s == KS - 1;
    uint4 b[Q], a[ND];
    load_b<T>(b, fr + s * SetWords<T>::v, lane);
    if constexpr (ST == kWords) {
      typename DigWord<T>::U u[2][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (tail && q >= 2) break;
        const uint4 w = A[(4 * s + q) * 32 + lane];
        u[0][q] = ((unsigned long long)w.y << 32) | w.x;
        u[1][q] = ((unsigned long long)w.w << 32) | w.z;
      }
      get_a<T>(a, u, !tail);
    } else if constexpr (ST == kDigits) {
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        if (tail) {
          const uint2 w = reinterpret_cast<const uint2*>(A + s * ND * 32)[i * 32 + lane];
          a[i] = make_uint4(w.x, w.y, 0u, 0u);
        } else {
          a[i] = A[(s * ND + i) * 32 + lane];
        }
      }
    } else {
#pragma unroll
      for (int i = 0; i < ND; ++i) a[i] = A[s * ND + i];
    }
    if (tail) {
      uint2 a8[ND];
#pragma unroll
      for (int i = 0; i < ND; ++i) a8[i] = make_uint2(a[i].x, a[i].y);
      dig::block8<T>(acc, a8, b);
    } else if (s == 0) {
      dig::block16<T, true>(acc, a, b);
    } else {
      dig::block16<T>(acc, a, b);
    }
  }
}
// A of k step s into its store.
template <class T, Store ST>
__device__ __forceinline__ void put_a(uint4* A, int s, bool full, int lane, const typename DigWord<T>::U (*u)[4]) {
  constexpr int ND = Fmt<T>::ND;
  if constexpr (ST == kWords) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (full || q < 2)
        A[(4 * s + q) * 32 + lane] = make_uint4((uint32_t)u[0][q], (uint32_t)(u[0][q] >> 32), (uint32_t)u[1][q],
                                                (uint32_t)(u[1][q] >> 32));
  } else if constexpr (ST == kDigits) {
    uint4 a[ND];
    get_a<T>(a, u, full);
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      if (full) A[(s * ND + i) * 32 + lane] = a[i];
      else reinterpret_cast<uint2*>(A + s * ND * 32)[i * 32 + lane] = make_uint2(a[i].x, a[i].y);
    }
  } else {
    get_a<T>(A + s * ND, u, full);
  }
}
// FP32: the activation of h2 slot (p, e), row r, back from the digits in registers (their unit is u): within 2^-30 of the
// row's largest.
__device__ __forceinline__ float from_digits(const uint4* A, int p, int e, int r, float u) {
  constexpr int ND = Fmt<float>::ND;
  float v = 0.f;
#pragma unroll
  for (int i = ND - 1; i >= 0; --i) {
    const uint4& w = A[(p >> 1) * ND + i];
    const uint32_t h = (p & 1) ? (r ? w.w : w.z) : (r ? w.y : w.x);
    const __half2 x = *reinterpret_cast<const __half2*>(&h);
    v += e ? __high2float(x) : __low2float(x);
  }
  return v * u;
}

// FP32: the digits of a tile's rows (g: r = 0, g + 8: r = 1) are relative to the row's largest activation: f = 2^(8 - e),
// u = 1 / f with |h| <= 2^e in the lane's slots and, by shuffles, those of the row's other three lanes.  With a fixed
// range a net whose activations are small lost bits (|h| ~ 1e-4: G 2e-4 off; now 8e-8, FMAs 1e-7).
template <int M>
__device__ __forceinline__ void row_scale(const float (*h)[2], float* f, float* u) {
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    float top = fabsf(h[0][r]);
#pragma unroll
    for (int p = 1; p < M; ++p) top = fmaxf(top, fabsf(h[p][r]));
    top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 1));
    top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
    f[r] = pow2t(8 - exp_above(top), 0.f);
    u[r] = unit_inv(f[r]);
  }
}

// Layers 1 and 2 of a tile: h1 [slot][row], h2 [n-tile][e][row] (rows g, g + 8; FP64), and the digits of h2
// in A (shared memory, FP64) or A (registers, FP32, which takes h2 back from them) with their units uh (FP32).
template <class T, Store ST>
__device__ __forceinline__ void layers12(const PairSmall<T>& sm, const uint4* __restrict__ fr,
                                         T x0, T x1, const dig::TanhTab* tab, uint4* A, int lane,
                                         typename Fmt<T>::V (*h1)[2], typename Fmt<T>::V (*h2)[2][2], T* uh) {
  constexpr int ND = Fmt<T>::ND;
  constexpr bool D = sizeof(T) == 8;
  using V = typename Fmt<T>::V;
  using U = typename DigWord<T>::U;
  const int t = lane & 3;
#pragma unroll
  for (int p = 0; p < kS1; ++p) {
    const T w = sm.w1[4 * p + t], b = sm.b1[4 * p + t];  // zero beyond unit 24: h1 = 0
    h1[p][0] = act1(x0, w, b, tab);
    h1[p][1] = act1(x1, w, b, tab);
  }
  T f[2] = {T(1), T(1)}, u1[2] = {T(1), T(1)};
  if constexpr (!D) row_scale<kS1>(h1, f, u1);
  uint4 A1r[D ? 1 : kK2 * ND];
  uint4* A1 = D ? A : A1r;
#pragma unroll
  for (int s = 0; s < kK2; ++s) {
    U u[2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 2; ++r) u[r][q] = 4 * s + q < kS1 ? dig_h1(h1[4 * s + q < kS1 ? 4 * s + q : 0][r], f[r]) : dig_h1(V(0), f[r]);
    put_a<T, ST>(A1, s, true, lane, u);
  }
  if (D) __syncwarp();
  U u[2][4];
  V hf[D ? 1 : 2 * kT2][2];  // FP32: h2, until the row's largest is known
#pragma unroll
  for (int p = 0; p < kT2; ++p) {
    float acc[Fmt<T>::NO][4];
    product<T, kK2, false, ST>(acc, A1, fr + (size_t)(kF2 + p * kK2) * SetWords<T>::v, lane);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const Out<T> o = sm.o2[8 * p + 2 * t + e];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const V h = h1[p][r] + act(acc, 2 * r + e, o, u1[r], tab);
        if constexpr (D) h2[p][e][r] = h;
        else hf[2 * p + e][r] = h;
      }
    }
  }
  if constexpr (!D) {
    row_scale<2 * kT2>(hf, f, uh);
#pragma unroll
    for (int p = 0; p < kT2; ++p) {
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int r = 0; r < 2; ++r) u[r][2 * (p & 1) + e] = dig_h2(hf[2 * p + e][r], f[r]);
      if ((p & 1) || p == kT2 - 1) put_a<T, ST>(A, p >> 1, p & 1, lane, u);
    }
  } else {
    __syncwarp();
#pragma unroll
    for (int s = 0; s < kK3; ++s) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int p = 2 * s + (q >> 1);
          u[r][q] = p < kT2 ? dig_h2(h2[p < kT2 ? p : 0][q & 1][r], f[r]) : dig_h2(V(0), f[r]);
        }
      put_a<T, ST>(A, s, s + 1 < kK3, lane, u);
    }
    __syncwarp();
  }
}
template <class T>
__device__ __forceinline__ typename Fmt<T>::V h2_of(const uint4* A, const typename Fmt<T>::V (*h2)[2][2], int p, int e, int r, const T* uh) {
  if constexpr (sizeof(T) == 8) return h2[p][e][r];
  else return from_digits(A, p, e, r, uh[r]);
}

__device__ __forceinline__ double to_t(long long v) { return (double)v; }  // times 2^-54 later
__device__ __forceinline__ float to_t(float v) { return v; }
template <class T> struct Unit { };
template <> struct Unit<double> { static constexpr double v = 1.0 / 18014398509481984.0; };  // 2^-54
template <> struct Unit<float> { static constexpr float v = 1.f; };

// A warp's work: task (atom i, share sub of its tiles).  The 16-row tiles of all neighbour types of the
// atom are numbered in one sequence; tile q belongs to the task with sub = q % sp.
// warps a CTA (one CTA an SM): FP64 needs 255 registers a thread, FP32 runs in 128
template <class T> struct FwdWarps { static constexpr int v = sizeof(T) == 8 ? 8 : 16; };
constexpr int kADigits = (kK3 - 1) * Fmt<double>::ND * 32 + Fmt<double>::ND * 16;  // FP64 digits of a tile, in uint4
constexpr int kAWords = (4 * (kK3 - 1) + 2) * 32, kZWords = (4 * (kK3T - 1) + 2) * 32;  // FP64 digit words
template <class T>
struct FwdWarp {  // shared memory of one warp
  uint4 A[sizeof(T) == 8 ? kADigits : 1];
  T G[16][34];
  T R[16][4];
};

// ------------------------------------------------------------------ forward
template <class T>
__global__ void __launch_bounds__(32 * FwdWarps<T>::v, 1) k_dig_fwd(DigArgs<T> a) {
  extern __shared__ __align__(16) unsigned char raw[];
  constexpr bool D = sizeof(T) == 8;
  constexpr int W = FwdWarps<T>::v;
  constexpr Store ST = D ? kDigits : kRegs;
  using V = typename Fmt<T>::V;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = lane & 3, g = lane >> 2;
  dig::TanhTab* tab = reinterpret_cast<dig::TanhTab*>(raw);
  if (D) {
    const uint4* src = reinterpret_cast<const uint4*>(a.tab);
    for (int q = threadIdx.x; q < (int)(sizeof(dig::TanhTab) / 16); q += 32 * W)
      reinterpret_cast<uint4*>(tab)[q] = src[q];
    __syncthreads();
  }
  FwdWarp<T>& sw = reinterpret_cast<FwdWarp<T>*>(raw + (D ? (sizeof(dig::TanhTab) + 15) / 16 * 16 : 0))[w];
  const long ntask = (long)a.N * a.sp;
  for (long task = (long)blockIdx.x * W + w; task < ntask; task += (long)gridDim.x * W) {
    const int i = (int)(task / a.sp), sub = (int)(task - (long)i * a.sp);
    const int ti = a.itype[i];
    T accT[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) accT[q][c] = T(0);
    int q0 = 0;  // tiles of the atom so far
    for (int tj = 0; tj < a.ntypes; ++tj) {
      const int cnt = a.nl_count[(size_t)i * a.ntypes + tj];
      const int nt = (cnt + 15) >> 4;
      const int pair = ti * a.ntypes + tj;
      const PairSmall<T>& sm = a.small[pair];
      const uint4* fr = a.frag + (size_t)pair * kFrags * SetWords<T>::v;
      int first = (sub - q0) % a.sp;
      if (first < 0) first += a.sp;
      q0 += nt;
      for (int tile = first; tile < nt; tile += a.sp) {
        const int base = tile * 16;
        __syncwarp();
        if (lane < 16) {
          Env<T> v;
#pragma unroll
          for (int c = 0; c < 4; ++c) v.R[c] = T(0);
          if (base + lane < cnt) {
            pair_vec<T>(a.nl_d, (size_t)i * a.S + a.sel_off[tj] + base + lane, v.d);
            env_row<T>(a, ti, v);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) sw.R[lane][c] = v.R[c];
        }
        __syncwarp();
        V h1[kS1][2], h2[D ? kT2 : 1][2][2];
        uint4 Ar[D ? 1 : kK3 * Fmt<T>::ND];
        uint4* A = D ? sw.A : Ar;
        T uh[2] = {T(1), T(1)};
        layers12<T, ST>(sm, fr, sw.R[g][0], sw.R[g + 8][0], tab, A, lane, h1, h2, uh);
#pragma unroll
        for (int grp = 0; grp < 4; ++grp) {
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int j = 4 * grp + jj;
            if (j >= kT3) break;
            float acc[Fmt<T>::NO][4];
            product<T, kK3, true, ST>(acc, A, fr + (size_t)(kF3 + j * kK3) * SetWords<T>::v, lane);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              V res;
              if (j < 12) {
                res = h2_of<T>(A, h2, j < 12 ? j >> 1 : 0, j & 1, r, uh);
              } else {  // unit 24 (lane 0 of the quad, its own) and unit 49 (held by lane 0, used by lane 1)
                const V o = __shfl_sync(0xffffffffu, h2_of<T>(A, h2, 6, 1, r, uh), lane & ~3);
                res = t == 0 ? h2_of<T>(A, h2, 6, 0, r, uh) : o;
              }
#pragma unroll
              for (int e = 0; e < 2; ++e)
                sw.G[g + 8 * r][8 * jj + 2 * t + e] = to_t(res + act(acc, 2 * r + e, sm.o3[8 * j + 2 * t + e], uh[r], tab));
            }
          }
          __syncwarp();
          if (grp < 3) {  // lane = unit
#pragma unroll
            for (int rr = 0; rr < 16; ++rr) {
              const T gv = sw.G[rr][lane];
#pragma unroll
              for (int c = 0; c < 4; ++c) accT[grp][c] = fma(sw.R[rr][c], gv, accT[grp][c]);
            }
          } else {        // n-tile 12 has four units: lane = (row pair, unit)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int rr = 2 * g + k;
              const T gv = sw.G[rr][t];
#pragma unroll
              for (int c = 0; c < 4; ++c) accT[3][c] = fma(sw.R[rr][c], gv, accT[3][c]);
            }
          }
          __syncwarp();
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) accT[3][c] += __shfl_xor_sync(0xffffffffu, accT[3][c], o);
#pragma unroll
    for (int grp = 0; grp < 4; ++grp) {
      const int j = 4 * grp + (grp < 3 ? lane >> 3 : 0), col = grp < 3 ? lane & 7 : lane;
      if (grp == 3 && lane >= 4) break;
      const int q = unit3m(j, col >> 1) + kN2 * (col & 1);
      T* dst = a.Tm + (size_t)i * 4 * kN3 + q;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const T v = accT[grp][c] * Unit<T>::v;
        if (a.sp == 1) dst[c * kN3] = v;
        else atomicAdd(dst + c * kN3, v);
      }
    }
  }
}

// ------------------------------------------------------------------ descriptor, dE/dT
// T (sums over neighbours, unscaled) -> T = (sum + padded slots) / S, D = T^T T[:, :16]; block per atom.
template <class T>
__global__ void __launch_bounds__(128) k_dig_desc(int N, int nt, T invS, const T* __restrict__ pad,
                                                  const int* __restrict__ itype, const int* __restrict__ cnt,
                                                  int4 sel, T* Tm, T* Dm) {
  __shared__ T s[4 * kN3];
  const int i = blockIdx.x, tid = threadIdx.x;
  const int ti = itype[i];
  const int sl[4] = {sel.x, sel.y, sel.z, sel.w};
  T* Ti = Tm + (size_t)i * 4 * kN3;
  for (int q = tid; q < 4 * kN3; q += 128) {
    T v = Ti[q];
    if (pad)
      for (int tj = 0; tj < nt; ++tj)
        v += T(sl[tj] - cnt[(size_t)i * nt + tj]) * pad[(size_t)(ti * nt + tj) * 4 * kN3 + q];
    v *= invS;
    s[q] = v;
    Ti[q] = v;
  }
  __syncthreads();
  for (int q = tid; q < kKD; q += 128) {
    const int aa = q >> 4, b = q & 15;
    T v = T(0);
#pragma unroll
    for (int c = 0; c < 4; ++c) v += s[c * kN3 + aa] * s[c * kN3 + b];
    Dm[(size_t)i * kKD + q] = v;
  }
}

// dT[a][c] = (1/S) (sum_b dD[a][b] T[c][b] + [a < 16] sum_a' dD[a'][a] T[c][a']), feature-major, and the
// largest |dT| of each component (the bound of the backward's row scales); block per atom.
template <class T>
__global__ void __launch_bounds__(128) k_dig_dT(int N, T invS, const T* __restrict__ Tm, const T* __restrict__ dD, T* dT,
                                                T* dTmax) {
  __shared__ T s[4 * kN3], sd[kKD + kN3];  // dD rows of 17: no bank conflicts down a column
  __shared__ T red[4][4];
  const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int q = tid; q < 4 * kN3; q += 128) s[q] = Tm[(size_t)i * 4 * kN3 + q];
  for (int q = tid; q < kKD; q += 128) sd[q + (q >> 4)] = dD[(size_t)i * kKD + q];
  __syncthreads();
  T v[4] = {T(0), T(0), T(0), T(0)};
  if (tid < kN3) {
#pragma unroll
    for (int b = 0; b < kM2; ++b) {
      const T x = sd[tid * 17 + b];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] += x * s[c * kN3 + b];
    }
    if (tid < kM2)
      for (int a2 = 0; a2 < kN3; ++a2) {
        const T x = sd[a2 * 17 + tid];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] += x * s[c * kN3 + a2];
      }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[c] *= invS;
      dT[((size_t)i * kN3 + tid) * 4 + c] = v[c];
      v[c] = fabs(v[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[c] = fmax(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
    if (lane == 0) red[w][c] = v[c];
  }
  __syncthreads();
  if (tid < 4) dTmax[(size_t)i * 4 + tid] = fmax(fmax(red[0][tid], red[1][tid]), fmax(red[2][tid], red[3][tid]));
}

// ------------------------------------------------------------------ backward
// FP64 keeps digit words and the residual part of dE/dh2 (r) in shared memory: 29.5 KB a warp, six warps an SM.
// FP32 holds the digits in registers, multiplies each k step of dz3 as soon as it exists and sums dE/dh2 in
// registers; shared memory is left to L1, which keeps the weights (100 KB a pair).
template <class T>
struct BwdWarp {
  static constexpr bool D = sizeof(T) == 8;
  uint4 A[D ? kAWords : 1];                                // digits of h1, h2, then dz2
  uint4 Z[D ? kZWords : 1];                                     // digits of dz3
  T r[D ? 2 * 2 * kT2 : 1][32];                                 // dG[m] + dG[m + 50], then dz2, lane-private
  union {
    struct {
      T R[16][4];                                               // R_hat scaled by the row's power of two
      T x[16];
    };
    T out[16][5];                                               // dR_hat, d s_hat (after the last read of R)
  };
  T env[6][16];                                                 // d, 1/r, switch and derivative of each row
  T g3[3][16];                                                  // dE/dd of each row
  int sd[16];
};
// Warps a CTA.  FP32: 12 (168 registers) with one atom type; 16 (128 registers, some spills) with more, whose
// weights (100 KB a pair) overflow L1 and leave more latency to hide: 32,000 Cu atoms 4.79 (12) and 5.10 ms (16),
// 2,331 water atoms 325 and 282 us.
constexpr int kBwdWarps64 = 6, kBwdWarps32 = 12, kBwdWarps32Types = 16;

// Product value of element e (FP64: orders joined in units of 2^40; FP32: weights are 2^(18 - sw) times their digits).
__device__ __forceinline__ double value(const float (*acc)[4], int e, double scale) {
  const dig::Pair64 p = dig::join(acc, e);
  return fma((double)p.hi, 4294967296.0, (double)p.lo) * scale;
}
__device__ __forceinline__ float value(const float (*acc)[4], int e, float scale) { return dig::join_f(acc, e) * scale; }
// Gradients are scaled to |v| <= 2^GradBits (1 - 1/128), the digits' whole range.
template <class T> struct GradBits { static constexpr int v = sizeof(T) == 8 ? 55 : 8; };
template <class T> struct ProdUnit { static constexpr int v = sizeof(T) == 8 ? 40 : 18; };

// g (1 - t^2) with t = tau 2^-54 (FP64) or tau (FP32)
__device__ __forceinline__ double times_sech2(double g, long long tau) {
  const double x = (double)tau;
  return fma(g * x, x * -3.0814879110195774e-33, g);  // 2^-108
}
__device__ __forceinline__ float times_sech2(float g, float tau) { return g * fmaf(-tau, tau, 1.f); }

// The value as FP64.  The conversion instruction takes the FP64 pipe for 64 clocks; a float's bits move by
// integer instructions (subnormals become zero).
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = (uint32_t)__float_as_int(v), e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
  const uint32_t x = e == 255u ? 0x7ffu : e + 896u;
  return __hiloint2double((int)((b & 0x80000000u) | (e == 0u ? 0u : (x << 20) | (m >> 3))), (int)(e == 0u ? 0u : m << 29));
}
// Sum over a tile's rows first, first + 2, ... of g (plain) or -g d, in FP64.  FP32 rows: exact products, and sums of three
// floats (70 bits and more, so no less than FP64's 53) that are widened once a tile; the FP64 form was 18% of the FP64
// pipe and a chain of 16 DFMAs.
__device__ __forceinline__ double tile_sum(const double* g, const double* d, bool plain, int first, int rows) {
  double s = 0.0;
  for (int k = first; k < rows; k += 2) s = fma(g[k], plain ? 1.0 : -d[k], s);
  return s;
}
__device__ __forceinline__ float two_sum(float& s, float x) {  // s += x; returns what was rounded off
  const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
  const float r = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
  s = t;
  return r;
}
__device__ __forceinline__ double tile_sum(const float* g, const float* d, bool plain, int first, int rows) {
  float s = 0.f, c = 0.f, l = 0.f;
  for (int k = first; k < rows; k += 2) {
    const float x = g[k], y = plain ? 1.f : -d[k];
    const float p = __fmul_rn(x, y), e = __fmaf_rn(x, y, -p);
    const float r = two_sum(s, p), q = two_sum(c, e);
    l = __fadd_rn(l, __fadd_rn(two_sum(c, r), q));
  }
  return (double)s + ((double)c + (double)l);
}

// Embedding backward with recompute, prod_force and the per-atom virial.  Everything downstream of
// dG = R_hat . dT carries the row's power of two 2^sd (a bound of |dG| from max |dT|), so dz3 is ready
// to be cut into digits and the products come out in one scale for the whole warp.
template <class T, int W>
__global__ void __launch_bounds__(32 * W, 1) k_dig_bwd(DigArgs<T> a) {
  extern __shared__ __align__(16) unsigned char raw[];
  constexpr bool D = sizeof(T) == 8;
  constexpr int ND = Fmt<T>::ND, Q = dig::Frag<T>::Q;
  constexpr Store ST = D ? kWords : kRegs;
  using V = typename Fmt<T>::V;
  using U = typename DigWord<T>::U;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = lane & 3, g = lane >> 2;
  dig::TanhTab* tab = reinterpret_cast<dig::TanhTab*>(raw);
  if (D) {
    const uint4* src = reinterpret_cast<const uint4*>(a.tab);
    for (int q = threadIdx.x; q < (int)(sizeof(dig::TanhTab) / 16); q += 32 * W) reinterpret_cast<uint4*>(tab)[q] = src[q];
    __syncthreads();
  }
  BwdWarp<T>& sw = reinterpret_cast<BwdWarp<T>*>(raw + (D ? (sizeof(dig::TanhTab) + 15) / 16 * 16 : 0))[w];
  const long ntask = (long)a.N * a.sp;
  for (long task = (long)blockIdx.x * W + w; task < ntask; task += (long)gridDim.x * W) {
    const int i = (int)(task / a.sp), sub = (int)(task - (long)i * a.sp);
    const int ti = a.itype[i];
    const T* dTi = a.dT + (size_t)i * kN3 * 4;
    T bmax[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) bmax[c] = a.dTmax[(size_t)i * 4 + c];
    int q0 = 0;
    bool any = false;
    double mine = 0.0;  // lanes 0..2: centre force, 3..11: virial, over even rows; 12..23: odd rows
    for (int tj = 0; tj < a.ntypes; ++tj) {
      const int cnt = a.nl_count[(size_t)i * a.ntypes + tj];
      const int nt = (cnt + 15) >> 4;
      const int pair = ti * a.ntypes + tj;
      const PairSmall<T>& sm = a.small[pair];
      const uint4* fr = a.frag + (size_t)pair * kFrags * SetWords<T>::v;
      int first = (sub - q0) % a.sp;
      if (first < 0) first += a.sp;
      q0 += nt;
      for (int tile = first; tile < nt; tile += a.sp) {
        const int base = tile * 16;
        const size_t e0 = (size_t)i * a.S + a.sel_off[tj] + base + lane;
        const bool row = lane < 16 && base + lane < cnt;
        any = true;
        __syncwarp();
        if (lane < 16) {
          Env<T> v;
#pragma unroll
          for (int c = 0; c < 4; ++c) v.R[c] = T(0);
          if (row) {
            pair_vec<T>(a.nl_d, e0, v.d);
            env_row<T>(a, ti, v);
          }
          T b = T(0);
#pragma unroll
          for (int c = 0; c < 4; ++c) b = fma(fabs(v.R[c]), bmax[c], b);
          const int sd = GradBits<T>::v - exp_above(b * T(1.0 + 1.0 / 128));
          const T f = pow2t(sd, T(0));
          sw.sd[lane] = sd;
          sw.x[lane] = v.R[0];
          if (row) {
#pragma unroll
            for (int c = 0; c < 3; ++c) sw.env[c][lane] = v.d[c];
            sw.env[3][lane] = v.rinv;
            sw.env[4][lane] = v.sw;
            sw.env[5][lane] = v.dsw;
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) sw.R[lane][c] = v.R[c] * f;
        }
        __syncwarp();
        V h1[kS1][2], h2[D ? kT2 : 1][2][2];
        uint4 Ar[D ? 1 : kK3 * ND];
        uint4* A = D ? sw.A : Ar;
        T uh[2] = {T(1), T(1)};
        layers12<T, ST>(sm, fr, sw.x[g], sw.x[g + 8], tab, A, lane, h1, h2, uh);
        T R[2][4], dR[2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            R[r][c] = sw.R[g + 8 * r][c];
            dR[r][c] = T(0);
          }
        // layer 3: G, dR_hat, dG, dz3 (digits), residual dG[m] + dG[m + 50]; then
        // dE/dh2 = residual + dz3 W3^T, dz2 = dE/dh2 (1 - t2^2), the residual part of dE/dh1
        T dh1[kS1][2];
        T dh2[D ? 1 : kT2][2][2];  // FP32: dE/dh2 in the units of dz3 W3^T, then dz2
        if constexpr (!D) {
#pragma unroll
          for (int p = 0; p < kT2; ++p)
#pragma unroll
            for (int e = 0; e < 2; ++e) dh2[p][e][0] = dh2[p][e][1] = T(0);
        }
        U u[2][4];
#pragma unroll
        for (int j = 0; j < kT3; ++j) {
          float acc[Fmt<T>::NO][4];
          product<T, kK3, true, ST>(acc, A, fr + (size_t)(kF3 + j * kK3) * SetWords<T>::v, lane);
          const int m = unit3m(j, t);
          T dt[2][4];
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int c = 0; c < 4; ++c) dt[e][c] = (j < 12 || m >= 0) ? dTi[(m + kN2 * e) * 4 + c] : T(0);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            V res;
            if (j < 12) {
              res = h2_of<T>(A, h2, j < 12 ? j >> 1 : 0, j & 1, r, uh);
            } else {
              const V o = __shfl_sync(0xffffffffu, h2_of<T>(A, h2, 6, 1, r, uh), lane & ~3);
              res = t == 0 ? h2_of<T>(A, h2, 6, 0, r, uh) : o;
            }
            T sum = T(0);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const V t3 = act(acc, 2 * r + e, sm.o3[8 * j + 2 * t + e], uh[r], tab);
              const T G = to_t(res + t3);
              T dg = T(0);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                dR[r][c] = fma(dt[e][c], G, dR[r][c]);
                dg = fma(R[r][c], dt[e][c], dg);
              }
              u[r][2 * (j & 1) + e] = dig_of(times_sech2(dg, t3));
              sum += dg;
            }
            if (j < 12) {
              if constexpr (D) sw.r[2 * j + r][lane] = sum;
              else dh2[j >> 1][j & 1][r] = fmaf(sum, unit_inv(sm.c3t[8 * (j >> 1) + 2 * t + (j & 1)]), dh2[j >> 1][j & 1][r]);
            } else {  // slot (6, 0) of lane 0 and, from lane 1, slot (6, 1)
              const T o = __shfl_sync(0xffffffffu, sum, (lane & ~3) + 1);
              if constexpr (D) {
                sw.r[24 + r][lane] = t == 0 ? sum : T(0);
                sw.r[26 + r][lane] = t == 0 ? o : T(0);
              } else {
                dh2[kT2 - 1][0][r] = fmaf(t == 0 ? sum : T(0), unit_inv(sm.c3t[8 * (kT2 - 1) + 2 * t]), dh2[kT2 - 1][0][r]);
                dh2[kT2 - 1][1][r] = fmaf(t == 0 ? o : T(0), unit_inv(sm.c3t[8 * (kT2 - 1) + 2 * t + 1]), dh2[kT2 - 1][1][r]);
              }
            }
          }
          if constexpr (D) {
            if ((j & 1) || j == kT3 - 1) put_a<T, ST>(sw.Z, j >> 1, j & 1, lane, u);
          } else if ((j & 1) || j == kT3 - 1) {  // this k step against every n-tile of W3^T
            uint4 za[ND];
            get_a<T>(za, u, j & 1);
#pragma unroll
            for (int p = 0; p < kT3T; ++p) {
              const uint4* set = fr + (size_t)(kF3T + p * kK3T + (j >> 1)) * SetWords<T>::v;
              if (j & 1) {
                uint4 b[Q];
                load_b<T>(b, set, lane);
                dig::block16<T, true>(acc, za, b);
              } else {
                dig::zero_acc<T>(acc);
                product<T, 1, true, ST>(acc, za, set, lane);
              }
#pragma unroll
              for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int r = 0; r < 2; ++r) dh2[p][e][r] += dig::join_f(acc, 2 * r + e);
            }
          }
        }
        __syncwarp();
        T top[2] = {T(0), T(0)};
#pragma unroll
        for (int p = 0; p < kT3T; ++p) {
          float acc[Fmt<T>::NO][4];
          if constexpr (D) product<T, kK3T, true, ST>(acc, sw.Z, fr + (size_t)(kF3T + p * kK3T) * SetWords<T>::v, lane);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            dh1[p][r] = T(0);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const T c3 = sm.c3t[8 * p + 2 * t + e];
              T g2;
              if constexpr (D) g2 = sw.r[4 * p + 2 * e + r][lane] + value(acc, 2 * r + e, c3);
              else g2 = dh2[p][e][r] * c3;
              const T dz = times_sech2(g2, h2_of<T>(A, h2, p, e, r, uh) - h1[p][r]);
              if constexpr (D) sw.r[4 * p + 2 * e + r][lane] = dz;
              else dh2[p][e][r] = dz;
              top[r] = fmax(top[r], fabs(dz));
              dh1[p][r] += g2;
            }
          }
        }
        int sd2[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          top[r] = fmax(top[r], __shfl_xor_sync(0xffffffffu, top[r], 1));
          top[r] = fmax(top[r], __shfl_xor_sync(0xffffffffu, top[r], 2));
          sd2[r] = GradBits<T>::v - exp_above(top[r] * T(1.0 + 1.0 / 128));
        }
        {
          const T f[2] = {pow2t(sd2[0], T(0)), pow2t(sd2[1], T(0))};
#pragma unroll
          for (int s = 0; s < kK2T; ++s) {
            U z[2][4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const int p = 2 * s + (q >> 1);
                T v = T(0);
                if (p < kT2) {
                  if constexpr (D) v = sw.r[4 * p + 2 * (q & 1) + r][lane];
                  else v = dh2[p < kT2 ? p : 0][q & 1][r];
                }
                z[r][q] = dig_of(v * f[r]);
              }
            put_a<T, ST>(A, s, s + 1 < kK2T, lane, z);  // the digits of h2 are no longer needed
          }
        }
        __syncwarp();
        // dE/dh1 = residual + dz2 W2^T, then d s_hat
        T ds[2] = {T(0), T(0)};
        {
          T sc[2];
#pragma unroll
          for (int r = 0; r < 2; ++r) sc[r] = pow2t(-sd2[r], T(0));
#pragma unroll
          for (int n = 0; n < kT2T; ++n) {
            float acc[Fmt<T>::NO][4];
            product<T, kK2T, true, ST>(acc, A, fr + (size_t)(kF2T + n * kK2T) * SetWords<T>::v, lane);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int p = 2 * n + e;
              if (p >= kS1) break;
              const T w1 = sm.w1[4 * p + t], c2 = sm.c2t[4 * p + t];
#pragma unroll
              for (int r = 0; r < 2; ++r) {
                const T g1 = dh1[p][r] + value(acc, 2 * r + e, c2 * sc[r]);
                ds[r] = fma(times_sech2(g1, h1[p][r]), w1, ds[r]);
              }
            }
          }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            ds[r] += __shfl_xor_sync(0xffffffffu, ds[r], o);
#pragma unroll
            for (int c = 0; c < 4; ++c) dR[r][c] += __shfl_xor_sync(0xffffffffu, dR[r][c], o);
          }
        if (t == 0)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            sw.out[g + 8 * r][4] = ds[r] * pow2t(-sw.sd[g + 8 * r], T(0));
#pragma unroll
            for (int c = 0; c < 4; ++c) sw.out[g + 8 * r][c] = dR[r][c] * Unit<T>::v;
          }
        __syncwarp();
        if (row) {
          T o[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) o[c] = sw.out[lane][c];
          o[0] += sw.out[lane][4];
#pragma unroll
          for (int c = 0; c < 4; ++c) o[c] *= a.stat[(a.ntypes + ti) * 4 + c];
          const T d[3] = {sw.env[0][lane], sw.env[1][lane], sw.env[2][lane]};
          const T rinv = sw.env[3][lane], sf = sw.env[4][lane], dsf = sw.env[5][lane];
          const T dsr = dsf * rinv - sf * rinv * rinv;
          const T qv = sf * rinv * rinv;
          const T dq = dsf * rinv * rinv - T(2) * sf * rinv * rinv * rinv;
          const T proj = o[1] * d[0] + o[2] * d[1] + o[3] * d[2];
          const T common = (o[0] * dsr + dq * proj) * rinv;
          const int jn = a.nl_j[e0];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const T g3 = common * d[c] + qv * o[1 + c];
            sw.g3[c][lane] = g3;
            atomicAdd(&a.force[3 * (size_t)jn + c], -widen(g3));
          }
        }
        __syncwarp();
        if (lane < 24) {  // k = c: sum of g_c; k = 3 + 3 p + q: -sum of g_p d_q
          const int k = lane < 12 ? lane : lane - 12;
          const int c = k < 3 ? k : (k - 3) / 3, q = k < 3 ? 0 : (k - 3) % 3;
          mine += tile_sum(sw.g3[c], sw.env[q], k < 3, lane >= 12, min(16, cnt - base));
        }
      }
    }
    if (any) {
      mine += __shfl_down_sync(0xffffffffu, mine, 12);
      if (lane < 3) atomicAdd(&a.force[3 * (size_t)i + lane], mine);
      else if (lane < 12) atomicAdd(&a.vir_atom[(size_t)i * 9 + lane - 3], mine);
    }
  }
}

// ------------------------------------------------------------------ weights
// Fixed-point form of a weight in the scale sw.
__device__ __forceinline__ unsigned long long weight_digits(double v, int sw, double) {
  return dig::biased(__double2ll_rn(v * dig::pow2d(sw)));
}
__device__ __forceinline__ float weight_digits(float v, int sw, float) {
  return v * __int_as_float((127 + sw - 18) << 23);  // |.| < 256
}

// B fragments of every pair: block (fragment set, pair), one warp.
template <class T>
__global__ void __launch_bounds__(32) k_dig_weights(const T* __restrict__ theta, const PairScale* scale, uint4* frag) {
  constexpr int Q = dig::Frag<T>::Q;
  const int lane = threadIdx.x, t = lane & 3, n = lane >> 2;  // B fragment: k rows 2t.., column n
  const int f = blockIdx.x, pair = blockIdx.y;
  const T* W = theta + (size_t)pair * kEmbParams;
  const PairScale& ps = scale[pair];
  const int tc = n >> 1, ec = n & 1;  // column n = 2 tc + ec
  typename DigWord<T>::U u[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {  // the lane's four k rows: 2t, 2t + 1, 2t + 8, 2t + 9
    const int hi = k >> 1, par = k & 1;
    T v = T(0);
    int sw = 0;
    if (f < kF3) {
      const int p = (f - kF2) / kK2, s = (f - kF2) % kK2;
      const int kk = 4 * (4 * s + 2 * hi + par) + t, m = unit2(p, tc, ec);
      if (m >= 0) sw = ps.sw2[m];
      if (kk < kN1 && m >= 0) v = W[kEW2 + kk * kN2 + m];
    } else if (f < kF3T) {
      const int j = (f - kF3) / kK3, s = (f - kF3) % kK3;
      const int m = 2 * s + hi < kT2 ? unit2(2 * s + hi, t, par) : -1, mo = unit3m(j, tc);
      if (mo >= 0) sw = ps.sw3[mo + kN2 * ec];
      if (m >= 0 && mo >= 0) v = W[kEW3 + m * kN3 + mo + kN2 * ec];
    } else if (f < kF2T) {
      const int p = (f - kF3T) / kK3T, s = (f - kF3T) % kK3T;
      const int j = 2 * s + hi;
      const int mi = j < kT3 ? unit3m(j, t) : -1, m = unit2(p, tc, ec);
      if (m >= 0) sw = ps.swt3[m];
      if (mi >= 0 && m >= 0) v = W[kEW3 + m * kN3 + mi + kN2 * par];
    } else {
      const int r = (f - kF2T) / kK2T, s = (f - kF2T) % kK2T;
      const int m = 2 * s + hi < kT2 ? unit2(2 * s + hi, t, par) : -1, k1 = 4 * (2 * r + ec) + tc;
      if (k1 < kN1) sw = ps.swt2[k1];
      if (m >= 0 && k1 < kN1) v = W[kEW2 + k1 * kN2 + m];
    }
    u[k] = weight_digits(v, sw, T(0));
  }
  uint32_t lo[2 * Q], hi[2 * Q];
  lo[2 * Q - 1] = hi[2 * Q - 1] = 0u;  // an odd number of digits
  split2(u[0], u[1], lo);
  split2(u[2], u[3], hi);
  uint4* dst = frag + ((size_t)pair * kFrags + f) * SetWords<T>::v;
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int q = 0; q < Q; ++q) dst[q * 32 + lane] = make_uint4(lo[2 * q], hi[2 * q], lo[2 * q + 1], hi[2 * q + 1]);
  } else {
    dst[lane] = make_uint4(lo[0], hi[0], lo[1], hi[1]);
    reinterpret_cast<uint2*>(dst + 32)[lane] = make_uint2(lo[2], hi[2]);
  }
}

__device__ __forceinline__ void set_out(Out<double>& o, double b, int, int zs, int s) {
  o.b = __double2ll_rn(b * dig::pow2d(zs));
  o.zs = zs;
  o.s = s;
}
__device__ __forceinline__ void set_out(Out<float>& o, float b, int sw, int, int) {
  o.b = b;
  o.c = pow2t(18 - sw, 0.f);
}

template <class T>
__global__ void __launch_bounds__(128) k_dig_small(const T* __restrict__ theta, const PairScale* scale, PairSmall<T>* out) {
  const int pair = blockIdx.x, q = threadIdx.x;
  const T* W = theta + (size_t)pair * kEmbParams;
  const PairScale& ps = scale[pair];
  PairSmall<T>& o = out[pair];
  if (q < 4 * kS1) {
    o.w1[q] = q < kN1 ? W[kEW1 + q] : T(0);
    o.b1[q] = q < kN1 ? W[kEb1 + q] : T(0);
    o.c2t[q] = q < kN1 ? pow2t(ProdUnit<T>::v - ps.swt2[q], T(0)) : T(1);
  }
  const int t = (q & 7) >> 1, e = q & 1;
  if (q < 8 * kT2) {
    const int m = unit2(q >> 3, t, e), k = max(m, 0);  // no unit: zero digits, the scale of unit 0
    set_out(o.o2[q], m >= 0 ? W[kEb2 + m] : T(0), ps.sw2[k], ps.zs2[k], ps.s2[k]);
    o.c3t[q] = m >= 0 ? pow2t(ProdUnit<T>::v - ps.swt3[m], T(0)) : T(1);
  }
  if (q < 8 * kT3) {
    const int m = unit3m(q >> 3, t), k = m >= 0 ? m + kN2 * e : 0;
    set_out(o.o3[q], m >= 0 ? W[kEb3 + k] : T(0), ps.sw3[k], ps.zs3[k], ps.s3[k]);
  }
}

// Smallest e with v <= 2^e.
int ceil_log2(double v) {
  int e = 0;
  const double f = std::frexp(v, &e);  // v = f 2^e, 0.5 <= f < 1
  return f == 0.5 ? e - 1 : e;
}

// 2^sw times weights of at most `top`: half of the digits' range (FP64), 2^26 (1 - 2^-8) of 2^26 (FP32).
int digit_scale(double top, bool fp64, int lowest) {
  const int e = top > 0.0 ? std::max(ceil_log2(fp64 ? top : top * (1.0 + 1.0 / 128)), lowest) : 0;
  return (fp64 ? Fmt<double>::BD * Fmt<double>::ND - 2 : Fmt<float>::BD * Fmt<float>::ND - 1) - e;
}

// No weight of a column (n of them, `stride` apart) above kSpread times the rms of its other nonzero ones.
bool even_column(const double* w, int n, int stride) {
  double top = 0.0, sum = 0.0;
  int num = 0;
  for (int k = 0; k < n; ++k) {
    const double v = std::fabs(w[(size_t)k * stride]);
    top = std::fmax(top, v);
    sum += v * v;
    num += v != 0.0;
  }
  return num <= 1 || top * top * (num - 1) <= dig::kSpread * dig::kSpread * (sum - top * top);
}

// Scales of one layer (K x N weights W, biases b, |inputs| <= in, FP64 activations with sh fraction bits): sw, zs and s
// of every column, swt of every row; false when the weights are outside the range the fixed-point layer covers
// (or not finite), or with `even` spread too far.
bool layer_scale(const double* W, const double* b, int K, int N, double in, bool fp64, bool even, int sh, int* sw, int* zs,
                 int* s, int* swt) {
  std::vector<double> row(K, 0.0);
  for (int n = 0; n < N; ++n) {
    double top = 0.0, sum = std::fabs(b[n]);
    for (int k = 0; k < K; ++k) {
      const double v = std::fabs(W[(size_t)k * N + n]);
      if (!(v <= 65536.0)) return false;
      top = std::fmax(top, v);
      row[k] = std::fmax(row[k], v);
      sum += in * v;
    }
    if (!(sum <= 1048576.0) || (even && !even_column(W + n, K, N))) return false;
    sw[n] = digit_scale(top, fp64, fp64 ? -12 : -100);
    zs[n] = std::min(56, 60 - (sum > 1.0 ? ceil_log2(sum) : 0));
    s[n] = 72 + zs[n] - sh - sw[n];
    if (fp64 && s[n] > 31) {  // large weights: fewer fraction bits in z
      zs[n] -= s[n] - 31;
      s[n] = 31;
    }
    if (fp64 && (s[n] < 1 || zs[n] < 40)) return false;
  }
  for (int k = 0; k < K; ++k) {
    if (even && !even_column(W + (size_t)k * N, N, 1)) return false;
    swt[k] = digit_scale(row[k], fp64, -100);
  }
  return true;
}

// FP64 activations have 54 fraction bits whatever their size, tanh an absolute error of 2^-55: on nets whose activations
// are small that is worse than FMAs and a relative tanh (rms of h1 0.5: G 7e-17 off against 1.7e-16; 0.27: 1.3 / 1.8e-16;
// 0.11: 3.1 / 1.9e-16; 0.01: 2.8e-15 / 1.9e-16).  True if the rms over units of h1 and of h2, over the inputs at 14
// distances up to r_c, is at least kActivations.
constexpr double kActivations = 0.2;
bool activations_large(const Model* m, const double* W, int ti) {
  double s1 = 0.0, s2 = 0.0;
  for (int k = 2; k < 16; ++k) {
    const double r = m->rc * (k + 0.5) / 16.0, u = (r - m->rs) / (m->rc - m->rs);
    const double sw = u <= 0.0 ? 1.0 : m->switch_kind == 1 ? 0.5 * std::cos(3.14159265358979323846 * u) + 0.5
                                                            : u * u * u * (-6.0 * u * u + 15.0 * u - 10.0) + 1.0;
    const double x = (sw / r - m->davg_host[4 * ti]) / m->dstd_host[4 * ti];
    double h1[kN1];
    for (int q = 0; q < kN1; ++q) {
      h1[q] = std::tanh(x * W[kEW1 + q] + W[kEb1 + q]);
      s1 += h1[q] * h1[q];
    }
    for (int n = 0; n < kN2; ++n) {
      double z = W[kEb2 + n];
      for (int q = 0; q < kN1; ++q) z += h1[q] * W[kEW2 + q * kN2 + n];
      const double h2 = h1[n % kN1] + std::tanh(z);
      s2 += h2 * h2;
    }
  }
  const double least = kActivations * kActivations * 14.0;
  return s1 >= least * kN1 && s2 >= least * kN2;
}

// A pair's scales stand before its constants and fragments.
size_t scale_bytes(int npairs) { return (sizeof(PairScale) * npairs + 255) / 256 * 256; }

template <class T>
dp_status upload(Model* m) {
  const int np = m->ntypes * m->ntypes;
  constexpr int bits = Fmt<T>::BD * Fmt<T>::ND;
  constexpr bool d = sizeof(T) == 8;
  std::vector<PairScale> sc(np);
  // The plain FP64 kernels keep all pairs of a centre type in shared memory, which holds three: four types multiply in
  // digits whatever their spread.
  const bool even = !d || m->ntypes <= 3;
  m->dig_ok = true;
  for (int p = 0; p < np; ++p) {
    const double* W = m->theta_host.data() + (size_t)p * kEmbParams;
    PairScale& q = sc[p];
    m->dig_ok = m->dig_ok && layer_scale(W + kEW2, W + kEb2, kN1, kN2, 1.0, d, even, bits - 2, q.sw2, q.zs2, q.s2, q.swt2) &&
                layer_scale(W + kEW3, W + kEb3, kN2, kN3, 2.0, d, even, bits - 3, q.sw3, q.zs3, q.s3, q.swt3) &&
                (!d || !even || activations_large(m, W, p / m->ntypes));
  }
  if (!m->dig_ok) return DP_OK;
  unsigned char* base = static_cast<unsigned char*>(m->dig_emb);
  PairScale* dsc = reinterpret_cast<PairScale*>(base);
  DP_CUDA_TRY(m, cudaMemcpy(dsc, sc.data(), sizeof(PairScale) * np, cudaMemcpyHostToDevice));
  const T* th = sizeof(T) == 8 ? reinterpret_cast<const T*>(m->w64) : reinterpret_cast<const T*>(m->w32);
  PairSmall<T>* sm = reinterpret_cast<PairSmall<T>*>(base + scale_bytes(np));
  uint4* fr = reinterpret_cast<uint4*>(base + scale_bytes(np) + sizeof(PairSmall<T>) * np);
  k_dig_weights<T><<<dim3(kFrags, np), 32>>>(th, dsc, fr);
  k_dig_small<T><<<np, 128>>>(th, dsc, sm);
  m->launches += 2;
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

template <class T>
DigArgs<T> make_args(Model* m, int N) {
  DigArgs<T> a{};
  const int np = m->ntypes * m->ntypes;
  a.N = N; a.ntypes = m->ntypes; a.S = m->S;
  for (int t = 0; t <= m->ntypes; ++t) a.sel_off[t] = m->sel_off[t];
  a.rc = (T)m->rc; a.rs = (T)m->rs; a.winv = (T)(1.0 / (m->rc - m->rs)); a.switch_kind = m->switch_kind;
  a.stat = sizeof(T) == 8 ? reinterpret_cast<const T*>(m->stat64) : reinterpret_cast<const T*>(m->stat32);
  unsigned char* base = static_cast<unsigned char*>(m->dig_emb);
  a.small = reinterpret_cast<const PairSmall<T>*>(base + scale_bytes(np));
  a.frag = reinterpret_cast<const uint4*>(base + scale_bytes(np) + sizeof(PairSmall<T>) * np);
  a.tab = static_cast<const dig::TanhTab*>(m->dig_tanh);
  a.itype = m->itype; a.nl_j = m->nl_j; a.nl_d = m->nl_d; a.nl_count = m->nl_count;
  a.Tm = static_cast<T*>(m->Tm);
  a.dT = static_cast<const T*>(m->dig_dT);
  a.dTmax = a.dT + (size_t)m->max_atoms * 4 * kN3;
  a.force = m->force; a.vir_atom = m->vir_atom;
  return a;
}

template <class T>
size_t fwd_smem() {
  return (sizeof(T) == 8 ? (sizeof(dig::TanhTab) + 15) / 16 * 16 : 0) + FwdWarps<T>::v * sizeof(FwdWarp<T>);
}
template <class T>
size_t bwd_smem(int warps) {
  return (sizeof(T) == 8 ? (sizeof(dig::TanhTab) + 15) / 16 * 16 : 0) + warps * sizeof(BwdWarp<T>);
}

// Tasks per atom: enough warp tasks (about 16 a resident warp) that the last wave is short; at most about one a
// tile (lists hold two thirds of S in water, a third in Cu), since a task's sums cost a few hundred atomics.
// A 192-atom water box has six tiles an atom: with four tasks half the warps took two tiles (forward 146 us).
int split_of(const Model* m, int N, int warps) {
  const long want = 16l * num_sms() * warps;
  const int most = std::max(1, m->S / 23);
  return (int)std::max(1l, std::min((long)most, (want + N - 1) / N));
}

template <class T>
dp_status forward(Model* m, int N) {
  DigArgs<T> a = make_args<T>(m, N);
  const size_t smem = fwd_smem<T>();
  const void* fn = reinterpret_cast<const void*>(k_dig_fwd<T>);
  DP_CUDA_TRY(m, ensure_smem(fn, smem, true));
  constexpr int W = FwdWarps<T>::v;
  const int per = blocks_per_sm(fn, 32 * W, smem);
  a.sp = split_of(m, N, W * per);
  if (a.sp > 1) DP_CUDA_TRY(m, cudaMemsetAsync(m->Tm, 0, sizeof(T) * 4 * kN3 * (size_t)N, m->stream));
  const int grid = (int)std::min((long)num_sms() * per, ((long)N * a.sp + W - 1) / W);
  k_dig_fwd<T><<<grid, 32 * W, smem, m->stream>>>(a);
  const T* pad = !m->has_pad ? nullptr
                             : (sizeof(T) == 8 ? reinterpret_cast<const T*>(m->pad64) : reinterpret_cast<const T*>(m->pad32));
  k_dig_desc<T><<<N, 128, 0, m->stream>>>(N, m->ntypes, T(1) / (T)m->S, pad, m->itype, m->nl_count,
                                          make_int4(m->sel[0], m->sel[1], m->sel[2], m->sel[3]), a.Tm,
                                          static_cast<T*>(m->Dm));
  m->launches += 2;
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

template <class T>
dp_status backward(Model* m, int N) {
  DigArgs<T> a = make_args<T>(m, N);
  k_dig_dT<T><<<N, 128, 0, m->stream>>>(N, T(1) / (T)m->S, a.Tm, static_cast<const T*>(m->dD), const_cast<T*>(a.dT),
                                        const_cast<T*>(a.dTmax));
  auto kern = k_dig_bwd<T, sizeof(T) == 8 ? kBwdWarps64 : kBwdWarps32>;
  int W = sizeof(T) == 8 ? kBwdWarps64 : kBwdWarps32;
  if constexpr (sizeof(T) == 4)
    if (m->ntypes > 1) {
      kern = k_dig_bwd<T, kBwdWarps32Types>;
      W = kBwdWarps32Types;
    }
  const size_t smem = bwd_smem<T>(W);
  const void* fn = reinterpret_cast<const void*>(kern);
  DP_CUDA_TRY(m, ensure_smem(fn, smem, true));
  const int per = blocks_per_sm(fn, 32 * W, smem);
  a.sp = split_of(m, N, W * per);
  DP_CUDA_TRY(m, cudaMemsetAsync(m->vir_atom, 0, sizeof(double) * 9 * (size_t)N, m->stream));
  const int grid = (int)std::min((long)num_sms() * per, ((long)N * a.sp + W - 1) / W);
  kern<<<grid, 32 * W, smem, m->stream>>>(a);
  m->launches += 2;
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

}  // namespace

size_t dig_emb_bytes(int ntypes, bool fp64) {
  const size_t np = (size_t)ntypes * ntypes;
  return scale_bytes((int)np) + np * (fp64 ? sizeof(PairSmall<double>) + (size_t)kFrags * SetWords<double>::v * 16
                                           : sizeof(PairSmall<float>) + (size_t)kFrags * SetWords<float>::v * 16);
}
size_t dig_tanh_bytes() { return sizeof(dig::TanhTab); }

// The table of tanh_fixed: Taylor coefficients at k / 64 in the working precision of long double, the
// degree-7 term economised over |d| <= 2^-7 (d^7 ~ h^7 (112 x^5 - 56 x^3 + 7 x) / 64, x = d / h).
// Built once per process (about 3 ms of extended-precision arithmetic).
static std::vector<dig::TanhTab> make_tanh_table() {
  std::vector<dig::TanhTab> buf(1);
  dig::TanhTab& tb = buf[0];
  // derivatives of tanh are (1 - t^2) q_n(t): q_1 = 1, q_{n+1} = d/dt [(1 - t^2) q_n]
  std::vector<std::vector<long double>> q(8);
  q[1] = {1.0L};
  for (int n = 2; n < 8; ++n) {
    std::vector<long double> p(q[n - 1].size() + 2, 0.0L);
    for (size_t k = 0; k < q[n - 1].size(); ++k) { p[k] += q[n - 1][k]; p[k + 2] -= q[n - 1][k]; }
    q[n].assign(p.size() - 1, 0.0L);
    for (size_t k = 1; k < p.size(); ++k) q[n][k - 1] = p[k] * (long double)k;
  }
  const long double h = 1.0L / 128.0L;
  for (int k = 0; k < dig::kTanhN; ++k) {
    const long double x = (long double)k / 64.0L, e = std::exp(-2.0L * x);
    const long double t = std::tanh(x), c1 = 4.0L * e / ((1.0L + e) * (1.0L + e));
    long double c[8] = {t, c1}, fact = 1.0L;
    for (int n = 2; n < 8; ++n) {
      fact *= n;
      long double s = 0.0L;
      for (size_t j = q[n].size(); j-- > 0;) s = s * t + q[n][j];
      c[n] = c1 * s / fact;
    }
    c[5] += c[7] * h * h * 112.0L / 64.0L;
    c[3] -= c[7] * h * h * h * h * 56.0L / 64.0L;
    c[1] += c[7] * h * h * h * h * h * h * 7.0L / 64.0L;
    const long double two62 = 4611686018427387904.0L;
    tb.a[k].x = std::llrint(c[0] * two62);
    tb.a[k].y = std::llrint(c[1] * two62);
    const long long c2 = std::llrint(c[2] * two62);
    tb.b[k].x = (int)(c2 & 0xffffffffll);
    tb.b[k].y = (int)(c2 >> 32);
    tb.b[k].z = (int)std::llrint(c[3] * 4294967296.0L);
    const float c4 = (float)c[4];
    std::memcpy(&tb.b[k].w, &c4, 4);
    tb.c[k] = make_float2((float)c[5], (float)c[6]);
  }
  return buf;
}
dp_status dig_upload_tanh(Model* m) {
  static const std::vector<dig::TanhTab> tab = make_tanh_table();
  DP_CUDA_TRY(m, cudaMemcpy(m->dig_tanh, tab.data(), sizeof(dig::TanhTab), cudaMemcpyHostToDevice));
  return DP_OK;
}

dp_status dig_upload(Model* m) { return m->prec == DP_FP64 ? upload<double>(m) : upload<float>(m); }
dp_status launch_dig_descriptor(Model* m, int N) {
  return m->prec == DP_FP64 ? forward<double>(m, N) : forward<float>(m, N);
}
dp_status launch_dig_embed_backward(Model* m, int N) {
  return m->prec == DP_FP64 ? backward<double>(m, N) : backward<float>(m, N);
}

}  // namespace dpg
