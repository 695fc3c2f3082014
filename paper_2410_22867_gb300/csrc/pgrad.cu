// Parameter gradient of the training loss
//   L = cE (E - E0)^2 + cF sum_k |F_k - F0_k|^2
// with respect to every network parameter theta (embedding nets, fitting nets,
// e_bias) of the model of Section II-A / Fig. 1, in FP64 or FP32.
//
// With alpha = 2 cE (E - E0) and w = 2 cF (F - F0) held fixed, and F = -dE/dx,
//   dL/dtheta = alpha dE/dtheta - d/dtheta [ sum_k w_k . dE/dx_k ],
// i.e. the gradient of Psi = alpha E - D_w E, where D_w E is the directional
// derivative of E along the displacement field w.  D_w E is computed by carrying
// a tangent (derivative along w) beside every value of the forward pass:
// pair vectors get d' = w_j - w_i, and the tangent runs through the environment
// row, the embedding net, T, the descriptor and the fitting net to E_i'.  A
// reverse sweep over that (value, tangent) computation then gives dPsi/dtheta.
//
// Work runs per chunk of centre atoms of one type (at most pg_cap atoms):
//   1. embedding forward with tangents -> T, T' per atom, layer by layer over row chunks;
//   2. descriptor D, D' per atom, stacked as the 2n rows [D; D'];
//   3. fitting net forward on the stacked rows (GEMMs), activations kept;
//   4. fitting reverse: adjoint rows [u_bar; v_bar] per layer, weight gradients as
//      GEMMs over the atoms, and [D_bar; D'_bar];
//   5. descriptor reverse -> T_bar, T'_bar per atom;
//   6. embedding reverse over the same row chunks (activations recomputed).
// The embedding layers run as tall, skinny GEMMs over neighbour rows (at most kPgRows at a time): a
// value and its tangent are consecutive rows 2 r and 2 r + 1, and one thread holds both for the two
// units that share a residual, so activations, residuals and the adjoint formulas are epilogues in
// registers.  One thread per row with its 225 activations in local memory took 17 ms of a
// 3,072-atom FP32 gradient; these take 3.1 ms.
// Weight gradients are accumulated with FP64 atomics.
#include "common.cuh"

namespace dpg {
namespace {

template <class T> __device__ __forceinline__ T tanh_t(T x);
template <> __device__ __forceinline__ float tanh_t<float>(float x) { return tanhf(x); }
template <> __device__ __forceinline__ double tanh_t<double>(double x) { return tanh(x); }

template <class T>
__device__ __forceinline__ void switch_t(T r, T rs, T rc, int kind, T& sw, T& dsw) {
  if (r < rs) { sw = T(1); dsw = T(0); return; }
  if (r >= rc) { sw = T(0); dsw = T(0); return; }
  const T wd = rc - rs;
  const T u = (r - rs) / wd;
  if (kind == 1) {
    const T pi = T(3.14159265358979323846);
    sw = T(0.5) * cos(pi * u) + T(0.5);
    dsw = T(-0.5) * pi * sin(pi * u) / wd;
  } else {
    const T u2 = u * u;
    sw = u2 * u * (T(-6) * u2 + T(15) * u - T(10)) + T(1);
    dsw = T(-30) * u2 * (u - T(1)) * (u - T(1)) / wd;
  }
}

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

template <class T>
struct PgArgs {
  int N, ntypes, S;
  int sel_off[kMaxTypes + 1];
  T rc, rs, invS;
  int switch_kind;
  const T* w;            // theta
  const T* stat;         // davg [nt][4], 1/dstd [nt][4]
  const int* nl_j;
  const void* nl_d;
  const int* nl_count;   // [N][nt]
  const double* wdir;    // [N][3] tangent direction w (internal order)
  const T* pad;          // [nt][nt][4][100] padded-slot term of T, or null (every davg is 0)
  int sel[kMaxTypes];
};

// Environment row R_hat and its tangent along d' (Jacobian of (s, s d/r), s = sw/r).
template <class T>
__device__ __forceinline__ void env_tangent(const PgArgs<T>& a, int ti, const T* d, const T* dd, T* R, T* Rd) {
  const T r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  T sw, dsw;
  switch_t<T>(r, a.rs, a.rc, a.switch_kind, sw, dsw);
  const T rinv = T(1) / r;
  const T s = sw * rinv;
  const T q = sw * rinv * rinv;
  const T rdot = (d[0] * dd[0] + d[1] * dd[1] + d[2] * dd[2]) * rinv;  // dr along d'
  const T sdot = (dsw * rinv - sw * rinv * rinv) * rdot;
  const T qdot = (dsw * rinv * rinv - T(2) * sw * rinv * rinv * rinv) * rdot;
  R[0] = s;
  Rd[0] = sdot;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    R[1 + c] = q * d[c];
    Rd[1 + c] = qdot * d[c] + q * dd[c];
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const T isd = a.stat[(a.ntypes + ti) * 4 + c];
    R[c] = (R[c] - a.stat[ti * 4 + c]) * isd;
    Rd[c] *= isd;
  }
}

template <class T>
__device__ __forceinline__ void row_geometry(const PgArgs<T>& a, int i, int ti, size_t e, T* R, T* Rd) {
  T d[3], dd[3];
  pair_vec<T>(a.nl_d, e, d);
  const int j = a.nl_j[e];
#pragma unroll
  for (int c = 0; c < 3; ++c) dd[c] = (T)(a.wdir[3 * (size_t)j + c] - a.wdir[3 * (size_t)i + c]);
  env_tangent<T>(a, ti, d, dd, R, Rd);
}

// Rows of a chunk: the neighbours of type tj of atoms [b0, b0 + nb), numbered by roff (exclusive offsets).
struct RowMap {
  int ti, tj, b0, nb, R;
  const int* roff;
};

// 1a / 6a. Environment row and tangent, and layer 1 with tangents, of every row of a chunk:
// geo [R][8] = (R_hat, R_hat'), atom [R] = local atom, H1 rows 2 r = h1, 2 r + 1 = h1'.
constexpr int kPgGeo = 8;
template <class T>
__global__ void __launch_bounds__(128) k_pg_rows(PgArgs<T> a, RowMap m, T* __restrict__ geo, int* __restrict__ atom,
                                                T* __restrict__ H1) {
  __shared__ T sx[128][2];
  const int r0 = blockIdx.x * 128, r = r0 + threadIdx.x;
  const T* W = a.w + (size_t)(m.ti * a.ntypes + m.tj) * kEmbParams;
  if (r < m.R) {
    int lo = 0, hi = m.nb - 1;  // last atom k with roff[k] <= r
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (m.roff[mid] <= r) lo = mid; else hi = mid - 1;
    }
    T R[4], Rd[4];
    row_geometry<T>(a, m.b0 + lo, m.ti, (size_t)(m.b0 + lo) * a.S + a.sel_off[m.tj] + (r - m.roff[lo]), R, Rd);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      geo[(size_t)r * kPgGeo + c] = R[c];
      geo[(size_t)r * kPgGeo + 4 + c] = Rd[c];
    }
    atom[r] = lo;
    sx[threadIdx.x][0] = R[0];
    sx[threadIdx.x][1] = Rd[0];
  }
  __syncthreads();
  const int rows = min(128, m.R - r0);
  for (int q = threadIdx.x; q < rows * kN1; q += 128) {
    const int rr = q / kN1, k = q - rr * kN1;
    const T w = W[kEW1 + k];
    const T h = tanh_t<T>(sx[rr][0] * w + W[kEb1 + k]);
    T* o = H1 + (size_t)(r0 + rr) * 2 * kN1 + k;
    o[0] = h;
    o[kN1] = (T(1) - h * h) * (sx[rr][1] * w);
  }
}

// Tall, skinny product of 2 R rows: C = A [2 R x K] W [K x N] (or W^T with TB: W is [N x K]), all of W and
// 128 (N = 100) or 256 (N = 50, 25) rows in shared memory (FP64: half as many).  320 threads (160): TC
// column groups of CN columns tc + TC j (so the columns m and m + N / 2 of a residual pair belong to one
// thread), row groups of 4 rows (two value / tangent pairs).  Per k a thread loads 4 + CN values for
// 4 CN multiply-adds.
template <class T, int N> struct Skinny {
  static constexpr int THREADS = sizeof(T) == 8 ? 160 : 320;
  static constexpr int TC = N == 100 ? 10 : 5, CN = N / TC, TR = THREADS / TC, ROWS = 4 * TR;
  static constexpr int CP = (CN + 3) / 4 * 4;  // columns of a thread, padded for 16-byte loads
};
template <class T, int K, int N> constexpr size_t skinny_smem() {
  return sizeof(T) * ((size_t)K * Skinny<T, N>::TC * Skinny<T, N>::CP + (size_t)K * (Skinny<T, N>::ROWS + 4));
}
template <class T, int K, int N, bool TB, class Epi>
__global__ void __launch_bounds__(Skinny<T, N>::THREADS) k_pg_layer(int R2, const T* __restrict__ A, const T* __restrict__ W, Epi epi) {
  using S = Skinny<T, N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sW = reinterpret_cast<T*>(smem_raw);         // [K][TC][CP]
  T* sA = sW + (size_t)K * S::TC * S::CP;         // [K][ROWS + 4]
  const int tid = threadIdx.x;
  const int row0 = blockIdx.x * S::ROWS;
  for (int q = tid; q < K * N; q += S::THREADS) {
    const int k = TB ? q % K : q / N, n = TB ? q / K : q % N;
    sW[((size_t)k * S::TC + n % S::TC) * S::CP + n / S::TC] = W[q];
  }
  for (int q = tid; q < S::ROWS * K; q += S::THREADS) {
    const int r = q / K, k = q - r * K;
    sA[(size_t)k * (S::ROWS + 4) + r] = row0 + r < R2 ? A[(size_t)row0 * K + q] : T(0);
  }
  __syncthreads();
  const int tc = tid % S::TC, tr = tid / S::TC;
  T acc[4][S::CN];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < S::CN; ++c) acc[r][c] = T(0);
#pragma unroll 5
  for (int k = 0; k < K; ++k) {
    T av[4], wv[S::CN];
#pragma unroll
    for (int r = 0; r < 4; ++r) av[r] = sA[(size_t)k * (S::ROWS + 4) + 4 * tr + r];
#pragma unroll
    for (int c = 0; c < S::CN; ++c) wv[c] = sW[((size_t)k * S::TC + tc) * S::CP + c];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < S::CN; ++c) acc[r][c] += av[r] * wv[c];
  }
  epi.template run<S::TC, S::CN>(row0 + 4 * tr, R2, tc, acc, reinterpret_cast<T*>(smem_raw));
}

// h2 = [h1, h1] + tanh(z2 + b2), h2' = [h1', h1'] + (1 - t2^2) z2'; keeps (t2, z2').
template <class T>
struct EpiL2 {
  const T* b;
  const T* H1;
  T* H2;
  T* TZ;
  template <int TC, int CN>
  __device__ __forceinline__ void run(int row, int R2, int tc, T (*acc)[CN], T*) const {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const size_t r = (size_t)row + 2 * p;
      if (r >= (size_t)R2) return;
#pragma unroll
      for (int c = 0; c < CN; ++c) {
        const int n = tc + TC * c, k = n % kN1;
        const T t = tanh_t<T>(acc[2 * p][c] + b[n]), zd = acc[2 * p + 1][c];
        H2[r * kN2 + n] = H1[r * kN1 + k] + t;
        H2[(r + 1) * kN2 + n] = H1[(r + 1) * kN1 + k] + (T(1) - t * t) * zd;
        if (TZ) {
          TZ[r * kN2 + n] = t;
          TZ[(r + 1) * kN2 + n] = zd;
        }
      }
    }
  }
};
// G = [h2, h2] + tanh(z3 + b3) and G' likewise.
template <class T>
struct EpiL3 {
  const T* b;
  const T* H2;
  T* G;
  template <int TC, int CN>
  __device__ __forceinline__ void run(int row, int R2, int tc, T (*acc)[CN], T*) const {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const size_t r = (size_t)row + 2 * p;
      if (r >= (size_t)R2) return;
#pragma unroll
      for (int c = 0; c < CN; ++c) {
        const int n = tc + TC * c, k = n % kN2;
        const T t = tanh_t<T>(acc[2 * p][c] + b[n]);
        G[r * kN3 + n] = H2[r * kN2 + k] + t;
        G[(r + 1) * kN3 + n] = H2[(r + 1) * kN2 + k] + (T(1) - t * t) * acc[2 * p + 1][c];
      }
    }
  }
};
// Adjoints of z3, z3' (into Y3) and the residual adjoints of h2, h2' (gb[m] + gb[m + 50], into HB).
template <class T>
struct EpiR3 {
  const T* b;
  const T* geo;
  const int* atom;
  const T* TB;  // [local atom][800]
  T invS;
  T* Y3;
  T* HB;
  template <int TC, int CN>
  __device__ __forceinline__ void run(int row, int R2, int tc, T (*acc)[CN], T*) const {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const size_t r = (size_t)row + 2 * p;
      if (r >= (size_t)R2) return;
      T g[kPgGeo];
#pragma unroll
      for (int c = 0; c < kPgGeo; ++c) g[c] = geo[(r / 2) * kPgGeo + c];
      const T* Tb = TB + (size_t)atom[r / 2] * 800;
#pragma unroll
      for (int c = 0; c < CN / 2; ++c) {
        T sb = T(0), sd = T(0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c + h * (CN / 2), n = tc + TC * cc;
          const T t = tanh_t<T>(acc[2 * p][cc] + b[n]), zd = acc[2 * p + 1][cc];
          T gb = T(0), gd = T(0);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const T u = Tb[x * kN3 + n], ud = Tb[400 + x * kN3 + n];
            gb += g[x] * u + g[4 + x] * ud;
            gd += g[x] * ud;
          }
          gb *= invS;
          gd *= invS;
          const T q = T(1) - t * t;
          Y3[r * kN3 + n] = (gb - T(2) * t * (gd * zd)) * q;
          Y3[(r + 1) * kN3 + n] = gd * q;
          sb += gb;
          sd += gd;
        }
        const int m = tc + TC * c;
        HB[r * kN2 + m] = sb;
        HB[(r + 1) * kN2 + m] = sd;
      }
    }
  }
};
// dE/dh2 = residual + Y3 W3^T; adjoints of z2, z2' (Y2) and the residual adjoints of h1, h1' (HB1).
template <class T>
struct EpiR2 {
  const T* HB;
  const T* TZ;
  T* Y2;
  T* HB1;
  template <int TC, int CN>
  __device__ __forceinline__ void run(int row, int R2, int tc, T (*acc)[CN], T*) const {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const size_t r = (size_t)row + 2 * p;
      if (r >= (size_t)R2) return;
#pragma unroll
      for (int c = 0; c < CN / 2; ++c) {
        T sb = T(0), sd = T(0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c + h * (CN / 2), n = tc + TC * cc;
          const T hb = HB[r * kN2 + n] + acc[2 * p][cc], hd = HB[(r + 1) * kN2 + n] + acc[2 * p + 1][cc];
          const T t = TZ[r * kN2 + n], zd = TZ[(r + 1) * kN2 + n];
          const T q = T(1) - t * t;
          Y2[r * kN2 + n] = (hb - T(2) * t * (hd * zd)) * q;
          Y2[(r + 1) * kN2 + n] = hd * q;
          sb += hb;
          sd += hd;
        }
        const int k = tc + TC * c;
        HB1[r * kN1 + k] = sb;
        HB1[(r + 1) * kN1 + k] = sd;
      }
    }
  }
};
// dE/dh1 = residual + Y2 W2^T, then the gradients of W1 and b1: sums over rows of x z1_bar + x' v1_bar and
// z1_bar, added up in shared memory (FP64) and with one atomic per column and block.
template <class T>
struct EpiR1 {
  const T* HB1;
  const T* H1;
  const T* geo;
  const T* w1;
  double* gw1;  // W1 then b1
  template <int TC, int CN>
  __device__ __forceinline__ void run(int row, int R2, int tc, T (*acc)[CN], T* smem) const {
    T sw[CN], sb[CN];
#pragma unroll
    for (int c = 0; c < CN; ++c) sw[c] = sb[c] = T(0);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const size_t r = (size_t)row + 2 * p;
      if (r < (size_t)R2) {
        const T x = geo[(r / 2) * kPgGeo], xd = geo[(r / 2) * kPgGeo + 4];
#pragma unroll
        for (int c = 0; c < CN; ++c) {
          const int k = tc + TC * c;
          const T hb = HB1[r * kN1 + k] + acc[2 * p][c], hd = HB1[(r + 1) * kN1 + k] + acc[2 * p + 1][c];
          const T h = H1[r * kN1 + k], q = T(1) - h * h;
          const T zb = (hb - T(2) * h * (hd * (xd * w1[k]))) * q, vb = hd * q;
          sw[c] += x * zb + xd * vb;
          sb[c] += zb;
        }
      }
    }
    __syncthreads();  // every thread is done with the operands
    T* s = smem;      // [row groups][2 kN1]
    const int tr = threadIdx.x / TC;
#pragma unroll
    for (int c = 0; c < CN; ++c) {
      s[tr * 2 * kN1 + tc + TC * c] = sw[c];
      s[tr * 2 * kN1 + kN1 + tc + TC * c] = sb[c];
    }
    __syncthreads();
    if (threadIdx.x < 2 * kN1) {
      double v = 0.0;
      for (int q = 0; q < (int)blockDim.x / TC; ++q) v += (double)s[q * 2 * kN1 + threadIdx.x];
      atomicAdd(gw1 + threadIdx.x, v);
    }
  }
};

// T += R_hat^T G and T' += R_hat'^T G + R_hat^T G' over the rows of each atom of the chunk (CTA per atom;
// sums over S added later): rows [roff[k], roff[k + 1]) of G.
template <class T>
__global__ void __launch_bounds__(128) k_pg_T(RowMap m, int a0, const T* __restrict__ geo, const T* __restrict__ G,
                                             T* TT) {
  __shared__ T sg[32][kPgGeo];
  const int k = blockIdx.x, q = threadIdx.x;
  const int rb = m.roff[k], re = m.roff[k + 1];
  T acc[4], accd[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = accd[c] = T(0);
  for (int r0 = rb; r0 < re; r0 += 32) {
    __syncthreads();
    for (int e = q; e < 32 * kPgGeo; e += 128) {
      const int r = r0 + e / kPgGeo;
      sg[e / kPgGeo][e % kPgGeo] = r < re ? geo[(size_t)r * kPgGeo + e % kPgGeo] : T(0);
    }
    __syncthreads();
    if (q < kN3)
      for (int r = r0; r < min(re, r0 + 32); ++r) {
        const T g = G[(size_t)2 * r * kN3 + q], gd = G[((size_t)2 * r + 1) * kN3 + q];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          acc[c] += sg[r - r0][c] * g;
          accd[c] += sg[r - r0][4 + c] * g + sg[r - r0][c] * gd;
        }
      }
  }
  if (q < kN3) {
    T* o = TT + (size_t)(m.b0 + k - a0) * 800 + q;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      o[c * kN3] += acc[c];
      o[400 + c * kN3] += accd[c];
    }
  }
}

// Padded slots (constant in the positions: T only) and the normaliser 1 / S; block per atom of the chunk.
template <class T>
__global__ void __launch_bounds__(128) k_pg_T_scale(PgArgs<T> a, int ti, int a0, T* TT) {
  const int li = blockIdx.x, i = a0 + li;
  for (int q = threadIdx.x; q < 800; q += 128) {
    T v = TT[(size_t)li * 800 + q];
    if (a.pad && q < 400)
      for (int tj = 0; tj < a.ntypes; ++tj)
        v += T(a.sel[tj] - a.nl_count[(size_t)i * a.ntypes + tj]) * a.pad[(size_t)(ti * a.ntypes + tj) * 4 * kN3 + q];
    TT[(size_t)li * 800 + q] = v * a.invS;
  }
}

// Weight and bias gradients of a layer: gW [KX x N] += X^T Y over the 2 R rows (value and tangent rows
// alike), gb [N] += column sums of the value rows of Y.  A block sums a range of rows in registers
// (thread: two columns of X, N / 10 of Y) and adds its result with FP64 atomics.
template <class T, int KX, int N>
__global__ void __launch_bounds__(320) k_pg_wgrad(int R2, int per, const T* __restrict__ X, const T* __restrict__ Y,
                                                 double* gW, double* gb) {
  constexpr int CN = N / 10, GX = (KX + 1) / 2, B = 32;  // GX groups of two X columns, then one for the bias
  __shared__ T sX[B][KX + 1], sY[B][N];
  const int tid = threadIdx.x, tc = tid % 10, tx = tid / 10;
  const int rb = blockIdx.x * per, re = min(R2, rb + per);
  T acc[2][CN];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < CN; ++c) acc[h][c] = T(0);
  for (int r0 = rb; r0 < re; r0 += B) {
    __syncthreads();
    const int nr = min(B, re - r0);
    for (int q = tid; q < B * KX; q += 320) sX[q / KX][q % KX] = q / KX < nr ? X[(size_t)r0 * KX + q] : T(0);
    for (int q = tid; q < B * N; q += 320) sY[q / N][q % N] = q / N < nr ? Y[(size_t)r0 * N + q] : T(0);
    __syncthreads();
    if (tx < GX) {
#pragma unroll 4
      for (int r = 0; r < B; ++r) {
        const T x0 = sX[r][2 * tx], x1 = 2 * tx + 1 < KX ? sX[r][2 * tx + 1] : T(0);
#pragma unroll
        for (int c = 0; c < CN; ++c) {
          const T y = sY[r][tc + 10 * c];
          acc[0][c] += x0 * y;
          acc[1][c] += x1 * y;
        }
      }
    } else if (tx == GX) {
      for (int r = 0; r < B; r += 2)
#pragma unroll
        for (int c = 0; c < CN; ++c) acc[0][c] += sY[r][tc + 10 * c];
    }
  }
  if (tx < GX) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (2 * tx + h < KX)
#pragma unroll
        for (int c = 0; c < CN; ++c) atomicAdd(gW + (2 * tx + h) * N + tc + 10 * c, (double)acc[h][c]);
  } else if (tx == GX) {
#pragma unroll
    for (int c = 0; c < CN; ++c) atomicAdd(gb + tc + 10 * c, (double)acc[0][c]);
  }
}

// 2. D = T^T T[:, :16] and D' = T'^T T< + T^T T'< as rows li and n + li of Y.
template <class T>
__global__ void k_pg_desc(int n, const T* TT, T* Y) {
  __shared__ T s[800];
  for (int li = blockIdx.x; li < n; li += gridDim.x) {
    __syncthreads();
    for (int q = threadIdx.x; q < 800; q += blockDim.x) s[q] = TT[(size_t)li * 800 + q];
    __syncthreads();
    const T* Tp = s;
    const T* Td = s + 400;
    for (int o = threadIdx.x; o < kKD; o += blockDim.x) {
      const int aa = o / kM2, b = o % kM2;
      T v = T(0), vd = T(0);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        v += Tp[c * kN3 + aa] * Tp[c * kN3 + b];
        vd += Td[c * kN3 + aa] * Tp[c * kN3 + b] + Tp[c * kN3 + aa] * Td[c * kN3 + b];
      }
      Y[(size_t)li * kKD + o] = v;
      Y[(size_t)(n + li) * kKD + o] = vd;
    }
  }
}

// 5. T_bar and T'_bar from D_bar (row li of Yb) and D'_bar (row n + li).
template <class T>
__global__ void k_pg_desc_bwd(int n, const T* TT, const T* Yb, T* TB) {
  __shared__ T s[800 + 2 * kKD];
  for (int li = blockIdx.x; li < n; li += gridDim.x) {
    __syncthreads();
    for (int q = threadIdx.x; q < 800; q += blockDim.x) s[q] = TT[(size_t)li * 800 + q];
    for (int q = threadIdx.x; q < kKD; q += blockDim.x) {
      s[800 + q] = Yb[(size_t)li * kKD + q];
      s[800 + kKD + q] = Yb[(size_t)(n + li) * kKD + q];
    }
    __syncthreads();
    const T* Tp = s;
    const T* Td = s + 400;
    const T* Db = s + 800;
    const T* Ddb = s + 800 + kKD;
    for (int o = threadIdx.x; o < 400; o += blockDim.x) {
      const int c = o / kN3, aa = o % kN3;
      T tb = T(0), tdb = T(0);
#pragma unroll
      for (int b = 0; b < kM2; ++b) {
        tb += Db[aa * kM2 + b] * Tp[c * kN3 + b] + Ddb[aa * kM2 + b] * Td[c * kN3 + b];
        tdb += Ddb[aa * kM2 + b] * Tp[c * kN3 + b];
      }
      if (aa < kM2) {
        for (int a2 = 0; a2 < kN3; ++a2) {
          tb += Db[a2 * kM2 + aa] * Tp[c * kN3 + a2] + Ddb[a2 * kM2 + aa] * Td[c * kN3 + a2];
          tdb += Ddb[a2 * kM2 + aa] * Tp[c * kN3 + a2];
        }
      }
      TB[(size_t)li * 800 + o] = tb;
      TB[(size_t)li * 800 + 400 + o] = tdb;
    }
  }
}

// 5b. Parameter gradient through the padded slots of centre type ti, one block per neighbour
//     type tj.  Every padded slot of segment tj holds the row R_pad = -davg[ti] / dstd[ti] and
//     G = N_{ti,tj}(R_pad_0), so with T_bar the adjoint of T (row li of TB, primal half):
//       G_bar[a] = (1/S) sum_li (sel[tj] - count_li,tj) sum_c T_bar_li[c][a] R_pad[c],
//     and the reverse of the embedding net at the single input R_pad_0 gives the parameter
//     gradients (FP64 atomics).  The input is a constant (davg, dstd are not parameters).
//     k_pg_pad_sum forms the sums over atoms first, 32 atoms a block (one block per tj walking all
//     atoms took 0.27 ms a call): gsum [tj][100], zeroed by the caller.
template <class T>
__global__ void __launch_bounds__(128) k_pg_pad_sum(PgArgs<T> a, int ti, int a0, int n, const T* __restrict__ TB,
                                                   double* gsum) {
  const int tj = blockIdx.x, tid = threadIdx.x;
  if (tid >= kN3) return;
  T Rp[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) Rp[c] = (T(0) - a.stat[ti * 4 + c]) * a.stat[(a.ntypes + ti) * 4 + c];
  T acc = T(0);
  for (int li = blockIdx.y * 32; li < min(n, blockIdx.y * 32 + 32); ++li) {
    const T np = T(a.sel[tj] - a.nl_count[(size_t)(a0 + li) * a.ntypes + tj]);
    const T* tb = TB + (size_t)li * 800;
    acc += np * (tb[tid] * Rp[0] + tb[kN3 + tid] * Rp[1] + tb[2 * kN3 + tid] * Rp[2] + tb[3 * kN3 + tid] * Rp[3]);
  }
  atomicAdd(gsum + tj * kN3 + tid, (double)acc);
}
template <class T>
__global__ void __launch_bounds__(128) k_pg_pad_rev(PgArgs<T> a, int ti, const double* __restrict__ gsum, double* grad) {
  const int tj = blockIdx.x, tid = threadIdx.x;
  const T* W = a.w + (size_t)(ti * a.ntypes + tj) * kEmbParams;
  double* gW = grad + (size_t)(ti * a.ntypes + tj) * kEmbParams;
  __shared__ T Rp[4], h1[kN1], t2[kN2], h2[kN2], gG[kN3], dz3[kN3], dh2[kN2], dz2[kN2];
  if (tid < 4) Rp[tid] = (T(0) - a.stat[ti * 4 + tid]) * a.stat[(a.ntypes + ti) * 4 + tid];
  __syncthreads();
  if (tid < kN3) gG[tid] = (T)gsum[tj * kN3 + tid] * a.invS;
  const T x = Rp[0];
  if (tid < kN1) h1[tid] = tanh_t<T>(x * W[kEW1 + tid] + W[kEb1 + tid]);
  __syncthreads();
  if (tid < kN2) {
    T z = W[kEb2 + tid];
    for (int k = 0; k < kN1; ++k) z += h1[k] * W[kEW2 + k * kN2 + tid];
    t2[tid] = tanh_t<T>(z);
    h2[tid] = h1[tid % kN1] + t2[tid];
  }
  __syncthreads();
  if (tid < kN3) {  // G[a] = h2[a % 50] + tanh(z3[a])
    T z = W[kEb3 + tid];
    for (int mm = 0; mm < kN2; ++mm) z += h2[mm] * W[kEW3 + mm * kN3 + tid];
    const T t3 = tanh_t<T>(z);
    dz3[tid] = gG[tid] * (T(1) - t3 * t3);
    atomicAdd(&gW[kEb3 + tid], (double)dz3[tid]);
  }
  __syncthreads();
  for (int q = tid; q < kN2 * kN3; q += blockDim.x)
    atomicAdd(&gW[kEW3 + q], (double)(h2[q / kN3] * dz3[q % kN3]));
  if (tid < kN2) {
    T v = gG[tid] + gG[tid + kN2];
    for (int aa = 0; aa < kN3; ++aa) v += W[kEW3 + tid * kN3 + aa] * dz3[aa];
    dh2[tid] = v;
    dz2[tid] = v * (T(1) - t2[tid] * t2[tid]);
    atomicAdd(&gW[kEb2 + tid], (double)dz2[tid]);
  }
  __syncthreads();
  for (int q = tid; q < kN1 * kN2; q += blockDim.x)
    atomicAdd(&gW[kEW2 + q], (double)(h1[q / kN2] * dz2[q % kN2]));
  if (tid < kN1) {
    T v = dh2[tid] + dh2[tid + kN1];
    for (int mm = 0; mm < kN2; ++mm) v += W[kEW2 + tid * kN2 + mm] * dz2[mm];
    const T dz1 = v * (T(1) - h1[tid] * h1[tid]);
    atomicAdd(&gW[kEb1 + tid], (double)dz1);
    atomicAdd(&gW[kEW1 + tid], (double)(x * dz1));
  }
}

// Plain tiled GEMM C[M x N] = op(A)[M x K] op(B)[K x N] (row-major storage, op = transpose
// when TA / TB).  OUT 0: store; 1: C += result; 2: atomicAdd into FP64 C, with the K range
// split over gridDim.z.
constexpr int kGM = 64, kGN = 64, kGK = 16;

template <class T, bool TA, bool TB, int OUT>
__global__ void __launch_bounds__(256) k_pg_gemm(int M, int N, int K, const T* __restrict__ A, int lda,
                                               const T* __restrict__ B, int ldb, void* Cv, int ldc) {
  __shared__ T As[kGK][kGM + 1];
  __shared__ T Bs[kGK][kGN + 1];
  const int m0 = blockIdx.y * kGM, n0 = blockIdx.x * kGN;
  const int kchunk = (K + gridDim.z - 1) / gridDim.z;
  const int kbeg = blockIdx.z * kchunk, kend = min(K, kbeg + kchunk);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T acc[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = T(0);
  for (int k0 = kbeg; k0 < kend; k0 += kGK) {
    for (int e = threadIdx.x; e < kGM * kGK; e += 256) {
      const int mm = TA ? e % kGM : e / kGK, kk = TA ? e / kGM : e % kGK;
      const int gm = m0 + mm, gk = k0 + kk;
      T v = T(0);
      if (gm < M && gk < kend) v = TA ? A[(size_t)gk * lda + gm] : A[(size_t)gm * lda + gk];
      As[kk][mm] = v;
    }
    for (int e = threadIdx.x; e < kGK * kGN; e += 256) {
      const int nn = TB ? e / kGK : e % kGN, kk = TB ? e % kGK : e / kGN;
      const int gn = n0 + nn, gk = k0 + kk;
      T v = T(0);
      if (gn < N && gk < kend) v = TB ? B[(size_t)gn * ldb + gk] : B[(size_t)gk * ldb + gn];
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      T av[4], bv[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) av[p] = As[kk][ty * 4 + p];
#pragma unroll
      for (int q = 0; q < 4; ++q) bv[q] = Bs[kk][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] += av[p] * bv[q];
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int gm = m0 + ty * 4 + p;
    if (gm >= M) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gn = n0 + tx + 16 * q;
      if (gn >= N) continue;
      const size_t o = (size_t)gm * ldc + gn;
      if (OUT == 2) {
        atomicAdd(static_cast<double*>(Cv) + o, (double)acc[p][q]);
      } else {
        T* C = static_cast<T*>(Cv);
        C[o] = (OUT == 1 ? C[o] : T(0)) + acc[p][q];
      }
    }
  }
}

// 3. Fitting activations on the stacked rows F = [z; z'] (raw GEMM output, 2n x 240):
//    layer 1: F <- [h1; v1], H <- [h1; h1'];  layer L > 1: F <- [k_L; v_L], and for L = 2
//    H <- H + [k2; (1 - k2^2) v2] (H then holds [h2; h2']).
template <class T>
__global__ void k_pg_fit_act(int n, int layer, const T* __restrict__ bias, T* F, T* H) {
  const size_t total = (size_t)n * kF;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int col = (int)(e % kF);
    const size_t rp = e, rt = e + total;
    const T k = tanh_t<T>(F[rp] + bias[col]);
    F[rp] = k;
    const T v = F[rt];
    if (layer == 1) {
      H[rp] = k;
      H[rt] = (T(1) - k * k) * v;
    } else if (layer == 2) {
      H[rp] += k;
      H[rt] += (T(1) - k * k) * v;
    }
  }
}

// 4a. Head: h3 = h2 + k3, h3' = h2' + (1 - k3^2) v3; gradient of w4 (sum over atoms of
//     alpha h3 - h3'); adjoints of (h3, h3') = (alpha w4, -w4) into G.
template <class T>
__global__ void k_pg_head(int n, const T* __restrict__ H, const T* __restrict__ F3, const T* __restrict__ w4,
                          const double* scal, T* G, double* gw4) {
  const T alpha = (T)scal[0];
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= kF) return;
  const size_t nt = (size_t)n * kF;
  double acc = 0.0;
  const T wv = w4[col];
  for (int r = blockIdx.y; r < n; r += gridDim.y) {
    const size_t e = (size_t)r * kF + col;
    const T k3 = F3[e], v3 = F3[e + nt];
    const T h3 = H[e] + k3;
    const T h3d = H[e + nt] + (T(1) - k3 * k3) * v3;
    acc += (double)(alpha * h3 - h3d);
    G[e] = alpha * wv;
    G[e + nt] = -wv;
  }
  atomicAdd(gw4 + col, acc);
}

// 4b. Layer reverse: from the adjoints (A, A') of (h_L, h_L') held in G and F_L = [k; v]:
//     k_bar = A - 2 k (A' v), u_bar = k_bar (1 - k^2), v_bar = A' (1 - k^2)  -> U = [u_bar; v_bar];
//     bias gradient += sum over atoms of u_bar.  For layer 2 also H <- [h1; h1'] from F1.
template <class T>
__global__ void k_pg_fit_rev(int n, int layer, const T* __restrict__ G, const T* __restrict__ FL,
                             const T* __restrict__ F1, T* U, T* H, double* gbias) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= kF) return;
  const size_t nt = (size_t)n * kF;
  double acc = 0.0;
  for (int r = blockIdx.y; r < n; r += gridDim.y) {
    const size_t e = (size_t)r * kF + col;
    const T k = FL[e], v = FL[e + nt];
    const T q = T(1) - k * k;
    const T Ap = G[e], At = G[e + nt];
    const T kb = Ap - T(2) * k * (At * v);
    const T ub = kb * q;
    U[e] = ub;
    U[e + nt] = At * q;
    acc += (double)ub;
    if (layer == 2) {
      const T h1 = F1[e];
      H[e] = h1;
      H[e + nt] = (T(1) - h1 * h1) * F1[e + nt];
    }
  }
  atomicAdd(gbias + col, acc);
}

// alpha * (number of atoms) into b4 and e_bias of the type.
__global__ void k_pg_counts(int n, const double* scal, double* gb4, double* gebias) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    atomicAdd(gb4, scal[0] * n);
    atomicAdd(gebias, scal[0] * n);
  }
}

// alpha, loss, and the tangent direction w = 2 cF (F - F0) in internal order.
__global__ void k_pg_setup(int N, const double* __restrict__ e_atom, const double* __restrict__ force,
                           const double* __restrict__ F0, const int* __restrict__ perm, double E0, double cE,
                           double cF, double* wdir, double* scal) {
  __shared__ double sE[32], sL[32];
  double e = 0.0, l = 0.0;
  for (int k = threadIdx.x; k < N; k += blockDim.x) {
    e += e_atom[k];
    const int u = perm[k];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double df = force[3 * (size_t)k + c] - F0[3 * (size_t)u + c];
      l += df * df;
      wdir[3 * (size_t)k + c] = 2.0 * cF * df;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, o);
    l += __shfl_xor_sync(0xffffffffu, l, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { sE[wid] = e; sL[wid] = l; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double E = 0.0, L = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { E += sE[q]; L += sL[q]; }
    scal[0] = 2.0 * cE * (E - E0);
    scal[1] = cE * (E - E0) * (E - E0) + cF * L;
    scal[2] = E;
  }
}

template <class T, bool TA, bool TB, int OUT>
void gemm(Model* m, int M, int N, int K, const T* A, int lda, const T* B, int ldb, void* C, int ldc, int splitk = 1) {
  if (M <= 0 || N <= 0 || K <= 0) return;
  dim3 grid(cdiv(N, kGN), cdiv(M, kGM), std::max(1, std::min(splitk, cdiv(K, kGK))));
  k_pg_gemm<T, TA, TB, OUT><<<grid, 256, 0, m->stream>>>(M, N, K, A, lda, B, ldb, C, ldc);
  m->launches += 1;
}

template <class T>
dp_status run_param_grad(Model* m, int N, double* grad) {
  const int nt = m->ntypes;
  PgArgs<T> a{};
  a.N = N; a.ntypes = nt; a.S = m->S;
  for (int t = 0; t <= nt; ++t) a.sel_off[t] = m->sel_off[t];
  a.rc = (T)m->rc; a.rs = (T)m->rs; a.invS = T(1) / (T)m->S; a.switch_kind = m->switch_kind;
  const T* theta = (sizeof(T) == 8) ? reinterpret_cast<const T*>(m->w64) : reinterpret_cast<const T*>(m->w32);
  a.w = theta;
  a.stat = (sizeof(T) == 8) ? reinterpret_cast<const T*>(m->stat64) : reinterpret_cast<const T*>(m->stat32);
  a.nl_j = m->nl_j; a.nl_d = m->nl_d; a.nl_count = m->nl_count; a.wdir = m->pg_w;
  a.pad = !m->has_pad ? nullptr
                      : (sizeof(T) == 8) ? reinterpret_cast<const T*>(m->pad64) : reinterpret_cast<const T*>(m->pad32);
  for (int t = 0; t < nt; ++t) a.sel[t] = m->sel[t];

  // host copies of the type ranges and per-atom neighbour counts (chunking)
  std::vector<int> cnt((size_t)N * nt), tc(kMaxTypes + 1);
  DP_CUDA_TRY(m, cudaMemcpyAsync(cnt.data(), m->nl_count, sizeof(int) * cnt.size(), cudaMemcpyDeviceToHost,
                                 m->stream));
  DP_CUDA_TRY(m, cudaMemcpyAsync(tc.data(), m->type_count, sizeof(int) * (kMaxTypes + 1), cudaMemcpyDeviceToHost,
                                 m->stream));
  DP_CUDA_TRY(m, cudaStreamSynchronize(m->stream));

  // row offsets of every (centre chunk, neighbour type, row chunk), uploaded once
  struct RowChunk { int ti, tj, a0, b0, nb, R; size_t off; };
  struct AtomChunk { int ti, a0, n; };
  std::vector<AtomChunk> achunks;
  std::vector<RowChunk> rchunks;
  std::vector<int> roffs;
  const int cap = m->pg_cap;
  for (int t = 0; t < nt; ++t)
    if (m->sel[t] > kPgSel) {
      m->last_error = "param_grad: sel larger than 16384";
      return DP_ERR_UNSUPPORTED;
    }
  int start = 0;
  for (int ti = 0; ti < nt; ++ti) {
    const int cnt_t = tc[ti];
    for (int c0 = 0; c0 < cnt_t; c0 += cap) {
      AtomChunk ac{ti, start + c0, std::min(cap, cnt_t - c0)};
      achunks.push_back(ac);
      for (int tj = 0; tj < nt; ++tj) {
        int b = ac.a0;
        const int bend = ac.a0 + ac.n;
        while (b < bend) {
          RowChunk rc{ti, tj, ac.a0, b, 0, 0, roffs.size()};
          int rows = 0;
          roffs.push_back(0);
          while (b < bend && rows + cnt[(size_t)b * nt + tj] <= m->pg_rows) {
            rows += cnt[(size_t)b * nt + tj];
            roffs.push_back(rows);
            ++b;
          }
          rc.nb = b - rc.b0;
          rc.R = rows;
          rchunks.push_back(rc);
        }
      }
    }
    start += cnt_t;
  }
  if (roffs.size() > m->pg_roff_cap) {
    m->last_error = "param_grad: row-offset table larger than allocated";
    return DP_ERR_CAPACITY;
  }
  if (!roffs.empty())
    DP_CUDA_TRY(m, cudaMemcpyAsync(m->pg_roff, roffs.data(), sizeof(int) * roffs.size(), cudaMemcpyHostToDevice,
                                   m->stream));

  // workspace: T and its adjoint, then one area that the fitting net (steps 2 to 5) and the neighbour rows
  // (steps 1 and 6) use in turn
  T* ws = static_cast<T*>(m->pg_ws);
  const size_t C = (size_t)cap;
  T* TT = ws;
  T* TB = TT + C * 800;
  T* Y = TB + C * 800;
  T* Yb = Y + 2 * C * kKD;
  T* F1 = Yb + 2 * C * kKD;
  T* F2 = F1 + 2 * C * kF;
  T* F3 = F2 + 2 * C * kF;
  T* H = F3 + 2 * C * kF;
  T* U = H + 2 * C * kF;
  T* G = U + 2 * C * kF;
  const size_t RW = (size_t)m->pg_rows;
  T* geo = Y;
  T* H1 = geo + RW * kPgGeo;
  T* H2 = H1 + 2 * RW * kN1;
  T* TZ = H2 + 2 * RW * kN2;
  T* Y3 = TZ + 2 * RW * kN2;   // G, G' of the forward; adjoints of z3, z3' of the reverse
  T* HB = Y3 + 2 * RW * kN3;
  T* Y2 = HB + 2 * RW * kN2;
  T* HB1 = Y2 + 2 * RW * kN2;
  int* atom = reinterpret_cast<int*>(HB1 + 2 * RW * kN1);

  const size_t emb_total = (size_t)nt * nt * kEmbParams;
  // one layer over the rows of a chunk
#define PG_LAYER(K_, N_, TB_, EPI_, A_, W_)                                                                  \
  do {                                                                                                       \
    auto fn_ = k_pg_layer<T, K_, N_, TB_, EPI_<T>>;                                                          \
    const size_t sm_ = skinny_smem<T, K_, N_>();                                                             \
    DP_CUDA_TRY(m, ensure_smem(reinterpret_cast<const void*>(fn_), sm_));                                    \
    fn_<<<cdiv(2 * rc.R, Skinny<T, N_>::ROWS), Skinny<T, N_>::THREADS, sm_, m->stream>>>(2 * rc.R, A_, W_, epi);                   \
    m->launches += 1;                                                                                        \
  } while (0)
  const int sms = num_sms();

  for (const AtomChunk& ac : achunks) {
    const int n = ac.n, ti = ac.ti;
    const size_t fb = emb_total + (size_t)ti * kFitParams;  // fitting block of ti
    const T* P = theta + fb;
    double* gP = grad + fb;
    // 1-2: T, T', D, D'
    DP_CUDA_TRY(m, cudaMemsetAsync(TT, 0, sizeof(T) * 800 * (size_t)n, m->stream));
    for (const RowChunk& rc : rchunks) {
      if (rc.ti != ti || rc.a0 != ac.a0 || rc.R == 0) continue;
      const T* W = theta + (size_t)(ti * nt + rc.tj) * kEmbParams;
      const RowMap rm{ti, rc.tj, rc.b0, rc.nb, rc.R, m->pg_roff + rc.off};
      k_pg_rows<T><<<cdiv(rc.R, 128), 128, 0, m->stream>>>(a, rm, geo, atom, H1);
      { EpiL2<T> epi{W + kEb2, H1, H2, nullptr}; PG_LAYER(kN1, kN2, false, EpiL2, H1, W + kEW2); }
      { EpiL3<T> epi{W + kEb3, H2, Y3}; PG_LAYER(kN2, kN3, false, EpiL3, H2, W + kEW3); }
      k_pg_T<T><<<rc.nb, 128, 0, m->stream>>>(rm, ac.a0, geo, Y3, TT);
      m->launches += 2;
    }
    k_pg_T_scale<T><<<n, 128, 0, m->stream>>>(a, ti, ac.a0, TT);
    k_pg_desc<T><<<std::min(n, 8 * sms), 128, 0, m->stream>>>(n, TT, Y);
    m->launches += 2;
    // 3: fitting forward on [D; D']
    const int M2 = 2 * n;
    const int eg = std::min(cdiv((long)n * kF, 256), 8 * sms);
    gemm<T, false, false, 0>(m, M2, kF, kKD, Y, kKD, P + kFW1, kF, F1, kF);
    k_pg_fit_act<T><<<eg, 256, 0, m->stream>>>(n, 1, P + kFb1, F1, H);
    gemm<T, false, false, 0>(m, M2, kF, kF, H, kF, P + kFW2, kF, F2, kF);
    k_pg_fit_act<T><<<eg, 256, 0, m->stream>>>(n, 2, P + kFb2, F2, H);
    gemm<T, false, false, 0>(m, M2, kF, kF, H, kF, P + kFW3, kF, F3, kF);
    k_pg_fit_act<T><<<eg, 256, 0, m->stream>>>(n, 3, P + kFb3, F3, H);
    m->launches += 3;
    // 4: fitting reverse
    const dim3 cg(cdiv(kF, 128), std::min(n, 64));
    k_pg_head<T><<<cg, 128, 0, m->stream>>>(n, H, F3, P + kFw4, m->pg_scal, G, gP + kFw4);
    k_pg_counts<<<1, 32, 0, m->stream>>>(n, m->pg_scal, gP + kFb4, grad + emb_total + (size_t)nt * kFitParams + ti);
    k_pg_fit_rev<T><<<cg, 128, 0, m->stream>>>(n, 3, G, F3, F1, U, H, gP + kFb3);
    m->launches += 3;
    const int sk = std::max(1, std::min(64, M2 / 256));
    gemm<T, true, false, 2>(m, kF, kF, M2, H, kF, U, kF, gP + kFW3, kF, sk);   // W3 grad: [h2; h2']^T U
    gemm<T, false, true, 1>(m, M2, kF, kF, U, kF, P + kFW3, kF, G, kF);        // G += U W3^T
    k_pg_fit_rev<T><<<cg, 128, 0, m->stream>>>(n, 2, G, F2, F1, U, H, gP + kFb2);
    m->launches += 1;
    gemm<T, true, false, 2>(m, kF, kF, M2, H, kF, U, kF, gP + kFW2, kF, sk);   // W2 grad: [h1; h1']^T U
    gemm<T, false, true, 1>(m, M2, kF, kF, U, kF, P + kFW2, kF, G, kF);        // G += U W2^T
    k_pg_fit_rev<T><<<cg, 128, 0, m->stream>>>(n, 1, G, F1, F1, U, H, gP + kFb1);
    m->launches += 1;
    gemm<T, true, false, 2>(m, kKD, kF, M2, Y, kKD, U, kF, gP + kFW1, kF, sk);  // W1 grad: [D; D']^T U
    gemm<T, false, true, 0>(m, M2, kKD, kF, U, kF, P + kFW1, kF, Yb, kKD);      // [D_bar; D'_bar] = U W1^T
    // 5: T_bar, T'_bar
    k_pg_desc_bwd<T><<<std::min(n, 8 * sms), 128, 0, m->stream>>>(n, TT, Yb, TB);
    m->launches += 1;
    if (a.pad) {
      double* gsum = m->pg_scal + 8;
      DP_CUDA_TRY(m, cudaMemsetAsync(gsum, 0, sizeof(double) * kN3 * nt, m->stream));
      k_pg_pad_sum<T><<<dim3(nt, cdiv(n, 32)), 128, 0, m->stream>>>(a, ti, ac.a0, n, TB, gsum);
      k_pg_pad_rev<T><<<nt, 128, 0, m->stream>>>(a, ti, gsum, grad);
      m->launches += 2;
    }
    // 6: embedding reverse over the rows
    for (const RowChunk& rc : rchunks) {
      if (rc.ti != ti || rc.a0 != ac.a0 || rc.R == 0) continue;
      const size_t eb = (size_t)(ti * nt + rc.tj) * kEmbParams;
      const T* W = theta + eb;
      double* gW = grad + eb;
      const RowMap rm{ti, rc.tj, rc.b0, rc.nb, rc.R, m->pg_roff + rc.off};
      k_pg_rows<T><<<cdiv(rc.R, 128), 128, 0, m->stream>>>(a, rm, geo, atom, H1);
      { EpiL2<T> epi{W + kEb2, H1, H2, TZ}; PG_LAYER(kN1, kN2, false, EpiL2, H1, W + kEW2); }
      {
        EpiR3<T> epi{W + kEb3, geo, atom, TB + (size_t)(rc.b0 - ac.a0) * 800, a.invS, Y3, HB};
        PG_LAYER(kN2, kN3, false, EpiR3, H2, W + kEW3);
      }
      { EpiR2<T> epi{HB, TZ, Y2, HB1}; PG_LAYER(kN3, kN2, true, EpiR2, Y3, W + kEW3); }
      { EpiR1<T> epi{HB1, H1, geo, W + kEW1, gW + kEW1}; PG_LAYER(kN2, kN1, true, EpiR1, Y2, W + kEW2); }
      // about two blocks an SM, at least 128 rows each
      const int per = std::max(128, cdiv(cdiv(2 * rc.R, 2 * sms), 32) * 32);
      k_pg_wgrad<T, kN2, kN3><<<cdiv(2 * rc.R, per), 320, 0, m->stream>>>(2 * rc.R, per, H2, Y3, gW + kEW3, gW + kEb3);
      k_pg_wgrad<T, kN1, kN2><<<cdiv(2 * rc.R, per), 320, 0, m->stream>>>(2 * rc.R, per, H1, Y2, gW + kEW2, gW + kEb2);
      m->launches += 3;
    }
  }
#undef PG_LAYER
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

}  // namespace

size_t param_grad_workspace_bytes(int cap, int rows, bool fp64) {
  const size_t fit = 2 * 2 * (size_t)kKD + 6 * 2 * (size_t)kF;  // per atom
  const size_t per_row = kPgGeo + 2 * (size_t)(kN1 + kN2 + kN2 + kN3 + kN2 + kN2 + kN1) + 1;
  return ((size_t)cap * 1600 + std::max((size_t)cap * fit, (size_t)rows * per_row)) * (fp64 ? 8 : 4);
}

dp_status launch_param_grad(Model* m, int N, const double* F0, double E0, double cE, double cF, double* grad,
                            double* loss) {
  DP_CUDA_TRY(m, cudaMemsetAsync(grad, 0, sizeof(double) * (size_t)m->ntheta, m->stream));
  k_pg_setup<<<1, 1024, 0, m->stream>>>(N, m->e_atom, m->force, F0, m->perm, E0, cE, cF, m->pg_w, m->pg_scal);
  m->launches += 1;
  DP_LAUNCH_CHECK(m);
  dp_status st = (m->prec == DP_FP64) ? run_param_grad<double>(m, N, grad) : run_param_grad<float>(m, N, grad);
  if (st != DP_OK) return st;
  if (loss) DP_CUDA_TRY(m, cudaMemcpyAsync(loss, m->pg_scal + 1, sizeof(double), cudaMemcpyDeviceToDevice, m->stream));
  return DP_OK;
}

}  // namespace dpg
