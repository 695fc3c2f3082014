// Tabulated embedding of the mixed precisions with the table in shared memory.
//
// The one-row-per-thread table kernels (mix_embed.cu, TAB) read six coefficients of 100 outputs of the
// row's own interval, 3.2 KB a row from a 0.8 MB table that L1 cannot hold: 18 GB through L2 for a
// 32,000-atom crystal, 2.48 ms forward and 2.50 ms backward.  Here a CTA keeps one half of a pair's outputs
// (50 of 100) as node data (value and h-scaled first and second derivative at the n + 1 nodes, 154 KB
// for 256 intervals) and a warp walks the neighbours of an atom with lane = two outputs: its
// shared-memory reads are consecutive, the six Hermite basis values of a row are the same for all
// outputs, and T (forward) or dR_hat, d s_hat (backward) are sums in registers.  A row outside the table
// (an input below the first or above the last node) is evaluated from the edge interval's coefficients: u intervals
// beyond the edge the Hermite basis values grow as u^5 and cancel, which costs all FP32 digits.  Half the CTAs hold
// outputs 0..49, half 50..99; the backward's force terms are linear in those sums, so each half adds its own.
// Bound by shared-memory wavefronts and issue (about 32 and 54 a row forward): 32,000 Cu atoms 2.48 -> 0.72 ms
// forward, 2.50 -> 1.23 ms backward.
#include "tc_common.cuh"

namespace dpg {
namespace {

constexpr int kHalf = kN3 / 2;        // outputs of a CTA
constexpr int kNode = 3 * kHalf;      // floats of a node
constexpr int kWarps = 16;

struct TabArgs {
  int N, ntypes, S, n;
  int sel_off[kMaxTypes + 1];
  float rc, rs, winv, x0, ih;
  int switch_kind;
  const float* stat;
  const float* nodes;        // [pair][2][n + 1][3][50]
  const float4* coef;        // [pair][n][100][2]: quintic coefficients (rows outside the table)
  const int* type_off;
  const int* type_count;
  const int* nl_j;
  const float4* nl_d;
  const int* nl_count;
  float* Tseg;               // [nt][N][400]
  const float4* dT;          // [N][100] paired: (x_m, x_m+50, y_m, y_m+50), (z.., w..)
  float* force32;            // [N][4]
  double* vir_rep;
  const int* irep;
};

__device__ __forceinline__ void switch_fn(const TabArgs& a, float r, float& sw, float& dsw) {
  if (r < a.rs) { sw = 1.f; dsw = 0.f; return; }
  if (r >= a.rc) { sw = 0.f; dsw = 0.f; return; }
  const float u = (r - a.rs) * a.winv;
  if (a.switch_kind == 1) {
    const float pi = 3.14159265358979323846f;
    sw = 0.5f * cosf(pi * u) + 0.5f;
    dsw = -0.5f * pi * sinf(pi * u) * a.winv;
  } else {
    const float u2 = u * u;
    sw = u2 * u * (-6.f * u2 + 15.f * u - 10.f) + 1.f;
    dsw = -30.f * u2 * (u - 1.f) * (u - 1.f) * a.winv;
  }
}

struct Row {
  float d[3], R[4], rinv, sw, dsw;
};
__device__ __forceinline__ void env_row(const TabArgs& a, int ti, float4 dv, Row& f) {
  f.d[0] = dv.x; f.d[1] = dv.y; f.d[2] = dv.z;
  const float r2 = dv.x * dv.x + dv.y * dv.y + dv.z * dv.z;
  f.rinv = rsqrtf(r2);
  switch_fn(a, r2 * f.rinv, f.sw, f.dsw);
  const float s = f.sw * f.rinv, sr = s * f.rinv;
  f.R[0] = s; f.R[1] = sr * dv.x; f.R[2] = sr * dv.y; f.R[3] = sr * dv.z;
#pragma unroll
  for (int c = 0; c < 4; ++c) f.R[c] = (f.R[c] - a.stat[ti * 4 + c]) * a.stat[(a.ntypes + ti) * 4 + c];
}

// The interval of x (edge intervals beyond the ends) and the quintic Hermite basis at u = (x - x_i) / h for
// (f, h f', h^2 f'') at its left and right node; D: the derivatives of the basis.  Outside the table the basis is
// zero and `out` is set.
__device__ __forceinline__ int basis(const TabArgs& a, float x, float& u, bool& out, float* H) {
  const float f = (x - a.x0) * a.ih;
  const int i = min(max((int)floorf(f), 0), a.n - 1);
  u = f - (float)i;
  out = !(u >= 0.f && u <= 1.f);
  if (out) {
#pragma unroll
    for (int k = 0; k < 6; ++k) H[k] = 0.f;
    return i;
  }
  const float u2 = u * u, u3 = u2 * u;
  const float s = u3 * fmaf(u, fmaf(6.f, u, -15.f), 10.f);
  H[0] = 1.f - s;
  H[1] = u + u3 * fmaf(u, fmaf(-3.f, u, 8.f), -6.f);
  H[2] = 0.5f * (u2 + u3 * fmaf(u, fmaf(-1.f, u, 3.f), -3.f));
  H[3] = s;
  H[4] = u3 * fmaf(u, fmaf(-3.f, u, 7.f), -4.f);
  H[5] = 0.5f * u3 * fmaf(u, fmaf(1.f, u, -2.f), 1.f);
  return i;
}
__device__ __forceinline__ void basis_d(float u, float* D) {
  const float u2 = u * u;
  const float s = u2 * fmaf(u, fmaf(30.f, u, -60.f), 30.f);
  D[0] = -s;
  D[1] = 1.f + u2 * fmaf(u, fmaf(-15.f, u, 32.f), -18.f);
  D[2] = u + u2 * fmaf(u, fmaf(-2.5f, u, 6.f), -4.5f);
  D[3] = s;
  D[4] = u2 * fmaf(u, fmaf(-15.f, u, 28.f), -12.f);
  D[5] = u2 * fmaf(u, fmaf(2.5f, u, -4.f), 1.5f);
}

// P(u) and P'(u) of outputs q and q + 1 from the coefficients of interval i.
__device__ __forceinline__ void poly2(const TabArgs& a, int pair, int i, int q, float u, float* g, float* gu) {
  const float4* p = a.coef + (((size_t)pair * a.n + i) * kN3 + q) * 2;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float4 lo = __ldg(p + 2 * k), hi = __ldg(p + 2 * k + 1);
    g[k] = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, hi.y, hi.x), lo.w), lo.z), lo.y), lo.x);
    gu[k] = fmaf(u, fmaf(u, fmaf(u, fmaf(u, 5.f * hi.y, 4.f * hi.x), 3.f * lo.w), 2.f * lo.z), lo.y);
  }
}

__device__ __forceinline__ void load_nodes(const TabArgs& a, int pair, int half, float* tab) {
  const float2* src = reinterpret_cast<const float2*>(a.nodes + ((size_t)pair * 2 + half) * (a.n + 1) * kNode);
  __syncthreads();  // every warp is done with the previous pair
  for (int q = threadIdx.x; q < (a.n + 1) * kNode / 2; q += 32 * kWarps) reinterpret_cast<float2*>(tab)[q] = src[q];
  __syncthreads();
}

// Two outputs (packed) at the lane's place in nodes i and i + 1: sum of basis times node data.
__device__ __forceinline__ uint64_t ld2(const float* p) { return *reinterpret_cast<const uint64_t*>(p); }
__device__ __forceinline__ uint64_t dup(float x) { return tc::f2(x, x); }

// ------------------------------------------------------------------ forward
// Partial T per neighbour type; G and R_hat are rounded to fp16 as in the T product of the other kernels.
__global__ void __launch_bounds__(32 * kWarps, 1) k_tab_fwd(TabArgs a) {
  extern __shared__ __align__(16) float sm[];
  float* tab = sm;
  float4(*rows)[32][3] = reinterpret_cast<float4(*)[32][3]>(sm + ((size_t)(a.n + 1) * kNode + 3) / 4 * 4);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = blockIdx.x & 1;
  const int wid = (blockIdx.x >> 1) * kWarps + w, nw = (gridDim.x >> 1) * kWarps;
  float4(*mine)[3] = rows[w];
  const int fo = 2 * min(lane, kHalf / 2 - 1);
  for (int pair = 0; pair < a.ntypes * a.ntypes; ++pair) {
    const int ti = pair / a.ntypes, tj = pair % a.ntypes;
    if (a.type_count[ti] == 0) continue;
    load_nodes(a, pair, half, tab);
    const int i1 = a.type_off[ti] + a.type_count[ti];
    for (int i = a.type_off[ti] + wid; i < i1; i += nw) {
      const int cnt = a.nl_count[(size_t)i * a.ntypes + tj];
      const float4* dp = a.nl_d + (size_t)i * a.S + a.sel_off[tj];
      uint64_t acc[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c] = dup(0.f);
      float4 nxt = lane < cnt ? dp[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      for (int b = 0; b < cnt; b += 32) {
        const float4 dv = nxt;
        if (b + 32 + lane < cnt) nxt = dp[b + 32 + lane];
        __syncwarp();
        bool out = false;
        if (b + lane < cnt) {
          Row f;
          float H[6], u;
          env_row(a, ti, dv, f);
          const int k = basis(a, f.R[0], u, out, H);
#pragma unroll
          for (int c = 0; c < 4; ++c) f.R[c] = __half2float(__float2half_rn(f.R[c]));
          mine[lane][0] = make_float4(H[0], H[1], H[2], H[3]);
          mine[lane][1] = make_float4(H[4], H[5], __int_as_float(k * kNode), f.R[0]);
          mine[lane][2] = make_float4(f.R[1], f.R[2], f.R[3], u);
        }
        unsigned far = __ballot_sync(0xffffffffu, out);
        __syncwarp();
        const int nr = min(32, cnt - b);
        for (; far; far &= far - 1) {
          const int r = __ffs(far) - 1;
          const float4 q = mine[r][1], s = mine[r][2];
          float g[2], gu[2];
          poly2(a, pair, __float_as_int(q.z) / kNode, half * kHalf + fo, s.w, g, gu);
          const float2 G = __half22float2(__floats2half2_rn(g[0], g[1]));
          const uint64_t gg = tc::f2(G.x, G.y);
          acc[0] = tc::f2fma(dup(q.w), gg, acc[0]);
          acc[1] = tc::f2fma(dup(s.x), gg, acc[1]);
          acc[2] = tc::f2fma(dup(s.y), gg, acc[2]);
          acc[3] = tc::f2fma(dup(s.z), gg, acc[3]);
        }
#pragma unroll 2
        for (int r = 0; r < nr; ++r) {
          const float4 p = mine[r][0], q = mine[r][1], s = mine[r][2];
          const float* t = tab + __float_as_int(q.z) + fo;
          uint64_t g = tc::f2mul(dup(p.x), ld2(t));
          uint64_t h = tc::f2mul(dup(p.w), ld2(t + kNode));
          g = tc::f2fma(dup(p.y), ld2(t + kHalf), g);
          h = tc::f2fma(dup(q.x), ld2(t + kNode + kHalf), h);
          g = tc::f2fma(dup(p.z), ld2(t + 2 * kHalf), g);
          h = tc::f2fma(dup(q.y), ld2(t + kNode + 2 * kHalf), h);
          g = tc::f2add(g, h);
          const float2 G = __half22float2(__floats2half2_rn(tc::f2lo(g), tc::f2hi(g)));
          g = tc::f2(G.x, G.y);
          acc[0] = tc::f2fma(dup(q.w), g, acc[0]);
          acc[1] = tc::f2fma(dup(s.x), g, acc[1]);
          acc[2] = tc::f2fma(dup(s.y), g, acc[2]);
          acc[3] = tc::f2fma(dup(s.z), g, acc[3]);
        }
      }
      if (lane < kHalf / 2) {
        float* o = a.Tseg + ((size_t)tj * a.N + i) * 400 + half * kHalf + 2 * lane;
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<uint64_t*>(o + c * kN3) = acc[c];
      }
    }
  }
}

// ------------------------------------------------------------------ backward
// Sums over the 32 lanes of v[row][5] for eight rows; lane 4 r (r = row's bit-reversed place) ends with row's sums.
__device__ __forceinline__ void reduce8(float (*v)[5], int lane, float* out) {
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const float send = h16 ? v[r][q] : v[r + 4][q], keep = h16 ? v[r + 4][q] : v[r][q];
      v[r][q] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const float send = h8 ? v[r][q] : v[r + 2][q], keep = h8 ? v[r + 2][q] : v[r][q];
      v[r][q] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const float send = h4 ? v[0][q] : v[1][q], keep = h4 ? v[1][q] : v[0][q];
    float x = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    out[q] = x;  // row ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)
  }
}

__global__ void __launch_bounds__(32 * kWarps, 1) k_tab_bwd(TabArgs a) {
  extern __shared__ __align__(16) float sm[];
  float* tab = sm;
  float4(*rows)[32][5] = reinterpret_cast<float4(*)[32][5]>(sm + ((size_t)(a.n + 1) * kNode + 3) / 4 * 4);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = blockIdx.x & 1;
  const int wid = (blockIdx.x >> 1) * kWarps + w, nw = (gridDim.x >> 1) * kWarps;
  float4(*mine)[5] = rows[w];
  const int fo = 2 * min(lane, kHalf / 2 - 1);
  float vacc[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) vacc[q] = 0.f;
  int vrep = -1;
  auto flush = [&]() {
    if (vrep >= 0) {
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        float v = vacc[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(&a.vir_rep[9 * vrep + q], (double)v);
        vacc[q] = 0.f;
      }
    }
  };
  for (int pair = 0; pair < a.ntypes * a.ntypes; ++pair) {
    const int ti = pair / a.ntypes, tj = pair % a.ntypes;
    if (a.type_count[ti] == 0) continue;
    load_nodes(a, pair, half, tab);
    float isd[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) isd[c] = a.stat[(a.ntypes + ti) * 4 + c];
    const int i1 = a.type_off[ti] + a.type_count[ti];
    for (int i = a.type_off[ti] + wid; i < i1; i += nw) {
      const int cnt = a.nl_count[(size_t)i * a.ntypes + tj];
      if (cnt == 0) continue;
      if (a.irep[i] != vrep) {
        flush();
        vrep = a.irep[i];
      }
      const size_t e0 = (size_t)i * a.S + a.sel_off[tj];
      // dE/dT of the lane's outputs m = fo, fo + 1 (of the first or second half of the 100)
      uint64_t dt[4];
      {
        const float4* p = a.dT + (size_t)i * kN3 + 2 * fo;
        const float4 a0 = p[0], a1 = p[1], b0 = p[2], b1 = p[3];
        const bool on = lane < kHalf / 2;  // idle lanes add nothing to the sums
        dt[0] = on ? (half ? tc::f2(a0.y, b0.y) : tc::f2(a0.x, b0.x)) : dup(0.f);
        dt[1] = on ? (half ? tc::f2(a0.w, b0.w) : tc::f2(a0.z, b0.z)) : dup(0.f);
        dt[2] = on ? (half ? tc::f2(a1.y, b1.y) : tc::f2(a1.x, b1.x)) : dup(0.f);
        dt[3] = on ? (half ? tc::f2(a1.w, b1.w) : tc::f2(a1.z, b1.z)) : dup(0.f);
      }
      float fi[3] = {0.f, 0.f, 0.f};
      for (int b = 0; b < cnt; b += 32) {
        Row f;
        const bool in = b + lane < cnt;
        bool out = false;
        __syncwarp();
        {
          float H[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, D[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          float u = 0.f;
          int k = 0;
          f.R[0] = f.R[1] = f.R[2] = f.R[3] = 0.f;
          if (in) {
            env_row(a, ti, a.nl_d[e0 + b + lane], f);
            k = basis(a, f.R[0], u, out, H);
            if (!out) basis_d(u, D);
          }
          mine[lane][0] = make_float4(H[0], H[1], H[2], H[3]);
          mine[lane][1] = make_float4(H[4], H[5], __int_as_float(k * kNode), f.R[0]);
          mine[lane][2] = make_float4(f.R[1], f.R[2], f.R[3], D[0]);
          mine[lane][3] = make_float4(D[1], D[2], D[3], D[4]);
          mine[lane][4] = make_float4(D[5], u, 0.f, 0.f);
        }
        unsigned far = __ballot_sync(0xffffffffu, out);
        __syncwarp();
        const int nr = min(32, cnt - b);
        float own[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // this lane's row
        for (int r0 = 0; r0 < nr; r0 += 8) {
          float v[8][5];
#pragma unroll
          for (int r = 0; r < 8; ++r) {  // rows past the last have a zero basis and R_hat
            const float4 p = mine[r0 + r][0], q = mine[r0 + r][1], s = mine[r0 + r][2], x = mine[r0 + r][3];
            const float d5 = mine[r0 + r][4].x;
            const float* t = tab + __float_as_int(q.z) + fo;
            const uint64_t n0 = ld2(t), n1 = ld2(t + kHalf), n2 = ld2(t + 2 * kHalf);
            const uint64_t n3 = ld2(t + kNode), n4 = ld2(t + kNode + kHalf), n5 = ld2(t + kNode + 2 * kHalf);
            uint64_t g = tc::f2mul(dup(p.x), n0), gd = tc::f2mul(dup(s.w), n0);
            g = tc::f2fma(dup(p.y), n1, g);
            gd = tc::f2fma(dup(x.x), n1, gd);
            g = tc::f2fma(dup(p.z), n2, g);
            gd = tc::f2fma(dup(x.y), n2, gd);
            g = tc::f2fma(dup(p.w), n3, g);
            gd = tc::f2fma(dup(x.z), n3, gd);
            g = tc::f2fma(dup(q.x), n4, g);
            gd = tc::f2fma(dup(x.w), n4, gd);
            g = tc::f2fma(dup(q.y), n5, g);
            gd = tc::f2fma(dup(d5), n5, gd);
            uint64_t dg = tc::f2mul(dup(q.w), dt[0]);
            dg = tc::f2fma(dup(s.x), dt[1], dg);
            dg = tc::f2fma(dup(s.y), dt[2], dg);
            dg = tc::f2fma(dup(s.z), dt[3], dg);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint64_t m = tc::f2mul(dt[c], g);
              v[r][c] = tc::f2lo(m) + tc::f2hi(m);
            }
            const uint64_t m = tc::f2mul(dg, gd);
            v[r][4] = tc::f2lo(m) + tc::f2hi(m);
          }
          float o[5];
          reduce8(v, lane, o);
          // the sums of row r0 + k sit in lanes whose bits 4, 3, 2 spell k: hand them to lane r0 + k
          const int k = lane & 7, src = (k & 4) * 4 + (k & 2) * 4 + (k & 1) * 4;
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            const float y = __shfl_sync(0xffffffffu, o[q], src);
            if ((lane & ~7) == r0) own[q] = y;
          }
        }
        for (; far; far &= far - 1) {
          const int r = __ffs(far) - 1;
          const float4 q = mine[r][1], s = mine[r][2];
          float g[2], gu[2], v[5];
          poly2(a, pair, __float_as_int(q.z) / kNode, half * kHalf + fo, mine[r][4].y, g, gu);
          const uint64_t gg = tc::f2(g[0], g[1]);
          uint64_t dg = tc::f2mul(dup(q.w), dt[0]);
          dg = tc::f2fma(dup(s.x), dt[1], dg);
          dg = tc::f2fma(dup(s.y), dt[2], dg);
          dg = tc::f2fma(dup(s.z), dt[3], dg);
#pragma unroll
          for (int c = 0; c < 5; ++c) {
            const uint64_t m = c < 4 ? tc::f2mul(dt[c], gg) : tc::f2mul(dg, tc::f2(gu[0], gu[1]));
            v[c] = lane < kHalf / 2 ? tc::f2lo(m) + tc::f2hi(m) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
            if (lane == r) own[c] = v[c];
          }
        }
        if (in) {
          own[0] += own[4] * a.ih;
#pragma unroll
          for (int c = 0; c < 4; ++c) own[c] *= isd[c];
          const float rinv = f.rinv;
          const float dsr = f.dsw * rinv - f.sw * rinv * rinv;
          const float qv = f.sw * rinv * rinv;
          const float dq = f.dsw * rinv * rinv - 2.f * f.sw * rinv * rinv * rinv;
          const float proj = own[1] * f.d[0] + own[2] * f.d[1] + own[3] * f.d[2];
          const float common = (own[0] * dsr + dq * proj) * rinv;
          float g3[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            g3[c] = common * f.d[c] + qv * own[1 + c];
            fi[c] += g3[c];
          }
          tc::red_add_v4(a.force32 + 4 * (size_t)a.nl_j[e0 + b + lane], -g3[0], -g3[1], -g3[2], 0.f);
#pragma unroll
          for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) vacc[3 * p + q] = fmaf(-g3[p], f.d[q], vacc[3 * p + q]);
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fi[c] += __shfl_xor_sync(0xffffffffu, fi[c], o);
      if (lane == 0) tc::red_add_v4(a.force32 + 4 * (size_t)i, fi[0], fi[1], fi[2], 0.f);
    }
  }
  flush();
}

// FP32 node data of the table: [pair][half][node][f, h f', h^2 f''][50] from the FP64 nodes [pair][node][100][3].
__global__ void k_tab_nodes32(int n, double h, const double* __restrict__ v, float* __restrict__ out) {
  const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;  // (pair, node, output)
  const int pair = blockIdx.y;
  if (idx >= (size_t)(n + 1) * kN3) return;
  const int q = (int)(idx % kN3), i = (int)(idx / kN3);
  const double* s = v + (((size_t)pair * (n + 1) + i) * kN3 + q) * 3;
  float* o = out + (((size_t)pair * 2 + q / kHalf) * (n + 1) + i) * kNode + q % kHalf;
  o[0] = (float)s[0];
  o[kHalf] = (float)(h * s[1]);
  o[2 * kHalf] = (float)(h * h * s[2]);
}

TabArgs make_args(Model* m, int N) {
  TabArgs a{};
  a.N = N; a.ntypes = m->ntypes; a.S = m->S; a.n = m->tab_n;
  for (int t = 0; t <= m->ntypes; ++t) a.sel_off[t] = m->sel_off[t];
  a.rc = (float)m->rc; a.rs = (float)m->rs; a.winv = 1.f / (a.rc - a.rs);
  a.x0 = (float)m->tab_x0; a.ih = (float)(1.0 / m->tab_h);
  a.switch_kind = m->switch_kind; a.stat = m->stat32; a.nodes = m->tab_nodes32;
  a.coef = reinterpret_cast<const float4*>(m->tab32);
  a.type_off = m->type_off; a.type_count = m->type_count; a.nl_j = m->nl_j;
  a.nl_d = static_cast<const float4*>(m->nl_d); a.nl_count = m->nl_count;
  a.Tseg = m->Tseg; a.dT = static_cast<const float4*>(m->dTm); a.force32 = m->force32;
  a.vir_rep = m->vir_rep; a.irep = m->irep;
  return a;
}
size_t tab_smem(int n, int vecs) { return (((size_t)(n + 1) * kNode + 3) / 4 * 4) * 4 + (size_t)kWarps * 32 * vecs * 16; }

}  // namespace

// The table of one half of the outputs fits shared memory beside the backward's row data (n <= 318), and
// there are enough neighbour slots to pay for loading it once per pair and CTA.
bool tab_smem_path(const Model* m, int N) {
  return m->tab_n > 0 && tab_smem(m->tab_n, 5) <= 227 * 1024 && (long)N * m->S >= kTabSlots;
}

dp_status launch_tab_nodes32(Model* m, int n, double h, const double* v, float* out) {
  k_tab_nodes32<<<dim3(cdiv((long)(n + 1) * kN3, 256), m->ntypes * m->ntypes), 256, 0, m->stream>>>(n, h, v, out);
  m->launches += 1;
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}
dp_status launch_tab_forward(Model* m, int N) {
  const size_t smem = tab_smem(m->tab_n, 3);
  DP_CUDA_TRY(m, ensure_smem(reinterpret_cast<const void*>(k_tab_fwd), smem));
  k_tab_fwd<<<num_sms() / 2 * 2, 32 * kWarps, smem, m->stream>>>(make_args(m, N));
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}
dp_status launch_tab_backward(Model* m, int N) {
  const size_t smem = tab_smem(m->tab_n, 5);
  DP_CUDA_TRY(m, ensure_smem(reinterpret_cast<const void*>(k_tab_bwd), smem));
  k_tab_bwd<<<num_sms() / 2 * 2, 32 * kWarps, smem, m->stream>>>(make_args(m, N));
  DP_LAUNCH_CHECK(m);
  return DP_OK;
}

}  // namespace dpg
