// Quadrature nodes row by row (FP32), shared by the tensor-core assembly and
// the adjoint contraction: direction patches built by the lanes of a warp in
// parallel, and the node geometry of node.cuh with everything that is constant
// along a row of a patch (fixed xi) taken out of the node.
//
// On a row the bilinear map is f(eta) = F0 + eta F1, F0 = a + b xi,
// F1 = c + d xi, so with N = F1 x F0
//   det[f, f_xi, f_eta] = N . b + eta N . d
// and every linear form m . f (the three s_X of the closed form, the receiving
// tangential momentum, the exit face's normal) is m . F0 + eta m . F1: one FMA
// per node instead of three multiply-adds on a normalised direction.  The
// closed form is homogeneous in d, so it is evaluated on f itself:
//   |OBC| = |ABC| s_A(f) / den(f),   L_O = D3 |f| / den(f).
// A node takes about 45 instructions plus the Zernike vectors (about 200 with
// the direct evaluation at every node).
#pragma once

#include "node.cuh"

namespace dfm {
namespace {

// Subdivision state of one warp: a stack of the polygons still to be split (12
// generator floats and nv | depth << 8 each; 13 words, so that lanes touching
// consecutive entries hit distinct banks) and the patches ready for
// quadrature.
constexpr int kPolyCap = 40;     // stack entries
constexpr int kPolyBatch = 8;    // polygons split side by side, four children each
constexpr int kRowPatches = 20;  // patches per chunk

struct PatchWarp {
  alignas(16) float patch[kRowPatches][12];  // a, b, c, d of Eq. (Parametr)
  float poly[kPolyCap][13];
  int sp, npatch;
};

// The lanes with `on` hold a polygon each: those with an edge longer than the
// threshold (depth < kMaxDepth) go onto the stack, the others become patches.
// A triangle repeats its first generator as the fourth.
__device__ __forceinline__ void sort_polygons(PatchWarp& S, const float (&v)[4][3], int nv, int depth, bool on,
                                              float cos_max, int lane, int& sp, int& np) {
  float minc = fminf(fminf(dotf(v[0], v[1]), dotf(v[1], v[2])), dotf(v[2], v[3]));
  if (nv == 4) minc = fminf(minc, dotf(v[3], v[0]));
  const bool split = on && minc < cos_max && depth < kMaxDepth;
  const bool leaf = on && !split;
  const unsigned ms = __ballot_sync(0xffffffffu, split), ml = __ballot_sync(0xffffffffu, leaf);
  const unsigned below = (1u << lane) - 1u;
  if (leaf) {
    float o[12];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o[c] = 0.25f * (v[0][c] + v[1][c] + v[2][c] + v[3][c]);
      o[3 + c] = 0.25f * (v[1][c] - v[0][c] + v[2][c] - v[3][c]);
      o[6 + c] = 0.25f * (v[2][c] + v[3][c] - v[0][c] - v[1][c]);
      o[9 + c] = 0.25f * (v[2][c] - v[3][c] + v[0][c] - v[1][c]);
    }
    float4* out = reinterpret_cast<float4*>(S.patch[np + __popc(ml & below)]);
#pragma unroll
    for (int u = 0; u < 3; ++u) out[u] = make_float4(o[4 * u], o[4 * u + 1], o[4 * u + 2], o[4 * u + 3]);
  }
  if (split) {
    float* q = S.poly[sp + __popc(ms & below)];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int x = 0; x < 3; ++x) q[3 * k + x] = v[k][x];
    q[12] = __int_as_float(nv | depth << 8);
  }
  sp += __popc(ms);
  np += __popc(ml);
}

// Lanes 0..3: the four non-empty direction regions (region_poly of node.cuh;
// every generator is a difference of two of the tet's vertices A, B, C, D).
__device__ __forceinline__ void start_regions(PatchWarp& S, const PairConst& pc, float cos_max, int lane) {
  const int r = lane & 3;
  const float* V = pc.A;  // A, B, C, D one after the other
  float v[4][3];
  auto gen = [&](int k, int p, int q) {
#pragma unroll
    for (int x = 0; x < 3; ++x) v[k][x] = V[3 * p + x] - V[3 * q + x];
    nrm3(v[k]);
  };
  gen(0, 3, 0);
  gen(1, r == 1 ? 1 : 3, r == 1 ? 0 : (r == 3 ? 2 : 1));
  gen(2, r == 0 ? 3 : (r == 3 ? 1 : 2), r == 1 ? 0 : (r == 2 ? 1 : 2));
  const int nv = r < 2 ? 3 : 4;
  gen(3, nv == 3 ? 3 : (r == 2 ? 2 : 1), 0);
  int sp = 0, np = 0;
  sort_polygons(S, v, nv, 0, lane < 4, cos_max, lane, sp, np);
  if (lane == 0) {
    S.sp = sp;
    S.npatch = np;
  }
  __syncwarp();
}

// Split polygons, up to kPolyBatch at a time with one lane per child (midpoint
// subdivision on the sphere, fill_patches of node.cuh), until the patch buffer
// is full or the stack is empty.  Returns the number of patches (0: done).
// Splitting n polygons grows the stack by at most 3 n; batches of several leave
// 12 entries free, which is what taking one polygon at a time to the deepest
// level can still add.
__device__ __forceinline__ int fill_patches_warp(PatchWarp& S, float cos_max, int lane) {
  int np = S.npatch;
  int sp = S.sp;
  __syncwarp();
  while (sp > 0 && np + 4 <= kRowPatches) {
    int n = (kPolyCap - 12 - sp) / 3;
    n = min(min(max(1, n), kPolyBatch), min(sp, (kRowPatches - np) >> 2));
    const int par = lane >> 2, c = lane & 3;
    const bool on = par < n;
    const float* P = S.poly[sp - 1 - (on ? par : 0)];
    const int tag = __float_as_int(P[12]);
    const int nv = tag & 0xff, depth = tag >> 8;
    const bool quad = nv == 4;
    // corner a and its neighbours b, d (a triangle's middle child: all three)
    const int ia = quad ? c : (c == 3 ? 0 : c);
    const int ib = quad ? (c + 1) & 3 : (ia == 2 ? 0 : ia + 1);
    const int id = quad ? (c + 3) & 3 : (ia == 0 ? 2 : ia - 1);
    float a[3], m1[3], m2[3], m3[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      a[x] = P[3 * ia + x];
      const float b = P[3 * ib + x], d = P[3 * id + x];
      m1[x] = a[x] + b;
      m2[x] = a[x] + d;
      m3[x] = quad ? P[x] + P[3 + x] + P[6 + x] + P[9 + x] : b + d;
    }
    nrm3(m1);
    nrm3(m2);
    nrm3(m3);
    // quadrilateral: (a, ab, centre, da); triangle (v0, v1, v2): (v0, 01, 20),
    // (01, v1, 12), (20, 12, v2), (01, 12, 20)
    float v[4][3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      v[0][x] = quad || c == 0 ? a[x] : (c == 1 ? m2[x] : m1[x]);
      v[1][x] = quad || c == 0 ? m1[x] : (c == 1 ? a[x] : (c == 2 ? m2[x] : m3[x]));
      v[2][x] = quad ? m3[x] : (c == 1 ? m1[x] : (c == 2 ? a[x] : m2[x]));
      v[3][x] = quad ? m2[x] : v[0][x];
    }
    __syncwarp();  // every parent is read before its entry is reused
    sp -= n;
    sort_polygons(S, v, nv, depth + 1, on, cos_max, lane, sp, np);
    __syncwarp();
  }
  if (lane == 0) {
    S.sp = sp;
    S.npatch = 0;
  }
  __syncwarp();
  return np;
}

// v as the sum of two FP32 numbers.  What all pairs share, Gauss weights and norms, is
// kept this way: the rounding of a pair's own constants averages out over a mesh,
// but one common to all entries is magnified by a solve at little damping (FP32
// weights alone add up to 3.0e-8 too much at q = 9 and 10, and 3.0e-8 too little at
// q = 8).
__device__ __forceinline__ float2 two_floats(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}
// x v, rounded once (a rounded x hi plus x lo would often round back)
__device__ __forceinline__ float times(float x, float2 v) { return fmaf(x, v.x, x * v.y); }

// 1 / x to FP32 rounding (the approximate reciprocal and one Newton step)
__device__ __forceinline__ float recip(float x) {
  float r = __fdividef(1.f, x);
  return fmaf(r, fmaf(-x, r, 1.f), r);
}

// phi2 (see node.cuh) in FP32: the series up to x = 1 (12 terms: the first one
// left out is below 2e-10 of the sum there), which also spares the closed
// form's cancellation just above its own limit
__device__ __forceinline__ float phi2_row(float x) {
  if (x < 1.f) {
    const float c[12] = {1.f / 2,       1.f / 6,        1.f / 24,        1.f / 120,        1.f / 720,         1.f / 5040,
                         1.f / 40320,   1.f / 362880,   1.f / 3628800,   1.f / 39916800,   1.f / 479001600,   1.f / 6227020800.f};
    float s = c[11];
#pragma unroll
    for (int i = 10; i >= 0; --i) s = fmaf(-x, s, c[i]);
    return s;
  }
  return (x - 1.f + expf(-x)) / (x * x);
}

// Packed FP32 pairs (two independent IEEE operations per instruction).
__device__ __forceinline__ float2 pair(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// What a row of a patch fixes: value at eta = 0 and slope of ...
struct RowConst {
  float2 x0, x1;    // (f_x, receiving tangential momentum along e1')
  float2 y0, y1;    // (f_y, the same along e2'; both times the refraction factor)
  float2 zd0, zd1;  // (f_z, det[f, f_xi, f_eta])
  float2 bc0, bc1;  // (s_B, s_C)
  float a0, a1;     // s_A
  float n0, n1;     // inward normal of the exit face . f (interfaces between media)
};

__device__ __forceinline__ void row_const(const float* cf, float xi, const PairConst& pc, RowConst& r) {
  float b[3], d[3], F0[3], F1[3];
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    b[x] = cf[3 + x];
    d[x] = cf[9 + x];
    F0[x] = fmaf(b[x], xi, cf[x]);
    F1[x] = fmaf(d[x], xi, cf[6 + x]);
  }
  const float n0 = F1[1] * F0[2] - F1[2] * F0[1];
  const float n1 = F1[2] * F0[0] - F1[0] * F0[2];
  const float n2 = F1[0] * F0[1] - F1[1] * F0[0];
  r.zd0 = pair(F0[2], n0 * b[0] + n1 * b[1] + n2 * b[2]);
  r.zd1 = pair(F1[2], n0 * d[0] + n1 * d[1] + n2 * d[2]);
  r.a0 = dotf(pc.mA, F0);
  r.a1 = dotf(pc.mA, F1);
  r.bc0 = pair(dotf(pc.mB, F0), dotf(pc.mC, F0));
  r.bc1 = pair(dotf(pc.mB, F1), dotf(pc.mC, F1));
  r.x0 = pair(F0[0], pc.qscale * dotf(pc.R1, F0));
  r.x1 = pair(F1[0], pc.qscale * dotf(pc.R1, F1));
  r.y0 = pair(F0[1], pc.qscale * dotf(pc.R2, F0));
  r.y1 = pair(F1[1], pc.qscale * dotf(pc.R2, F1));
  r.n0 = dotf(pc.ndst, F0);
  r.n1 = dotf(pc.ndst, F1);
}

// One node of a row: tangential momenta px = (source, receiving) along the
// first frame axes and py along the second, L_O, and base = jac s_A / den times
// the media weight (zero outside the regions' support, s_A <= 0), so that the
// node's weight is w_i w_j 2 |ABC| base phi2(mu L_O).
struct RowNode {
  float2 px, py;
  float LO, base;
};

__device__ __forceinline__ RowNode row_node(const RowConst& r, float eta, float D3, int kind, const PairConst& pc) {
  RowNode o;
  const float2 e2 = pair(eta, eta);
  const float2 fx = fma2(e2, r.x1, r.x0), fy = fma2(e2, r.y1, r.y0), zd = fma2(e2, r.zd1, r.zd0);
  const float2 bc = fma2(e2, r.bc1, r.bc0);
  const float sA = fmaf(eta, r.a1, r.a0);
  const float r2 = fmaf(fx.x, fx.x, fmaf(fy.x, fy.x, zd.x * zd.x));
  // 1 / |f| to FP32 rounding: one Newton step, r2 being within [1/4, 1].  rsqrtf alone
  // is 4.9e-9 too small on average there, and base has its fourth power
  float ri = rsqrtf(r2);
  ri = fmaf(0.5f * ri, fmaf(-r2 * ri, ri, 1.f), ri);
  const bool ok = sA > 1e-30f;  // den >= s_A: its reciprocal stays finite
  const float inv = ok ? recip(sA + fmaxf(bc.x, 0.f) + fmaxf(bc.y, 0.f)) : 0.f;
  const float ri2 = ri * ri;
  o.LO = D3 * (r2 * ri) * inv;
  o.base = ok ? fabsf(zd.x * zd.y) * (ri2 * ri2) * (sA * inv) : 0.f;
  o.px = mul2(fx, pair(ri, ri));
  o.py = mul2(fy, pair(ri, ri));
  if (kind > 0) {
    const float cos_r = -fmaf(eta, r.n1, r.n0) * ri;
    o.base *= kind == 1 ? transmission_prob<float>(cos_r, pc.c_ratio, pc.z_src, pc.z_dst)
                        : reflection_prob<float>(cos_r, pc.c_ratio, pc.z_src, pc.z_dst);
  }
  return o;
}

// zernike<NP> (node.cuh) at two points at once, c0 times: the source and the
// receiving momentum of a node run the same recursion, so packed instructions
// serve both, and the node's weight rides in c0.
template <int NP>
__device__ __forceinline__ void zernike2(float2 px, float2 py, float2 c0, float2* Z) {
  const float2 r2 = fma2(px, px, mul2(py, py));
  const float2 npy = pair(-py.x, -py.y), minus = pair(-1.f, -1.f), two_r2 = pair(2.f * r2.x, 2.f * r2.y);
  float2 Q[NP + 1][NP + 1];
  float2 cr[NP + 1], ci[NP + 1];
  cr[0] = c0;
#pragma unroll
  for (int m = 1; m <= NP; ++m) {
    if (m == 1) {
      cr[1] = mul2(c0, px);
      ci[1] = mul2(c0, py);
    } else {
      cr[m] = fma2(ci[m - 1], npy, mul2(cr[m - 1], px));
      ci[m] = fma2(cr[m - 1], py, mul2(ci[m - 1], px));
    }
  }
#pragma unroll
  for (int n = 0; n <= NP; ++n) {
#pragma unroll
    for (int m = n & 1; m <= n; m += 2) {
      if (m == n) Q[n][m] = pair(1.f, 1.f);
      else if (n == 2) Q[n][m] = fma2(two_r2, pair(1.f, 1.f), minus);
      else if (m == 0) Q[n][m] = fma2(two_r2, Q[n - 1][1], mul2(Q[n - 2][0], minus));
      else if (m == n - 2) Q[n][m] = fma2(r2, pair(1.f, 1.f), fma2(Q[n - 2][m], minus, Q[n - 1][m - 1]));
      else Q[n][m] = fma2(r2, Q[n - 1][m + 1], fma2(Q[n - 2][m], minus, Q[n - 1][m - 1]));
      const int i = n * (n + 2) / 2;
      if (m == 0) {
        Z[i] = n == 0 ? c0 : mul2(Q[n][0], c0);
      } else {
        const int ip = (n * (n + 2) + m) / 2, im = (n * (n + 2) - m) / 2;
        Z[ip] = m == n ? cr[m] : mul2(Q[n][m], cr[m]);
        Z[im] = m == n ? ci[m] : mul2(Q[n][m], ci[m]);
      }
    }
  }
}

// Rows of a chunk are handed to the 32 lanes in passes: 32 rows with one lane
// each, or, for the remainder, t rows with g = 32 / t lanes each (16 when at
// least 16 are left: two half-empty passes cost less than a full-length one).
struct RowPass {
  int rows, per;  // rows taken, lanes per row
};
__device__ __forceinline__ RowPass next_pass(int left) {
  RowPass p;
  p.rows = left >= 32 ? 32 : (left >= 16 ? 16 : left);
  p.per = 32 / p.rows;
  return p;
}

}  // namespace
}  // namespace dfm
