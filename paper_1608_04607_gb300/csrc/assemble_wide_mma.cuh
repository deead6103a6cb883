// Assembly of the bases above N_p = 8 (piecewise-constant spatial basis) with
// the block sums on tensor cores.  Included by wide.cu.
//
// One block of 16 warps per (face pair, tile of test functions).  Per pass of 64
// quadrature nodes every warp first evaluates its share of the next pass's
// vectors into the other staging buffer (Z(p) or w Z(p') of 32 nodes, the
// functions of a quarter of the m), then forms its part of the present pass's
// product as in assemble_mma.cuh: FP16 hi + lo parts of both factors, hi on a grid
// on which the tensor cores' sums are exact, three mma.sync m16n8k16 products per
// 16 nodes started at zero for every 32 nodes, whose weights are scaled by a power
// of two, then added to FP32 sums.  A warp
// owns 2 x TN tiles of 16 x 8 entries.
//
// The Zernike functions come m-major out of the radial recurrence, cosine and
// sine together, and are staged in that order (one 4-byte store for the pair of
// hi parts, one for the lo parts); the epilogue sends rows and columns back to
// the basis order.  N_p = 16 takes 3 x 2 x 200 MMAs per 32 nodes, 2,400 cycles of an
// SM of its 6,400: the rest goes to the latencies of the recurrences and of the
// FP16 splits in front of the barrier of each pass.  N_p = 16, 768 tets: 71.3 ms
// by assemble_wide_kernel (FP32 FMAs), 38.6 ms here.  Half of the warps evaluating
// before their products and half after: 47.2 ms, instruction fetches.
#pragma once

#include "assemble_mma.cuh"

namespace dfm {
namespace {

// warps, nodes and tiles: launch_geometry.h (shared with a host-side check)
constexpr int kWmWarps = geom::kWideMmaWarps;
constexpr int kWmNodes = geom::kWideMmaNodes;  // per pass
using geom::WideMma;

// The Zernike functions of order <= Np with |m| = sub mod 4 at (px, py), times
// s: hi and lo FP16 parts at positions [r0, r0 + rows) of the staged order, into
// hi and lo.  s_pos[m]: position of the first function of m.  The recurrence of
// zernike_wide.h with its coefficients from a table (Q_n = (A rho^2 + B) Q_{n-2} +
// C Q_{n-4}, entry s_pos[m] / 2 + (n - m) / 2, m = 0 from kRadial0 on) in a loop,
// four steps unrolled so that conversions of several functions are in flight:
// 36.9 ms at N_p = 16, 768 tets, when this was chosen; 43.5 ms not unrolled, 38.5 ms
// unrolled over m and n for each m mod 4, code that outgrows the instruction caches.
constexpr int kRadial0 = 128;
__device__ __forceinline__ void stage_zernike(int Np, float px, float py, float s, int sub, const short* s_pos,
                                              const float4* s_rad, int r0, int rows, __half* hi, __half* lo) {
  const float r2 = px * px + py * py;
  // (px + i py)^sub s and the step to the next m, (px + i py)^4
  float cr = s, ci = 0.f;
  for (int k = 0; k < sub; ++k) {
    const float t = cr * px - ci * py;
    ci = cr * py + ci * px;
    cr = t;
  }
  const float sr = px * px - py * py, si = 2.f * px * py;
  const float fr = sr * sr - si * si, fi = 2.f * sr * si;
  int m = sub;
  if (m == 0) {
    const int pos0 = s_pos[0] - r0, cnt = (Np >> 1) + 1;
    float qa = 0.f, qb = 1.f;
#pragma unroll 2
    for (int k = 0; k < cnt; ++k) {
      const float4 t = s_rad[kRadial0 + k];
      const float qn = fmaf(t.x, r2, t.y) * qb + t.z * qa;
      qa = qb;
      qb = qn;
      const int pos = pos0 + k;
      if ((unsigned)pos < (unsigned)rows) {
        const float v = qn * cr, h = (v + kSplitStep) - kSplitStep;
        hi[pos] = __float2half_rn(h);
        lo[pos] = __float2half_rn(v - h);
      }
    }
    const float t = cr * fr - ci * fi;
    ci = cr * fi + ci * fr;
    cr = t;
    m = 4;
  }
  for (; m <= Np; m += 4) {
    const int pos0 = s_pos[m];
    const float4* tab = s_rad + (pos0 >> 1);
    // functions of this m within [r0, r0 + rows): k0 <= k < k1 (r0 and rows are even)
    const int cnt = ((Np - m) >> 1) + 1;
    const int k1 = min(cnt, (r0 + rows - pos0) >> 1), k0 = max(0, (r0 - pos0) >> 1);
    float qa = 0.f, qb = 1.f;
    if (k1 > k0) {
      for (int k = 0; k < k0; ++k) {
        const float4 t = tab[k];
        const float qn = fmaf(t.x, r2, t.y) * qb + t.z * qa;
        qa = qb;
        qb = qn;
      }
      __half* ph = hi + (pos0 - r0);
      __half* pl = lo + (pos0 - r0);
#pragma unroll 4
      for (int k = k0; k < k1; ++k) {
        const float4 t = tab[k];
        const float qn = fmaf(t.x, r2, t.y) * qb + t.z * qa;
        qa = qb;
        qb = qn;
        const float v0 = qn * cr, v1 = qn * ci;
        const float h0 = (v0 + kSplitStep) - kSplitStep, h1 = (v1 + kSplitStep) - kSplitStep;
        *reinterpret_cast<__half2*>(ph + 2 * k) = __floats2half2_rn(h0, h1);
        *reinterpret_cast<__half2*>(pl + 2 * k) = __floats2half2_rn(v0 - h0, v1 - h1);
      }
    }
    const float t = cr * fr - ci * fi;
    ci = cr * fi + ci * fr;
    cr = t;
  }
}

template <int TN>
__global__ void __launch_bounds__(32 * kWmWarps, 1)
assemble_wide_mma_kernel(const PairConst* __restrict__ pairs, const double* __restrict__ gl_x,
                         const double* __restrict__ gl_w, int q, float cos_max, float* __restrict__ vals,
                         int64_t row_stride, unsigned long long* __restrict__ node_count, int moment, WideMma G) {
  extern __shared__ __align__(16) __half stg[];  // [2][64][ldq] hi, lo; [2][64][ldp] hi, lo
  __shared__ PatchWarp P;
  __shared__ PairConst pc;
  __shared__ float s_x[kMaxQ], s_inv[2][2], s_w00[2];
  __shared__ float2 s_w[kMaxQ];
  __shared__ short s_idx[256];  // basis index of a staged position, -1 for the pad
  __shared__ short s_pos[geom::kWideMaxNp + 1];  // position of the first function of m
  __shared__ float4 s_rad[kRadial0 + geom::kWideMaxNp / 2 + 1];
  __shared__ int s_np;
  if (pairs[blockIdx.x].kind < 0) return;  // the whole block: no block for this pair in this part
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int qb = kWmNodes * G.ldq, pb = kWmNodes * G.ldp;  // halves of one part of one buffer
  __half* sq = stg;            // + buf 2 qb: hi, then lo
  __half* sp = stg + 4 * qb;   // + buf 2 pb
  if (tid < (int)(sizeof(PairConst) / 4)) reinterpret_cast<int*>(&pc)[tid] = reinterpret_cast<const int*>(pairs + blockIdx.x)[tid];
  if (tid < q) {
    s_x[tid] = (float)gl_x[tid];
    s_w[tid] = two_floats(gl_w[tid]);
  }
  if (tid < 256) s_idx[tid] = -1;
  __syncthreads();
  if (tid <= G.Np) {  // thread m writes the positions of its functions
    const int m = tid, c0 = G.Np / 2 + 1;
    int pos = m == 0 ? 0 : (c0 + 1) / 2 * 2;
    for (int k = 1; k < m; ++k) pos += 2 * ((G.Np - k) / 2 + 1);
    s_pos[m] = (short)pos;
    for (int n = m; n <= G.Np; n += 2) {
      // radial recurrence (zernike_wide.h): K1 Q_n = (K2 rho^2 + K3) Q_{n-2} + K4 Q_{n-4}
      float4 t = make_float4(0.f, 1.f, 0.f, 0.f);
      if (n == m + 2) t = make_float4((float)(m + 2), (float)(-(m + 1)), 0.f, 0.f);
      if (n > m + 2) {
        const float k1 = (float)((n + m) * (n - m) * (n - 2) / 2);
        t.x = (float)(2 * n * (n - 1) * (n - 2)) / k1;
        t.y = (float)(-m * m * (n - 1) - n * (n - 1) * (n - 2)) / k1;
        t.z = (float)(-n * (n + m - 2) * (n - m - 2) / 2) / k1;
      }
      s_rad[m == 0 ? kRadial0 + n / 2 : pos >> 1] = t;
      if (m == 0) {
        s_idx[pos++] = (short)(n * (n + 2) / 2);
      } else {
        s_idx[pos++] = (short)((n * (n + 2) + m) / 2);
        s_idx[pos++] = (short)((n * (n + 2) - m) / 2);
      }
    }
  }
  if (warp == 0) start_regions(P, pc, cos_max, lane);
  const int r0 = blockIdx.y * G.rows;
  const int wm = warp % G.WM, wn = warp / G.WM;
  const int NT = (G.total + 7) / 8;
  const int n0 = wn * TN, nn = wn < G.WN ? min(TN, NT - n0) : 0;  // this warp's column tiles
  const float mu = pc.mu, D3 = pc.D[2], area2 = 2.f * pc.area_src;
  const int kind = pc.kind, qq = q * q;
  float acc[TN][2][4];
#pragma unroll
  for (int n = 0; n < TN; ++n)
#pragma unroll
    for (int m = 0; m < 2; ++m) acc[n][m][0] = acc[n][m][1] = acc[n][m][2] = acc[n][m][3] = 0.f;
  unsigned long long pair_nodes = 0;
  float w00 = 0.f;  // this lane's part of entry (0, 0), the sum of the weights (of its half of the nodes)
  // stages pass `pass` of the chunk's nodes: warp 4 sub + part the functions of m =
  // sub mod 4, part 0 and 1 Z(p) of nodes 0..31 and 32..63, 2 and 3 w Z(p')
  auto evaluate = [&](int pass, int nodes) {
    const int part = warp & 3, sub = warp >> 2, half = part & 1, buf = pass & 1;
    const int kl = 32 * half + lane, k = pass * kWmNodes + kl;
    const int kc = min(k, nodes - 1);
    const int pi = kc / qq, rem = kc - pi * qq, i = rem / q, j = rem - i * q;
    RowConst rc;
    row_const(P.patch[pi], s_x[i], pc, rc);
    const RowNode g = row_node(rc, s_x[j], D3, kind, pc);
    if (part < 2) {
      __half* h = sp + buf * 2 * pb + kl * G.ldp;
      stage_zernike(G.Np, g.px.x, g.py.x, 1.f, sub, s_pos, s_rad, 0, 256, h, h + pb);
    } else {
      const float sk = moment == 0 ? phi2_row(mu * g.LO) : moment_factor(moment, mu, g.LO);
      const float w = k < nodes ? times(times(area2 * g.base * sk, s_w[i]), s_w[j]) : 0.f;
      w00 += w;
      // power of two that brings the 32 nodes' largest |w| into [1, 2)
      const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(w)));
      const unsigned ex = min(max(top >> 23, 1u), 253u);
      if (lane == 0 && sub == 0) s_inv[buf][half] = __uint_as_float(ex << 23);
      __half* h = sq + buf * 2 * qb + kl * G.ldq;
      stage_zernike(G.Np, g.px.y, g.py.y, w * __uint_as_float((254u - ex) << 23), sub, s_pos, s_rad, r0, G.rows, h, h + qb);
    }
  };
  const int arow = (lane & 7) + ((lane >> 4) << 3), acol = 32 * wm + (((lane >> 3) & 1) << 3);
  while (true) {
    __syncthreads();
    if (warp == 0) {
      const int np = fill_patches_warp(P, cos_max, lane);
      if (lane == 0) s_np = np;
    }
    __syncthreads();
    const int npatch = s_np;
    if (npatch == 0) break;
    const int nodes = npatch * qq, passes = (nodes + kWmNodes - 1) / kWmNodes;
    pair_nodes += nodes;
    evaluate(0, nodes);
    __syncthreads();
    for (int pass = 0; pass < passes; ++pass) {
      if (pass + 1 < passes) evaluate(pass + 1, nodes);
      const int buf = pass & 1;
      if (nn > 0) {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const __half* qh = sq + buf * 2 * qb + 32 * h * G.ldq;
          const __half* ph = sp + buf * 2 * pb + (32 * h + lane) * G.ldp + 8 * n0;
          const float inv = s_inv[buf][h];
          uint32_t ah[2][2][4], al[2][2][4];
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
              const int o = (16 * ks + arow) * G.ldq + 16 * m + acol;
              ldsm4_trans(ah[m][ks], qh + o);
              ldsm4_trans(al[m][ks], qh + qb + o);
            }
#pragma unroll
          for (int n = 0; n < TN; ++n) {
            if (n < nn) {
              uint32_t bh[4], bl[4];
              ldsm4_trans(bh, ph + 8 * n);
              ldsm4_trans(bl, ph + pb + 8 * n);
              uint32_t bs[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) bs[i] = add_half2(bh[i], bl[i]);
#pragma unroll
              for (int m = 0; m < 2; ++m) {
                float t[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                  mma_f16(t, ah[m][ks], bh[2 * ks], bh[2 * ks + 1]);
                  mma_f16(u, al[m][ks], bs[2 * ks], bs[2 * ks + 1]);
                  mma_f16(u, ah[m][ks], bl[2 * ks], bl[2 * ks + 1]);
                }
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                  const float2 v = __fadd2_rn(pair(u[e], u[e + 1]), pair(t[e], t[e + 1]));
                  const float2 s = fma2(v, pair(inv, inv), pair(acc[n][m][e], acc[n][m][e + 1]));
                  acc[n][m][e] = s.x;
                  acc[n][m][e + 1] = s.y;
                }
              }
            }
          }
        }
      }
      __syncthreads();
    }
  }
  if (tid == 0 && blockIdx.y == 0) atomicAdd(node_count, pair_nodes);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) w00 += __shfl_xor_sync(0xffffffffu, w00, o);
  if (lane == 0 && (warp == 2 || warp == 3)) s_w00[warp - 2] = w00;  // parts 2 and 3, the weights of either half
  __syncthreads();
  // epilogue: basis order, row i scaled by lambda N_i / sqrt(|T_l||T_l'|)
  float* out = vals + (int64_t)pc.out_row * row_stride + (int64_t)pc.slot * G.nb * G.nb;
  const int g8 = lane >> 2, t4 = lane & 3;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int r = r0 + 32 * wm + 16 * m + g8 + 8 * hh;
      const int a = r < 256 ? s_idx[r] : -1;
      if (a < 0) continue;
      const float s = (float)((double)pc.scale * zernike_invnorm(a));
#pragma unroll
      for (int n = 0; n < TN; ++n)
        if (n < nn)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int b = s_idx[8 * (n0 + n) + 2 * t4 + e];
            if (b >= 0) out[(int64_t)a * G.nb + b] = (a + b == 0 ? s_w00[0] + s_w00[1] : acc[n][m][2 * hh + e]) * s;
          }
    }
}

int launch_assemble_wide_mma(int Np, const PairConst* pairs, int64_t npairs, const double* glx, const double* glw,
                             int q, float cos_max, float* vals, int64_t row_stride, unsigned long long* nodes,
                             int moment, cudaStream_t st) {
  const WideMma g = geom::wide_mma_geometry(Np);
  if (g.TN < 2 || g.TN > geom::kWideMmaMaxTn || g.smem > 222 * 1024)
    return set_error(DFM_ERR_UNSUPPORTED, "dfm_assemble: wide assembly tile does not fit a block");
  auto go = [&](auto kernel) -> int {
    DFM_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem));
    {
      ::dfm::KernelTimer timer_(DFM_KERNEL_ASSEMBLE, st);
      kernel<<<dim3((unsigned)npairs, (unsigned)g.ntile), 32 * kWmWarps, g.smem, st>>>(
          pairs, glx, glw, q, cos_max, vals, row_stride, nodes, moment, g);
    }
    DFM_LAUNCHED();
    DFM_CUDA_CHECK(cudaGetLastError());
    return DFM_OK;
  };
  switch (g.TN) {
    case 2: return go(assemble_wide_mma_kernel<2>);
    case 3: return go(assemble_wide_mma_kernel<3>);
    case 4: return go(assemble_wide_mma_kernel<4>);
    case 5: return go(assemble_wide_mma_kernel<5>);
    case 6: return go(assemble_wide_mma_kernel<6>);
    case 7: return go(assemble_wide_mma_kernel<7>);
    default: return go(assemble_wide_mma_kernel<8>);
  }
}

}  // namespace
}  // namespace dfm
