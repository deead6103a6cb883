// FP32 assembly of the operator blocks (N_p <= 8) with the block sums on
// tensor cores.  Included by assemble.cu.
//
// One warp per face pair.  Lanes evaluate one quadrature node each (row by
// row, row_node.cuh); the block is the sum over nodes of w Z(p') Z(p)^T, an
// N_b x N_b product over some 1,400 (N_p = 4) to 2,700 (N_p = 8) nodes.  Per pass of
// 32 nodes each staged value x is split into two FP16 parts x = hi + lo and the
// pass's product is three mma.sync m16n8k16 products, hi hi, lo (hi + lo) and hi lo,
// started at zero and added to the FP32 sums on the CUDA cores.
//
// The tensor cores round their sums towards zero, which would make every entry
// too small by a common factor, and a solve at little damping magnifies such a
// loss some hundred times.  So hi hi is made exact: hi is a multiple of 2^-9,
// |Z(p)| <= 1, and the weights of a pass are scaled by a power of two to a maximum
// in [1, 2), so |w Z(p')| < 2.  All products are then multiples of 2^-18, and 32 of
// them add up to at most 2^6 = 2^24 such units, which FP32 holds without
// rounding.  The other two products have sums of their own, 2^-9 of it, and so has
// their loss.  lo is rounded to nearest at 2^-22 at most, so a staged value is
// exact to 2^-22 of its pass's largest (not of itself).  The scale is taken out by
// the FMA that adds the pass.  Entry (0, 0), the one such a solve hangs on, is the
// sum of the weights, and is added up lane by lane beside the products: 32 sums of
// some 45 terms lose less to rounding than one.
//
// Measured (GB300): 48,000 tets at N_p = 4 in 10.5 ms against 23.8 ms for the
// rank-1 form on CUDA cores, 24,576 tets at N_p = 8 in 37.0 against 87.0 ms; error
// against 64 bits (2-norm, 1,296 and 384 tets) 2.4e-7 against 5.7e-7 at N_p = 4,
// 4.3e-7 against 8.3e-7 at N_p = 8.  (Parts split relative to each value, hi hi not
// exact: 10.2 and 35.7 ms, every entry 7e-8 too small.)
// What bounds it: issue and the FP32, ALU and shared-memory pipes together at
// N_p = 4; at N_p = 8 the latency of the MMA chains (108 MMAs of 8 cycles in a pass
// of some 1,800), with 255 registers and 8 warps per SM.  N_p = 7 likewise: 11.8
// ms at 10,368 tets, 12.4 ms with 168 registers and 12 warps.  More warps at
// N_p <= 4 gain nothing (24 per SM: 10.5 ms).
#pragma once

#include <algorithm>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "row_node.cuh"

namespace dfm {
namespace {

template <int NP>
struct MmaTile {
  static constexpr int NB = (NP + 1) * (NP + 2) / 2;
  static constexpr int MT = (NB + 15) / 16;  // 16-row tiles of test functions
  static constexpr int NT = (NB + 7) / 8;    // 8-column tiles of trial functions
  // staged halves per node: the MMA tiles' width, a row stride of an odd
  // number of 16-byte units (ldmatrix and the 16-byte stores then touch
  // distinct bank groups)
  static constexpr int W = MT * 16;
  static constexpr int LD = W / 8 % 2 ? W : W + 8;
};

// Shared memory of one warp.
template <int NP>
struct MmaWarp {
  PatchWarp P;
  PairConst pc;
  // Z(p') times the scaled weight, and Z(p): hi and lo parts, one row per node
  alignas(16) __half qh[32 * MmaTile<NP>::LD];
  alignas(16) __half ql[32 * MmaTile<NP>::LD];
  alignas(16) __half ph[32 * MmaTile<NP>::LD];
  alignas(16) __half pl[32 * MmaTile<NP>::LD];
};

// x + kSplitStep - kSplitStep is x rounded to a multiple of 2^-9 (|x| <= 2): FP32
// has units of 2^-9 between 2^14 and 2^15, of which this is the middle
constexpr float kSplitStep = 24576.f;

// hi and lo FP16 parts of the values v[0..NB) of a node (x: Z(p), y: w Z(p');
// zero up to a multiple of 8) into its four staged rows.  What the last m-tile
// reads beyond that is left as it is: it reaches only block rows past N_b.
template <int NB>
__device__ __forceinline__ void stage_split(__half* ph, __half* pl, __half* qh, __half* ql, const float2* v) {
  const float2 minus = pair(-1.f, -1.f), step = pair(kSplitStep, kSplitStep), back = pair(-kSplitStep, -kSplitStep);
  auto bits = [](__half2 h) { return reinterpret_cast<const uint32_t&>(h); };
#pragma unroll
  for (int u = 0; u < (NB + 7) / 8; ++u) {
    uint32_t h0[4], l0[4], h1[4], l1[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int b = 8 * u + 2 * e;
      if (b >= NB) {
        h0[e] = l0[e] = h1[e] = l1[e] = 0u;
        continue;
      }
      const float2 s = v[b], t = b + 1 < NB ? v[b + 1 < NB ? b + 1 : b] : pair(0.f, 0.f);
      const float2 hs = __fadd2_rn(__fadd2_rn(s, step), back), ht = __fadd2_rn(__fadd2_rn(t, step), back);
      const float2 ds = fma2(hs, minus, s), dt = fma2(ht, minus, t);
      h0[e] = bits(__floats2half2_rn(hs.x, ht.x));
      h1[e] = bits(__floats2half2_rn(hs.y, ht.y));
      l0[e] = bits(__floats2half2_rn(ds.x, dt.x));
      l1[e] = bits(__floats2half2_rn(ds.y, dt.y));
    }
    *reinterpret_cast<uint4*>(ph + 8 * u) = make_uint4(h0[0], h0[1], h0[2], h0[3]);
    *reinterpret_cast<uint4*>(pl + 8 * u) = make_uint4(l0[0], l0[1], l0[2], l0[3]);
    *reinterpret_cast<uint4*>(qh + 8 * u) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
    *reinterpret_cast<uint4*>(ql + 8 * u) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
  }
}

__device__ __forceinline__ void ldsm4_trans(uint32_t r[4], const __half* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p))
               : "memory");
}

__device__ __forceinline__ void mma_f16(float d[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t add_half2(uint32_t a, uint32_t b) {
  const __half2 v = __hadd2(reinterpret_cast<const __half2&>(a), reinterpret_cast<const __half2&>(b));
  return reinterpret_cast<const uint32_t&>(v);
}

// acc += inv * (staged Z(p'))^T (staged Z(p)) over the 32 nodes of a pass.
// ldmatrix.trans of the node-major rows gives both operands: the A fragment
// of (m-tile, 16 nodes) from four 8 x 8 pieces, and the B fragments of both
// 16-node halves of an n-tile from one instruction.  With hi + lo of Z(p) in FP16
// as the other factor of the first of the two mixed products, lo lo is in it too.
// An m-tile's two sums side by side, or with three m-tiles one after the other
// over all of them, keep the fewest registers: 6.3 against 6.5 ms (10,368
// tets, N_p = 6) and 36.7 against 38.8 ms (24,576 tets, N_p = 8) the other way round.
template <int NP>
__device__ __forceinline__ void pass_product(const MmaWarp<NP>& S, int lane, float inv,
                                             float (&acc)[MmaTile<NP>::NT][MmaTile<NP>::MT][4]) {
  using TL = MmaTile<NP>;
  constexpr int MT = TL::MT, NT = TL::NT, LD = TL::LD;
  uint32_t ah[MT][2][4], al[MT][2][4];
  // pieces (nodes 0-7, m 0-7), (nodes 0-7, m 8-15), (nodes 8-15, m 0-7), (nodes 8-15, m 8-15)
  const int arow = (lane & 7) + ((lane >> 4) << 3), acol = ((lane >> 3) & 1) << 3;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      const int o = (16 * ks + arow) * LD + 16 * mt + acol;
      ldsm4_trans(ah[mt][ks], S.qh + o);
      ldsm4_trans(al[mt][ks], S.ql + o);
    }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    uint32_t bh[4], bl[4], bs[4];  // (nodes 0-7, 8-15, 16-23, 24-31) x 8 columns
    ldsm4_trans(bh, S.ph + lane * LD + 8 * nt);
    ldsm4_trans(bl, S.pl + lane * LD + 8 * nt);
#pragma unroll
    for (int i = 0; i < 4; ++i) bs[i] = add_half2(bh[i], bl[i]);
    auto add = [&](int mt, float2 u0, float2 u1) {
      float* a = acc[nt][mt];
      u0 = fma2(u0, pair(inv, inv), pair(a[0], a[1]));
      u1 = fma2(u1, pair(inv, inv), pair(a[2], a[3]));
      a[0] = u0.x, a[1] = u0.y, a[2] = u1.x, a[3] = u1.y;
    };
    if constexpr (MT <= 2) {
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        float t[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          mma_f16(t, ah[mt][ks], bh[2 * ks], bh[2 * ks + 1]);
          mma_f16(u, al[mt][ks], bs[2 * ks], bs[2 * ks + 1]);
          mma_f16(u, ah[mt][ks], bl[2 * ks], bl[2 * ks + 1]);
        }
        add(mt, __fadd2_rn(pair(u[0], u[1]), pair(t[0], t[1])), __fadd2_rn(pair(u[2], u[3]), pair(t[2], t[3])));
      }
    } else {
      float t[MT][4];
      auto start = [&]() {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) t[mt][0] = t[mt][1] = t[mt][2] = t[mt][3] = 0.f;
      };
      auto product = [&](const uint32_t (&a)[MT][2][4], const uint32_t (&b)[4]) {
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) mma_f16(t[mt], a[mt][ks], b[2 * ks], b[2 * ks + 1]);
      };
      auto finish = [&]() {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) add(mt, pair(t[mt][0], t[mt][1]), pair(t[mt][2], t[mt][3]));
      };
      start();
      product(ah, bh);
      finish();
      start();
      product(al, bs);
      product(ah, bl);
      finish();
    }
  }
}

// moment k: L_O^k phi2^(k)(mu L_O).  A call of its own: inlined, its Gauss rule
// would take the registers of every assembly.
__device__ __noinline__ float moment_factor(int moment, float mu, float LO) {
  float sk = phi2_deriv<float>(moment, mu * LO);
  for (int e = 0; e < moment; ++e) sk *= LO;
  return sk;
}

template <int NP, typename TO>
__global__ void __launch_bounds__(kWarps * 32, NP >= 7 ? 2 : (NP >= 5 ? 4 : 5))
assemble_mma_kernel(const PairConst* __restrict__ pairs, int64_t npairs, const double* __restrict__ gl_x,
                    const double* __restrict__ gl_w, int q, float cos_max, TO* __restrict__ vals, int64_t row_stride,
                    unsigned long long* __restrict__ node_count, unsigned long long* __restrict__ counter, int moment) {
  using TL = MmaTile<NP>;
  constexpr int NB = TL::NB, MT = TL::MT, NT = TL::NT, LD = TL::LD;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  MmaWarp<NP>* smem = reinterpret_cast<MmaWarp<NP>*>(dyn_smem);
  float* s_x = reinterpret_cast<float*>(smem + kWarps);
  float2* s_w = reinterpret_cast<float2*>(s_x + kMaxQ);
  float2* s_ninv = s_w + kMaxQ;
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;
  MmaWarp<NP>& S = smem[wid];
  if (threadIdx.x < q) {
    s_x[threadIdx.x] = (float)gl_x[threadIdx.x];
    s_w[threadIdx.x] = two_floats(gl_w[threadIdx.x]);
  }
  if (threadIdx.x < NB) s_ninv[threadIdx.x] = two_floats(zernike_invnorm(threadIdx.x));
  __syncthreads();
  const int g8 = lane >> 2, t4 = lane & 3;
  const float qinv = 1.f / (float)q;
  unsigned long long my_nodes = 0;
  // resident warps take pairs off a shared counter, the next one fetched while
  // this one runs: pairs differ in patch count, and the Gauss table and norms
  // above are set up once per block
  unsigned long long p = (unsigned long long)blockIdx.x * kWarps + wid;
  while (p < (unsigned long long)npairs) {
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(counter, 1ull) + (unsigned long long)gridDim.x * kWarps;
    for (int i = lane; i < (int)(sizeof(PairConst) / 4); i += 32)
      reinterpret_cast<int*>(&S.pc)[i] = reinterpret_cast<const int*>(pairs + p)[i];
    __syncwarp();
    const int kind = S.pc.kind;
    if (kind >= 0) {  // else no block for this pair in this part
      float acc[NT][MT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) acc[nt][mt][0] = acc[nt][mt][1] = acc[nt][mt][2] = acc[nt][mt][3] = 0.f;
      float w00 = 0.f;  // this lane's part of entry (0, 0)
      start_regions(S.P, S.pc, cos_max, lane);
      const float mu = S.pc.mu, D3 = S.pc.D[2], area2 = 2.f * S.pc.area_src;
      while (true) {
        const int npatch = fill_patches_warp(S.P, cos_max, lane);
        if (npatch == 0) break;
        const int rows = npatch * q;
        my_nodes += (unsigned long long)(rows * q);
        for (int base = 0; base < rows;) {
          const RowPass ps = next_pass(rows - base);
          const int rl = lane / ps.per;
          const bool live = rl < ps.rows;
          const int row = base + (live ? rl : ps.rows - 1);
          const int pi = (int)(((float)row + 0.5f) * qinv), i = row - pi * q;  // exact: row < 20 x 32
          RowConst rc;
          row_const(S.P.patch[pi], s_x[i], S.pc, rc);
          const float wi = live ? times(area2, s_w[i]) : 0.f;
          base += ps.rows;
          for (int j0 = 0; j0 < q; j0 += ps.per) {
            const int j = j0 + (lane - rl * ps.per);
            const bool on = j < q;
            const int jc = on ? j : q - 1;
            const RowNode g = row_node(rc, s_x[jc], D3, kind, S.pc);
            const float sk = moment == 0 ? phi2_row(mu * g.LO) : moment_factor(moment, mu, g.LO);
            const float w = on ? times(wi * g.base * sk, s_w[jc]) : 0.f;
            w00 += w;
            // power of two that brings the pass's largest |w| into [1, 2)
            const unsigned top = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(w)));
            const unsigned ex = min(max(top >> 23, 1u), 253u);
            const float scale = __uint_as_float((254u - ex) << 23), inv = __uint_as_float(ex << 23);
            float2 Z[NB];
            zernike2<NP>(g.px, g.py, pair(1.f, w * scale), Z);
            stage_split<NB>(S.ph + lane * LD, S.pl + lane * LD, S.qh + lane * LD, S.ql + lane * LD, Z);
            __syncwarp();
            pass_product<NP>(S, lane, inv, acc);
            __syncwarp();
          }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w00 += __shfl_xor_sync(0xffffffffu, w00, o);
      if (lane == 0) acc[0][0][0] = w00;
      // epilogue: scale row a by lambda N_a / sqrt(|T_l||T_l'|) and store
      TO* out = vals + (int64_t)S.pc.out_row * row_stride + (int64_t)S.pc.slot * NB * NB;
      const float sp = S.pc.scale;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int a = 16 * mt + g8 + 8 * h;
          if (a >= NB) continue;
          const float s = times(sp, s_ninv[a]);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int b = 8 * nt + 2 * t4 + e;
              if (b >= NB) continue;
              const float v = acc[nt][mt][2 * h + e] * s;
              if constexpr (std::is_same<TO, __nv_bfloat16>::value)
                out[a * NB + b] = __float2bfloat16_rn(v);
              else
                out[a * NB + b] = v;
            }
        }
    }
    p = __shfl_sync(0xffffffffu, next, 0);
    __syncwarp();  // the pair's constants are read before the next ones arrive
  }
  if (lane == 0 && my_nodes) atomicAdd(node_count, my_nodes);
}

template <int NP, typename TO>
int launch_assemble_mma(const PairConst* pairs, int64_t npairs, const double* glx, const double* glw, int q,
                        float cos_max, TO* vals, int64_t row_stride, unsigned long long* nodes, int moment,
                        cudaStream_t st) {
  constexpr size_t smem = sizeof(MmaWarp<NP>) * kWarps + (3 * kMaxQ + 2 * 64) * sizeof(float);
  static_assert(smem <= 220 * 1024, "assembly shared memory");
  static_assert(sizeof(MmaWarp<NP>) % 16 == 0, "16-byte aligned staging rows");
  DFM_CUDA_CHECK(
      cudaFuncSetAttribute(assemble_mma_kernel<NP, TO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int dev = 0, nsm = 0, per_sm = 0;
  DFM_CUDA_CHECK(cudaGetDevice(&dev));
  DFM_CUDA_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  DFM_CUDA_CHECK(
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, assemble_mma_kernel<NP, TO>, kWarps * 32, smem));
  const int64_t blocks = std::min<int64_t>((npairs + kWarps - 1) / kWarps, (int64_t)nsm * std::max(per_sm, 1));
  unsigned long long* counter = nodes + 1;
  DFM_CUDA_CHECK(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st));
  {
    ::dfm::KernelTimer timer_(DFM_KERNEL_ASSEMBLE, st);
    assemble_mma_kernel<NP, TO><<<(unsigned)blocks, kWarps * 32, smem, st>>>(pairs, npairs, glx, glw, q, cos_max, vals,
                                                                             row_stride, nodes, counter, moment);
  }
  DFM_LAUNCHED();
  DFM_CUDA_CHECK(cudaGetLastError());
  return DFM_OK;
}

}  // namespace
}  // namespace dfm
