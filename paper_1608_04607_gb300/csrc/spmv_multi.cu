// Forward application y = x0 + alpha sum_k coef_k B_k x of FP32 operators to
// FP32 right-hand sides on tensor cores: the block Krylov operator of the
// many-source solves, the damping moments of the per-source ones, and single
// vectors of the larger bases.
//
// Per operator row the product is Y (NB x R) = sum over operators and the row's
// three blocks of B X, a dense contraction.  Every FP32 operand is split into
// two TF32 parts (hi, lo, 11 significant bits each), in three mma.sync m16n8k8
// products, lo hi + hi lo + hi hi; lo lo, at most 2^-23 of the product, is left out.
// A solve magnifies what all results lose in common, so nothing here is rounded one
// way more than once: x's hi part is rounded to nearest (with both chopped, lo lo is
// positive wherever the product is: 1.5e-7 of it lost on average), and the tensor
// cores, which round towards zero, add up eight hi hi products from zero, the rest
// being added on the CUDA cores (chains over a block: another 2e-7 at 45 functions).
// One truncation is left, 4.3e-8 on average at most; results are measured 8e-9 off in
// common, 1e-7 (3 functions) to 2.7e-7 (45) with hi chopped and block-long chains,
// at the same times: 494 against 521 us for 16 right-hand sides (24,576 tets, 45
// functions), 111 against 104 us for one (16,464 tets, 28 functions).
//
// Work is taken by source tet: the four rows that tet t sends to (recv[4t + l'],
// one contiguous row of each operator) read the same 4 NB coefficients of every
// right-hand side, so these are fetched once for four rows.  Producer warps
// (tet j of the block to producer j mod P) stream tets through a ring, four row
// stages and one coefficient slot each, by bulk copies (TMA); a consumer warp
// owns one 16-row tile of test functions of one row of every G-th tet.  The
// ring's depth is a multiple of P and of G, so every barrier's previous phase
// was consumed by the very warps that wait for it (no phase is ever read two
// behind).  Waits are bounded; a time-out sets the operator's error flag.
//
// HBM bounds it where enough bytes are in flight (about 110 KB per SM at 2.5 us
// under load), so one block per SM takes all of its shared memory.  One producer
// warp spends 0.7 us per tet plus 30 ns per copy, more than the small bases' rows
// take to arrive, hence up to four; and a row is spread over its m-tiles because
// with one warp per row the two-tet ring of the large bases had no stage left to
// fill ahead while it was being consumed.
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "dfm_internal.cuh"
#include "tma_pipe.cuh"

namespace dfm {
namespace {

using namespace pipe;

// ring and warps: launch_geometry.h (shared with a host-side check)
constexpr int kMaxOps = geom::kMultiMaxOps, kMaxRhs = geom::kMultiMaxRhs, kMaxD = geom::kMultiMaxDepth;
constexpr int kHead = geom::kMultiHead, kMaxProducers = geom::kMultiMaxProducers;
using geom::multi_max_groups;
using geom::multi_m_tiles;
using geom::multi_slot_stride;
static_assert(10 * kMaxD * 8 <= kHead, "barriers");

struct Ops {
  const float* vals[kMaxOps];
  float coef[kMaxRhs][kMaxOps];
};

// An operator entry: hi its top 11 significant bits, lo the rest (exact, 13 bits)
// plus half a unit of TF32's last place, which the multiplier's own truncation to
// TF32 turns into rounding to nearest.  Three instructions (cvt.rna twice takes
// five).
__device__ __forceinline__ void split_entry(float x, uint32_t& hi, uint32_t& lo) {
  hi = __float_as_uint(x) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi)) + 0x1000u;
}
// A coefficient: hi rounded to 11 significant bits, lo the rest (exact, 12 bits and
// its sign).  What is not finite, or rounds to infinity, gives a result that is not
// finite.
__device__ __forceinline__ void split_coefficient(float x, uint32_t& hi, uint32_t& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}

// d += A B, or d = A B
__device__ __forceinline__ void mma_tf32_k8(float d[4], const uint32_t a[4], const uint32_t b[2]) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void mma_tf32_k8_first(float d[4], const uint32_t a[4], const uint32_t b[2]) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
}

// s += t, two elements per instruction
__device__ __forceinline__ void add4(float (&s)[4], const float (&t)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    const float2 v = __fadd2_rn(make_float2(s[e], s[e + 1]), make_float2(t[e], t[e + 1]));
    s[e] = v.x;
    s[e + 1] = v.y;
  }
}

// One output in FP32 FMAs: rows `blk` (a row of the three blocks of K operators
// `stride` apart) times the coefficients x, the exit face's left out, times the operators'
// weights.  The split parts of an infinite coefficient cancel, so outputs that are
// not finite are formed again as written.
__device__ __noinline__ float plain_output(const float* blk, int64_t stride, int nb, int K, const float* x, int exit_face,
                                           const float* weight) {
  float s = 0.f;
  for (int k = 0; k < K; ++k)
    for (int f = 0; f < 3; ++f)
      for (int b = 0; b < nb; ++b) {
        const float v = x[(f + (f >= exit_face ? 1 : 0)) * nb + b];
        s = fmaf(blk[k * stride + f * nb * nb + b], weight ? v * weight[k] : v, s);
      }
  return s;
}

// COMBO: K operators with per-right-hand-side weights; else one, weight 1
template <int NB, int NT, bool COMBO>
__global__ void __launch_bounds__(32 * (kMaxProducers + 4 * multi_m_tiles(NB) * multi_max_groups(NB)), 1)
spmv_multi_kernel(const __grid_constant__ Ops ops, int K, int64_t row_stride, const int32_t* __restrict__ recv,
                  int nt, int64_t nrows, const float* __restrict__ x, const float* x0, float* y, int R,
                  float alpha, int P, int G, int logD, int logX, int reverse, int keep_from, int* __restrict__ err) {
  constexpr int MT = multi_m_tiles(NB), KK = (NB + 7) / 8, XS = multi_slot_stride(NB);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw);
  uint64_t* empty = full + 4 * kMaxD;
  uint64_t* xfull = empty + 4 * kMaxD;
  uint64_t* xempty = xfull + kMaxD;
  float* stage0 = reinterpret_cast<float*>(smem_raw + kHead);
  const int NX = 1 << logX, S = 4 << logD, logS = logD + 2;
  const int stage_f = K * (int)row_stride;  // floats per row stage
  float* slot0 = stage0 + S * stage_f;
  const int slot_f = R * XS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], MT);  // the row's m-tiles
    }
    for (int s = 0; s < NX; ++s) {
      mbar_init(&xfull[s], 1);
      mbar_init(&xempty[s], 4 * MT);  // the four rows of a tet
    }
    mbar_init_fence();
  }
  __syncthreads();
  // tets and rows of this block are counted in 32 bits (rows < 2^31 in all)
  const int mine = nt > blockIdx.x ? (nt - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  auto tet_of = [&](int j) -> int64_t {
    const int q = blockIdx.x + j * (int)gridDim.x;
    return reverse ? nt - 1 - q : q;
  };
  if (warp < P) {
    // ---------------- producers ----------------
    const uint64_t pol_last = l2_policy_evict_last(), pol_first = l2_policy_evict_first();
    const unsigned xb = 4 * NB * 4, vb = (unsigned)(row_stride * 4);
    // lanes 0..3 own the four rows of a tet (their stage's barriers and copies),
    // lanes 0..R-1 one right-hand side's coefficients each: issued row after row
    // by one lane, the waits and copies of a tet cost four times as long
    bool ok = true;
    int last = -1;  // last tet issued
    const int lp = lane & 3;
    // the row map of eight of this warp's tets at a time (lane: tet lane / 4, face
    // lane % 4), one batch ahead of their use
    auto load_map = [&](int u0) -> int32_t {
      const int j = warp + (u0 + (lane >> 2)) * P;
      return j < mine ? recv[4 * tet_of(j) + lp] : 0;
    };
    int32_t map = load_map(0), next_map = load_map(8);
    for (int j = warp, u = 0; j < mine; j += P, ++u) {
      const int64_t t = tet_of(j);
      if (u && !(u & 7)) {
        map = next_map;
        next_map = load_map(u + 8);
      }
      const int64_t row = __shfl_sync(0xffffffffu, map, 4 * (u & 7) + lp);
      const int i = 4 * j + lp, s = i & (S - 1), xs = j & (NX - 1);
      if (lane < 4 && i >= S) ok = mbar_wait_bounded(&empty[s], (unsigned)(((i >> logS) - 1) & 1));
      if (j >= NX) ok = mbar_wait_bounded(&xempty[xs], (unsigned)(((j >> logX) - 1) & 1)) && ok;
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      if (lane == 0) mbar_arrive_expect_tx(&xfull[xs], R * xb);
      __syncwarp();
      if (lane < R)
        bulk_copy_g2s(slot0 + xs * slot_f + lane * XS, x + ((int64_t)lane * nrows + 4 * t) * NB, xb, &xfull[xs]);
      if (lane < 4) {
        const uint64_t pol = (int)blockIdx.x + j * (int)gridDim.x >= keep_from ? pol_last : pol_first;
        mbar_arrive_expect_tx(&full[s], (unsigned)K * vb);
        for (int k = 0; k < K; ++k)
          bulk_copy_g2s_hint(stage0 + s * stage_f + k * (int)row_stride, ops.vals[k] + row * row_stride, vb, &full[s], pol);
      }
      last = j;
    }
    if (!ok && lane == 0) atomicOr(err, 1);
    // drain: this warp's issued copies must have landed before the block's shared
    // memory goes away (earlier tets of a stage landed before it was reused)
    if (lane == 0)
      for (int j = last; j >= 0 && j > last - NX; j -= P) {
        mbar_wait_bounded(&xfull[j & (NX - 1)], (unsigned)((j >> logX) & 1));
        for (int i = 4 * j; i < 4 * j + 4; ++i)
          if (i > 4 * last + 3 - S) mbar_wait_bounded(&full[i & (S - 1)], (unsigned)((i >> logS) & 1));
      }
    return;
  }
  // ---------------- consumers ----------------
  const int c = warp - P;
  const int g = lane >> 2, t4 = lane & 3;
  const int a0 = 16 * (c % MT) + g, lp = (c / MT) & 3;  // test functions a0, a0 + 8 of the row across face lp
  int j = c / (4 * MT);
  int32_t next_row = j < mine ? recv[4 * tet_of(j) + lp] : 0;
  for (; j < mine; j += G) {
    const int i = 4 * j + lp;
    const int s = i & (S - 1), xs = j & (NX - 1);
    const int64_t row = next_row;
    if (j + G < mine) next_row = recv[4 * tet_of(j + G) + lp];
    // x0 of this lane's outputs, ahead of the wait and the products
    float base[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int a = a0 + (e & 2 ? 8 : 0), r = 8 * n + 2 * t4 + (e & 1);
        base[n][e] = (x0 && a < NB && r < R) ? x0[((int64_t)r * nrows + row) * NB + a] : 0.f;
      }
    bool ok = mbar_wait_bounded(&full[s], (unsigned)((i >> logS) & 1));
    ok = ok && mbar_wait_bounded(&xfull[xs], (unsigned)((j >> logX) & 1));
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) {
      if (lane == 0) atomicOr(err, 1);
      break;
    }
    const float* xq[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n)  // columns past R repeat the last one; they are not stored
      xq[n] = slot0 + xs * slot_f + min(8 * n + g, R - 1) * XS + t4;
    float acc[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
    const int nops = COMBO ? K : 1;
    for (int k = 0; k < nops; ++k) {
      float cf[NT];
#pragma unroll
      for (int n = 0; n < NT; ++n) cf[n] = COMBO ? ops.coef[min(8 * n + g, R - 1)][k] : 1.f;
      const float* vals = stage0 + s * stage_f + k * (int)row_stride + a0 * NB + t4;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const int l = f + (f >= lp ? 1 : 0);
        const float* blk = vals + f * NB * NB;
        float tl[NT][4];
#pragma unroll
        for (int kk = 0; kk < KK; ++kk) {
          // this lane's contraction indices 8 kk + t4 and 8 kk + t4 + 4; beyond
          // NB both operands are zero (what follows a block in memory is not)
          const bool in0 = 8 * kk + 3 < NB || 8 * kk + t4 < NB, in1 = 8 * kk + 7 < NB || 8 * kk + t4 + 4 < NB;
          const float* p = blk + 8 * kk;
          const float v[4] = {in0 ? p[0] : 0.f, in0 ? p[8 * NB] : 0.f, in1 ? p[4] : 0.f, in1 ? p[8 * NB + 4] : 0.f};
          uint32_t ah[4], al[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) split_entry(v[e], ah[e], al[e]);
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            float u0 = in0 ? xq[n][l * NB + 8 * kk] : 0.f, u1 = in1 ? xq[n][l * NB + 8 * kk + 4] : 0.f;
            if (COMBO) {
              u0 *= cf[n];
              u1 *= cf[n];
            }
            uint32_t xh[2], xl[2];
            split_coefficient(u0, xh[0], xl[0]);
            split_coefficient(u1, xh[1], xl[1]);
            float th[4];
            mma_tf32_k8_first(th, ah, xh);
            if (kk == 0) mma_tf32_k8_first(tl[n], al, xh);
            else mma_tf32_k8(tl[n], al, xh);
            mma_tf32_k8(tl[n], ah, xl);
            add4(acc[n], th);
          }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) add4(acc[n], tl[n]);
      }
    }
    float zero = 0.f;  // NaN if an output is not finite
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) zero = fmaf(acc[n][e], 0.f, zero);
    if (zero != 0.f) {
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int a = a0 + (e & 2 ? 8 : 0), r = 8 * n + 2 * t4 + (e & 1);
          if (a < NB && r < R && !(fabsf(acc[n][e]) <= 3.402823466e38f))
            acc[n][e] = plain_output(stage0 + s * stage_f + a * NB, row_stride, NB, nops,
                                     slot0 + xs * slot_f + r * XS, lp, COMBO ? ops.coef[r] : nullptr);
        }
    }
    __syncwarp();  // the row's stage and the tet's slot are read
    if (lane == 0) {
      mbar_arrive(&empty[s]);
      mbar_arrive(&xempty[xs]);
    }
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int a = a0 + (e & 2 ? 8 : 0), r = 8 * n + 2 * t4 + (e & 1);
        if (a < NB && r < R) y[((int64_t)r * nrows + row) * NB + a] = fmaf(alpha, acc[n][e], base[n][e]);
      }
  }
}

template <int NB>
int launch_multi(const dfm_op* op, const Ops& ops, int K, bool combo, const float* x, const float* x0, float* y,
                 int R, float alpha, const geom::Multi& g, cudaStream_t st) {
  int dev = 0, nsm = 0;
  DFM_CUDA_CHECK(cudaGetDevice(&dev));
  DFM_CUDA_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  if (op->nrows >= int64_t(1) << 31) return set_error(DFM_ERR_UNSUPPORTED, "dfm_apply: too many rows");
  const int nt = (int)(op->nrows / 4);
  auto go = [&](auto kernel) -> int {
    DFM_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem));
    const int grid = std::min(nt, nsm), threads = 32 * (g.producers + 4 * multi_m_tiles(NB) * g.groups);
    // operator bytes kept in L2 for the next application, which sweeps the other way (as in spmv.cu)
    const int keep = (int)std::max<int64_t>(0, nt - (64ll << 20) / (4 * K * op->row_stride * 4));
    {
      ::dfm::KernelTimer timer_(DFM_KERNEL_SPMV, st);
      kernel<<<(unsigned)grid, threads, g.smem, st>>>(ops, K, op->row_stride, op->recv ? op->recv : op->mesh->recv,
                                                       nt, op->nrows, x, x0, y, R, alpha, g.producers, g.groups,
                                                       g.log_depth, g.log_slots,
                                                       next_sweep_direction(op->vals), keep, op->dev_err);
    }
    DFM_LAUNCHED();
    DFM_CUDA_CHECK(cudaGetLastError());
    return DFM_OK;
  };
  if (R > 8) return combo ? go(spmv_multi_kernel<NB, 2, true>) : go(spmv_multi_kernel<NB, 2, false>);
  return combo ? go(spmv_multi_kernel<NB, 1, true>) : go(spmv_multi_kernel<NB, 1, false>);
}

}  // namespace

bool apply_multi_supported(const dfm_op* op, int K, int R) {
  return op->precision == DFM_F32 && geom::multi_faster(op->nb, K, std::min(R, kMaxRhs));
}

int apply_multi(const dfm_op* op, const dfm_op* const* combo_ops, int K, const double* coef, const float* x,
                const float* x0, float* y, int R, double alpha, cudaStream_t st) {
  const int64_t stride = op->nrows * (int64_t)op->nb;
  for (int r0 = 0; r0 < R; r0 += kMaxRhs) {
    const int Rl = std::min(kMaxRhs, R - r0);
    const geom::Multi g = geom::multi_geometry(op->nb, K, Rl);
    Ops ops{};
    for (int k = 0; k < K; ++k)
      ops.vals[k] = reinterpret_cast<const float*>(combo_ops ? combo_ops[k]->vals : op->vals);
    for (int r = 0; r < Rl; ++r)
      for (int k = 0; k < K; ++k) ops.coef[r][k] = coef ? (float)coef[(int64_t)(r0 + r) * K + k] : 1.f;
    const float* xr = x + r0 * stride;
    const float* x0r = x0 ? x0 + r0 * stride : nullptr;
    float* yr = y + r0 * stride;
    int rc;
    switch (op->nb) {
      case 3: rc = launch_multi<3>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 6: rc = launch_multi<6>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 10: rc = launch_multi<10>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 15: rc = launch_multi<15>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 21: rc = launch_multi<21>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 28: rc = launch_multi<28>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 36: rc = launch_multi<36>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      case 45: rc = launch_multi<45>(op, ops, K, coef != nullptr, xr, x0r, yr, Rl, (float)alpha, g, st); break;
      default: rc = set_error(DFM_ERR_UNSUPPORTED, "dfm_apply: unsupported basis size");
    }
    if (rc) return rc;
  }
  return DFM_OK;
}

}  // namespace dfm
