// Adjoint gradient of a receiver functional with respect to per-tet damping,
// and the interior density functional it is built from (Sec. 4.1, Eq. IntDens).
//
// J(rho) = g . rho with (I - B) rho = rho0.  With (I - B)^T lambda = g,
//   dJ/dmu_t = lambda^T (dB/dmu_t) rho + (dg/dmu_t) . rho.
// B depends on mu_t only through the damped areas S = 2 |OBC| phi2(mu L_O) of
// the 12 face pairs of tet t (Sec. 3.3), so
//   dB/dmu_t (pair) = lambda_pair N_{n'm'} / sqrt(|T_l||T_l'|) sum_nodes w J 2|OBC| L_O phi2'(mu L_O) Z(p') Z(p)^T.
// The contraction lambda_R^T dB rho_J is computed on the fly: per node the
// scalar c = w' (Z(p') . lambda_s) is accumulated into u = sum c Z(p), and the
// pair contributes u . rho_J for every right-hand side; dB is never formed.
#include <math.h>

#include <algorithm>
#include <vector>

#include "dfm_internal.cuh"
#include "interior_rule.cuh"
#include "node.cuh"
#include "row_node.cuh"

namespace dfm {
namespace {

constexpr int kCWarps = 4;      // warps per block in the contraction kernel
constexpr int kManyRhs = 8;     // right-hand sides from which the lanes split over them

// d/dx phi2(x) = (2 - x - (x + 2) e^{-x}) / x^3 = sum_j (-1)^(j+1) (j+1) x^j / (j+3)!
// in FP32: eleven terms of the series below x = 1, where the closed form cancels
// (the first one left out is below 1e-9 of the sum)
__device__ __forceinline__ float phi2_prime_row(float x) {
  if (x < 1.f) {
    const float c[11] = {-1.f / 6,          2.f / 24,          -3.f / 120,          4.f / 720,
                         -5.f / 5040,       6.f / 40320,       -7.f / 362880,       8.f / 3628800,
                         -9.f / 39916800,   10.f / 479001600,  -11.f / 6227020800.f};
    float s = c[10];
#pragma unroll
    for (int i = 9; i >= 0; --i) s = fmaf(x, s, c[i]);
    return s;
  }
  return (2.f - x - (x + 2.f) * expf(-x)) / (x * x * x);
}

template <int NP>
struct ContractWarp {
  static constexpr int NB = (NP + 1) * (NP + 2) / 2, NB4 = (NB + 3) / 4 * 4;
  PatchWarp P;
  PairConst pc;
  alignas(16) float lam[NB4];  // lambda of the receiving row times the test-side normalisation
  // the lanes' sums of c Z(p), one row per lane of an odd stride; then their total
  float u[32 * (NB | 1)];
};

// One warp per face pair, nodes row by row (row_node.cuh); resident warps take
// pairs off a shared counter as in the assembly.  Per node both Zernike vectors
// come from one packed recursion.  Measured: 6,000 tets at N_p = 4 in
// 0.77 ms against 1.4 ms with every node's geometry evaluated on its own and a
// shuffle reduction per basis function.  Issue bounds it.
template <int NP>
__global__ void __launch_bounds__(kCWarps * 32, NP >= 7 ? 3 : (NP >= 5 ? 4 : 5))
contract_kernel(const PairConst* __restrict__ pairs, int64_t npairs, const double* __restrict__ gl_x,
                const double* __restrict__ gl_w, int q, float cos_max, const double* __restrict__ lam,
                const double* __restrict__ rho, int R, int64_t nrows, int64_t nt, double* __restrict__ dJ,
                unsigned long long* __restrict__ counter) {
  constexpr int NB = (NP + 1) * (NP + 2) / 2, NB4 = ContractWarp<NP>::NB4, LD = NB | 1;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  ContractWarp<NP>* smem = reinterpret_cast<ContractWarp<NP>*>(dyn_smem);
  __shared__ float s_x[kMaxQ], s_w[kMaxQ];
  __shared__ double s_ninv[64];
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;
  ContractWarp<NP>& S = smem[wid];
  if (threadIdx.x < q) {
    s_x[threadIdx.x] = (float)gl_x[threadIdx.x];
    s_w[threadIdx.x] = (float)gl_w[threadIdx.x];
  }
  if (threadIdx.x < NB) s_ninv[threadIdx.x] = zernike_invnorm(threadIdx.x);
  __syncthreads();
  const float qinv = 1.f / (float)q;
  unsigned long long p = (unsigned long long)blockIdx.x * kCWarps + wid;
  while (p < (unsigned long long)npairs) {
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(counter, 1ull) + (unsigned long long)gridDim.x * kCWarps;
    for (int i = lane; i < (int)(sizeof(PairConst) / 4); i += 32)
      reinterpret_cast<int*>(&S.pc)[i] = reinterpret_cast<const int*>(pairs + p)[i];
    __syncwarp();
    const int kind = S.pc.kind;
    if (kind >= 0) {  // else no block for this pair in this part
      const int64_t t = (int64_t)(p / 12);
      const int64_t J = 4 * t + (int64_t)((p % 12) / 3);
      for (int a = lane; a < NB4; a += 32)
        S.lam[a] = a < NB ? (float)(lam[(int64_t)S.pc.out_row * NB + a] * (double)S.pc.scale * s_ninv[a]) : 0.f;
      start_regions(S.P, S.pc, cos_max, lane);
      const float mu = S.pc.mu, D3 = S.pc.D[2], area2 = 2.f * S.pc.area_src;
      float u[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) u[b] = 0.f;
      while (true) {
        const int npatch = fill_patches_warp(S.P, cos_max, lane);
        if (npatch == 0) break;
        const int rows = npatch * q;
        for (int base = 0; base < rows;) {
          const RowPass ps = next_pass(rows - base);
          const int rl = lane / ps.per;
          const bool live = rl < ps.rows;
          const int row = base + (live ? rl : ps.rows - 1);
          const int pi = (int)(((float)row + 0.5f) * qinv), i = row - pi * q;  // exact: row < 20 x 32
          RowConst rc;
          row_const(S.P.patch[pi], s_x[i], S.pc, rc);
          const float wi = live ? s_w[i] * area2 : 0.f;
          base += ps.rows;
          for (int j0 = 0; j0 < q; j0 += ps.per) {
            const int j = j0 + (lane - rl * ps.per);
            const bool on = j < q;
            const int jc = on ? j : q - 1;
            const RowNode g = row_node(rc, s_x[jc], D3, kind, S.pc);
            const float w = on ? wi * s_w[jc] * g.base * (g.LO * phi2_prime_row(mu * g.LO)) : 0.f;
            float2 Z[NB];
            zernike2<NP>(g.px, g.py, pair(1.f, 1.f), Z);
            float sq[4] = {0.f, 0.f, 0.f, 0.f};  // four chains
#pragma unroll
            for (int v = 0; v < NB4 / 4; ++v) {
              const float4 l4 = *reinterpret_cast<const float4*>(S.lam + 4 * v);
              const float la[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (4 * v + e < NB) sq[e] = fmaf(Z[4 * v + e < NB ? 4 * v + e : 0].y, la[e], sq[e]);
            }
            const float c = w * ((sq[0] + sq[1]) + (sq[2] + sq[3]));
#pragma unroll
            for (int b = 0; b < NB; ++b) u[b] = fmaf(c, Z[b].x, u[b]);
          }
        }
      }
      // sum over the lanes: lane b adds column b (and b + 32) of the staged rows
#pragma unroll
      for (int b = 0; b < NB; ++b) S.u[lane * LD + b] = u[b];
      __syncwarp();
      float t0 = 0.f, t1 = 0.f;
      for (int k = 0; k < 32; ++k) {
        if (lane < NB) t0 += S.u[k * LD + lane];
        if (NB > 32 && lane + 32 < NB) t1 += S.u[k * LD + lane + 32];
      }
      __syncwarp();
      if (R < kManyRhs) {
        // the lanes share a right-hand side: one product each, summed by shuffles
        for (int r = 0; r < R; ++r) {
          const double* x = rho + ((int64_t)r * nrows + J) * NB;
          double s = lane < NB ? (double)t0 * x[lane] : 0.0;
          if (NB > 32 && lane + 32 < NB) s = fma((double)t1, x[lane + 32], s);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (lane == 0) atomicAdd(&dJ[(int64_t)r * nt + t], s);
        }
      } else {
        // a right-hand side per lane
        if (lane < NB) S.u[lane] = t0;
        if (NB > 32 && lane + 32 < NB) S.u[lane + 32] = t1;
        __syncwarp();
        for (int r = lane; r < R; r += 32) {
          const double* x = rho + ((int64_t)r * nrows + J) * NB;
          double s = 0.0;
          for (int b = 0; b < NB; ++b) s = fma((double)S.u[b], x[b], s);
          atomicAdd(&dJ[(int64_t)r * nt + t], s);
        }
      }
    }
    p = __shfl_sync(0xffffffffu, next, 0);
    __syncwarp();  // the pair's constants are read before the next ones arrive
  }
}

// dJ[r][t] += sum_{l,a} dg[4t+l][a] rho_r[4t+l][a]  (rows with dg == 0 are skipped)
__global__ void explicit_term_kernel(const double* __restrict__ dg, const double* __restrict__ rho, int R, int nb,
                                     int64_t nrows, int64_t nt, double* __restrict__ dJ) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const double* d = dg + 4 * t * nb;
  bool any = false;
  for (int i = 0; i < 4 * nb; ++i) any |= (d[i] != 0.0);
  if (!any) return;
  for (int r = 0; r < R; ++r) {
    const double* x = rho + ((int64_t)r * nrows + 4 * t) * nb;
    double s = 0.0;
    for (int i = 0; i < 4 * nb; ++i) s = fma(d[i], x[i], s);
    dJ[(int64_t)r * nt + t] += s;
  }
}

// Interior density coefficients at the centroid of tet e (Eq. IntDens), FP64.
// One warp per (listed tet, face): collapsed tensor Gauss on the face.
template <int NP>
__global__ void interior_density_kernel(const double* __restrict__ V, const int32_t* __restrict__ tets,
                                        const FaceGeom* __restrict__ geom, const double* __restrict__ mu_tet,
                                        double mu_uniform, const int64_t* __restrict__ list,
                                        const double* __restrict__ weights, int n, const double* __restrict__ gl_x,
                                        const double* __restrict__ gl_w, int nq, double* __restrict__ gvec,
                                        double* __restrict__ dgvec) {
  constexpr int NB = (NP + 1) * (NP + 2) / 2;
  const int lane = threadIdx.x & 31;
  const int64_t wg = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (wg >= 4 * (int64_t)n) return;
  const int i = (int)(wg >> 2);
  const int l = (int)(wg & 3);
  const int64_t e = list[i];
  const double wt = weights ? weights[i] : 1.0;
  const int32_t* tv = tets + 4 * e;
  double r[3] = {0, 0, 0};
  for (int v = 0; v < 4; ++v)
    for (int c = 0; c < 3; ++c) r[c] += 0.25 * V[3 * (int64_t)tv[v] + c];
  const FaceGeom F = geom[4 * e + l];
  double p[3][3];
  for (int k = 0; k < 3; ++k)
    for (int c = 0; c < 3; ++c) p[k][c] = V[3 * (int64_t)tv[(l + 1 + k) & 3] + c];
  const double mu = mu_tet ? mu_tet[e] : mu_uniform;
  double g[NB], dg[NB], Z[NB];
#pragma unroll
  for (int a = 0; a < NB; ++a) g[a] = dg[a] = 0.0;
  for (int k = lane; k < nq * nq; k += 32) {
    const int ii = k / nq, jj = k - ii * nq;
    const double u = 0.5 * (1.0 + gl_x[ii]);
    const double v = (1.0 - u) * 0.5 * (1.0 + gl_x[jj]);
    const double w = gl_w[ii] * gl_w[jj] * 0.25 * (1.0 - u) * 2.0 * F.area;
    double rs[3];
    for (int c = 0; c < 3; ++c) rs[c] = r[c] - (p[0][c] + u * (p[1][c] - p[0][c]) + v * (p[2][c] - p[0][c]));
    const double dist = sqrt(rs[0] * rs[0] + rs[1] * rs[1] + rs[2] * rs[2]);
    const double id = 1.0 / dist;
    const double d0 = rs[0] * id, d1 = rs[1] * id, d2 = rs[2] * id;
    const double cosv = d0 * F.n[0] + d1 * F.n[1] + d2 * F.n[2];
    const double ker = w * cosv * exp(-mu * dist) * id * id;
    zernike<NP, double>(d0 * F.e1[0] + d1 * F.e1[1] + d2 * F.e1[2], d0 * F.e2[0] + d1 * F.e2[1] + d2 * F.e2[2], Z);
#pragma unroll
    for (int a = 0; a < NB; ++a) {
      g[a] = fma(ker, Z[a], g[a]);
      dg[a] = fma(-dist * ker, Z[a], dg[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < NB; ++a)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      g[a] += __shfl_xor_sync(0xffffffffu, g[a], o);
      dg[a] += __shfl_xor_sync(0xffffffffu, dg[a], o);
    }
  if (lane == 0) {
    const double s = wt / sqrt(F.area);
    for (int a = 0; a < NB; ++a) {
      atomicAdd(&gvec[(4 * e + l) * NB + a], s * g[a]);
      if (dgvec) atomicAdd(&dgvec[(4 * e + l) * NB + a], s * dg[a]);
    }
  }
}

template <int NP>
int launch_contract_np(const PairConst* pairs, int64_t npairs, const double* glx, const double* glw, int q,
                       float cos_max, const double* lam, const double* rho, int R, int64_t nrows, int64_t nt,
                       double* dJ, unsigned long long* counter, cudaStream_t st) {
  constexpr size_t smem = sizeof(ContractWarp<NP>) * kCWarps;
  int dev = 0, nsm = 0, per_sm = 0;
  DFM_CUDA_CHECK(cudaGetDevice(&dev));
  DFM_CUDA_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  DFM_CUDA_CHECK(cudaFuncSetAttribute(contract_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  DFM_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, contract_kernel<NP>, kCWarps * 32, smem));
  const int64_t blocks = std::min<int64_t>((npairs + kCWarps - 1) / kCWarps, (int64_t)nsm * std::max(per_sm, 1));
  DFM_CUDA_CHECK(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st));
  {
    ::dfm::KernelTimer timer_(DFM_KERNEL_CONTRACT, st);
    contract_kernel<NP><<<(unsigned)blocks, kCWarps * 32, smem, st>>>(pairs, npairs, glx, glw, q, cos_max, lam, rho, R,
                                                                      nrows, nt, dJ, counter);
  }
  DFM_LAUNCHED();
  DFM_CUDA_CHECK(cudaGetLastError());
  return DFM_OK;
}

int launch_contract(int Np, const PairConst* pairs, int64_t npairs, const double* glx, const double* glw, int q,
                    float cos_max, const double* lam, const double* rho, int R, int64_t nrows, int64_t nt, double* dJ,
                    unsigned long long* counter, cudaStream_t st) {
#define CASE(N) \
  case N: return launch_contract_np<N>(pairs, npairs, glx, glw, q, cos_max, lam, rho, R, nrows, nt, dJ, counter, st);
  switch (Np) {
    CASE(0) CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8)
    default: return set_error(DFM_ERR_ARG, "dfm_adjoint: Np must be in 0..8");
  }
#undef CASE
}

// ---------------------------------------------------------------------------
// The same functional with the split polar rule of interior_rule.cuh (6 nq^2
// nodes per face), which stays accurate when the centroid is close to a face.
//
// FP64 arithmetic is what this costs (2 FP64 lanes per SM), so the work is
// split by what it depends on:
//  - per (face, edge): the foot of the centroid, the edge's line and the two
//    pieces' ranges, by one lane, kept in shared memory;
//  - per line (edge, piece, azimuth node): direction, Jacobian, and the angle
//    Phi up to the edge, by the lane that owns the line;
//  - per node of a line: with p = -sin(phi) (ex, ey) the Zernike function is
//    R_n^m(sin phi) times an angular factor of the line, and R_n^m is a
//    polynomial in u = 1 - 2 sin^2(phi) (n even) or sin(phi) times one (n odd),
//    so a node only adds its kernel weight times u^k and sin(phi) u^k to the
//    N_p + 1 moments of the line (u in [-1, 1] keeps the coefficients, and with
//    them the rounding, small: their absolute values sum to at most 8.5 up to
//    N_p = 8, where powers of sin^2 would reach 321);
//  - phi_b = Phi x_b with the Gauss nodes symmetric about Phi / 2: sine and
//    cosine of the lower half by their series (phi <= pi / 4), of the upper half
//    by the addition theorems.
// Measured: 6,000 tets at N_p = 4 in 8.4 ms against 67.8 ms with every node
// evaluated on its own.  FP64 issue bounds it: some 50 FP64 instructions per node
// (12 for its sine and cosine, 17 for 1 / c and the exponential, 21 for the moments)
// and 260 per line are 8.0 ms at two lanes per SM.
// ---------------------------------------------------------------------------

// coefficients of R_n^m in powers of u = 1 - 2 rho^2, after taking out one rho
// for odd n; m >= 0, N_p <= 8
struct RadialTable {
  double c[9][9][5];
};
constexpr RadialTable radial_table() {
  RadialTable t{};
  for (int n = 0; n <= 8; ++n)
    for (int m = n & 1; m <= n; m += 2)
      for (int s = 0; s <= (n - m) / 2; ++s) {
        // (-1)^s (n - s)! / (s! ((n + m)/2 - s)! ((n - m)/2 - s)!) rho^(n - 2s)
        double f = s & 1 ? -1.0 : 1.0;
        for (int i = 2; i <= n - s; ++i) f *= i;
        for (int i = 2; i <= s; ++i) f /= i;
        for (int i = 2; i <= (n + m) / 2 - s; ++i) f /= i;
        for (int i = 2; i <= (n - m) / 2 - s; ++i) f /= i;
        const int j = (n - 2 * s) / 2;  // rho^(2 j) = ((1 - u) / 2)^j
        double b = 1.0;
        for (int i = 0; i < j; ++i) b *= 0.5;
        for (int k = 0; k <= j; ++k) {
          t.c[n][m][k] += f * b;
          b = -b * (j - k) / (k + 1);
        }
      }
  return t;
}

// 1 / x in FP64: the hardware's approximate reciprocal (about 20 bits) and two
// Newton steps
__device__ __forceinline__ double recip64(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// sine and cosine of x in [0, pi / 4] (Taylor; the first terms left out are
// below 5e-17)
__device__ __forceinline__ void sincos_quarter(double x, double* s, double* c) {
  const double z = x * x;
  double a = -1.0 / 1307674368000.0, b = 1.0 / 20922789888000.0;
  a = fma(a, z, 1.0 / 6227020800.0);
  a = fma(a, z, -1.0 / 39916800.0);
  a = fma(a, z, 1.0 / 362880.0);
  a = fma(a, z, -1.0 / 5040.0);
  a = fma(a, z, 1.0 / 120.0);
  a = fma(a, z, -1.0 / 6.0);
  b = fma(b, z, -1.0 / 87178291200.0);
  b = fma(b, z, 1.0 / 479001600.0);
  b = fma(b, z, -1.0 / 3628800.0);
  b = fma(b, z, 1.0 / 40320.0);
  b = fma(b, z, -1.0 / 720.0);
  b = fma(b, z, 1.0 / 24.0);
  b = fma(b, z, -0.5);
  *s = fma(a * z, x, x);
  *c = fma(b, z, 1.0);
}

// e^-x for x in [0, 1/16] (Taylor; the first term left out is below 3e-19)
__device__ __forceinline__ double exp_small(double x) {
  double s = -1.0 / 362880.0;
  s = fma(s, x, 1.0 / 40320.0);
  s = fma(s, x, -1.0 / 5040.0);
  s = fma(s, x, 1.0 / 720.0);
  s = fma(s, x, -1.0 / 120.0);
  s = fma(s, x, 1.0 / 24.0);
  s = fma(s, x, -1.0 / 6.0);
  s = fma(s, x, 0.5);
  s = fma(s, x, -1.0);
  return fma(s, x, 1.0);
}

// One edge of a face: its line (distance d from the foot F, unit direction t,
// foot M of the perpendicular from F), cc = sqrt(h^2 + d^2), the ranges of the
// two pieces in s, and the sign of the triangle (0: it adds nothing).
struct PolarEdge {
  double d, cc, Mx, My, tx, ty, s0, s1, s2, sgn;
};

// moments of one line: U_k = sum ker u^k, V_k = sum ker rho u^k, and the same
// with ker R
template <int NP>
struct LineMoments {
  static constexpr int NU = NP / 2 + 1, NV = (NP + 1) / 2;
  double U[NU], V[NV > 0 ? NV : 1], UR[NU], VR[NV > 0 ? NV : 1];
};

template <int NP>
__device__ __forceinline__ void add_node(LineMoments<NP>& L, double s, double c, double w, double h, double mu,
                                         bool small) {
  using M = LineMoments<NP>;
  const double R = h * recip64(c);
  const double x = mu * R;
  double k = w * s * (small ? exp_small(x) : exp(-x));
  double kR = k * R;
  const double u = fma(-2.0 * s, s, 1.0);
  double v = k * s, vR = kR * s;
#pragma unroll
  for (int i = 0; i < M::NU; ++i) {
    L.U[i] += k;
    L.UR[i] += kR;
    if (i + 1 < M::NU) k *= u, kR *= u;
  }
#pragma unroll
  for (int i = 0; i < M::NV; ++i) {
    L.V[i] += v;
    L.VR[i] += vR;
    if (i + 1 < M::NV) v *= u, vR *= u;
  }
}

// LP lanes per (listed tet, face), each taking every LP-th of its 6 nq lines
template <int NP, int LP>
__global__ void __launch_bounds__(128)
interior_density_polar_kernel(const double* __restrict__ V, const int32_t* __restrict__ tets,
                              const FaceGeom* __restrict__ geom, const double* __restrict__ mu_tet, double mu_uniform,
                              const int64_t* __restrict__ list, const double* __restrict__ weights, int n,
                              const double* __restrict__ gl_x, const double* __restrict__ gl_w, int nq,
                              double* __restrict__ gvec, double* __restrict__ dgvec) {
  constexpr int NB = (NP + 1) * (NP + 2) / 2;
  constexpr int FB = 128 / LP;  // faces per block
  constexpr RadialTable RT = radial_table();
  __shared__ PolarEdge s_edge[FB][3];
  __shared__ double s_h[FB];
  __shared__ double s_x[64], s_w[64];
  const int gl = threadIdx.x / LP, lane = threadIdx.x % LP;
  const int64_t unit = (int64_t)blockIdx.x * FB + gl;
  const bool live = unit < 4 * (int64_t)n;
  const int i = live ? (int)(unit >> 2) : 0;
  const int l = (int)(unit & 3);
  const int64_t e = list[i];
  if (threadIdx.x < nq) {
    s_x[threadIdx.x] = 0.5 * (gl_x[threadIdx.x] + 1.0);
    s_w[threadIdx.x] = 0.5 * gl_w[threadIdx.x];
  }
  const FaceGeom* F = geom + 4 * e + l;
  if (lane < 3) {
    const int32_t* tv = tets + 4 * e;
    double r[3] = {0, 0, 0}, p[3][3];
    for (int v = 0; v < 4; ++v)
      for (int c = 0; c < 3; ++c) r[c] += 0.25 * V[3 * (int64_t)tv[v] + c];
    for (int k = 0; k < 3; ++k)
      for (int c = 0; c < 3; ++c) p[k][c] = V[3 * (int64_t)tv[(l + 1 + k) & 3] + c];
    double h = 0.0, on = 0.0, u[3], v[3];
    for (int c = 0; c < 3; ++c) {
      h += (r[c] - p[0][c]) * F->n[c];
      u[c] = p[1][c] - p[0][c];
      v[c] = p[2][c] - p[0][c];
    }
    on = (u[1] * v[2] - u[2] * v[1]) * F->n[0] + (u[2] * v[0] - u[0] * v[2]) * F->n[1] +
         (u[0] * v[1] - u[1] * v[0]) * F->n[2];
    // the edge's end points in the face plane, F at the origin
    const int ka = lane, kb = lane == 2 ? 0 : lane + 1;
    double Ax = 0, Ay = 0, Bx = 0, By = 0;
    for (int c = 0; c < 3; ++c) {
      const double fc = r[c] - h * F->n[c];
      const double pa = ka == 0 ? p[0][c] : (ka == 1 ? p[1][c] : p[2][c]);
      const double pb = kb == 0 ? p[0][c] : (kb == 1 ? p[1][c] : p[2][c]);
      Ax += (pa - fc) * F->e1[c];
      Ay += (pa - fc) * F->e2[c];
      Bx += (pb - fc) * F->e1[c];
      By += (pb - fc) * F->e2[c];
    }
    PolarEdge E;
    const double len = sqrt((Bx - Ax) * (Bx - Ax) + (By - Ay) * (By - Ay));
    E.tx = len > 0.0 ? (Bx - Ax) / len : 1.0;
    E.ty = len > 0.0 ? (By - Ay) / len : 0.0;
    E.d = fabs(Ax * E.ty - Ay * E.tx);
    const double cr = Ax * By - Ay * Bx;
    E.sgn = (cr > 0.0 ? 1.0 : (cr < 0.0 ? -1.0 : 0.0)) * (on >= 0.0 ? 1.0 : -1.0);
    if (len == 0.0 || E.d < 1e-15 * len) {
      E.sgn = 0.0;
      E.d = 1.0;  // keeps the line's arithmetic finite
    }
    const double uA = Ax * E.tx + Ay * E.ty, uB = Bx * E.tx + By * E.ty;
    E.Mx = Ax - uA * E.tx;
    E.My = Ay - uA * E.ty;
    E.cc = sqrt(h * h + E.d * E.d);
    E.s0 = atan2(uA, E.cc);
    E.s2 = atan2(uB, E.cc);
    E.s1 = (E.s0 < 0.0 && E.s2 > 0.0) ? 0.0 : 0.5 * (E.s0 + E.s2);
    s_edge[gl][lane] = E;
    if (lane == 0) s_h[gl] = h;
  }
  __syncthreads();
  const double h = s_h[gl];
  const double mu = mu_tet ? mu_tet[e] : mu_uniform;
  double g[NB], dg[NB];
#pragma unroll
  for (int a = 0; a < NB; ++a) g[a] = dg[a] = 0.0;
  const int half = nq / 2;
  for (int line = lane; line < 6 * nq; line += LP) {
    const int pc = line / nq, a = line - pc * nq;
    const PolarEdge& E = s_edge[gl][pc >> 1];
    const double s0 = pc & 1 ? E.s1 : E.s0, ds = (pc & 1 ? E.s2 : E.s1) - s0;
    double sn, cs;
    sincos(s0 + ds * s_x[a], &sn, &cs);
    const double ics = recip64(cs);
    const double uu = E.cc * sn * ics;
    const double ell2 = fma(uu, uu, E.d * E.d);
    const double ell = sqrt(ell2), iell = 1.0 / ell;
    const double ex = -(E.Mx + uu * E.tx) * iell, ey = -(E.My + uu * E.ty) * iell;
    const double ih = 1.0 / sqrt(fma(h, h, ell2));
    const double sP = ell * ih, cP = h * ih;
    const double Phi = atan2(ell, h);
    // dpsi = d du / ell^2, du = c ds / cos^2(s)
    const double J = E.sgn * ds * s_w[a] * E.cc * E.d * ics * ics * iell * iell * Phi;
    const bool small = fabs(mu) * h <= 0.0625 * cP;  // every mu R of the line is at most mu h / cos(Phi)
    LineMoments<NP> L;
#pragma unroll
    for (int k = 0; k < LineMoments<NP>::NU; ++k) L.U[k] = L.UR[k] = 0.0;
#pragma unroll
    for (int k = 0; k < LineMoments<NP>::NV; ++k) L.V[k] = L.VR[k] = 0.0;
    for (int b = 0; b < half; ++b) {
      double sl, cl;
      sincos_quarter(Phi * s_x[b], &sl, &cl);
      add_node<NP>(L, sl, cl, s_w[b], h, mu, small);
      add_node<NP>(L, fma(sP, cl, -cP * sl), fma(cP, cl, sP * sl), s_w[nq - 1 - b], h, mu, small);
    }
    if (nq & 1) {
      double sl, cl;
      sincos_quarter(0.5 * Phi, &sl, &cl);
      add_node<NP>(L, sl, cl, s_w[half], h, mu, small);
    }
    double cm = J, sm = 0.0;  // J Re, Im of the line's (-ex - i ey)^m
#pragma unroll
    for (int m = 0; m <= NP; ++m) {
      if (m > 0) {
        const double t = cm * ex - sm * ey;
        sm = cm * ey + sm * ex;
        cm = t;
      }
#pragma unroll
      for (int nn = m; nn <= NP; nn += 2) {
        double S = 0.0, T = 0.0;
#pragma unroll
        for (int k = 0; k <= nn / 2; ++k) {
          const double c = RT.c[nn][m][k];
          if (c == 0.0) continue;
          S = fma(c, nn & 1 ? L.V[k < LineMoments<NP>::NV ? k : 0] : L.U[k], S);
          T = fma(c, nn & 1 ? L.VR[k < LineMoments<NP>::NV ? k : 0] : L.UR[k], T);
        }
        const int ip = (nn * (nn + 2) + m) / 2, im = (nn * (nn + 2) - m) / 2;
        g[ip] = fma(cm, S, g[ip]);
        dg[ip] = fma(-cm, T, dg[ip]);
        if (m > 0) {
          g[im] = fma(sm, S, g[im]);
          dg[im] = fma(-sm, T, dg[im]);
        }
      }
    }
  }
  const double s = live ? (weights ? weights[i] : 1.0) / sqrt(F->area) : 0.0;
#pragma unroll
  for (int a = 0; a < NB; ++a) {
#pragma unroll
    for (int o = LP / 2; o > 0; o >>= 1) {
      g[a] += __shfl_xor_sync(0xffffffffu, g[a], o);
      dg[a] += __shfl_xor_sync(0xffffffffu, dg[a], o);
    }
    if (live && lane == a % LP) {
      atomicAdd(&gvec[(4 * e + l) * NB + a], s * g[a]);
      if (dgvec) atomicAdd(&dgvec[(4 * e + l) * NB + a], s * dg[a]);
    }
  }
}

template <int NP>
void launch_polar(const dfm_mesh* mesh, const double* mu, double mu_uniform, const int64_t* list, const double* w,
                  int n, const double* glx, const double* glw, int nq, double* gvec, double* dgvec, cudaStream_t st) {
  // sixteen lanes per face take the 144 lines of the default rule in nine full
  // rounds; a whole warp per face where that still leaves SM partitions idle, at up
  // to two faces for each of the four (48 tets at N_p = 4: 120 against 187 us)
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    nsm = 0;
  if (4 * (int64_t)n > 8 * (int64_t)nsm)
    interior_density_polar_kernel<NP, 16><<<(unsigned)((4 * (int64_t)n + 7) / 8), 128, 0, st>>>(
        mesh->verts, mesh->tets, mesh->geom, mu, mu_uniform, list, w, n, glx, glw, nq, gvec, dgvec);
  else
    interior_density_polar_kernel<NP, 32><<<(unsigned)n, 128, 0, st>>>(
        mesh->verts, mesh->tets, mesh->geom, mu, mu_uniform, list, w, n, glx, glw, nq, gvec, dgvec);
}

// out[r][e] = sum over tet e's four rows of gvec . rho_r: one warp per (r, e),
// the lanes striding over the 4 nb contiguous coefficients of the tet
__global__ void tet_density_kernel(const double* __restrict__ g, const double* __restrict__ rho, int64_t nt,
                                   int nb, int64_t units, double* __restrict__ out) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= units) return;  // blockDim is a multiple of 32: whole warps leave together
  const int64_t r = w / nt, e = w - r * nt;
  const double* gp = g + 4 * e * nb;
  const double* xp = rho + (r * 4 * nt + 4 * e) * nb;
  double acc = 0.0;
  for (int k = lane; k < 4 * nb; k += 32) acc = fma(gp[k], xp[k], acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) out[w] = acc;
}

}  // namespace
}  // namespace dfm

using namespace dfm;

extern "C" int dfm_interior_density(const dfm_mesh* mesh, int Np, const double* mu, double mu_uniform,
                                    const int64_t* tets_host, const double* weights_host, int n, int nq, double* gvec,
                                    double* dgvec, void* stream) {
  if (!mesh || !tets_host || !gvec || n < 1 || !basis_ok(Np, geom::kWideMaxNp))
    return set_error(DFM_ERR_ARG, "dfm_interior_density: bad argument");
  const int ns = basis_ns(Np);
  Np = basis_np(Np);
  // nq < 0: the split polar rule with |nq| points per direction; nq = 0: the
  // same rule with 24 points (accurate for centroids close to a face, as on
  // thin tets); nq > 0: the flat collapsed Gauss rule of that order
  if (nq == 0) nq = -24;
  const bool polar = nq < 0;
  if (polar) nq = -nq;
  if (nq < 2 || nq > 64) return set_error(DFM_ERR_ARG, "dfm_interior_density: |nq| must be in 2..64");
  if (!mu && !(mu_uniform >= 0)) return set_error(DFM_ERR_ARG, "dfm_interior_density: mu_uniform must be >= 0");
  for (int i = 0; i < n; ++i)
    if (tets_host[i] < 0 || tets_host[i] >= mesh->nt) return set_error(DFM_ERR_ARG, "dfm_interior_density: bad tet id");
  cudaStream_t st = as_stream(stream);
  // small stream-ordered scratch: tet list, weights, Gauss table
  char* buf = nullptr;
  const size_t bytes = sizeof(int64_t) * n + sizeof(double) * n + 2 * 64 * sizeof(double) + 256;
  DFM_CUDA_CHECK(cudaMallocAsync(reinterpret_cast<void**>(&buf), bytes, st));
  int64_t* list = reinterpret_cast<int64_t*>(buf);
  double* w = reinterpret_cast<double*>(buf + sizeof(int64_t) * n);
  double* glx = w + n;
  double* glw = glx + 64;
  DFM_CUDA_CHECK(cudaMemcpyAsync(list, tets_host, sizeof(int64_t) * n, cudaMemcpyHostToDevice, st));
  if (weights_host) DFM_CUDA_CHECK(cudaMemcpyAsync(w, weights_host, sizeof(double) * n, cudaMemcpyHostToDevice, st));
  int rc = gauss_legendre_device(nq, glx, glw, st);
  if (rc) return rc;
  const int64_t threads = 4 * (int64_t)n * 32;
  const unsigned blocks = (unsigned)((threads + 127) / 128);
  const double* wp = weights_host ? w : nullptr;
#define CASE(N)                                                                                                  \
  case N:                                                                                                        \
    if (polar)                                                                                                   \
      launch_polar<N>(mesh, mu, mu_uniform, list, wp, n, glx, glw, nq, gvec, dgvec, st);                         \
    else                                                                                                         \
      interior_density_kernel<N><<<blocks, 128, 0, st>>>(mesh->verts, mesh->tets, mesh->geom, mu, mu_uniform, list, \
                                                         wp, n, glx, glw, nq, gvec, dgvec);                      \
    break;
  switch (ns == 1 ? Np : -1) {
    CASE(0) CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8)
    default:  // Np = 9..20, and the linear spatial basis (wide.cu)
      rc = launch_interior_density_wide(Np, ns, polar, mesh, mu, mu_uniform, list, wp, n, glx, glw, nq, gvec, dgvec,
                                        st);
      if (rc) {
        cudaFreeAsync(buf, st);
        return rc;
      }
  }
#undef CASE
  if (Np <= 8 && ns == 1) DFM_LAUNCHED();
  DFM_CUDA_CHECK(cudaGetLastError());
  DFM_CUDA_CHECK(cudaFreeAsync(buf, st));
  return DFM_OK;
}

extern "C" int dfm_tet_density(const dfm_mesh* mesh, int Np, const double* gvec, const double* rho, int R,
                               double* out, void* stream) {
  if (!mesh || !gvec || !rho || !out || R < 1 || !basis_ok(Np, geom::kWideMaxNp))
    return set_error(DFM_ERR_ARG, "dfm_tet_density: bad argument");
  const int64_t units = (int64_t)R * mesh->nt;
  const int64_t blocks = (units + 7) / 8;  // 8 warps per block
  if (blocks > 0x7fffffff) return set_error(DFM_ERR_ARG, "dfm_tet_density: too many right-hand sides");
  cudaStream_t st = as_stream(stream);
  tet_density_kernel<<<(unsigned)blocks, 256, 0, st>>>(gvec, rho, mesh->nt, basis_size(Np), units, out);
  DFM_LAUNCHED();
  DFM_CUDA_CHECK(cudaGetLastError());
  return DFM_OK;
}

extern "C" int dfm_adjoint(const dfm_op* op, const dfm_params* params, const double* rho, int R, const double* gvec,
                           const double* dgvec, double* lambda_out, double* dJ_dmu, const dfm_solve_opts* opts,
                           void* stream, dfm_solve_info* info) {
  if (!op || !params || !rho || !gvec || !lambda_out || !dJ_dmu || !opts || R < 1)
    return set_error(DFM_ERR_ARG, "dfm_adjoint: bad argument");
  if (basis_np(params->Np) != op->Np || basis_ns(params->Np) != op->ns)
    return set_error(DFM_ERR_ARG, "dfm_adjoint: params->Np differs from the operator's");
  if (op->Np > 8 || op->ns > 1)
    return set_error(DFM_ERR_UNSUPPORTED,
                     "dfm_adjoint: the dB/dmu contraction is built for Np <= 8 and the piecewise-constant basis");
  const dfm_mesh* mesh = op->mesh;
  cudaStream_t st = as_stream(stream);
  // 1. adjoint equation (I - B)^T lambda = g
  dfm_solve_opts o = *opts;
  o.transpose = 1;
  o.use_x0 = opts->use_x0 ? 1 : 0;  // lambda_out holds the initial guess
  int rc = dfm_solve(op, gvec, 1, lambda_out, &o, stream, info);
  if (rc != DFM_OK && rc != DFM_ERR_NOT_CONVERGED) return rc;
  const int solve_rc = rc;
  // 2. per-pair constants for the operator's damping, then the fused contraction
  const int q = params->quad_order ? params->quad_order : params->Np + 6;
  if (q < 1 || q > kMaxQ) return set_error(DFM_ERR_ARG, "dfm_adjoint: quad_order must be in 1..32");
  const double deg = params->max_patch_deg > 0 ? params->max_patch_deg : 60.0;
  const float cos_max = (float)cos(deg * M_PI / 180.0);
  const int64_t npairs = 12 * mesh->nt;
  dfm_op* mop = const_cast<dfm_op*>(op);
  const int64_t need = npairs * (int64_t)sizeof(PairConst) + 2 * 64 * (int64_t)sizeof(double) + 256;
  if (mop->work_bytes < need) return set_error(DFM_ERR_ARG, "dfm_adjoint: operator has no assembly workspace");
  PairConst* pairs = reinterpret_cast<PairConst*>(mop->work);
  double* glx = reinterpret_cast<double*>(reinterpret_cast<char*>(mop->work) + npairs * sizeof(PairConst));
  double* glw = glx + 64;
  // (after the table: the assembly's node count, which stays, and a work counter)
  rc = gauss_legendre_device(q, glx, glw, st);
  if (rc) return rc;
  DFM_CUDA_CHECK(cudaMemsetAsync(dJ_dmu, 0, sizeof(double) * R * mesh->nt, st));
  // part 0: the blocks received across each exit face; part 1 (heterogeneous
  // media): the blocks reflected at interfaces; both cross tet t
  const bool media = params->c || params->rho_f;
  if (media != (op->rop != nullptr))
    return set_error(DFM_ERR_ARG, "dfm_adjoint: params->c / rho_f differ from the operator's assembly");
  for (int part = 0; part < (media ? 2 : 1); ++part) {
    pair_setup_kernel<<<(unsigned)((mesh->nrows + 127) / 128), 128, 0, st>>>(mesh->verts, mesh->tets, mesh->recv,
                                                                       mesh->refl, mesh->geom, params->mu,
                                                                       params->mu_uniform, mesh->nrows, pairs, params->c,
                                                                       params->rho_f, part);
    DFM_LAUNCHED();
    DFM_CUDA_CHECK(cudaGetLastError());
    rc = launch_contract(op->Np, pairs, npairs, glx, glw, q, cos_max, lambda_out, rho, R, op->nrows, mesh->nt,
                         dJ_dmu, reinterpret_cast<unsigned long long*>(glw + 64) + 1, st);
    if (rc) return rc;
  }
  if (dgvec) {
    explicit_term_kernel<<<(unsigned)((mesh->nt + 127) / 128), 128, 0, st>>>(dgvec, rho, R, op->nb, op->nrows,
                                                                              mesh->nt, dJ_dmu);
    DFM_LAUNCHED();
    DFM_CUDA_CHECK(cudaGetLastError());
  }
  return solve_rc;
}
