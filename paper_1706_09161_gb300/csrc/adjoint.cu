// Discrete adjoint of the time step and parameter gradients of a snapshot loss.
//
// With the parameters fixed, one time step of Algorithm 1 is linear in the
// populations f: C = <1|f>, F_mu = K_mu C along axis mu, feq = E(C, F) (Eqs. Feq,
// CoeffA_FADE3D), f* = f - Omega (f - feq) (Eqs. LBE_Ket / MRT-Coll), push streaming
// (Eq. Def_Translation) and the walls (Eq. Dirichlet_BC, affine).  Its transpose, in
// reverse order, with mu = dL/df(t+1):
//   walls      each known population b at a wall node z:  mu_b - (1/k) sum_{unknown u} mu_u
//   streaming  lambda*_q(y) = (walls^T mu)_q(y + e_q), 0 where y + e_q leaves the domain
//   collision  lambda_f = (I - Omega)^T lambda*,  lambda_feq = Omega^T lambda*
//   equilibrium lambda_C += lambda_feq_0 + sum_mu a_mu (lambda_feq_{2mu+1} - lambda_feq_{2mu+2})
//              lambda_F_mu = -w_0 lambda_feq_0 + w_i (lambda_feq_{2mu+1} + lambda_feq_{2mu+2})
//   operator   lambda_C += sum_mu K_mu^T lambda_F_mu   (the SIMT GEMM with K and K^T swapped)
//   moment     dL/df_q(t) = lambda_f_q + lambda_C (+ the snapshot residual 2 (C - obs)).
// Parameter gradients (sums over steps of lambda^T dA/dtheta f):
//   alpha_mu, p_mu : <dK_mu/dtheta, G_mu>,  G_mu[n][l] = sum_t sum_lines lambda_F(n) C_t(l)
//   D_mumu        : - sum lambda*^T (dOmega/dD_mumu) (f - feq)
//   u_mu          : sum (dt/dx)(w_i/e^2) C (lambda_feq_{2mu+1} - lambda_feq_{2mu+2})
// plus the initial condition f(0) = feq(C0, K C0).  Forward states are recomputed from
// checkpoints taken every `ckpt` steps, each kernel writing its slot of the segment; the last
// segment's states come from the forward pass itself.  A backward step is two launches: the
// step's adjoint and the operator's transpose.  Gradient sums are FP64, in FP32 forms those over a
// node's populations as pairs of floats; G_mu is one GEMM per checkpoint segment (FP32 forms:
// products summed in FP32 over 16 terms, then as pairs of floats in a block, which keep about 48
// bits, and in FP64 over blocks).  256^2, 300 steps, 10 snapshots, checkpoints every 100, through the Python call:
// 25.2 ms when slots were copied, the sums formed by passes of their own and G accumulated in
// FP64; 12.8 ms now.
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "lbm_internal.h"
#include "simt_dev.cuh"
#include "two_float.cuh"

namespace lbm {
namespace {

constexpr int kThreads = 256;

template <typename real>
struct AdjConst {
  int n[3];
  long long nodes;
  real omT[kMaxQ][kMaxQ];       // Omega^T
  // dOmega / dD_mumu = da db^T (MRT: rank one); BGK: a multiple of the identity, which the
  // host applies to the sum of lambda*^T (f - feq)
  int bgk;
  real da[3][kMaxQ], db[3][kMaxQ];
  real w0, wi;
  real advw[3];                 // dfeq_{2mu+1}/dC = (dt/dx) u_mu w_i / e^2
  real cu;                      // dfeq_{2mu+1}/du_mu per unit C = (dt/dx) w_i / e^2
};

__device__ __forceinline__ void evec(int q, int& ex, int& ey, int& ez) {
  ex = (q == 1) - (q == 2);
  ey = (q == 3) - (q == 4);
  ez = (q == 5) - (q == 6);
}

// dL/df of a later time, as the kernels that made it left it: dL/df_q = lf_q + r with
// r = lcl + sum_mu lcf_mu (+ the snapshot residual 2 (C - obs)), r the same for every q.
template <typename real>
struct LamIn {
  const real* lf;   // [q][node]
  const real* lcl;  // lambda_C of the equilibrium
  const real* lcf;  // [mu][node]: K_mu^T lambda_F_mu
  const real* C;    // concentration of that time and its observation (null: no snapshot)
  const real* obs;
};

template <typename real, int D>
__device__ __forceinline__ real lam_common(const LamIn<real>& in, long long nodes, long long node) {
  real r = in.lcl[node];
#pragma unroll
  for (int mu = 0; mu < D; ++mu) r += in.lcf[mu * nodes + node];
  if (in.obs) r += static_cast<real>(2) * (in.C[node] - in.obs[node]);
  return r;
}

// (1/k) sum of mu over the k unknown (wall-filled) populations of node (x, y, z); 0 inside
template <typename real, int D>
__device__ __forceinline__ real wall_nu(const AdjConst<real>& c, const real* __restrict__ lf, real r, long long node,
                                        int x, int y, int z) {
  constexpr int Q = 2 * D + 1;
  real s = static_cast<real>(0);
  int k = 0;
#pragma unroll
  for (int q = 1; q < Q; ++q) {
    int ex, ey, ez;
    evec(q, ex, ey, ez);
    const int sx = x - ex, sy = y - ey, sz = z - ez;
    if (sx < 0 || sx >= c.n[0] || sy < 0 || sy >= c.n[1] || sz < 0 || sz >= c.n[2]) {
      s += lf[q * c.nodes + node] + r;
      ++k;
    }
  }
  return k ? s / static_cast<real>(k) : static_cast<real>(0);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Adds the block's sums of v[0..K) to part[blockIdx.x * K + k] (fixed order, so repeated
// calls with the same grid accumulate deterministically).
template <int K>
__device__ __forceinline__ void block_accumulate(const double* v, double* __restrict__ part) {
  __shared__ double s[K][kThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const double w = warp_sum(v[k]);
    if (lane == 0) s[k][wid] = w;
  }
  __syncthreads();
  if (threadIdx.x < K) {
    double acc = 0.0;
    for (int i = 0; i < kThreads / 32; ++i) acc += s[threadIdx.x][i];
    part[blockIdx.x * K + threadIdx.x] += acc;
  }
}

// (sum of x[q] y[q]) z to FP64's precision: FP32 terms as an unevaluated pair of floats, products by
// FMA and sums by TwoSum (Ogita, Rump, Oishi 2005), which leaves the FP64 pipe one addition and two
// conversions
template <int Q>
__device__ __forceinline__ double wide_dot(const double* x, const double* y, double z) {
  double s = x[0] * y[0];
#pragma unroll
  for (int q = 1; q < Q; ++q) s += x[q] * y[q];
  return s * z;
}
template <int Q>
__device__ __forceinline__ double wide_dot(const float* x, const float* y, float z) {
  float hi = __fmul_rn(x[0], y[0]), lo = __fmaf_rn(x[0], y[0], -hi);
#pragma unroll
  for (int q = 1; q < Q; ++q) {
    const float p = __fmul_rn(x[q], y[q]), pe = __fmaf_rn(x[q], y[q], -p);
    float s, e;
    two_sum(hi, p, s, e);
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, pe));
  }
  const float p = __fmul_rn(hi, z), e = __fmaf_rn(lo, z, __fmaf_rn(hi, z, -p));
  return static_cast<double>(p) + (isfinite(p) ? static_cast<double>(e) : 0.0);
}

// Adds the warp's FP64 sums of v[0..K) to part[warp * K + k] (fixed order; the same grid
// accumulates deterministically over calls).  Each exchange halves the values a lane carries,
// so K = 4 takes 6 FP64 additions instead of 20: the pipe (a warp instruction holds it for 16
// clocks) is what these sums cost.
template <int K>
__device__ __forceinline__ void warp_accumulate(const double* val, double* __restrict__ part) {
  constexpr int P = K <= 4 ? 4 : 8;
  const int tid = threadIdx.x, lane = tid & 31;
  double v[P];
#pragma unroll
  for (int k = 0; k < P; ++k) v[k] = k < K ? val[k] : 0.0;
  int m = 16;
#pragma unroll
  for (int w = P / 2; w >= 1; w /= 2, m /= 2) {
    const bool up = lane & m;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const double keep = up ? v[j + w] : v[j], send = up ? v[j] : v[j + w];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, m);
    }
  }
#pragma unroll
  for (int o = 16 / P; o >= 1; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  const int k = lane / (32 / P);
  if (lane % (32 / P) == 0 && k < K)
    part[(blockIdx.x * (long long)(blockDim.x / 32) + tid / 32) * K + k] += v[0];
}

// One backward step: dL/df(t) of populations (lf, lcl and lambda_F; the operator's transpose
// follows) from dL/df(t + 1) and the forward state at t, and the step's part of the u and D
// gradients.  Bound by memory latency and the FP64 pipe; the sum lambda_f + lambda_C of the
// later step is formed on the fly for the node and its neighbours (cached reads), which saves
// a pass over the populations, and the FP64 work is three operations per summed value.
// 256^2, single cold-cache launches: 14.5 us and 3.4 us for the pass, now 9.9 us.
constexpr int kStepThreads = 128;

template <typename real, int D>
__global__ void __launch_bounds__(kStepThreads)
adj_step_kernel(const __grid_constant__ AdjConst<real> c, const real* __restrict__ f, const real* __restrict__ F,
                const __grid_constant__ LamIn<real> in, real* __restrict__ lf, real* __restrict__ lcl,
                real* __restrict__ lF, long long lFs, double* __restrict__ part) {
  constexpr int Q = 2 * D + 1;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // lcf comes from the previous kernel
  const long long nodes = c.nodes;
  const long long node = blockIdx.x * (long long)kStepThreads + threadIdx.x;
  double g[2 * D];
#pragma unroll
  for (int k = 0; k < 2 * D; ++k) g[k] = 0.0;
  if (node < nodes) {
    const int n0 = c.n[0], n1 = c.n[1];
    const int x = static_cast<int>(node % n0);
    const int y = static_cast<int>((node / n0) % n1);
    const int z = static_cast<int>(node / ((long long)n0 * n1));
    // forward state of this node
    real fv[Q], Fv[D];
#pragma unroll
    for (int q = 0; q < Q; ++q) fv[q] = f[q * nodes + node];
#pragma unroll
    for (int mu = 0; mu < D; ++mu) Fv[mu] = F[mu * nodes + node];
    // lambda* (adjoint of the post-collision populations of this node)
    real ls[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      int ex, ey, ez;
      evec(q, ex, ey, ez);
      const int tx = x + ex, ty = y + ey, tz = z + ez;
      if (tx < 0 || tx >= n0 || ty < 0 || ty >= n1 || tz < 0 || tz >= c.n[2]) {
        ls[q] = static_cast<real>(0);
      } else {
        const long long t = tx + (long long)n0 * (ty + (long long)n1 * tz);
        const real r = lam_common<real, D>(in, nodes, t);
        ls[q] = (in.lf[q * nodes + t] + r) - wall_nu<real, D>(c, in.lf, r, t, tx, ty, tz);
      }
    }
    real C = fv[0];
#pragma unroll
    for (int q = 1; q < Q; ++q) C += fv[q];
    real sumF = Fv[0];
#pragma unroll
    for (int mu = 1; mu < D; ++mu) sumF += Fv[mu];
    real dl[Q];  // f - feq
    dl[0] = fv[0] - (C - c.w0 * sumF);
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      const real a = c.wi * Fv[mu], b = c.advw[mu] * C;
      dl[2 * mu + 1] = fv[2 * mu + 1] - (a + b);
      dl[2 * mu + 2] = fv[2 * mu + 2] - (a - b);
    }
    // collision transpose
    real le[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      real acc = c.omT[i][0] * ls[0];
#pragma unroll
      for (int j = 1; j < Q; ++j) acc += c.omT[i][j] * ls[j];
      le[i] = acc;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) lf[q * nodes + node] = ls[q] - le[q];
    real lc = le[0];
#pragma unroll
    for (int mu = 0; mu < D; ++mu) lc += c.advw[mu] * (le[2 * mu + 1] - le[2 * mu + 2]);
    lcl[node] = lc;
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      lF[mu * lFs + node] = -c.w0 * le[0] + c.wi * (le[2 * mu + 1] + le[2 * mu + 2]);
      g[mu] = static_cast<double>(C) * static_cast<double>(le[2 * mu + 1] - le[2 * mu + 2]);
    }
    if (c.bgk) {
#pragma unroll
      for (int q = 0; q < Q; ++q) g[D] += static_cast<double>(ls[q]) * static_cast<double>(dl[q]);
    } else {
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        real b = c.db[mu][0] * dl[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) b += c.db[mu][q] * dl[q];
        g[D + mu] = wide_dot<Q>(c.da[mu], ls, b);
      }
    }
  }
  warp_accumulate<2 * D>(g, part);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// f(0) = feq(C0, K C0): lambda_F of the initial fractional terms and the u-gradient part
template <typename real, int D>
__global__ void __launch_bounds__(kStepThreads)
adj_init_kernel(const __grid_constant__ AdjConst<real> c, const real* __restrict__ C0,
                const __grid_constant__ LamIn<real> in, real* __restrict__ lF, double* __restrict__ part) {
  const long long nodes = c.nodes;
  const long long node = blockIdx.x * (long long)kStepThreads + threadIdx.x;
  double g[2 * D];
#pragma unroll
  for (int k = 0; k < 2 * D; ++k) g[k] = 0.0;
  if (node < nodes) {
    const real r = lam_common<real, D>(in, nodes, node);
    const real l0 = in.lf[node] + r;
    const real C = C0[node];
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      const real a = in.lf[(2 * mu + 1) * nodes + node] + r, b = in.lf[(2 * mu + 2) * nodes + node] + r;
      lF[mu * nodes + node] = -c.w0 * l0 + c.wi * (a + b);
      g[mu] = static_cast<double>(C) * static_cast<double>(a - b);
    }
  }
  warp_accumulate<2 * D>(g, part);
}

// G_mu[n][l] += sum_t sum_lines lambda_F_mu,t(line, n) C_t(line, l) over the steps of one
// checkpoint segment, as one SIMT GEMM whose reduction index runs over (step, line).
// The element (row n, reduction index jk = j * kin + k) of either operand sits at
// j * sj + n * ldn + k * ldk; the three axes map onto this as
//   x: ldn = 1,       ldk = n0, kin = steps * lines, nj = 1   (step stride nodes = lines * n0)
//   y: ldn = n0,      ldk = 1,  kin = n0, sj = n0 n1, nj = steps * n2
//   z: ldn = n0 n1,   ldk = 1,  kin = n0 n1, sj = nodes, nj = steps.
// Each block owns a 64x64 tile of G and one slice of the reduction index; partial sums go
// to their own slab and are added in slab order (deterministic).
struct GLayout {
  int side;
  int vec;  // quads of the reduction index (or of rows, x axis) never straddle and are aligned
  long long kin, sj, ldn, ldk, ktotal, kchunk;
};

constexpr int GB = 64, GK = 16;

template <typename real, bool NCONTIG>
__global__ void __launch_bounds__(256)
adj_G_gemm64(const GLayout L, const real* __restrict__ A, const real* __restrict__ B, double* __restrict__ part) {
  __shared__ real As[GK][GB + 4];
  __shared__ real Bs[GK][GB + 4];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int n0 = blockIdx.y * GB, l0 = blockIdx.x * GB;
  const long long kb = blockIdx.z * L.kchunk;
  const long long ke = min(kb + L.kchunk, L.ktotal);
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  constexpr int R = (GB * GK) / 256;
  // NCONTIG: consecutive threads walk the row index (contiguous); else the reduction index.
  // (j, k) of each loaded reduction index is stepped by GK per slice (no division in the loop)
  long long jj[R], kq[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = tid + r * 256;
    const long long jk = kb + (NCONTIG ? (e / GB) : (e % GK));
    jj[r] = jk / L.kin;
    kq[r] = jk - jj[r] * L.kin;
  }
  for (long long k0 = kb; k0 < ke; k0 += GK) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int e = tid + r * 256;
      const int rr = NCONTIG ? (e % GB) : (e / GK);
      const int kk = NCONTIG ? (e / GB) : (e % GK);
      real a = static_cast<real>(0), b = static_cast<real>(0);
      if (k0 + kk < ke) {
        const long long base = jj[r] * L.sj + kq[r] * L.ldk;
        if (n0 + rr < L.side) a = A[base + (long long)(n0 + rr) * L.ldn];
        if (l0 + rr < L.side) b = B[base + (long long)(l0 + rr) * L.ldn];
      }
      As[kk][rr] = a;
      Bs[kk][rr] = b;
      kq[r] += GK;
      while (kq[r] >= L.kin) {
        kq[r] -= L.kin;
        ++jj[r];
      }
    }
    __syncthreads();
    real sub[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sub[i][j] = static_cast<real>(0);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      real a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sub[i][j] += a[i] * b[j];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += static_cast<double>(sub[i][j]);
    __syncthreads();
  }
  double* slab = part + (size_t)blockIdx.z * L.side * L.side;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = n0 + ty + 16 * i;
    if (n >= L.side) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int l = l0 + tx + 16 * j;
      if (l < L.side) slab[(size_t)n * L.side + l] = acc[i][j];
    }
  }
}

// FP32 form of the same product: 64 x 32 tile of G per block of 64 threads, 8 x 4 outputs per
// thread, packed FMAs from swizzled shared memory (as the SIMT operator's kernel).  The
// products of one 16-deep slice are summed in FP32 and the slices' sums added to a pair of
// floats by TwoSum (Knuth), which keeps about 48 bits without the FP64 pipe: the conversions
// and additions of FP64 accumulators took eight times the FMAs' time.  Slabs hold the pairs.
// 256^2, 15 steps, both axes, single cold-cache launches: 570 us before, 105 us now.
constexpr int GM = 64, GN = 32;

template <bool NCONTIG>
__global__ void __launch_bounds__(64)
adj_G_gemm32(const GLayout L, const float* __restrict__ A, const float* __restrict__ B, float2* __restrict__ part) {
  constexpr int LA = GM * GK / 4 / 64, LB = GN * GK / 4 / 64;
  __shared__ __align__(16) float As[2][GK * GM];
  __shared__ __align__(16) float Bs[2][GK * GN];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int n0 = blockIdx.y * GM, l0 = blockIdx.x * GN;
  const long long kb = blockIdx.z * L.kchunk;
  const long long ke = min(kb + L.kchunk, L.ktotal);
  const bool vec = L.vec;
  // reduction index of a quad's first element as (j, k), stepped by GK per slice
  // (NCONTIG: rows are contiguous and j = 0 always)
  const int kq = 4 * (tid % (GK / 4));
  long long jj = 0, kk0 = kb + kq;
  if (!NCONTIG) {
    jj = kk0 / L.kin;
    kk0 -= jj * L.kin;
  }
  float4 ra[LA], rb[LB];
  auto quad = [&](const float* p, int row0, int e, int width, long long k0) -> float4 {
    if (NCONTIG) {  // four rows at one reduction index
      const long long k = k0 + e / (width / 4);
      const int row = row0 + 4 * (e % (width / 4));
      return load4(p + k * L.ldk + row, k < ke ? L.side - row : 0, vec);
    }
    const int row = row0 + e / (GK / 4);  // four reduction indices of one row
    const long long left = row < L.side ? ke - (k0 + kq) : 0;
    const float* q = p + row * L.ldn;
    if (vec) return load4(q + jj * L.sj + kk0, left < 4 ? (int)left : 4, true);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    long long j = jj, k = kk0;
    float* o = &v.x;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (u < left) o[u] = q[j * L.sj + k];
      if (++k == L.kin) {
        k = 0;
        ++j;
      }
    }
    return v;
  };
  auto fetch = [&](long long k0) {
#pragma unroll
    for (int i = 0; i < LA; ++i) ra[i] = quad(A, n0, tid + i * 64, GM, k0);
#pragma unroll
    for (int i = 0; i < LB; ++i) rb[i] = quad(B, l0, tid + i * 64, GN, k0);
    kk0 += GK;
    if (!NCONTIG)
      while (kk0 >= L.kin) {
        kk0 -= L.kin;
        ++jj;
      }
  };
  auto put = [&](float* s, const float4& v, int e, int width) {
    if (NCONTIG) {
      const int k = e / (width / 4);
      *reinterpret_cast<float4*>(s + k * width + ((4 * (e % (width / 4))) ^ (8 * (k / 4)))) = v;
    } else {
      const int q = e % (GK / 4);
      float* p = s + 4 * q * width + ((e / (GK / 4)) ^ (8 * q));
      p[0] = v.x;
      p[width] = v.y;
      p[2 * width] = v.z;
      p[3 * width] = v.w;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int i = 0; i < LA; ++i) put(As[buf], ra[i], tid + i * 64, GM);
#pragma unroll
    for (int i = 0; i < LB; ++i) put(Bs[buf], rb[i], tid + i * 64, GN);
  };
  unsigned long long hi[8][2], lo[8][2];  // rows 32 (i / 4) + 4 ty + i % 4, packed column pairs 4 tx + 2 j
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) hi[i][j] = lo[i][j] = 0ull;
  const unsigned long long m1 = twice(-1.0f);
  fetch(kb);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (long long k0 = kb; k0 < ke; k0 += GK) {
    const bool more = k0 + GK < ke;
    if (more) fetch(k0 + GK);
    unsigned long long sub[8][2];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) sub[i][j] = 0ull;
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      const int sw = 8 * (kk / 4);
      float4 a[2];
#pragma unroll
      for (int g = 0; g < 2; ++g) a[g] = *reinterpret_cast<const float4*>(&As[buf][kk * GM + 32 * g + ((4 * ty) ^ sw)]);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk * GN + ((4 * tx) ^ sw)]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 q = a[i / 4];
        const unsigned long long av = twice((i & 3) == 0 ? q.x : (i & 3) == 1 ? q.y : (i & 3) == 2 ? q.z : q.w);
        sub[i][0] = ffma2(av, b.x, sub[i][0]);
        sub[i][1] = ffma2(av, b.y, sub[i][1]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {  // TwoSum, differences as exact-product FMAs
        const unsigned long long h = hi[i][j], x = sub[i][j];
        const unsigned long long s = fadd2(h, x);
        const unsigned long long bp = ffma2(h, m1, s);
        const unsigned long long u = ffma2(ffma2(bp, m1, s), m1, h);
        lo[i][j] = fadd2(lo[i][j], fadd2(u, ffma2(bp, m1, x)));
        hi[i][j] = s;
      }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  float2* slab = part + (size_t)blockIdx.z * L.side * L.side;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int n = n0 + 32 * (i / 4) + 4 * ty + (i & 3);
    if (n >= L.side) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int l = l0 + 4 * tx + j, sh = 32 * (j & 1);
      if (l < L.side)
        slab[(size_t)n * L.side + l] = make_float2(__uint_as_float((unsigned)(hi[i][j / 2] >> sh)),
                                                   __uint_as_float((unsigned)(lo[i][j / 2] >> sh)));
    }
  }
}

__global__ void adj_G_reduce64(long long count, int nslab, const double* __restrict__ part, double* __restrict__ G) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int z = 0; z < nslab; ++z) acc += part[(size_t)z * count + i];
    G[i] += acc;
  }
}

// the slabs' pairs added in FP64, in slab order (a non-finite sum has no meaningful lo)
__global__ void adj_G_reduce32(long long count, int nslab, const float2* __restrict__ part, double* __restrict__ G) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int z = 0; z < nslab; ++z) {
      const float2 v = part[(size_t)z * count + i];
      acc += isfinite(v.x) ? static_cast<double>(v.x) + static_cast<double>(v.y) : static_cast<double>(v.x);
    }
    G[i] += acc;
  }
}

// slabs of the reduction split for one side x side G: enough blocks to fill the GPU (FP64: two
// of 256 threads per SM; FP32: six of 64), at least 1024 reduction indices per block
constexpr int kMaxSlabs = 64;

int g_slabs(int side, long long ktotal, bool f64) {
  const long long sms = device_sms();
  const long long tn = (side + (f64 ? GB : GN) - 1) / (f64 ? GB : GN), tm = (side + GB - 1) / GB;
  long long z = ((f64 ? 2 : 6) * sms + tm * tn - 1) / (tm * tn);
  z = std::min<long long>(z, std::max<long long>(1, ktotal / 1024));
  return static_cast<int>(std::max<long long>(1, std::min<long long>(z, kMaxSlabs)));
}

// reduction length of G_mu over `steps` steps
long long g_ktotal(const lbm_s* h, int mu, int steps) { return h->sp.nodes / h->sp.n[mu] * steps; }

// G_mu += sum over `steps` consecutive steps (operand step stride = nodes)
template <typename real>
cudaError_t accumulate_G(const lbm_s* h, int mu, int steps, const real* lF, const real* C, double* G, double* part,
                         cudaStream_t s) {
  const long long n0 = h->sp.n[0], n1 = h->sp.n[1];
  const long long nodes = h->sp.nodes;
  GLayout L{};
  L.side = h->sp.n[mu];
  L.ktotal = g_ktotal(h, mu, steps);
  if (mu == 0) {
    L.ldn = 1; L.ldk = n0; L.kin = L.ktotal; L.sj = 0;
  } else if (mu == 1) {
    L.ldn = n0; L.ldk = 1; L.kin = n0; L.sj = n0 * n1;
  } else {
    L.ldn = n0 * n1; L.ldk = 1; L.kin = n0 * n1; L.sj = nodes;
  }
  const bool aligned = reinterpret_cast<uintptr_t>(lF) % 16 == 0 && reinterpret_cast<uintptr_t>(C) % 16 == 0;
  L.vec = aligned && n0 % 4 == 0;  // rows, steps and reduction runs are then whole aligned quads
  const int nslab = g_slabs(L.side, L.ktotal, sizeof(real) == 8);
  L.kchunk = ((L.ktotal + nslab - 1) / nslab + GK - 1) / GK * GK;
  const int tm = (L.side + GB - 1) / GB;
  const long long count = (long long)L.side * L.side;
  const int rb = static_cast<int>(std::min<long long>((count + 255) / 256, 1216));
  if constexpr (sizeof(real) == 8) {
    const dim3 grid(tm, tm, nslab);
    if (mu == 0) adj_G_gemm64<real, true><<<grid, 256, 0, s>>>(L, lF, C, part);
    else adj_G_gemm64<real, false><<<grid, 256, 0, s>>>(L, lF, C, part);
    adj_G_reduce64<<<rb, 256, 0, s>>>(count, nslab, part, G);
  } else {
    const dim3 grid((L.side + GN - 1) / GN, tm, nslab);
    float2* pairs = reinterpret_cast<float2*>(part);
    if (mu == 0) adj_G_gemm32<true><<<grid, 64, 0, s>>>(L, lF, C, pairs);
    else adj_G_gemm32<false><<<grid, 64, 0, s>>>(L, lF, C, pairs);
    adj_G_reduce32<<<rb, 256, 0, s>>>(count, nslab, pairs, G);
  }
  return cudaGetLastError();
}

// sum (C - obs)^2 into *out (FP64; partial sums per block then one block)
template <typename real>
__global__ void __launch_bounds__(kThreads)
adj_loss_partials(long long nodes, const real* __restrict__ C, const real* __restrict__ obs, double* __restrict__ part) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < nodes; i += (long long)gridDim.x * kThreads) {
    const double r = static_cast<double>(C[i]) - static_cast<double>(obs[i]);
    acc += r * r;
  }
  double v[1] = {acc};
  // reuse the fixed-order block reduction on a zeroed slot
  if (threadIdx.x == 0) part[blockIdx.x] = 0.0;
  __syncthreads();
  block_accumulate<1>(v, part);
}

__global__ void __launch_bounds__(32) adj_sum_kernel(const double* __restrict__ part, int n, double* __restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) acc += part[i];
  acc = warp_sum(acc);
  if (threadIdx.x == 0) *out = acc;
}

template <typename real>
AdjConst<real> make_adj(const lbm_s* h, const double dOm[3][kMaxQ][kMaxQ]) {
  AdjConst<real> c{};
  for (int i = 0; i < 3; ++i) c.n[i] = h->sp.n[i];
  c.nodes = h->sp.nodes;
  for (int i = 0; i < kMaxQ; ++i)
    for (int j = 0; j < kMaxQ; ++j) c.omT[i][j] = static_cast<real>(h->sp.omega[j][i]);
  c.bgk = h->prm.collision == LBM_BGK;
  for (int mu = 0; mu < h->d && !c.bgk; ++mu) {
    // dOmega/dD_mumu = -M^-1 Lambda E_mu Lambda M is an outer product: its row and column
    // through the largest entry
    int i0 = 0, j0 = 0;
    for (int i = 0; i < h->Q; ++i)
      for (int j = 0; j < h->Q; ++j)
        if (std::fabs(dOm[mu][i][j]) > std::fabs(dOm[mu][i0][j0])) i0 = i, j0 = j;
    for (int i = 0; i < h->Q; ++i) {
      c.da[mu][i] = static_cast<real>(dOm[mu][i][j0] / dOm[mu][i0][j0]);
      c.db[mu][i] = static_cast<real>(dOm[mu][i0][i]);
    }
  }
  c.w0 = static_cast<real>(h->sp.w0);
  c.wi = static_cast<real>(h->sp.wi);
  for (int mu = 0; mu < 3; ++mu) c.advw[mu] = static_cast<real>(h->sp.adv[mu] * h->sp.wi);
  const double e2 = (h->d == 2) ? 1.0 / 3.0 : 1.0 / 4.0;
  c.cu = static_cast<real>((h->prm.dt / h->prm.dx) * h->sp.wi / e2);
  return c;
}

// the gradient's device buffers, from the handle's allocator, released on scope exit
// (after the handle's stream has drained)
struct Buffers {
  const lbm_s* h;
  std::vector<void*> ptrs;
  void* get(size_t bytes) {
    void* p = nullptr;
    if (dev_alloc(h, &p, bytes) != cudaSuccess) return nullptr;
    ptrs.push_back(p);
    return p;
  }
  ~Buffers() {
    if (!ptrs.empty() && h->stream) cudaStreamSynchronize(h->stream);
    for (void* p : ptrs) dev_free(h, p);
  }
};

template <typename real, int D>
int run_adjoint(lbm_s* h, const AdjHooks& hooks, int nsnap, const int* snaps, const double* obs_host, int ckpt,
                const double dOm[3][kMaxQ][kMaxQ], double* loss, double* G_host, double* gpart_host) {
  constexpr int Q = 2 * D + 1;
  cudaStream_t s = h->stream;
  const long long nodes = h->sp.nodes;
  const size_t E = sizeof(real);
  const int T = snaps[nsnap - 1];
  const int nck = T / ckpt + 1;
  const int seglen = ckpt < T ? ckpt : (T > 0 ? T : 1);
  const int nb = static_cast<int>((nodes + kThreads - 1) / kThreads);
  const int sb = static_cast<int>((nodes + kStepThreads - 1) / kStepThreads);  // blocks of a backward step
  const size_t gwarps = (size_t)sb * (kStepThreads / 32);
  Buffers B{h, {}};
  real* obs = static_cast<real*>(B.get(E * nodes * nsnap));
  real* ck = static_cast<real*>(B.get(E * Q * nodes * nck));
  real* sf = static_cast<real*>(B.get(E * Q * nodes * seglen));
  real* sF = static_cast<real*>(B.get(E * D * nodes * seglen));
  real* sC = static_cast<real*>(B.get(E * nodes * seglen));
  real* lf[2] = {static_cast<real*>(B.get(E * Q * nodes)), static_cast<real*>(B.get(E * Q * nodes))};
  real* lcl[2] = {static_cast<real*>(B.get(E * nodes)), static_cast<real*>(B.get(E * nodes))};
  real* Cb = static_cast<real*>(B.get(E * nodes));  // C at the end of the segment in hand
  // lambda_F of every step of a segment, [mu][step][node], for one G product per segment
  real* slF = static_cast<real*>(B.get(E * D * nodes * seglen));
  real* lcf = static_cast<real*>(B.get(E * D * nodes));
  size_t gsz = 0;
  for (int mu = 0; mu < D; ++mu) gsz += (size_t)h->sp.n[mu] * h->sp.n[mu];
  double* G = static_cast<double*>(B.get(sizeof(double) * gsz));
  size_t gslab = 0;
  for (int mu = 0; mu < D; ++mu)
    gslab = std::max(gslab, (size_t)g_slabs(h->sp.n[mu], g_ktotal(h, mu, seglen), sizeof(real) == 8) * h->sp.n[mu] * h->sp.n[mu]);
  double* Gpart = static_cast<double*>(B.get(sizeof(double) * gslab));
  double* gpart = static_cast<double*>(B.get(sizeof(double) * gwarps * 2 * D));
  double* lpart = static_cast<double*>(B.get(sizeof(double) * nb));
  double* lossd = static_cast<double*>(B.get(sizeof(double) * nsnap));
  if (!obs || !ck || !sf || !sF || !sC || !lf[0] || !lf[1] || !lcl[0] || !lcl[1] || !Cb || !slF || !lcf || !G || !Gpart || !gpart || !lpart ||
      !lossd)
    return LBM_ENOMEM;
#define CK(x)                                    \
  do {                                           \
    if ((x) != cudaSuccess) return LBM_ECUDA;    \
  } while (0)
  // observations in the working precision
  for (int k = 0; k < nsnap; ++k) {
    CK(cudaMemcpyAsync(h->dev.stage, obs_host + (size_t)k * nodes, sizeof(double) * nodes, cudaMemcpyHostToDevice, s));
    CK(launch_convert_in(h->dev.stage, obs + (size_t)k * nodes, (int)E, nodes, s));
    CK(cudaStreamSynchronize(s));
  }
  CK(cudaMemsetAsync(G, 0, sizeof(double) * gsz, s));
  CK(cudaMemsetAsync(gpart, 0, sizeof(double) * gwarps * 2 * D, s));
  CK(cudaMemsetAsync(lossd, 0, sizeof(double) * nsnap, s));
  const AdjConst<real> c = make_adj<real>(h, dOm);
  auto snap_index = [&](int t) {
    for (int k = 0; k < nsnap; ++k)
      if (snaps[k] == t) return k;
    return -1;
  };
  auto loss_at = [&](int k, const real* C) -> cudaError_t {
    adj_loss_partials<real><<<nb, kThreads, 0, s>>>(nodes, C, obs + (size_t)k * nodes, lpart);
    adj_sum_kernel<<<1, 32, 0, s>>>(lpart, nb, lossd + k);
    return cudaGetLastError();
  };

  // window maps of the segment's slots for the TMA-fed marches
  std::vector<CUtensorMap> maps(h->cs_plan ? 2 * (size_t)seglen : 0);
  for (size_t i = 0; i < maps.size() / 2; ++i)
    if (!cs_encode_slot(h, sf + i * Q * nodes, sF + i * D * nodes, &maps[2 * i], &maps[2 * i + 1])) return LBM_ECUDA;

  // steps t0 .. t1 - 1 from the populations f0 into the segment's slots, each kernel writing its
  // slot; with f_end also the step into t1 (C to Cb)
  auto run_segment = [&](int t0, int t1, const void* f0, void* f_end) -> int {
    CK(cudaMemcpyAsync(sf, f0, E * Q * nodes, cudaMemcpyDeviceToDevice, s));
    CK(launch_moment(h, sf, sC, s));
    for (int i = 0; i < t1 - t0; ++i) {
      const bool last = i + 1 == t1 - t0;
      real* F = sF + (size_t)i * D * nodes;
      CK(launch_frac_simt(h, sC + (size_t)i * nodes, F, s));
      if (last && !f_end) break;
      const CsSlot slot{F, maps.empty() ? nullptr : &maps[2 * i], maps.empty() ? nullptr : &maps[2 * i + 1]};
      CK(launch_collide_stream(h, sf + (size_t)i * Q * nodes, last ? f_end : sf + (size_t)(i + 1) * Q * nodes,
                               last ? Cb : sC + (size_t)(i + 1) * nodes, s, 0, &slot));
    }
    return LBM_OK;
  };

  // ---- forward pass from the initial state: checkpoints every ckpt steps, losses; the last
  // segment's steps stay in the slots
  int rc = hooks.reset(h);
  if (rc) return rc;
  int cur = h->cur;
  const int nseg = (T + ckpt - 1) / ckpt;
  const int tl = nseg > 0 ? (nseg - 1) * ckpt : 0;  // first step of the last segment
  for (int t = 0; t < tl; ++t) {
    if (t % ckpt == 0)
      CK(cudaMemcpyAsync(ck + (size_t)(t / ckpt) * Q * nodes, h->dev.f[cur], E * Q * nodes, cudaMemcpyDeviceToDevice, s));
    const int k0 = snap_index(t);
    if (k0 >= 0) CK(loss_at(k0, static_cast<const real*>(h->dev.C)));
    if ((rc = hooks.step(h, cur, s))) return rc;
  }
  if (T > 0) {
    if ((rc = run_segment(tl, T, h->dev.f[cur], h->dev.f[cur ^ 1]))) return rc;
    for (int t = tl; t < T; ++t)
      if (const int k0 = snap_index(t); k0 >= 0) CK(loss_at(k0, sC + (size_t)(t - tl) * nodes));
  } else {
    CK(cudaMemcpyAsync(Cb, h->dev.C, E * nodes, cudaMemcpyDeviceToDevice, s));
  }
  CK(loss_at(snap_index(T), Cb));

  // ---- backward, segment by segment; lambda(T) = 2 (C(T) - obs)
  int lc = 0;
  CK(cudaMemsetAsync(lf[0], 0, E * Q * nodes, s));
  CK(cudaMemsetAsync(lcl[0], 0, E * nodes, s));
  CK(cudaMemsetAsync(lcf, 0, E * D * nodes, s));
  auto lam_at = [&](int t, const real* C) {
    const int k = snap_index(t);
    return LamIn<real>{lf[lc], lcl[lc], lcf, C, k >= 0 ? obs + (size_t)k * nodes : nullptr};
  };
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sb);
  cfg.blockDim = dim3(kStepThreads);
  cfg.stream = s;
  cudaLaunchAttribute pdl[1];
  pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = pdl;
  cfg.numAttrs = 1;
  for (int seg = nseg - 1; seg >= 0; --seg) {
    const int t0 = seg * ckpt, t1 = std::min(t0 + ckpt, T);
    if (seg < nseg - 1) {
      CK(cudaMemcpyAsync(Cb, sC, E * nodes, cudaMemcpyDeviceToDevice, s));
      if ((rc = run_segment(t0, t1, ck + (size_t)seg * Q * nodes, nullptr))) return rc;
    }
    const long long lFs = (long long)seglen * nodes;
    for (int t = t1 - 1; t >= t0; --t) {
      const int i = t - t0;
      real* lFi = slF + (size_t)i * nodes;
      const LamIn<real> in = lam_at(t + 1, t + 1 == t1 ? Cb : sC + (size_t)(i + 1) * nodes);
      CK(cudaLaunchKernelEx(&cfg, adj_step_kernel<real, D>, c, (const real*)(sf + (size_t)i * Q * nodes),
                            (const real*)(sF + (size_t)i * D * nodes), in, lf[lc ^ 1], lcl[lc ^ 1], lFi, lFs, gpart));
      CK(launch_frac_simt_T(h, lFi, lFs, lcf, s));
      lc ^= 1;
    }
    size_t goff = 0;
    for (int mu = 0; mu < D; ++mu) {
      CK(accumulate_G<real>(h, mu, t1 - t0, slF + (size_t)mu * lFs, sC, G + goff, Gpart, s));
      goff += (size_t)h->sp.n[mu] * h->sp.n[mu];
    }
  }
  // ---- the initial condition f(0) = feq(C0, K C0)
  adj_init_kernel<real, D><<<sb, kStepThreads, 0, s>>>(c, static_cast<const real*>(h->dev.C0),
                                                       lam_at(0, T > 0 ? sC : Cb), slF, gpart);
  CK(cudaGetLastError());
  {
    size_t goff = 0;
    for (int mu = 0; mu < D; ++mu) {
      CK(accumulate_G<real>(h, mu, 1, slF + (size_t)mu * nodes, static_cast<const real*>(h->dev.C0), G + goff, Gpart,
                            s));
      goff += (size_t)h->sp.n[mu] * h->sp.n[mu];
    }
  }
  std::vector<double> lossv(nsnap);
  CK(cudaMemcpyAsync(lossv.data(), lossd, sizeof(double) * nsnap, cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(G_host, G, sizeof(double) * gsz, cudaMemcpyDeviceToHost, s));
  std::vector<double> gp(gwarps * 2 * D);
  CK(cudaMemcpyAsync(gp.data(), gpart, sizeof(double) * gp.size(), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
#undef CK
  double L = 0.0;
  for (double v : lossv) L += v;
  *loss = L;
  double sum[2 * D];
  for (int k = 0; k < 2 * D; ++k) {
    sum[k] = 0.0;
    for (size_t w = 0; w < gwarps; ++w) sum[k] += gp[w * 2 * D + k];
  }
  for (int mu = 0; mu < D; ++mu) {
    gpart_host[mu] = static_cast<double>(c.cu) * sum[mu];
    gpart_host[D + mu] = c.bgk ? -dOm[mu][0][0] * sum[D] : -sum[D + mu];
  }
  return LBM_OK;
}

}  // namespace

int adjoint_grad(lbm_s* h, const AdjHooks& hooks, int nsnap, const int* snaps, const double* obs, int ckpt,
                 const double dOm[3][kMaxQ][kMaxQ], double* loss, double* G, double* gsum) {
  if (h->elem == 8) {
    return (h->d == 2) ? run_adjoint<double, 2>(h, hooks, nsnap, snaps, obs, ckpt, dOm, loss, G, gsum)
                       : run_adjoint<double, 3>(h, hooks, nsnap, snaps, obs, ckpt, dOm, loss, G, gsum);
  }
  return (h->d == 2) ? run_adjoint<float, 2>(h, hooks, nsnap, snaps, obs, ckpt, dOm, loss, G, gsum)
                     : run_adjoint<float, 3>(h, hooks, nsnap, snaps, obs, ckpt, dOm, loss, G, gsum);
}

}  // namespace lbm
