// Fused equilibrium + collision + streaming + Dirichlet walls + new concentration.
//
// One launch performs the rest of Algorithm 1's time step after the fractional terms:
//           equilibrium   feq = A + (C/e^2)(dt/dx) u_mu |e_mu w>            Eqs. (Feq), (CoeffA_FADE3D)
//           collision     f* = f - Omega (f - feq)                          Eqs. (LBE_Ket), (MRT-Coll)
//           streaming     f_i(x + e_i, t+dt) = f*_i(x, t)                   Eq. (Def_Translation)
//           walls         f_b = C_wall - sum_{i != b} f_i                   Eq. (Dirichlet_BC)
//           moment        C = <1|f>
// Populations are stored after streaming and boundary treatment, so a CTA
// collides its nodes plus a one-node ring and gathers ("pulls") each population
// from the node it came from; the ring's collisions are recomputed by the
// neighbouring CTAs and their loads mostly hit L2.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "lbm_internal.h"
#include "tc_dev.cuh"
#include "two_float.cuh"

namespace lbm {
namespace {

template <int D> struct Lat;
template <> struct Lat<2> { static constexpr int Q = 5; };
template <> struct Lat<3> { static constexpr int Q = 7; };

// MRT change of basis, Eq. (MatrixD2): entry (i, q) of M for D2Q5 (D = 2) or D3Q7 (D = 3),
// and the squared norm of row i (the rows are orthogonal: M^-1 = M^T diag(1 / norm))
__host__ __device__ constexpr int mom(int D, int i, int q) {
  if (i == 0) return 1;
  if (i <= D) return q == 2 * i - 1 ? 1 : (q == 2 * i ? -1 : 0);  // flux moments
  if (D == 2) return i == 3 ? (q == 0 ? 4 : -1) : (q == 0 ? 0 : (q <= 2 ? 1 : -1));
  if (i == 4) return q == 0 ? 6 : -1;
  if (i == 5) return q == 0 ? 0 : (q <= 2 ? 2 : -1);
  return (q == 0 || q <= 2) ? 0 : (q <= 4 ? 1 : -1);
}
__host__ __device__ constexpr int mom_norm(int D, int i) {
  int n = 0;
  for (int q = 0; q < 2 * D + 1; ++q) n += mom(D, i, q) * mom(D, i, q);
  return n;
}
static_assert(mom_norm(2, 3) == 20 && mom_norm(3, 4) == 42 && mom_norm(3, 5) == 12 && mom_norm(3, 6) == 4,
              "moment rows of Eq. (MatrixD2)");

// Per-step constants in the working precision (no FP64 arithmetic per node on the
// FP32 forms; GB300's FP64 rate is a small fraction of its FP32 rate).
template <typename real>
struct KConst {
  int n[3];
  long long nodes;
  real omega[kMaxQ][kMaxQ];
  real w0, wi;
  real advw[3];  // (dt/dx) u_mu w_i / e^2
  real C_wall;
  int ksum;           // F holds ksum partial sums (split-K operator), added in order
  long long pstride;  // elements between partial sums
  real sfree[3];      // MRT rates of the free moments d+1..Q-1 over the squared norms of their rows of M
                      // (spatially varying coefficients)
};

// Coefficients that vary from node to node (lbm_set_fields), working precision, [k][node]:
//   coll: BGK 1/lambda(x); MRT the symmetric rate block R(x) = lambdabar(x)^-1 of the flux
//         moments, entries (00, 01, 11) in 2-D, (00, 01, 02, 11, 12, 22) in 3-D
//   advw: (dt/dx) u_mu(x) w_i / e^2, the advective factor of Eq. (Feq)
//   g:    g_mu(x); the kernel writes G_mu = g_mu(x) C(x), the operator's input along mu
//   src:  S(x) of a source S_c(x, t) = S(x) exp(rate t) (or null), added after the collision
//         as w_i S_c dt (Eq. LBE_Ket); cw: wall values C_w(x) of C_0(x, t) = C_w(x) exp(rate t)
//         (or null: the constant C_wall); tf: this launch's time factors, tf[0] =
//         exp(rate_S t) dt at the step's start t, tf[1] = exp(rate_w (t + dt)) at its end.
template <typename real>
struct FieldPtrs {
  const real* coll;
  const real* advw;
  const real* g;
  real* G;
  const real* src;
  const real* cw;
  const double* tf;
  // tensor-core forms with g(x): the operand parts of g_mu(x) C per axis ([mu][part], pitch
  // gldp), written in place of those of C
  void* gs[3][3];
  int gsplit;
  int gldp;
};

template <typename real>
KConst<real> make_const(const StepParams& sp) {
  KConst<real> k{};
  for (int i = 0; i < 3; ++i) k.n[i] = sp.n[i];
  k.nodes = sp.nodes;
  for (int i = 0; i < kMaxQ; ++i)
    for (int j = 0; j < kMaxQ; ++j) k.omega[i][j] = static_cast<real>(sp.omega[i][j]);
  k.w0 = static_cast<real>(sp.w0);
  k.wi = static_cast<real>(sp.wi);
  for (int i = 0; i < 3; ++i) k.advw[i] = static_cast<real>(sp.adv[i] * sp.wi);
  k.C_wall = static_cast<real>(sp.C_wall);
  k.ksum = sp.ksum;
  k.pstride = (sp.n[2] > 1 ? 3 : 2) * sp.nodes;
  const int d = sp.n[2] > 1 ? 3 : 2;
  for (int i = 0; i < d; ++i) k.sfree[i] = static_cast<real>(sp.sfree[i] / mom_norm(d, d + 1 + i));
  return k;
}

// F_mu at `node`: the sum of the operator's ksum partial sums, in order
template <typename real>
__device__ __forceinline__ real frac_term(const KConst<real>& sp, const real* __restrict__ F, int mu, long long node) {
  const real* p = F + (long long)mu * sp.nodes + node;
  real acc = p[0];
  for (int s = 1; s < sp.ksum; ++s) acc += p[s * sp.pstride];
  return acc;
}

// The FP32 collision matrix of a block's problem in shared memory, rows padded to 8: the
// grouped (batched) 2-D kernels stage it here and read each row in 128-bit loads
// (collide_node<float, 2, true, KS = true>).
__shared__ float4 s_om_rows[kMaxQ][2];

// Equilibrium and collision of one node.  f: populations (in), fs: post-collision (out).
// KS: the matrix is read from s_om_rows (same products in the same order: bit-identical).
template <typename real, int D, bool MRT, bool KS = false>
__device__ __forceinline__ void collide_node(const KConst<real>& sp, const real* f, const real* F, real* fs) {
  constexpr int Q = Lat<D>::Q;
  real C = f[0];
#pragma unroll
  for (int q = 1; q < Q; ++q) C += f[q];
  real sumF = F[0];
#pragma unroll
  for (int mu = 1; mu < D; ++mu) sumF += F[mu];
  real feq[Q];
  feq[0] = C - sp.w0 * sumF;
#pragma unroll
  for (int mu = 0; mu < D; ++mu) {
    const real a = sp.wi * F[mu];
    const real b = sp.advw[mu] * C;
    feq[2 * mu + 1] = a + b;
    feq[2 * mu + 2] = a - b;
  }
  if (!MRT) {
    const real om = sp.omega[0][0];
#pragma unroll
    for (int q = 0; q < Q; ++q) fs[q] = f[q] - om * (f[q] - feq[q]);
  } else {
    real dl[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) dl[q] = f[q] - feq[q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      real acc;
      if constexpr (KS) {
        static_assert(Q == 5 && sizeof(real) == 4, "rows of the 2-D FP32 matrix");
        const float4 a = s_om_rows[i][0];
        acc = a.x * dl[0];
        acc += a.y * dl[1];
        acc += a.z * dl[2];
        acc += a.w * dl[3];
        acc += s_om_rows[i][1].x * dl[4];
      } else {
        acc = sp.omega[i][0] * dl[0];
#pragma unroll
        for (int j = 1; j < Q; ++j) acc += sp.omega[i][j] * dl[j];
      }
      fs[i] = f[i] - acc;
    }
  }
}

// One node's coefficients (FieldPtrs): relaxation rate or rate block R, advective factors, source.
template <typename real, int D, bool MRT>
struct NodeCoef {
  static constexpr int NR = MRT ? D * (D + 1) / 2 : 1;
  real coll[NR], adv[D], src;
};

// MRT collision in moment space with the rates of the node: f* = f - M^-1 Lambda(x) M dl,
// dl = f - feq, Lambda(x) = diag(1, R(x), s_free) (Eqs. MRT-Coll, MatrixS, D_ab).  The squared
// norms of M's rows are in the rates (sfree) or powers of two; the conserved moment, dm[0], is
// rounding only.  No division: an FP32 one by 5 or 20 is a dozen instructions, an FP64 one a
// chain on the narrow FP64 pipe.
template <typename real, int D>
__device__ __forceinline__ void collide_moments(const KConst<real>& sp, const real* coll, const real* f, const real* dl,
                                                real* fs) {
  constexpr int Q = Lat<D>::Q;
  real dm[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    real acc = static_cast<real>(mom(D, i, 0)) * dl[0];
#pragma unroll
    for (int q = 1; q < Q; ++q)
      if (mom(D, i, q) != 0) acc += static_cast<real>(mom(D, i, q)) * dl[q];
    dm[i] = acc;
  }
  real dmp[Q];  // Lambda dm over the rows' norms
  dmp[0] = dm[0] * (static_cast<real>(1) / static_cast<real>(mom_norm(D, 0)));
#pragma unroll
  for (int a = 0; a < D; ++a) {
    real acc = static_cast<real>(0);
#pragma unroll
    for (int b = 0; b < D; ++b) {
      const int lo = a < b ? a : b, hi = a < b ? b : a;  // packed upper triangle, row by row
      const real t = coll[lo * D - lo * (lo - 1) / 2 + hi - lo];
      acc = b == 0 ? t * dm[1] : acc + t * dm[1 + b];
    }
    dmp[1 + a] = acc * static_cast<real>(0.5);
  }
#pragma unroll
  for (int k = D + 1; k < Q; ++k) dmp[k] = sp.sfree[k - D - 1] * dm[k];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    real acc = static_cast<real>(0);
#pragma unroll
    for (int i = 0; i < Q; ++i)
      if (mom(D, i, q) != 0) acc += static_cast<real>(mom(D, i, q)) * dmp[i];
    fs[q] = f[q] - acc;
  }
}

// Equilibrium and collision of one node with coefficients of that node:
// Eq. (Feq) with u(x); BGK f* = f - (f - feq)/lambda(x); MRT in moment space.
template <typename real, int D, bool MRT>
__device__ __forceinline__ void collide_node_field(const KConst<real>& sp, const FieldPtrs<real>& fp,
                                                   const NodeCoef<real, D, MRT>& c, const real* f, const real* F,
                                                   real* fs) {
  constexpr int Q = Lat<D>::Q;
  real C = f[0];
#pragma unroll
  for (int q = 1; q < Q; ++q) C += f[q];
  real sumF = F[0];
#pragma unroll
  for (int mu = 1; mu < D; ++mu) sumF += F[mu];
  real dl[Q];
  dl[0] = f[0] - (C - sp.w0 * sumF);
#pragma unroll
  for (int mu = 0; mu < D; ++mu) {
    const real a = sp.wi * F[mu];
    const real b = c.adv[mu] * C;
    dl[2 * mu + 1] = f[2 * mu + 1] - (a + b);
    dl[2 * mu + 2] = f[2 * mu + 2] - (a - b);
  }
  if (!MRT) {
    const real om = c.coll[0];
#pragma unroll
    for (int q = 0; q < Q; ++q) fs[q] = f[q] - om * dl[q];
  } else {
    collide_moments<real, D>(sp, c.coll, f, dl, fs);
  }
  if (fp.src) {  // |w> S_c(x, t) dt, Eq. (LBE_Ket)
    const real sv = c.src * static_cast<real>(fp.tf[0]);
    fs[0] += sp.w0 * sv;
#pragma unroll
    for (int q = 1; q < Q; ++q) fs[q] += sp.wi * sv;
  }
}

// Operands of the split-precision fractional operator, x-pitch ldp: bf16 parts C = hi + lo
// (SPLIT = 1) or hi + lo + lo2 (SPLIT = 3); tf32 (SPLIT = 2): C itself in hi (FP32).
struct SplitOut {
  void* hi;
  void* lo;
  int ldp;
  // tf32 on the TMA-fed marches: C again (FP32), regrouped along y (index 0) and z (index 1)
  // in groups of 4, the K-major operands of the y and z axes: element (x, y, z) at
  // thi[0][((z tg1 + y/4) tpx + x) 4 + y%4] and thi[1][((z/4 n1 + y) tpx + x) 4 + z%4]
  float* thi[2];
  int tg1;  // groups of 4 along y
  int tpx;  // x pitch (n0 rounded up to 16)
  void* lo2;  // bf16 with C in three parts (SPLIT = 3): the third part
};

// Per-problem entry of a grouped (batched) collide-stream launch.
struct BatchCS {
  KConst<float> k;
  const float* f[2];  // population buffers; the launch's parity picks input and output
  const float* F;
  float* C;
  SplitOut so;
  int* flag;
  double* mpart;              // the problem's mass partials, one per warp
  int v, strips, rows, items; // 2-D: strip march (StripGrid)
  int bx;                     // 3-D: tile columns in x
};

// SPLIT: 1 = bf16 hi + lo, 3 = bf16 in three parts (each the rounding of what the previous
// ones left: the three add up to C exactly), 2 = tf32: C itself in FP32 (the operator splits
// it into tf32 hi + lo in shared memory)
template <int SPLIT, typename real>
__device__ __forceinline__ void write_split(const SplitOut& so, long long o, real C) {
  const float c = static_cast<float>(C);
  if (SPLIT == 1 || SPLIT == 3) {
    const __nv_bfloat16 h = __float2bfloat16_rn(c);
    const float r1 = c - __bfloat162float(h);
    const __nv_bfloat16 l = __float2bfloat16_rn(r1);
    static_cast<__nv_bfloat16*>(so.hi)[o] = h;
    static_cast<__nv_bfloat16*>(so.lo)[o] = l;
    if (SPLIT == 3) static_cast<__nv_bfloat16*>(so.lo2)[o] = __float2bfloat16_rn(r1 - __bfloat162float(l));
  } else if (SPLIT == 2) {
    static_cast<float*>(so.hi)[o] = c;
  }
}

// Mass of the new concentration (the moment C = <1|f> of Algorithm 1), as a by-product of the step.
// Every thread adds the C it wrote; each warp reduces its threads' sums in a fixed order
// (xor shuffles: every lane ends with the same value) and lane 0 stores the warp's partial
// at part[slot * warps + warp]; the handle adds the partials of the latest step in one
// small fixed-order FP64 pass when asked (lbm_mass).  FP32 concentrations are carried as an
// unevaluated sum hi + lo of two floats, combined by TwoSum (Knuth), which keeps the sum
// exact up to the rounding of lo (of order u^2 per addition, u = 2^-24) without FP64
// arithmetic, and the partial is stored as the pair (hi, lo) in the 8-byte slot: the final
// pass forms hi + lo in FP64.  The FP64 pipe is narrow (a warp instruction on it holds an
// SM sub-partition for tens of cycles): the FP64 per-node sum had cost 3-12% of the
// collide-stream kernels, and even the three FP64 operations per warp of a double partial
// kept that pipe 11% busy at the tail of the 512^2 kernel.  FP64 concentrations are summed
// and stored in FP64.  No block-wide barrier.  part may be null (no partial wanted).
template <int WARPS = kMassSlots, typename real>
__device__ __forceinline__ void block_mass(SumAcc<real>& macc, double* part, int slot) {
  macc.warp_reduce();
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  if ((tid & 31) == 0 && part) macc.store(part + (long long)slot * WARPS + (tid >> 5));
}

// Thread block: 16 warps own a 32 x 16 tile of nodes (one node per thread, full
// 128-byte rows), and three more warps collide the one-node ring the pull needs: the
// x-ring (16 + 16 nodes, one warp) and the rows below and above (one warp each).
// The block marches along z through a chunk of planes, colliding every plane once; the
// in-plane movers (e_1..e_4) of the current plane go through shared memory, the z
// movers (e_5, e_6) stay in registers (previous plane's f*_5, next plane's f*_6).
// In 2-D the block handles one plane.  Each node is loaded ~1.19 times per step.
constexpr int TX = 32, TY = 16, HALO_WARPS = 3;
static_assert(kMassSlots * 32 == TX * (TY + HALO_WARPS), "one mass partial per warp of a block");

template <typename real, int D, bool MRT, bool FLD = false>
__device__ __forceinline__ void collide_at(const KConst<real>& sp, const real* __restrict__ f_in,
                                           const real* __restrict__ F, bool inside, long long node, real* fs,
                                           const FieldPtrs<real>& fp) {
  constexpr int Q = Lat<D>::Q;
  if (!inside) {
#pragma unroll
    for (int q = 0; q < Q; ++q) fs[q] = static_cast<real>(0);
    return;
  }
  const long long nodes = sp.nodes;
  real f[Q], Fv[D];
#pragma unroll
  for (int q = 0; q < Q; ++q) f[q] = f_in[q * nodes + node];
#pragma unroll
  for (int mu = 0; mu < D; ++mu) Fv[mu] = frac_term(sp, F, mu, node);
  if constexpr (FLD) {
    NodeCoef<real, D, MRT> c;
#pragma unroll
    for (int k = 0; k < NodeCoef<real, D, MRT>::NR; ++k) c.coll[k] = fp.coll[k * nodes + node];
#pragma unroll
    for (int mu = 0; mu < D; ++mu) c.adv[mu] = fp.advw[mu * nodes + node];
    c.src = fp.src ? fp.src[node] : static_cast<real>(0);
    collide_node_field<real, D, MRT>(sp, fp, c, f, Fv, fs);
  } else collide_node<real, D, MRT>(sp, f, Fv, fs);
}

// Asynchronous prefetch of the 2-D march (FP32): every thread copies the populations and
// fractional terms of its node in the next two tiles into its own column of a
// shared-memory ring (cp.async, 4 bytes each), so the loads of later tiles are in
// flight while the current one is processed.
constexpr int NT = TX * (TY + HALO_WARPS);
constexpr int PIPE_STAGES = 3;
constexpr int PIPE_VALS = 7;  // D2Q5: 5 populations + 2 fractional terms
constexpr int PIPE_SMEM = PIPE_STAGES * PIPE_VALS * NT * 4;

__device__ __forceinline__ void cp_async4(float* smem, const float* gmem) {
  const uint32_t sa = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}

// Programmatic dependent launch: let the next kernel of the stream be scheduled.  A grid
// that fits in one wave does this at block start (its dependents' prologues overlap it);
// a longer grid does it at block end, so that early dependents do not take SMs that its
// later waves need.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Warps of a block that owns a TXX x TYY tile: one thread per owned node and per ring node.
__host__ __device__ constexpr int march_warps(int txx, int tyy) { return (txx * tyy + 2 * (txx + tyy) + 31) / 32; }
static_assert(march_warps(TX, TY) == TY + HALO_WARPS, "32 x 16 tiles: 16 owner and 3 ring warps");

// One block's column (TXX x TYY tile bx, by; planes z0 .. z1-1) of one problem.
template <typename real, int D, bool MRT, int SPLIT, bool FLD = false, int TXX = TX, int TYY = TY>
__device__ __forceinline__ void march_body(const KConst<real>& sp, const real* __restrict__ f_in,
                                           const real* __restrict__ F, real* __restrict__ f_out,
                                           real* __restrict__ C_out, int* __restrict__ flag, const SplitOut& so,
                                           int bx, int by, int z0, int z1, double* mpart, int mslot,
                                           const FieldPtrs<real> fp = FieldPtrs<real>{}) {
  constexpr int Q = Lat<D>::Q;
  // movers of the current plane on the tile plus ring: [buffer][mover 1..4][y+1][x+1]
  __shared__ real s_m[2][4][TYY + 2][TXX + 2];
  const int n0 = sp.n[0], n1 = sp.n[1], n2 = sp.n[2];
  const long long nodes = sp.nodes;
  const long long plane = (long long)n0 * n1;
  const int tid = threadIdx.x + 32 * threadIdx.y, lane = threadIdx.x;
  const int x0 = bx * TXX, y0 = by * TYY;

  // the node this thread collides every plane, and where its movers go.  (The 3-D FP32 marches have 48
  // registers: a variable for the ring's side, kept through the planes, made the grouped one spill, 4
  // problems of 48^3 65 -> 80 us.)
  int gx, gy;
  const bool owner = TXX == 32 ? threadIdx.y < TYY : tid < TXX * TYY;
  const int ring = tid - TXX * TYY;
  if (owner) {
    gx = x0 + (TXX == 32 ? lane : tid % TXX);
    gy = y0 + (TXX == 32 ? (int)threadIdx.y : tid / TXX);
  } else if (ring < 2 * TYY) {
    gx = ring / TYY ? x0 + TXX : x0 - 1;
    gy = y0 + ring % TYY;
  } else {
    gx = x0 + (ring - 2 * TYY) % TXX;
    gy = ring < 2 * TYY + TXX ? y0 - 1 : y0 + TYY;
  }
  const int sx = gx - x0 + 1, sy = gy - y0 + 1;
  // programmatic dependent launch: the operator's F (and the previous step's f) must be
  // complete before any load
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr bool spare = march_warps(TXX, TYY) * 32 > TXX * TYY + 2 * (TXX + TYY);  // threads past the ring, idle
  const bool in_xy = (!spare || ring < 2 * (TXX + TYY)) && gx >= 0 && gx < n0 && gy >= 0 && gy < n1;
  const long long col = gx + (long long)n0 * gy;
  bool bad = false;
  SumAcc<real> macc;

  real cur[Q], nxt[Q];
  real prev5 = static_cast<real>(0);
  if (owner) {
    if (D == 3) {
      real t[Q];
      collide_at<real, D, MRT, FLD>(sp, f_in, F, in_xy && z0 > 0, col + (z0 - 1) * plane, t, fp);
      prev5 = t[5];
    }
    collide_at<real, D, MRT, FLD>(sp, f_in, F, in_xy, col + z0 * plane, cur, fp);
  }
  int buf = 0;
  for (int z = z0; z < z1; ++z) {
    if (owner) {
      if (D == 3) collide_at<real, D, MRT, FLD>(sp, f_in, F, in_xy && z + 1 < n2, col + (z + 1) * plane, nxt, fp);
      s_m[buf][0][sy][sx] = cur[1];
      s_m[buf][1][sy][sx] = cur[2];
      s_m[buf][2][sy][sx] = cur[3];
      s_m[buf][3][sy][sx] = cur[4];
    } else {
      real h[Q];
      collide_at<real, D, MRT, FLD>(sp, f_in, F, in_xy, col + z * plane, h, fp);
      // the ring: left and right columns, rows below and above, each moving into the tile
      if (ring < 2 * TYY) {
        if (ring < TYY) s_m[buf][0][sy][sx] = h[1];
        else s_m[buf][1][sy][sx] = h[2];
      } else if (ring < 2 * TYY + TXX) {
        s_m[buf][2][sy][sx] = h[3];
      } else if (!spare || ring < 2 * (TXX + TYY)) {
        s_m[buf][3][sy][sx] = h[4];
      }
    }
    __syncthreads();
    if (owner && in_xy) {
      real fv[Q];
      bool known[Q];
      fv[0] = cur[0];
      known[0] = true;
      known[1] = gx > 0;
      known[2] = gx + 1 < n0;
      known[3] = gy > 0;
      known[4] = gy + 1 < n1;
      fv[1] = s_m[buf][0][sy][sx - 1];
      fv[2] = s_m[buf][1][sy][sx + 1];
      fv[3] = s_m[buf][2][sy - 1][sx];
      fv[4] = s_m[buf][3][sy + 1][sx];
      if (D == 3) {
        known[5] = z > 0;
        known[6] = z + 1 < n2;
        fv[5] = prev5;
        fv[6] = nxt[6];
      }
      real sum_known = static_cast<real>(0);
      int n_unknown = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if (known[q]) {
          sum_known += fv[q];
        } else {
          fv[q] = static_cast<real>(0);
          ++n_unknown;
        }
      }
      real C = sum_known;
      if (n_unknown > 0) {
        // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit; the
        // wall value varies with position and time when given (Section 2.5)
        real cwall = sp.C_wall;
        if (FLD && fp.cw) cwall = fp.cw[col + z * plane] * static_cast<real>(fp.tf[1]);
        const real fill = (cwall - sum_known) / static_cast<real>(n_unknown);
#pragma unroll
        for (int q = 0; q < Q; ++q)
          if (!known[q]) fv[q] = fill;
        C = fv[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) C += fv[q];
      }
      const long long node = col + z * plane;
#pragma unroll
      for (int q = 0; q < Q; ++q) f_out[q * nodes + node] = fv[q];
      if (SPLIT == 0 || C_out) C_out[node] = C;
      if (SPLIT && FLD && fp.gsplit) {
#pragma unroll
        for (int mu = 0; mu < D; ++mu) {
          SplitOut sm{};
          sm.hi = fp.gs[mu][0];
          sm.lo = fp.gs[mu][1];
          sm.lo2 = fp.gs[mu][2];
          write_split<SPLIT>(sm, ((long long)z * n1 + gy) * fp.gldp + gx, fp.g[mu * nodes + node] * C);
        }
      } else if (SPLIT) {
        write_split<SPLIT>(so, ((long long)z * n1 + gy) * so.ldp + gx, C);
      }
      if (FLD && fp.G) {  // the SIMT operator's inputs of the next step: g_mu(x) C, one field per axis
#pragma unroll
        for (int mu = 0; mu < D; ++mu) fp.G[mu * nodes + node] = fp.g[mu * nodes + node] * C;
      }
      bad |= !isfinite(C);
      macc.add(C);
    }
    if (owner && D == 3) {
      prev5 = cur[5];
#pragma unroll
      for (int q = 0; q < Q; ++q) cur[q] = nxt[q];
    }
    buf ^= 1;
  }
  // one flag update per warp at most
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 1);
  block_mass<march_warps(TXX, TYY)>(macc, mpart, mslot);
}

// movers of the current tile plus ring for the 2-D FP32 marches: [buffer][mover 1..4][y+1][x+1]
// (one array per kernel, whichever 2-D march it runs)
__shared__ float s_m2[2][4][TY + 2][TX + 2];

// 2-D FP32: the block walks `ychunk` consecutive 32 x 16 tiles up the y axis (tile
// rows tr0 .. tr0 + ychunk - 1 of column bx), each thread prefetching its node of the
// next two tiles through the cp.async ring while the current tile is collided.  The
// per-tile work is that of march_body with one plane.
template <bool MRT, int SPLIT>
__device__ __forceinline__ void march2_pipe(const KConst<float>& sp, const float* __restrict__ f_in,
                                            const float* __restrict__ F, float* __restrict__ f_out,
                                            float* __restrict__ C_out, int* __restrict__ flag, const SplitOut& so,
                                            int ychunk, int bx, int byc, float* stage, double* mpart, int mslot) {
  constexpr int D = 2, Q = 5;
  auto& s_m = s_m2;
  const int n0 = sp.n[0], n1 = sp.n[1];
  const long long nodes = sp.nodes;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int tid = wy * TX + lane;
  const int tr0 = byc * ychunk;
  const int tr1 = min(tr0 + ychunk, (n1 + TY - 1) / TY);
  // this thread's node relative to the tile origin: owners, x-ring, rows below / above
  const bool owner = wy < TY;
  int dx, dy;
  if (owner) {
    dx = lane;
    dy = wy;
  } else if (wy == TY) {
    dx = (lane < 16) ? -1 : TX;
    dy = lane & 15;
  } else {
    dx = lane;
    dy = (wy == TY + 1) ? -1 : TY;
  }
  const int gx = bx * TX + dx;
  const int sx = dx + 1, sy = dy + 1;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const bool in_x = gx >= 0 && gx < n0;
  auto issue = [&](int tr, int slot) {
    const int gy = tr * TY + dy;
    if (in_x && gy >= 0 && gy < n1) {
      const long long node = gx + (long long)n0 * gy;
      float* st = stage + (size_t)slot * PIPE_VALS * NT + tid;
#pragma unroll
      for (int q = 0; q < Q; ++q) cp_async4(st + q * NT, f_in + q * nodes + node);
      if (sp.ksum == 1) {
#pragma unroll
        for (int mu = 0; mu < D; ++mu) cp_async4(st + (Q + mu) * NT, F + mu * nodes + node);
      }
    }
    cp_async_commit();
  };
  issue(tr0, 0);
  if (tr0 + 1 < tr1) issue(tr0 + 1, 1); else cp_async_commit();
  bool bad = false;
  SumAcc<float> macc;
  int buf = 0;
  for (int tr = tr0; tr < tr1; ++tr) {
    const int slot = (tr - tr0) % PIPE_STAGES;
    if (tr + 2 < tr1) issue(tr + 2, (tr - tr0 + 2) % PIPE_STAGES); else cp_async_commit();
    cp_async_wait<2>();  // this thread's copies for tile row tr have landed
    const int gy = tr * TY + dy;
    const bool inside = in_x && gy >= 0 && gy < n1;
    float fs[Q];
    if (inside) {
      const float* st = stage + (size_t)slot * PIPE_VALS * NT + tid;
      float fv[Q], Fv[D];
#pragma unroll
      for (int q = 0; q < Q; ++q) fv[q] = st[q * NT];
      if (sp.ksum == 1) {
#pragma unroll
        for (int mu = 0; mu < D; ++mu) Fv[mu] = st[(Q + mu) * NT];
      } else {  // split-K partials: summed here, in order
#pragma unroll
        for (int mu = 0; mu < D; ++mu) Fv[mu] = frac_term(sp, F, mu, gx + (long long)n0 * gy);
      }
      collide_node<float, D, MRT>(sp, fv, Fv, fs);
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) fs[q] = 0.f;
    }
    if (owner) {
      s_m[buf][0][sy][sx] = fs[1];
      s_m[buf][1][sy][sx] = fs[2];
      s_m[buf][2][sy][sx] = fs[3];
      s_m[buf][3][sy][sx] = fs[4];
    } else if (wy == TY) {
      if (lane < 16) s_m[buf][0][sy][sx] = fs[1];  // moves +x into the tile
      else s_m[buf][1][sy][sx] = fs[2];            // moves -x into the tile
    } else if (wy == TY + 1) {
      s_m[buf][2][sy][sx] = fs[3];                 // moves +y into the tile
    } else {
      s_m[buf][3][sy][sx] = fs[4];                 // moves -y into the tile
    }
    __syncthreads();
    if (owner && inside) {
      float fv[Q];
      bool known[Q];
      fv[0] = fs[0];
      known[0] = true;
      known[1] = gx > 0;
      known[2] = gx + 1 < n0;
      known[3] = gy > 0;
      known[4] = gy + 1 < n1;
      fv[1] = s_m[buf][0][sy][sx - 1];
      fv[2] = s_m[buf][1][sy][sx + 1];
      fv[3] = s_m[buf][2][sy - 1][sx];
      fv[4] = s_m[buf][3][sy + 1][sx];
      float sum_known = 0.f;
      int n_unknown = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if (known[q]) {
          sum_known += fv[q];
        } else {
          fv[q] = 0.f;
          ++n_unknown;
        }
      }
      float C = sum_known;
      if (n_unknown > 0) {
        // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit
        const float fill = (sp.C_wall - sum_known) / static_cast<float>(n_unknown);
#pragma unroll
        for (int q = 0; q < Q; ++q)
          if (!known[q]) fv[q] = fill;
        C = fv[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) C += fv[q];
      }
      const long long node = gx + (long long)n0 * gy;
#pragma unroll
      for (int q = 0; q < Q; ++q) f_out[q * nodes + node] = fv[q];
      if (SPLIT == 0 || C_out) C_out[node] = C;
      if (SPLIT) write_split<SPLIT>(so, (long long)gy * so.ldp + gx, C);
      bad |= !isfinite(C);
      macc.add(C);
    }
    buf ^= 1;
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 1);
  block_mass(macc, mpart, mslot);
}

// ---------------------------------------------------------------------------- 2-D FP32 strip march
// One warp owns a strip of 32 V nodes along x (V = 2 adjacent nodes per lane where rows are
// whole 8-byte pairs, else 1) and marches up a chunk of rows, colliding every row once: the y
// movers (e_3, e_4) stay in registers (previous row's f*_3, next row's f*_4), the x movers
// (e_1, e_2) go to the neighbouring lane by shuffle, and the strip's two ring columns are
// collided 16 rows at a time, one node per lane.  No shared memory, no barrier and no block:
// warps are independent, each with the next two rows' loads in flight.  A chunk of R rows
// collides (R + 2) / R + 1 / (32 V) of its nodes.  Serves the batches, where there are rows
// enough to keep every SM's warps busy (16 problems of 128^2 to 1024^2: 69 us with the TMA-fed
// blocks of 19 warps, 335 instructions per node; 59 us and 165 here); a single 512^2 lattice is a chain of
// latencies in which the TMA-fed blocks are the faster form (512^2 bf16x6 step 12.4 us against
// 13.4 us with strips of two rows).
template <int V, bool MRT, bool FLD>
struct StripRow {
  float f[5][V], F[2][V];
  float coll[MRT ? 3 : 1][V], adv[2][V], src[V];  // FLD
};

template <int V>
__device__ __forceinline__ void load_v(float (&d)[V], const float* __restrict__ p) {
  if constexpr (V == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    d[0] = t.x;
    d[1] = t.y;
  } else {
    d[0] = *p;
  }
}

template <int V>
__device__ __forceinline__ void store_v(float* __restrict__ p, const float (&d)[V]) {
  if constexpr (V == 2) *reinterpret_cast<float2*>(p) = make_float2(d[0], d[1]);
  else *p = d[0];
}

// the values of V neighbouring nodes from offset `o` on, zeros where !ok
template <int V, bool MRT, bool FLD>
__device__ __forceinline__ void strip_load(long long nodes, const float* __restrict__ f, const float* __restrict__ F,
                                           const FieldPtrs<float>& fp, long long o, bool ok,
                                           StripRow<V, MRT, FLD>& r) {
  constexpr int NR = MRT ? 3 : 1;
  if (ok) {
#pragma unroll
    for (int q = 0; q < 5; ++q) load_v<V>(r.f[q], f + q * nodes + o);
#pragma unroll
    for (int mu = 0; mu < 2; ++mu) load_v<V>(r.F[mu], F + mu * nodes + o);
    if constexpr (FLD) {
#pragma unroll
      for (int k = 0; k < NR; ++k) load_v<V>(r.coll[k], fp.coll + k * nodes + o);
#pragma unroll
      for (int mu = 0; mu < 2; ++mu) load_v<V>(r.adv[mu], fp.advw + mu * nodes + o);
      if (fp.src) load_v<V>(r.src, fp.src + o);
    }
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
      for (int q = 0; q < 5; ++q) r.f[q][v] = 0.f;
      r.F[0][v] = r.F[1][v] = 0.f;
      if constexpr (FLD) {
#pragma unroll
        for (int k = 0; k < NR; ++k) r.coll[k][v] = 0.f;
        r.adv[0][v] = r.adv[1][v] = r.src[v] = 0.f;
      }
    }
  }
}

// equilibrium and collision of the V nodes of a loaded row
template <int V, bool MRT, bool KS, bool FLD>
__device__ __forceinline__ void strip_collide(const KConst<float>& sp, const FieldPtrs<float>& fp,
                                              const StripRow<V, MRT, FLD>& r, float (&fs)[5][V]) {
#pragma unroll
  for (int v = 0; v < V; ++v) {
    float f[5], o[5];
    const float F[2] = {r.F[0][v], r.F[1][v]};
#pragma unroll
    for (int q = 0; q < 5; ++q) f[q] = r.f[q][v];
    if constexpr (FLD) {
      NodeCoef<float, 2, MRT> c;
#pragma unroll
      for (int k = 0; k < NodeCoef<float, 2, MRT>::NR; ++k) c.coll[k] = r.coll[k][v];
      c.adv[0] = r.adv[0][v];
      c.adv[1] = r.adv[1][v];
      c.src = r.src[v];
      collide_node_field<float, 2, MRT>(sp, fp, c, f, F, o);
    } else {
      collide_node<float, 2, MRT, KS>(sp, f, F, o);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) fs[q][v] = o[q];
  }
}

// operands of V neighbouring values at element o (write_split of each, packed stores)
template <int SPLIT, int V>
__device__ __forceinline__ void write_split_v(const SplitOut& so, long long o, const float (&c)[V]) {
  if constexpr (SPLIT == 2) {
    store_v<V>(static_cast<float*>(so.hi) + o, c);
  } else if constexpr (V == 1) {
    write_split<SPLIT>(so, o, c[0]);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(c[0], c[1]);
    const float r0 = c[0] - __low2float(h), r1 = c[1] - __high2float(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(r0, r1);
    *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(so.hi) + o) = h;
    *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(so.lo) + o) = l;
    if constexpr (SPLIT == 3)
      *reinterpret_cast<__nv_bfloat162*>(static_cast<__nv_bfloat16*>(so.lo2) + o) =
          __floats2bfloat162_rn(r0 - __low2float(l), r1 - __high2float(l));
  }
}

// the warp's strip (nodes x0 .. x0 + 32 V - 1), rows y0 .. y1 - 1; its mass partial to mpart[slot]
template <int V, bool MRT, int SPLIT, bool KS, bool FLD = false>
__device__ __forceinline__ void strip_march(const KConst<float>& sp, const float* __restrict__ f_in,
                                            const float* __restrict__ F, float* __restrict__ f_out,
                                            float* __restrict__ C_out, int* __restrict__ flag, const SplitOut& so,
                                            int x0, int y0, int y1, double* mpart, int slot,
                                            const FieldPtrs<float>& fp = FieldPtrs<float>{}) {
  const int n0 = sp.n[0], n1 = sp.n[1], lane = threadIdx.x & 31;
  const long long nodes = sp.nodes;
  const int gx = x0 + V * lane;
  const bool in_x = gx < n0;  // (n0 is a multiple of V)
  const bool side = x0 == 0 || x0 + 32 * V >= n0;
  StripRow<V, MRT, FLD> row[2];
  auto load = [&](int y, StripRow<V, MRT, FLD>& r) {
    strip_load(nodes, f_in, F, fp, (long long)y * n0 + gx, in_x && y >= 0 && y < n1, r);
  };
  load(y0 - 1, row[0]);
  load(y0, row[1]);
  // ring columns of rows yb .. yb + 15: lane r the left column's f*_1 of row yb + r, lane 16 + r
  // the right column's f*_2
  float h = 0.f;
  auto ring = [&](int yb) {
    const int hx = lane < 16 ? x0 - 1 : x0 + 32 * V, hy = yb + (lane & 15);
    StripRow<1, MRT, FLD> r;
    float o[5][1];
    strip_load(nodes, f_in, F, fp, (long long)hy * n0 + hx, hx >= 0 && hx < n0 && hy < y1, r);
    strip_collide<1, MRT, KS, FLD>(sp, fp, r, o);
    h = lane < 16 ? o[1][0] : o[2][0];
  };
  ring(y0);
  SumAcc<float> macc;
  float bad = 0.f;
  float c[4][V], p3[V];  // f*_0..3 of the last collided row, f*_3 of the one before
#pragma unroll
  for (int v = 0; v < V; ++v) c[0][v] = c[1][v] = c[2][v] = c[3][v] = p3[v] = 0.f;
  auto advance = [&](int y, StripRow<V, MRT, FLD>& r) {
    const int yo = y - 1;  // the row that is complete now
    float g[2][V];         // g_mu of that row
    if constexpr (FLD) {
      if (in_x && yo >= y0 && (fp.gsplit || fp.G)) {
#pragma unroll
        for (int mu = 0; mu < 2; ++mu) load_v<V>(g[mu], fp.g + mu * nodes + (long long)yo * n0 + gx);
      }
    }
    float n[5][V];
    strip_collide<V, MRT, KS, FLD>(sp, fp, r, n);
    if (y + 2 <= y1) load(y + 2, r);
    if (yo >= y0) {
      const int k = (yo - y0) & 15;
      if (yo > y0 && k == 0) ring(yo);
      const float hl = __shfl_sync(0xffffffffu, h, k), hr = __shfl_sync(0xffffffffu, h, 16 + k);
      const float up = __shfl_up_sync(0xffffffffu, c[1][V - 1], 1), dn = __shfl_down_sync(0xffffffffu, c[2][0], 1);
      float o[5][V], C[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        o[0][v] = c[0][v];
        o[1][v] = v == 0 ? (lane == 0 ? hl : up) : c[1][v > 0 ? v - 1 : 0];
        o[2][v] = v == V - 1 ? (lane == 31 ? hr : dn) : c[2][v < V - 1 ? v + 1 : 0];
        o[3][v] = p3[v];
        o[4][v] = n[4][v];
        C[v] = 0.f;
      }
      if (!side && yo > 0 && yo + 1 < n1) {  // no wall within reach (warp-uniform)
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int q = 0; q < 5; ++q) C[v] += o[q][v];
      } else {
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const bool known[5] = {true, gx + v > 0, gx + v + 1 < n0, yo > 0, yo + 1 < n1};
          int n_unknown = 0;
#pragma unroll
          for (int q = 0; q < 5; ++q) {
            if (known[q]) {
              C[v] += o[q][v];
            } else {
              o[q][v] = 0.f;
              ++n_unknown;
            }
          }
          if (n_unknown > 0) {
            // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit; the
            // wall value varies with position and time when given (Section 2.5)
            float cwall = sp.C_wall;
            if (FLD && fp.cw && in_x) cwall = fp.cw[(long long)yo * n0 + gx + v] * static_cast<float>(fp.tf[1]);
            const float fill = (cwall - C[v]) / static_cast<float>(n_unknown);
#pragma unroll
            for (int q = 0; q < 5; ++q)
              if (!known[q]) o[q][v] = fill;
            C[v] = o[0][v];
#pragma unroll
            for (int q = 1; q < 5; ++q) C[v] += o[q][v];
          }
        }
      }
      if (in_x) {
        const long long node = (long long)yo * n0 + gx;
#pragma unroll
        for (int q = 0; q < 5; ++q) store_v<V>(f_out + q * nodes + node, o[q]);
        if (SPLIT == 0 || C_out) store_v<V>(C_out + node, C);
        bool parts = SPLIT != 0;
        if constexpr (FLD) {
          if (fp.gsplit || fp.G) {  // the operator's inputs of the next step: g_mu(x) C, one per axis
#pragma unroll
            for (int mu = 0; mu < 2; ++mu) {
              float G[V];
#pragma unroll
              for (int v = 0; v < V; ++v) G[v] = g[mu][v] * C[v];
              if (fp.G) store_v<V>(fp.G + mu * nodes + node, G);
              if constexpr (SPLIT == 1 || SPLIT == 3) {
                SplitOut sm{};
                sm.hi = fp.gs[mu][0];
                sm.lo = fp.gs[mu][1];
                sm.lo2 = fp.gs[mu][2];
                if (fp.gsplit) write_split_v<SPLIT, V>(sm, (long long)yo * fp.gldp + gx, G);
              }
            }
          }
          if (fp.gsplit) parts = false;
        }
        if constexpr (SPLIT != 0)
          if (parts) write_split_v<SPLIT, V>(so, (long long)yo * so.ldp + gx, C);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          bad = __fmaf_rn(C[v], 0.f, bad);  // NaN once a C is not finite
          macc.add(C[v]);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      p3[v] = c[3][v];
#pragma unroll
      for (int q = 0; q < 4; ++q) c[q][v] = n[q][v];
    }
  };
  for (int y = y0 - 1; y <= y1; y += 2) {
    advance(y, row[0]);
    if (y + 1 <= y1) advance(y + 1, row[1]);
  }
  if (__any_sync(0xffffffffu, bad != 0.f) && lane == 0) atomicOr(flag, 1);
  macc.warp_reduce();
  if (lane == 0 && mpart) macc.store(mpart + slot);
}

// rows of a chunk: kStripRows per unit of the tunable chunk
constexpr int kStripRows = 2, kStripWarps = 4;

// how a 2-D problem's nodes are dealt to warps: item = chunk * strips + strip
struct StripGrid {
  int v, strips, rows, items;
};
StripGrid strip_grid(const int* n, int chunk) {
  StripGrid g;
  g.v = n[0] % 2 == 0 ? 2 : 1;
  g.strips = (n[0] + 32 * g.v - 1) / (32 * g.v);
  g.rows = std::min(kStripRows * std::min(chunk, n[1]), n[1]);  // (chunk may be any positive int)
  g.items = g.strips * ((n[1] + g.rows - 1) / g.rows);
  return g;
}

// linear index of this block in its grid (the slot of its mass partial)
__device__ __forceinline__ int block_linear() {
  return static_cast<int>(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z));
}

template <bool MRT, int SPLIT>
__global__ void __launch_bounds__(TX*(TY + HALO_WARPS), 2)
collide_stream_march2_kernel(const KConst<float> sp, const float* __restrict__ f_in, const float* __restrict__ F,
                             float* __restrict__ f_out, float* __restrict__ C_out, int* __restrict__ flag,
                             SplitOut so, int ychunk, int early, double* mpart) {
  extern __shared__ __align__(16) float pipe_stage[];
  if (early) pdl_trigger();
  march2_pipe<MRT, SPLIT>(sp, f_in, F, f_out, C_out, flag, so, ychunk, blockIdx.x, blockIdx.y, pipe_stage, mpart,
                          block_linear());
  if (!early) pdl_trigger();
}

// A single large 2-D FP32 lattice whose coefficients vary from node to node, on strips: 14 values
// in and 6 to 18 out per node, bound by the latency of its loads from L2.  Against one block of
// 32 x 16 nodes per tile: 512^2 bf16x6 step 17.6 -> 14.7 us, 1000 x 900 51.7 -> 40.5.
template <int V, bool MRT, int SPLIT>
__global__ void __launch_bounds__(32 * kStripWarps, 4)
collide_stream_fields2_kernel(const __grid_constant__ KConst<float> sp, const float* __restrict__ f_in,
                              const float* __restrict__ F, float* __restrict__ f_out, float* __restrict__ C_out,
                              int* __restrict__ flag, const __grid_constant__ SplitOut so,
                              const __grid_constant__ FieldPtrs<float> fp, const StripGrid g, int early,
                              double* mpart) {
  if (early) pdl_trigger();
  // programmatic dependent launch: the operator's F (and the previous step's f) must be
  // complete before any load
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int item = blockIdx.x * kStripWarps + (threadIdx.x >> 5);
  if (item < g.items) {
    const int y0 = item / g.strips * g.rows;
    strip_march<V, MRT, SPLIT, false, true>(sp, f_in, F, f_out, C_out, flag, so, item % g.strips * 32 * V, y0,
                                            min(y0 + g.rows, sp.n[1]), mpart, item, fp);
  }
  if (!early) pdl_trigger();
}

template <typename real, int D, bool MRT, int SPLIT, bool FLD = false, int TXX = TX, int TYY = TY>
__global__ void __launch_bounds__(32 * march_warps(TXX, TYY), sizeof(real) == 4 ? 2 : 1)
collide_stream_march_kernel(const KConst<real> sp, const real* __restrict__ f_in, const real* __restrict__ F,
                            real* __restrict__ f_out, real* __restrict__ C_out, int* __restrict__ flag, SplitOut so,
                            int nz, int early, double* mpart, const FieldPtrs<real> fp = FieldPtrs<real>{}) {
  // z chunk blockIdx.z of nz (boundaries bz * n2 / nz): concurrent blocks march the same
  // z window, so the ring loads of neighbouring columns hit L2
  const int n2 = sp.n[2];
  const int bz = blockIdx.z;
  const int z0 = static_cast<int>((long long)bz * n2 / nz), z1 = static_cast<int>((long long)(bz + 1) * n2 / nz);
  if (early) pdl_trigger();
  march_body<real, D, MRT, SPLIT, FLD, TXX, TYY>(sp, f_in, F, f_out, C_out, flag, so, blockIdx.x, blockIdx.y, z0, z1,
                                                 mpart, block_linear(), fp);
  if (!early) pdl_trigger();
}

// ---------------------------------------------------------------------------- TMA-fed 3-D march
// FP32 forms with n0 % 4 == 0, bound by HBM: per plane, one thread loads the block's 40 x 18
// window of all Q populations and all d fractional terms (tile, one-node ring, x aligned down
// to a 16-byte boundary) with two 4-D TMA box loads into a 3-stage shared-memory ring, up to
// three planes ahead of the plane being collided.  Nodes outside the domain arrive as zeros
// (TMA out-of-bounds fill), which the collision maps to zero movers, exactly as the plain march
// treats them.  Measured against one node per thread (608 threads, two barriers per plane, two
// planes ahead, 410 instructions per node) with its z chunks: 256^3 bf16x6 231 -> 209 us (1315 MB
// with C, which a call's last step stores: 93% of the measured copy rate), tf32x3 247 -> 227, 160 x 128 x 100 43 -> 33.
constexpr int TW = TX + 8, TH = TY + 2;  // staged window: x from x0 - 4, y from y0 - 1
constexpr int TMA_STAGES = 3;
constexpr uint32_t TMA_F_BYTES = 7u * TH * TW * 4;   // D3Q7 populations
constexpr uint32_t TMA_FF_BYTES = 3u * TH * TW * 4;  // fractional terms
constexpr uint32_t TMA_TX = TMA_F_BYTES + TMA_FF_BYTES;  // bytes landing per plane
constexpr uint32_t TMA_FF_OFF = (TMA_F_BYTES + 127) / 128 * 128;  // 128-byte aligned box starts
constexpr uint32_t TMA_STAGE = (TMA_FF_OFF + TMA_FF_BYTES + 127) / 128 * 128;
constexpr size_t TMA_SMEM = (size_t)TMA_STAGES * TMA_STAGE + 128 /*align*/ + 64 /*barriers*/;
constexpr long long kTmaWaitNs = 2000000000LL;

struct CsPlan {
  CUtensorMap f[2];  // populations, dims (n0, n1, n2, Q), box (TW, TH, 1, Q)
  CUtensorMap F;     // fractional terms, dims (n0, n1, n2, d), box (TW, TH, 1, d)
};

__device__ __forceinline__ uint32_t cs_smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool cs_mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(cs_smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait: false (and bit 2 of the flag) after kTmaWaitNs of %globaltimer
__device__ __forceinline__ bool cs_mbar_wait(uint64_t* bar, uint32_t parity, int* flag) {
  if (cs_mbar_try(bar, parity)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (cs_mbar_try(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > (unsigned long long)kTmaWaitNs) {
      atomicOr(flag, 2);
      return false;
    }
  }
}

__device__ __forceinline__ void cs_tma_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(cs_smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(cs_smem_u32(bar))
      : "memory");
}

// Two x-neighbours per thread: 8 owner warps (a half-warp per row of the tile), one warp of
// ring pairs (the rows below and above) and one of single ring nodes (the columns left and
// right).  x movers go to the neighbouring lane by shuffle, y movers through shared memory in
// three buffers (one barrier per plane: a buffer is rewritten only after the next plane's
// barrier), z movers stay in registers.
constexpr int T3_WARPS = TX * TY / 64 + 2;

template <bool MRT, int SPLIT>
__global__ void __launch_bounds__(32 * T3_WARPS, 2)
collide_stream_tma3_kernel(const __grid_constant__ KConst<float> sp, const __grid_constant__ CUtensorMap map_f,
                           const __grid_constant__ CUtensorMap map_F, float* __restrict__ f_out,
                           float* __restrict__ C_out, int* __restrict__ flag, const __grid_constant__ SplitOut so, int nz,
                           int early, double* mpart) {
  constexpr int D = 3, Q = 7;
  extern __shared__ uint8_t cs_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(cs_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)TMA_STAGES * TMA_STAGE);
  __shared__ __align__(8) float s_up[3][TY + 1][TX];  // f*_3 of row r - 1 at [r]
  __shared__ __align__(8) float s_dn[3][TY + 1][TX];  // f*_4 of row r at [r]
  __shared__ float s_x[3][2][TY];                     // f*_1 of the left column, f*_2 of the right one
  // tf32: C of the last two planes, the source of the copy regrouped along y
  __shared__ __align__(8) float s_c[SPLIT == 2 ? 2 : 1][SPLIT == 2 ? TY : 1][TX];
  const bool wT = SPLIT == 2 && so.thi[0] != nullptr;
  const int n0 = sp.n[0], n1 = sp.n[1], n2 = sp.n[2];
  const long long nodes = sp.nodes;
  const long long plane = (long long)n0 * n1;
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int bz = blockIdx.z;
  const int z0 = static_cast<int>((long long)bz * n2 / nz), z1 = static_cast<int>((long long)(bz + 1) * n2 / nz);
  if (early) pdl_trigger();

  const bool owner = warp < TX * TY / 64;
  const int xp = 2 * (lane & 15), row = 2 * warp + (lane >> 4);  // owner's place in the tile
  const int gx = x0 + xp, gy = y0 + row;
  // place in the staged window: owners and row ring pairs (x aligned to 8 bytes), column ring nodes
  int lx = xp + 4, ly = row + 1;
  if (warp == T3_WARPS - 2) ly = lane < 16 ? 0 : TY + 1;
  if (warp == T3_WARPS - 1) {
    lx = lane < 16 ? 3 : TX + 4;
    ly = (lane & 15) + 1;
  }
  const float* win = reinterpret_cast<const float*>(ring) + ly * TW + lx;

  // plane p lives in stage (p - z0 + 1) % 3; its k-th use of that stage completes phase k
  auto stage_of = [&](int p) { return (p - z0 + 1) % TMA_STAGES; };
  auto parity_of = [&](int p) { return static_cast<uint32_t>(((p - z0 + 1) / TMA_STAGES) & 1); };
  auto issue = [&](int p) {
    const int s = stage_of(p);
    uint8_t* st = ring + (size_t)s * TMA_STAGE;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(cs_smem_u32(&full[s])),
                 "r"(TMA_TX)
                 : "memory");
    cs_tma_4d(st, &map_f, x0 - 4, y0 - 1, p, 0, &full[s]);
    cs_tma_4d(st + TMA_FF_OFF, &map_F, x0 - 4, y0 - 1, p, 0, &full[s]);
  };
  auto collide_pair = [&](int p, float (&fs)[2][Q]) {
    cs_mbar_wait(&full[stage_of(p)], parity_of(p), flag);
    const float* st = win + stage_of(p) * (TMA_STAGE / 4);
    float fv[2][Q], Fv[2][D];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const float2 t = *reinterpret_cast<const float2*>(st + q * (TH * TW));
      fv[0][q] = t.x;
      fv[1][q] = t.y;
    }
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      const float2 t = *reinterpret_cast<const float2*>(st + TMA_FF_OFF / 4 + mu * (TH * TW));
      Fv[0][mu] = t.x;
      Fv[1][mu] = t.y;
    }
    collide_node<float, D, MRT>(sp, fv[0], Fv[0], fs[0]);
    collide_node<float, D, MRT>(sp, fv[1], Fv[1], fs[1]);
  };
  // plane p's movers into buffer b; the owners' populations stay in fs
  auto movers = [&](int p, int b, float (&fs)[2][Q]) {
    if (owner) {
      collide_pair(p, fs);
      *reinterpret_cast<float2*>(&s_up[b][row + 1][xp]) = make_float2(fs[0][3], fs[1][3]);
      *reinterpret_cast<float2*>(&s_dn[b][row][xp]) = make_float2(fs[0][4], fs[1][4]);
    } else if (p >= z1) {
      return;  // only the owners' f*_6 of the plane past the chunk is needed
    } else if (warp == T3_WARPS - 2) {
      float h[2][Q];
      collide_pair(p, h);
      if (lane < 16) *reinterpret_cast<float2*>(&s_up[b][0][xp]) = make_float2(h[0][3], h[1][3]);  // moves +y into the tile
      else *reinterpret_cast<float2*>(&s_dn[b][TY][xp]) = make_float2(h[0][4], h[1][4]);           // moves -y into it
    } else {
      cs_mbar_wait(&full[stage_of(p)], parity_of(p), flag);
      const float* st = win + stage_of(p) * (TMA_STAGE / 4);
      float fv[Q], Fv[D], h[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) fv[q] = st[q * (TH * TW)];
#pragma unroll
      for (int mu = 0; mu < D; ++mu) Fv[mu] = st[TMA_FF_OFF / 4 + mu * (TH * TW)];
      collide_node<float, D, MRT>(sp, fv, Fv, h);
      s_x[b][lane >> 4][lane & 15] = lane < 16 ? h[1] : h[2];  // moves +x, -x into the tile
    }
  };

  if (tid == 0) {
    for (int s = 0; s < TMA_STAGES; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cs_smem_u32(&full[s])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // programmatic dependent launch: f and F come from the previous kernels
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0) {
    issue(z0 - 1);
    issue(z0);
    issue(z0 + 1);  // z0 + 1 <= z1: needed by the owners' first iteration
  }
  SumAcc<float> macc;
  float bad = 0.f;
  float c[2][Q], p5[2] = {0.f, 0.f};  // plane z: f*_q of this pair; f*_5 of plane z - 1
  float tz[2][4] = {};                // tf32: C of the current group of four planes
#pragma unroll
  for (int v = 0; v < 2; ++v)
#pragma unroll
    for (int q = 0; q < Q; ++q) c[v][q] = 0.f;
  if (owner) {
    collide_pair(z0 - 1, c);
    p5[0] = c[0][5];
    p5[1] = c[1][5];
  }
  movers(z0, 0, c);
  __syncthreads();  // planes z0 - 1 and z0 are read: their stages take z0 + 2 and z0 + 3
  if (tid == 0) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (z0 + 2 <= z1) issue(z0 + 2);
    if (z0 + 3 <= z1) issue(z0 + 3);
  }
  // tf32: plane p of s_c to the copy regrouped along y: 32 x 4 groups of 16 bytes
  auto flush_y = [&](int p) {
    const int x = tid & 31, yq = 4 * (tid >> 5);
    if (tid < 4 * TX && x0 + x < n0 && y0 + yq < n1) {
      const float* r = &s_c[p & 1][SPLIT == 2 ? yq : 0][x];
      const long long o = (((long long)p * so.tg1 + ((y0 + yq) >> 2)) * so.tpx + x0 + x) * 4;
      *reinterpret_cast<float4*>(so.thi[0] + o) = make_float4(r[0], r[TX], r[2 * TX], r[3 * TX]);
    }
  };
  const bool in_xy = gx < n0 && gy < n1;  // (owners; n0 is a multiple of 4)
  const bool side = x0 == 0 || x0 + TX >= n0 || y0 == 0 || y0 + TY >= n1;
  const unsigned off = static_cast<unsigned>(gy * n0 + gx);
  int b = 0;
  for (int z = z0; z < z1; ++z) {
    float n[2][Q];
    const int bn = b == 2 ? 0 : b + 1;
    movers(z + 1, bn, n);
    __syncthreads();
    // plane z + 1 is read by everyone: its stage takes plane z + 4
    if (tid == 0 && z + 4 <= z1) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(z + 4);
    }
    if (SPLIT == 2 && wT && z > z0) flush_y(z - 1);
    if (owner) {
      const float up = __shfl_up_sync(0xffffffffu, c[1][1], 1), dn = __shfl_down_sync(0xffffffffu, c[0][2], 1);
      const float2 y3 = *reinterpret_cast<const float2*>(&s_up[b][row][xp]);
      const float2 y4 = *reinterpret_cast<const float2*>(&s_dn[b][row + 1][xp]);
      float o[2][Q], C[2] = {0.f, 0.f};
      o[0][0] = c[0][0];
      o[1][0] = c[1][0];
      o[0][1] = xp == 0 ? s_x[b][0][row] : up;
      o[1][1] = c[0][1];
      o[0][2] = c[1][2];
      o[1][2] = xp == TX - 2 ? s_x[b][1][row] : dn;
      o[0][3] = y3.x;
      o[1][3] = y3.y;
      o[0][4] = y4.x;
      o[1][4] = y4.y;
      o[0][5] = p5[0];
      o[1][5] = p5[1];
      o[0][6] = n[0][6];
      o[1][6] = n[1][6];
      if (!side && z > 0 && z + 1 < n2) {  // no wall within reach (block-uniform)
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int q = 0; q < Q; ++q) C[v] += o[v][q];
      } else {
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const bool known[Q] = {true, gx + v > 0, gx + v + 1 < n0, gy > 0, gy + 1 < n1, z > 0, z + 1 < n2};
          int n_unknown = 0;
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            if (known[q]) {
              C[v] += o[v][q];
            } else {
              o[v][q] = 0.f;
              ++n_unknown;
            }
          }
          if (n_unknown > 0) {
            // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit
            const float fill = (sp.C_wall - C[v]) / static_cast<float>(n_unknown);
#pragma unroll
            for (int q = 0; q < Q; ++q)
              if (!known[q]) o[v][q] = fill;
            C[v] = o[v][0];
#pragma unroll
            for (int q = 1; q < Q; ++q) C[v] += o[v][q];
          }
        }
      }
      if (in_xy) {
        float* fz = f_out + z * plane;
#pragma unroll
        for (int q = 0; q < Q; ++q) *reinterpret_cast<float2*>(fz + q * nodes + off) = make_float2(o[0][q], o[1][q]);
        if (SPLIT == 0 || C_out) *reinterpret_cast<float2*>(C_out + z * plane + off) = make_float2(C[0], C[1]);
        if constexpr (SPLIT == 2) {
          *reinterpret_cast<float2*>(static_cast<float*>(so.hi) + ((long long)z * n1 + gy) * so.ldp + gx) =
              make_float2(C[0], C[1]);
        } else if constexpr (SPLIT != 0) {
          write_split_v<SPLIT, 2>(so, ((long long)z * n1 + gy) * so.ldp + gx, C);
        }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          bad = __fmaf_rn(C[v], 0.f, bad);  // NaN once a C is not finite
          macc.add(C[v]);
        }
      } else {
        C[0] = C[1] = 0.f;  // zero outside the domain
      }
      if (SPLIT == 2 && wT) {
        *reinterpret_cast<float2*>(&s_c[z & 1][SPLIT == 2 ? row : 0][xp]) = make_float2(C[0], C[1]);
        // z copy: each node's group of four planes, or the part of it that lies in this chunk
        const int k = z & 3;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (j == k) {
            tz[0][j] = C[0];
            tz[1][j] = C[1];
          }
        if (in_xy && (k == 3 || z + 1 == z1)) {
          const int first = max(z0 - (z & ~3), 0);
          float* t = so.thi[1] + (((long long)(z >> 2) * n1 + gy) * so.tpx + gx) * 4;
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            if (first == 0 && k == 3) {
              *reinterpret_cast<float4*>(t + 4 * v) = make_float4(tz[v][0], tz[v][1], tz[v][2], tz[v][3]);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j >= first && j <= k) t[4 * v + j] = tz[v][j];
            }
          }
        }
      }
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        p5[v] = c[v][5];
#pragma unroll
        for (int q = 0; q < Q; ++q) c[v][q] = n[v][q];
      }
    }
    b = bn;
  }
  if (SPLIT == 2 && wT) {
    __syncthreads();
    flush_y(z1 - 1);
  }
  // every issued plane (up to z1) was waited for by the owners; after a timeout make sure
  // no copy is still in flight into this block's shared memory before it exits
  if (tid == 0)
    for (int p = (z1 - 2 > z0 - 1 ? z1 - 2 : z0 - 1); p <= z1; ++p) cs_mbar_wait(&full[stage_of(p)], parity_of(p), flag);
  if (__any_sync(0xffffffffu, bad != 0.f) && lane == 0) atomicOr(flag, 1);
  block_mass<T3_WARPS>(macc, mpart, block_linear());
  if (!early) pdl_trigger();
}

// ---------------------------------------------------------------------------- TMA-fed 2-D march
// FP32 forms with n0 % 4 == 0: the block walks `ychunk` tiles up y; per tile one thread
// loads the 40 x 18 window of the 5 populations and the 2 fractional terms with two 3-D
// TMA box loads into a 3-stage ring, two tiles ahead.
constexpr uint32_t TMA2_F_BYTES = 5u * TH * TW * 4;
constexpr uint32_t TMA2_FF_OFF = (TMA2_F_BYTES + 127) / 128 * 128;
// with ks split-K partial sums the fractional-term window holds 2 ks planes; two stages
// then (the ring must leave room for two blocks per SM up to ks = 4)
__host__ __device__ constexpr uint32_t tma2_ff_bytes(int ks) { return 2u * ks * TH * TW * 4; }
__host__ __device__ constexpr uint32_t tma2_stage(int ks) {
  return (TMA2_FF_OFF + tma2_ff_bytes(ks) + 127) / 128 * 128;
}
__host__ __device__ constexpr int tma2_nst(int ks) { return ks > 1 ? 2 : TMA_STAGES; }
__host__ __device__ constexpr size_t tma2_smem(int ks) {
  return (size_t)tma2_nst(ks) * tma2_stage(ks) + 128 /*align*/ + 64 /*barriers*/;
}

__device__ __forceinline__ void cs_tma_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(cs_smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(cs_smem_u32(bar))
      : "memory");
}

// The collide-stream phase of the fused step (blocks of 32 x 19 threads, one node per thread).
template <bool MRT>
__device__ __forceinline__ void march2_tma(const KConst<float>& sp, const CUtensorMap* map_f,
                                           const CUtensorMap* map_F, float* __restrict__ f_out,
                                           float* __restrict__ C_out, int* __restrict__ flag, const SplitOut& so,
                                           int ychunk, int bx, int byc, uint8_t* raw, double* mpart, int mslot) {
  constexpr int D = 2, Q = 5;
  auto& s_m = s_m2;
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 127) & ~uintptr_t(127));
  const int ks = sp.ksum;
  const int nst = tma2_nst(ks);
  const uint32_t stg = tma2_stage(ks);
  const uint32_t tx = TMA2_F_BYTES + tma2_ff_bytes(ks);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)nst * stg);
  const int n0 = sp.n[0], n1 = sp.n[1];
  const long long nodes = sp.nodes;
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int tid = wy * TX + lane;
  const int x0 = bx * TX;
  const int tr0 = byc * ychunk;
  const int tr1 = min(tr0 + ychunk, (n1 + TY - 1) / TY);
  const bool owner = wy < TY;
  int dx, dy;
  if (owner) {
    dx = lane;
    dy = wy;
  } else if (wy == TY) {
    dx = (lane < 16) ? -1 : TX;
    dy = lane & 15;
  } else {
    dx = lane;
    dy = (wy == TY + 1) ? -1 : TY;
  }
  const int gx = x0 + dx;
  const int sx = dx + 1, sy = dy + 1;
  const int lx = dx + 4, ly = dy + 1;  // position in the staged window
  const bool in_x = gx >= 0 && gx < n0;
  auto stage_of = [&](int t) { return (t - tr0) % nst; };
  auto parity_of = [&](int t) { return static_cast<uint32_t>(((t - tr0) / nst) & 1); };
  auto issue = [&](int t) {
    const int s = stage_of(t);
    uint8_t* st = ring + (size_t)s * stg;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(cs_smem_u32(&full[s])), "r"(tx)
                 : "memory");
    cs_tma_3d(st, map_f, x0 - 4, t * TY - 1, 0, &full[s]);
    cs_tma_3d(st + TMA2_FF_OFF, map_F, x0 - 4, t * TY - 1, 0, &full[s]);
  };
  if (tid == 0) {
    for (int s = 0; s < nst; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cs_smem_u32(&full[s])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");  // f and F come from the previous kernels
  if (tid == 0)
    for (int t = tr0; t < tr1 && t < tr0 + nst; ++t) issue(t);
  bool bad = false;
  SumAcc<float> macc;
  int buf = 0;
  for (int tr = tr0; tr < tr1; ++tr) {
    cs_mbar_wait(&full[stage_of(tr)], parity_of(tr), flag);
    const float* st = reinterpret_cast<const float*>(ring + (size_t)stage_of(tr) * stg);
    float fs[Q];
    {
      float fv[Q], Fv[D];
#pragma unroll
      for (int q = 0; q < Q; ++q) fv[q] = st[(q * TH + ly) * TW + lx];
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        // planes of the window: partial s of axis mu at plane s * D + mu, added in order of s
        float acc = st[TMA2_FF_OFF / 4 + (mu * TH + ly) * TW + lx];
        for (int k = 1; k < ks; ++k) acc += st[TMA2_FF_OFF / 4 + ((k * D + mu) * TH + ly) * TW + lx];
        Fv[mu] = acc;
      }
      collide_node<float, D, MRT>(sp, fv, Fv, fs);
    }
    if (owner) {
      s_m[buf][0][sy][sx] = fs[1];
      s_m[buf][1][sy][sx] = fs[2];
      s_m[buf][2][sy][sx] = fs[3];
      s_m[buf][3][sy][sx] = fs[4];
    } else if (wy == TY) {
      if (lane < 16) s_m[buf][0][sy][sx] = fs[1];  // moves +x into the tile
      else s_m[buf][1][sy][sx] = fs[2];            // moves -x into the tile
    } else if (wy == TY + 1) {
      s_m[buf][2][sy][sx] = fs[3];                 // moves +y into the tile
    } else {
      s_m[buf][3][sy][sx] = fs[4];                 // moves -y into the tile
    }
    __syncthreads();
    // tile row tr is read by everyone: its stage takes tile row tr + nst
    if (tid == 0 && tr + nst < tr1) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(tr + nst);
    }
    const int gy = tr * TY + dy;
    if (owner && in_x && gy < n1) {
      float fv[Q];
      bool known[Q];
      fv[0] = fs[0];
      known[0] = true;
      known[1] = gx > 0;
      known[2] = gx + 1 < n0;
      known[3] = gy > 0;
      known[4] = gy + 1 < n1;
      fv[1] = s_m[buf][0][sy][sx - 1];
      fv[2] = s_m[buf][1][sy][sx + 1];
      fv[3] = s_m[buf][2][sy - 1][sx];
      fv[4] = s_m[buf][3][sy + 1][sx];
      float C = 0.f;
      if (x0 > 0 && x0 + TX < n0 && tr * TY > 0 && tr * TY + TY < n1) {  // no wall within reach (block-uniform)
#pragma unroll
        for (int q = 0; q < Q; ++q) C += fv[q];
      } else {
        int n_unknown = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          if (known[q]) {
            C += fv[q];
          } else {
            fv[q] = 0.f;
            ++n_unknown;
          }
        }
        if (n_unknown > 0) {
          // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit
          const float fill = (sp.C_wall - C) / static_cast<float>(n_unknown);
#pragma unroll
          for (int q = 0; q < Q; ++q)
            if (!known[q]) fv[q] = fill;
          C = fv[0];
#pragma unroll
          for (int q = 1; q < Q; ++q) C += fv[q];
        }
      }
      const long long node = gx + (long long)n0 * gy;
#pragma unroll
      for (int q = 0; q < Q; ++q) f_out[q * nodes + node] = fv[q];
      C_out[node] = C;
      write_split<1>(so, (long long)gy * so.ldp + gx, C);
      bad |= !isfinite(C);
      macc.add(C);
    }
    buf ^= 1;
  }
  // after a timeout no copy may still be landing in this block's shared memory
  if (tid == 0) {
    for (int t = (tr1 - nst > tr0 ? tr1 - nst : tr0); t < tr1; ++t)
      cs_mbar_wait(&full[stage_of(t)], parity_of(t), flag);
    for (int s = 0; s < nst; ++s)  // the barrier words may hold other data afterwards
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(cs_smem_u32(&full[s])) : "memory");
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 1);
  block_mass(macc, mpart, mslot);
}

// The two-kernel step's form: two x-neighbours per thread, warps as in collide_stream_tma3_kernel.
// A 512^2 lattice sits in L2: the kernel is a chain of window load, collision and stores, in which
// the instructions per node count (one node per thread, 19 warps: 335).  512^2 bf16x6 step 12.5 ->
// 11.2 us, FP32 23.2 -> 22.4.
template <bool MRT, int SPLIT>
__global__ void __launch_bounds__(32 * T3_WARPS, 2)
collide_stream_tma2_kernel(const __grid_constant__ KConst<float> sp, const __grid_constant__ CUtensorMap map_f,
                           const __grid_constant__ CUtensorMap map_F, float* __restrict__ f_out,
                           float* __restrict__ C_out, int* __restrict__ flag, const __grid_constant__ SplitOut so,
                           int ychunk, int early, double* mpart) {
  constexpr int D = 2, Q = 5;
  extern __shared__ uint8_t cs_raw2[];
  __shared__ __align__(8) float s_up[2][TY + 1][TX];  // f*_3 of row r - 1 at [r]
  __shared__ __align__(8) float s_dn[2][TY + 1][TX];  // f*_4 of row r at [r]
  __shared__ float s_x[2][2][TY];                     // f*_1 of the left column, f*_2 of the right one
  // tf32: C of the last two tile rows (slot t & 1), the source of the copy regrouped along y
  __shared__ __align__(8) float s_c[SPLIT == 2 ? 2 : 1][SPLIT == 2 ? TY : 1][TX];
  if (early) pdl_trigger();
  const bool wT = SPLIT == 2 && so.thi[0] != nullptr;
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(cs_raw2) + 127) & ~uintptr_t(127));
  const int ks = sp.ksum;
  const int nst = tma2_nst(ks);
  const uint32_t stg = tma2_stage(ks);
  const uint32_t tx = TMA2_F_BYTES + tma2_ff_bytes(ks);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)nst * stg);
  const int n0 = sp.n[0], n1 = sp.n[1];
  const long long nodes = sp.nodes;
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int x0 = blockIdx.x * TX;
  const int tr0 = blockIdx.y * ychunk;
  const int tr1 = min(tr0 + ychunk, (n1 + TY - 1) / TY);
  const bool owner = warp < TX * TY / 64;
  const int xp = 2 * (lane & 15), row = 2 * warp + (lane >> 4);  // owner's place in the tile
  const int gx = x0 + xp;
  // place in the staged window: owners and row ring pairs (x aligned to 8 bytes), column ring nodes
  int lx = xp + 4, ly = row + 1;
  if (warp == T3_WARPS - 2) ly = lane < 16 ? 0 : TY + 1;
  if (warp == T3_WARPS - 1) {
    lx = lane < 16 ? 3 : TX + 4;
    ly = (lane & 15) + 1;
  }
  const float* win = reinterpret_cast<const float*>(ring) + ly * TW + lx;
  auto stage_of = [&](int t) { return (t - tr0) % nst; };
  auto parity_of = [&](int t) { return static_cast<uint32_t>(((t - tr0) / nst) & 1); };
  auto issue = [&](int t) {
    const int s = stage_of(t);
    uint8_t* st = ring + (size_t)s * stg;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(cs_smem_u32(&full[s])), "r"(tx)
                 : "memory");
    cs_tma_3d(st, &map_f, x0 - 4, t * TY - 1, 0, &full[s]);
    cs_tma_3d(st + TMA2_FF_OFF, &map_F, x0 - 4, t * TY - 1, 0, &full[s]);
  };
  // tf32: tile row t to the y copy (element (x, y) at thi[0][(y/4 tpx + x) 4 + y%4]): warp w < 4
  // writes y group 4t + w for the tile's 32 x (512 contiguous bytes)
  auto flush_y = [&](int t) {
    const int yq = 4 * warp;
    if (warp < TY / 4 && x0 + lane < n0 && t * TY + yq < n1) {
      const float* r = &s_c[t & 1][SPLIT == 2 ? yq : 0][lane];
      const long long o = ((long long)((t * TY + yq) >> 2) * so.tpx + x0 + lane) * 4;
      *reinterpret_cast<float4*>(so.thi[0] + o) = make_float4(r[0], r[TX], r[2 * TX], r[3 * TX]);
    }
  };
  if (tid == 0) {
    for (int s = 0; s < nst; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(cs_smem_u32(&full[s])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");  // f and F come from the previous kernels
  if (tid == 0)
    for (int t = tr0; t < tr1 && t < tr0 + nst; ++t) issue(t);
  SumAcc<float> macc;
  float bad = 0.f;
  int b = 0;
  for (int tr = tr0; tr < tr1; ++tr, b ^= 1) {
    cs_mbar_wait(&full[stage_of(tr)], parity_of(tr), flag);
    const float* st = win + stage_of(tr) * (stg / 4);
    const float* sF = st + TMA2_FF_OFF / 4;  // partial k of axis mu at plane k * D + mu, added in order of k
    float fs[2][Q];
    if (warp < T3_WARPS - 1) {
      float fv[2][Q], Fv[2][D];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float2 t = *reinterpret_cast<const float2*>(st + q * (TH * TW));
        fv[0][q] = t.x;
        fv[1][q] = t.y;
      }
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        float2 t = *reinterpret_cast<const float2*>(sF + mu * (TH * TW));
        for (int k = 1; k < ks; ++k) {
          const float2 u = *reinterpret_cast<const float2*>(sF + (k * D + mu) * (TH * TW));
          t.x += u.x;
          t.y += u.y;
        }
        Fv[0][mu] = t.x;
        Fv[1][mu] = t.y;
      }
      collide_node<float, D, MRT>(sp, fv[0], Fv[0], fs[0]);
      collide_node<float, D, MRT>(sp, fv[1], Fv[1], fs[1]);
      if (owner || lane < 16)  // moves +y: the tile's rows, and the row below into the tile
        *reinterpret_cast<float2*>(&s_up[b][owner ? row + 1 : 0][xp]) = make_float2(fs[0][3], fs[1][3]);
      if (owner || lane >= 16)  // moves -y: the tile's rows, and the row above into the tile
        *reinterpret_cast<float2*>(&s_dn[b][owner ? row : TY][xp]) = make_float2(fs[0][4], fs[1][4]);
    } else {
      float fv[Q], Fv[D], h[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) fv[q] = st[q * (TH * TW)];
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        Fv[mu] = sF[mu * (TH * TW)];
        for (int k = 1; k < ks; ++k) Fv[mu] += sF[(k * D + mu) * (TH * TW)];
      }
      collide_node<float, D, MRT>(sp, fv, Fv, h);
      s_x[b][lane >> 4][lane & 15] = lane < 16 ? h[1] : h[2];  // moves +x, -x into the tile
    }
    __syncthreads();
    // tile row tr is read by everyone: its stage takes tile row tr + nst
    if (tid == 0 && tr + nst < tr1) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(tr + nst);
    }
    if (SPLIT == 2 && wT && tr > tr0) flush_y(tr - 1);  // its slot is rewritten only after the next barrier
    if (owner) {
      const int gy = tr * TY + row;
      const float up = __shfl_up_sync(0xffffffffu, fs[1][1], 1), dn = __shfl_down_sync(0xffffffffu, fs[0][2], 1);
      const float2 y3 = *reinterpret_cast<const float2*>(&s_up[b][row][xp]);
      const float2 y4 = *reinterpret_cast<const float2*>(&s_dn[b][row + 1][xp]);
      float o[2][Q], C[2] = {0.f, 0.f};
      o[0][0] = fs[0][0];
      o[1][0] = fs[1][0];
      o[0][1] = xp == 0 ? s_x[b][0][row] : up;
      o[1][1] = fs[0][1];
      o[0][2] = fs[1][2];
      o[1][2] = xp == TX - 2 ? s_x[b][1][row] : dn;
      o[0][3] = y3.x;
      o[1][3] = y3.y;
      o[0][4] = y4.x;
      o[1][4] = y4.y;
      if (x0 > 0 && x0 + TX < n0 && tr * TY > 0 && tr * TY + TY < n1) {  // no wall within reach (block-uniform)
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int q = 0; q < Q; ++q) C[v] += o[v][q];
      } else {
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const bool known[Q] = {true, gx + v > 0, gx + v + 1 < n0, gy > 0, gy + 1 < n1};
          int n_unknown = 0;
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            if (known[q]) {
              C[v] += o[v][q];
            } else {
              o[v][q] = 0.f;
              ++n_unknown;
            }
          }
          if (n_unknown > 0) {
            // Eq. (Dirichlet_BC); with k unknown populations each takes 1/k of the deficit
            const float fill = (sp.C_wall - C[v]) / static_cast<float>(n_unknown);
#pragma unroll
            for (int q = 0; q < Q; ++q)
              if (!known[q]) o[v][q] = fill;
            C[v] = o[v][0];
#pragma unroll
            for (int q = 1; q < Q; ++q) C[v] += o[v][q];
          }
        }
      }
      if (gx < n0 && gy < n1) {  // (n0 is a multiple of 4)
        const long long node = gx + (long long)n0 * gy;
#pragma unroll
        for (int q = 0; q < Q; ++q) *reinterpret_cast<float2*>(f_out + q * nodes + node) = make_float2(o[0][q], o[1][q]);
        if (SPLIT == 0 || C_out) *reinterpret_cast<float2*>(C_out + node) = make_float2(C[0], C[1]);
        if constexpr (SPLIT != 0) write_split_v<SPLIT, 2>(so, (long long)gy * so.ldp + gx, C);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          bad = __fmaf_rn(C[v], 0.f, bad);  // NaN once a C is not finite
          macc.add(C[v]);
        }
      } else {
        C[0] = C[1] = 0.f;  // zero outside the domain
      }
      if (SPLIT == 2 && wT)
        *reinterpret_cast<float2*>(&s_c[tr & 1][SPLIT == 2 ? row : 0][xp]) = make_float2(C[0], C[1]);
    }
  }
  if (SPLIT == 2 && wT) {
    __syncthreads();
    flush_y(tr1 - 1);
  }
  // every issued tile row was waited for by every warp; after a timeout no copy may still be
  // landing in this block's shared memory
  if (tid == 0)
    for (int t = (tr1 - nst > tr0 ? tr1 - nst : tr0); t < tr1; ++t)
      cs_mbar_wait(&full[stage_of(t)], parity_of(t), flag);
  if (__any_sync(0xffffffffu, bad != 0.f) && lane == 0) atomicOr(flag, 1);
  block_mass<T3_WARPS>(macc, mpart, block_linear());
  if (!early) pdl_trigger();
}

int ychunk_for(long long tiles, int by);

// ---------------------------------------------------------------------------- fused 2-D step
// Small 2-D problems on the bf16 split: one cooperative launch runs many whole steps.
// Every block of (32, 19) threads is resident (one per SM); per step
//   phase A  warps 0-3 run operator work items (tile, contraction slice) of the per-tile
//            plan, storing partial tiles of F (op_item);
//   barrier  all blocks;
//   phase B  the block runs TMA-fed collide-stream items (tile column, tile rows), which
//            add the partial tiles in rank order (march2_tma);
//   barrier  all blocks.
// The arithmetic is that of the two-kernel step with the same plan, so the results are
// identical; the kernel boundaries (completion, flush, launch of the next grid) become
// grid barriers.  A barrier wait is bounded: after 2 s it sets bit 2 of the flag and the
// block continues, so every block reaches the end.
__device__ __forceinline__ void grid_sync(unsigned int* gbar, unsigned int target, int* flag) {
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    __threadfence();
    atomicAdd(gbar, 1u);
    unsigned int v;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(gbar) : "memory");
      if (v >= target) break;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t - t0 > (unsigned long long)kTmaWaitNs) {
        atomicOr(flag, 2);
        break;
      }
    }
    __threadfence();
    asm volatile("fence.proxy.async.global;" ::: "memory");  // this block's next TMA reads
  }
  __syncthreads();
}

template <int BN, int KS, bool MRT>
__global__ void __launch_bounds__(NT, 1)
lbm_fused2_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ TcParams P, const KConst<float> sp,
                  const __grid_constant__ CUtensorMap mf0, const __grid_constant__ CUtensorMap mf1,
                  const __grid_constant__ CUtensorMap mF, float* f0, float* f1, float* C, SplitOut so, int ychunk,
                  int nsteps, int parity, unsigned int* gbar, int* flag, double* mpart) {
  extern __shared__ uint8_t fused_raw[];
  __shared__ uint32_t tmem_slot;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(fused_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.y * TX + threadIdx.x;
  if (threadIdx.y == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(512)  // op_item's accumulator regions (at most 512 columns)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int G = gridDim.x;
  const int op_items = P.total_tiles * KS;
  const int bxn = (sp.n[0] + TX - 1) / TX, byn = (sp.n[1] + TY - 1) / TY;
  const int cs_items = bxn * ((byn + ychunk - 1) / ychunk);
  unsigned int target = 0;
  for (int st = 0; st < nsteps; ++st) {
    if (tid < 128)
      for (int it = blockIdx.x; it < op_items; it += G) op_item<2, BN, KS>(maps, P, it, smem, tmem, tid);
    target += G;
    grid_sync(gbar, target, flag);
    const int par = parity ^ (st & 1);
    const CUtensorMap* mf = par ? &mf1 : &mf0;
    float* fo = par ? f0 : f1;
    for (int it = blockIdx.x; it < cs_items; it += G) {
      march2_tma<MRT>(sp, mf, &mF, fo, C, flag, so, ychunk, it % bxn, it / bxn, smem, mpart, it);
      __syncthreads();
    }
    target += G;
    grid_sync(gbar, target, flag);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.y == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

template <int BN, int KS>
size_t fused_smem() {
  const size_t a = Cfg<2, BN, KS>::SMEM, b = tma2_smem(KS);
  return (a > b ? a : b) + 1024;
}

template <int BN, int KS, bool MRT>
cudaError_t fused_attr(int* blocks_per_sm) {
  static std::atomic<unsigned long long> attr{0};
  if (const cudaError_t e = smem_attr_once(attr, lbm_fused2_kernel<BN, KS, MRT>, (int)fused_smem<BN, KS>()); e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, lbm_fused2_kernel<BN, KS, MRT>, NT,
                                                       fused_smem<BN, KS>());
}

template <int BN, int KS, bool MRT>
cudaError_t fused_launch(const lbm_s* h, int nsteps, int grid, cudaStream_t s) {
  const TcPlan* p = h->tc;
  const CsPlan* pl = static_cast<const CsPlan*>(h->cs_plan);
  const KConst<float> sp = make_const<float>(h->sp);
  SplitOut so{h->dev.Chi, h->dev.Clo, tc_split_pitch(h)};
  const int bx = (h->sp.n[0] + TX - 1) / TX, by = (h->sp.n[1] + TY - 1) / TY;
  const int ychunk = h->cs_chunk > 0 ? std::min(h->cs_chunk, by) : ychunk_for((long long)bx * by, by);
  h->cs_nparts = kMassSlots * bx * ((by + ychunk - 1) / ychunk);  // per collide-stream item
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(TX, TY + HALO_WARPS);
  cfg.dynamicSmemBytes = fused_smem<BN, KS>();
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lbm_fused2_kernel<BN, KS, MRT>, p->maps, p->prm, sp, pl->f[0], pl->f[1], pl->F,
                            static_cast<float*>(h->dev.f[0]), static_cast<float*>(h->dev.f[1]),
                            static_cast<float*>(h->dev.C), so, ychunk, nsteps, h->cur, h->fused_bar, h->dev.flag,
                            h->cs_part);
}

// Grouped form for a batch of independent problems: one launch covers every block of
// every problem; block_map[b] = (problem, block within it), one load per block.  The
// problem's constants are staged in shared memory.
__host__ __device__ constexpr int batch_threads(int d) { return d == 2 ? 32 * kStripWarps : NT; }

template <int D, bool MRT, int SPLIT>
__global__ void __launch_bounds__(batch_threads(D), D == 2 ? 4 : 2)
collide_stream_batch_kernel(const BatchCS* __restrict__ tab, const int2* __restrict__ block_map, int parity, int keep_C) {
  __shared__ KConst<float> s_k;
  const int2 pb = __ldg(&block_map[blockIdx.x]);
  const BatchCS& e = tab[pb.x];
  const int tid = threadIdx.y * TX + threadIdx.x;
  constexpr int words = sizeof(KConst<float>) / sizeof(int);
  for (int i = tid; i < words; i += batch_threads(D))
    reinterpret_cast<int*>(&s_k)[i] = reinterpret_cast<const int*>(&e.k)[i];
  if (D == 2 && MRT && tid < kMaxQ * 8) {
    const int r = tid >> 3, c = tid & 7;
    reinterpret_cast<float*>(&s_om_rows[r][0])[c] = c < kMaxQ ? e.k.omega[r][c] : 0.0f;
  }
  __syncthreads();
  float* fo = const_cast<float*>(e.f[parity ^ 1]);
  float* Co = SPLIT == 0 || keep_C ? e.C : nullptr;
  if constexpr (D == 2) {
    const int item = pb.y * kStripWarps + (tid >> 5);
    if (item < e.items) {
      const int x = item % e.strips * 32 * e.v, y0 = item / e.strips * e.rows, y1 = min(y0 + e.rows, s_k.n[1]);
      if (e.v == 2) strip_march<2, MRT, SPLIT, true>(s_k, e.f[parity], e.F, fo, Co, e.flag, e.so, x, y0, y1, e.mpart, item);
      else strip_march<1, MRT, SPLIT, true>(s_k, e.f[parity], e.F, fo, Co, e.flag, e.so, x, y0, y1, e.mpart, item);
    }
  } else {
    march_body<float, D, MRT, SPLIT>(s_k, e.f[parity], e.F, fo, Co, e.flag, e.so, pb.y % e.bx, pb.y / e.bx, 0,
                                     e.k.n[2], e.mpart, pb.y);
  }
}

// Re-initialisation, f = feq(C, F(C)), bound by HBM: then C = <1|f>, so that the first step sees
// the C that the populations carry, and the operands of that C for the operator's next launch,
// all in one pass over the nodes.  In passes of their own the sum read the Q populations again and
// the operands C (256^3 bf16x6, 16 steps from a reset: 5772 -> 5646 us, tf32x3 6491 -> 6379).
template <typename real, int D, int SPLIT>
__global__ void init_state_kernel(const __grid_constant__ KConst<real> sp, const real* __restrict__ F,
                                  real* __restrict__ C, real* __restrict__ f, const __grid_constant__ SplitOut so,
                                  const __grid_constant__ FieldPtrs<real> fp) {
  const long long nodes = sp.nodes;
  const int n0 = sp.n[0], x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= n0) return;
  const int rows = static_cast<int>(nodes / n0);
  for (int row = blockIdx.y * blockDim.y + threadIdx.y; row < rows; row += gridDim.y * blockDim.y) {
    const long long i = (long long)row * n0 + x;
    const real c = C[i];
    real sumF = static_cast<real>(0);
    real Fv[D];
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      Fv[mu] = frac_term(sp, F, mu, i);
      sumF += Fv[mu];
    }
    real m = c - sp.w0 * sumF;
    f[i] = m;
#pragma unroll
    for (int mu = 0; mu < D; ++mu) {
      const real a = sp.wi * Fv[mu];
      const real b = (fp.advw ? fp.advw[mu * nodes + i] : sp.advw[mu]) * c;  // u(x) when it varies
      f[(2 * mu + 1) * nodes + i] = a + b;
      f[(2 * mu + 2) * nodes + i] = a - b;
      m += a + b;
      m += a - b;
    }
    C[i] = m;
    if constexpr (SPLIT != 0) {
      if (!fp.gsplit) write_split<SPLIT>(so, (long long)row * so.ldp + x, m);
    }
    if (fp.G || fp.gsplit) {  // g_mu(x) C per axis
#pragma unroll
      for (int mu = 0; mu < D; ++mu) {
        const real G = fp.g[mu * nodes + i] * m;
        if (fp.G) fp.G[mu * nodes + i] = G;
        if constexpr (SPLIT != 0) {
          SplitOut sm{};
          sm.hi = fp.gs[mu][0];
          sm.lo = fp.gs[mu][1];
          sm.lo2 = fp.gs[mu][2];
          if (fp.gsplit) write_split<SPLIT>(sm, (long long)row * fp.gldp + x, G);
        }
      }
    }
  }
}

// G_mu = g_mu(x) C, the operator's inputs when g varies in space
template <typename real>
__global__ void scale_fields_kernel(long long nodes, int d, const real* __restrict__ C, const real* __restrict__ g,
                                    real* __restrict__ G) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
       i += (long long)gridDim.x * blockDim.x)
    for (int mu = 0; mu < d; ++mu) G[mu * nodes + i] = g[mu * nodes + i] * C[i];
}

template <typename real, int Q>
__global__ void moment_kernel(long long nodes, const real* __restrict__ f, real* __restrict__ C) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nodes;
       i += (long long)gridDim.x * blockDim.x) {
    real c = f[i];
#pragma unroll
    for (int q = 1; q < Q; ++q) c += f[q * nodes + i];
    C[i] = c;
  }
}

template <bool MRT, int SPLIT>
cudaError_t launch_tma3(const cudaLaunchConfig_t& cfg, const KConst<float>& sp, const CUtensorMap& mf,
                        const CUtensorMap& mF, float* fo, float* Co, int* flag, const SplitOut& so, int nz,
                        int early, double* mpart) {
  static std::atomic<unsigned long long> attr{0};
  if (const cudaError_t e = smem_attr_once(attr, collide_stream_tma3_kernel<MRT, SPLIT>, (int)TMA_SMEM); e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, collide_stream_tma3_kernel<MRT, SPLIT>, sp, mf, mF, fo, Co, flag, so, nz, early,
                            mpart);
}

template <bool MRT, int SPLIT>
cudaError_t launch_tma2(const cudaLaunchConfig_t& cfg, const KConst<float>& sp, const CUtensorMap& mf,
                        const CUtensorMap& mF, float* fo, float* Co, int* flag, const SplitOut& so, int ychunk,
                        int early, double* mpart) {
  static std::atomic<unsigned long long> attr{0};
  if (const cudaError_t e = smem_attr_once(attr, collide_stream_tma2_kernel<MRT, SPLIT>, (int)tma2_smem(8)); e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, collide_stream_tma2_kernel<MRT, SPLIT>, sp, mf, mF, fo, Co, flag, so, ychunk,
                            early, mpart);
}

// at most two blocks per SM resident: the grid runs in one wave
bool one_wave(const dim3& g) { return (long long)g.x * g.y * g.z <= 2LL * device_sms(); }

// Let the next kernel (the operator) be scheduled at block start: only where this grid runs in
// one wave and the operator takes one block per SM (the tensor-core forms), or where both grids
// together are small (64^2 FP32 step 6.56 us without, 6.22 with the early trigger, 100^2 7.51 and
// 7.34).  The SIMT operator's small blocks, launched early beside a larger grid, pile up on the SMs
// that it leaves first (512^2 FP32 32.8 us with the early trigger, 22.9 without).
int early_trigger(const lbm_s* h, const dim3& g) {
  if (h->tc) return one_wave(g) ? 1 : 0;
  return one_wave(dim3(g.x * g.y * g.z + (unsigned)std::min(simt_blocks(h), 1LL << 30), 1, 1)) ? 1 : 0;
}

// 2-D FP32 lattices with coefficients per node: rows of a warp's strip in units of kStripRows, or 0
// for the plain march.  That one collides each node once and is the faster form where its blocks
// fit one wave (step, strips / plain: 64^2 bf16x6 7.9 / 6.8 us, 300^2 13.0 / 11.9, 300^2 FP32
// 18.1 / 15.7); beyond, its second wave costs more than the strips' extra rows (512^2 bf16x6
// 14.7 / 17.6, FP32 24.5 / 26.7, 1000 x 900 bf16x6 40.5 / 51.7).  The strips take the fewest rows
// that fit one wave (1000 x 900 with 2 / 4 / 6 / 8 rows: 44.3 / 42.6 / 40.6 / 44.5 us), at most 8.
int fields2_built_in(const lbm_s* h) {
  if (one_wave(dim3((h->sp.n[0] + TX - 1) / TX, (h->sp.n[1] + TY - 1) / TY, 1))) return 0;
  int c = 1;
  while (c < 4 && strip_grid(h->sp.n, c).items > 4LL * kStripWarps * device_sms()) ++c;
  return c;
}
int fields2_chunk(const lbm_s* h) { return h->fld_chunk > 0 ? h->fld_chunk : fields2_built_in(h); }

template <bool MRT, int SPLIT>
cudaError_t launch_march2(const cudaLaunchConfig_t& cfg, const KConst<float>& sp, const float* fi, const float* F,
                          float* fo, float* Co, int* flag, const SplitOut& so, int ychunk, int early, double* mpart) {
  static std::atomic<unsigned long long> attr{0};
  if (const cudaError_t e = smem_attr_once(attr, collide_stream_march2_kernel<MRT, SPLIT>, PIPE_SMEM); e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, collide_stream_march2_kernel<MRT, SPLIT>, sp, fi, F, fo, Co, flag, so, ychunk,
                            early, mpart);
}

// z chunks of the 3-D march over `cols` tile columns.  With waves enough, chunks of 16 planes:
// long chunks leave a long last wave, short ones re-collide two planes each (256^3 bf16x6 march
// with 7 / 9 / 16 / 24 / 38 chunks: 231 / 216 / 209 / 210 / 217 us).  Else the count that
// maximises the wave efficiency (blocks / 304 over its ceiling, two blocks per SM) per plane
// collided, chunks of at least 4 planes (with fewer blocks than the GPU holds, a block's chain
// of planes is the whole time: 48^3 in 18 blocks of 18 planes 23 us, in 72 of 6 12.6 us)
int z_chunks(long long cols, int n2) {
  if (n2 < 8) return 1;
  if (cols * (n2 / 16) >= 8LL * device_sms()) return (n2 + 15) / 16;
  const int sms = device_sms();
  int best = 1;
  double best_eff = 0.0;
  for (int nz = 1; nz <= n2 / 4; ++nz) {
    const double waves = static_cast<double>(cols * nz) / (2 * sms);
    const double eff = waves / std::ceil(waves);
    const double zc = static_cast<double>(n2) / nz;
    const double score = eff * zc / (zc + 2.0);
    if (score > best_eff + 1e-9) {
      best_eff = score;
      best = nz;
    }
  }
  return best;
}

// FP64 march: block tile and z chunks.  The FP64 pipe bounds it (a warp instruction holds the
// SM's pipe for 16 clocks, about 45 of them per collided node), so the plan with the smallest
// share on the busiest SM wins: ceil(blocks / SMs) blocks of march_warps warps over the planes
// of a chunk plus two (the chunk's first and last neighbours are collided again), plus the
// unhidden load and barrier latency of each plane of one block.  Measured against 32 x 16 tiles
// and chunks of at least 16 planes: 64^2 (8 blocks before, 128 now) 14.5 -> 8.4 us alone and the
// whole step 12.5 -> 7.3 us; 80^3 (75 blocks of 19 warps before) 160 -> 81 us.
struct March64Plan {
  int tile;  // 0: 32 x 16, 1: 16 x 16, 2: 8 x 4
  int bx, by, nz;
};
constexpr int kTile64[3][2] = {{TX, TY}, {16, 16}, {8, 4}};

March64Plan march64_plan(const lbm_s* h, int chunk) {
  const int n0 = h->sp.n[0], n1 = h->sp.n[1], n2 = h->sp.n[2];
  const long long sms = device_sms();
  March64Plan best{};
  double best_cost = -1.0;
  for (int t = 0; t < 3; ++t) {
    const int bx = (n0 + kTile64[t][0] - 1) / kTile64[t][0], by = (n1 + kTile64[t][1] - 1) / kTile64[t][1];
    for (int nz = 1; nz <= n2; ++nz) {
      if (chunk > 0 && h->d == 3 && nz != std::min(chunk, n2)) continue;
      const double planes = h->d == 2 ? 1.0 : static_cast<double>((n2 + nz - 1) / nz) + 2.0;
      const double blocks = static_cast<double>(((long long)bx * by * nz + sms - 1) / sms);
      const double cost = planes * (blocks * march_warps(kTile64[t][0], kTile64[t][1]) * 45 * 16 + 1500);
      if (best_cost < 0.0 || cost < best_cost) {
        best_cost = cost;
        best = {t, bx, by, nz};
      }
    }
  }
  return best;
}

template <int D, bool MRT, bool FLD, int TXX, int TYY>
cudaError_t launch_march64(cudaLaunchConfig_t& cfg, const KConst<double>& sp, const double* fi, const double* F,
                           double* fo, double* Co, int* flag, int nz, double* mp, const FieldPtrs<double>& fp) {
  cfg.blockDim = dim3(32, march_warps(TXX, TYY));
  return cudaLaunchKernelEx(&cfg, collide_stream_march_kernel<double, D, MRT, 0, FLD, TXX, TYY>, sp, fi, F, fo, Co,
                            flag, SplitOut{}, nz, 0, mp, fp);
}

template <int D, bool MRT, bool FLD>
cudaError_t launch_march64_any(const lbm_s* h, cudaLaunchConfig_t& cfg, const KConst<double>& sp, const double* fi,
                               const double* F, double* fo, double* Co, const FieldPtrs<double>& fp) {
  const March64Plan pl = march64_plan(h, h->cs_chunk);
  cfg.gridDim = dim3(pl.bx, pl.by, pl.nz);
  h->cs_nparts = march_warps(kTile64[pl.tile][0], kTile64[pl.tile][1]) * pl.bx * pl.by * pl.nz;
  int* flag = h->dev.flag;
  double* mp = h->cs_part;
  if (pl.tile == 0) return launch_march64<D, MRT, FLD, TX, TY>(cfg, sp, fi, F, fo, Co, flag, pl.nz, mp, fp);
  if (pl.tile == 1) return launch_march64<D, MRT, FLD, 16, 16>(cfg, sp, fi, F, fo, Co, flag, pl.nz, mp, fp);
  return launch_march64<D, MRT, FLD, 8, 4>(cfg, sp, fi, F, fo, Co, flag, pl.nz, mp, fp);
}

// tile rows per 2-D block: ceil(tiles / 304) (one wave of two blocks per SM), at most by
int ychunk_for(long long tiles, int by) {
  const long long w = 2LL * device_sms();
  const long long c = (tiles + w - 1) / w;
  return static_cast<int>(std::max<long long>(1, std::min<long long>(c, by)));
}

// which operand split of the new C the collide-stream kernel writes (write_split codes)
int cs_split_code(const lbm_s* h) {
  if (h->tc == nullptr) return 0;
  if (!bf16_parts(h->prm.precision)) return 2;
  return h->prm.precision == LBM_FP32_BF16SPLIT6 ? 3 : 1;
}

template <typename real>
FieldPtrs<real> field_ptrs(const lbm_s* h, int tk) {
  FieldPtrs<real> fp{static_cast<const real*>(h->fld.coll), static_cast<const real*>(h->fld.advw),
                     static_cast<const real*>(h->fld.g),    static_cast<real*>(h->fld.G),
                     static_cast<const real*>(h->fld.src),  static_cast<const real*>(h->fld.cw),
                     h->fld.tf ? h->fld.tf + 2 * tk : nullptr, {}, 0, 0};
  if (h->tc && h->tc->gvar && h->tc->elem == 2) {  // bf16: the parts of g_mu(x) C per axis
    fp.gsplit = 1;
    fp.gldp = h->tc->ldp;
    for (int mu = 0; mu < 3; ++mu)
      for (int k = 0; k < 3; ++k) fp.gs[mu][k] = h->tc->gp[mu][k];
  }
  return fp;
}

template <typename real, int D, bool MRT>
cudaError_t launch_cs(const lbm_s* h, const void* f_in, void* f_out, void* C_out, cudaStream_t s, int tk,
                      const CsSlot* slot) {
  const KConst<real> sp = make_const<real>(h->sp);
  SplitOut so{h->dev.Chi, h->dev.Clo, tc_split_pitch(h)};
  so.lo2 = h->dev.Cl2;
  const int split = cs_split_code(h);
  const real* fi = static_cast<const real*>(f_in);
  const real* F = static_cast<const real*>(slot ? slot->F : h->dev.F);
  real* fo = static_cast<real*>(f_out);
  real* Co = static_cast<real*>(C_out);
  int* flag = h->dev.flag;
  double* mp = h->cs_part;
  const int bx = (sp.n[0] + TX - 1) / TX, by = (sp.n[1] + TY - 1) / TY;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(TX, TY + HALO_WARPS);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = h->pdl ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (h->fld.on) {
    // coefficients per node: strips in 2-D, the plain march in 3-D
    const FieldPtrs<real> fp = field_ptrs<real>(h, tk);
    if constexpr (sizeof(real) == 8) return launch_march64_any<D, MRT, true>(h, cfg, sp, fi, F, fo, Co, fp);
    const int chunk = D == 2 ? fields2_chunk(h) : 0;
    if constexpr (D == 2 && sizeof(real) == 4)
    if (chunk > 0) {
      const StripGrid g = strip_grid(sp.n, chunk);
      cfg.gridDim = dim3((g.items + kStripWarps - 1) / kStripWarps);
      cfg.blockDim = dim3(32 * kStripWarps);
      h->cs_nparts = g.items;
      auto go = [&](auto v2, auto v1) {
        return cudaLaunchKernelEx(&cfg, g.v == 2 ? v2 : v1, sp, fi, F, fo, Co, flag, so, fp, g, h->pdl && h->tc ? 1 : 0, mp);
      };
      // the tensor-core forms' march also writes the operator's operands of the new C
      if (split == 0) return go(collide_stream_fields2_kernel<2, MRT, 0>, collide_stream_fields2_kernel<1, MRT, 0>);
      if (split == 1) return go(collide_stream_fields2_kernel<2, MRT, 1>, collide_stream_fields2_kernel<1, MRT, 1>);
      if (split == 2) return go(collide_stream_fields2_kernel<2, MRT, 2>, collide_stream_fields2_kernel<1, MRT, 2>);
      return go(collide_stream_fields2_kernel<2, MRT, 3>, collide_stream_fields2_kernel<1, MRT, 3>);
    }
    if constexpr (sizeof(real) == 4) {
      const int nz = D == 2 ? 1 : h->cs_chunk > 0 ? std::min(h->cs_chunk, sp.n[2]) : z_chunks((long long)bx * by, sp.n[2]);
      cfg.gridDim = dim3(bx, by, nz);
      h->cs_nparts = kMassSlots * bx * by * nz;
      const int early = early_trigger(h, cfg.gridDim);
      auto go = [&](auto k) { return cudaLaunchKernelEx(&cfg, k, sp, fi, F, fo, Co, flag, so, nz, early, mp, fp); };
      if (split == 0) return go(collide_stream_march_kernel<real, D, MRT, 0, true>);
      if (split == 1) return go(collide_stream_march_kernel<real, D, MRT, 1, true>);
      if (split == 2) return go(collide_stream_march_kernel<real, D, MRT, 2, true>);
      return go(collide_stream_march_kernel<real, D, MRT, 3, true>);
    }
  }
  if constexpr (sizeof(real) == 8)
    return launch_march64_any<D, MRT, false>(h, cfg, sp, fi, F, fo, Co, FieldPtrs<double>{});
  if constexpr (D == 2 && sizeof(real) == 4) {
    // tile rows per block: about one wave of two blocks per SM, unless tuned
    const int ychunk = h->cs_chunk > 0 ? std::min(h->cs_chunk, by) : ychunk_for((long long)bx * by, by);
    cfg.gridDim = dim3(bx, (by + ychunk - 1) / ychunk, 1);
    h->cs_nparts = kMassSlots * static_cast<int>(cfg.gridDim.x * cfg.gridDim.y);
    const int early = early_trigger(h, cfg.gridDim);
    if (h->cs_plan) {
      const CsPlan* pl = static_cast<const CsPlan*>(h->cs_plan);
      const CUtensorMap& mf = slot ? *static_cast<const CUtensorMap*>(slot->map_f) : pl->f[f_in == h->dev.f[0] ? 0 : 1];
      const CUtensorMap& mF = slot ? *static_cast<const CUtensorMap*>(slot->map_F) : pl->F;
      cfg.dynamicSmemBytes = tma2_smem(h->sp.ksum);
      cfg.blockDim = dim3(32, T3_WARPS);
      h->cs_nparts = T3_WARPS * static_cast<int>(cfg.gridDim.x * cfg.gridDim.y);
      if (split == 0) return launch_tma2<MRT, 0>(cfg, sp, mf, mF, fo, Co, flag, so, ychunk, early, mp);
      if (split == 1) return launch_tma2<MRT, 1>(cfg, sp, mf, mF, fo, Co, flag, so, ychunk, early, mp);
      if (split == 3) return launch_tma2<MRT, 3>(cfg, sp, mf, mF, fo, Co, flag, so, ychunk, early, mp);
      so.thi[0] = static_cast<float*>(h->tc->ct_hi[1]);  // the y operand of the tf32 operator
      so.tg1 = h->tc->tg[1];
      so.tpx = h->tc->tpx;
      return launch_tma2<MRT, 2>(cfg, sp, mf, mF, fo, Co, flag, so, ychunk, early, mp);
    }
    cfg.dynamicSmemBytes = PIPE_SMEM;
    if (split == 0) return launch_march2<MRT, 0>(cfg, sp, fi, F, fo, Co, flag, so, ychunk, early, mp);
    if (split == 1) return launch_march2<MRT, 1>(cfg, sp, fi, F, fo, Co, flag, so, ychunk, early, mp);
    if (split == 3) return launch_march2<MRT, 3>(cfg, sp, fi, F, fo, Co, flag, so, ychunk, early, mp);
    return launch_march2<MRT, 2>(cfg, sp, fi, F, fo, Co, flag, so, ychunk, early, mp);
  }
  if constexpr (sizeof(real) == 4) {
  const int nz = h->cs_chunk > 0 ? std::min(h->cs_chunk, sp.n[2]) : z_chunks((long long)bx * by, sp.n[2]);
  cfg.gridDim = dim3(bx, by, nz);
  h->cs_nparts = kMassSlots * bx * by * nz;
  const int early = early_trigger(h, cfg.gridDim);
  if constexpr (D == 3 && sizeof(real) == 4) {
    if (h->cs_plan) {
      // TMA-fed march: the map of whichever population buffer is the input
      const CsPlan* pl = static_cast<const CsPlan*>(h->cs_plan);
      const CUtensorMap& mf = slot ? *static_cast<const CUtensorMap*>(slot->map_f) : pl->f[f_in == h->dev.f[0] ? 0 : 1];
      const CUtensorMap& mF = slot ? *static_cast<const CUtensorMap*>(slot->map_F) : pl->F;
      cfg.dynamicSmemBytes = TMA_SMEM;
      cfg.blockDim = dim3(32, T3_WARPS);
      h->cs_nparts = T3_WARPS * bx * by * nz;
      if (split == 0) return launch_tma3<MRT, 0>(cfg, sp, mf, mF, fo, Co, flag, so, nz, early, mp);
      if (split == 1) return launch_tma3<MRT, 1>(cfg, sp, mf, mF, fo, Co, flag, so, nz, early, mp);
      if (split == 3) return launch_tma3<MRT, 3>(cfg, sp, mf, mF, fo, Co, flag, so, nz, early, mp);
      for (int a = 0; a < 2; ++a) {  // the y and z operands of the tf32 operator
        so.thi[a] = static_cast<float*>(h->tc->ct_hi[a + 1]);
      }
      so.tg1 = h->tc->tg[1];
      so.tpx = h->tc->tpx;
      return launch_tma3<MRT, 2>(cfg, sp, mf, mF, fo, Co, flag, so, nz, early, mp);
    }
  }
  if (split == 0)
    return cudaLaunchKernelEx(&cfg, collide_stream_march_kernel<real, D, MRT, 0>, sp, fi, F, fo, Co, flag, so, nz,
                              early, mp, FieldPtrs<real>{});
  if (split == 1)
    return cudaLaunchKernelEx(&cfg, collide_stream_march_kernel<real, D, MRT, 1>, sp, fi, F, fo, Co, flag, so, nz,
                              early, mp, FieldPtrs<real>{});
  if (split == 3)
    return cudaLaunchKernelEx(&cfg, collide_stream_march_kernel<real, D, MRT, 3>, sp, fi, F, fo, Co, flag, so, nz,
                              early, mp, FieldPtrs<real>{});
  return cudaLaunchKernelEx(&cfg, collide_stream_march_kernel<real, D, MRT, 2>, sp, fi, F, fo, Co, flag, so, nz,
                            early, mp, FieldPtrs<real>{});
  }
}

int grid_for(long long n) {
  long long b = (n + 255) / 256;
  const long long cap = 16LL * device_sms();
  if (b > cap) b = cap;
  return static_cast<int>(b < 1 ? 1 : b);
}

}  // namespace

// tf32 handles on the TMA-fed marches: the collide-stream kernel writes the regrouped split
bool cs_writes_T(const lbm_s* h) {
  return !h->is_batch() && h->elem == 4 && h->cs_plan != nullptr && h->tc != nullptr && h->tc->elem == 4 &&
         h->prm.precision == LBM_FP32_TF32SPLIT && !h->fld.on;  // the field march writes x-major operands only
}

cudaError_t launch_collide_stream(const lbm_s* h, const void* f_in, void* f_out, void* C_out, cudaStream_t s, int tk,
                                  const CsSlot* slot) {
  const bool mrt = h->prm.collision == LBM_MRT;
  if (h->elem == 8) {
    if (h->d == 2) return mrt ? launch_cs<double, 2, true>(h, f_in, f_out, C_out, s, tk, slot)
                              : launch_cs<double, 2, false>(h, f_in, f_out, C_out, s, tk, slot);
    return mrt ? launch_cs<double, 3, true>(h, f_in, f_out, C_out, s, tk, slot)
               : launch_cs<double, 3, false>(h, f_in, f_out, C_out, s, tk, slot);
  }
  if (h->d == 2) return mrt ? launch_cs<float, 2, true>(h, f_in, f_out, C_out, s, tk, slot)
                            : launch_cs<float, 2, false>(h, f_in, f_out, C_out, s, tk, slot);
  return mrt ? launch_cs<float, 3, true>(h, f_in, f_out, C_out, s, tk, slot)
             : launch_cs<float, 3, false>(h, f_in, f_out, C_out, s, tk, slot);
}

constexpr int kBatchChunk = 4;  // units of kStripRows per warp

// window map of `planes` fields (x fastest, `base` their first) for the TMA-fed marches:
// (n0, n1, planes) in 2-D, (n0, n1, n2, planes) in 3-D
bool encode_window(const lbm_s* h, CUtensorMap* m, const void* base, unsigned long long planes) {
  const unsigned long long n0 = h->sp.n[0], n1 = h->sp.n[1], n2 = h->sp.n[2], nodes = h->sp.nodes;
  if (h->d == 2) {
    const unsigned long long dims[3] = {n0, n1, planes}, strides[2] = {n0 * 4, nodes * 4};
    const unsigned int box[3] = {TW, TH, (unsigned int)planes};
    return encode_f32_map(m, 3, const_cast<void*>(base), dims, strides, box);
  }
  const unsigned long long dims[4] = {n0, n1, n2, planes}, strides[3] = {n0 * 4, n0 * n1 * 4, nodes * 4};
  const unsigned int box[4] = {TW, TH, 1, (unsigned int)planes};
  return encode_f32_map(m, 4, const_cast<void*>(base), dims, strides, box);
}

// window maps of a handle: its population buffers and its fractional terms ([partial][axis][node])
bool encode_maps(const lbm_s* h, CUtensorMap* mf, CUtensorMap* mF) {
  return encode_window(h, &mf[0], h->dev.f[0], h->Q) && encode_window(h, &mf[1], h->dev.f[1], h->Q) &&
         encode_window(h, mF, h->dev.F, (unsigned long long)h->d * h->sp.ksum);
}

bool cs_encode_slot(const lbm_s* h, const void* f, const void* F, void* map_f, void* map_F) {
  return encode_window(h, static_cast<CUtensorMap*>(map_f), f, h->Q) &&
         encode_window(h, static_cast<CUtensorMap*>(map_F), F, h->d);
}

// the fused step for this handle's plan: 0 (not covered) or the blocks per SM it gets
namespace {
template <int BN, int KS>
cudaError_t fused_call(lbm_s* h, int nsteps, int grid, cudaStream_t s, int* occ) {
  const bool mrt = h->prm.collision == LBM_MRT;
  if (occ) return mrt ? fused_attr<BN, KS, true>(occ) : fused_attr<BN, KS, false>(occ);
  return mrt ? fused_launch<BN, KS, true>(h, nsteps, grid, s) : fused_launch<BN, KS, false>(h, nsteps, grid, s);
}

cudaError_t fused_any(lbm_s* h, int nsteps, int grid, cudaStream_t s, int* occ) {
  int bn = 0, ks = 0, persist = 0;
  tc_config(h, &bn, &ks, &persist);
  if (persist) return cudaErrorNotSupported;
  if (bn == 64 && ks == 2) return fused_call<64, 2>(h, nsteps, grid, s, occ);
  if (bn == 64 && ks == 4) return fused_call<64, 4>(h, nsteps, grid, s, occ);
  if (bn == 128 && ks == 2) return fused_call<128, 2>(h, nsteps, grid, s, occ);
  if (bn == 128 && ks == 4) return fused_call<128, 4>(h, nsteps, grid, s, occ);
  return cudaErrorNotSupported;
}
}  // namespace

int fused_prepare(lbm_s* h) {
  h->fused_grid = 0;
  if (h->is_batch() || h->d != 2 || h->prm.precision != LBM_FP32_BF16SPLIT || !h->tc || !h->cs_plan) return LBM_ENOTSUP;
  if (!tc_tma_store(h)) return LBM_ENOTSUP;
  int occ = 0;
  if (fused_any(h, 0, 0, nullptr, &occ) != cudaSuccess || occ < 1) return LBM_ENOTSUP;
  if (!h->fused_bar && dev_alloc(h, (void**)&h->fused_bar, sizeof(unsigned int)) != cudaSuccess) return LBM_ENOMEM;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  h->fused_grid = sms * occ;
  return LBM_OK;
}

cudaError_t launch_fused(lbm_s* h, int nsteps, cudaStream_t s) {
  if (h->fused_grid < 1) return cudaErrorNotSupported;
  const cudaError_t e = cudaMemsetAsync(h->fused_bar, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  return fused_any(h, nsteps, h->fused_grid, s, nullptr);
}

int cs_prepare(lbm_s* h) {
  if (h->elem != 4 || h->sp.n[0] % 4 != 0) return LBM_OK;
  CsPlan* pl = new (std::nothrow) CsPlan();
  if (!pl) return LBM_ENOMEM;
  if (encode_maps(h, pl->f, &pl->F)) h->cs_plan = pl;
  else delete pl;  // the cp.async (2-D) or plain (3-D) march serves the handle
  return LBM_OK;
}

void cs_release(lbm_s* h) {
  delete static_cast<CsPlan*>(h->cs_plan);
  h->cs_plan = nullptr;
}

bool cs_one_wave(const lbm_s* h) {
  if (h->elem == 8) {
    const March64Plan pl = march64_plan(h, h->cs_chunk);
    return one_wave(dim3(pl.bx, pl.by, pl.nz));
  }
  const int bx = (h->sp.n[0] + TX - 1) / TX, by = (h->sp.n[1] + TY - 1) / TY;
  if (h->d == 2 && h->elem == 4 && h->fld.on) {
    const int chunk = fields2_chunk(h);  // strips: four blocks to an SM
    if (chunk > 0) return strip_grid(h->sp.n, chunk).items <= 4LL * kStripWarps * device_sms();
    return one_wave(dim3(bx, by, 1));
  }
  if (h->d == 2 && h->elem == 4) {
    const int ychunk = h->cs_chunk > 0 ? std::min(h->cs_chunk, by) : ychunk_for((long long)bx * by, by);
    return one_wave(dim3(bx, (by + ychunk - 1) / ychunk, 1));
  }
  const int nz = h->cs_chunk > 0 ? std::min(h->cs_chunk, h->sp.n[2]) : z_chunks((long long)bx * by, h->sp.n[2]);
  return one_wave(dim3(bx, by, nz));
}

long long cs_max_parts(const lbm_s* h) {
  long long most = h->d == 2 && h->elem == 4 ? strip_grid(h->sp.n, 1).items : 0;
  for (int t = 0; t < (h->elem == 8 ? 3 : 1); ++t) {  // one block per tile and plane at most
    const long long bx = (h->sp.n[0] + kTile64[t][0] - 1) / kTile64[t][0], by = (h->sp.n[1] + kTile64[t][1] - 1) / kTile64[t][1];
    most = std::max(most, march_warps(kTile64[t][0], kTile64[t][1]) * bx * by * h->sp.n[2]);
  }
  return most;
}

int cs_chunk_default(const lbm_s* h) {
  const int bx = (h->sp.n[0] + TX - 1) / TX, by = (h->sp.n[1] + TY - 1) / TY;
  if (h->is_batch()) return kBatchChunk;
  if (h->d == 2 && h->elem == 4 && h->fld.on) return fields2_built_in(h);
  if (h->d == 2) return h->elem == 4 ? ychunk_for((long long)bx * by, by) : 1;
  return h->elem == 8 ? march64_plan(h, 0).nz : z_chunks((long long)bx * by, h->sp.n[2]);
}

int cs_batch_prepare(lbm_s* b) {
  const int P = static_cast<int>(b->subs.size());
  std::vector<BatchCS> tab(P);
  std::vector<int2> map;
  std::vector<int> nparts(P);
  int total = 0;
  for (int i = 0; i < P; ++i) {
    lbm_s* h = b->subs[i];
    if (h->elem != 4) return LBM_EINVAL;
    BatchCS& e = tab[i];
    e.k = make_const<float>(h->sp);
    e.f[0] = static_cast<const float*>(h->dev.f[0]);
    e.f[1] = static_cast<const float*>(h->dev.f[1]);
    e.F = static_cast<const float*>(h->dev.F);
    e.C = static_cast<float*>(h->dev.C);
    e.so = SplitOut{h->dev.Chi, h->dev.Clo, tc_split_pitch(h)};
    e.so.lo2 = h->dev.Cl2;
    e.flag = h->dev.flag;
    e.mpart = h->cs_part;
    e.bx = (h->sp.n[0] + TX - 1) / TX;
    int blocks = e.bx * ((h->sp.n[1] + TY - 1) / TY);  // 3-D: one column each, the whole z extent
    nparts[i] = kMassSlots * blocks;
    if (h->d == 2) {
      const StripGrid g = strip_grid(h->sp.n, b->cs_chunk > 0 ? b->cs_chunk : kBatchChunk);
      e.v = g.v;
      e.strips = g.strips;
      e.rows = g.rows;
      e.items = nparts[i] = g.items;
      blocks = (g.items + kStripWarps - 1) / kStripWarps;
    }
    for (int k = 0; k < blocks; ++k) map.push_back(make_int2(i, k));
    total += blocks;
  }
  // the tables in force stay until the new ones are whole
  void* d_tab = nullptr;
  void* d_map = nullptr;
  int rc = LBM_OK;
  if (dev_alloc(b, &d_tab, sizeof(BatchCS) * P) != cudaSuccess || dev_alloc(b, &d_map, sizeof(int2) * total) != cudaSuccess)
    rc = LBM_ENOMEM;
  else if (cudaMemcpy(d_tab, tab.data(), sizeof(BatchCS) * P, cudaMemcpyHostToDevice) != cudaSuccess ||
           cudaMemcpy(d_map, map.data(), sizeof(int2) * total, cudaMemcpyHostToDevice) != cudaSuccess ||
           cudaStreamSynchronize(b->stream) != cudaSuccess)  // no launch in flight reads the old ones
    rc = LBM_ECUDA;
  dev_free(b, rc ? d_tab : b->batch_cs);
  dev_free(b, rc ? d_map : static_cast<void*>(b->batch_cs_start));
  if (rc) return rc;
  b->batch_cs = d_tab;
  b->batch_cs_start = static_cast<int*>(d_map);
  b->batch_cs_blocks = total;
  for (int i = 0; i < P; ++i) b->subs[i]->cs_nparts = nparts[i];
  return LBM_OK;
}

cudaError_t launch_collide_stream_batch(const lbm_s* b, int parity, cudaStream_t s, bool keep_C) {
  const lbm_s* h0 = b->subs[0];
  const bool mrt = h0->prm.collision == LBM_MRT;
  const int split = cs_split_code(h0);  // 0, 1 or 3 (batches have no tf32 form)
  const BatchCS* tab = static_cast<const BatchCS*>(b->batch_cs);
  const int P = static_cast<int>(b->subs.size());
  const dim3 block(TX, batch_threads(h0->d) / TX);
  const int g = b->batch_cs_blocks;
#define LBM_CSB(D_, M_, S_) \
  collide_stream_batch_kernel<D_, M_, S_><<<g, block, 0, s>>>(tab, reinterpret_cast<const int2*>(b->batch_cs_start), parity, keep_C || split == 0)
  if (h0->d == 2) {
    if (mrt) { if (split == 3) LBM_CSB(2, true, 3); else if (split) LBM_CSB(2, true, 1); else LBM_CSB(2, true, 0); }
    else { if (split == 3) LBM_CSB(2, false, 3); else if (split) LBM_CSB(2, false, 1); else LBM_CSB(2, false, 0); }
  } else {
    if (mrt) { if (split == 3) LBM_CSB(3, true, 3); else if (split) LBM_CSB(3, true, 1); else LBM_CSB(3, true, 0); }
    else { if (split == 3) LBM_CSB(3, false, 3); else if (split) LBM_CSB(3, false, 1); else LBM_CSB(3, false, 0); }
  }
#undef LBM_CSB
  return cudaGetLastError();
}

template <typename real, int D>
cudaError_t launch_init(const lbm_s* h, void* f, cudaStream_t s) {
  SplitOut so{h->dev.Chi, h->dev.Clo, tc_split_pitch(h)};
  so.lo2 = h->dev.Cl2;
  const FieldPtrs<real> fp = h->fld.on ? field_ptrs<real>(h, 0) : FieldPtrs<real>{};
  const KConst<real> sp = make_const<real>(h->sp);
  auto go = [&](auto k) {
    k<<<row_grid(h), row_block(h), 0, s>>>(sp, static_cast<const real*>(h->dev.F), static_cast<real*>(h->dev.C), static_cast<real*>(f), so, fp);
    return cudaGetLastError();
  };
  if constexpr (sizeof(real) == 4) {
    const int split = cs_split_code(h);
    if (split == 1) return go(init_state_kernel<real, D, 1>);
    if (split == 2) return go(init_state_kernel<real, D, 2>);
    if (split == 3) return go(init_state_kernel<real, D, 3>);
  }
  return go(init_state_kernel<real, D, 0>);
}

cudaError_t launch_init_state(const lbm_s* h, void* f, cudaStream_t s) {
  const cudaError_t e = h->elem == 8 ? (h->d == 2 ? launch_init<double, 2>(h, f, s) : launch_init<double, 3>(h, f, s))
                                     : (h->d == 2 ? launch_init<float, 2>(h, f, s) : launch_init<float, 3>(h, f, s));
  if (e != cudaSuccess || !h->tc) return e;
  return launch_split_T(h, s);  // tf32: the operands regrouped along y and z
}

cudaError_t launch_scale_fields(const lbm_s* h, cudaStream_t s) {
  if (!h->fld.G) return cudaSuccess;  // tensor-core forms: g is uniform and folded into K
  const int g = grid_for(h->sp.nodes);
  if (h->elem == 8)
    scale_fields_kernel<double><<<g, 256, 0, s>>>(h->sp.nodes, h->d, (const double*)h->dev.C, (const double*)h->fld.g,
                                                  (double*)h->fld.G);
  else
    scale_fields_kernel<float><<<g, 256, 0, s>>>(h->sp.nodes, h->d, (const float*)h->dev.C, (const float*)h->fld.g,
                                                 (float*)h->fld.G);
  return cudaGetLastError();
}

cudaError_t launch_moment(const lbm_s* h, const void* f, void* C, cudaStream_t s) {
  const int g = grid_for(h->sp.nodes);
  if (h->elem == 8) {
    if (h->Q == 5) moment_kernel<double, 5><<<g, 256, 0, s>>>(h->sp.nodes, (const double*)f, (double*)C);
    else moment_kernel<double, 7><<<g, 256, 0, s>>>(h->sp.nodes, (const double*)f, (double*)C);
  } else {
    if (h->Q == 5) moment_kernel<float, 5><<<g, 256, 0, s>>>(h->sp.nodes, (const float*)f, (float*)C);
    else moment_kernel<float, 7><<<g, 256, 0, s>>>(h->sp.nodes, (const float*)f, (float*)C);
  }
  return cudaGetLastError();
}

}  // namespace lbm
