// Fractional terms on CUDA cores (FP64 and plain-FP32 forms).
//
// Algorithm 1 (fractional terms) / Section 2.4, Eq. (XXminus_discret): along every
// lattice line of axis mu, F_mu[n] = sum_l K_mu[n][l] C[l].  Viewed over all
// lines this is one dense GEMM per axis:
//   axis x (fastest):  F[r][n] = sum_l C[r][l] K[n][l]     = C  * K^T   (rows r = other coords)
//   axis y, z:         F[b][n][c] = sum_l K[n][l] C[b][l][c] = K * C_b  (b = outer planes, c = inner)
// Both are written as a row-major GEMM D = A B (A: M x K, B: K x N), batched over b with
// strides; K and K^T are both stored, so that B, and A on the y and z axes, are read with
// their output index contiguous.  One launch covers every axis: a table maps each block to
// (axis, batch, tile, contraction slice).
//
// FP32: small problems split the contraction over the ks blocks of a thread-block cluster,
// which add their partial tiles in slice order through distributed shared memory.
#include <algorithm>
#include <atomic>
#include <climits>

#include "cluster_dev.cuh"
#include "lbm_internal.h"
#include "simt_dev.cuh"

namespace lbm {
namespace {

struct GemmAxis {
  const void* A;
  const void* B;
  void* C;
  long long lda, sA, ldb, sB, ldc, sC;
  int M, N, K;
  int tm, tn;          // tiles along M and N
  int amode;           // 0: A(m, k) at m * lda + k; 1: at k * lda + m
  int vec;             // FP32: bit 0/1/2: A/B/C rows and extents are whole aligned groups of four
  long long begin;     // first block of this axis
};

struct GemmPlan {
  GemmAxis ax[3];
  int naxes;
  int ks;              // contraction slices per tile (FP32: the blocks of one cluster)
  int sub;             // FP32: parts of a slice with an accumulation chain of their own, added in order
  long long total;
  int early;           // one-wave grid: let the next kernel be scheduled at block start
};

// block b of the plan: axis, batch index, tile origin
struct BlockAt {
  int a, m0, n0;
  long long bz;
};

__device__ __forceinline__ BlockAt locate_block(const GemmPlan& P, long long b, int BM, int BN) {
  int a = 0;
  while (a + 1 < P.naxes && b >= P.ax[a + 1].begin) ++a;
  const GemmAxis& X = P.ax[a];
  b = (b - X.begin) / P.ks;
  const long long per = (long long)X.tm * X.tn;
  const long long bz = b / per;
  const int r = static_cast<int>(b - bz * per);
  return BlockAt{a, (r / X.tn) * BM, (r % X.tn) * BN, bz};
}

// ---------------------------------------------------------------------------- FP32
// A block of 8 TY threads owns a tile of 4 RG TY x 32 CG outputs, 4 RG x 4 CG per thread.
// Bound by FP32 issue once the grid fills the GPU, so the inner loop is packed fma.rn.f32x2
// (two outputs of a row per instruction, each rounded as an FMA), which leaves issue slots for
// the shared loads and for doubling A's values into packed operands.  (Staging A doubled in
// shared memory instead made the loop shared-memory bound: 16 wavefronts per 16 clocks of
// FMAs; 256^3 operator 584 us against 484.)  A thread's outputs come in groups of four rows
// and columns, so that all shared and global accesses are 128-bit; the staged A is swizzled
// so that transposing C's rows into it is free of bank conflicts.  Rounds of SBK contraction
// steps (groups of 16), double buffered through registers.  Each output's products are added in contraction
// order within its part of a slice, whichever tile serves it.
// Measured with the rules below, before (64 x 64 or 32 x 32 tiles of scalar FMAs, partial sums
// added by the consumer) and after: step of 512^2 32.2 -> 22.9 us, 256^2 13.8 -> 9.6 us,
// operator of 256^3 845 -> 484 us (66% of the FP32 pipe's rate), of 1024^2 98 us.
constexpr int kSlice = 32;  // contraction slices of a split, and their parts, start at multiples of this

__device__ __forceinline__ void store4(float* p, float4 v, int left, bool vec) {
  if (left >= 4 && vec) {
    *reinterpret_cast<float4*>(p) = v;
    return;
  }
  if (left > 0) p[0] = v.x;
  if (left > 1) p[1] = v.y;
  if (left > 2) p[2] = v.z;
  if (left > 3) p[3] = v.w;
}

template <int RG, int CG, int TY, int SBK, bool SUB>
__global__ void __launch_bounds__(8 * TY) frac_simt32_kernel(const __grid_constant__ GemmPlan P);

template <int RG, int CG, int TY, int SBK, bool SUB = false>
struct F32Cfg {
  static constexpr int THREADS = 8 * TY, AMODE = 1;
  static constexpr int BM = 4 * RG * TY, BN = 32 * CG;
  static auto kernel() { return frac_simt32_kernel<RG, CG, TY, SBK, SUB>; }
};

template <int RG, int CG, int TY, int SBK, bool SUB>
__global__ void __launch_bounds__(8 * TY)
frac_simt32_kernel(const __grid_constant__ GemmPlan P) {
  using G = F32Cfg<RG, CG, TY, SBK, SUB>;
  constexpr int THREADS = G::THREADS, BM = G::BM, BN = G::BN, R = 4 * RG;
  constexpr int LA = BM * SBK / 4 / THREADS;       // float4 loads per thread
  constexpr int LB = BN * SBK / 4 / THREADS;
  __shared__ __align__(16) float s_mem[2 * SBK * (BM + BN) > BM * BN ? 2 * SBK * (BM + BN) : BM * BN];
  float* As = s_mem;                          // [2][SBK][BM]: (k, m) at column m ^ 8 ((k / 4) % 4)
  float* Bs = s_mem + 2 * SBK * BM;           // [2][SBK][BN]
  // programmatic dependent launch: C (read) and F (written) belong to the previous kernel
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (P.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const BlockAt at = locate_block(P, blockIdx.x, BM, BN);
  const GemmAxis& X = P.ax[at.a];
  const int ks = P.ks, rank = static_cast<int>(blockIdx.x) % ks;  // (an axis begins at a multiple of ks)
  const int m0 = at.m0, n0 = at.n0;
  const float* __restrict__ A = static_cast<const float*>(X.A) + at.bz * X.sA;
  const float* __restrict__ B = static_cast<const float*>(X.B) + at.bz * X.sB;
  float* __restrict__ Cm = static_cast<float*>(X.C) + at.bz * X.sC;
  const int M = X.M, N = X.N, amode = X.amode;
  const bool va = X.vec & 1, vb = X.vec & 2, vc = X.vec & 4;
  const int nkb = (X.K + kSlice - 1) / kSlice;
  // part j of the contraction (sub parts to a slice) starts here
  const int sub = SUB ? P.sub : 1;
  auto part = [&](int j) { return j * nkb / (ks * sub) * kSlice; };
  const int kbeg = part(rank * sub);
  const int K = min(X.K, part((rank + 1) * sub));
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;

  float4 ra[LA], rb[LB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * THREADS;
      if (amode == 0) {  // four k of one row
        const int m = m0 + e / 4 % BM, k = k0 + 16 * (e / (4 * BM)) + 4 * (e % 4);
        ra[i] = load4(A + m * X.lda + k, m < M ? K - k : 0, va);
      } else {           // four rows at one k
        const int k = k0 + e / (BM / 4), m = m0 + 4 * (e % (BM / 4));
        ra[i] = load4(A + k * X.lda + m, k < K ? M - m : 0, va);
      }
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + i * THREADS;
      const int k = k0 + e / (BN / 4), n = n0 + 4 * (e % (BN / 4));
      rb[i] = load4(B + k * X.ldb + n, k < K ? N - n : 0, vb);
    }
  };
  auto stash = [&](int buf) {
    float* as = As + buf * SBK * BM;
    float* bs = Bs + buf * SBK * BN;
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * THREADS;
      const float4 v = ra[i];
      if (amode == 0) {
        const int kq = 4 * (e / (4 * BM)) + e % 4;
        float* p = as + 4 * kq * BM + ((e / 4 % BM) ^ (8 * (kq % 4)));
        p[0] = v.x;
        p[BM] = v.y;
        p[2 * BM] = v.z;
        p[3 * BM] = v.w;
      } else {
        const int k = e / (BM / 4);
        *reinterpret_cast<float4*>(as + k * BM + ((4 * (e % (BM / 4))) ^ (8 * (k / 4 % 4)))) = v;
      }
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + i * THREADS;
      *reinterpret_cast<float4*>(bs + (e / (BN / 4)) * BN + 4 * (e % (BN / 4))) = rb[i];
    }
  };

  unsigned long long acc[R][2 * CG];  // rows 4 ty + i (groups 4 TY apart), packed column pairs 4 tx + 2 j (groups 32 apart)
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < 2 * CG; ++j) acc[i][j] = 0ull;

  // the finished parts of the slice (SUB: it may have more than one)
  unsigned long long sum[SUB ? R : 1][SUB ? 2 * CG : 1] = {};
  int j = 1, kpart = SUB ? part(rank * sub + 1) : INT_MAX;
  auto close_part = [&]() {  // acc joins the finished parts
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int h = 0; h < 2 * CG; ++h) {
        sum[SUB ? i : 0][SUB ? h : 0] = fadd2(sum[SUB ? i : 0][SUB ? h : 0], acc[i][h]);
        acc[i][h] = 0ull;
      }
  };

  fetch(kbeg);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < K; k0 += SBK) {
    if (SUB && k0 >= kpart) {
      close_part();
      while (k0 >= kpart) kpart = ++j < sub ? part(rank * sub + j) : INT_MAX;
    }
    const bool more = k0 + SBK < K;
    if (more) fetch(k0 + SBK);
    const float* as = As + buf * SBK * BM;
    const float* bs = Bs + buf * SBK * BN + 4 * tx;
#pragma unroll
    for (int kk = 0; kk < SBK; ++kk) {
      if (kk > 0 && kk % 16 == 0 && k0 + kk >= K) break;  // the rest of the round is past the end
      float4 a[RG];
      ulonglong2 b[CG];
#pragma unroll
      for (int g = 0; g < RG; ++g)
        a[g] = *reinterpret_cast<const float4*>(as + kk * BM + 4 * TY * g + ((4 * ty) ^ (8 * (kk / 4 % 4))));
#pragma unroll
      for (int h = 0; h < CG; ++h) b[h] = *reinterpret_cast<const ulonglong2*>(bs + kk * BN + 32 * h);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 q = a[i / 4];
        const unsigned long long av = twice((i & 3) == 0 ? q.x : (i & 3) == 1 ? q.y : (i & 3) == 2 ? q.z : q.w);
#pragma unroll
        for (int h = 0; h < CG; ++h) {
          acc[i][2 * h] = ffma2(av, b[h].x, acc[i][2 * h]);
          acc[i][2 * h + 1] = ffma2(av, b[h].y, acc[i][2 * h + 1]);
        }
      }
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  if (SUB) {
    close_part();
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int h = 0; h < 2 * CG; ++h) acc[i][h] = sum[SUB ? i : 0][SUB ? h : 0];
  }
  auto row_of = [&](int i) { return 4 * TY * (i / 4) + 4 * ty + (i & 3); };
  auto quad = [&](int i, int h) {
    float4 v;
    v.x = __uint_as_float((unsigned)acc[i][2 * h]);
    v.y = __uint_as_float((unsigned)(acc[i][2 * h] >> 32));
    v.z = __uint_as_float((unsigned)acc[i][2 * h + 1]);
    v.w = __uint_as_float((unsigned)(acc[i][2 * h + 1] >> 32));
    return v;
  };
  if (ks == 1) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int gm = m0 + row_of(i);
      if (gm >= M) continue;
#pragma unroll
      for (int h = 0; h < CG; ++h) {
        const int gn = n0 + 32 * h + 4 * tx;
        store4(Cm + gm * X.ldc + gn, quad(i, h), N - gn, vc);
      }
    }
  } else {
    // the cluster's partial tiles, added in slice order: block `rank` sums and stores its
    // share of the rows (every block reaches both cluster barriers)
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int h = 0; h < CG; ++h) *reinterpret_cast<float4*>(s_mem + row_of(i) * BN + 32 * h + 4 * tx) = quad(i, h);
    cluster_arrive();
    cluster_wait();
    const int rows = BM / ks;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(s_mem));
    for (int e = tid; e < rows * (BN / 4); e += THREADS) {
      const int m = rank * rows + e / (BN / 4), n = 4 * (e % (BN / 4));
      const uint32_t off = base + 4u * (m * BN + n);
      float4 v = ld_cluster_f4(off, 0);
      for (int r = 1; r < ks; ++r) {
        const float4 w = ld_cluster_f4(off, r);
        v.x += w.x;
        v.y += w.y;
        v.z += w.z;
        v.w += w.w;
      }
      if (m0 + m < M) store4(Cm + (m0 + m) * X.ldc + n0 + n, v, N - (n0 + n), vc);
    }
    cluster_arrive();
    cluster_wait();  // peers have read this block's tile before it leaves
  }
  if (!P.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------- FP64, small FP32
// FP64 is bound by the FP64 pipe (2 FMA per clock and SM: a warp instruction holds it for 16
// clocks), so what counts is that every SM gets the same share of the tiles and that no
// tile is padding; shared-memory and issue costs hide behind the pipe.  256 threads per
// block; tiles of T x T outputs, T = 32 (2 x 2 per thread), 16 (1 each) or 8 (1 each, four
// thread groups taking a quarter of each contraction slice).  Measured against tiles of 64 and
// 32 alone: operator of 64^2 (8 blocks of 32 x 32 before, 128 of 8 x 8 now) 23 -> 7 us with the
// launch, of 80^3 (each side of 80 padded to 128 before) 409 -> 207 us, 95% of the FP64 pipe
// (246 while whole rounds of 32 contraction steps were multiplied, 450^2 369 for 357).
// FP32 (T = 32): the unsplit operator of small grids, batch members above all, is a chain of load
// latencies in too few blocks to hide them; the 256 threads here have four times the loads in
// flight of the packed kernel's 64 (operator and march of 3 problems of 224^2: 65 us per step with
// the packed kernel, 45 so; 8 of 128^2 110 and 75).
template <typename real, int T, bool SUB>
__global__ void __launch_bounds__(256) frac_plain_kernel(const __grid_constant__ GemmPlan P);

template <typename real, int T, bool SUB = false>
struct PlainCfg {
  static constexpr int THREADS = 256;
  static constexpr int BM = T, BN = T, AMODE = 0;
  static auto kernel() { return frac_plain_kernel<real, T, SUB>; }
  static constexpr int BK = 32;
  static constexpr int KSL = T == 8 ? 4 : 1;     // in-block contraction groups
  static constexpr int TR = T == 32 ? 2 : 1;     // outputs per thread along either side
  static constexpr int L = (T * BK + 255) / 256; // elements per thread and operand
};

template <typename real, int T, bool SUB>
__global__ void __launch_bounds__(256)
frac_plain_kernel(const __grid_constant__ GemmPlan P) {
  using G = PlainCfg<real, T, SUB>;
  constexpr int BK = G::BK, TR = G::TR, KSL = G::KSL, PK = BK / KSL;
  static_assert(G::AMODE == 0, "A is read with k contiguous");
  __shared__ real As[2][T][BK + 1];
  __shared__ real Bs[2][BK][T];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (P.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const BlockAt at = locate_block(P, blockIdx.x, G::BM, G::BN);
  const GemmAxis& X = P.ax[at.a];
  const int m0 = at.m0, n0 = at.n0;
  const real* __restrict__ A = static_cast<const real*>(X.A) + at.bz * X.sA;
  const real* __restrict__ B = static_cast<const real*>(X.B) + at.bz * X.sB;
  real* __restrict__ Cm = static_cast<real*>(X.C) + at.bz * X.sC;
  const int M = X.M, N = X.N, K = X.K;
  const int tid = threadIdx.x;
  const int grp = tid / (256 / KSL), t = tid % (256 / KSL);
  const int ty = t / (T / TR), tx = t % (T / TR);

  real ra[G::L], rb[G::L];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < G::L; ++i) {
      const int e = tid + i * 256;
      const int m = m0 + e / BK, ka = k0 + e % BK;
      ra[i] = (m < M && ka < K) ? A[m * X.lda + ka] : static_cast<real>(0);
      const int kb = k0 + e / T, n = n0 + e % T;
      rb[i] = (kb < K && n < N) ? B[kb * X.ldb + n] : static_cast<real>(0);
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int i = 0; i < G::L; ++i) {
      const int e = tid + i * 256;
      As[buf][e / BK][e % BK] = ra[i];
      Bs[buf][e / T][e % T] = rb[i];
    }
  };
  real acc[TR][TR];
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int j = 0; j < TR; ++j) acc[i][j] = static_cast<real>(0);
  // the finished parts of the contraction (SUB, as in the packed kernel)
  real sum[TR][TR] = {};
  const int nkb = (K + kSlice - 1) / kSlice;
  int part = 1, kpart = SUB ? nkb / P.sub * kSlice : INT_MAX;
  auto close_part = [&]() {
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int j = 0; j < TR; ++j) {
        sum[i][j] += acc[i][j];
        acc[i][j] = static_cast<real>(0);
      }
  };
  fetch(0);
  stash(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    if (SUB && k0 >= kpart) {
      close_part();
      while (k0 >= kpart) kpart = ++part < P.sub ? part * nkb / P.sub * kSlice : INT_MAX;
    }
    const bool more = k0 + BK < K;
    if (more) fetch(k0 + BK);
    // (nothing past the end is multiplied: half a round, or a group's share of it)
#pragma unroll
    for (int q = 0; q < PK; ++q) {
      const int kk = grp * PK + q;
      if (q % 16 == 0 && k0 + kk >= K) break;
      real av[TR], bv[TR];
#pragma unroll
      for (int i = 0; i < TR; ++i) av[i] = As[buf][ty * TR + i][kk];
#pragma unroll
      for (int j = 0; j < TR; ++j) bv[j] = Bs[buf][kk][tx * TR + j];
#pragma unroll
      for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < TR; ++j) acc[i][j] += av[i] * bv[j];
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  if (SUB) {
    close_part();
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
      for (int j = 0; j < TR; ++j) acc[i][j] = sum[i][j];
  }
  if (KSL > 1) {  // the groups' sums, in contraction order (the operand buffers are idle)
    real* red = &As[0][0][0];
    red[grp * T * T + t] = acc[0][0];
    __syncthreads();
    if (grp == 0)
      for (int g = 1; g < KSL; ++g) acc[0][0] += red[g * T * T + t];
  }
  if (grp == 0) {
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const int gm = m0 + ty * TR + i;
#pragma unroll
      for (int j = 0; j < TR; ++j) {
        const int gn = n0 + tx * TR + j;
        if (gm < M && gn < N) Cm[gm * X.ldc + gn] = acc[i][j];
      }
    }
  }
  if (!P.early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------- host

void add_axis(GemmPlan& P, int BM, int BN, int M, int N, int K, int batch, int amode, const void* A, long long lda, long long sA,
              const void* B, long long ldb, long long sB, void* C, long long ldc, long long sC) {
  // (blocks of this axis = tiles x batch x P.ks)
  GemmAxis& X = P.ax[P.naxes++];
  X.A = A; X.B = B; X.C = C;
  X.lda = lda; X.sA = sA; X.ldb = ldb; X.sB = sB; X.ldc = ldc; X.sC = sC;
  X.M = M; X.N = N; X.K = K;
  X.amode = amode;
  auto quads = [](const void* p, long long ld, long long s) {
    return reinterpret_cast<uintptr_t>(p) % 16 == 0 && ld % 4 == 0 && s % 4 == 0;
  };
  X.vec = (quads(A, lda, sA) ? 1 : 0) | (quads(B, ldb, sB) ? 2 : 0) | (quads(C, ldc, sC) ? 4 : 0);
  X.tm = (M + BM - 1) / BM;
  X.tn = (N + BN - 1) / BN;
  X.begin = P.total;
  P.total += (long long)X.tm * X.tn * batch * P.ks;
}

// transpose = false: F_mu = K_mu applied along mu to C_mu, transpose = true: K_mu^T; the
// input of axis mu is the field at C + mu * cstride (cstride = 0: one input for every axis);
// BM x BN output tiles.  am = 1 (the packed kernel) reads the y and z axes' A (K_mu) from the other
// stored orientation, with the output index contiguous.
template <typename real>
GemmPlan make_plan(const lbm_s* h, const real* C, real* F, bool transpose, long long cstride, int BM, int BN, int ks, int am) {
  const int n0 = h->sp.n[0], n1 = h->sp.n[1], n2 = h->sp.n[2];
  const long long nodes = h->sp.nodes;
  const real* K = static_cast<const real*>(transpose ? h->dev.KT : h->dev.K);
  const real* KT = static_cast<const real*>(transpose ? h->dev.K : h->dev.KT);
  const real* KA = am ? KT : K;
  GemmPlan P{};
  P.ks = ks;
  P.sub = 1;
  long long koff = 0;
  // axis x: F_0 = C (rows x n0) * K_0^T
  add_axis(P, BM, BN, (int)(nodes / n0), n0, n0, 1, 0, C, n0, 0, KT + koff, n0, 0, F, n0, 0);
  koff += (long long)n0 * n0;
  // axis y: for each z-plane b, F_1[b] = K_1 * C[b]  (C[b] is n1 x n0)
  add_axis(P, BM, BN, n1, n0, n1, n2, am, KA + koff, n1, 0, C + cstride, n0, (long long)n1 * n0, F + nodes, n0,
           (long long)n1 * n0);
  koff += (long long)n1 * n1;
  // axis z: F_2 = K_2 * C  (C is n2 x (n1 n0))
  if (h->d == 3)
    add_axis(P, BM, BN, n2, n0 * n1, n2, 1, am, KA + koff, n2, 0, C + 2 * cstride, (long long)n0 * n1, 0, F + 2 * nodes,
             (long long)n0 * n1, 0);
  return P;
}

long long count_tiles(const lbm_s* h, int BM, int BN) {
  const long long n0 = h->sp.n[0], n1 = h->sp.n[1], n2 = h->sp.n[2];
  auto tiles = [=](long long m, long long n) { return ((m + BM - 1) / BM) * ((n + BN - 1) / BN); };
  long long t = tiles(h->sp.nodes / n0, n0) + tiles(n1, n0) * n2;
  if (h->d == 3) t += tiles(n2, n0 * n1);
  return t;
}


// FP32 block tiles: 32 x 32 where 64 x 64 tiles (times the contraction split) leave SMs
// without two blocks; else 128 x 64 unless its padding exceeds that of 64 x 64 tiles by 2%.
// The 32 x 32 tiles of a split run in rounds of 32 steps (a chain may end there); unsplit (batch
// members, short lines), up to two tiles per SM, on the plain kernel, and beyond in rounds of 64 (3 problems side by side, us
// per step, packed with rounds of 32 / 64 / plain: 224^2 65 / 58 / 45, 320^2 76 / 62 / 63, 416^2
// 94 / 84 / 97, 512^2 110 / 101 / 140).
template <class F>
auto with_tile32(const lbm_s* h, int ks, const F& f) {
  const long long t64 = count_tiles(h, 64, 64);
  if (t64 * ks < 2LL * device_sms()) {
    const bool sub = h->simt_sub > 1;
    if (ks == 1 && count_tiles(h, 32, 32) <= 2LL * device_sms())
      return sub ? f(PlainCfg<float, 32, true>{}) : f(PlainCfg<float, 32>{});
    // (several chains take 127 registers in rounds of 32: beyond six blocks per SM they no longer spread
    // evenly, 320^2 with 5.3 of them 11.8 us per step against 12.5 in rounds of 16, 352^2 with 6.4 19.6
    // against 13.2)
    if (sub && count_tiles(h, 32, 32) * ks > 6LL * device_sms()) return f(F32Cfg<1, 1, 8, 16, true>{});
    if (sub) return f(F32Cfg<1, 1, 8, 32, true>{});
    return ks > 1 ? f(F32Cfg<1, 1, 8, 32>{}) : f(F32Cfg<1, 1, 8, 64>{});
  }
  if (200 * count_tiles(h, 128, 64) > 102 * t64) return f(F32Cfg<2, 2, 8, 16>{});
  return f(F32Cfg<2, 2, 16, 16>{});
}

// FP64 tile side: the smallest share of the busiest SM, ceil(tiles / SMs) T^2 outputs, with
// the smaller tiles' extra shared and L2 reads weighted in
int tile64(const lbm_s* h) {
  const long long sms = device_sms();
  int best = 32;
  double best_cost = 0.0;
  for (int T : {32, 16, 8}) {
    const double cost = static_cast<double>((count_tiles(h, T, T) + sms - 1) / sms) * T * T * (T == 8 ? 1.3 : T == 16 ? 1.05 : 1.0);
    if (T == 32 || cost < best_cost) {
      best = T;
      best_cost = cost;
    }
  }
  return best;
}

// the grid of `blocks` blocks is resident at once (one wave).  Asked of the driver once per kernel
// and device: every launch needs the answer.
template <class Cfg>
bool blocks_fit(long long blocks) {
  static std::atomic<int> known[64];  // blocks per SM + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  int v = known[dev & 63].load(std::memory_order_relaxed);
  if (v == 0) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Cfg::kernel(), Cfg::THREADS, 0) != cudaSuccess)
      return false;
    known[dev & 63].store(v = per_sm + 1, std::memory_order_relaxed);
  }
  return blocks <= (long long)(v - 1) * device_sms();
}

template <typename real>
cudaError_t frac_all_axes(const lbm_s* h, const real* C, real* F, cudaStream_t s, bool transpose = false,
                          long long cstride = 0) {
  // programmatic dependent launch: the forward operator overlaps the previous collide-stream
  // kernel's tail where the handle has it on, the transpose that of the adjoint's step
  const bool pdl = transpose || h->pdl;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if constexpr (sizeof(real) == 8) {
    const int T = tile64(h);
    const GemmPlan P = make_plan<real>(h, C, F, transpose, cstride, T, T, 1, 0);
    cfg.gridDim = dim3(static_cast<unsigned>(P.total), 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    if (T == 32) return cudaLaunchKernelEx(&cfg, frac_plain_kernel<double, 32, false>, P);
    if (T == 16) return cudaLaunchKernelEx(&cfg, frac_plain_kernel<double, 16, false>, P);
    return cudaLaunchKernelEx(&cfg, frac_plain_kernel<double, 8, false>, P);
  } else {
    const int ks = h->simt_ks;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = ks;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    if (ks > 1) cfg.numAttrs = 2;
    return with_tile32(h, ks, [&](auto G) {
      GemmPlan P = make_plan<real>(h, C, F, transpose, cstride, G.BM, G.BN, ks, G.AMODE);
      // 2-D only: the 3-D marches' long blocks, launched early, would pile up two to an SM on
      // the SMs this grid leaves first (measured: 48^3 step 24 -> 37 us)
      P.early = !transpose && pdl && h->d == 2 && blocks_fit<decltype(G)>(P.total);
      P.sub = h->simt_sub;
      cfg.gridDim = dim3(static_cast<unsigned>(P.total), 1, 1);
      cfg.blockDim = dim3(G.THREADS, 1, 1);
      return cudaLaunchKernelEx(&cfg, G.kernel(), P);
    });
  }
}

}  // namespace

bool simt_one_wave(const lbm_s* h) {
  if (h->elem == 8) {
    const int T = tile64(h);
    const long long b = count_tiles(h, T, T);
    return T == 32 ? blocks_fit<PlainCfg<double, 32>>(b)
                   : T == 16 ? blocks_fit<PlainCfg<double, 16>>(b) : blocks_fit<PlainCfg<double, 8>>(b);
  }
  return with_tile32(h, h->simt_ks, [&](auto G) {
    return blocks_fit<decltype(G)>(count_tiles(h, G.BM, G.BN) * h->simt_ks);
  });
}

// Blocks that are launched early go to the SMs that the kernel before leaves first, several to an SM.
// Where an SM's share of the FP64 operator (two FMAs per clock) is some 4 us, the launch gap that this
// hides is worth more; beyond, the pile is the longer (step in us, launched early / not; runs of
// captured graphs, then of single launches: 24^3 7,700 FMAs per SM 21.9 / 22.4 and 22.4 / 27.9, 96^2
// 12,300 10.7 / 10.1 and 10.0 / 14.6, 32^3 24,600 33.0 / 27.4 and 33.5 / 32.0, 175^2 45.8 / 34.8 and
// 37.8 / 39.1, 256^2 330 / 83 and 144 / 88).
bool simt64_short(const lbm_s* h) {
  const int T = tile64(h);
  const long long per_sm = (count_tiles(h, T, T) + device_sms() - 1) / device_sms();
  return per_sm * T * T * std::max(h->sp.n[0], std::max(h->sp.n[1], h->sp.n[2])) <= 16384;
}

long long simt_blocks(const lbm_s* h) {
  if (h->elem == 8) return count_tiles(h, tile64(h), tile64(h));
  return with_tile32(h, h->simt_ks, [&](auto G) { return count_tiles(h, G.BM, G.BN) * h->simt_ks; });
}

// The split doubles while 64 x 64 tiles leave SMs without a block, or, up to four slices, while
// every slice keeps 80 contraction steps and the tiles leave fewer than eight blocks per SM
// (measured, us per step with 1/2/4/8 slices: 256^2 16.3 / 11.9 / 9.8 / 9.7, 384^2 22.1 / 16.7 /
// 14.7 / 16.0, 512^2 32.4 / 26.4 / 22.8 / 26.1, 700 x 600 52 / 48 / 40 / 48, 1024^2 123 / 117 / 105 /
// 117; 3-D with 1/2: 48^3 15.7 / 17.5, 64^3 15.8 / 18.6, 72^3 28.7 / 39.2).  The longer axis sets
// the most slices in 2-D (by the shorter one: 1000 x 60 29.3 us against 14.5, 53 x 1001 35.8 and 15.2).
// 2-D lines of at most 64 stay whole: the cluster costs more than the half of the contraction that it
// takes off a block (32 steps from a reset, two slices / plain unsplit in two chains: 48^2 331 / 291 us, 64^2 322 / 284).
int simt_ksplit(const lbm_s* h) {
  if (h->elem != 4) return 1;
  const long long tiles = count_tiles(h, 64, 64), sms = device_sms();
  int kmin = 1 << 30, kmax = 0;
  for (int mu = 0; mu < h->d; ++mu) {
    kmin = std::min(kmin, h->sp.n[mu]);
    kmax = std::max(kmax, h->sp.n[mu]);
  }
  // 2-D: as many slices as the longer axis has, the shorter one's last slices then being empty
  const int kbs = ((h->d == 2 ? kmax : kmin) + kSlice - 1) / kSlice;
  int ks = 1;
  while (kmax > (h->d == 2 ? 64 : 0) && ks * 2 <= 8 && ks * 2 <= kbs &&
         (tiles * ks < sms - sms / 10 || (ks < 4 && tiles * ks < 8 * sms && kmin >= 160 * ks))) ks *= 2;
  return ks;
}

// Parts of a slice that are summed on their own with the built-in split (one that is asked for is taken
// as it is, and a batch's members are unsplit).  An FP32 chain of additions rounds at the scale of its running sum, so the
// contraction is cut in as many chains as fill the GPU with two 64 x 64 tiles per SM, at least 32
// steps each; where the built-in split has fewer slices than that (300^2 four of eight, 64^3 one of
// two), a block sums its part of them one after the other.  Error of C against 64 bits, one chain
// per slice / so: 64^3, 8 steps, 1.6e-7 / 1.4e-7.  The registers for it are there in the 32 x 32 tiles,
// which serve every such grid.
int simt_sub(const lbm_s* h) {
  if (h->elem != 4) return 1;
  const long long tiles = count_tiles(h, 64, 64);
  int kmin = 1 << 30;
  for (int mu = 0; mu < h->d; ++mu) kmin = std::min(kmin, h->sp.n[mu]);
  const int kbs = (kmin + kSlice - 1) / kSlice;
  int chains = 1;
  while (chains * 2 <= 8 && chains * 2 <= kbs && tiles * chains < 2LL * device_sms()) chains *= 2;
  return tiles * h->simt_ks < 2LL * device_sms() ? std::max(1, chains / h->simt_ks) : 1;
}

cudaError_t launch_frac_simt_T(const lbm_s* h, const void* in, long long in_stride, void* out, cudaStream_t s) {
  if (h->elem == 8)
    return frac_all_axes<double>(h, static_cast<const double*>(in), static_cast<double*>(out), s, true, in_stride);
  return frac_all_axes<float>(h, static_cast<const float*>(in), static_cast<float*>(out), s, true, in_stride);
}

cudaError_t launch_frac_simt(const lbm_s* h, const void* C, void* F, cudaStream_t s) {
  // spatially varying g: the input along mu is G_mu = g_mu(x) C (Eq. Fg), one field per axis
  const long long cs = (h->fld.on && h->fld.G) ? h->sp.nodes : 0;
  if (h->fld.on && h->fld.G) C = h->fld.G;
  if (h->elem == 8)
    return frac_all_axes<double>(h, static_cast<const double*>(C), static_cast<double*>(F), s, false, cs);
  return frac_all_axes<float>(h, static_cast<const float*>(C), static_cast<float*>(F), s, false, cs);
}

}  // namespace lbm
