// Active-active orbital rotation of the integrals and its adjoint
// (Sec. III.A: the integrals depend on kappa through U = exp(kappa);
// Sec. III.B, Eq. vdedk2: dE/dkappa = sum dH/dkappa contracted with the RDMs).
//
// Forward:  h' = U^T h U,  (pq|rs)' = sum U_ap U_bq U_cr U_ds (ab|cd)
//           as four quarter transforms out[J][p] = sum_a in[a][J] M[a][p]
//           that each rotate the leading index to the back.
// Backward: dE/dh = U g1 U^T, dE/d(ab|cd) = sum D_pqrs U_ap U_bq U_cr U_ds
//           with D = rdm2/2, and dE/dU = h U g1^T + h^T U g1 + 4 sum_bcd
//           (xb|cd) T[d][c][b][y], T = D with its first three indices
//           back-transformed (the four index positions of a real state with
//           8-fold symmetric integrals contribute equally, so the position
//           left out is the last: T is three quarter transforms of D, and
//           the fourth gives dE/d(ab|cd));
//           dE/dkappa = L_exp(kappa^T, dE/dU), the Frechet derivative of
//           exp at kappa^T, by the derivative of every step of exp.
// The quarter transforms (the n^5 part) run on the bf16 tensor cores as
// exact digit products rounded once to FP64 (qtrans_tc.cu); the n x n
// matrix work stays on the FP64 pipe.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "hci_internal.cuh"

namespace {

// ---------------------------------------------------------------------------
// n x n matrix chains (n <= 64) in one launch: one thread-block cluster, each
// CTA owning a block of the entries of every matrix; a product reads its
// operands from global memory (L2) into shared memory, and the cluster's
// barrier separates the products that depend on one another.
//
// exp(X) is the Taylor polynomial of degree 16 of X = kappa / 2^s, |X|_1 <=
// 1/2 (remainder below 3e-20), with its blocks of four powers by Horner's rule in
// X^4 (Paterson and Stockmeyer, SIAM J. Comput. 1973): 6 products where the
// term-by-term rule takes 17, then s squarings.  On FP64 issue alone a
// product of 44 x 44 matrices takes 1.4 us over 16 SMs; as separate launches
// (6.9 us a product, 1.5 us a Horner step, and the host's wait for the norm)
// exp took 200 us; the whole chain, h' = U^T h U included, takes 46 us at 44
// orbitals and 15 us at 10 (one CTA).
// ---------------------------------------------------------------------------
constexpr int CLM_T = 128;          // threads per CTA: one warp per FP64 pipe
constexpr int CLM_NU = 4;           // entries per thread at most (8 CTAs: 16 x 32 of 64 x 64)
constexpr int CLM_BI = 16, CLM_BJ = 32;

// Without .aligned, which asks that a warp's threads execute the barrier
// together: cl_mm's loops and epilogues end thread by thread (a block of
// 5 x 5 entries, the triangle of h), and nothing says where the warp meets
// again.
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ int cl_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int cl_size() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

// this CTA's block of every matrix
struct Tile {
  int i0, j0, ni, nj, cnt;
  int rn, rj;            // ceil(2^18 / n), ceil(2^18 / nj)
};
__device__ __forceinline__ Tile cl_tile(int n) {
  const int c = cl_size(), r = cl_rank();
  const int R = c >= 4 ? 4 : 1, C = c / R;
  const int bi = (n + R - 1) / R, bj = (n + C - 1) / C;
  Tile t;
  t.i0 = (r % R) * bi;
  t.j0 = (r / R) * bj;
  t.ni = min(bi, n - t.i0);
  t.nj = min(bj, n - t.j0);
  if (t.ni < 0) t.ni = 0;
  if (t.nj < 0) t.nj = 0;
  t.cnt = t.ni * t.nj;
  t.rn = ((1 << 18) + n - 1) / n;
  t.rj = t.nj > 0 ? ((1 << 18) + t.nj - 1) / t.nj : 0;
  return t;
}

struct MM {
  const double* A;
  const double* B;
  int tA, tB;            // transposed
};

// epi(u, i, j, v) for every entry (i, j) of the CTA's block, v = sum over the
// terms of (op(A) op(B))_ij, u < CLM_NU the thread's entry number (the same
// entry in every call).  Operands written in this kernel are read through
// L2, after cl_sync.
template <int NT, class F>
__device__ __forceinline__ void cl_mm(int n, const Tile& t, const MM (&terms)[NT], double* sA, double* sB, F epi) {
  double acc[CLM_NU], acc2[CLM_NU];     // two chains: one alone waits for its own latency
#pragma unroll
  for (int u = 0; u < CLM_NU; ++u) acc[u] = acc2[u] = 0.0;
  const int na = t.ni * n, nb = n * t.nj, most = na > nb ? na : nb;
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    const MM& m = terms[q];
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < most; e += CLM_T) {
      // e / n and e / nj by multiplication (exact for e < 2^12)
      const int i = (e * t.rn) >> 18, k = e - i * n, kb = (e * t.rj) >> 18, j = e - kb * t.nj;
      double va = 0.0, vb = 0.0;
      if (e < na) va = __ldcg(m.tA ? m.A + k * n + t.i0 + i : m.A + (t.i0 + i) * n + k);
      if (e < nb) vb = __ldcg(m.tB ? m.B + (t.j0 + j) * n + kb : m.B + kb * n + t.j0 + j);
      if (e < na) sA[e] = va;
      if (e < nb) sB[e] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < CLM_NU; ++u) {
      const int o = threadIdx.x + u * CLM_T;
      if (o >= t.cnt) break;
      const int i = (o * t.rj) >> 18, j = o - i * t.nj;
      const double* a = sA + i * n;
      const double* b = sB + j;
      double v = acc[u], v2 = acc2[u];
      int k = 0;
#pragma unroll 4
      for (; k + 2 <= n; k += 2) {
        v = fma(a[k], b[k * t.nj], v);
        v2 = fma(a[k + 1], b[(k + 1) * t.nj], v2);
      }
      if (k < n) v = fma(a[k], b[k * t.nj], v);
      acc[u] = v;
      acc2[u] = v2;
    }
  }
#pragma unroll
  for (int u = 0; u < CLM_NU; ++u) {
    const int o = threadIdx.x + u * CLM_T;
    if (o >= t.cnt) break;
    const int i = (o * t.rj) >> 18;
    epi(u, t.i0 + i, t.j0 + (o - i * t.nj), acc[u] + acc2[u]);
  }
}

// 1 / k!
__device__ constexpr double INV_FACT[17] = {
    1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320, 1.0 / 362880, 1.0 / 3628800,
    1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0, 1.0 / 87178291200.0, 1.0 / 1307674368000.0,
    1.0 / 20922789888000.0};

// Work matrices of the chains (n x n each) and their status words.
enum { W_X = 0, W_X2, W_X3, W_X4, W_S0, W_S1, W_S2, W_E, W_F, W_T, W_T2, W_UT, W_UTH, W_GU, W_FWD_COUNT = W_T + 1,
       W_D1 = W_GU + 1, W_D2, W_D3, W_D4, W_DS0, W_DS1, W_DS2, W_DE, W_DF, W_COUNT };
struct RotStatus {
  int nonfinite;     // |kappa|_1 is not finite: every later kernel of the call returns at once, so that the
                     // outputs stay as they were
  int timeout;       // a quarter transform gave up waiting for its products
  int squarings;
  int bad_gradient;  // dE/dU is infinite
};

struct ChainArgs {
  int n;
  const double* kappa;
  const double* h;
  double* U;
  double* h_out;        // forward: U^T h U, exactly symmetric
  const double* g1;     // backward
  double* dh;           // backward: U g1 U^T, or NULL
  int want_gu;          // backward: h-part of dE/dU
  double* ws;
  RotStatus* status;
};

template <bool BWD>
__global__ void __launch_bounds__(CLM_T) k_exp_chain(ChainArgs A) {
  __shared__ double sA[CLM_BI * HCI_MAXORB], sB[HCI_MAXORB * CLM_BJ];
  __shared__ double s_nrm[CLM_T];
  const int n = A.n, nn = n * n, tid = threadIdx.x;
  double* ws = A.ws;
  auto W = [&](int k) { return ws + (size_t)k * nn; };
  // 1-norm, by every CTA for itself: thread = column, rows in halves
  {
    const int j = tid & 63, half = tid >> 6;
    double c = 0.0;
    if (j < n)
      for (int i = half; i < n; i += 2) c += fabs(A.kappa[i * n + j]);
    s_nrm[tid] = c;
    __syncthreads();
    if (tid < 64) s_nrm[tid] += s_nrm[tid + 64];
    __syncthreads();
    if (tid < 32) {
      double v = fmax(fmax(0.0, s_nrm[tid]), s_nrm[tid + 32]);
      for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (tid == 0) s_nrm[0] = v;
    }
    __syncthreads();
  }
  const double nrm = s_nrm[0];
  if (!isfinite(nrm)) {
    if (cl_rank() == 0 && tid == 0) A.status->nonfinite = 1;
    return;   // the same in every CTA
  }
  int s = 0;
  while (ldexp(nrm, -s) > 0.5) ++s;
  const double sc = ldexp(1.0, -s);
  if (cl_rank() == 0 && tid == 0) A.status->squarings = s;
  const Tile t = cl_tile(n);
  double x[CLM_NU], x2[CLM_NU], x3[CLM_NU];
  const MM m2[1] = {{A.kappa, A.kappa, 0, 0}};
  cl_mm(n, t, m2, sA, sB, [&](int u, int i, int j, double v) {
    x[u] = A.kappa[i * n + j] * sc;
    x2[u] = v * sc * sc;
    if (BWD) W(W_X)[i * n + j] = x[u];
    W(W_X2)[i * n + j] = x2[u];
  });
  cl_sync();
  const MM m3[1] = {{W(W_X2), A.kappa, 0, 0}};
  cl_mm(n, t, m3, sA, sB, [&](int u, int i, int j, double v) {
    x3[u] = v * sc;
    if (BWD) W(W_X3)[i * n + j] = x3[u];
  });
  const MM m4[1] = {{W(W_X2), W(W_X2), 0, 0}};
  auto blk = [&](int b, int u, int i, int j) {
    double v = i == j ? INV_FACT[b] : 0.0;
    v = fma(INV_FACT[b + 1], x[u], v);
    v = fma(INV_FACT[b + 2], x2[u], v);
    return fma(INV_FACT[b + 3], x3[u], v);
  };
  cl_mm(n, t, m4, sA, sB, [&](int u, int i, int j, double v) {
    W(W_X4)[i * n + j] = v;
    W(W_S0)[i * n + j] = fma(INV_FACT[16], v, blk(12, u, i, j));
  });
  cl_sync();
  const MM h1[1] = {{W(W_X4), W(W_S0), 0, 0}}, h2[1] = {{W(W_X4), W(W_S1), 0, 0}}, h3[1] = {{W(W_X4), W(W_S2), 0, 0}};
  cl_mm(n, t, h1, sA, sB, [&](int u, int i, int j, double v) { W(W_S1)[i * n + j] = v + blk(8, u, i, j); });
  cl_sync();
  cl_mm(n, t, h2, sA, sB, [&](int u, int i, int j, double v) { W(W_S2)[i * n + j] = v + blk(4, u, i, j); });
  cl_sync();
  auto store_u = [&](int i, int j, double v) {
    A.U[i * n + j] = v;
    if (BWD) {
      W(W_UT)[j * n + i] = v;
      W(W_UTH)[j * n + i] = 0.5 * v;
    }
  };
  cl_mm(n, t, h3, sA, sB, [&](int u, int i, int j, double v) {
    v += blk(0, u, i, j);
    W(W_E)[i * n + j] = v;
    if (s == 0) store_u(i, j, v);
  });
  cl_sync();
  // squarings (the backward keeps W_E, the exponential of the scaled matrix)
  int from = W_E, to = W_F;
  for (int q = 0; q < s; ++q) {
    const MM sq[1] = {{W(from), W(from), 0, 0}};
    cl_mm(n, t, sq, sA, sB, [&](int u, int i, int j, double v) {
      W(to)[i * n + j] = v;
      if (q == s - 1) store_u(i, j, v);
    });
    cl_sync();
    const int old = from;
    from = to;
    to = old == W_E ? W_T : old;
  }
  if (!BWD) {
    const MM a[1] = {{A.h, A.U, 0, 0}};
    cl_mm(n, t, a, sA, sB, [&](int u, int i, int j, double v) { W(W_S0)[i * n + j] = v; });
    cl_sync();
    // the upper triangle's values on both sides
    const MM b[1] = {{A.U, W(W_S0), 1, 0}};
    cl_mm(n, t, b, sA, sB, [&](int u, int i, int j, double v) {
      if (i <= j) {
        A.h_out[i * n + j] = v;
        A.h_out[j * n + i] = v;
      }
    });
  } else {
    const MM a[1] = {{A.g1, A.U, 0, 1}}, b[1] = {{A.h, A.U, 0, 0}}, c[1] = {{A.h, A.U, 1, 0}};
    if (A.dh) cl_mm(n, t, a, sA, sB, [&](int u, int i, int j, double v) { W(W_D1)[i * n + j] = v; });
    if (A.want_gu) {
      cl_mm(n, t, b, sA, sB, [&](int u, int i, int j, double v) { W(W_T)[i * n + j] = v; });
      cl_mm(n, t, c, sA, sB, [&](int u, int i, int j, double v) { W(W_T2)[i * n + j] = v; });
    }
    cl_sync();
    if (A.want_gu) {
      const MM d[2] = {{W(W_T), A.g1, 0, 1}, {W(W_T2), A.g1, 0, 0}};
      cl_mm(n, t, d, sA, sB, [&](int u, int i, int j, double v) { W(W_GU)[i * n + j] = v; });
    }
    if (A.dh) {
      cl_sync();          // dh may be g1's or h's own buffer
      const MM e[1] = {{A.U, W(W_D1), 0, 0}};
      cl_mm(n, t, e, sA, sB, [&](int u, int i, int j, double v) { A.dh[i * n + j] = v; });
    }
  }
}

// dkappa = L_exp(kappa^T, G), G = W_GU: the derivative of every step of the
// chain above at X^T (whose powers are the stored ones transposed) along
// dX = G / 2^s; 12 products.  dkappa is left as it is when G is infinite.
__global__ void __launch_bounds__(CLM_T) k_exp_adjoint(ChainArgs A, double* __restrict__ dkappa) {
  __shared__ double sA[CLM_BI * HCI_MAXORB], sB[HCI_MAXORB * CLM_BJ];
  if (A.status->nonfinite) return;
  const int n = A.n, nn = n * n, s = A.status->squarings;
  const double sc = ldexp(1.0, -s);
  double* ws = A.ws;
  auto W = [&](int k) { return ws + (size_t)k * nn; };
  const Tile t = cl_tile(n);
  double d1[CLM_NU], d2[CLM_NU], d3[CLM_NU];
  // products with G itself, scaled in the epilogue
  const MM p2[2] = {{W(W_X), W(W_GU), 1, 0}, {W(W_GU), W(W_X), 0, 1}};
  cl_mm(n, t, p2, sA, sB, [&](int u, int i, int j, double v) {
    const double g = __ldcg(W(W_GU) + i * n + j);
    if (isinf(g)) A.status->bad_gradient = 1;
    d1[u] = g * sc;
    d2[u] = v * sc;
    W(W_D1)[i * n + j] = d1[u];
    W(W_D2)[i * n + j] = d2[u];
  });
  cl_sync();
  if (__ldcg(&A.status->bad_gradient)) return;   // written before the barrier only: the same in every CTA
  const MM p3[2] = {{W(W_X2), W(W_D1), 1, 0}, {W(W_D2), W(W_X), 0, 1}};
  cl_mm(n, t, p3, sA, sB, [&](int u, int i, int j, double v) { d3[u] = v; });
  const MM p4[2] = {{W(W_X2), W(W_D2), 1, 0}, {W(W_D2), W(W_X2), 0, 1}};
  auto blk = [&](int b, int u) {
    return fma(INV_FACT[b + 1], d1[u], fma(INV_FACT[b + 2], d2[u], INV_FACT[b + 3] * d3[u]));
  };
  cl_mm(n, t, p4, sA, sB, [&](int u, int i, int j, double v) {
    W(W_D4)[i * n + j] = v;
    W(W_DS0)[i * n + j] = fma(INV_FACT[16], v, blk(12, u));
  });
  cl_sync();
  const MM q1[2] = {{W(W_X4), W(W_DS0), 1, 0}, {W(W_D4), W(W_S0), 0, 1}};
  cl_mm(n, t, q1, sA, sB, [&](int u, int i, int j, double v) { W(W_DS1)[i * n + j] = v + blk(8, u); });
  cl_sync();
  const MM q2[2] = {{W(W_X4), W(W_DS1), 1, 0}, {W(W_D4), W(W_S1), 0, 1}};
  cl_mm(n, t, q2, sA, sB, [&](int u, int i, int j, double v) { W(W_DS2)[i * n + j] = v + blk(4, u); });
  cl_sync();
  const MM q3[2] = {{W(W_X4), W(W_DS2), 1, 0}, {W(W_D4), W(W_S2), 0, 1}};
  cl_mm(n, t, q3, sA, sB, [&](int u, int i, int j, double v) {
    v += blk(0, u);
    if (s == 0) dkappa[i * n + j] = v;
    else W(W_DE)[i * n + j] = v;
  });
  // E <- E^2, dE <- E^T dE + dE E^T
  int e0 = W_E, e1 = W_F, f0 = W_DE, f1 = W_DF;
  for (int q = 0; q < s; ++q) {
    cl_sync();
    const MM r[2] = {{W(e0), W(f0), 1, 0}, {W(f0), W(e0), 0, 1}};
    cl_mm(n, t, r, sA, sB, [&](int u, int i, int j, double v) {
      if (q == s - 1) dkappa[i * n + j] = v;
      else W(f1)[i * n + j] = v;
    });
    if (q < s - 1) {
      const MM sq[1] = {{W(e0), W(e0), 0, 0}};
      cl_mm(n, t, sq, sA, sB, [&](int u, int i, int j, double v) { W(e1)[i * n + j] = v; });
    }
    int w = e0; e0 = e1; e1 = w;
    w = f0; f0 = f1; f1 = w;
  }
}

// The solver reads different permutations of one integral (heat-bath lists,
// Slater-Condon rules), so every permutation must hold the same bits: each
// element of the 8-fold orbit of (pq|rs) takes the value of the orbit's
// representative ((a,b) = sorted (p,q), (c,d) = sorted (r,s), pairs ordered
// so that (a,b) <= (c,d)), and h_pq = h_qp takes the value of h_min,max.  In
// place: a representative is only ever rewritten with its own value.
__global__ void k_sym8(int n, double* __restrict__ eri, const RotStatus* __restrict__ status) {
  if (status->nonfinite) return;
  const int64_t n2 = (int64_t)n * n, n4 = n2 * n2;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
    const int s = (int)(t % n), r = (int)((t / n) % n), q = (int)((t / n2) % n), p = (int)(t / (n2 * n));
    int a = p < q ? p : q, b = p < q ? q : p, c = r < s ? r : s, d = r < s ? s : r;
    if (a * n + b > c * n + d) {
      const int ta = a, tb = b;
      a = c; b = d; c = ta; d = tb;
    }
    const int64_t rep = (((int64_t)a * n + b) * n + c) * n + d;
    if (rep != t) eri[t] = eri[rep];
  }
}
// part[b][x][y] = block b's share of sum_J eri[J][x] T[y][J], J = (d, c, b):
// the leading pair's symmetry of eri, (dc|bx) = (cd|bx), leaves the pairs
// d <= c with T[y][d][c][b] + T[y][c][d][b] (d < c), half the FP64 products
// that bound this contraction.  Every block takes an equal share of the
// n^2 (n + 1) / 2 rows, NT_CH staged at a time; thread t owns entries
// t, t + 256, ... (44 orbitals: 302 us for all of J, 156 us so with
// three blocks per SM, 170 with two).
constexpr int NT_CH = 48;
template <int NACC>
__global__ void __launch_bounds__(256) k_gemm_nt_part(int n, int64_t rows, const double* __restrict__ eri,
                                                      const double* __restrict__ T, double* __restrict__ part) {
  extern __shared__ double sm[];
  double* sE = sm;                 // [NT_CH][n] (x fastest)
  double* sT = sm + NT_CH * n;     // [NT_CH][n + 1] (y fastest)
  const int nn = n * n, ld = n + 1;
  const int64_t n3 = (int64_t)nn * n;
  const int64_t r0 = rows * blockIdx.x / gridDim.x, r1 = rows * (blockIdx.x + 1) / gridDim.x;
  double acc[NACC];
#pragma unroll
  for (int u = 0; u < NACC; ++u) acc[u] = 0.0;
  for (int64_t rr = r0; rr < r1; rr += NT_CH) {
    const int cnt = r1 - rr < NT_CH ? (int)(r1 - rr) : NT_CH;
    __syncthreads();
    // row q = (pair t = c (c + 1) / 2 + d with d <= c, b)
    for (int e = threadIdx.x; e < cnt * n; e += 256) {
      const int k = e / n, x = e - k * n;
      const int64_t q = rr + k;
      const int tp = (int)(q / n), b = (int)(q - (int64_t)tp * n);
      int c = (int)((sqrtf(8.0f * (float)tp + 1.0f) - 1.0f) * 0.5f);
      while (c * (c + 1) / 2 > tp) --c;
      while ((c + 1) * (c + 2) / 2 <= tp) ++c;
      const int d = tp - c * (c + 1) / 2;
      sE[k * n + x] = eri[((int64_t)(d * n + c) * n + b) * n + x];
    }
    for (int e = threadIdx.x; e < cnt * n; e += 256) {
      const int y = e / cnt, k = e - y * cnt;
      const int64_t q = rr + k;
      const int tp = (int)(q / n), b = (int)(q - (int64_t)tp * n);
      int c = (int)((sqrtf(8.0f * (float)tp + 1.0f) - 1.0f) * 0.5f);
      while (c * (c + 1) / 2 > tp) --c;
      while ((c + 1) * (c + 2) / 2 <= tp) ++c;
      const int d = tp - c * (c + 1) / 2;
      double v = T[(int64_t)y * n3 + (int64_t)(d * n + c) * n + b];
      if (d != c) v += T[(int64_t)y * n3 + (int64_t)(c * n + d) * n + b];
      sT[k * ld + y] = v;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NACC; ++u) {
      const int o = threadIdx.x + 256 * u;
      if (o < nn) {
        const int x = o % n, y = o / n;
        double v = acc[u];
#pragma unroll 8
        for (int k = 0; k < cnt; ++k) v = fma(sE[k * n + x], sT[k * ld + y], v);
        acc[u] = v;
      }
    }
  }
#pragma unroll
  for (int u = 0; u < NACC; ++u) {
    const int o = threadIdx.x + 256 * u;
    if (o < nn) part[(int64_t)blockIdx.x * nn + o] = acc[u];
  }
}

// out[x][y] += scale * sum of the parts' [y][x], 32 entries per block, the
// parts in eight slices
__global__ void __launch_bounds__(256) k_sum_parts(int n, int nparts, const double* __restrict__ part, double scale,
                                                   double* __restrict__ out) {
  __shared__ double red[8][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane, nn = n * n;
  double s = 0.0;
  if (o < nn)
#pragma unroll 4
    for (int b = w; b < nparts; b += 8) s += part[(int64_t)b * nn + o];
  red[w][lane] = s;
  __syncthreads();
  if (w == 0 && o < nn) {
    s = 0.0;
    for (int k = 0; k < 8; ++k) s += red[k][lane];
    out[(o % n) * n + o / n] += scale * s;
  }
}

struct Scratch {
  cudaStream_t st;
  void* ptrs[16];
  int count = 0;
  int64_t left = hci_fail_alloc_env();   // host-side fault injection (tests)
  double* get(size_t doubles) {
    void* p = nullptr;
    if (left == 0) return nullptr;
    if (left > 0) --left;
    if (cudaMallocAsync(&p, doubles * 8 + 64, st) != cudaSuccess) return nullptr;
    ptrs[count++] = p;
    return reinterpret_cast<double*>(p);
  }
  ~Scratch() {
    for (int i = 0; i < count; ++i) cudaFreeAsync(ptrs[i], st);
  }
};

inline unsigned blocks(int64_t work, int b = 256) { return (unsigned)((work + b - 1) / b); }

// CTAs of a chain's cluster: one for 16 orbitals or fewer (a product is then
// shorter than the cluster's barrier), else 16 where the device can hold
// such a cluster (an opt-in size), or the portable 8.  Looked up once per
// device.
int chain_ctas(int n) {
  if (n <= 16) return 1;
  static std::atomic<int> known[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
  int c = known[dev].load();
  if (c) return c;
  c = 8;
  const void* fns[3] = {(const void*)k_exp_chain<false>, (const void*)k_exp_chain<true>, (const void*)k_exp_adjoint};
  bool ok = true;
  for (const void* f : fns) ok = ok && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  if (ok) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(CLM_T);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 16;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int nc = 0;
    for (const void* f : fns) {
      ok = ok && cudaOccupancyMaxActiveClusters(&nc, f, &cfg) == cudaSuccess && nc >= 1;
    }
    if (ok) c = 16;
  }
  cudaGetLastError();
  known[dev].store(c);
  return c;
}

template <class... P, class... Q>
cudaError_t launch_chain(cudaStream_t st, int n, void (*k)(P...), Q... args) {
  cudaLaunchConfig_t cfg = {};
  const int c = chain_ctas(n);
  cfg.gridDim = dim3((unsigned)c);
  cfg.blockDim = dim3(CLM_T);
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)c;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  hci_count_launch();
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// out[J*n + p] = sum_a in[a*N3 + J] * M[a*n + p], J < N3 = n^3
#define QTRANS(who, in, M, out, flag, skip)                                                  \
  do {                                                                                       \
    if (qtrans_tc(st, n, in, M, out, flag, skip) != HCI_OK)                                      \
      return hci_fail(nullptr, HCI_ERR_CUDA, who ": quarter transform launch failed: %s",     \
                      cudaGetErrorString(cudaGetLastError()));                               \
  } while (0)

// the call's status words read and judged (synchronises st)
hci_status chain_status(const char* who, cudaStream_t st, const RotStatus* dev) {
  RotStatus h = {};
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, dev, sizeof h, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return hci_fail(nullptr, HCI_ERR_CUDA, "%s: %s", who, cudaGetErrorString(e));
  if (h.nonfinite) return hci_fail(nullptr, HCI_ERR_INVALID, "%s: matrix exponential failed", who);
  if (h.bad_gradient) return hci_fail(nullptr, HCI_ERR_INVALID, "%s: Frechet exponential failed", who);
  if (h.timeout)
    return hci_fail(nullptr, HCI_ERR_CUDA, "%s: a quarter transform gave up waiting for its tensor-core products", who);
  return HCI_OK;
}

// ws: W_FWD_COUNT n x n matrices and the status words; t4: n^4
hci_status rotate_core(const char* who, cudaStream_t st, int n, const double* kappa, const double* h, const double* eri,
                       double* U, double* h_out, double* eri_out, double* ws, double* t4) {
  RotStatus* status = reinterpret_cast<RotStatus*>(ws + (size_t)W_FWD_COUNT * n * n);
  ChainArgs A = {};
  A.n = n; A.kappa = kappa; A.h = h; A.U = U; A.h_out = h_out; A.ws = ws; A.status = status;
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(RotStatus), st);
  if (e == cudaSuccess) e = launch_chain(st, n, k_exp_chain<false>, A);
  if (e != cudaSuccess) return hci_fail(nullptr, HCI_ERR_CUDA, "%s: %s", who, cudaGetErrorString(e));
  QTRANS("hci_rotate", eri, U, t4, &status->timeout, &status->nonfinite);
  QTRANS("hci_rotate", t4, U, eri_out, &status->timeout, &status->nonfinite);
  QTRANS("hci_rotate", eri_out, U, t4, &status->timeout, &status->nonfinite);
  QTRANS("hci_rotate", t4, U, eri_out, &status->timeout, &status->nonfinite);
  // exact permutational symmetry of the rotated integrals (see k_sym8)
  HCI_LAUNCH(k_sym8, (unsigned)std::min<int64_t>(blocks((int64_t)n * n * n * n), 4096), 256, 0, st)(n, eri_out, status);
  return chain_status(who, st, status);
}

}  // namespace

extern "C" hci_status hci_rotate(int norb, const double* kappa, const double* h, const double* eri, double* U,
                                 double* h_out, double* eri_out, void* stream) {
  const int n = norb;
  if (n < 1 || n > HCI_MAXORB) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate: norb=%d outside [1,64]", n);
  if (!kappa || !h || !eri || !U || !h_out || !eri_out)
    return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate: null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  Scratch S{st};
  const size_t n2 = (size_t)n * n, n4 = n2 * n2;
  double *ws = S.get(W_FWD_COUNT * n2 + 2), *t4 = S.get(n4);
  if (!ws || !t4)
    return hci_fail(nullptr, HCI_ERR_NOMEM, "hci_rotate: allocation failed%s",
                    S.left == 0 ? " (injected by HCI_FAIL_ALLOC_AFTER)" : "");
  return rotate_core("hci_rotate", st, n, kappa, h, eri, U, h_out, eri_out, ws, t4);
}

extern "C" hci_status hci_rotate_backward(int norb, const double* kappa, const double* h, const double* eri,
                                          const double* rdm1, const double* rdm2, double* dh, double* deri,
                                          double* dkappa, void* stream) {
  const int n = norb;
  if (n < 1 || n > HCI_MAXORB)
    return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate_backward: norb=%d outside [1,64]", n);
  if (!kappa || !h || !eri || !rdm1 || !rdm2)
    return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate_backward: null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  Scratch S{st};
  const size_t n2 = (size_t)n * n, n4 = n2 * n2;
  const int64_t rows = (int64_t)n2 * (n + 1) / 2;
  const int nparts = (int)std::min<int64_t>(3 * hci_nsm(), (rows + 15) / 16);
  double *ws = S.get(W_COUNT * n2 + 2), *U = S.get(n2), *ta = S.get(n4), *tb = S.get(n4);
  double* part = dkappa ? S.get((size_t)nparts * n2) : nullptr;
  if (!ws || !U || !ta || !tb || (dkappa && !part))
    return hci_fail(nullptr, HCI_ERR_NOMEM, "hci_rotate_backward: allocation failed%s",
                    S.left == 0 ? " (injected by HCI_FAIL_ALLOC_AFTER)" : "");
  RotStatus* status = reinterpret_cast<RotStatus*>(ws + W_COUNT * n2);
  ChainArgs A = {};
  A.n = n; A.kappa = kappa; A.h = h; A.U = U; A.g1 = rdm1; A.dh = dh; A.want_gu = dkappa != nullptr; A.ws = ws;
  A.status = status;
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(RotStatus), st);
  if (e == cudaSuccess) e = launch_chain(st, n, k_exp_chain<true>, A);
  if (e != cudaSuccess) return hci_fail(nullptr, HCI_ERR_CUDA, "hci_rotate_backward: %s", cudaGetErrorString(e));
  // D = rdm2 / 2 back-transformed: the half goes into the first U^T; three
  // transforms leave T[y][d][c][b] in ta, the fourth is dE/d(dc|ba)
  const double *Ut = ws + (size_t)W_UT * n2, *Uth = ws + (size_t)W_UTH * n2;
  if (deri || dkappa) {
    QTRANS("hci_rotate_backward", rdm2, Uth, ta, &status->timeout, &status->nonfinite);
    QTRANS("hci_rotate_backward", ta, Ut, tb, &status->timeout, &status->nonfinite);
    QTRANS("hci_rotate_backward", tb, Ut, ta, &status->timeout, &status->nonfinite);
  }
  if (dkappa) {
    const size_t sm = (size_t)NT_CH * (2 * n + 1) * 8;
    if (n2 <= 2048) {
      HCI_LAUNCH(k_gemm_nt_part<8>, nparts, 256, sm, st)(n, rows, eri, ta, part);
    } else {
      cudaFuncSetAttribute(k_gemm_nt_part<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, NT_CH * 129 * 8);
      HCI_LAUNCH(k_gemm_nt_part<16>, nparts, 256, sm, st)(n, rows, eri, ta, part);
    }
    HCI_LAUNCH(k_sum_parts, (unsigned)((n2 + 31) / 32), 256, 0, st)(n, nparts, part, 4.0, ws + (size_t)W_GU * n2);
    e = launch_chain(st, n, k_exp_adjoint, A, dkappa);
    if (e != cudaSuccess) return hci_fail(nullptr, HCI_ERR_CUDA, "hci_rotate_backward: %s", cudaGetErrorString(e));
  }
  if (deri) QTRANS("hci_rotate_backward", ta, Ut, deri, &status->timeout, &status->nonfinite);
  return chain_status("hci_rotate_backward", st, status);
}

extern "C" hci_status hci_qtrans(int norb, const double* in, const double* M, double* out, int check,
                                 void* stream) {
  const int n = norb;
  if (n < 1 || n > HCI_MAXORB) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_qtrans: norb=%d outside [1,64]", n);
  if (!in || !M || !out) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_qtrans: null pointer");
  cudaStream_t st = (cudaStream_t)stream;
  QTRANS("hci_qtrans", in, M, out, nullptr, nullptr);
  if (check && qtrans_tc_check(st) != HCI_OK)
    return hci_fail(nullptr, HCI_ERR_CUDA, "hci_qtrans: a quarter transform gave up waiting for its tensor-core products");
  return HCI_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free rotation.
//
// Some callers cannot allocate device memory at the time they need the
// rotation: code running inside another framework's memory pool that forbids
// foreign allocations, or a host thread that must not perform a
// cudaMalloc/cudaFree (each may synchronise the device).  For them
// hci_rotate_noalloc computes exactly what hci_rotate computes, with its
// scratch (the n^4 intermediate of the quarter transforms and the work
// matrices of exp(kappa)) in the file-scope device array below instead of
// stream-ordered allocations.  The array is part of this library's module:
// every GPU that loads the library holds it until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr int NOALLOC_MAXORB = 32;
constexpr size_t NOALLOC_T4 = (size_t)NOALLOC_MAXORB * NOALLOC_MAXORB * NOALLOC_MAXORB * NOALLOC_MAXORB;
constexpr size_t NOALLOC_M = (size_t)NOALLOC_MAXORB * NOALLOC_MAXORB;
constexpr size_t NOALLOC_DOUBLES = NOALLOC_T4 + W_FWD_COUNT * NOALLOC_M + 32;   // 8.08 MiB

static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_DOUBLES];

constexpr int NOALLOC_MAXDEV = 64;
struct NoallocSlot {
  unsigned long long ctx_id = 0;   // context the address was looked up in (0: none)
  double* ptr = nullptr;
};
static NoallocSlot g_noalloc_slot[NOALLOC_MAXDEV];
static std::mutex g_noalloc_mu;

// Identity of the calling thread's current CUDA context (a driver-assigned id
// that is never reused), 0 when it cannot be read.  The driver entry points
// are fetched through the runtime, so the library does not link libcuda.
unsigned long long current_context_id() {
  typedef CUresult (*GetCurrent)(CUcontext*);
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    void* a = nullptr;
    void* b = nullptr;
    cudaDriverEntryPointQueryResult qa, qb;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa) == cudaSuccess &&
        qa == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrent>(a);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) == cudaSuccess &&
        qb == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetId>(b);
    cudaGetLastError();
    looked_up = true;
  }
  if (!get_current || !get_id) return 0;
  CUcontext c = nullptr;
  unsigned long long id = 0;
  if (get_current(&c) != CUDA_SUCCESS || !c) return 0;
  if (get_id(c, &id) != CUDA_SUCCESS) return 0;
  return id;
}

// Device address of the scratch array in the current context.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// with cudaGetSymbolAddress (with the device current) once per device and
// context: the cached address is used again only while the same context is
// current, so a device reset or another context gets its own look-up.
hci_status noalloc_scratch(double** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return hci_fail(nullptr, HCI_ERR_CUDA, "hci_rotate_noalloc: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= NOALLOC_MAXDEV)
    return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate_noalloc: device %d outside [0,%d)", dev, NOALLOC_MAXDEV);
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  NoallocSlot& slot = g_noalloc_slot[dev];
  unsigned long long id = current_context_id();
  if (!slot.ptr || id == 0 || slot.ctx_id != id) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return hci_fail(nullptr, HCI_ERR_CUDA, "hci_rotate_noalloc: cudaGetSymbolAddress failed: %s",
                      cudaGetErrorString(e));
    if (id == 0) id = current_context_id();   // the look-up made the primary context current
    slot.ptr = reinterpret_cast<double*>(p);
    slot.ctx_id = id;
  }
  *out = slot.ptr;
  return HCI_OK;
}

}  // namespace

extern "C" hci_status hci_rotate_noalloc(int norb, const double* kappa, const double* h, const double* eri, double* U,
                                         double* h_out, double* eri_out, void* stream) {
  const int n = norb;
  if (n < 1 || n > NOALLOC_MAXORB)
    return hci_fail(nullptr, HCI_ERR_INVALID,
                    "hci_rotate_noalloc: norb=%d outside [1,%d] (the static scratch holds one %d^4 intermediate)", n,
                    NOALLOC_MAXORB, NOALLOC_MAXORB);
  if (!kappa || !h || !eri || !U || !h_out || !eri_out)
    return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rotate_noalloc: null pointer");
  double* base = nullptr;
  hci_status s = noalloc_scratch(&base);
  if (s != HCI_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  // every scratch element read below is written first in the same call, so
  // nothing has to be cleared; calls that overlap on the GPU share the array
  // and race
  return rotate_core("hci_rotate_noalloc", st, n, kappa, h, eri, U, h_out, eri_out, base + NOALLOC_T4, base);
}
