// FP64 Davidson for the lowest eigenpair on a fixed determinant space:
// the minimum of the energy functional Eq. (variational) with the
// normalisation multiplier (Sec. II.A: after each enlargement of V the new
// ground state is found with Davidson's method).  Vector operations, the
// subspace eigenproblem (one block) and the phase convention all run on the
// GPU; the host reads one report (Ritz value, residual norm, why a chain ended)
// per DAV_AHEAD iterations, or per iteration where products cannot be queued
// ahead (locked roots, a spin parity, one-orientation and direct graphs).
#include <cmath>

#include "hci_internal.cuh"

namespace {

constexpr int MAXSUB = 24;          // subspace size before restart (<= 32)
constexpr int DAV_KEEP = 4;         // Ritz vectors kept for the next, grown space
constexpr int LDG = 32;             // leading dimension of the subspace matrix
constexpr int DBLOCK = 256;
// Iterations queued before the host waits for their reports.  A wait leaves
// the GPU idle for about 35 us (the copy back, the host, the next launches),
// as long as an iteration's own kernels on a small space; the kernels queued
// behind the converged one return at once (about 14 us per iteration).
constexpr int DAV_AHEAD = 4;

// what the host reads of an iteration
struct DavReport {
  double theta;           // Ritz value
  double ols[3];          // |r|^2, x . M^-1 r, x . M^-1 x (Olsen correction)
  int stall;              // a correction fell inside the subspace
  int stop;               // chained iterations: nothing queued after this is to run
  int it, k;              // Ritz steps taken, the last one's subspace size
};

struct DavDev {
  double G[LDG * LDG];
  float X[LDG * LDG];        // FP32 eigenvectors of the last subspace matrix (kx x kx), start of the next
  double Y[DAV_KEEP][LDG];   // the lowest eigenvectors of the subspace matrix, orthonormal (k_lowest<DAV_KEEP>)
  double y[LDG];
  double dots[LDG];
  DavReport rep;
  double nrm2;
  double eps, unit;           // k_pass: the Olsen step, 1 / norm of the correction (0: it lies in the subspace)
  int kx, ky;             // sizes of X and of y (0: none)
  unsigned int ticket;    // blocks of the running reduction that have finished
};

// ---------------------------------------------------------------------------
// Grid-wide sums of NA accumulators per thread.
//
// The vector passes below are bound by FP64 issue long before memory (a
// warp's FP64 instruction takes 64 cycles of its sub-partition): a plain
// shuffle tree costs 5 additions per accumulator and warp, more than the
// products themselves at a few elements per thread.  warp_sums halves the
// values held per lane at every step instead (27 additions for 24
// accumulators, not 120), and the reducing passes run one or two blocks per
// SM, so that each warp reduces once for several elements.
// ---------------------------------------------------------------------------
template <int H, int OFF>
__device__ __forceinline__ void warp_sums(double* a, int lane) {
  if constexpr (OFF > 0) {
    if constexpr (H % 2 == 0) {
      const bool up = lane & OFF;
#pragma unroll
      for (int q = 0; q < H / 2; ++q) {
        const double keep = up ? a[q + H / 2] : a[q], give = up ? a[q] : a[q + H / 2];
        a[q] = keep + __shfl_xor_sync(0xffffffffu, give, OFF);
      }
      warp_sums<H / 2, OFF / 2>(a, lane);
    } else {
#pragma unroll
      for (int q = 0; q < H; ++q) a[q] += __shfl_xor_sync(0xffffffffu, a[q], OFF);
      warp_sums<H, OFF / 2>(a, lane);
    }
  }
}
// lanes that hold sums after warp_sums: first index of a lane's values
// (`left` values, the same in the lanes that differ only in `spare` bits)
template <int H, int OFF>
__device__ __forceinline__ int sums_base(int lane, int& left, int& spare) {
  left = H;
  if constexpr (OFF > 0) {
    if constexpr (H % 2 == 0) {
      const int b = (lane & OFF) ? H / 2 : 0;
      return b + sums_base<H / 2, OFF / 2>(lane, left, spare);
    } else {
      spare = 2 * OFF - 1;
    }
  }
  return 0;
}

// Sums of acc[0 .. NA) over the grid, taken by the last block to finish (a
// ticket counter) from the blocks' partial sums, in a fixed order, so that
// the result does not depend on the order in which blocks finish.  True in
// that block, whose threads t < NA then hold sum t in *total.  Blocks of the
// grid: (x, y), partial sums at [x][j0 .. j0 + NA) for the y-th group.
template <int NA>
__device__ __forceinline__ bool grid_sums(double* acc, int j0, int ncol, double* partial, unsigned int* ticket,
                                          double* total) {
  __shared__ double red[DBLOCK / 32][LDG];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  warp_sums<NA, 16>(acc, lane);
  int left = 0, spare = 0;
  const int base = sums_base<NA, 16>(lane, left, spare);
  if ((lane & spare) == 0)
    for (int q = 0; q < left; ++q) red[wid][base + q] = acc[q];
  __syncthreads();
  if (threadIdx.x < NA && j0 + (int)threadIdx.x < ncol) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < DBLOCK / 32; ++w) s += red[w][threadIdx.x];
    partial[(int64_t)blockIdx.x * LDG + j0 + threadIdx.x] = s;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1u;
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  // the columns rounded up to a power of two share the block's threads, so
  // that a thread adds few partial sums (304 blocks: 2 for one column, 38
  // for 24), four loads in flight
  int cp = 1;
  while (cp < ncol) cp <<= 1;
  const int col = threadIdx.x & (cp - 1);
  double s = 0.0;
  if (col < ncol) {
    const double* pc = partial + col;
#pragma unroll 4
    for (int b = threadIdx.x / cp; b < (int)gridDim.x; b += DBLOCK / cp) s += __ldcg(pc + (int64_t)b * LDG);
  }
  for (int o = cp; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane < cp) red[wid][lane] = s;
  __syncthreads();
  s = 0.0;
  if ((int)threadIdx.x < ncol)
#pragma unroll
    for (int w = 0; w < DBLOCK / 32; ++w) s += red[w][threadIdx.x];
  *total = s;
  if (threadIdx.x == 0) *ticket = 0u;
  return true;
}

// out[j] = V_j . w (j < k <= 32), vectors in groups of DOTS_GROUP (blockIdx.y
// = group).  With gcol >= 0 out[j] is also stored as G[j][gcol] = G[gcol][j],
// j <= gcol.
constexpr int DOTS_GROUP = 8;

__global__ void __launch_bounds__(DBLOCK) k_dots(const double* __restrict__ V, int64_t ld, int k,
                                                 const double* __restrict__ w, int64_t n, double* __restrict__ partial,
                                                 double* __restrict__ out, DavDev* __restrict__ gd, int gcol) {
  const int j0 = blockIdx.y * DOTS_GROUP;
  const int kg = k - j0 < DOTS_GROUP ? k - j0 : DOTS_GROUP;
  const double* Vg = V + (int64_t)j0 * ld;
  double acc[DOTS_GROUP];
#pragma unroll
  for (int j = 0; j < DOTS_GROUP; ++j) acc[j] = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double wv = w[i];
#pragma unroll
    for (int j = 0; j < DOTS_GROUP; ++j)
      if (j < kg) acc[j] = fma(Vg[(int64_t)j * ld + i], wv, acc[j]);
  }
  double s;
  if (!grid_sums<DOTS_GROUP>(acc, j0, k, partial, &gd->ticket, &s)) return;
  const int j = threadIdx.x;
  if (j < k) {
    out[j] = s;
    if (gcol >= 0 && j <= gcol) {
      gd->G[j * LDG + gcol] = s;
      gd->G[gcol * LDG + j] = s;
    }
  }
}

// The vector passes of one iteration between the Ritz step and the next
// product, each one launch over the k subspace vectors (NA >= the number of
// sums):
//   OLSEN: t <- t - eps u (the Olsen correction, see k_ritz), dots_j = V_j . t
//   ORTH:  t <- t - sum_j dots_j V_j, dots_j = V_j . t of the result (the
//          second Gram-Schmidt pass's products, from the values of V_j that
//          the first one's subtraction has in registers), and with |t|^2 of
//          it |t|^2 - sum_j dots_j^2, the norm^2 that the second subtraction
//          leaves (dots_j is rounding beside t, the V_j are orthonormal):
//          unit = 1 / the norm.  A correction of norm^2 at most 1e-26 lies in
//          the subspace: unit = 0
//   UNIT:  V_k <- (t - sum_j dots_j V_j) unit, no sums
//   GCOL:  after W_k = H V_k: G[j][k] = G[k][j] = V_j . W_k, j <= k, and with
//          unit = 0 stall = stop = 1.
// Bound by FP64 issue (2 k + 1 operations per element) at 1e5 elements, by
// the k vectors' bytes beyond L2, and by their launch and reduction (6.3 us)
// on small spaces.  (12e,12o) space, 1.4e5 elements, k from 17 to 24: 15.1,
// 20.7, 9.8 and 15.1 us; with |V_k|^2 summed in a pass of its own and the
// scaling left to GCOL 17.0, 22.9, 11.5 and 22.8.
enum { PASS_OLSEN = 0, PASS_ORTH = 1, PASS_UNIT = 2, PASS_GCOL = 3 };

template <int OP, int NA>
__global__ void __launch_bounds__(DBLOCK, OP == PASS_UNIT ? 2 : 1) k_pass(double* __restrict__ V, const double* __restrict__ W, int64_t ld,
                                                    int k, int64_t n, double* __restrict__ t,
                                                    const double* __restrict__ u, DavDev* __restrict__ d,
                                                    double* __restrict__ partial) {
  __shared__ double cs[LDG];
  if (d->rep.stop) return;
  if (threadIdx.x < LDG) cs[threadIdx.x] = d->dots[threadIdx.x];
  __syncthreads();
  const double eps = OP == PASS_OLSEN ? d->eps : 0.0, f = d->unit;
  const int nv = OP == PASS_GCOL ? k + 1 : k;            // vectors read
  const int ns = OP == PASS_ORTH ? NA : nv;              // sums; ORTH (k < NA): the last is |t|^2
  constexpr int NS = OP == PASS_UNIT ? 1 : NA;
  double acc[NS];
#pragma unroll
  for (int j = 0; j < NS; ++j) acc[j] = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double v[NA];
#pragma unroll
    for (int j = 0; j < NA; ++j) v[j] = j < nv && (OP != PASS_ORTH || j < NA - 1) ? V[(int64_t)j * ld + i] : 0.0;
    double w;
    if (OP == PASS_OLSEN) {
      w = fma(-eps, u[i], t[i]);
      t[i] = w;
    } else if (OP == PASS_GCOL) {
      w = W[(int64_t)k * ld + i];
    } else {
      w = t[i];
#pragma unroll
      for (int j = 0; j < NA; ++j)
        if (j < k) w = fma(-cs[j], v[j], w);
      if (OP == PASS_ORTH) t[i] = w;
      else V[(int64_t)k * ld + i] = f != 0.0 ? w * f : 0.0;
    }
    if (OP != PASS_UNIT) {
#pragma unroll
      for (int j = 0; j < NS; ++j)
        if (OP == PASS_ORTH && j == NA - 1) acc[j] = fma(w, w, acc[j]);
        else if (j < nv) acc[j] = fma(v[j], w, acc[j]);
    }
  }
  if (OP == PASS_UNIT) return;
  double s;
  if (!grid_sums<NS>(acc, 0, ns, partial, &d->ticket, &s)) return;
  const int j = threadIdx.x;
  if (OP == PASS_GCOL) {
    if (j <= k) {
      d->G[j * LDG + k] = s;
      d->G[k * LDG + j] = s;
    }
    if (j == 0 && f == 0.0) d->rep.stall = d->rep.stop = 1;
    return;
  }
  if (j < k) d->dots[j] = s;
  if (OP == PASS_ORTH && j < 32) {
    double q = j < k ? -s * s : j == NA - 1 ? s : 0.0;
    for (int o = 16; o; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    // here and not in every thread of UNIT: a warp's FP64 root and division
    // cost as much as its share of the pass
    if (j == 0) d->unit = q > 1e-26 ? 1.0 / sqrt(q) : 0.0;
  }
}

// ---------------------------------------------------------------------------
// Lowest eigenpair(s) of the k x k subspace matrix G, one block.
//
// FP64 is the scarce unit: a warp's FP64 instruction takes 64 cycles of its
// sub-partition whatever its active lanes, so a full FP64 Jacobi (about 70
// of them per round, 23 rounds per sweep) is bound by that pipe.  Only the
// lowest pair is needed, so FP64 is kept for the residual and everything
// else runs in FP32 on G shifted by G_00 (which takes the large common part
// of the energies away).
//
// NV = 1 (lowest_newton), from the last lowest vector y: y is turned by the
// 2 x 2 problem of y and the newly added direction, then
//   rho = y.Gy / y.y,  r = Gy - rho y                       (FP64)
//   y <- y - B^-1 r,   B = G - rho + s y y^T                (FP32 inverse)
// until the next residual is predicted below 2e-16 of the spectrum's
// spread.  B lifts y by the spread s, so it is positive definite exactly
// when no other eigenvalue lies below rho: its pivots (Gauss-Jordan, one
// row per lane) decide whether the pair found is the lowest one.  A pivot
// below 1e-5 s (a neighbour too close for FP32), or no convergence, and
// every NV > 1 call, takes the second way.
//
// Second way: Jacobi in FP32 (round-robin schedule; thread (s, t) owns the
// 2 x 2 block of pairs s and t, reads it and both pairs' rotations from one
// copy of A and writes the rotated block to the other, so that a round takes
// one barrier), started from the last eigenvectors when the matrix is the
// last one or that bordered by one row and column, then the same refinement
// of the NV lowest vectors, one warp each, with the FP32 eigenvectors x_m:
//   y <- y - sum_{m != lowest} x_m (x_m . r) / (e_m - rho).
// Neighbours closer than 2e-5 of the spread, or no convergence: FP64 Jacobi.
//
// (12e,12o) space, k up to 24, about 840 calls: 219 us per call with an
// FP64 Jacobi started from the last eigenvectors, 45 us by the second way,
// 12.4 us by the first.  Against a Jacobi in quad precision, 2700 calls of
// Davidson runs on 240 random matrices (gaps from 0.02 to 1 of a spectrum of
// 6, offsets of -40 and -8000): vector error at most 5e-16 and residual 1e-15 (the FP64 Jacobi 2e-14
// and 4e-14, with the offset 2e-12 and 3e-12), since only the residual is
// rounded in FP64 and it is formed on the shifted matrix.
constexpr int LW_X = 160;             // threads below: 2 x 2 blocks of A; from here on: rows of X
constexpr int LW_T = 320;
constexpr float LW_SKIP = 1e-6f;      // rotations below this angle are skipped
constexpr float LW_GAP = 2e-5f;       // least gap (of the spread) that FP32 resolves

// pair t of round r, m players (index m - 1 stays, the others rotate)
__device__ __forceinline__ void rr_pair(int r, int t, int m, int& p, int& q) {
  int a = r, b = m - 1;
  if (t > 0) {
    a = r + t;
    if (a >= m - 1) a -= m - 1;
    b = r - t;
    if (b < 0) b += m - 1;
  }
  p = a < b ? a : b;
  q = a < b ? b : a;
}

__device__ __forceinline__ bool rot32(const float (*a)[LDG + 1], int p, int q, float& c, float& s) {
  const float apq = a[p][q], dd = a[q][q] - a[p][p];
  c = 1.0f;
  s = 0.0f;
  if (fabsf(apq) <= LW_SKIP * fabsf(dd)) return false;
  const float e2 = 2.0f * apq, h = dd * dd + e2 * e2;
  const float t = __fdividef(copysignf(e2, dd * e2), fabsf(dd) + h * rsqrtf(h));
  c = rsqrtf(1.0f + t * t);
  s = t * c;
  return true;
}

// Full FP64 Jacobi of A (overwritten; diagonal = eigenvalues), Q = vectors
__device__ void jacobi_fp64(int k, double (*A)[LDG + 1], double (*Q)[LDG + 1], double* rc, double* rs, int* rp,
                            int* rq) {
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int m = (k + 1) & ~1;          // even number of players (index k is a dummy when k is odd)
  const int npairs = m / 2;
  for (int sweep = 0; sweep < 50 && k > 1; ++sweep) {
    int rotated = 0;
    for (int r = 0; r < m - 1; ++r) {
      int active = 0;
      if (threadIdx.x < npairs) {
        const int t = threadIdx.x;
        int p, q;
        rr_pair(r, t, m, p, q);
        double c = 1.0, sn = 0.0;
        if (q < k) {
          const double apq = A[p][q], app = A[p][p], aqq = A[q][q];
          const double g = 100.0 * fabs(apq);
          // an element too small to change either diagonal partner (even
          // scaled by 100) is zeroed
          if (!((fabs(app) + g == fabs(app) && fabs(aqq) + g == fabs(aqq)) || fabs(apq) < 1e-300)) {
            // tan of the rotation angle without the division for tau (the
            // entries are Rayleigh quotients of normalised vectors, far
            // from overflow)
            const double dd = aqq - app, e2 = 2.0 * apq;
            const double tt = copysign(1.0, dd) * e2 / (fabs(dd) + sqrt(dd * dd + e2 * e2));
            c = rsqrt(1.0 + tt * tt);
            sn = tt * c;
            active = 1;
          }
        }
        rp[t] = p; rq[t] = q; rc[t] = c; rs[t] = active ? sn : 0.0;
        if (!active && q < k) { A[p][q] = 0.0; A[q][p] = 0.0; }
      }
      rotated |= __syncthreads_or(active);
      // columns: A <- A J, Q <- Q J (lane = row)
      if (l < k) {
        for (int t = w; t < npairs; t += nw) {
          const double s2 = rs[t];
          if (s2 == 0.0) continue;
          const int p = rp[t], q = rq[t];
          const double c2 = rc[t];
          const double alp = A[l][p], alq = A[l][q];
          A[l][p] = c2 * alp - s2 * alq;
          A[l][q] = s2 * alp + c2 * alq;
          const double vlp = Q[l][p], vlq = Q[l][q];
          Q[l][p] = c2 * vlp - s2 * vlq;
          Q[l][q] = s2 * vlp + c2 * vlq;
        }
      }
      __syncthreads();
      // rows: A <- J^T A (lane = column)
      if (l < k) {
        for (int t = w; t < npairs; t += nw) {
          const double s2 = rs[t];
          if (s2 == 0.0) continue;
          const int p = rp[t], q = rq[t];
          const double c2 = rc[t];
          const double apl = A[p][l], aql = A[q][l];
          A[p][l] = c2 * apl - s2 * aql;
          A[q][l] = s2 * apl + c2 * aql;
        }
      }
      __syncthreads();
      if (threadIdx.x < npairs && rs[threadIdx.x] != 0.0) {
        A[rp[threadIdx.x]][rq[threadIdx.x]] = 0.0;
        A[rq[threadIdx.x]][rp[threadIdx.x]] = 0.0;
      }
      __syncthreads();
    }
    if (!rotated) break;
  }
}

// The first way (see above) for k <= K: G64 / G32 the shifted matrix, zero
// beyond k; on success y0 = the normalised lowest vector, *rho0 its shifted
// eigenvalue.  All threads of the block call it; warp 0 decides.
template <int K>
__device__ bool lowest_newton(int k, const double (*G64)[LDG + 1], const float (*G32)[LDG + 1], const double* yprev,
                              int ky, double (*P)[LDG + 1], double* y0, double* rho0) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr unsigned ALL = 0xffffffffu;
  double y = 0.0;
  if (w == 0) {
    if (ky == k - 1) {
      y = lane < ky ? yprev[lane] : 0.0;
      // 2 x 2 problem of y and e_{k-1}
      double g = 0.0;
      if (lane < ky) g = y * G64[lane][k - 1];
      float gf = (float)g, hf = 0.0f;
      for (int j = 0; j < ky; ++j) hf = fmaf(G32[lane][j], __shfl_sync(ALL, (float)y, j), hf);
      hf *= (float)y;
      for (int b = 16; b; b >>= 1) {
        gf += __shfl_xor_sync(ALL, gf, b);
        hf += __shfl_xor_sync(ALL, hf, b);
      }
      const float dd = G32[k - 1][k - 1] - hf, e2 = 2.0f * gf;
      // lowest vector of [[hf, gf], [gf, hf + dd]]: (1, t) with t below
      const float q = sqrtf(fmaf(dd, dd, e2 * e2));
      if (dd >= 0.0f) {
        const float t = e2 == 0.0f ? 0.0f : -e2 / (dd + q);
        if (lane == k - 1) y = t;
      } else {
        const float t = e2 == 0.0f ? 0.0f : -e2 / (q - dd);
        y = lane == k - 1 ? 1.0 : y * (double)t;
      }
    } else {
      // no vector of the last matrix: its lowest diagonal element
      const float dl = lane < k ? G32[lane][lane] : INFINITY;
      float mn = dl;
      for (int b = 16; b; b >>= 1) mn = fminf(mn, __shfl_xor_sync(ALL, mn, b));
      const int at = __ffs(__ballot_sync(ALL, dl == mn)) - 1;
      y = lane == at ? 1.0 : 0.0;
    }
    y0[lane] = y;
  }
  float inv[K];
  float prev = 0.0f, scale = 0.0f;
  bool fresh = false;
  int verdict = 0;                      // 1: converged, 2: give up
  for (int it = 0; it < 10; ++it) {
    __syncthreads();
    if (w < 4) {
      double g = 0.0;
      for (int j = w; j < k; j += 4) g = fma(G64[lane][j], y0[j], g);
      P[w][lane] = g;
    }
    __syncthreads();
    if (w == 0) {
      const double g = (P[0][lane] + P[1][lane]) + (P[2][lane] + P[3][lane]);
      // y.y in the lower half of the warp, y.g in the upper
      const double a = y * y, c = y * g;
      const bool up = lane & 16;
      double t = (up ? c : a) + __shfl_xor_sync(ALL, up ? a : c, 16);
      for (int b = 8; b; b >>= 1) t += __shfl_xor_sync(ALL, t, b);
      const double s0 = __shfl_sync(ALL, t, 0), s1 = __shfl_sync(ALL, t, 16);
      const double rho = s1 / s0;
      const float rf = (float)(g - rho * y);
      if (!fresh) {
        // B^-1 at this y (row per lane)
        const float yf = (float)y, dg = (float)(G64[lane][lane] - rho);
        float sc = lane < k ? fabsf(dg) : 0.0f;
        for (int b = 16; b; b >>= 1) sc = fmaxf(sc, __shfl_xor_sync(ALL, sc, b));
        scale = sc;
        const float sy = sc / (float)s0 * yf;
#pragma unroll
        for (int m = 0; m < K; ++m) {
          const float ym = __shfl_sync(ALL, yf, m);
          inv[m] = fmaf(sy, ym, m == lane ? dg : G32[lane][m]);
          if (m >= k) inv[m] = m == lane ? sc : 0.0f;   // padding: a multiple of the identity
        }
        bool pos = sc > 0.0f;
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const float piv = __shfl_sync(ALL, inv[j], j);
          pos = pos && piv > 1e-5f * sc;
          const float ip = 1.0f / piv;
          const float f = lane == j ? 0.0f : inv[j];
#pragma unroll
          for (int m = 0; m < K; ++m)
            if (m != j) {
              const float rj = __shfl_sync(ALL, inv[m], j) * ip;
              inv[m] = lane == j ? rj : fmaf(-f, rj, inv[m]);
            }
          inv[j] = lane == j ? ip : -f * ip;
        }
        if (!pos) verdict = 2;
        fresh = true;
      }
      float de = 0.0f;
#pragma unroll
      for (int m = 0; m < K; ++m) de = fmaf(inv[m], __shfl_sync(ALL, rf, m), de);
      float rr = rf * rf, d2 = lane < k ? de * de : 0.0f;
      for (int b = 16; b; b >>= 1) {
        rr += __shfl_xor_sync(ALL, rr, b);
        d2 += __shfl_xor_sync(ALL, d2, b);
      }
      if (lane < k) y -= (double)de;
      const float s0f = (float)s0, rn = sqrtf(rr / s0f);
      d2 /= s0f;
      if (verdict == 0) {
        const float ratio = it > 0 ? fminf(rn / prev, 1.0f) : 1.0f;
        if (rn * ratio <= 2e-16f * scale && d2 < 1e-6f) verdict = 1;
        else if (it >= 3 && rn > 0.5f * prev) verdict = rn <= 1e-14f * scale ? 1 : 2;
        else if (!(d2 < 1.0f)) verdict = 2;
      }
      if (d2 > 1e-4f) fresh = false;    // y moved by more than 1e-2: invert again
      prev = rn;
      if (verdict == 1) {
        double q = y * y;
        for (int b = 16; b; b >>= 1) q += __shfl_xor_sync(ALL, q, b);
        y *= 1.0 / sqrt(q);
        if (lane == 0) *rho0 = rho;
      }
      y0[lane] = y;
    }
    const int v = __syncthreads_or(w == 0 ? verdict : 0);
    if (v) return __syncthreads_or(w == 0 && verdict == 1) != 0;
  }
  return false;
}

// NV = 1: theta, y = the lowest eigenpair.  NV > 1: also Y[0 .. min(NV, k))
// = the lowest eigenvectors, ascending, orthonormal.
template <int NV>
__global__ void __launch_bounds__(LW_T) k_lowest(DavDev* d, int k) {
  __shared__ double G[LDG][LDG + 1];
  __shared__ float A[2][LDG][LDG + 1];
  __shared__ float X[LDG][LDG + 1];
  __shared__ float ev[LDG];
  __shared__ int order[LDG];
  __shared__ double Ys[NV][LDG], th[NV];
  __shared__ float Rs[NV][LDG], Cs[NV][LDG];
  __shared__ double A64[LDG][LDG + 1], Q64[LDG][LDG + 1];
  __shared__ double rc[LDG / 2], rs[LDG / 2];
  __shared__ int rp[LDG / 2], rq[LDG / 2];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (NV == 1 && d->rep.stop) return;
  const double sh = d->G[0];
  const int kx = (d->kx == k || d->kx == k - 1) ? d->kx : 0, ky = d->ky;
  for (int e = tid; e < LDG * LDG; e += LW_T) {
    const int i = e / LDG, j = e % LDG;
    const double g = (i < k && j < k) ? d->G[e] - (i == j ? sh : 0.0) : 0.0;
    G[i][j] = g;
    A[0][i][j] = (float)g;
    A[1][i][j] = 0.0f;
    X[i][j] = (i < kx && j < kx) ? d->X[e] : (i == j ? 1.0f : 0.0f);
  }
  if (tid < LDG) order[tid] = tid;
  __syncthreads();
  if (NV == 1) {
    bool ok;
    if (k == 1) {
      if (tid < LDG) Ys[0][tid] = tid == 0 ? 1.0 : 0.0;
      if (tid == 0) th[0] = 0.0;
      __syncthreads();
      ok = G[0][0] == 0.0;               // false for a non-finite matrix
    } else if (k <= 8) {
      ok = lowest_newton<8>(k, G, A[0], d->y, ky, Q64, Ys[0], th);
    } else if (k <= 16) {
      ok = lowest_newton<16>(k, G, A[0], d->y, ky, Q64, Ys[0], th);
    } else {
      ok = lowest_newton<MAXSUB>(k, G, A[0], d->y, ky, Q64, Ys[0], th);
    }
    if (ok) {
      if (w == 0) d->y[lane] = Ys[0][lane];
      if (tid == 0) {
        d->rep.theta = th[0] + sh;
        d->ky = k;
      }
      return;
    }
  }
  if (kx > 0) {
    for (int e = tid; e < k * k; e += LW_T) {
      const int i = e / k, j = e % k;
      float t = 0.0f;
      for (int m = 0; m < k; ++m) t = fmaf(A[0][i][m], X[m][j], t);
      A[1][i][j] = t;
    }
    __syncthreads();
    for (int e = tid; e < k * k; e += LW_T) {
      const int i = e / k, j = e % k;
      float t = 0.0f;
      for (int m = 0; m < k; ++m) t = fmaf(X[m][i], A[1][m][j], t);
      A[0][i][j] = t;
    }
    __syncthreads();
  }
  int cur = 0;
  if (k > 1) {
    const int m = (k + 1) & ~1, np = m / 2;
    int idle = 0, r = 0;
    for (int round = 0; round < 40 * (m - 1); ++round) {
      const float(*a)[LDG + 1] = A[cur];
      float(*b)[LDG + 1] = A[cur ^ 1];
      bool act = false;
      if (tid < np * np) {
        const int si = tid / np, ti = tid - si * np;
        int p1, q1, p2, q2;
        rr_pair(r, si, m, p1, q1);
        rr_pair(r, ti, m, p2, q2);
        float c1, s1, c2, s2;
        act = rot32(a, p1, q1, c1, s1);
        rot32(a, p2, q2, c2, s2);
        const float xpp = a[p1][p2], xpq = a[p1][q2], xqp = a[q1][p2], xqq = a[q1][q2];
        const float ypp = c2 * xpp - s2 * xpq, ypq = s2 * xpp + c2 * xpq;
        const float yqp = c2 * xqp - s2 * xqq, yqq = s2 * xqp + c2 * xqq;
        b[p1][p2] = c1 * ypp - s1 * yqp;
        b[p1][q2] = c1 * ypq - s1 * yqq;
        b[q1][p2] = s1 * ypp + c1 * yqp;
        b[q1][q2] = s1 * ypq + c1 * yqq;
      } else if (tid >= LW_X) {
        for (int it = tid - LW_X; it < np * k; it += LW_T - LW_X) {
          const int ti = it / k, l = it - ti * k;
          int p, q;
          rr_pair(r, ti, m, p, q);
          float c, s;
          if (rot32(a, p, q, c, s)) {
            const float u = X[l][p], v = X[l][q];
            X[l][p] = c * u - s * v;
            X[l][q] = s * u + c * v;
          }
        }
      }
      const int any = __syncthreads_or(act);
      cur ^= 1;
      idle = any ? 0 : idle + 1;
      if (idle >= m - 1) break;
      if (++r == m - 1) r = 0;
    }
  }
  if (w == 0) {
    const float e = lane < k ? A[cur][lane][lane] : 0.0f;
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const float o = __shfl_sync(0xffffffffu, e, j);
      rank += (o < e || (o == e && j < lane)) ? 1 : 0;
    }
    if (lane < k) {
      ev[lane] = e;
      order[rank] = lane;
    }
  }
  __syncthreads();
  const int kk = k < NV ? k : NV;
  const float spread = ev[order[k - 1]] - ev[order[0]];
  bool good = true;
  for (int t = 0; t < kk && t + 1 < k; ++t) good = good && ev[order[t + 1]] - ev[order[t]] > LW_GAP * spread;
  if (good && w < kk) {
    // warp w refines the w-th lowest vector; lane = row
    const int o = order[w];
    double y = lane < k ? (double)X[lane][o] : 0.0, rho = 0.0;
    float prev = 0.0f;
    good = false;
    for (int it = 0; it < 12; ++it) {
      Ys[w][lane] = y;
      __syncwarp();
      double g = 0.0;
      for (int j = 0; j < k; ++j) g = fma(G[lane][j], Ys[w][j], g);
      double s0 = y * y, s1 = y * g;
      for (int b = 16; b; b >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, b);
        s1 += __shfl_xor_sync(0xffffffffu, s1, b);
      }
      rho = s1 / s0;
      const float rf = (float)(g - rho * y);
      float rr = rf * rf;
      for (int b = 16; b; b >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, b);
      const float rn = sqrtf(rr);
      Rs[w][lane] = rf;
      __syncwarp();
      float am = 0.0f;
      if (lane < k && lane != o) {
        for (int i = 0; i < k; ++i) am = fmaf(X[i][lane], Rs[w][i], am);
        am = -am / (ev[lane] - (float)rho);
      }
      Cs[w][lane] = am;
      __syncwarp();
      float de = 0.0f;
      for (int j = 0; j < k; ++j) de = fmaf(X[lane][j], Cs[w][j], de);
      if (lane < k) y += (double)de;
      const float ratio = it > 0 ? fminf(rn / prev, 1.0f) : 1.0f;
      if (rn * ratio <= 2e-16f * spread) { good = true; break; }
      if (it >= 3 && rn > 0.5f * prev) { good = rn <= 1e-14f * spread; break; }
      prev = rn;
    }
    double s0 = y * y;
    for (int b = 16; b; b >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, b);
    Ys[w][lane] = y * (1.0 / sqrt(s0));
    if (lane == 0) th[w] = rho + sh;
  }
  if (__syncthreads_and(good)) {
    if (NV > 1 && w == 0) {
      // orthogonal to about the refinement's accuracy: one Gram-Schmidt pass
      for (int t = 1; t < kk; ++t) {
        double y = Ys[t][lane];
        for (int u = 0; u < t; ++u) {
          double dt = Ys[u][lane] * y;
          for (int b = 16; b; b >>= 1) dt += __shfl_xor_sync(0xffffffffu, dt, b);
          y = fma(-dt, Ys[u][lane], y);
        }
        double s0 = y * y;
        for (int b = 16; b; b >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, b);
        Ys[t][lane] = y * (1.0 / sqrt(s0));
        __syncwarp();
      }
    }
  } else {
    for (int e = tid; e < LDG * LDG; e += LW_T) {
      A64[e / LDG][e % LDG] = G[e / LDG][e % LDG];
      Q64[e / LDG][e % LDG] = e / LDG == e % LDG ? 1.0 : 0.0;
    }
    __syncthreads();
    jacobi_fp64(k, A64, Q64, rc, rs, rp, rq);
    if (tid == 0) {
      bool used[LDG];
      for (int j = 0; j < k; ++j) used[j] = false;
      for (int t = 0; t < kk; ++t) {
        int b = -1;
        for (int j = 0; j < k; ++j)
          if (!used[j] && (b < 0 || A64[j][j] < A64[b][b])) b = j;
        used[b] = true;
        order[t] = b;
        th[t] = A64[b][b] + sh;
      }
    }
    __syncthreads();
    if (w < kk) Ys[w][lane] = lane < k ? Q64[lane][order[w]] : 0.0;
    for (int e = tid; e < LDG * LDG; e += LW_T) X[e / LDG][e % LDG] = (float)Q64[e / LDG][e % LDG];
  }
  __syncthreads();
  for (int e = tid; e < LDG * LDG; e += LW_T) d->X[e] = X[e / LDG][e % LDG];
  if (w == 0) {
    d->y[lane] = Ys[0][lane];
    if (NV > 1)
      for (int t = 0; t < kk; ++t) d->Y[t % DAV_KEEP][lane] = Ys[t % NV][lane];
  }
  if (tid == 0) {
    d->rep.theta = th[0];
    d->kx = d->ky = k;
  }
}

// x = V y, wy = W y, r = wy - theta x, t = M^-1 r and u = M^-1 x with M =
// theta - diag (guarded away from zero), and the sums r^2, x t and x u of
// the Olsen correction t - eps u, eps = (x M^-1 r) / (x M^-1 x), which is
// orthogonal to x to first order.  2 k + 16 FP64 operations per element (one
// division, not two) bound it at 1e5 elements, 16 k bytes beyond L2: 22.1 ->
// 15.4 us on the (12e,12o) space.
__global__ void __launch_bounds__(DBLOCK) k_ritz(const double* __restrict__ V, const double* __restrict__ W, int64_t ld,
                                                 int k, DavDev* __restrict__ d, const double* __restrict__ diag,
                                                 int64_t n, double* __restrict__ x, double* __restrict__ wy,
                                                 double* __restrict__ t, double* __restrict__ u,
                                                 double* __restrict__ partial, int chained, double tol) {
  __shared__ double ys[LDG];
  if (d->rep.stop) return;
  if (threadIdx.x < LDG) ys[threadIdx.x] = d->y[threadIdx.x];
  __syncthreads();
  const double theta = d->rep.theta;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double xv = 0.0, wv = 0.0;
    const double* v = V + i;
    const double* w = W + i;
    int j = 0;
    for (; j + 4 <= k; j += 4) {
      const double v0 = v[0], v1 = v[ld], v2 = v[2 * ld], v3 = v[3 * ld];
      const double w0 = w[0], w1 = w[ld], w2 = w[2 * ld], w3 = w[3 * ld];
      xv = fma(ys[j], v0, xv);
      wv = fma(ys[j], w0, wv);
      xv = fma(ys[j + 1], v1, xv);
      wv = fma(ys[j + 1], w1, wv);
      xv = fma(ys[j + 2], v2, xv);
      wv = fma(ys[j + 2], w2, wv);
      xv = fma(ys[j + 3], v3, xv);
      wv = fma(ys[j + 3], w3, wv);
      v += 4 * ld;
      w += 4 * ld;
    }
    for (; j < k; ++j, v += ld, w += ld) {
      xv = fma(ys[j], v[0], xv);
      wv = fma(ys[j], w[0], wv);
    }
    const double r = wv - theta * xv;
    double den = theta - diag[i];
    if (fabs(den) < 1e-8) den = den >= 0.0 ? 1e-8 : -1e-8;
    const double inv = 1.0 / den, tv = r * inv, uv = xv * inv;
    x[i] = xv;
    wy[i] = wv;
    t[i] = tv;
    u[i] = uv;
    acc[0] = fma(r, r, acc[0]);
    acc[1] = fma(xv, tv, acc[1]);
    acc[2] = fma(xv, uv, acc[2]);
  }
  double s;
  if (!grid_sums<4>(acc, 0, 3, partial, &d->ticket, &s)) return;
  if (threadIdx.x < 3) d->rep.ols[threadIdx.x] = s;
  if (threadIdx.x >= 32) return;
  const double num = __shfl_sync(0xffffffffu, s, 1), den = __shfl_sync(0xffffffffu, s, 2);
  if (threadIdx.x == 0) {
    d->eps = den != 0.0 ? num / den : 0.0;
    d->rep.it += 1;
    d->rep.k = k;
    // a residual that is not finite ends the chain too; a tolerance that is not
    // a number is never met, here as on the host
    if (chained && (sqrt(s) <= tol || !isfinite(s) || !isfinite(theta))) d->rep.stop = 1;
  }
}

// The kk <= DAV_KEEP lowest Ritz vectors of the current subspace (ascending Ritz value)
// and their H products: Qo[t] = sum_j Y[t][j] V[j], Wo[t] likewise from W.
__global__ void __launch_bounds__(DBLOCK) k_keep(const double* __restrict__ V, const double* __restrict__ W,
                                                 int64_t ld, int k, const DavDev* __restrict__ d, int kk, int64_t n,
                                                 double* __restrict__ Qo, double* __restrict__ Wo) {
  __shared__ double ys[DAV_KEEP][LDG];
  for (int e = threadIdx.x; e < kk * k; e += blockDim.x) ys[e / k][e % k] = d->Y[e / k][e % k];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double qv[DAV_KEEP], wv[DAV_KEEP];
#pragma unroll
    for (int t = 0; t < DAV_KEEP; ++t) { qv[t] = 0.0; wv[t] = 0.0; }
    for (int j = 0; j < k; ++j) {
      const double vj = V[(int64_t)j * ld + i], wj = W[(int64_t)j * ld + i];
#pragma unroll
      for (int t = 0; t < DAV_KEEP; ++t)
        if (t < kk) {
          qv[t] = fma(ys[t][j], vj, qv[t]);
          wv[t] = fma(ys[t][j], wj, wv[t]);
        }
    }
#pragma unroll
    for (int t = 0; t < DAV_KEEP; ++t)
      if (t < kk) {
        Qo[(int64_t)t * ld + i] = qv[t];
        Wo[(int64_t)t * ld + i] = wv[t];
      }
  }
}

// Spin-flip partners (S_z = 0 sector): partner[i] = internal id of the
// determinant with the alpha and beta strings of internal id i exchanged;
// *missing counts determinants whose partner is not in the space.
__global__ void k_flip_partner(const ulonglong2* __restrict__ keys_int, const ulonglong2* __restrict__ sorted,
                               const int32_t* __restrict__ s2i, int64_t n, int32_t* __restrict__ partner,
                               unsigned long long* __restrict__ missing) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const ulonglong2 k = keys_int[i];
    const ulonglong2 f = make_ulonglong2(k.y, k.x);
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      const ulonglong2 m = sorted[mid];
      if (m.x < f.x || (m.x == f.x && m.y < f.y)) lo = mid + 1;
      else hi = mid;
    }
    if (lo < n && sorted[lo].x == f.x && sorted[lo].y == f.y) {
      partner[i] = s2i[lo];
    } else {
      partner[i] = -1;
      atomicAdd(missing, 1ull);
    }
  }
}

// Projection on spin parity p: v_i <- (v_i + p v_partner(i)) / 2, each pair
// once (from its lower id, both entries written); alpha = beta determinants
// keep v_i for p = +1 and vanish for p = -1.  The two entries of a pair end
// up with exactly equal magnitudes.
__global__ void k_parity_project(double* __restrict__ v, const int32_t* __restrict__ partner, int64_t n, double p) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = partner[i];
    if (j == i) {
      if (p < 0.0) v[i] = 0.0;
    } else if (j > i) {
      const double a = v[i], b = v[j];
      const double s = 0.5 * (a + p * b);
      v[i] = s;
      v[j] = p * s;
    }
  }
}

// t <- t - eps u (the Olsen correction, see k_ritz)
__global__ void __launch_bounds__(DBLOCK) k_olsen(const DavDev* __restrict__ d, int64_t n,
                                                  const double* __restrict__ u, double* __restrict__ t) {
  const double den_x = d->rep.ols[2];
  const double eps = den_x != 0.0 ? d->rep.ols[1] / den_x : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    t[i] = fma(-eps, u[i], t[i]);
}

// v[i] += a * (a hash of i mapped to [-1, 1)): a start component in every
// symmetry sector (deflated roots need not share the lowest diagonal
// determinant's symmetry)
__global__ void k_add_hash(double* __restrict__ v, int64_t n, double a) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t x = (uint64_t)i + 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    v[i] += a * ((double)(x >> 11) * (2.0 / 9007199254740992.0) - 1.0);
  }
}

// t -= sum_j dots_j V_j
__global__ void k_orth(const double* __restrict__ V, int64_t ld, int k, const DavDev* __restrict__ d,
                       double* __restrict__ t, int64_t n) {
  __shared__ double cs[LDG];
  if (threadIdx.x < LDG) cs[threadIdx.x] = d->dots[threadIdx.x];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double v = t[i];
    for (int j = 0; j < k; ++j) v = fma(-cs[j], V[(int64_t)j * ld + i], v);
    t[i] = v;
  }
}

// x *= 1/sqrt(*s2) (and y likewise if given)
__global__ void k_scale_by(double* __restrict__ x, double* __restrict__ y, int64_t n, const double* __restrict__ s2) {
  double f = 1.0 / sqrt(*s2);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] *= f;
    if (y) y[i] *= f;
  }
}

__global__ void k_scale_const(double* __restrict__ x, int64_t n, double f) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] *= f;
}

// y = x / sqrt(|x|^2) with |x|^2 = d->nrm2 read on the device (the
// normalised correction into its subspace slot); a correction of norm^2 at
// most 1e-26 lies in the subspace: y = 0 and d->stall = 1
__global__ void k_scale_unit(const double* __restrict__ x, int64_t n, DavDev* __restrict__ d, double* __restrict__ y) {
  const double nrm2 = d->nrm2;
  const bool ok = nrm2 > 1e-26;
  const double f = ok ? 1.0 / sqrt(nrm2) : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = ok ? x[i] * f : 0.0;
  if (!ok && blockIdx.x == 0 && threadIdx.x == 0) d->rep.stall = 1;
}

// best (value, index) over the grid: the largest value, the lowest index on
// ties; true in the last block to finish, whose thread 0 gets it
__device__ __forceinline__ bool grid_best(double& bv, int64_t& bi, double* pv, int64_t* pi, unsigned int* ticket) {
  __shared__ double sv[DBLOCK / 32];
  __shared__ int64_t si[DBLOCK / 32];
  __shared__ bool s_last;
  auto block_best = [&]() {
    for (int o = 16; o; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int64_t oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = bv; si[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 1; w < DBLOCK / 32; ++w)
        if (sv[w] > bv || (sv[w] == bv && si[w] < bi)) { bv = sv[w]; bi = si[w]; }
  };
  block_best();
  if (threadIdx.x == 0) {
    pv[blockIdx.x] = bv;
    pi[blockIdx.x] = bi;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  bv = -INFINITY;
  bi = INT64_MAX;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += DBLOCK) {
    const double v = __ldcg(pv + b);
    const int64_t q = __ldcg(pi + b);
    if (v > bv || (v == bv && q < bi)) { bv = v; bi = q; }
  }
  block_best();
  if (threadIdx.x == 0) *ticket = 0u;
  return true;
}

// sign of the entry of largest magnitude (first index on ties)
__global__ void __launch_bounds__(DBLOCK) k_phase_sign(const double* __restrict__ x, int64_t n, double* __restrict__ pv,
                                                       int64_t* __restrict__ pi, DavDev* __restrict__ d,
                                                       double* __restrict__ sgn) {
  double bv = -1.0;
  int64_t bi = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = fabs(x[i]);
    if (a > bv) { bv = a; bi = i; }
  }
  if (grid_best(bv, bi, pv, pi, &d->ticket) && threadIdx.x == 0) *sgn = x[bi] < 0.0 ? -1.0 : 1.0;
}

__global__ void k_apply_sign(double* __restrict__ x, int64_t n, const double* __restrict__ sgn) {
  const double s = *sgn;
  if (s > 0.0) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = -x[i];
}

// x[i] = 1 at the smallest diagonal element (first on ties); x zeroed before
__global__ void __launch_bounds__(DBLOCK) k_unit_min_diag(double* __restrict__ x, const double* __restrict__ diag,
                                                          int64_t n, double* __restrict__ pv, int64_t* __restrict__ pi,
                                                          DavDev* __restrict__ d) {
  double bv = -INFINITY;
  int64_t bi = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (-diag[i] > bv) { bv = -diag[i]; bi = i; }
  if (grid_best(bv, bi, pv, pi, &d->ticket) && threadIdx.x == 0) x[bi] = 1.0;
}

struct Dav {
  hci_ctx* ctx;
  int64_t n, ld;
  double *V, *W, *x, *wy, *t, *u, *part;
  DavDev* d;
  int nblk;     // blocks of the elementwise passes
  // blocks of the reducing passes: each warp pays the reduction once, so few
  // blocks (one per SM: 18.6 / 24.8 us for OLSEN / ORTH at 1.2e5 elements
  // and k = 22, two 20.6 / 28.1, three 30.7 / 37.8); k_ritz, which also
  // stores four vectors, takes two (65.9 us at 5e5 elements, one 84.2)
  int rblk, rblk2;

  // out[j] = Vb_j . w, j < k; with gcol >= 0 also column gcol of G
  hci_status dots(const double* Vb, int k, const double* w, double* out, int gcol = -1) {
    const dim3 grid((unsigned)rblk, (unsigned)((k + DOTS_GROUP - 1) / DOTS_GROUP));
    HCI_LAUNCH(k_dots, grid, DBLOCK, 0, ctx->st)(Vb, ld, k, w, n, part, out, d, gcol);
    HCI_CUDA(ctx, cudaGetLastError());
    return HCI_OK;
  }
  template <int OP>
  hci_status pass(int k) {
    const int na = k + (OP == PASS_ORTH || OP == PASS_GCOL);
    const int g = OP == PASS_UNIT ? nblk : rblk;
    if (na <= 8)
      HCI_LAUNCH((k_pass<OP, 8>), g, DBLOCK, 0, ctx->st)(V, W, ld, k, n, t, u, d, part);
    else if (na <= 16)
      HCI_LAUNCH((k_pass<OP, 16>), g, DBLOCK, 0, ctx->st)(V, W, ld, k, n, t, u, d, part);
    else
      HCI_LAUNCH((k_pass<OP, MAXSUB>), g, DBLOCK, 0, ctx->st)(V, W, ld, k, n, t, u, d, part);
    HCI_CUDA(ctx, cudaGetLastError());
    return HCI_OK;
  }
  hci_status sigma(int slot) {
    return sigma_apply(ctx, V + (int64_t)slot * ld, W + (int64_t)slot * ld, 1, &d->rep.stop);
  }
};

}  // namespace

// Spin-flip partners of the cached space (built once per graph epoch);
// HCI_ERR_INVALID when the space is not closed under the flip.
static hci_status parity_prepare(hci_ctx* ctx, int64_t nV) {
  const Graph& G = ctx->graph;
  if (ctx->partner_epoch == G.epoch && ctx->d_partner.bytes >= (size_t)nV * 4) return HCI_OK;
  HCI_TRY(ensure_buf(ctx, ctx->d_partner, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  unsigned long long* miss = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 8);
  HCI_CUDA(ctx, cudaMemsetAsync(miss, 0, 8, ctx->st));
  HCI_LAUNCH(k_flip_partner, grid_for(nV, 256), 256, 0, ctx->st)(
      reinterpret_cast<const ulonglong2*>(G.keys_int.p), reinterpret_cast<const ulonglong2*>(G.keys.p),
      reinterpret_cast<const int32_t*>(G.s2i.p), nV, bp<int32_t>(ctx->d_partner), miss);
  HCI_CUDA(ctx, cudaGetLastError());
  unsigned long long h = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&h, miss, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  if (h) return hci_fail(ctx, HCI_ERR_INVALID, "spin parity: %llu determinants of V lack their spin-flip partner", h);
  ctx->partner_epoch = G.epoch;
  return HCI_OK;
}

static void parity_project(hci_ctx* ctx, double* v, int64_t nV, int nblk) {
  if (ctx->spin_parity == 0) return;
  HCI_LAUNCH(k_parity_project, nblk, DBLOCK, 0, ctx->st)(v, bp<int32_t>(ctx->d_partner), nV,
                                                        (double)ctx->spin_parity);
}

// The Davidson loop; with m > 0 locked vectors L (orthonormal, internal
// order, leading dimension (nV + 31) & ~31) the start vector and every
// correction are kept orthogonal to them, so the iteration converges to the
// lowest eigenpair of H in their complement (the next root when L holds the
// lower ones).
static hci_status davidson_core(hci_ctx* ctx, const uint64_t* keys, int64_t nV, double* c_inout, double* energy,
                                double tol, int maxit, int* iters, const double* L, int m) {
  if (iters) *iters = 0;
  HCI_TRY(graph_ensure(ctx, keys, nV));
  if (ctx->spin_parity != 0) HCI_TRY(parity_prepare(ctx, nV));
  prof_tic(ctx, HCI_PH_DAVIDSON);
  Dav D;
  D.ctx = ctx;
  D.n = nV;
  D.ld = (nV + 31) & ~(int64_t)31;
  D.nblk = grid_for(nV, DBLOCK, ctx->nsm * 8);
  D.rblk = grid_for(nV, DBLOCK, ctx->nsm);
  D.rblk2 = grid_for(nV, DBLOCK, ctx->nsm * 2);
  HCI_TRY(ensure_buf(ctx, ctx->d_vb, (size_t)D.ld * (MAXSUB + 4) * 8));
  HCI_TRY(ensure_buf(ctx, ctx->d_wb, (size_t)D.ld * MAXSUB * 8));
  HCI_TRY(ensure_buf(ctx, ctx->d_part, (size_t)(D.nblk + 1) * LDG * 8));
  HCI_TRY(ensure_buf(ctx, ctx->d_small, sizeof(DavDev) + (size_t)(D.nblk + 1) * 16));
  D.V = bp<double>(ctx->d_vb);
  D.W = bp<double>(ctx->d_wb);
  D.x = D.V + (int64_t)MAXSUB * D.ld;
  D.wy = D.x + D.ld;
  D.t = D.wy + D.ld;
  D.u = D.t + D.ld;
  D.part = bp<double>(ctx->d_part);
  D.d = bp<DavDev>(ctx->d_small);
  double* amax_v = reinterpret_cast<double*>(bp<char>(ctx->d_small) + sizeof(DavDev));
  int64_t* amax_i = reinterpret_cast<int64_t*>(amax_v + D.nblk);
  const double* diag = bp<double>(ctx->graph.diag);
  cudaStream_t st = ctx->st;
  HCI_CUDA(ctx, cudaMemsetAsync(D.d, 0, sizeof(DavDev), st));
  // A single-root run on the space the last one converged on, or on a space
  // grown from it, starts from that run's lowest Ritz vectors (zero on the
  // new determinants) with their H products: the old rows of those are
  // unchanged and the new rows cost one pass over the new rows' entries per
  // vector, so the warm start is taken when that is at most one product.
  const Graph& G = ctx->graph;
  DavKeep& K = ctx->dkeep;
  // A zero start vector asks for a cold start: the kept vectors are not used.
  double c0n2 = 0.0;
  {
    HCI_TRY(D.dots(c_inout, 1, c_inout, &D.d->nrm2));
    HCI_CUDA(ctx, cudaMemcpyAsync(&c0n2, &D.d->nrm2, 8, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
  }
  const bool same = K.valid && K.epoch == G.epoch && K.nV == nV;
  const bool grown = K.valid && !G.direct && G.parent == K.epoch && G.nold == K.nV &&
                     (double)G.tail_entries * K.k <= (double)(G.nstored > 0 ? G.nstored : 1);
  int kwarm = (m == 0 && c0n2 > 0.0 && (same || grown)) ? K.k : 0;
  if (kwarm > 0) {
    for (int j = 0; j < kwarm; ++j) {
      double* vj = D.V + (int64_t)j * D.ld;
      double* wj = D.W + (int64_t)j * D.ld;
      HCI_CUDA(ctx, cudaMemcpyAsync(vj, bp<double>(K.Q) + (int64_t)j * K.ld, (size_t)K.nV * 8,
                                    cudaMemcpyDeviceToDevice, st));
      HCI_CUDA(ctx, cudaMemcpyAsync(wj, bp<double>(K.W) + (int64_t)j * K.ld, (size_t)K.nV * 8,
                                    cudaMemcpyDeviceToDevice, st));
      if (nV > K.nV) {
        HCI_CUDA(ctx, cudaMemsetAsync(vj + K.nV, 0, (size_t)(nV - K.nV) * 8, st));
        HCI_TRY(sigma_tail(ctx, K.nV, vj, wj));
      }
    }
    for (int j = 0; j < kwarm; ++j) {
      HCI_TRY(D.dots(D.V, j + 1, D.W + (int64_t)j * D.ld, D.d->dots, j));
    }
  }
  // start vector, in the graph's internal order (after the kept vectors)
  double* V0 = D.V + (int64_t)kwarm * D.ld;
  HCI_TRY(to_internal(ctx, c_inout, V0, 1));
  double nrm2 = c0n2;
  if (ctx->spin_parity != 0 && nrm2 > 0.0 && std::isfinite(nrm2)) {
    // the start vector's part of the requested spin parity
    parity_project(ctx, V0, nV, D.nblk);
    HCI_TRY(D.dots(V0, 1, V0, &D.d->nrm2));
    HCI_CUDA(ctx, cudaMemcpyAsync(&nrm2, &D.d->nrm2, 8, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
    if (!(nrm2 > 1e-20)) nrm2 = 0.0;
  }
  if (!(nrm2 > 0.0) || !std::isfinite(nrm2)) {
    HCI_CUDA(ctx, cudaMemsetAsync(V0, 0, (size_t)nV * 8, st));
    HCI_LAUNCH(k_unit_min_diag, D.rblk, DBLOCK, 0, st)(V0, diag, nV, amax_v, amax_i, D.d);
    if (m > 0 || ctx->spin_parity != 0)
      HCI_LAUNCH(k_add_hash, D.nblk, DBLOCK, 0, st)(V0, nV, 1e-2 / std::sqrt((double)nV));
    if (ctx->spin_parity != 0) {
      parity_project(ctx, V0, nV, D.nblk);
      HCI_TRY(D.dots(V0, 1, V0, &D.d->nrm2));
      HCI_CUDA(ctx, cudaMemcpyAsync(&nrm2, &D.d->nrm2, 8, cudaMemcpyDeviceToHost, st));
      HCI_CUDA(ctx, cudaStreamSynchronize(st));
      if (!(nrm2 > 1e-20)) return hci_fail(ctx, HCI_ERR_INVALID, "hci_davidson: no state of spin parity %+d in V",
                                           ctx->spin_parity);
      HCI_LAUNCH(k_scale_const, D.nblk, DBLOCK, 0, st)(V0, nV, 1.0 / std::sqrt(nrm2));
    }
  } else {
    HCI_LAUNCH(k_scale_const, D.nblk, DBLOCK, 0, st)(V0, nV, 1.0 / std::sqrt(nrm2));
  }
  bool add_start = true;
  if (kwarm > 0) {
    // the start vector joins the kept ones only with what they do not span
    for (int pass = 0; pass < 2; ++pass) {
      HCI_TRY(D.dots(D.V, kwarm, V0, D.d->dots));
      HCI_LAUNCH(k_orth, D.nblk, DBLOCK, 0, st)(D.V, D.ld, kwarm, D.d, V0, nV);
    }
    HCI_TRY(D.dots(V0, 1, V0, &D.d->nrm2));
    HCI_CUDA(ctx, cudaMemcpyAsync(&nrm2, &D.d->nrm2, 8, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
    add_start = nrm2 > 1e-16;
    if (add_start) HCI_LAUNCH(k_scale_const, D.nblk, DBLOCK, 0, st)(V0, nV, 1.0 / std::sqrt(nrm2));
  }
  if (m > 0) {
    // start orthogonal to the locked vectors (else the unit vector at the
    // lowest diagonal element, made orthogonal)
    for (int attempt = 0; attempt < 2; ++attempt) {
      for (int pass = 0; pass < 2; ++pass) {
        HCI_TRY(D.dots(L, m, D.V, D.d->dots));
        HCI_LAUNCH(k_orth, D.nblk, DBLOCK, 0, st)(L, D.ld, m, D.d, D.V, nV);
      }
      HCI_TRY(D.dots(D.V, 1, D.V, &D.d->nrm2));
      HCI_CUDA(ctx, cudaMemcpyAsync(&nrm2, &D.d->nrm2, 8, cudaMemcpyDeviceToHost, st));
      HCI_CUDA(ctx, cudaStreamSynchronize(st));
      if (nrm2 > 1e-20) break;
      if (attempt == 1) return hci_fail(ctx, HCI_ERR_INVALID, "hci_davidson_roots: no start vector outside the roots");
      HCI_CUDA(ctx, cudaMemsetAsync(D.V, 0, (size_t)nV * 8, st));
      HCI_LAUNCH(k_unit_min_diag, D.rblk, DBLOCK, 0, st)(D.V, diag, nV, amax_v, amax_i, D.d);
      HCI_LAUNCH(k_add_hash, D.nblk, DBLOCK, 0, st)(D.V, nV, 1e-2 / std::sqrt((double)nV));
      parity_project(ctx, D.V, nV, D.nblk);
    }
    HCI_LAUNCH(k_scale_const, D.nblk, DBLOCK, 0, st)(D.V, nV, 1.0 / std::sqrt(nrm2));
  }
  int k = kwarm;
  if (add_start) {
    HCI_TRY(D.sigma(k));
    HCI_TRY(D.dots(D.V, k + 1, D.W + (int64_t)k * D.ld, D.d->dots, k));
    ++k;
  }
  bool converged = false;
  double theta = 0.0, rn = 0.0;
  int it = 0;
  // Without locked vectors or spin parity an iteration is one chain of
  // launches, and several are queued at a time: a kernel of the chain returns
  // at once when an earlier one found convergence, an unusable residual or a
  // correction inside the subspace (rep.stop).  The one-orientation and
  // direct products do not look at the flag and go one at a time.
  const bool plain = m == 0 && ctx->spin_parity == 0;
  const int ahead = plain && !G.half && !G.direct ? DAV_AHEAD : 1;
  DavReport rep = {};
  auto ritz = [&]() -> hci_status {
    HCI_LAUNCH(k_lowest<1>, 1, LW_T, 0, st)(D.d, k);
    HCI_LAUNCH(k_ritz, D.rblk2, DBLOCK, 0, st)(D.V, D.W, D.ld, k, D.d, diag, nV, D.x, D.wy, D.t, D.u, D.part,
                                              plain ? 1 : 0, tol);
    HCI_CUDA(ctx, cudaGetLastError());
    return HCI_OK;
  };
  auto report = [&]() -> hci_status {
    HCI_CUDA(ctx, cudaMemcpyAsync(&rep, &D.d->rep, sizeof rep, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
    theta = rep.theta;
    rn = std::sqrt(rep.ols[0]);
    if (!std::isfinite(theta) || !std::isfinite(rn))
      return hci_fail(ctx, HCI_ERR_CUDA, "hci_davidson: non-finite Ritz value or residual");
    return HCI_OK;
  };
  // the correction of the last Ritz step, orthogonalised twice and
  // normalised, as vector k, with its product
  auto expand = [&]() -> hci_status {
    HCI_TRY(D.pass<PASS_OLSEN>(k));
    HCI_TRY(D.pass<PASS_ORTH>(k));
    HCI_TRY(D.pass<PASS_UNIT>(k));
    HCI_TRY(D.sigma(k));
    HCI_TRY(D.pass<PASS_GCOL>(k));
    ++k;
    return HCI_OK;
  };
  auto expand_locked = [&]() -> hci_status {
    HCI_LAUNCH(k_olsen, D.nblk, DBLOCK, 0, st)(D.d, nV, D.u, D.t);
    parity_project(ctx, D.t, nV, D.nblk);
    for (int pass = 0; pass < 2; ++pass) {
      HCI_TRY(D.dots(D.V, k, D.t, D.d->dots));
      HCI_LAUNCH(k_orth, D.nblk, DBLOCK, 0, st)(D.V, D.ld, k, D.d, D.t, nV);
      if (m > 0) {
        HCI_TRY(D.dots(L, m, D.t, D.d->dots));
        HCI_LAUNCH(k_orth, D.nblk, DBLOCK, 0, st)(L, D.ld, m, D.d, D.t, nV);
      }
    }
    HCI_TRY(D.dots(D.t, 1, D.t, &D.d->nrm2));
    HCI_LAUNCH(k_scale_unit, D.nblk, DBLOCK, 0, st)(D.t, nV, D.d, D.V + (int64_t)k * D.ld);
    HCI_TRY(D.sigma(k));
    HCI_TRY(D.dots(D.V, k + 1, D.W + (int64_t)k * D.ld, D.d->dots, k));
    ++k;
    return HCI_OK;
  };
  while (it < maxit) {
    const int before = it;
    int queued = 1;
    // Vectors kept from this very space have usually converged on it: nothing
    // is queued behind the first step then (a converged call 361 us with three
    // iterations queued in vain, 325 us so).
    const int most = same && kwarm > 0 && it == 0 ? 1 : ahead;
    HCI_TRY(ritz());
    for (; queued < most && it + queued < maxit && k < MAXSUB; ++queued) {
      HCI_TRY(expand());
      HCI_TRY(ritz());
    }
    HCI_TRY(report());
    it = plain ? rep.it : it + 1;
    if (plain && rep.stop) {
      // products queued behind the stop did not run
      const int64_t skipped = (queued - 1) - (it - before - (rep.stall ? 0 : 1));
      ctx->st_counts[HCI_ST_SIGMA_CALLS] -= skipped;
      ctx->st_counts[HCI_ST_SIGMA_ROWS] -= skipped * G.nV;
      ctx->st_counts[HCI_ST_SIGMA_NNZ] -= skipped * G.nnz;
      // a correction inside the subspace: the Ritz pair before it is final
      k = rep.k;
      converged = rn <= tol;
      HCI_CUDA(ctx, cudaMemsetAsync(&D.d->rep.stop, 0, sizeof(int), st));
      break;
    }
    if (!plain && rep.stall) {
      // the last correction lay in the subspace (it was added as zeros):
      // drop it, take the Ritz pair of the subspace before it and stop
      --k;
      HCI_TRY(ritz());
      HCI_TRY(report());
      converged = rn <= tol;
      if (!converged) --it;   // not a step of its own: counted as the chain above counts
      break;
    }
    if (rn <= tol) {
      converged = true;
      break;
    }
    if (it >= maxit) break;
    if (k == MAXSUB) {
      // restart from the current Ritz vector
      HCI_CUDA(ctx, cudaMemcpyAsync(D.V, D.x, (size_t)nV * 8, cudaMemcpyDeviceToDevice, st));
      HCI_CUDA(ctx, cudaMemcpyAsync(D.W, D.wy, (size_t)nV * 8, cudaMemcpyDeviceToDevice, st));
      HCI_TRY(D.dots(D.V, 1, D.V, &D.d->nrm2));
      HCI_LAUNCH(k_scale_by, D.nblk, DBLOCK, 0, st)(D.V, D.W, nV, &D.d->nrm2);
      HCI_TRY(D.dots(D.V, 1, D.W, D.d->dots, 0));
      k = 1;
    }
    HCI_TRY(plain ? expand() : expand_locked());
  }
  if (iters) *iters = it;
  // the lowest Ritz vectors for a later run on this space or a grown one
  K.valid = false;
  if (m == 0 && converged) {
    const int kk = k < DAV_KEEP ? k : DAV_KEEP;
    if (ensure_buf(ctx, K.Q, (size_t)D.ld * kk * 8) == HCI_OK && ensure_buf(ctx, K.W, (size_t)D.ld * kk * 8) == HCI_OK) {
      HCI_LAUNCH(k_lowest<DAV_KEEP>, 1, LW_T, 0, st)(D.d, k);
      HCI_LAUNCH(k_keep, D.nblk, DBLOCK, 0, st)(D.V, D.W, D.ld, k, D.d, kk, nV, bp<double>(K.Q), bp<double>(K.W));
      K.valid = true;
      K.epoch = G.epoch;
      K.nV = nV;
      K.ld = D.ld;
      K.k = kk;
    }
  }
  // final vector: normalise, back to the caller's order, fix the phase
  // there (largest |c|, first sorted position on ties); with a spin parity
  // projected once more, so that the entries of a flip pair have equal
  // magnitudes exactly
  parity_project(ctx, D.x, nV, D.nblk);
  HCI_TRY(D.dots(D.x, 1, D.x, &D.d->nrm2));
  HCI_LAUNCH(k_scale_by, D.nblk, DBLOCK, 0, st)(D.x, nullptr, nV, &D.d->nrm2);
  HCI_TRY(to_sorted(ctx, D.x, c_inout, 1));
  HCI_LAUNCH(k_phase_sign, D.rblk, DBLOCK, 0, st)(c_inout, nV, amax_v, amax_i, D.d, &D.d->dots[0]);
  HCI_LAUNCH(k_apply_sign, D.nblk, DBLOCK, 0, st)(c_inout, nV, &D.d->dots[0]);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_DAVIDSON);
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  *energy = theta;
  if (!converged && rn > tol)
    return hci_fail(ctx, HCI_ERR_NOT_CONVERGED, "hci_davidson: residual %.3e > tol %.3e after %d iterations", rn, tol,
                    it);
  return HCI_OK;
}

extern "C" hci_status hci_set_spin_parity(hci_ctx* ctx, int parity) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_set_spin_parity: null context");
  if (parity < -1 || parity > 1) return hci_fail(ctx, HCI_ERR_INVALID, "hci_set_spin_parity: parity %d not in {-1, 0, 1}", parity);
  if (parity != 0 && ctx->na != ctx->nb)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_set_spin_parity: needs n_alpha = n_beta (S_z = 0), got %d and %d", ctx->na,
                    ctx->nb);
  if (parity != ctx->spin_parity) ctx->dkeep.valid = false;
  ctx->spin_parity = parity;
  return HCI_OK;
}

extern "C" hci_status hci_davidson(hci_ctx* ctx, const uint64_t* keys, int64_t nV, double* c_inout, double* energy,
                                   double tol, int maxit, int* iters) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_davidson: null context");
  if (nV <= 0 || !keys || !c_inout || !energy)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_davidson: empty space or null pointer");
  return davidson_core(ctx, keys, nV, c_inout, energy, tol, maxit, iters, nullptr, 0);
}

extern "C" hci_status hci_davidson_roots(hci_ctx* ctx, const uint64_t* keys, int64_t nV, int nroots, double* c_inout,
                                         double* energies, double tol, int maxit, int* iters) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_davidson_roots: null context");
  if (nV <= 0 || !keys || !c_inout || !energies)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_davidson_roots: empty space or null pointer");
  if (nroots < 1 || nroots > nV || nroots > LDG)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_davidson_roots: nroots must lie in [1, min(nV, %d)]", LDG);
  if (iters) *iters = 0;
  HCI_TRY(graph_ensure(ctx, keys, nV));
  const int64_t ld = (nV + 31) & ~(int64_t)31;
  HCI_TRY(ensure_buf(ctx, ctx->d_lock, (size_t)ld * nroots * 8));
  double* L = bp<double>(ctx->d_lock);
  int total = 0;
  for (int r = 0; r < nroots; ++r) {
    int it = 0;
    hci_status s = davidson_core(ctx, keys, nV, c_inout + (int64_t)r * nV, &energies[r], tol, maxit, &it, L, r);
    total += it;
    if (iters) *iters = total;
    if (s != HCI_OK) return s;
    HCI_TRY(to_internal(ctx, c_inout + (int64_t)r * nV, L + (int64_t)r * ld, 1));
  }
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  return HCI_OK;
}
