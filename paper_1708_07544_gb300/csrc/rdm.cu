// Spin-summed variational 1- and 2-RDMs accumulated over the connections of
// V (Sec. IV: the variational RDMs reuse the single/double connections of
// the Hamiltonian build; Gamma^{c,c} of Eq. vdedk2).
//
//   rdm1[p,q]     = sum_s  <a+_ps a_qs>
//   rdm2[p,q,r,s] = sum_st <a+_ps a+_rt a_st a_qs>
//
// For a connection D_i = phase * (excitation of D_j) with weight
// w = c_i c_j phase, the non-zero operator strings are:
//   single a->b (spin S), each spectator k occupied in D_j (spin T):
//     rdm1[b,a] += w; rdm2[b,a,k,k] += w; rdm2[k,k,b,a] += w;
//     if T == S: rdm2[k,a,b,k] -= w; rdm2[b,k,k,a] -= w
//   double a->c, b->d (holes a<b, particles c<d in one spin, or a->c alpha
//   and b->d beta): rdm2[c,a,d,b] += w; rdm2[d,b,c,a] += w;
//     same spin only: rdm2[c,b,d,a] -= w; rdm2[d,a,c,b] -= w
// One orientation of each connected pair is accumulated (the graph stores
// one, or both) and the other added as its transpose.  The diagonal part is
// reduced through the weighted
// occupation correlation M[sp][tq] = sum_i c_i^2 n_sp(i) n_tq(i), summed from
// the orbitals in which each determinant differs from the aufbau one.
#include "hci_internal.cuh"
#include "rdm_acc.cuh"

namespace {

constexpr int R_WARPS = 8;


// A determinant with its coefficient, one 32-byte sector, gathered by one
// 32-byte load per lane: gathers and additions each take a lane's turn in
// the L1's address stage (one per clock per SM), which bounds the kernels
// below, so the key and the coefficient take one turn instead of two.
struct __align__(32) DetC {
  uint64_t a, b;
  double c;
  uint64_t pad;
};
__global__ void k_pack_det(const ulonglong2* __restrict__ V, const double* __restrict__ c, int64_t nV,
                           DetC* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nV; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = DetC{V[i].x, V[i].y, c[i], 0ull};
}
__device__ __forceinline__ void load_det(const DetC* p, ulonglong2& k, double& c) {
  uint64_t x, y, z, u;
  asm volatile("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(x), "=l"(y), "=l"(z), "=l"(u) : "l"(p));
  k = make_ulonglong2(x, y);
  c = __longlong_as_double((long long)z);
}

// Chunks of RQ_CHUNK stored entries from a queue, whatever rows they belong to
// (a row of 1e5 entries left to one warp is a tail several times as long as
// all the rest).  One-orientation graphs: every stored entry is one
// orientation of a connected pair; both-orientation graphs: the entries with
// j > i are.  The pairs to accumulate are queued per
// warp (half of a full row's entries are the other orientation's) and looked
// at 32 at a time; alpha-beta doubles, most of them, are added at once,
// same-spin doubles and singles (whose spectators loop) are queued again by
// kind, so that no lane waits through another kind's code.  (44e,44o), 4.9e8
// pairs: 15.4 ms with every kind in place and 2 to 4 atomics per double,
// 5.2 ms so.
constexpr int RQ_CHUNK = 2048;

__global__ void __launch_bounds__(R_WARPS * 32) k_rdm_offdiag(int n, const DetC* __restrict__ V, int64_t nV,
                                                              const int64_t* __restrict__ rowptr,
                                                              const int64_t* __restrict__ rowstart,
                                                              const __grid_constant__ SegTab T, int both, RdmAcc R,
                                                              unsigned long long* __restrict__ queue) {
  __shared__ int2 s_q[R_WARPS][3][64];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int2(*q)[64] = s_q[threadIdx.x >> 5];
  int nq = 0, ns = 0, n1 = 0;        // queued pairs, same-spin doubles, singles
  auto shift = [&](int2* w, int& cnt, int m) {
    const int2 rest = lane + m < cnt ? w[lane + m] : make_int2(0, 0);
    __syncwarp();
    if (lane + m < cnt) w[lane] = rest;
    cnt -= m;
    __syncwarp();
  };
  auto take_kind = [&](int kind, int& cnt, int m) {
    __syncwarp();
    if (lane < m) {
      const int2 p = q[kind][lane];
      ulonglong2 ki, kj;
      double ci, cj;
      load_det(V + p.x, ki, ci);
      load_det(V + p.y, kj, cj);
      const double cc = ci * cj;
      if (cc != 0.0) {
        if (kind == 2) rdm_single(R, n, ki, kj, cc);
        else if (ki.y == kj.y) rdm_same(R, n, ki.x, kj.x, cc);
        else rdm_same(R, n, ki.y, kj.y, cc);
      }
    }
    shift(q[kind], cnt, m);
  };
  auto take = [&](int m) {   // the first m <= 32 queued pairs
    __syncwarp();
    bool same = false, one = false;
    int2 p = make_int2(0, 0);
    if (lane < m) {
      p = q[0][lane];
      ulonglong2 ki, kj;
      double ci, cj;
      load_det(V + p.x, ki, ci);
      load_det(V + p.y, kj, cj);
      const int da = __popcll(ki.x ^ kj.x), db = __popcll(ki.y ^ kj.y);
      one = da + db == 2;
      same = !one && da != db;
      const double cc = ci * cj;
      if (!one && !same && cc != 0.0) rdm_mixed(R, n, ki, kj, cc);
    }
    const unsigned bs = __ballot_sync(0xffffffffu, same), b1 = __ballot_sync(0xffffffffu, one);
    if (same) q[1][ns + __popc(bs & lt)] = p;
    if (one) q[2][n1 + __popc(b1 & lt)] = p;
    ns += __popc(bs);
    n1 += __popc(b1);
    shift(q[0], nq, m);
    if (ns >= 32) take_kind(1, ns, 32);
    if (n1 >= 32) take_kind(2, n1, 32);
  };
  const int64_t total = rowptr[nV];
  while (true) {
    unsigned long long qi = 0;
    if (lane == 0) qi = atomicAdd(queue, (unsigned long long)RQ_CHUNK);
    const int64_t e0 = (int64_t)__shfl_sync(0xffffffffu, qi, 0);
    if (e0 >= total) break;
    const int64_t e1 = e0 + RQ_CHUNK < total ? e0 + RQ_CHUNK : total;
    int64_t e = e0;
    for (int64_t i = row_of_entry(rowptr, nV, e0); e < e1; ++i) {
      const int64_t lo = rowptr[i], hi = rowptr[i + 1] < e1 ? rowptr[i + 1] : e1;
      const int64_t rs = rowstart[i], off = e - lo, len = hi - e;
      e = hi;
      if (len <= 0 || V[i].c == 0.0) continue;
      const int32_t* col = T.col[rs >> GRAPH_SEG_SHIFT] + (rs & GRAPH_SEG_MASK) + off;
      int32_t jn = lane < len ? __ldcs(col + lane) : -1;
      for (int64_t k0 = 0; k0 < len; k0 += 32) {
        const int32_t j = jn;
        jn = k0 + 32 + lane < len ? __ldcs(col + k0 + 32 + lane) : -1;
        const bool ok = j >= 0 && (!both || j > i);
        const unsigned b = __ballot_sync(0xffffffffu, ok);
        if (ok) q[0][nq + __popc(b & lt)] = make_int2((int)i, j);
        nq += __popc(b);
        if (nq >= 32) take(32);
      }
    }
  }
  if (nq > 0) take(nq);
  if (ns > 0) take_kind(1, ns, ns);
  if (n1 > 0) take_kind(2, n1, n1);
}

// Single-excitation spectator sums: Xt[b][a][k] over both spins,
// Xx[b][a][k] over the excitation's own spin (spectator k != a).
__device__ __forceinline__ double rdm_xt(const RdmAcc& R, int n, int b, int a, int k) {
  const int64_t ba = (int64_t)b * n + a;
  const double s = R.S1[ba] + R.S1[(int64_t)n * n + ba];
  const int occ = (int)((R.ref_a >> k) & 1ull) + (int)((R.ref_b >> k) & 1ull) - (k == a);
  return s * occ + R.Ds[ba * n + k] + R.Do[ba * n + k];
}
__device__ __forceinline__ double rdm_xx(const RdmAcc& R, int n, int b, int a, int k) {
  const int64_t ba = (int64_t)b * n + a;
  const int oa = (int)((R.ref_a >> k) & 1ull) - (k == a), ob = (int)((R.ref_b >> k) & 1ull) - (k == a);
  return R.S1[ba] * oa + R.S1[(int64_t)n * n + ba] * ob + R.Ds[ba * n + k];
}
// the single-excitation terms of one orientation at (p,q,r,s)
__device__ __forceinline__ double rdm_single_terms(const RdmAcc& R, int n, int p, int q, int r, int s) {
  double v = 0.0;
  if (r == s) v += rdm_xt(R, n, p, q, r);
  if (p == q) v += rdm_xt(R, n, r, s, p);
  if (s == p) v -= rdm_xx(R, n, r, q, p);
  if (q == r) v -= rdm_xx(R, n, p, s, q);
  return v;
}

// the doubles of one orientation at (p,q,r,s): alpha-beta pairs in both
// orders, same-spin pairs with the sign of their particles' and holes' order
__device__ __forceinline__ double rdm_double_terms(const RdmAcc& R, int n, int p, int q, int r, int s) {
  const int64_t pq = (int64_t)p * n + q, rs = (int64_t)r * n + s, n2 = (int64_t)n * n;
  double v = R.Hm[pq * n2 + rs] + R.Hm[rs * n2 + pq];
  if (p != r && q != s) {
    const int np = n * (n - 1) / 2;
    const double x = R.Hs[(int64_t)(p < r ? tri_index(p, r) : tri_index(r, p)) * np +
                          (q < s ? tri_index(q, s) : tri_index(s, q))];
    v += (p < r) == (q < s) ? x : -x;
  }
  return v;
}

// rdm2 += doubles + single terms, rdm1 += S1 (the accumulated orientation), and
// with sym also their transposes (the other orientation of every pair)
__global__ void k_rdm_finish(int n, RdmAcc R, double* __restrict__ r1, double* __restrict__ r2, int sym) {
  const int64_t n2 = (int64_t)n * n, n4 = n2 * n2;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x) {
    const int s = (int)(t % n), r = (int)((t / n) % n), q = (int)((t / n2) % n), p = (int)(t / (n2 * n));
    double v = rdm_double_terms(R, n, p, q, r, s) + rdm_single_terms(R, n, p, q, r, s);
    if (sym) v += rdm_double_terms(R, n, q, p, s, r) + rdm_single_terms(R, n, q, p, s, r);
    r2[t] += v;
    if (t < n2) {
      const int pp = (int)(t / n), qq = (int)(t % n);
      double w = R.S1[t] + R.S1[n2 + t];
      if (sym) w += R.S1[(int64_t)qq * n + pp] + R.S1[n2 + (int64_t)qq * n + pp];
      r1[t] += w;
    }
  }
}

// Transition density of screened perturbative pairs: <V[src[j]]| op |tgt[j]>
// with weight c[src[j]] d[j] (pairs with d = 0 skipped).
__global__ void k_rdm_pairs(int n, const ulonglong2* __restrict__ V, const double* __restrict__ c,
                            const ulonglong2* __restrict__ tgt, const int32_t* __restrict__ src,
                            const double* __restrict__ d, int64_t m, RdmAcc R) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
    const double dj = d[j];
    if (dj == 0.0) continue;
    const int32_t i = src[j];
    rdm_accumulate(R, n, V[i], tgt[j], c[i] * dj);
  }
}

// Occupation correlation sum_a w_a n(a) n(a)^T, w_a = d_a^2, of determinants
// tgt[j] (j = 0 .. m - 1, or the listed j = list[0 .. *nlist)), over spin orbitals
// (alpha 0..n-1, beta n..2n-1), split about the aufbau occupations n_R:
// n(a) = n_R + delta_a.  A changed spin orbital k has delta_k = s_k, -1 when
// n_R holds it and +1 when not, so only the weights P_kl = sum of w over the
// targets that change both k and l are accumulated (k <= l, P_kk among them),
// with W = sum w: about 36 additions per target.  They go to L2 as FP64
// reductions without return, spread over DD_COPIES copies [W, P (2n x 2n)]
// so that the frontier orbitals' entries do not queue up at one address.
// The same sums with w = c_i^2 over V are the diagonal part of the RDMs
// (3.0e5 determinants: 82 + 700 + 21 us by string groups, 34 us so).
// FP64 additions in shared memory are compare-and-swap loops: block-local
// copies there took 71.4 ms for the pairs of a (44e,44o) state at eps2 = 2e-5,
// this 4.7 ms.
constexpr int DD_COPIES = 64;

__global__ void __launch_bounds__(256) k_dd_acc(int n, const ulonglong2* __restrict__ tgt, const double* __restrict__ d,
                                                int64_t m, const int64_t* __restrict__ list,
                                                const unsigned long long* __restrict__ nlist, uint64_t ra, uint64_t rb,
                                                double* __restrict__ acc) {
  const int mm = 2 * n;
  double* A = acc + (int64_t)(blockIdx.x % DD_COPIES) * (1 + mm * mm);
  double* P = A + 1;
  double wsum = 0.0;
  const int64_t nt = list ? (int64_t)*nlist : m;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nt; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = list ? list[q] : q;
    const double dj = d[j];
    if (dj == 0.0) continue;
    const ulonglong2 key = tgt[j];
    const double w = dj * dj;
    wsum += w;
    const uint64_t da = key.x ^ ra, db = key.y ^ rb;
    for (uint64_t x = da; x; x &= x - 1) {
      double* row = P + (__ffsll((long long)x) - 1) * mm;
      for (uint64_t y = x; y; y &= y - 1) atomicAdd(row + __ffsll((long long)y) - 1, w);
      for (uint64_t y = db; y; y &= y - 1) atomicAdd(row + n + __ffsll((long long)y) - 1, w);
    }
    for (uint64_t x = db; x; x &= x - 1) {
      double* row = P + (n + __ffsll((long long)x) - 1) * mm + n;
      for (uint64_t y = x; y; y &= y - 1) atomicAdd(row + __ffsll((long long)y) - 1, w);
    }
  }
  for (int o = 16; o; o >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
  if ((threadIdx.x & 31) == 0 && wsum != 0.0) atomicAdd(A, wsum);
}

// sum[t] = sum of the copies' entries t, in order
__global__ void k_dd_sum(int cnt, const double* __restrict__ acc, double* __restrict__ sum) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= cnt) return;
  double s = 0.0;
#pragma unroll 8
  for (int c = 0; c < DD_COPIES; ++c) s += acc[(int64_t)c * cnt + t];
  sum[t] = s;
}

// M = W n_R n_R^T + n_R u^T + u n_R^T + Q, u_k = s_k P_kk, Q_kl = s_k s_l
// P_kl, the layout k_diag_rdm reads
__global__ void k_dd_matrix(int n, const double* __restrict__ sum, uint64_t ra, uint64_t rb, double* __restrict__ M) {
  const int mm = 2 * n;
  const double W = sum[0];
  const double* P = sum + 1;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < mm * mm; t += gridDim.x * blockDim.x) {
    const int k = t / mm, l = t % mm;
    const double nk = (k < n ? ((ra >> k) & 1ull) : ((rb >> (k - n)) & 1ull)) ? 1.0 : 0.0;
    const double nl = (l < n ? ((ra >> l) & 1ull) : ((rb >> (l - n)) & 1ull)) ? 1.0 : 0.0;
    const double sk = 1.0 - 2.0 * nk, sl = 1.0 - 2.0 * nl;
    const double p = k < l ? P[k * mm + l] : P[l * mm + k];
    M[t] = W * nk * nl + nk * (sl * P[l * mm + l]) + (sk * P[k * mm + k]) * nl + sk * sl * p;
  }
}

// diagonal contributions from M
__global__ void k_diag_rdm(int n, const double* __restrict__ M, double* __restrict__ r1, double* __restrict__ r2) {
  const int m = 2 * n;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += gridDim.x * blockDim.x) {
    const int p = t / n, q = t % n;
    double coul = 0.0;
    for (int s = 0; s < 2; ++s)
      for (int u = 0; u < 2; ++u)
        if (!(p == q && s == u)) coul += M[(s * n + p) * m + u * n + q];
    r2[(((int64_t)p * n + p) * n + q) * n + q] += coul;
    if (p != q) {
      double ex = M[p * m + q] + M[(n + p) * m + n + q];
      r2[(((int64_t)p * n + q) * n + q) * n + p] -= ex;
    } else {
      r1[p * n + p] += M[p * m + p] + M[(n + p) * m + n + p];
    }
  }
}

}  // namespace

static RdmAcc ctx_acc(hci_ctx* ctx) {
  return rdm_acc_at(bp<double>(ctx->s_rdmh), (size_t)ctx->n, ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull),
                    ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull));
}

extern "C" hci_status hci_rdm12(hci_ctx* ctx, const uint64_t* keys, int64_t nV, const double* c, double* rdm1,
                                double* rdm2) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_rdm12: null context");
  if (nV <= 0 || !keys || !c || !rdm1 || !rdm2)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_rdm12: empty space or null pointer");
  HCI_TRY(graph_ensure(ctx, keys, nV));
  const int n = ctx->n;
  cudaStream_t st = ctx->st;
  prof_tic(ctx, HCI_PH_RDM);
  const size_t n2 = (size_t)n * n, n4 = n2 * n2;
  HCI_CUDA(ctx, cudaMemsetAsync(rdm1, 0, n2 * 8, st));
  HCI_CUDA(ctx, cudaMemsetAsync(rdm2, 0, n4 * 8, st));
  prof_tic(ctx, HCI_PH_RDM_DIAG);
  // diagonal part: M[s*n+p][t*n+q] = sum_i c_i^2 n_sp(i) n_tq(i)
  const int cnt = 1 + 4 * n * n;
  HCI_TRY(ensure_buf(ctx, ctx->s_rdmw, ((size_t)(DD_COPIES + 1) * cnt + 4 * n2) * 8));
  double* acc = bp<double>(ctx->s_rdmw);
  double* sum = acc + (size_t)DD_COPIES * cnt;
  double* M = sum + cnt;
  const uint64_t ra = ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull);
  const uint64_t rb = ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull);
  HCI_CUDA(ctx, cudaMemsetAsync(acc, 0, (size_t)DD_COPIES * cnt * 8, st));
  HCI_LAUNCH(k_dd_acc, grid_for(nV, 256, ctx->nsm * 8), 256, 0, st)(n, bp<ulonglong2>(ctx->graph.keys), c, nV, nullptr,
                                                                   nullptr, ra, rb, acc);
  HCI_LAUNCH(k_dd_sum, (unsigned)((cnt + 255) / 256), 256, 0, st)(cnt, acc, sum);
  HCI_LAUNCH(k_dd_matrix, grid_for((int64_t)4 * n2, 256), 256, 0, st)(n, sum, ra, rb, M);
  HCI_LAUNCH(k_diag_rdm, grid_for((int64_t)n2, 256), 256, 0, st)(n, M, rdm1, rdm2);
  prof_toc(ctx, HCI_PH_RDM_DIAG);
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  unsigned long long* queue = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 56);
  HCI_CUDA(ctx, cudaMemsetAsync(queue, 0, 8, st));
  // the connections are stored by internal id
  HCI_TRY(ensure_buf(ctx, ctx->d_perm, (size_t)nV * 40 + 32));
  DetC* det = bp<DetC>(ctx->d_perm);
  double* ci = reinterpret_cast<double*>(det + nV);
  HCI_TRY(to_internal(ctx, c, ci, 1));
  HCI_TRY(ensure_buf(ctx, ctx->s_rdmh, rdm_acc_doubles(n) * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(ctx->s_rdmh.p, 0, rdm_acc_doubles(n) * 8, st));
  const RdmAcc R = ctx_acc(ctx);
  if (ctx->graph.direct)
    HCI_TRY(direct_rdm(ctx, ci, R));   // connections searched again, one orientation each
  else {
    HCI_LAUNCH(k_pack_det, grid_for(nV, 256), 256, 0, st)(bp<ulonglong2>(ctx->graph.keys_int), ci, nV, det);
    HCI_LAUNCH(k_rdm_offdiag, ctx->nsm * 8, R_WARPS * 32, 0, st)(n, det, nV, bp<int64_t>(ctx->graph.rowptr),
                                                                 bp<int64_t>(ctx->graph.rowstart), ctx->graph.tab(),
                                                                 ctx->graph.half ? 0 : 1, R, queue);
  }
  HCI_LAUNCH(k_rdm_finish, grid_for((int64_t)n4, 256, ctx->nsm * 8), 256, 0, st)(n, R, rdm1, rdm2, 1);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_RDM);
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  return HCI_OK;
}

namespace {
// <S^2> = -N (N - 4) / 4 - 1/2 sum_pq rdm2[p,q,q,p], from S^2 = S_z^2 +
// (S_+ S_- + S_- S_+) / 2 written with the spin-summed 2-RDM of hci_rdm12
__global__ void k_spin_square(const double* __restrict__ rdm2, int n, int nelec, double* __restrict__ out) {
  __shared__ double red[256];
  double s = 0.0;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int p = t / n, q = t % n;
    s += rdm2[(((int64_t)p * n + q) * n + q) * n + p];
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = -0.25 * nelec * (nelec - 4.0) - 0.5 * red[0];
}
}  // namespace

extern "C" hci_status hci_spin_square(hci_ctx* ctx, const double* rdm2, double* s2) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_spin_square: null context");
  if (!rdm2 || !s2) return hci_fail(ctx, HCI_ERR_INVALID, "hci_spin_square: null pointer");
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  double* d = reinterpret_cast<double*>(bp<char>(ctx->s_counter) + 32);
  HCI_LAUNCH(k_spin_square, 1, 256, 0, ctx->st)(rdm2, ctx->n, ctx->na + ctx->nb, d);
  HCI_CUDA(ctx, cudaGetLastError());
  HCI_CUDA(ctx, cudaMemcpyAsync(s2, d, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  return HCI_OK;
}

// Density matrices of the perturbative correction, accumulated over the
// hash classes of hci_pt2: begin (clear), pairs (once per class), finish.
hci_status pt2_rdm_begin(hci_ctx* ctx) {
  const size_t n = (size_t)ctx->n, m = 2 * n;
  HCI_TRY(ensure_buf(ctx, ctx->s_rdmh, rdm_acc_doubles(n) * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(ctx->s_rdmh.p, 0, rdm_acc_doubles(n) * 8, ctx->st));
  // the copies, their sum and M
  HCI_TRY(ensure_buf(ctx, ctx->p2_dd, ((DD_COPIES + 1) * (1 + m * m) + m * m) * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(ctx->p2_dd.p, 0, DD_COPIES * (1 + m * m) * 8, ctx->st));
  return HCI_OK;
}

hci_status pt2_rdm_pairs(hci_ctx* ctx, const ulonglong2* V, const double* c, const ulonglong2* tgt, const int32_t* src,
                         const double* d, int64_t m, const int64_t* list, const unsigned long long* nlist) {
  if (m <= 0) return HCI_OK;
  const int n = ctx->n;
  RdmAcc R = ctx_acc(ctx);
  HCI_LAUNCH(k_rdm_pairs, grid_for(m, 256), 256, 0, ctx->st)(n, V, c, tgt, src, d, m, R);
  HCI_LAUNCH(k_dd_acc, grid_for(m, 256, ctx->nsm * 8), 256, 0, ctx->st)(n, tgt, d, m, list, nlist, R.ref_a, R.ref_b,
                                                                       bp<double>(ctx->p2_dd));
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

hci_status pt2_rdm_finish(hci_ctx* ctx, double* r1dd, double* r2dd, double* r1dc, double* r2dc) {
  const int n = ctx->n, mm = 2 * n;
  const size_t n2 = (size_t)n * n, n4 = n2 * n2;
  cudaStream_t st = ctx->st;
  RdmAcc R = ctx_acc(ctx);
  HCI_CUDA(ctx, cudaMemsetAsync(r1dc, 0, n2 * 8, st));
  HCI_CUDA(ctx, cudaMemsetAsync(r2dc, 0, n4 * 8, st));
  HCI_LAUNCH(k_rdm_finish, grid_for((int64_t)n4, 256, ctx->nsm * 8), 256, 0, st)(n, R, r1dc, r2dc, 0);
  const int cnt = 1 + mm * mm;
  double* acc = bp<double>(ctx->p2_dd);
  double* sum = acc + (int64_t)DD_COPIES * cnt;
  double* M = sum + cnt;
  HCI_LAUNCH(k_dd_sum, (unsigned)((cnt + 255) / 256), 256, 0, st)(cnt, acc, sum);
  HCI_LAUNCH(k_dd_matrix, grid_for((int64_t)mm * mm, 256), 256, 0, st)(n, sum, R.ref_a, R.ref_b, M);
  HCI_CUDA(ctx, cudaMemsetAsync(r1dd, 0, n2 * 8, st));
  HCI_CUDA(ctx, cudaMemsetAsync(r2dd, 0, n4 * 8, st));
  HCI_LAUNCH(k_diag_rdm, grid_for((int64_t)n2, 256), 256, 0, st)(n, M, r1dd, r2dd);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}
