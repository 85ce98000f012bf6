// Selection step of variational HCI (Sec. II.A, Eq. criteria, Fig. 1b):
// heat-bath walk over the sorted double-excitation lists, exact singles
// behind an upper-bound screen, sort-based deduplication against V, and the
// sorted merge V^{mu+1} = V^mu + C^mu.
#include <algorithm>
#include <cmath>
#include <vector>

#include "hci_internal.cuh"

namespace {

constexpr int SEL_WARPS = 8;          // warps per CTA in the walk kernels
constexpr int WALK_CHUNK = 256;       // list entries per walk work item

struct WalkArgs {
  int n, na, nb;
  const ulonglong2* keys;
  const double* c;
  int64_t nV;
  double eps1;
  int accept_all;
  const double* opp_mag;
  const uint16_t* opp_tgt;
  int Lo;
  const double* same_mag;
  const uint16_t* same_tgt;
  int Ls;
  double max_dbl;        // largest magnitude in any list
  const double* list_max; // [n*n] opposite-spin then [n(n-1)/2] same-spin list maxima
  const double* h;
  const double* jk_same;
  const double* j_opp;
  const double* single_bound;
  const uint16_t* single_pr;       // singles by descending bound, the bounds and the tables of the
  const float* single_bf;          // tight bound rounded up to FP32
  const float* single_f32;
  const float4* single_max;        // per sorted single: |F_R| alpha, beta, largest same- and other-spin term
  ulonglong2* out;
  int64_t cap;
  unsigned long long* counter;     // [0] candidates, [1] next det (work queue)
  unsigned long long* walkstat;    // [0] list entries walked, [1] exact singles
  int4* items;                     // walk work items {det, code, start, end}
  int64_t item_cap;
  unsigned long long* nitems;
  const double* f_ref;             // [2][n][n] single-excitation rows of the aufbau determinant
  uint64_t ref_a, ref_b;
  // perturbative mode (vals != nullptr): every emitted target also gets its
  // term H_ai c_i, emitted only when |H_ai c_i| > eps1 and the target's hash
  // class is `part` of `npart`
  double* vals;
  int32_t* srcs;         // perturbative mode with sources: source determinant of each pair; vals then
                         // holds the element H_ai instead of the term H_ai c_i
  int npart, part;
};

// perturbative mode: keep the term and the target?
__device__ __forceinline__ bool pt_keep(const WalkArgs& A, ulonglong2 key, double term) {
  return fabs(term) > A.eps1 && (A.npart <= 1 || (int)(key_mix(key) % (uint64_t)A.npart) == A.part);
}

__device__ __forceinline__ void tri_decode_dev(int t, int& lo, int& hi) {
  int h = (int)((1.0 + sqrt(1.0 + 8.0 * (double)t)) * 0.5);
  while (h * (h - 1) / 2 > t) --h;
  while ((h + 1) * h / 2 <= t) ++h;
  hi = h;
  lo = t - h * (h - 1) / 2;
}

// Emitted keys (with terms and sources) of a warp, gathered in shared memory
// and appended 64 or more at a time: an append per 32 tried targets is bound
// by the one counter's atomic rate (1e7 of them: 5 ms).
constexpr int EM_CAP = 96, EM_FLUSH = 64;
struct EmitBuf {
  ulonglong2 key[EM_CAP];
  double term[EM_CAP];
  int32_t src[EM_CAP];
};

__device__ __forceinline__ void emit_flush(EmitBuf& B, int& cnt, const WalkArgs& A) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  if (cnt == 0) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(&A.counter[0], (unsigned long long)cnt);
  base = __shfl_sync(0xffffffffu, base, 0);
  for (int k = lane; k < cnt; k += 32) {
    const unsigned long long idx = base + k;
    if ((int64_t)idx < A.cap) {
      A.out[idx] = B.key[k];
      if (A.vals) A.vals[idx] = B.term[k];
      if (A.srcs) A.srcs[idx] = B.src[k];
    }
  }
  cnt = 0;
  __syncwarp();
}

// one optional key (and term) per lane
__device__ __forceinline__ void warp_emit(bool emit, ulonglong2 key, double term, int src, EmitBuf& B, int& cnt,
                                          const WalkArgs& A) {
  const unsigned m = __ballot_sync(0xffffffffu, emit);
  if (!m) return;
  if (emit) {
    const int at = cnt + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
    B.key[at] = key;
    if (A.vals) B.term[at] = term;
    if (A.srcs) B.src[at] = src;
  }
  cnt += __popc(m);
  if (cnt >= EM_FLUSH) emit_flush(B, cnt, A);
}

// The warp's next determinants, one per lane (nV or above: none), or -1 at
// the queue's end: 32 of them, or about nV / warps where that is less, so that
// a small set of large coefficients (a sample's draws, a first selection) is
// spread over every warp.  An atomic per determinant would bound spaces of
// small coefficients; those of a fetch lie far apart, because determinants of
// large coefficients are neighbours (32 consecutive ones: 3.9 ms of k_singles
// where these take 0.3).  Fourteen selections of (12e,12o) spaces: 1.75 ms of
// k_walk_plan with 32 always, 1.23 so.
__device__ __forceinline__ int64_t next_dets(const WalkArgs& A) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * SEL_WARPS, each = (A.nV + warps - 1) / warps;
  const int per = each < 1 ? 1 : each < 32 ? (int)each : 32;
  const int64_t stride = (A.nV + per - 1) / per;
  unsigned long long q = 0;
  if (lane == 0) q = atomicAdd(&A.counter[1], 1ull);
  q = __shfl_sync(0xffffffffu, q, 0);
  if ((int64_t)q >= stride) return -1;
  return lane < per ? (int64_t)q + lane * stride : A.nV;
}

// Compact the occupied orbitals of a spin string into smem (ascending).
__device__ __forceinline__ void occ_list(uint64_t s, int n, int* occ) {
  const int lane = threadIdx.x & 31;
  int base = 0;
  for (int p0 = 0; p0 < n; p0 += 32) {
    int p = p0 + lane;
    bool o = p < n && ((s >> p) & 1ull);
    unsigned m = __ballot_sync(0xffffffffu, o);
    if (o) occ[base + __popc(m & ((1u << lane) - 1u))] = p;
    base += __popc(m);
  }
  __syncwarp();
}

// Doubles, planning pass: 32 determinants at a time from a queue (an atomic
// each would bound a space of small coefficients, most of which the largest
// element cannot lift over the threshold), one warp per remaining one.  For
// every occupied pair whose largest element passes in FP32 (maximum and
// coefficient rounded up, threshold down) the length L of the list prefix
// with |v||c_i| > eps1 is found by binary search in FP64 (four pairs of a
// lane side by side: the dependent loads of a single determinant of large
// coefficient are the kernel's tail), and the prefix is cut into work items of at most WALK_CHUNK entries, so that a determinant
// with a large coefficient (whose prefixes cover most of the lists) is
// spread over many warps.
constexpr int PLAN_ILP = 4;

__global__ void __launch_bounds__(SEL_WARPS * 32) k_walk_plan(WalkArgs A) {
  // shared: list maxima (n*n + n(n-1)/2), then the triangular decode table
  // t -> (lo, hi) of occupied-pair indices (bytes)
  extern __shared__ float s_max[];
  __shared__ int s_occ[SEL_WARPS][2][HCI_MAXORB];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nmax = A.n * A.n + A.n * (A.n - 1) / 2;
  unsigned char* s_tlo = reinterpret_cast<unsigned char*>(s_max + nmax);
  const int ntri = HCI_MAXORB * (HCI_MAXORB - 1) / 2;
  unsigned char* s_thi = s_tlo + ntri;
  for (int t = threadIdx.x; t < nmax; t += blockDim.x) s_max[t] = __double2float_ru(A.list_max[t]);
  for (int t = threadIdx.x; t < ntri; t += blockDim.x) {
    int lo, hi;
    tri_decode_dev(t, lo, hi);
    s_tlo[t] = (unsigned char)lo;
    s_thi[t] = (unsigned char)hi;
  }
  __syncthreads();
  int* occA = s_occ[w][0];
  int* occB = s_occ[w][1];
  const int Paa = A.na * (A.na - 1) / 2, Pbb = A.nb * (A.nb - 1) / 2, Pab = A.na * A.nb;
  const int P = Paa + Pbb + Pab;
  const int nn = A.n * A.n;
  const float epsf = __double2float_rd(A.eps1);
  unsigned long long walked = 0;
  while (true) {
    const int64_t i_l = next_dets(A);
    if (i_l < 0) break;
    const double absc_l = i_l < A.nV ? fabs(A.c[i_l]) : 0.0;
    unsigned go = __ballot_sync(0xffffffffu, i_l < A.nV && (A.accept_all || A.max_dbl * absc_l > A.eps1));
    while (go) {
      const int from = __ffs(go) - 1;
      go &= go - 1;
      const int64_t i = __shfl_sync(0xffffffffu, i_l, from);
      const double absc = __shfl_sync(0xffffffffu, absc_l, from);
      const float cf = __double2float_ru(absc);
      const ulonglong2 k = A.keys[i];
      __syncwarp();
      occ_list(k.x, A.n, occA);
      occ_list(k.y, A.n, occB);
      for (int base = 0; base < P; base += 32 * PLAN_ILP) {
        int code[PLAN_ILP], L[PLAN_ILP], hi[PLAN_ILP];
        const double* mag[PLAN_ILP];
#pragma unroll
        for (int u = 0; u < PLAN_ILP; ++u) {
          const int t = base + 32 * u + lane;
          int kind = 0, p = 0, q = 0, listid = 0;
          L[u] = hi[u] = 0;
          mag[u] = A.opp_mag;
          if (t < P) {
            int len;
            float first;
            if (t < Paa + Pbb) {
              const bool al = t < Paa;
              const int u2 = al ? t : t - Paa;
              const int* occ = al ? occA : occB;
              kind = al ? 0 : 1;
              p = occ[s_tlo[u2]]; q = occ[s_thi[u2]];
              listid = q * (q - 1) / 2 + p;
              first = s_max[nn + listid];
              mag[u] = A.same_mag + (int64_t)listid * A.Ls; len = A.Ls;
            } else {
              const int u2 = t - Paa - Pbb;
              p = occA[u2 / A.nb]; q = occB[u2 % A.nb]; kind = 2;
              listid = p * A.n + q;
              first = s_max[listid];
              mag[u] = A.opp_mag + (int64_t)listid * A.Lo; len = A.Lo;
            }
            if (A.accept_all) L[u] = hi[u] = len;
            else if (__fmul_ru(first, cf) > epsf) hi[u] = len;
          }
          code[u] = kind | (p << 2) | (q << 8) | (listid << 14);
        }
        // the searches side by side: entries [0, L) pass, [hi, len) fail
        while (true) {
          bool more = false;
#pragma unroll
          for (int u = 0; u < PLAN_ILP; ++u) more = more || L[u] < hi[u];
          if (!more) break;
          double v[PLAN_ILP];
#pragma unroll
          for (int u = 0; u < PLAN_ILP; ++u) v[u] = L[u] < hi[u] ? mag[u][(L[u] + hi[u]) >> 1] : 0.0;
#pragma unroll
          for (int u = 0; u < PLAN_ILP; ++u)
            if (L[u] < hi[u]) {
              const int mid = (L[u] + hi[u]) >> 1;
              if (v[u] * absc > A.eps1) L[u] = mid + 1;
              else hi[u] = mid;
            }
        }
#pragma unroll
        for (int u = 0; u < PLAN_ILP; ++u) {
          walked += L[u];
          // work items of at most WALK_CHUNK entries (det, kind|p|q|list, start, end)
          const int nit = (L[u] + WALK_CHUNK - 1) / WALK_CHUNK;
          if (!__any_sync(0xffffffffu, nit > 0)) continue;
          int incl = nit;
          for (int o = 1; o < 32; o <<= 1) {
            int t2 = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t2;
          }
          unsigned long long base_it = 0;
          if (lane == 31) base_it = atomicAdd(A.nitems, (unsigned long long)incl);
          base_it = __shfl_sync(0xffffffffu, base_it, 31);
          for (int j = 0; j < nit; ++j) {
            const unsigned long long idx = base_it + (incl - nit) + j;
            if ((int64_t)idx < A.item_cap)
              A.items[idx] = make_int4((int)i, code[u], j * WALK_CHUNK, min(L[u], (j + 1) * WALK_CHUNK));
          }
        }
      }
    }
  }
  for (int o = 16; o; o >>= 1) walked += __shfl_xor_sync(0xffffffffu, walked, o);
  if (lane == 0 && walked) atomicAdd(&A.walkstat[0], walked);
}

// Walk the planned list ranges: one warp per work item; every target whose
// orbitals are empty in the source determinant is emitted.  In perturbative
// mode the element is the list's magnitude with the sign kept beside the
// target and the determinant's two phases, one FP64 product per target.
__global__ void __launch_bounds__(SEL_WARPS * 32) k_walk_exec(WalkArgs A, int64_t nitems) {
  __shared__ EmitBuf s_emit[SEL_WARPS];
  const int lane = threadIdx.x & 31;
  EmitBuf& B = s_emit[threadIdx.x >> 5];
  int cnt = 0;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t it = warp; it < nitems; it += nwarps) {
    const int4 w = A.items[it];
    const ulonglong2 k = A.keys[w.x];
    const int sk = w.y & 3, sp = (w.y >> 2) & 63, sq = (w.y >> 8) & 63, sl = w.y >> 14;
    const uint16_t* tg = sk == 2 ? A.opp_tgt + (int64_t)sl * A.Lo : A.same_tgt + (int64_t)sl * A.Ls;
    const double* mg = sk == 2 ? A.opp_mag + (int64_t)sl * A.Lo : A.same_mag + (int64_t)sl * A.Ls;
    const double ci = A.vals ? A.c[w.x] : 0.0;
    for (int k0 = w.z; k0 < w.w; k0 += 32) {
      const int e = k0 + lane;
      bool emit = false;
      ulonglong2 key = k;
      double term = 0.0, elem = 0.0;
      if (e < w.w) {
        const uint16_t tt = tg[e];
        const int r = tt & 63, s2 = (tt >> 8) & 63;
        const uint64_t sa = sk == 1 ? k.y : k.x, sb = sk == 0 ? k.x : k.y;   // strings of p -> r and q -> s
        emit = !((sa >> r) & 1ull) && !((sb >> s2) & 1ull);
        if (emit) {
          const uint64_t ma = (1ull << sp) ^ (1ull << r), mb = (1ull << sq) ^ (1ull << s2);
          if (sk != 1) key.x ^= sk == 0 ? ma ^ mb : ma;
          if (sk != 0) key.y ^= sk == 1 ? ma ^ mb : mb;
          if (A.vals) {
            // signed <D_a|H|D_i> (same rule as the graph's elements), times c_i
            const int odd = bits_between(sa, sp, r) + bits_between(sk == 2 ? sb : sa ^ ma, sq, s2) + (tt >> 15);
            elem = flip_sign(mg[e], odd);
            term = elem * ci;
            emit = pt_keep(A, key, term);
          }
        }
      }
      warp_emit(emit, key, A.srcs ? elem : term, w.x, B, cnt, A);
    }
  }
  emit_flush(B, cnt, A);
}

// Upper bound, in FP32 rounded up, of |H_ai| of the single p->r (spin S) of
// a determinant D from the aufbau reference R: H = F_R + sum over the
// orbitals where D and R differ of +-(pr|kk)-(pk|kr) (same spin) or +-(pr|kk)
// (other spin), so |H| is at most |F_R| plus the absolute values of those few
// terms; the margins cover the rounding of both FP64 sums (at most 2n+1
// terms bounded by the loose bound).
__device__ __forceinline__ float single_tight(const WalkArgs& A, int spin, int p, int r, uint64_t s, uint64_t o) {
  const int n = A.n;
  const uint64_t ds = s ^ (spin == 0 ? A.ref_a : A.ref_b);
  const uint64_t dot = o ^ (spin == 0 ? A.ref_b : A.ref_a);
  const int64_t n3 = (int64_t)n * n * n;
  const float* js = A.single_f32 + ((int64_t)p * n + r) * n;
  const float* jo = js + n3;
  float t = A.single_f32[2 * n3 + ((int64_t)spin * n + p) * n + r];
  for (uint64_t x = ds; x; x &= x - 1) t = __fadd_ru(t, js[__ffsll((long long)x) - 1]);
  for (uint64_t x = dot; x; x &= x - 1) t = __fadd_ru(t, jo[__ffsll((long long)x) - 1]);
  t = __fadd_ru(t, __fmul_ru(2e-13f, __double2float_ru(A.single_bound[p * n + r])));
  return __fmul_ru(t, 1.000002f);
}

// Singles.  FP64 operations bound this kernel (64 cycles of a sub-partition
// each, whatever the active lanes), so they are left to the few singles that
// need them, 32 at a time:
//  1. 32 determinants from the queue; each one's prefix of the singles sorted
//     by their determinant-independent bound (FP32, bound and coefficient
//     rounded up); the prefix's singles that are occupied -> empty are queued;
//  2. queued singles against the determinant's own bound (single_tight);
//  3. the rest in FP64: in selection exactly, in the summation order of the
//     textbook rule (k ascending, same spin then opposite spin per k), so
//     that decisions are bit-identical to it; in perturbative mode from the
//     aufbau value plus the orbitals where the strings differ.
// The queues (per warp) run on from one determinant to the next.  (44e,44o),
// 4.1e5 determinants at eps1 = 1.5e-4: 914 us with one determinant per warp
// and FP64 bounds, 439 us so.
constexpr int SQ_CAP = 64;

__global__ void __launch_bounds__(SEL_WARPS * 32) k_singles(WalkArgs A) {
  extern __shared__ float s_bf[];              // n*n bounds, then the n*n packed singles
  __shared__ EmitBuf s_emit[SEL_WARPS];
  __shared__ uint64_t s_q1[SEL_WARPS][SQ_CAP], s_q2[SEL_WARPS][SQ_CAP];   // determinant << 20 | spin << 16 | r << 8 | p
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int n = A.n, nn = n * n;
  uint16_t* s_pr = reinterpret_cast<uint16_t*>(s_bf + nn);
  for (int t = threadIdx.x; t < nn; t += blockDim.x) {
    s_bf[t] = A.single_bf[t];
    s_pr[t] = A.single_pr[t];
  }
  __syncthreads();
  EmitBuf& B = s_emit[w];
  uint64_t* q1 = s_q1[w];
  uint64_t* q2 = s_q2[w];
  int cnt = 0, n1 = 0, n2 = 0;
  unsigned long long exact = 0;
  const float epsf = __double2float_rd(A.eps1);

  // the first m <= 32 entries of q2 evaluated
  auto evaluate = [&](int m) {
    __syncwarp();
    bool emit = false;
    ulonglong2 key = make_ulonglong2(0, 0);
    double term = 0.0, elem = 0.0;
    int64_t i = 0;
    if (lane < m) {
      const uint64_t q = q2[lane];
      const int p = (int)(q & 63), r = (int)((q >> 8) & 63), spin = (int)((q >> 16) & 1);
      i = (int64_t)(q >> 20);
      key = A.keys[i];
      const uint64_t s = spin == 0 ? key.x : key.y, o = spin == 0 ? key.y : key.x;
      const double* js = A.jk_same + ((int64_t)p * n + r) * n;
      const double* jo = A.j_opp + ((int64_t)p * n + r) * n;
      double v;
      if (A.vals) {
        const uint64_t rs = spin == 0 ? A.ref_a : A.ref_b, ro = spin == 0 ? A.ref_b : A.ref_a;
        v = A.f_ref[((int64_t)spin * n + p) * n + r];
        for (uint64_t mm = s & ~rs; mm; mm &= mm - 1) v += js[__ffsll((long long)mm) - 1];
        for (uint64_t mm = rs & ~s; mm; mm &= mm - 1) v -= js[__ffsll((long long)mm) - 1];
        for (uint64_t mm = o & ~ro; mm; mm &= mm - 1) v += jo[__ffsll((long long)mm) - 1];
        for (uint64_t mm = ro & ~o; mm; mm &= mm - 1) v -= jo[__ffsll((long long)mm) - 1];
        elem = flip_sign(v, bits_between(s, p, r));
        term = elem * A.c[i];
        emit = true;
      } else {
        v = A.h[p * n + r];
#pragma unroll 4
        for (int x = 0; x < n; ++x) {
          if ((s >> x) & 1ull) v += js[x];
          if ((o >> x) & 1ull) v += jo[x];
        }
        emit = fabs(v) * fabs(A.c[i]) > A.eps1;
      }
      const uint64_t flip = (1ull << p) ^ (1ull << r);
      if (spin == 0) key.x ^= flip;
      else key.y ^= flip;
      if (A.vals) emit = pt_keep(A, key, term);
    }
    if (!A.vals) exact += m;
    warp_emit(emit, key, A.srcs ? elem : term, (int)i, B, cnt, A);
    // the entries behind move to the front
    __syncwarp();
    const uint64_t q = lane + m < n2 ? q2[lane + m] : 0;
    __syncwarp();
    if (lane + m < n2) q2[lane] = q;
    n2 -= m;
    __syncwarp();
  };
  // the first m <= 32 entries of q1 against their own bounds
  auto screen = [&](int m) {
    __syncwarp();
    bool pass = false;
    uint64_t q = 0;
    if (lane < m) {
      q = q1[lane];
      pass = true;
      if (!A.accept_all) {
        const int p = (int)(q & 63), r = (int)((q >> 8) & 63), spin = (int)((q >> 16) & 1);
        const int64_t i = (int64_t)(q >> 20);
        const ulonglong2 k = A.keys[i];
        const float t = single_tight(A, spin, p, r, spin == 0 ? k.x : k.y, spin == 0 ? k.y : k.x);
        pass = __fmul_ru(t, __double2float_ru(fabs(A.c[i]))) > epsf;
      }
    }
    const unsigned b = __ballot_sync(0xffffffffu, pass);
    if (pass) q2[n2 + __popc(b & lt)] = q;
    n2 += __popc(b);
    if (n2 >= 32) evaluate(32);
    __syncwarp();
    const uint64_t rest = lane + m < n1 ? q1[lane + m] : 0;
    __syncwarp();
    if (lane + m < n1) q1[lane] = rest;
    n1 -= m;
    __syncwarp();
  };

  while (true) {
    const int64_t i_l = next_dets(A);
    if (i_l < 0) break;
    const bool in = i_l < A.nV;
    int len = 0;                                 // singles of this lane's determinant to look at
    if (in) {
      if (A.accept_all) {
        len = nn;
      } else {
        const float cf = __double2float_ru(fabs(A.c[i_l]));
        int lo = 0, hi = nn;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (__fmul_ru(s_bf[mid], cf) > epsf) lo = mid + 1;
          else hi = mid;
        }
        len = lo;
      }
    }
    unsigned go = __ballot_sync(0xffffffffu, len > 0);
    while (go) {
      const int from = __ffs(go) - 1;
      go &= go - 1;
      const uint64_t i = (uint64_t)__shfl_sync(0xffffffffu, i_l, from);
      const int L = __shfl_sync(0xffffffffu, len, from);
      const ulonglong2 k = A.keys[i];
      const float cf = __double2float_ru(fabs(A.c[i]));
      const float da = (float)__popcll(k.x ^ A.ref_a), db = (float)__popcll(k.y ^ A.ref_b);
      for (int e0 = 0; e0 < L; e0 += 32) {
        const int e = e0 + lane;
        const int pr = e < L ? s_pr[e] : 0;
        const float4 mx = e < L ? A.single_max[e] : make_float4(0.f, 0.f, 0.f, 0.f);
        const int p = pr & 63, r = pr >> 8;
#pragma unroll
        for (int spin = 0; spin < 2; ++spin) {
          const uint64_t s = spin == 0 ? k.x : k.y;
          bool ok = e < L && ((s >> p) & 1ull) && !((s >> r) & 1ull);
          if (!A.accept_all) {
            const float t = __fmaf_ru(spin == 0 ? da : db, mx.z, __fmaf_ru(spin == 0 ? db : da, mx.w, spin == 0 ? mx.x : mx.y));
            ok = ok && !(__fmul_ru(t, cf) <= epsf);   // not a number: 0 changed orbitals of a term beyond FP32
          }
          const unsigned b = __ballot_sync(0xffffffffu, ok);
          if (A.accept_all && !A.vals) {
            ulonglong2 key = k;
            const uint64_t flip = (1ull << p) ^ (1ull << r);
            if (spin == 0) key.x ^= flip;
            else key.y ^= flip;
            warp_emit(ok, key, 0.0, (int)i, B, cnt, A);
          } else if (b) {
            if (ok) q1[n1 + __popc(b & lt)] = (i << 20) | ((uint64_t)spin << 16) | (uint64_t)pr;
            n1 += __popc(b);
            if (n1 >= 32) screen(32);
          }
        }
      }
    }
  }
  if (n1 > 0) screen(n1);
  if (n2 > 0) evaluate(n2);
  emit_flush(B, cnt, A);
  if (lane == 0 && exact) atomicAdd(&A.walkstat[1], exact);
}

__device__ __forceinline__ bool key_less(ulonglong2 a, ulonglong2 b) {
  return a.x < b.x || (a.x == b.x && a.y < b.y);
}

// number of elements of sorted arr[0,n) strictly less than key
__device__ __forceinline__ int64_t lower_bound(const ulonglong2* __restrict__ arr, int64_t n, ulonglong2 key) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (key_less(arr[mid], key)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// flag = first of its run in the sorted candidates and not already in V
// c[m + t] = c[t] with the alpha and beta strings exchanged
__global__ void k_flip_append(ulonglong2* __restrict__ c, int64_t m) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    const ulonglong2 k = c[t];
    c[m + t] = make_ulonglong2(k.y, k.x);
  }
}

__global__ void k_flag_new(const ulonglong2* __restrict__ cand, int64_t m, const ulonglong2* __restrict__ V,
                           int64_t nV, int64_t* __restrict__ flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 k = cand[i];
    int64_t f = 0;
    if (i == 0 || !key_eq(k, cand[i - 1])) {
      int64_t pos = lower_bound(V, nV, k);
      f = (pos < nV && key_eq(V[pos], k)) ? 0 : 1;
    }
    flag[i] = f;
  }
}

__global__ void k_compact(const ulonglong2* __restrict__ cand, int64_t m, const int64_t* __restrict__ flag,
                          const int64_t* __restrict__ pos, ulonglong2* __restrict__ out, int64_t cap) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    if (flag[i] && pos[i] < cap) out[pos[i]] = cand[i];
  }
}

__global__ void k_merge_old(const ulonglong2* __restrict__ V, const double* __restrict__ c, int64_t nV,
                            const ulonglong2* __restrict__ N, int64_t nN, ulonglong2* __restrict__ out,
                            double* __restrict__ outc) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nV; i += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 k = V[i];
    int64_t pos = i + lower_bound(N, nN, k);
    out[pos] = k;
    if (outc) outc[pos] = c ? c[i] : 0.0;
  }
}

__global__ void k_merge_new(const ulonglong2* __restrict__ V, int64_t nV, const ulonglong2* __restrict__ N,
                            int64_t nN, ulonglong2* __restrict__ out, double* __restrict__ outc) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nN; j += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 k = N[j];
    int64_t pos = j + lower_bound(V, nV, k);
    out[pos] = k;
    if (outc) outc[pos] = 0.0;
  }
}

}  // namespace

static hci_status run_walk(hci_ctx* ctx, WalkArgs& A, int64_t* total) {
  HCI_TRY(ensure_buf(ctx, ctx->s_walkstat, 64));
  A.walkstat = bp<unsigned long long>(ctx->s_walkstat);
  A.nitems = A.walkstat + 2;
  HCI_CUDA(ctx, cudaMemsetAsync(A.walkstat, 0, 16, ctx->st));
  prof_tic(ctx, HCI_PH_WALK);
  HCI_CUDA(ctx, cudaMemsetAsync(A.counter, 0, 16, ctx->st));
  const int grid = ctx->nsm * 8;
  const size_t smw = (size_t)(A.n * A.n + A.n * (A.n - 1) / 2) * 4 + HCI_MAXORB * (HCI_MAXORB - 1);
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_walk_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
  for (int attempt = 0; attempt < 2; ++attempt) {
    HCI_TRY(ensure_buf(ctx, ctx->s_items, (size_t)(ctx->s_items.bytes > 0 ? ctx->s_items.bytes : (1 << 20) * 16)));
    A.items = bp<int4>(ctx->s_items);
    A.item_cap = (int64_t)(ctx->s_items.bytes / 16);
    HCI_CUDA(ctx, cudaMemsetAsync(A.counter + 1, 0, 8, ctx->st));
    HCI_CUDA(ctx, cudaMemsetAsync(A.nitems, 0, 8, ctx->st));
    HCI_LAUNCH(k_walk_plan, grid, SEL_WARPS * 32, smw, ctx->st)(A);
    HCI_CUDA(ctx, cudaGetLastError());
    unsigned long long ni = 0;
    HCI_CUDA(ctx, cudaMemcpyAsync(&ni, A.nitems, 8, cudaMemcpyDeviceToHost, ctx->st));
    HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
    if ((int64_t)ni <= A.item_cap) {
      if (ni > 0) HCI_LAUNCH(k_walk_exec, grid, SEL_WARPS * 32, 0, ctx->st)(A, (int64_t)ni);
      break;
    }
    HCI_TRY(ensure_buf(ctx, ctx->s_items, (size_t)(ni + ni / 8 + 1024) * 16));
  }
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_WALK);
  prof_tic(ctx, HCI_PH_SINGLES);
  HCI_CUDA(ctx, cudaMemsetAsync(A.counter + 1, 0, 8, ctx->st));
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_singles, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024));
  HCI_LAUNCH(k_singles, grid, SEL_WARPS * 32, (size_t)A.n * A.n * 6, ctx->st)(A);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_SINGLES);
  unsigned long long cnt = 0, ws[2] = {0, 0};
  HCI_CUDA(ctx, cudaMemcpyAsync(&cnt, A.counter, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaMemcpyAsync(ws, A.walkstat, 16, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  ctx->st_counts[HCI_ST_WALK_ENTRIES] += (int64_t)ws[0];
  ctx->st_counts[HCI_ST_SINGLES_EXACT] += (int64_t)ws[1];
  *total = (int64_t)cnt;
  return HCI_OK;
}

extern "C" hci_status hci_select(hci_ctx* ctx, double eps1, const uint64_t* keys, const double* c, int64_t nV,
                                 uint64_t* new_keys, int64_t cap, int64_t* n_new) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_select: null context");
  if (!n_new) return hci_fail(ctx, HCI_ERR_INVALID, "hci_select: n_new is NULL");
  *n_new = 0;
  if (nV < 0 || cap < 0) return hci_fail(ctx, HCI_ERR_INVALID, "hci_select: negative size");
  if (nV > 0 && (!keys || !c)) return hci_fail(ctx, HCI_ERR_INVALID, "hci_select: null keys or c");
  if (cap > 0 && !new_keys) return hci_fail(ctx, HCI_ERR_INVALID, "hci_select: null new_keys");
  if (nV == 0) return HCI_OK;
  HCI_TRY(hci_build_lists(ctx));
  int ok = 0;
  HCI_TRY(check_sorted(ctx, keys, nV, &ok));
  if (!ok) return hci_fail(ctx, HCI_ERR_INVALID, "hci_select: keys are not strictly ascending");
  Lists& L = ctx->lists;
  WalkArgs A;
  A.n = ctx->n; A.na = ctx->na; A.nb = ctx->nb;
  A.keys = reinterpret_cast<const ulonglong2*>(keys);
  A.c = c; A.nV = nV; A.eps1 = eps1; A.accept_all = eps1 <= 0.0 ? 1 : 0;
  A.opp_mag = bp<double>(L.opp_mag); A.opp_tgt = bp<uint16_t>(L.opp_tgt); A.Lo = L.len_opp;
  A.same_mag = bp<double>(L.same_mag); A.same_tgt = bp<uint16_t>(L.same_tgt); A.Ls = L.len_same;
  A.max_dbl = L.max_opp > L.max_same ? L.max_opp : L.max_same;
  A.h = bp<double>(ctx->h); A.jk_same = bp<double>(ctx->jk_same); A.j_opp = bp<double>(ctx->j_opp);
  A.single_bound = bp<double>(L.single_bound);
  A.single_pr = bp<uint16_t>(L.single_pr); A.single_bf = bp<float>(L.single_bf);
  A.single_f32 = bp<float>(L.single_f32); A.single_max = bp<float4>(L.single_max);
  A.list_max = bp<double>(L.list_max);
  A.f_ref = bp<double>(L.f_ref);
  A.ref_a = ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull);
  A.ref_b = ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull);
  A.vals = nullptr; A.srcs = nullptr; A.npart = 1; A.part = 0;
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  A.counter = bp<unsigned long long>(ctx->s_counter);
  // candidate buffer: grow and rerun when the first guess overflows
  int64_t guess = ctx->s_cand.bytes / 16;
  if (guess < (int64_t)1 << 16) guess = (int64_t)1 << 16;
  HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)guess * 16));
  A.out = bp<ulonglong2>(ctx->s_cand);
  A.cap = (int64_t)(ctx->s_cand.bytes / 16);
  int64_t m = 0;
  HCI_TRY(run_walk(ctx, A, &m));
  if (m > A.cap) {
    HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)(m + m / 8 + 1024) * 16));
    A.out = bp<ulonglong2>(ctx->s_cand);
    A.cap = (int64_t)(ctx->s_cand.bytes / 16);
    int64_t m2 = 0;
    HCI_TRY(run_walk(ctx, A, &m2));
    if (m2 != m) return hci_fail(ctx, HCI_ERR_CUDA, "hci_select: candidate count changed between runs");
  }
  if (ctx->spin_parity != 0 && m > 0) {
    // spin parity: every selected determinant brings its spin-flip partner
    HCI_TRY(ensure_buf(ctx, ctx->s_cand2, (size_t)2 * m * 16));
    HCI_CUDA(ctx, cudaMemcpyAsync(ctx->s_cand2.p, ctx->s_cand.p, (size_t)m * 16, cudaMemcpyDeviceToDevice, ctx->st));
    HCI_LAUNCH(k_flip_append, grid_for(m, 256), 256, 0, ctx->st)(bp<ulonglong2>(ctx->s_cand2), m);
    HCI_CUDA(ctx, cudaGetLastError());
    std::swap(ctx->s_cand, ctx->s_cand2);
    m *= 2;
  }
  ctx->last_candidates = m;
  ctx->st_counts[HCI_ST_SELECT_CALLS] += 1;
  ctx->st_counts[HCI_ST_SELECT_SOURCES] += nV;
  ctx->st_counts[HCI_ST_CANDIDATES] += m;
  if (m == 0) return HCI_OK;
  prof_tic(ctx, HCI_PH_DEDUP);
  HCI_TRY(ensure_buf(ctx, ctx->s_cand2, (size_t)m * 16));
  HCI_TRY(sort_keys(ctx, bp<uint64_t>(ctx->s_cand), bp<uint64_t>(ctx->s_cand2), m, ctx->n, ctx->n));
  HCI_TRY(ensure_buf(ctx, ctx->s_flags, (size_t)(2 * m + 1) * 8));
  int64_t* flag = bp<int64_t>(ctx->s_flags);
  int64_t* pos = flag + m;
  int64_t* total = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 16);
  HCI_LAUNCH(k_flag_new, grid_for(m, 256), 256, 0, ctx->st)(bp<ulonglong2>(ctx->s_cand), m,
                                                    reinterpret_cast<const ulonglong2*>(keys), nV, flag);
  HCI_CUDA(ctx, cudaGetLastError());
  HCI_TRY(scan_i64(ctx, flag, pos, m, total));
  prof_toc(ctx, HCI_PH_DEDUP);
  int64_t cnt = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&cnt, total, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  *n_new = cnt;
  if (cnt > cap)
    return hci_fail(ctx, HCI_ERR_CAPACITY, "hci_select: %lld new determinants exceed cap %lld", (long long)cnt,
                    (long long)cap);
  HCI_LAUNCH(k_compact, grid_for(m, 256), 256, 0, ctx->st)(bp<ulonglong2>(ctx->s_cand), m, flag, pos,
                                                   reinterpret_cast<ulonglong2*>(new_keys), cap);
  HCI_CUDA(ctx, cudaGetLastError());
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  return HCI_OK;
}

extern "C" hci_status hci_merge(hci_ctx* ctx, const uint64_t* keys, const double* c, int64_t nV,
                                const uint64_t* new_keys, int64_t n_new, uint64_t* out_keys, double* out_c) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_merge: null context");
  if (nV < 0 || n_new < 0) return hci_fail(ctx, HCI_ERR_INVALID, "hci_merge: negative size");
  if ((nV + n_new) > 0 && !out_keys) return hci_fail(ctx, HCI_ERR_INVALID, "hci_merge: null out_keys");
  const ulonglong2* V = reinterpret_cast<const ulonglong2*>(keys);
  const ulonglong2* N = reinterpret_cast<const ulonglong2*>(new_keys);
  ulonglong2* O = reinterpret_cast<ulonglong2*>(out_keys);
  prof_tic(ctx, HCI_PH_MERGE);
  if (nV > 0)
    HCI_LAUNCH(k_merge_old, grid_for(nV, 256), 256, 0, ctx->st)(V, c, nV, N, n_new, O, out_c);
  if (n_new > 0)
    HCI_LAUNCH(k_merge_new, grid_for(n_new, 256), 256, 0, ctx->st)(V, nV, N, n_new, O, out_c);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_MERGE);
  return HCI_OK;
}

// ---------------------------------------------------------------------------
// Second-order Epstein-Nesbet correction with screening (Sec. II.B,
// Eq. pt_hci): the walk and the singles emit every target D_a with its term
// H_ai c_i when |H_ai c_i| > eps2; the (target, term) pairs are grouped by
// target, targets in V are dropped, and each remaining target contributes
// (sum of its terms)^2 / (E0 - H_aa).  The targets are processed in hash
// classes so that at most max_pairs pairs are held at once.
// ---------------------------------------------------------------------------
namespace {

// Aufbau reference R for diagonal elements by differences, over spin
// orbitals k (alpha 0..n-1, beta n..2n-1): g_kl = (kk|ll) - [same spin] (kl|lk),
// F_k = h_kk + sum_{l in R, l != k} g_kl, E_R = e_core + sum_{k in R} h_kk +
// sum_{k<l in R} g_kl.  A spin orbital k where a determinant differs from R
// is emptied (d_k = -1) when R holds it, else filled (d_k = +1), so the
// signs go into the table: out = [E_R, d_k F_k (2n), d_k d_l g_kl (2n x 2n)].
// One block per k; k_pt2_eref adds E_R.
__global__ void k_pt2_ref(int n, const double* __restrict__ h, const double* __restrict__ eri, uint64_t ra, uint64_t rb,
                          double* __restrict__ out) {
  extern __shared__ double s_g[];
  const int m = 2 * n, k = blockIdx.x, p = k % n;
  auto occ = [&](int l) { return (l < n ? (ra >> l) : (rb >> (l - n))) & 1ull; };
  const double dk = occ(k) ? -1.0 : 1.0;
  for (int l = threadIdx.x; l < m; l += blockDim.x) {
    const int q = l % n;
    double v = eri[(((int64_t)p * n + p) * n + q) * n + q];
    if ((k < n) == (l < n)) v -= eri[(((int64_t)p * n + q) * n + q) * n + p];
    if (k == l) v = 0.0;
    s_g[l] = v;
    out[1 + m + k * m + l] = dk * (occ(l) ? -v : v);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double f = h[p * n + p];
    for (int l = 0; l < m; ++l)
      if (occ(l)) f += s_g[l];
    out[1 + k] = dk * f;
  }
}
// E_R = e_core + sum_{k in R} (h_kk + F_k) / 2
__global__ void k_pt2_eref(int n, const double* __restrict__ h, double ecore, uint64_t ra, uint64_t rb,
                           double* __restrict__ out) {
  const int lane = threadIdx.x;
  double e = 0.0;
  for (int k = lane; k < 2 * n; k += 32)
    if ((k < n ? (ra >> k) : (rb >> (k - n))) & 1ull) e += h[(k % n) * n + (k % n)] - out[1 + k];
  for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0) out[0] = ecore + 0.5 * e;
}

// H_aa = E_R + sum_k d_k F_k + sum_{k<l} d_k d_l g_kl over the spin orbitals
// where D_a differs from R
__device__ __forceinline__ double pt2_diag(const double* s_ref, int n, ulonglong2 key, uint64_t ra, uint64_t rb) {
  const int m = 2 * n;
  const double* F = s_ref + 1;
  const double* g = s_ref + 1 + m;
  const uint64_t da = key.x ^ ra, db = key.y ^ rb;
  double e = s_ref[0];
  for (uint64_t x = da; x; x &= x - 1) {
    const int k = __ffsll((long long)x) - 1;
    const double* gk = g + k * m;
    e += F[k];
    for (uint64_t y = x & (x - 1); y; y &= y - 1) e += gk[__ffsll((long long)y) - 1];
    for (uint64_t y = db; y; y &= y - 1) e += gk[n + __ffsll((long long)y) - 1];
  }
  for (uint64_t x = db; x; x &= x - 1) {
    const int k = __ffsll((long long)x) - 1;
    const double* gk = g + (n + k) * m + n;
    e += F[n + k];
    for (uint64_t y = x & (x - 1); y; y &= y - 1) e += gk[__ffsll((long long)y) - 1];
  }
  return e;
}

// Hash table of the determinants of V (their positions; -1 empty), at least
// twice as many slots, linear probing: one or two look-ups tell whether a
// target belongs to V, where a binary search takes log2 nV dependent ones.
__global__ void k_space_insert(const ulonglong2* __restrict__ V, int64_t nV, int32_t* __restrict__ tab, uint64_t mask) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nV; i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t h = key_mix(V[i]) & mask;
    for (uint64_t probe = 0; probe <= mask; ++probe, h = (h + 1) & mask)
      if (atomicCAS(&tab[h], -1, (int32_t)i) == -1) break;
  }
}
__device__ __forceinline__ bool in_space(const ulonglong2* __restrict__ V, const int32_t* __restrict__ tab,
                                         uint64_t mask, ulonglong2 key) {
  uint64_t h = key_mix(key) & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe, h = (h + 1) & mask) {
    const int32_t j = tab[h];
    if (j < 0) return false;
    if (key_eq(V[j], key)) return true;
  }
  return false;
}

// list = the first pairs of the targets outside V (in any order; *count of
// them); with dpair, 0 on every pair of a target in V
__global__ void __launch_bounds__(256) k_pt2_targets(const ulonglong2* __restrict__ t, int64_t m, uint64_t gmask,
                                                     const ulonglong2* __restrict__ V, const int32_t* __restrict__ tab,
                                                     uint64_t tmask, int64_t* __restrict__ list,
                                                     unsigned long long* __restrict__ count,
                                                     double* __restrict__ dpair) {
  __shared__ int s_n[8];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t i0 = (int64_t)blockIdx.x * 256; i0 < m; i0 += (int64_t)gridDim.x * 256) {
    const int64_t i = i0 + threadIdx.x;
    bool ext = false;
    if (i < m) {
      const ulonglong2 key = t[i];
      if (first_of_key(t, i, key, gmask)) {
        ext = !in_space(V, tab, tmask, key);
        if (!ext && dpair)
          for (int64_t e = i; e < m; e = next_of_key(t, e, m, key, gmask)) dpair[e] = 0.0;
      }
    }
    const unsigned b = __ballot_sync(0xffffffffu, ext);
    if (lane == 0) s_n[w] = __popc(b);
    __syncthreads();
    if (threadIdx.x == 0) {
      int tot = 0;
      for (int q = 0; q < 8; ++q) {
        const int c = s_n[q];
        s_n[q] = tot;
        tot += c;
      }
      s_base = tot ? atomicAdd(count, (unsigned long long)tot) : 0ull;
    }
    __syncthreads();
    if (ext) list[s_base + s_n[w] + __popc(b & ((1u << lane) - 1u))] = i;
    __syncthreads();
  }
}

// One listed target per thread: its terms summed, sum^2 / (e0 - H_aa) added
// to the block's part_e, and with dpair the first-order coefficient d_a on
// every pair of the target.  The list's order and that of a target's pairs
// come from atomic counters, so E2 is a sum of the same terms in an order that
// differs from run to run.  Bound by FP64
// issue (about 55 operations per target, most of them H_aa's), so the targets
// are listed first: taken in place, where only the first pair of a run works,
// 2 to 3 lanes of 4 idle through all of them.
__global__ void __launch_bounds__(256) k_pt2_terms(const ulonglong2* __restrict__ t, const double* __restrict__ v,
                                                   int64_t m, uint64_t gmask, const int64_t* __restrict__ list,
                                                   const unsigned long long* __restrict__ count, int n,
                                                   const double* __restrict__ ref, uint64_t ra, uint64_t rb, double e0,
                                                   double* __restrict__ part_e, double* __restrict__ dpair,
                                                   const double* __restrict__ cvec, const int32_t* __restrict__ src) {
  extern __shared__ double s_ref[];
  __shared__ double red_e[8];
  const int nref = 1 + 2 * n + 4 * n * n;
  for (int u = threadIdx.x; u < nref; u += blockDim.x) s_ref[u] = ref[u];
  __syncthreads();
  double esum = 0.0;
  const int64_t nt = (int64_t)*count;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nt; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = list[q];
    const ulonglong2 key = t[i];
    double num = 0.0;
    for (int64_t e = i; e < m; e = next_of_key(t, e, m, key, gmask)) num += src ? v[e] * cvec[src[e]] : v[e];
    const double da = num / (e0 - pt2_diag(s_ref, n, key, ra, rb));
    esum = fma(num, da, esum);
    if (dpair)
      for (int64_t e = i; e < m; e = next_of_key(t, e, m, key, gmask)) dpair[e] = da;
  }
  for (int o = 16; o; o >>= 1) esum += __shfl_xor_sync(0xffffffffu, esum, o);
  if ((threadIdx.x & 31) == 0) red_e[threadIdx.x >> 5] = esum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double e = 0.0;
    for (int w = 0; w < 8; ++w) e += red_e[w];
    part_e[blockIdx.x] = e;
  }
}

__global__ void k_pt2_total(const double* __restrict__ part_e, int np, double* __restrict__ out) {
  double e = 0.0;
  for (int b = threadIdx.x; b < np; b += 32) e += part_e[b];
  for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (threadIdx.x == 0) *out = e;
}

// dE2/dc_i = 2 sum over the screened pairs of d_a H_ai (the pairs fixed)
__global__ void k_pt2_grad(const int32_t* __restrict__ src, const double* __restrict__ elem,
                           const double* __restrict__ d, int64_t m, double* __restrict__ g) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
    if (d[j] != 0.0) atomicAdd(&g[src[j]], 2.0 * d[j] * elem[j]);
}

constexpr int PT2_SUM_BLOCKS = 1024;

// part[b] = sum of a[] over block b's contiguous slice, in order
__global__ void k_sum_slices_d(const double* __restrict__ a, int64_t m, double* __restrict__ part) {
  __shared__ double red[256];
  const int64_t per = (m + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * per, hi = lo + per < m ? lo + per : m;
  double s = 0.0;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) s += a[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_sum_parts_d(const double* __restrict__ part, int np, double* __restrict__ out) {
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int b = 0; b < np; ++b) s += part[b];
    *out = s;
  }
}

}  // namespace

// Walk arguments of the perturbative modes: sources keys/c (nV of them),
// terms kept when |H_ai c_i| > eps (every single and double when eps < 0).
static hci_status pt_walk_args(hci_ctx* ctx, WalkArgs& A, const uint64_t* keys, const double* c, int64_t nV,
                               double eps) {
  Lists& L = ctx->lists;
  A = WalkArgs{};
  A.n = ctx->n; A.na = ctx->na; A.nb = ctx->nb;
  A.keys = reinterpret_cast<const ulonglong2*>(keys);
  A.c = c; A.nV = nV; A.eps1 = eps; A.accept_all = eps <= 0.0 ? 1 : 0;
  A.opp_mag = bp<double>(L.opp_mag); A.opp_tgt = bp<uint16_t>(L.opp_tgt); A.Lo = L.len_opp;
  A.same_mag = bp<double>(L.same_mag); A.same_tgt = bp<uint16_t>(L.same_tgt); A.Ls = L.len_same;
  A.max_dbl = L.max_opp > L.max_same ? L.max_opp : L.max_same;
  A.h = bp<double>(ctx->h); A.jk_same = bp<double>(ctx->jk_same); A.j_opp = bp<double>(ctx->j_opp);
  A.single_bound = bp<double>(L.single_bound);
  A.single_pr = bp<uint16_t>(L.single_pr); A.single_bf = bp<float>(L.single_bf);
  A.single_f32 = bp<float>(L.single_f32); A.single_max = bp<float4>(L.single_max);
  A.list_max = bp<double>(L.list_max);
  A.f_ref = bp<double>(L.f_ref);
  A.ref_a = ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull);
  A.ref_b = ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull);
  A.srcs = nullptr;
  A.vals = nullptr;
  A.npart = 1;
  A.part = 0;
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  A.counter = bp<unsigned long long>(ctx->s_counter);
  return HCI_OK;
}

extern "C" hci_status hci_pt2(hci_ctx* ctx, double eps2, const uint64_t* keys, const double* c, int64_t nV,
                              double e0, int64_t max_pairs, double* e2, int64_t* n_ext, double* rdm1_dd,
                              double* rdm2_dd, double* rdm1_dc, double* rdm2_dc, double* grad_c) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_pt2: null context");
  if (!e2) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: e2 is NULL");
  *e2 = 0.0;
  if (n_ext) *n_ext = 0;
  if (nV < 0 || max_pairs < 0) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: negative size");
  if (nV > 0 && (!keys || !c)) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: null keys or c");
  const int nrdm = (rdm1_dd != nullptr) + (rdm2_dd != nullptr) + (rdm1_dc != nullptr) + (rdm2_dc != nullptr);
  if (nrdm != 0 && nrdm != 4) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: give all four density matrices or none");
  const bool want_rdm = nrdm == 4;
  const bool want_src = want_rdm || grad_c != nullptr;
  if (grad_c && nV > 0) HCI_CUDA(ctx, cudaMemsetAsync(grad_c, 0, (size_t)nV * 8, ctx->st));
  if (want_rdm) {
    const size_t n2 = (size_t)ctx->n * ctx->n;
    HCI_CUDA(ctx, cudaMemsetAsync(rdm1_dd, 0, n2 * 8, ctx->st));
    HCI_CUDA(ctx, cudaMemsetAsync(rdm2_dd, 0, n2 * n2 * 8, ctx->st));
    HCI_CUDA(ctx, cudaMemsetAsync(rdm1_dc, 0, n2 * 8, ctx->st));
    HCI_CUDA(ctx, cudaMemsetAsync(rdm2_dc, 0, n2 * n2 * 8, ctx->st));
    HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  }
  if (nV == 0) return HCI_OK;
  HCI_TRY(hci_build_lists(ctx));
  int ok = 0;
  HCI_TRY(check_sorted(ctx, keys, nV, &ok));
  if (!ok) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: keys are not strictly ascending");
  cudaStream_t st = ctx->st;
  const int n = ctx->n;
  WalkArgs A;
  HCI_TRY(pt_walk_args(ctx, A, keys, c, nV, eps2));
  if (want_rdm) HCI_TRY(pt2_rdm_begin(ctx));
  // aufbau reference of the diagonal elements
  const size_t nref = 1 + 2 * (size_t)n + 4 * (size_t)n * n;
  HCI_TRY(ensure_buf(ctx, ctx->p2_ref, nref * 8 + (PT2_SUM_BLOCKS + 2) * 8));
  double* ref = bp<double>(ctx->p2_ref);
  HCI_LAUNCH(k_pt2_ref, 2 * n, 64, (size_t)2 * n * 8, st)(n, bp<double>(ctx->h), bp<double>(ctx->eri), A.ref_a, A.ref_b,
                                                         ref);
  HCI_LAUNCH(k_pt2_eref, 1, 32, 0, st)(n, bp<double>(ctx->h), ctx->ecore, A.ref_a, A.ref_b, ref);
  HCI_CUDA(ctx, cudaGetLastError());
  // hash table of V
  uint64_t tsize = 1024;
  while (tsize < 2 * (uint64_t)nV) tsize <<= 1;
  HCI_TRY(ensure_buf(ctx, ctx->p2_tab, (size_t)tsize * 4));
  HCI_CUDA(ctx, cudaMemsetAsync(ctx->p2_tab.p, 0xFF, (size_t)tsize * 4, st));
  HCI_LAUNCH(k_space_insert, grid_for(nV, 256), 256, 0, st)(A.keys, nV, bp<int32_t>(ctx->p2_tab), tsize - 1);
  HCI_CUDA(ctx, cudaGetLastError());
  const int64_t per = max_pairs > 0 ? max_pairs : ((int64_t)1 << 28);
  double acc = 0.0;
  int64_t next_total = 0;
  // one hash class of targets: walk into the pair buffer (walked again with
  // a larger buffer if it was too small), sort, reduce
  auto run_class = [&](int npart, int pc, int64_t* m_out, bool reduce) -> hci_status {
    A.npart = npart;
    A.part = pc;
    int64_t m = 0;
    for (int attempt = 0; attempt < 2; ++attempt) {
      A.out = bp<ulonglong2>(ctx->s_cand);
      A.vals = bp<double>(ctx->p2_vals);
      A.cap = (int64_t)std::min(ctx->s_cand.bytes / 16, ctx->p2_vals.bytes / 8);
      if (want_src) {
        HCI_TRY(ensure_buf(ctx, ctx->p2_src, (size_t)A.cap * 4));
        A.srcs = bp<int32_t>(ctx->p2_src);
      }
      HCI_TRY(run_walk(ctx, A, &m));
      if (m <= A.cap || (npart == 1 && m > per)) break;
      HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)(m + m / 8 + 4096) * 16));
      HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)(m + m / 8 + 4096) * 8));
    }
    *m_out = m;
    if (npart == 1 && m > per) return HCI_OK;   // too many for one class: the caller splits the targets
    if (m > A.cap) return hci_fail(ctx, HCI_ERR_CUDA, "hci_pt2: pair count changed between walks");
    if (!reduce || m == 0) return HCI_OK;
    HCI_TRY(ensure_buf(ctx, ctx->s_cand2, (size_t)m * 16));
    HCI_TRY(ensure_buf(ctx, ctx->p2_vals2, (size_t)m * 8));
    int32_t* src = nullptr;
    int32_t* src2 = nullptr;
    double* dpair = nullptr;
    if (want_src) {
      HCI_TRY(ensure_buf(ctx, ctx->p2_src2, (size_t)m * 4));
      HCI_TRY(ensure_buf(ctx, ctx->p2_d, (size_t)m * 8));
      src = bp<int32_t>(ctx->p2_src);
      src2 = bp<int32_t>(ctx->p2_src2);
      dpair = bp<double>(ctx->p2_d);
    }
    int gbits = 0;
    HCI_TRY(group_pairs(ctx, bp<uint64_t>(ctx->s_cand), bp<uint64_t>(ctx->s_cand2), bp<double>(ctx->p2_vals),
                        bp<double>(ctx->p2_vals2), src, src2, m, &gbits));
    const uint64_t gmask = ((uint64_t)1 << gbits) - 1;
    const int tb = grid_for(m, 256, ctx->nsm * 8);
    // [E2, targets outside V], the blocks' sums, the list of the targets
    HCI_TRY(ensure_buf(ctx, ctx->s_flags, (size_t)(2 + tb + m) * 8));
    double* esum = bp<double>(ctx->s_flags);
    unsigned long long* count = reinterpret_cast<unsigned long long*>(esum + 1);
    double* part_e = esum + 2;
    int64_t* list = reinterpret_cast<int64_t*>(part_e + tb);
    HCI_CUDA(ctx, cudaMemsetAsync(count, 0, 8, st));
    HCI_LAUNCH(k_pt2_targets, grid_for(m, 256), 256, 0, st)(bp<ulonglong2>(ctx->s_cand), m, gmask, A.keys,
                                                          bp<int32_t>(ctx->p2_tab), tsize - 1, list, count, dpair);
    const size_t sm = nref * 8;
    HCI_CUDA(ctx, cudaFuncSetAttribute(k_pt2_terms, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    HCI_LAUNCH(k_pt2_terms, tb, 256, sm, st)(bp<ulonglong2>(ctx->s_cand), bp<double>(ctx->p2_vals), m, gmask, list,
                                             count, n, ref, A.ref_a, A.ref_b, e0, part_e, dpair, c, src);
    if (grad_c)
      HCI_LAUNCH(k_pt2_grad, grid_for(m, 256), 256, 0, st)(src, bp<double>(ctx->p2_vals), dpair, m, grad_c);
    if (want_rdm)
      HCI_TRY(pt2_rdm_pairs(ctx, A.keys, c, bp<ulonglong2>(ctx->s_cand), src, dpair, m, list, count));
    HCI_LAUNCH(k_pt2_total, 1, 32, 0, st)(part_e, tb, esum);
    HCI_CUDA(ctx, cudaGetLastError());
    double hs = 0.0;
    unsigned long long hc = 0;
    HCI_CUDA(ctx, cudaMemcpyAsync(&hs, esum, 8, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaMemcpyAsync(&hc, count, 8, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
    acc += hs;
    next_total += (int64_t)hc;
    return HCI_OK;
  };
  HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)4096 * 16));
  HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)4096 * 8));
  // all targets at once when they fit max_pairs; else hash classes
  int64_t total = 0;
  HCI_TRY(run_class(1, 0, &total, true));
  if (total > per) {
    const int64_t np64 = (total + per - 1) / per;
    if (np64 > (1 << 20))
      return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2: max_pairs too small for %lld pairs", (long long)total);
    const int npart = (int)np64;
    const int64_t cap = total / npart + total / (8 * (int64_t)npart) + 4096;
    HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)cap * 16));
    HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)cap * 8));
    for (int pc = 0; pc < npart; ++pc) {
      int64_t m = 0;
      HCI_TRY(run_class(npart, pc, &m, true));
    }
  }
  if (want_rdm) {
    HCI_TRY(pt2_rdm_finish(ctx, rdm1_dd, rdm2_dd, rdm1_dc, rdm2_dc));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
  }
  *e2 = acc;
  if (n_ext) *n_ext = next_total;
  return HCI_OK;
}

// ---------------------------------------------------------------------------
// Semistochastic second-order correction (Sec. II.B, Eq. semistoc):
// E2 ~ E2^D(eps2_det) + mean over samples of [E2^S(eps2) - E2^S(eps2_det)],
// both stochastic terms of a sample taken from the same draws.  A sample is
// n_draws determinants of V drawn with replacement, D_i with probability
// p_i = W_i / sum W (integer weights W_i proportional to |c_i|); the drawn
// determinants are walked like V in the deterministic correction, and every
// target outside V contributes the unbiased multinomial estimate of the
// cited semistochastic HCI work, grouped as
//   (S^2 - T + (N_d - 1) U) / (N_d (N_d - 1) (E0 - H_aa)),
// S = sum_j f_j x_j, T = sum_j (f_j x_j)^2, U = sum_j f_j x_j^2,
// x_j = H_aj c_j, f_j = w_j / p_j (w_j = times D_j was drawn).
// Draw k of sample s uses the first word r of Philox4x64-10 at counter
// (k, s, 0, 0) and key (seed, 0): u = floor(r sum W / 2^64), and the drawn
// index is the i with prefix_{i-1} <= u < prefix_i of the inclusive prefix
// sums of W.  Weights, prefix sums and the draw are exact integer
// arithmetic, so the draws do not depend on the summation order.
// ---------------------------------------------------------------------------
namespace {

// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 64x64->128 multiplications by fixed odd constants, the halves mixed with
// the other two words and the key; the key is bumped by two Weyl
// constants between rounds.
__device__ __forceinline__ uint64_t philox4x64_first(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                                     uint64_t k0, uint64_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B97F4A7C15ull;
      k1 += 0xBB67AE8584CAA73Bull;
    }
    const uint64_t m0 = 0xD2E7470EE14C6C93ull, m1 = 0xCA5A826395121157ull;
    const uint64_t hi0 = __umul64hi(m0, c0), lo0 = m0 * c0;
    const uint64_t hi1 = __umul64hi(m1, c2), lo1 = m1 * c2;
    const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
  }
  return c0;
}

// largest |c_i| (bit pattern of a non-negative double orders like the value)
__global__ void k_abs_max(const double* __restrict__ c, int64_t n, unsigned long long* __restrict__ mx) {
  unsigned long long m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(c[i]));
    m = b > m ? b : m;
  }
  for (int o = 16; o; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
    m = v > m ? v : m;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(mx, m);
}

// W_i = ceil(|c_i| 2^(B - E)), 2^(E-1) <= max|c| < 2^E: W_i >= 1 iff c_i != 0, W_i <= 2^B, sum W <= 2^62
__global__ void k_ss_weights(const double* __restrict__ c, int64_t n, const unsigned long long* __restrict__ mx,
                             int B, int64_t* __restrict__ W) {
  int e = 0;
  frexp(__longlong_as_double((long long)*mx), &e);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    W[i] = (int64_t)ceil(ldexp(fabs(c[i]), B - e));
}

// draws: key (x = sample, y = drawn index) for the sort, and the index alone
__global__ void k_ss_draw(const int64_t* __restrict__ excl, int64_t nV,
                          const int64_t* __restrict__ total, uint64_t seed, int64_t nd, int64_t m,
                          ulonglong2* __restrict__ out, int32_t* __restrict__ draws) {
  const uint64_t tot = (uint64_t)*total;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = t / nd, k = t - s * nd;
    const uint64_t r = philox4x64_first((uint64_t)k, (uint64_t)s, 0ull, 0ull, seed, 0ull);
    const uint64_t u = __umul64hi(r, tot);
    // the i with excl[i] <= u < excl[i] + W[i] is the last i with
    // excl[i] <= u (a zero weight shares its start with the next entry, and
    // the last entry ends at the total > u, so that i has W[i] > 0)
    int64_t lo = 0, hi = nV;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((uint64_t)excl[mid] <= u) lo = mid + 1;
      else hi = mid;
    }
    const int64_t i = lo - 1;
    out[t] = make_ulonglong2((unsigned long long)s, (unsigned long long)i);
    if (draws) draws[t] = (int32_t)i;
  }
}

__global__ void k_run_first(const ulonglong2* __restrict__ k, int64_t m, int64_t* __restrict__ flag) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x)
    flag[t] = (t == 0 || !key_eq(k[t], k[t - 1])) ? 1 : 0;
}

// distinct (sample, index) runs of the sorted draws: index, sample, first position
__global__ void k_ss_compact(const ulonglong2* __restrict__ k, int64_t m, const int64_t* __restrict__ flag,
                             const int64_t* __restrict__ pos, int32_t* __restrict__ d_idx, int32_t* __restrict__ d_s,
                             int64_t* __restrict__ d_start) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x)
    if (flag[t]) {
      const int64_t j = pos[t];
      d_idx[j] = (int32_t)k[t].y;
      d_s[j] = (int32_t)k[t].x;
      d_start[j] = t;
    }
}

// seg[s] = first distinct run of sample s (s = 0..ns)
__global__ void k_ss_seg(const int32_t* __restrict__ d_s, int64_t nd, int ns, int64_t* __restrict__ seg) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s <= ns; s += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = nd;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (d_s[mid] < s) lo = mid + 1;
      else hi = mid;
    }
    seg[s] = lo;
  }
}

// the sources of one sample: key, c, f = w / p with p = W_i / sum W
__global__ void k_ss_gather(int64_t j0, int64_t j1, int64_t ndist, int64_t m, const int32_t* __restrict__ d_idx,
                            const int64_t* __restrict__ d_start, const ulonglong2* __restrict__ keys,
                            const double* __restrict__ c, const int64_t* __restrict__ W,
                            const int64_t* __restrict__ total, ulonglong2* __restrict__ sk, double* __restrict__ sc,
                            double* __restrict__ sf) {
  const double tot = (double)*total;
  for (int64_t j = j0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < j1;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = (j + 1 < ndist ? d_start[j + 1] : m) - d_start[j];
    const int32_t i = d_idx[j];
    const double p = (double)W[i] / tot;
    sk[j - j0] = keys[i];
    sc[j - j0] = c[i];
    sf[j - j0] = (double)w / p;
  }
}

// One listed target per thread (grouped pairs; element H_aj and source j on
// each pair): its estimate with the eps2 screen (every emitted pair) and with
// eps2_det, on its first pair; the other pairs' places are zero beforehand.
// FP64 issue bounds it, so the targets are listed first as for k_pt2_terms:
// taken in place, where only the first pair of a run works, ten samples of
// 1000 draws from 3.4e4 (22e,22o) determinants took 50 ms, 16.8 so.
__global__ void __launch_bounds__(256) k_ss_terms(const ulonglong2* __restrict__ t, const double* __restrict__ v,
                                                  const int32_t* __restrict__ src, int64_t m, uint64_t gmask,
                                                  const int64_t* __restrict__ list,
                                                  const unsigned long long* __restrict__ count,
                                                  const double* __restrict__ sc, const double* __restrict__ sf,
                                                  double eps2_det, double nd, int n, const double* __restrict__ ref,
                                                  uint64_t ra, uint64_t rb, double e0, double* __restrict__ out_t,
                                                  double* __restrict__ out_d) {
  extern __shared__ double s_ref[];
  const int nref = 1 + 2 * n + 4 * n * n;
  for (int u = threadIdx.x; u < nref; u += blockDim.x) s_ref[u] = ref[u];
  __syncthreads();
  const int64_t nt = (int64_t)*count;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nt; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = list[q];
    const ulonglong2 key = t[i];
    double S[2] = {0.0, 0.0}, T[2] = {0.0, 0.0}, U[2] = {0.0, 0.0};
    for (int64_t e = i; e < m; e = next_of_key(t, e, m, key, gmask)) {
      const int32_t j = src[e];
      const double x = v[e] * sc[j], f = sf[j];
      for (int k = 0; k < 2; ++k) {
        if (k == 1 && !(fabs(x) > eps2_det)) break;
        S[k] += f * x;
        T[k] += (f * x) * (f * x);
        U[k] += f * x * x;
      }
    }
    const double den = nd * (nd - 1.0) * (e0 - pt2_diag(s_ref, n, key, ra, rb));
    out_t[i] = (S[0] * S[0] - T[0] + (nd - 1.0) * U[0]) / den;
    out_d[i] = (S[1] * S[1] - T[1] + (nd - 1.0) * U[1]) / den;
  }
}

}  // namespace

extern "C" hci_status hci_pt2_stochastic(hci_ctx* ctx, const uint64_t* keys, const double* c, int64_t nV, double e0,
                                         double eps2, double eps2_det, int64_t n_draws, int n_samples,
                                         uint64_t seed, int64_t max_pairs, double* result, double* sample_e2,
                                         int32_t* draws) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_pt2_stochastic: null context");
  if (!result) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: result is NULL");
  result[0] = result[1] = result[2] = 0.0;
  if (nV < 0 || max_pairs < 0) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: negative size");
  if (n_draws < 2 || n_samples < 1)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: need n_draws >= 2 and n_samples >= 1");
  if (n_draws * (int64_t)n_samples > INT32_MAX)
    return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: n_draws * n_samples exceeds 2^31 - 1");
  if (!(eps2 <= eps2_det)) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: eps2 must not exceed eps2_det");
  if (nV > INT32_MAX) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: more than 2^31 - 1 determinants");
  if (sample_e2)
    for (int s = 0; s < 2 * n_samples; ++s) sample_e2[s] = 0.0;
  if (nV == 0) return HCI_OK;
  if (!keys || !c) return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: null keys or c");
  // deterministic part (also checks the keys and builds the lists)
  double e2d = 0.0;
  HCI_TRY(hci_pt2(ctx, eps2_det, keys, c, nV, e0, max_pairs, &e2d, nullptr, nullptr, nullptr, nullptr, nullptr,
                  nullptr));
  cudaStream_t st = ctx->st;
  const int n = ctx->n;
  const int64_t nd = n_draws, m = nd * n_samples;
  // weights, their exclusive prefix sums and total
  HCI_TRY(ensure_buf(ctx, ctx->ss_w, (size_t)(2 * nV + 2) * 8));
  int64_t* W = bp<int64_t>(ctx->ss_w);
  int64_t* excl = W + nV;
  int64_t* total = excl + nV;
  unsigned long long* mx = reinterpret_cast<unsigned long long*>(total + 1);
  HCI_CUDA(ctx, cudaMemsetAsync(mx, 0, 8, st));
  HCI_LAUNCH(k_abs_max, grid_for(nV, 256, ctx->nsm * 8), 256, 0, st)(c, nV, mx);
  // weight scale 2^B: 2^40, or less so that nV 2^B <= 2^62
  int lg = 0;
  while (((int64_t)1 << lg) < nV) ++lg;
  const int B = lg <= 22 ? 40 : 62 - lg;
  HCI_LAUNCH(k_ss_weights, grid_for(nV, 256, ctx->nsm * 8), 256, 0, st)(c, nV, mx, B, W);
  HCI_TRY(scan_i64(ctx, W, excl, nV, total));
  int64_t tot_h = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&tot_h, total, 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  if (tot_h == 0) {   // c = 0: every estimate is 0
    result[2] = e2d;
    result[0] = e2d;
    if (draws) HCI_CUDA(ctx, cudaMemsetAsync(draws, 0, (size_t)m * 4, st));
    return HCI_OK;
  }
  // draws, sorted by (sample, index), and their distinct runs
  HCI_TRY(ensure_buf(ctx, ctx->ss_draw, (size_t)m * 16));
  HCI_TRY(ensure_buf(ctx, ctx->ss_draw2, (size_t)m * 16));
  ulonglong2* dk = bp<ulonglong2>(ctx->ss_draw);
  HCI_LAUNCH(k_ss_draw, grid_for(m, 256, ctx->nsm * 8), 256, 0, st)(excl, nV, total, seed, nd, m, dk, draws);
  int sbits = 1, ibits = 1;
  while (sbits < 32 && ((int64_t)1 << sbits) < n_samples) ++sbits;
  while (ibits < 32 && ((int64_t)1 << ibits) < nV) ++ibits;
  HCI_TRY(sort_keys(ctx, bp<uint64_t>(ctx->ss_draw), bp<uint64_t>(ctx->ss_draw2), m, sbits, ibits));
  HCI_TRY(ensure_buf(ctx, ctx->ss_run, (size_t)m * (8 + 8 + 8 + 4 + 4) + (size_t)(n_samples + 1) * 8));
  int64_t* flag = bp<int64_t>(ctx->ss_run);
  int64_t* pos = flag + m;
  int64_t* d_start = pos + m;
  int32_t* d_idx = reinterpret_cast<int32_t*>(d_start + m);
  int32_t* d_s = d_idx + m;
  int64_t* seg = reinterpret_cast<int64_t*>(d_s + m);
  int64_t* ndist_dev = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 48);
  HCI_LAUNCH(k_run_first, grid_for(m, 256, ctx->nsm * 8), 256, 0, st)(dk, m, flag);
  HCI_TRY(scan_i64(ctx, flag, pos, m, ndist_dev));
  HCI_LAUNCH(k_ss_compact, grid_for(m, 256, ctx->nsm * 8), 256, 0, st)(dk, m, flag, pos, d_idx, d_s, d_start);
  int64_t ndist = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&ndist, ndist_dev, 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  HCI_LAUNCH(k_ss_seg, 1, 256, 0, st)(d_s, ndist, n_samples, seg);
  std::vector<int64_t> seg_h((size_t)n_samples + 1);
  HCI_CUDA(ctx, cudaMemcpyAsync(seg_h.data(), seg, (size_t)(n_samples + 1) * 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  int64_t maxsrc = 0;
  for (int s = 0; s < n_samples; ++s) maxsrc = std::max(maxsrc, seg_h[s + 1] - seg_h[s]);
  HCI_TRY(ensure_buf(ctx, ctx->ss_src, (size_t)maxsrc * 32));
  ulonglong2* sk = bp<ulonglong2>(ctx->ss_src);
  double* sc = reinterpret_cast<double*>(sk + maxsrc);
  double* sf = sc + maxsrc;
  // the reference of the diagonal elements and the hash table of V (written
  // by hci_pt2 above)
  uint64_t tsize = 1024;
  while (tsize < 2 * (uint64_t)nV) tsize <<= 1;
  WalkArgs A;
  HCI_TRY(pt_walk_args(ctx, A, reinterpret_cast<const uint64_t*>(sk), sc, 0, eps2));
  const size_t nref = 1 + 2 * (size_t)n + 4 * (size_t)n * n;
  double* ref = bp<double>(ctx->p2_ref);
  double* part = ref + nref;
  double* dsum = part + PT2_SUM_BLOCKS;
  const int64_t per = max_pairs > 0 ? max_pairs : ((int64_t)1 << 28);
  const ulonglong2* Vk = reinterpret_cast<const ulonglong2*>(keys);
  const size_t smref = nref * 8;
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_ss_terms, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smref));
  HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)4096 * 16));
  HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)4096 * 8));
  std::vector<double> est((size_t)n_samples * 2, 0.0);
  // one hash class of one sample's targets: walk (again with a larger
  // buffer if it was too small), sort, estimate, sum
  auto run_class = [&](int s, int npart, int pc, int64_t* m_out) -> hci_status {
    A.npart = npart;
    A.part = pc;
    int64_t mp = 0;
    for (int attempt = 0; attempt < 2; ++attempt) {
      A.out = bp<ulonglong2>(ctx->s_cand);
      A.vals = bp<double>(ctx->p2_vals);
      A.cap = (int64_t)std::min(ctx->s_cand.bytes / 16, ctx->p2_vals.bytes / 8);
      HCI_TRY(ensure_buf(ctx, ctx->p2_src, (size_t)A.cap * 4));
      A.srcs = bp<int32_t>(ctx->p2_src);
      HCI_TRY(run_walk(ctx, A, &mp));
      if (mp <= A.cap || (npart == 1 && mp > per)) break;
      HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)(mp + mp / 8 + 4096) * 16));
      HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)(mp + mp / 8 + 4096) * 8));
    }
    *m_out = mp;
    if (npart == 1 && mp > per) return HCI_OK;
    if (mp > A.cap) return hci_fail(ctx, HCI_ERR_CUDA, "hci_pt2_stochastic: pair count changed between walks");
    if (mp == 0) return HCI_OK;
    HCI_TRY(ensure_buf(ctx, ctx->s_cand2, (size_t)mp * 16));
    HCI_TRY(ensure_buf(ctx, ctx->p2_vals2, (size_t)mp * 8));
    HCI_TRY(ensure_buf(ctx, ctx->p2_src2, (size_t)mp * 4));
    HCI_TRY(ensure_buf(ctx, ctx->p2_d, (size_t)mp * 8));
    int gbits = 0;
    HCI_TRY(group_pairs(ctx, bp<uint64_t>(ctx->s_cand), bp<uint64_t>(ctx->s_cand2), bp<double>(ctx->p2_vals),
                        bp<double>(ctx->p2_vals2), bp<int32_t>(ctx->p2_src), bp<int32_t>(ctx->p2_src2), mp, &gbits));
    double* ct = bp<double>(ctx->p2_vals2);
    double* cd = bp<double>(ctx->p2_d);
    const uint64_t gmask = ((uint64_t)1 << gbits) - 1;
    HCI_TRY(ensure_buf(ctx, ctx->s_flags, (size_t)(1 + mp) * 8));
    unsigned long long* count = bp<unsigned long long>(ctx->s_flags);
    int64_t* list = reinterpret_cast<int64_t*>(count + 1);
    HCI_CUDA(ctx, cudaMemsetAsync(count, 0, 8, st));
    HCI_LAUNCH(k_pt2_targets, grid_for(mp, 256), 256, 0, st)(bp<ulonglong2>(ctx->s_cand), mp, gmask, Vk,
                                                           bp<int32_t>(ctx->p2_tab), tsize - 1, list, count, nullptr);
    HCI_CUDA(ctx, cudaMemsetAsync(ct, 0, (size_t)mp * 8, st));
    HCI_CUDA(ctx, cudaMemsetAsync(cd, 0, (size_t)mp * 8, st));
    HCI_LAUNCH(k_ss_terms, grid_for(mp, 256, ctx->nsm * 8), 256, smref, st)(
        bp<ulonglong2>(ctx->s_cand), bp<double>(ctx->p2_vals), bp<int32_t>(ctx->p2_src), mp, gmask, list, count, sc, sf,
        eps2_det, (double)nd, n, ref, A.ref_a, A.ref_b, e0, ct, cd);
    HCI_LAUNCH(k_sum_slices_d, PT2_SUM_BLOCKS, 256, 0, st)(ct, mp, part);
    HCI_LAUNCH(k_sum_parts_d, 1, 32, 0, st)(part, PT2_SUM_BLOCKS, dsum);
    HCI_LAUNCH(k_sum_slices_d, PT2_SUM_BLOCKS, 256, 0, st)(cd, mp, part);
    HCI_LAUNCH(k_sum_parts_d, 1, 32, 0, st)(part, PT2_SUM_BLOCKS, dsum + 1);
    HCI_CUDA(ctx, cudaGetLastError());
    double hs[2] = {0.0, 0.0};
    HCI_CUDA(ctx, cudaMemcpyAsync(hs, dsum, 16, cudaMemcpyDeviceToHost, st));
    HCI_CUDA(ctx, cudaStreamSynchronize(st));
    est[2 * (size_t)s] += hs[0];
    est[2 * (size_t)s + 1] += hs[1];
    return HCI_OK;
  };
  for (int s = 0; s < n_samples; ++s) {
    const int64_t j0 = seg_h[s], j1 = seg_h[s + 1];
    if (j1 <= j0) continue;
    HCI_LAUNCH(k_ss_gather, grid_for(j1 - j0, 256), 256, 0, st)(j0, j1, ndist, m, d_idx, d_start, Vk, c, W, total,
                                                                sk, sc, sf);
    A.nV = j1 - j0;
    int64_t tot_pairs = 0;
    HCI_TRY(run_class(s, 1, 0, &tot_pairs));
    if (tot_pairs > per) {
      const int64_t np64 = (tot_pairs + per - 1) / per;
      if (np64 > (1 << 20))
        return hci_fail(ctx, HCI_ERR_INVALID, "hci_pt2_stochastic: max_pairs too small for %lld pairs",
                        (long long)tot_pairs);
      const int npart = (int)np64;
      const int64_t cap = tot_pairs / npart + tot_pairs / (8 * (int64_t)npart) + 4096;
      HCI_TRY(ensure_buf(ctx, ctx->s_cand, (size_t)cap * 16));
      HCI_TRY(ensure_buf(ctx, ctx->p2_vals, (size_t)cap * 8));
      for (int pc = 0; pc < npart; ++pc) {
        int64_t mp = 0;
        HCI_TRY(run_class(s, npart, pc, &mp));
      }
    }
  }
  // Eq. (semistoc): E2^D plus the mean difference, and its standard error
  double mean = 0.0;
  for (int s = 0; s < n_samples; ++s) mean += est[2 * (size_t)s] - est[2 * (size_t)s + 1];
  mean /= n_samples;
  double var = 0.0;
  for (int s = 0; s < n_samples; ++s) {
    const double d = est[2 * (size_t)s] - est[2 * (size_t)s + 1] - mean;
    var += d * d;
  }
  result[0] = e2d + mean;
  result[1] = n_samples > 1 ? std::sqrt(var / (n_samples - 1) / n_samples) : 0.0;
  result[2] = e2d;
  if (sample_e2)
    for (size_t u = 0; u < est.size(); ++u) sample_e2[u] = est[u];
  return HCI_OK;
}
