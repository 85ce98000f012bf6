// Connection graph of a determinant space and the FP64 sigma H c.
//
// Sec. IV: the Hamiltonian on V is built from all pairs of determinants of V
// that differ by a single or double excitation.  Instead of generating the
// ~N^2 n^2 excitations of each row and looking them up, the determinants are
// grouped by alpha string (V is sorted by (alpha, beta)) and by beta string
// (a second, beta-major order), and connections are found by XOR/popcount
// scans:
//   (A) same alpha string, beta differs by 1 or 2 electrons;
//   (B) same beta string, alpha differs by 1 or 2 electrons;
//   (C) alpha differs by a single (via the single-excitation neighbours of
//       each distinct alpha string) and beta differs by a single.
// The three sets are disjoint.  Two stored forms (hci_set_sigma_mode):
//   both orientations: every row holds all of its connections in a row pool
//     with slack (12 B per ordered pair); H c is a pure gather over the
//     rows, and growing the space appends the new rows' transposes to the
//     old rows in place;
//   one orientation: each connected pair is stored once, in the row of the
//     determinant with the larger internal id (ids are insertion order), in
//     one segment per build or extension (half the memory; growing the
//     space only appends rows), and H c adds each entry to both of its rows
//     (a row sum plus an FP64 atomic scatter into the other row).
#include <algorithm>
#include <vector>

#include "hci_internal.cuh"
#include "rdm_acc.cuh"

namespace {

constexpr int G_WARPS = 8;
// blocks of the row search: six per SM, all resident at 40 registers
inline int rows_grid(const hci_ctx* ctx) { return ctx->nsm * 6; }
constexpr int64_t ROW_SCR = 8192;    // scratch entries per warp of the staged row search
constexpr int64_t ROW_SAMPLE = 2048; // work items counted to size the staging buffer
// pair checks per work item of the row search (see k_item_count)
constexpr int64_t ITEM_COST = 16384;

__device__ __forceinline__ bool key_less(ulonglong2 a, ulonglong2 b) {
  return a.x < b.x || (a.x == b.x && a.y < b.y);
}
__device__ __forceinline__ int64_t lower_bound_k(const ulonglong2* __restrict__ arr, int64_t n, ulonglong2 key) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (key_less(arr[mid], key)) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// grouping
// ---------------------------------------------------------------------------
// word = 0: group by .x (alpha) of keys; word = 1: by .x of swapped keys
__global__ void k_run_flags(const ulonglong2* __restrict__ keys, int64_t n, int64_t* __restrict__ flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = (i == 0 || keys[i].x != keys[i - 1].x) ? 1 : 0;
}

// group index per element, unique strings and group starts
__global__ void k_groups(const ulonglong2* __restrict__ keys, int64_t n, const int64_t* __restrict__ flag,
                         const int64_t* __restrict__ excl, int32_t* __restrict__ gidx, uint64_t* __restrict__ uniq,
                         int64_t* __restrict__ start) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t g = excl[i] + flag[i] - 1;
    gidx[i] = (int32_t)g;
    if (flag[i]) {
      uniq[g] = keys[i].x;
      start[g] = i;
    }
  }
}

__global__ void k_set_last(int64_t* start, const int64_t* ngroups_dev, int64_t n) {
  start[*ngroups_dev] = n;
}

__global__ void k_store_at(int64_t* arr, int64_t idx, const int64_t* val) { arr[idx] = *val; }

__global__ void k_swap_keys(const ulonglong2* __restrict__ in, int64_t n, ulonglong2* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 k = in[i];
    out[i] = make_ulonglong2(k.y, k.x);
  }
}

// permb[k] = index in V of the k-th determinant in beta-major order;
// ib[permb[k]] = beta group of position k
__global__ void k_perm_b(const ulonglong2* __restrict__ bkeys, int64_t n, const ulonglong2* __restrict__ V,
                         const int32_t* __restrict__ bgroup_of_pos, int32_t* __restrict__ permb,
                         int32_t* __restrict__ ib, int32_t* __restrict__ posb, uint64_t* __restrict__ ba) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    ulonglong2 s = bkeys[k];
    int64_t j = lower_bound_k(V, n, make_ulonglong2(s.y, s.x));
    permb[k] = (int32_t)j;
    ib[j] = bgroup_of_pos[k];
    posb[j] = (int32_t)k;
    ba[k] = s.y;
  }
}

__global__ void k_pack_beta(const ulonglong2* __restrict__ V, int64_t n, uint64_t* __restrict__ vb) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    vb[i] = V[i].y;
}

// Open-addressing hash set of the distinct strings (value = group index),
// linear probing; table size is a power of two >= 2 x entries, so probing
// always ends at an empty slot.
constexpr uint64_t HASH_EMPTY = ~0ull;

__device__ __forceinline__ uint64_t hash_str(uint64_t x) {
  x ^= x >> 33; x *= 0xff51afd7ed558ccdull; x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ull; x ^= x >> 33;
  return x;
}

__global__ void k_hash_insert(const uint64_t* __restrict__ u, int64_t nu, unsigned long long* __restrict__ tab,
                              int32_t* __restrict__ val, uint64_t mask) {
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < nu; g += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = u[g];
    uint64_t h = hash_str(key) & mask;
    for (uint64_t probe = 0; probe <= mask; ++probe) {
      const unsigned long long prev = atomicCAS(&tab[h], (unsigned long long)HASH_EMPTY, (unsigned long long)key);
      if (prev == HASH_EMPTY || prev == key) {
        val[h] = (int32_t)g;
        break;
      }
      h = (h + 1) & mask;
    }
  }
}

__device__ __forceinline__ int32_t hash_find(const unsigned long long* __restrict__ tab, const int32_t* __restrict__ val,
                                             uint64_t mask, uint64_t key) {
  uint64_t h = hash_str(key) & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    const unsigned long long t = tab[h];
    if (t == key) return val[h];
    if (t == HASH_EMPTY) return -1;
    h = (h + 1) & mask;
  }
  return -1;
}

// ---------------------------------------------------------------------------
// Slater-Condon element <D_i|H|D_j> for a known connection
// ---------------------------------------------------------------------------
struct HamView {
  int n;
  const double* h;
  const double* eri;
  const double* jk_same;   // [p][r][k] (pr|kk) - (pk|kr)
  const double* j_opp;     // [p][r][k] (pr|kk)
  const double* f_ref;     // [spin][p][r] single p->r of the aufbau determinant
  uint64_t ref_a, ref_b;   // aufbau alpha / beta strings
};

__device__ __forceinline__ double eri4(const HamView& H, int p, int r, int q, int s) {
  return H.eri[(((int64_t)p * H.n + r) * H.n + q) * H.n + s];
}

// single p->r in spin string sj (other spin string oj), both of D_j; spin 0
// = alpha.  h_pr + sum_{k in sj} [(pr|kk) - (pk|kr)] + sum_{k in oj} (pr|kk)
// is taken as the aufbau determinant's value plus the terms of the orbitals
// where sj and oj differ from the aufbau strings (a few for a selected
// determinant, instead of a pass over all n orbitals).
__device__ __forceinline__ double single_el(const HamView& H, uint64_t sj, uint64_t oj, int p, int r, int spin) {
  const uint64_t rs = spin ? H.ref_b : H.ref_a, ro = spin ? H.ref_a : H.ref_b;
  double v = H.f_ref[((int64_t)spin * H.n + p) * H.n + r];
  const double* js = H.jk_same + ((int64_t)p * H.n + r) * H.n;
  const double* jo = H.j_opp + ((int64_t)p * H.n + r) * H.n;
  for (uint64_t m = sj & ~rs; m; m &= m - 1) v += js[__ffsll((long long)m) - 1];
  for (uint64_t m = rs & ~sj; m; m &= m - 1) v -= js[__ffsll((long long)m) - 1];
  for (uint64_t m = oj & ~ro; m; m &= m - 1) v += jo[__ffsll((long long)m) - 1];
  for (uint64_t m = ro & ~oj; m; m &= m - 1) v -= jo[__ffsll((long long)m) - 1];
  return flip_sign(v, bits_between(sj, p, r));
}

__device__ __forceinline__ double same_double_el(const HamView& H, uint64_t sj, uint64_t x) {
  uint64_t holes = sj & x, parts = x & ~sj;
  int p = __ffsll((long long)holes) - 1; holes &= holes - 1;
  int q = __ffsll((long long)holes) - 1;
  int r = __ffsll((long long)parts) - 1; parts &= parts - 1;
  int s = __ffsll((long long)parts) - 1;
  const uint64_t t = sj ^ (1ull << p) ^ (1ull << r);
  return flip_sign(eri4(H, p, r, q, s) - eri4(H, p, s, q, r), bits_between(sj, p, r) + bits_between(t, q, s));
}

__device__ double connection_el(const HamView& H, ulonglong2 ki, ulonglong2 kj) {
  uint64_t xa = ki.x ^ kj.x, xb = ki.y ^ kj.y;
  int da = __popcll(xa), db = __popcll(xb);
  if (da == 0) {
    if (db == 2) {
      int p = __ffsll((long long)(kj.y & xb)) - 1, r = __ffsll((long long)(ki.y & xb)) - 1;
      return single_el(H, kj.y, kj.x, p, r, 1);
    }
    return same_double_el(H, kj.y, xb);
  }
  if (db == 0) {
    if (da == 2) {
      int p = __ffsll((long long)(kj.x & xa)) - 1, r = __ffsll((long long)(ki.x & xa)) - 1;
      return single_el(H, kj.x, kj.y, p, r, 0);
    }
    return same_double_el(H, kj.x, xa);
  }
  int p = __ffsll((long long)(kj.x & xa)) - 1, r = __ffsll((long long)(ki.x & xa)) - 1;
  int q = __ffsll((long long)(kj.y & xb)) - 1, s = __ffsll((long long)(ki.y & xb)) - 1;
  return flip_sign(eri4(H, p, r, q, s), bits_between(kj.x, p, r) + bits_between(kj.y, q, s));
}

// ---------------------------------------------------------------------------
// row traversal: (A) alpha group, (B) beta group, (C) alpha-single x beta-single
// ---------------------------------------------------------------------------
struct GraphArgs {
  const ulonglong2* V;     // alpha-major keys
  int64_t nV;
  int n, na, nb;
  const int32_t* ia;       // alpha group of each det
  const int64_t* ga;       // alpha group starts [nua+1]
  const int32_t* ib;       // beta group of each det
  const int64_t* gb;       // beta group starts (beta-major positions) [nub+1]
  const int32_t* permb;    // beta-major position -> det
  const uint64_t* vb;      // beta string of each det, alpha-major order (packed)
  const uint64_t* ba;      // alpha string of each det, beta-major order (packed)
  const int32_t* posb;     // det -> its beta-major position
  const int64_t* anbr_ptr; // single-excitation neighbours of each distinct alpha string
  const int32_t* anbr;
  const int64_t* bnbr_ptr; // ... of each distinct beta string
  const int32_t* bnbr;
  const int64_t* costa;    // cost of the alpha-side (C) search per distinct alpha string
  const int64_t* costb;
  const int4* items;       // work items {row, its number in the row list, part, parts}
  int64_t nitems;
  const int64_t* offs;     // fill pass: output offset per item
  int32_t* col;
  int64_t* cnt;            // count / staged pass: entries per item
  int32_t* scr;            // staged pass: scr_cap entries of scratch per warp of the grid
  int64_t scr_cap;
  int32_t* stage;          // staged pass: items, each contiguous, at itoff[q]
  int64_t stage_cap;
  int64_t* itoff;
  unsigned long long* stage_ctl;  // [0] next free staging entry, [1] items left to the fill pass
  const int32_t* s2i;      // sorted position -> internal id (columns are stored as internal ids)
  int lower;               // one-orientation form: a row keeps the connections with a smaller id
  unsigned long long* queue;
  HamView H;
  // direct traversals (no stored rows), vectors by sorted position
  const double* dc;             // input vector
  double* dpart;                // sigma: each item's share of its row's sum
  unsigned long long* dnnz;     // sigma: connections visited (may be null)
  RdmAcc R;                     // RDMs: accumulators
};

// A group of size m is scanned when that is cheaper than L binary searches.
__device__ __forceinline__ bool use_lookup(int64_t m, int L) {
  int lg = 64 - __clzll((long long)(m + 1));
  return m > (int64_t)L * lg;
}

// Row search modes: count only, fill at a known offset, or staged fill
// (into the warp's scratch, capped at scr_cap entries, still counting past it).
// With A.lower these three keep only the connections j whose internal id is
// below the row's (the one-orientation form).  Direct traversals evaluate
// every connection as it is found: ROWS_SIGMA adds H_ij c_j into the row's
// sum, ROWS_RDM accumulates <D_i| op |D_j> c_i c_j for j > i (the other
// orientation is added as the transpose).
constexpr int ROWS_COUNT = 0, ROWS_FILL = 1, ROWS_STAGED = 2, ROWS_SIGMA = 3, ROWS_RDM = 4;

// per-row state: row (sorted position), its internal id, c_i, partial sum
struct RowAcc {
  int64_t i;
  int32_t id;
  double ci;
  double acc;
};

template <int MODE>
__device__ __forceinline__ void visit(const GraphArgs& A, ulonglong2 ki, int64_t j, bool ok, int64_t& w,
                                      int32_t* out, RowAcc& ra) {
  const int lane = threadIdx.x & 31;
  int32_t id = 0;
  if (MODE == ROWS_COUNT || MODE == ROWS_FILL || MODE == ROWS_STAGED) {
    if (ok && (A.lower || MODE != ROWS_COUNT)) {
      id = A.s2i[j];
      if (A.lower) ok = id < ra.id;
    }
  }
  unsigned m = __ballot_sync(0xffffffffu, ok);
  if ((MODE == ROWS_FILL || MODE == ROWS_STAGED) && ok) {
    int64_t pos = w + __popc(m & ((1u << lane) - 1u));
    if (MODE == ROWS_FILL || pos < A.scr_cap) out[pos] = id;
  }
  if (MODE == ROWS_SIGMA && ok) ra.acc = fma(connection_el(A.H, ki, A.V[j]), A.dc[j], ra.acc);
  if (MODE == ROWS_RDM && ok && j > ra.i) {
    const double cc = ra.ci * A.dc[j];
    if (cc != 0.0) rdm_accumulate(A.R, A.n, ki, A.V[j], cc);
  }
  w += __popc(m);
}

// (C) from one side.  BETA == false: neighbours are alpha strings, groups are
// alpha groups (members j = position, other-spin value V[j].y); BETA == true:
// neighbours are beta strings, groups live in beta-major order (members
// j = permb[pos], other-spin value ba[pos]).  Small groups are scanned
// (flattened, 32 groups at a time); large groups are probed with binary
// searches for the L single excitations of the other-spin string.
template <int MODE, bool BETA>
__device__ __forceinline__ void mixed_side(const GraphArgs& A, ulonglong2 ki, int g, int64_t& w, int32_t* out,
                                           int64_t* s_start, int64_t* s_pref, int64_t* s_size, const int* occ_o,
                                           const int* vir_o, int nocc_o, int nvir_o, RowAcc& ra, int part, int parts) {
  const int lane = threadIdx.x & 31;
  const int64_t* ptr = BETA ? A.bnbr_ptr : A.anbr_ptr;
  const int32_t* nbr = BETA ? A.bnbr : A.anbr;
  const int64_t* gs = BETA ? A.gb : A.ga;
  const uint64_t mine = BETA ? ki.x : ki.y;     // other-spin string of row i
  const int L = nocc_o * nvir_o;
  int64_t nb0 = ptr[g], nb1 = ptr[g + 1];
  if (parts > 1) {
    const int64_t len = nb1 - nb0, b = nb0;
    nb0 = b + len * part / parts;
    nb1 = b + len * (part + 1) / parts;
  }
  for (int64_t c0 = nb0; c0 < nb1; c0 += 32) {
    const int64_t cidx = c0 + lane;
    int64_t st = 0, sz = 0;
    bool look = false;
    if (cidx < nb1) {
      const int gg = nbr[cidx];
      st = gs[gg];
      sz = gs[gg + 1] - st;
      look = use_lookup(sz, L);
    }
    const int64_t ssz = look ? 0 : sz;
    int64_t inc = ssz;
    for (int o = 1; o < 32; o <<= 1) {
      int64_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    s_start[lane] = st;
    s_size[lane] = sz;
    s_pref[lane + 1] = inc;
    if (lane == 0) s_pref[0] = 0;
    __syncwarp();
    const int64_t total = s_pref[32];
    for (int64_t v0 = 0; v0 < total; v0 += 32) {
      const int64_t v = v0 + lane;
      bool ok = false;
      int64_t j = -1;
      if (v < total) {
        int lo = 0, hi = 31;
        while (lo < hi) {
          int mid = (lo + hi + 1) >> 1;
          if (s_pref[mid] <= v) lo = mid;
          else hi = mid - 1;
        }
        const int64_t pos = s_start[lo] + (v - s_pref[lo]);
        uint64_t other;
        if (BETA) { j = A.permb[pos]; other = A.ba[pos]; }
        else { j = pos; other = A.vb[pos]; }
        ok = __popcll(mine ^ other) == 2;
      }
      visit<MODE>(A, ki, j, ok, w, out, ra);
    }
    unsigned lk = __ballot_sync(0xffffffffu, look);
    while (lk) {
      const int src = __ffs(lk) - 1;
      lk &= lk - 1;
      const int64_t st2 = s_start[src], sz2 = s_size[src];
      for (int t0 = 0; t0 < L; t0 += 32) {
        const int t = t0 + lane;
        bool ok = false;
        int64_t j = -1;
        if (t < L) {
          const uint64_t want = mine ^ (1ull << occ_o[t / nvir_o]) ^ (1ull << vir_o[t % nvir_o]);
          int64_t lo = 0, hi = sz2;
          while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            const uint64_t x = BETA ? A.ba[st2 + mid] : A.vb[st2 + mid];
            if (x < want) lo = mid + 1;
            else hi = mid;
          }
          if (lo < sz2) {
            const uint64_t x = BETA ? A.ba[st2 + lo] : A.vb[st2 + lo];
            if (x == want) { ok = true; j = BETA ? A.permb[st2 + lo] : st2 + lo; }
          }
        }
        visit<MODE>(A, ki, j, ok, w, out, ra);
      }
    }
    __syncwarp();
  }
}

__device__ __forceinline__ int occ_vir_lists(uint64_t s, int n, int* occ, int* vir) {
  const int lane = threadIdx.x & 31;
  int bo = 0, bv = 0;
  for (int p0 = 0; p0 < n; p0 += 32) {
    const int p = p0 + lane;
    const bool in = p < n;
    const bool o = in && ((s >> p) & 1ull);
    const unsigned mo = __ballot_sync(0xffffffffu, o);
    const unsigned mv = __ballot_sync(0xffffffffu, in && !o);
    const unsigned lt = (1u << lane) - 1u;
    if (o) occ[bo + __popc(mo & lt)] = p;
    if (in && !o) vir[bv + __popc(mv & lt)] = p;
    bo += __popc(mo);
    bv += __popc(mv);
  }
  __syncwarp();
  return bo;
}

// Work items of the row search: a row whose search takes more than ITEM_COST
// pair checks (the members of its alpha and beta groups and the cost of its
// cheaper mixed side) is cut into parts, part p of P taking the p-th share
// of both groups and of the neighbour list, so that no warp is left with the
// search of the aufbau determinant's row when all others are done (half of
// the direct product on 3e4 pentacene determinants).
__global__ void k_item_count(GraphArgs A, const int32_t* __restrict__ rowlist, int64_t nrows, int64_t* __restrict__ cnt) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = rowlist ? (int64_t)rowlist[q] : q;
    const int ga = A.ia[i], gb = A.ib[i];
    const int64_t ca = A.costa[ga], cb = A.costb[gb];
    const int64_t cost = (A.ga[ga + 1] - A.ga[ga]) + (A.gb[gb + 1] - A.gb[gb]) + (ca <= cb ? ca : cb);
    const int64_t parts = (cost + ITEM_COST - 1) / ITEM_COST;
    cnt[q] = parts < 1 ? 1 : parts > 4096 ? 4096 : parts;
  }
}
__global__ void k_item_fill(const int32_t* __restrict__ rowlist, int64_t nrows, const int64_t* __restrict__ first,
                            int4* __restrict__ items) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t f = first[q];
    const int parts = (int)(first[q + 1] - f);
    const int i = rowlist ? rowlist[q] : (int)q;
    for (int p = 0; p < parts; ++p) items[f + p] = make_int4(i, (int)q, p, parts);
  }
}

// the p-th of P shares of [b, e)
__device__ __forceinline__ void share(int64_t& b, int64_t& e, int p, int P) {
  if (P > 1) {
    const int64_t len = e - b, b0 = b;
    b = b0 + len * p / P;
    e = b0 + len * (p + 1) / P;
  }
}

// One warp per item taken from a queue.  ROWS_STAGED: the entries go to the
// warp's scratch; at the item's end one atomic reserves its range of the
// staging buffer and they are copied there (itoff[q] = its start, or -1 when
// the item outgrew the scratch or the staging buffer; cnt[q] is exact either
// way).
template <int MODE>
__global__ void __launch_bounds__(G_WARPS * 32, MODE <= ROWS_STAGED ? 6 : 5) k_rows(GraphArgs A) {
  __shared__ int64_t s_start[G_WARPS][32];
  __shared__ int64_t s_size[G_WARPS][32];
  __shared__ int64_t s_pref[G_WARPS][33];
  __shared__ int s_occ[G_WARPS][HCI_MAXORB];
  __shared__ int s_vir[G_WARPS][HCI_MAXORB];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  while (true) {
    unsigned long long qi = 0;
    if (lane == 0) qi = atomicAdd(A.queue, 1ull);
    const int64_t q = (int64_t)__shfl_sync(0xffffffffu, qi, 0);
    if (q >= A.nitems) break;
    const int4 it = A.items[q];
    const int64_t i = it.x;
    const int part = it.z, parts = it.w;
    const ulonglong2 ki = A.V[i];
    int64_t w = MODE == ROWS_FILL ? A.offs[q] : 0;
    int32_t* out = MODE == ROWS_FILL ? A.col
                   : MODE == ROWS_STAGED ? A.scr + (int64_t)(blockIdx.x * G_WARPS + wid) * A.scr_cap
                                         : nullptr;
    RowAcc ra{i, A.s2i[i], (MODE == ROWS_SIGMA || MODE == ROWS_RDM) ? A.dc[i] : 0.0, 0.0};
    // (A) same alpha string
    {
      const int g = A.ia[i];
      int64_t b = A.ga[g], e = A.ga[g + 1];
      share(b, e, part, parts);
      for (int64_t j0 = b; j0 < e; j0 += 64) {
        const int64_t j = j0 + lane, j2 = j + 32;
        const uint64_t x1 = j < e ? A.vb[j] : 0ull, x2 = j2 < e ? A.vb[j2] : 0ull;
        bool ok = false, ok2 = false;
        if (j < e && j != i) {
          const int d = __popcll(ki.y ^ x1);
          ok = d == 2 || d == 4;
        }
        if (j2 < e && j2 != i) {
          const int d = __popcll(ki.y ^ x2);
          ok2 = d == 2 || d == 4;
        }
        visit<MODE>(A, ki, j, ok, w, out, ra);
        if (j0 + 32 < e) visit<MODE>(A, ki, j2, ok2, w, out, ra);
      }
    }
    // (B) same beta string
    {
      const int g = A.ib[i];
      int64_t b = A.gb[g], e = A.gb[g + 1];
      share(b, e, part, parts);
      const int64_t mypos = A.posb[i];
      for (int64_t k0 = b; k0 < e; k0 += 64) {
        const int64_t k = k0 + lane, k2 = k + 32;
        const uint64_t x1 = k < e ? A.ba[k] : 0ull, x2 = k2 < e ? A.ba[k2] : 0ull;
        bool ok = false, ok2 = false;
        if (k < e && k != mypos) {
          const int d = __popcll(ki.x ^ x1);
          ok = d == 2 || d == 4;
        }
        if (k2 < e && k2 != mypos) {
          const int d = __popcll(ki.x ^ x2);
          ok2 = d == 2 || d == 4;
        }
        const int64_t j = ok ? (int64_t)A.permb[k] : -1;
        visit<MODE>(A, ki, j, ok, w, out, ra);
        if (k0 + 32 < e) {
          const int64_t j2 = ok2 ? (int64_t)A.permb[k2] : -1;
          visit<MODE>(A, ki, j2, ok2, w, out, ra);
        }
      }
    }
    // (C) single in alpha and single in beta, from the cheaper side
    {
      const int ga_i = A.ia[i], gb_i = A.ib[i];
      if (A.costa[ga_i] <= A.costb[gb_i]) {
        const int no = occ_vir_lists(ki.y, A.n, s_occ[wid], s_vir[wid]);
        mixed_side<MODE, false>(A, ki, ga_i, w, out, s_start[wid], s_pref[wid], s_size[wid], s_occ[wid],
                                s_vir[wid], no, A.n - no, ra, part, parts);
      } else {
        const int no = occ_vir_lists(ki.x, A.n, s_occ[wid], s_vir[wid]);
        mixed_side<MODE, true>(A, ki, gb_i, w, out, s_start[wid], s_pref[wid], s_size[wid], s_occ[wid],
                               s_vir[wid], no, A.n - no, ra, part, parts);
      }
    }
    if (MODE == ROWS_COUNT && lane == 0) A.cnt[q] = w;
    if (MODE == ROWS_SIGMA) {
      double a = ra.acc;
      for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) {
        A.dpart[q] = a;
        if (A.dnnz) atomicAdd(A.dnnz, (unsigned long long)w);
      }
    }
    if (MODE == ROWS_STAGED) {
      __syncwarp();
      int64_t base = -1;
      if (lane == 0) {
        A.cnt[q] = w;
        if (w <= A.scr_cap) {
          const int64_t b = (int64_t)atomicAdd(A.stage_ctl, (unsigned long long)w);
          if (b + w <= A.stage_cap) base = b;
        }
        if (base < 0) atomicAdd(A.stage_ctl + 1, 1ull);
        A.itoff[q] = base;
      }
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base >= 0)
        for (int64_t t = lane; t < w; t += 32) A.stage[base + t] = out[t];
      __syncwarp();
    }
  }
}

// direct product: a row's sum is its items' shares in order
__global__ void k_row_sums(const int64_t* __restrict__ first, int64_t nV, const double* __restrict__ part,
                           const double* __restrict__ diag, const double* __restrict__ c, double* __restrict__ sigma) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nV; i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int64_t q = first[i]; q < first[i + 1]; ++q) s += part[q];
    sigma[i] = fma(diag[i], c[i], s);
  }
}

// out[t] = a SAMP_SHARE-th of items[t * n / ns], an evenly strided sample of ns
// items (a whole one of ITEM_COST checks keeps its warp for 200 us)
constexpr int SAMP_SHARE = 8;
__global__ void k_stride_sample(const int4* __restrict__ items, int64_t n, int64_t ns, int4* __restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < ns) {
    int4 it = items[t * n / ns];
    it.z = it.z * SAMP_SHARE + (int)(t % SAMP_SHARE);
    it.w *= SAMP_SHARE;
    out[t] = it;
  }
}

// row offsets from the items': rp[q] = itp[first[q]], q <= nrows; len[q] its
// entries (or NULL)
__global__ void k_row_offsets(const int64_t* __restrict__ first, const int64_t* __restrict__ itp, int64_t nrows,
                              int64_t* __restrict__ rp, int64_t* __restrict__ len) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q <= nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = itp[first[q]];
    rp[q] = o;
    if (len && q < nrows) len[q] = itp[first[q + 1]] - o;
  }
}

// where item u's entries go: its row's place plus its offset in the row
__device__ __forceinline__ int64_t item_place(const int4* __restrict__ items, const int64_t* __restrict__ first,
                                              const int64_t* __restrict__ itp, const int64_t* __restrict__ rowoff, int64_t u) {
  const int q = items[u].y;
  return rowoff[q] + itp[u] - itp[first[q]];
}

// Staged items placed (itoff >= 0), one warp per item: copied from the
// staging buffer to their row's place in col
__global__ void k_copy_staged(const int4* __restrict__ items, int64_t nitems, const int64_t* __restrict__ first,
                              const int64_t* __restrict__ itp, const int64_t* __restrict__ itoff,
                              const int64_t* __restrict__ rowoff, const int32_t* __restrict__ stage,
                              int32_t* __restrict__ col) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = warp; u < nitems; u += nwarps) {
    const int64_t off = itoff[u];
    if (off < 0) continue;
    const int64_t b = item_place(items, first, itp, rowoff, u), len = itp[u + 1] - itp[u];
    int64_t t = lane;
    for (; t + 96 < len; t += 128) {
      const int32_t v0 = stage[off + t], v1 = stage[off + t + 32], v2 = stage[off + t + 64], v3 = stage[off + t + 96];
      col[b + t] = v0; col[b + t + 32] = v1; col[b + t + 64] = v2; col[b + t + 96] = v3;
    }
    for (; t < len; t += 32) col[b + t] = stage[off + t];
  }
}

// items the staged pass could not keep (or, with itoff NULL, every item) and
// their places, for the fill pass (any order: each is written at its own)
__global__ void k_collect_left(const int4* __restrict__ items, int64_t nitems, const int64_t* __restrict__ first,
                               const int64_t* __restrict__ itp, const int64_t* __restrict__ itoff,
                               const int64_t* __restrict__ rowoff, unsigned long long* __restrict__ counter,
                               int4* __restrict__ left, int64_t* __restrict__ left_off) {
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nitems; u += (int64_t)gridDim.x * blockDim.x)
    if (!itoff || itoff[u] < 0) {
      const unsigned long long m = atomicAdd(counter, 1ull);
      left[m] = items[u];
      left_off[m] = item_place(items, first, itp, rowoff, u);
    }
}

// Matrix elements of filled rows (the search only records the columns): row
// q has the logical entries [rowptr[q], rowptr[q+1]), kept from start[q] on
// (start NULL: at rowptr[q]) in col/val.  Chunks of RV_CHUNK entries whatever
// rows they belong to, four entries per lane in flight; bound by the latency
// of the gathered keys and integrals.  Phases flip the sign bit: with FP64
// products for them, and a warp per row, 1100 us for the 7e7 entries of a
// pentacene space, 966 us so.
constexpr int RV_CHUNK = 1024;
__global__ void __launch_bounds__(256, 4) k_row_values(const int32_t* __restrict__ rowlist, int64_t nrows,
                                                    const int64_t* __restrict__ rowptr,
                                                    const int64_t* __restrict__ start, const int32_t* __restrict__ col,
                                                    double* __restrict__ val, const ulonglong2* __restrict__ Vrow,
                                                    const ulonglong2* __restrict__ V, HamView H) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = rowptr[nrows];
  for (int64_t e0 = warp * RV_CHUNK; e0 < total; e0 += nwarps * RV_CHUNK) {
    const int64_t e1 = e0 + RV_CHUNK < total ? e0 + RV_CHUNK : total;
    int64_t e = e0;
    for (int64_t q = row_of_entry(rowptr, nrows, e0); e < e1; ++q) {
      const int64_t lo = rowptr[q], hi = rowptr[q + 1] < e1 ? rowptr[q + 1] : e1;
      if (hi <= e) continue;
      const ulonglong2 ki = Vrow[rowlist ? (int64_t)rowlist[q] : q];
      const int64_t b = (start ? start[q] : lo) + (e - lo), len = hi - e;
      e = hi;
      int64_t k = lane;
      for (; k + 96 < len; k += 128) {
        const ulonglong2 k0 = V[col[b + k]], k1 = V[col[b + k + 32]], k2 = V[col[b + k + 64]],
                         k3 = V[col[b + k + 96]];
        val[b + k] = connection_el(H, ki, k0);
        val[b + k + 32] = connection_el(H, ki, k1);
        val[b + k + 64] = connection_el(H, ki, k2);
        val[b + k + 96] = connection_el(H, ki, k3);
      }
      for (; k < len; k += 32) val[b + k] = connection_el(H, ki, V[col[b + k]]);
    }
  }
}

// single-excitation neighbours (within the distinct strings) of each
// distinct string with nocc electrons; count pass (out == nullptr) or fill
// pass.  The nocc * (n - nocc) occupied -> empty pairs are enumerated from
// per-warp occupied / empty lists, p-major, so each list is in (p, r) order.
// With scr, the count pass also writes string g's list at scr + g L (L =
// nocc (n - nocc), its largest possible length), for k_compact_nbrs.
__global__ void __launch_bounds__(256) k_alpha_nbrs(int n, int nocc, const uint64_t* __restrict__ ua, int64_t nua,
                                                    const int64_t* __restrict__ ptr, int64_t* __restrict__ cnt,
                                                    int32_t* __restrict__ out,
                                                    const unsigned long long* __restrict__ tab,
                                                    const int32_t* __restrict__ tval, uint64_t mask,
                                                    int32_t* __restrict__ scr) {
  __shared__ int s_occ[8][HCI_MAXORB];
  __shared__ int s_vir[8][HCI_MAXORB];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int nvir = n - nocc, L = nocc * nvir;
  for (int64_t g = warp; g < nua; g += nwarps) {
    const uint64_t s = ua[g];
    occ_vir_lists(s, n, s_occ[wid], s_vir[wid]);
    int64_t w = out ? ptr[g] : 0;
    int64_t c = 0;
    for (int t0 = 0; t0 < L; t0 += 32) {
      const int t = t0 + lane;
      int32_t idx = -1;
      if (t < L) idx = hash_find(tab, tval, mask, s ^ (1ull << s_occ[wid][t / nvir]) ^ (1ull << s_vir[wid][t % nvir]));
      const bool hit = idx >= 0;
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (out && hit) out[w + c + __popc(m & ((1u << lane) - 1u))] = idx;
      if (scr && hit) scr[g * L + c + __popc(m & ((1u << lane) - 1u))] = idx;
      c += __popc(m);
    }
    if (!out && lane == 0) cnt[g] = c;
    __syncwarp();
  }
}

// list of string g from its padded slot scr + g L to out + ptr[g]
__global__ void __launch_bounds__(256) k_compact_nbrs(const int32_t* __restrict__ scr, int L,
                                                      const int64_t* __restrict__ ptr, int64_t nua,
                                                      int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = warp; g < nua; g += nwarps) {
    const int64_t b = ptr[g], len = ptr[g + 1] - b;
    for (int64_t k = lane; k < len; k += 32) out[b + k] = scr[g * L + k];
  }
}

// cost[u] = sum over the neighbours v of string u of min(scan, lookup) cost
__global__ void k_nbr_cost(const int64_t* __restrict__ ptr, const int32_t* __restrict__ nbr,
                           const int64_t* __restrict__ gs, int64_t nu, int L, int64_t* __restrict__ cost) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = warp; u < nu; u += nwarps) {
    int64_t c = 0;
    for (int64_t k = ptr[u] + lane; k < ptr[u + 1]; k += 32) {
      const int g = nbr[k];
      const int64_t m = gs[g + 1] - gs[g];
      const int lg = 64 - __clzll((long long)(m + 1));
      c += use_lookup(m, L) ? (int64_t)L * lg : m;
    }
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cost[u] = c;
  }
}

// ---------------------------------------------------------------------------
// incremental update: V' = V + N (V's keys all present in V')
// ---------------------------------------------------------------------------
__global__ void k_find_old(const ulonglong2* __restrict__ oldk, int64_t nold, const ulonglong2* __restrict__ V,
                           int64_t nV, int64_t* __restrict__ pos_old, int64_t* __restrict__ mark,
                           unsigned long long* __restrict__ missing) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nold; i += (int64_t)gridDim.x * blockDim.x) {
    const ulonglong2 k = oldk[i];
    const int64_t p = lower_bound_k(V, nV, k);
    if (p < nV && V[p].x == k.x && V[p].y == k.y) {
      pos_old[i] = p;
      mark[p] = 1;
    } else {
      pos_old[i] = -1;
      atomicAdd(missing, 1ull);
    }
  }
}

__global__ void k_not(const int64_t* __restrict__ mark, int64_t n, int64_t* __restrict__ flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = 1 - mark[i];
}

__global__ void k_compact_idx(const int64_t* __restrict__ flag, const int64_t* __restrict__ pos, int64_t n,
                              int32_t* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (flag[i]) out[pos[i]] = (int32_t)i;
}

// rows of V' appended after the nold rows already stored: row nold + q has
// rp[q+1] - rp[q] entries starting at offset rp[q] of segment seg, and the
// prefix continues from base (rp[nrows] = the segment's size); with
// nold = 0, base = 0 and rp = rowptr this writes the table of a fresh graph
__global__ void k_append_rows(int64_t nold, int64_t nrows, const int64_t* rp, int64_t base, int seg,
                              int64_t* rowptr, int64_t* __restrict__ rowstart) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q <= nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = rp[q];
    rowptr[nold + q] = base + o;
    if (q < nrows) rowstart[nold + q] = ((int64_t)seg << GRAPH_SEG_SHIFT) | o;
  }
}

// per new row: number of entries whose column is an old determinant; also
// the histogram of those columns (entries to append to old rows)
__global__ void k_count_old_cols(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int64_t nrows,
                                 int64_t nold, int64_t* __restrict__ cnt, int64_t* __restrict__ hist) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t q = warp; q < nrows; q += nwarps) {
    int64_t c = 0;
    for (int64_t k = rp[q] + lane; k < rp[q + 1]; k += 32) {
      const int32_t j = col[k];
      if (j < nold) {
        ++c;
        atomicAdd((unsigned long long*)&hist[j], 1ull);
      }
    }
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[q] = c;
  }
}

// T records {x = old column (row to append to) | emitting new row q << 32,
// y = entry index in the new rows' CSR}, written in CSR order
// (deterministic); the sort keys on the low 32 bits of x only
__global__ void k_emit_T(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, int64_t nrows,
                         int64_t nold, const int64_t* __restrict__ base, ulonglong2* __restrict__ T) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t q = warp; q < nrows; q += nwarps) {
    int64_t w = base[q];
    for (int64_t k0 = rp[q]; k0 < rp[q + 1]; k0 += 32) {
      const int64_t k = k0 + lane;
      bool ok = false;
      int32_t j = 0;
      if (k < rp[q + 1]) {
        j = col[k];
        ok = j < nold;
      }
      const unsigned m = __ballot_sync(0xffffffffu, ok);
      if (ok)
        T[w + __popc(m & ((1u << lane) - 1u))] = make_ulonglong2((uint64_t)j | ((uint64_t)q << 32), (uint64_t)k);
      w += __popc(m);
    }
  }
}

// ---------------------------------------------------------------------------
// row pool: each row owns [rowstart, rowstart + rowcap) of the col/val
// pools; rowlen <= rowcap entries are live.  Slack lets later updates append
// in place; rows that outgrow it move to the end of the pool.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t slack_cap(int64_t len) { return len + len / 4 + 8; }

__global__ void k_caps(const int64_t* __restrict__ len, int64_t n, int64_t* __restrict__ cap) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    cap[i] = slack_cap(len[i]);
}

// Plan of V' = V + N: new length of every row, its capacity, whether it stays
// (start2 = old start) or needs a new range of `need` entries (start2 = -1).
__global__ void k_plan_rows(const int64_t* __restrict__ start_old, const int64_t* __restrict__ len_old,
                            const int64_t* __restrict__ cap_old, int64_t nold, const int64_t* __restrict__ rpN,
                            int64_t nnew, const int64_t* __restrict__ hist, int repack, int64_t* __restrict__ start2,
                            int64_t* __restrict__ len2, int64_t* __restrict__ cap2, int64_t* __restrict__ need) {
  const int64_t tot = nold + nnew;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    if (t < nold) {
      const int64_t L = len_old[t] + hist[t];
      len2[t] = L;
      if (!repack && L <= cap_old[t]) {
        start2[t] = start_old[t];
        cap2[t] = cap_old[t];
        need[t] = 0;
      } else {
        start2[t] = -1;
        cap2[t] = slack_cap(L);
        need[t] = cap2[t];
      }
    } else {
      const int64_t q = t - nold;
      const int64_t L = rpN[q + 1] - rpN[q];
      len2[t] = L;
      start2[t] = -1;
      cap2[t] = slack_cap(L);
      need[t] = cap2[t];
    }
  }
}

__global__ void k_assign_starts(int64_t* __restrict__ start2, const int64_t* __restrict__ rel, int64_t n, int64_t base) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    if (start2[i] < 0) start2[i] = base + rel[i];
}

// Rows copied to their places: row r's entries from start_src[r] of the source
// to start_dst[r] of the destination, unless that is where they are (columns
// are stable internal ids).  Bound by the 24 bytes per entry it moves; every
// warp takes MOVE_CHUNK consecutive entries (logical offsets rowptr), whatever
// rows they belong to: with a row per warp the aufbau determinant's row was
// all of it on a small space (113 and 19 us for the old and the new rows of
// an extension of 10 to 24 orbital spaces, 17 us each so).
constexpr int64_t MOVE_CHUNK = 1024;

__global__ void __launch_bounds__(256) k_move_rows(const int64_t* __restrict__ rowptr, int64_t nrows,
                                                   const int64_t* __restrict__ start_src, const int32_t* col_src,
                                                   const double* val_src, const int64_t* __restrict__ start_dst,
                                                   int32_t* col_dst, double* val_dst) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t total = rowptr[nrows];
  for (int64_t c0 = warp * MOVE_CHUNK; c0 < total; c0 += nwarps * MOVE_CHUNK) {
    const int64_t c1 = c0 + MOVE_CHUNK < total ? c0 + MOVE_CHUNK : total;
    int64_t r = row_of_entry(rowptr, nrows, c0), lo = rowptr[r];
    for (int64_t e = c0; e < c1; ++r) {
      const int64_t hi = rowptr[r + 1], end = hi < c1 ? hi : c1;
      const int64_t s = start_src[r] - lo, d = start_dst[r] - lo;
      if (s != d || col_src != col_dst) {
        int64_t k = e + lane;
        for (; k + 96 < end; k += 128) {
          const int32_t j0 = col_src[s + k], j1 = col_src[s + k + 32], j2 = col_src[s + k + 64], j3 = col_src[s + k + 96];
          const double v0 = val_src[s + k], v1 = val_src[s + k + 32], v2 = val_src[s + k + 64], v3 = val_src[s + k + 96];
          col_dst[d + k] = j0; col_dst[d + k + 32] = j1; col_dst[d + k + 64] = j2; col_dst[d + k + 96] = j3;
          val_dst[d + k] = v0; val_dst[d + k + 32] = v1; val_dst[d + k + 64] = v2; val_dst[d + k + 96] = v3;
        }
        for (; k < end; k += 32) {
          col_dst[d + k] = col_src[s + k];
          val_dst[d + k] = val_src[s + k];
        }
      }
      e = end;
      lo = hi;
    }
  }
}

// the transposes of the new rows' entries behind the old rows' own, one
// thread each (T is sorted by row; tstart[r] = the row's first)
__global__ void k_append_T(const ulonglong2* __restrict__ T, int64_t nT, const int64_t* __restrict__ tstart,
                           const int64_t* __restrict__ start, const int64_t* __restrict__ len_old, int64_t nold,
                           const double* __restrict__ valN, int32_t* __restrict__ col_dst, double* __restrict__ val_dst) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nT; k += (int64_t)gridDim.x * blockDim.x) {
    const ulonglong2 t = T[k];
    const int64_t r = (int64_t)(t.x & 0xffffffffull);
    const int64_t at = start[r] + len_old[r] + (k - tstart[r]);
    col_dst[at] = (int32_t)(nold + (int64_t)(t.x >> 32));
    val_dst[at] = valN[t.y];
  }
}

// sorted <-> internal maps of V' and the keys in internal order
__global__ void k_build_perm(const int64_t* __restrict__ pos_old, const int32_t* __restrict__ s2i_old, int64_t nold,
                             const int32_t* __restrict__ newrows, int64_t nnew, const ulonglong2* __restrict__ V,
                             int32_t* __restrict__ s2i, int32_t* __restrict__ i2s, ulonglong2* __restrict__ keys_int) {
  const int64_t tot = nold + nnew;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    if (t < nold) {
      const int64_t p = pos_old[t];
      const int32_t id = s2i_old[t];
      s2i[p] = id;
      i2s[id] = (int32_t)p;
    } else {
      const int64_t q = t - nold;
      const int32_t p = newrows[q];
      const int64_t id = nold + q;
      s2i[p] = (int32_t)id;
      i2s[id] = p;
      keys_int[id] = V[p];
    }
  }
}

__global__ void k_iota(int32_t* __restrict__ a, int32_t* __restrict__ b, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    a[i] = b[i] = (int32_t)i;
}

// out[t] = in[idx[t]] for nvec vectors of length n
__global__ void k_gather_vec(const double* __restrict__ in, const int32_t* __restrict__ idx, int64_t n, int nvec,
                             double* __restrict__ out) {
  const int64_t tot = n * nvec;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = t / n, i = t % n;
    out[t] = in[v * n + idx[i]];
  }
}


// Diagonal <D|H|D> (includes e_core) as its difference from the aufbau
// determinant R,
//   E_R + sum_k d_k F_k + sum_{k<l} d_k d_l ((kk|ll) - [same spin] (kl|lk))
// over the spin orbitals where D differs from R (d = -1 emptied, +1 filled):
// a few dozen FP64 additions per determinant, where the sum over all
// occupied pairs takes 700 (1.2e5 determinants of 22 electrons: 101 us, now
// under 40) to 1400.
__global__ void __launch_bounds__(256) k_diag(int n, uint64_t ra, uint64_t rb, const double* __restrict__ h,
                                              const double* __restrict__ eri, const double* __restrict__ f_ref,
                                              double ecore, const ulonglong2* __restrict__ V, int64_t nV,
                                              double* __restrict__ out) {
  extern __shared__ double sm[];
  __shared__ double s_eref;
  double* J = sm;              // (kk|ll)
  double* A = J + n * n;       // (kk|ll) - (kl|lk)
  double* F = A + n * n;       // f_ref's diagonal, alpha then beta
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int k = t / n, l = t % n;
    const double j = eri[(((int64_t)k * n + k) * n + l) * n + l];
    J[t] = j;
    A[t] = j - eri[(((int64_t)k * n + l) * n + l) * n + k];
  }
  for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) F[t] = f_ref[((int64_t)(t / n) * n + t % n) * n + t % n];
  __syncthreads();
  if (threadIdx.x < 32) {
    double e = 0.0;
    for (int t = threadIdx.x; t < 2 * n; t += 32)
      if ((t < n ? ra >> t : rb >> (t - n)) & 1) e += h[(t % n) * n + t % n] + F[t];
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (threadIdx.x == 0) s_eref = fma(0.5, e, ecore);
  }
  __syncthreads();
  const double eref = s_eref;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nV; i += (int64_t)gridDim.x * blockDim.x) {
    const ulonglong2 key = V[i];
    const uint64_t da = key.x ^ ra, db = key.y ^ rb;
    double e1 = 0.0, e2 = 0.0;
    for (uint64_t x = da; x; x &= x - 1) {
      const int k = __ffsll((long long)x) - 1, sk = (int)(ra >> k);
      e1 += flip_sign(F[k], sk);
      for (uint64_t y = x & (x - 1); y; y &= y - 1) {
        const int l = __ffsll((long long)y) - 1;
        e2 += flip_sign(A[k * n + l], sk ^ (int)(ra >> l));
      }
      for (uint64_t y = db; y; y &= y - 1) {
        const int l = __ffsll((long long)y) - 1;
        e2 += flip_sign(J[k * n + l], sk ^ (int)(rb >> l));
      }
    }
    for (uint64_t x = db; x; x &= x - 1) {
      const int k = __ffsll((long long)x) - 1, sk = (int)(rb >> k);
      e1 += flip_sign(F[n + k], sk);
      for (uint64_t y = x & (x - 1); y; y &= y - 1) {
        const int l = __ffsll((long long)y) - 1;
        e2 += flip_sign(A[k * n + l], sk ^ (int)(rb >> l));
      }
    }
    out[i] = eref + (e1 + e2);
  }
}

// Both-orientation form: sigma = diag .* c + offdiag * c.  The connections are
// cut into equal shares (logical entries [w, w + 1) x chunk), whatever rows
// they belong to, and a block's warps take its shares in turn.  A warp owns
// the rows that start in a share and sums the last one up to the share's end;
// the share's head, the rest of a row that started earlier, goes to head[w],
// which k_sigma_heads adds to the row in the order of the shares.  (WHOLE: a
// share takes its last row to the row's end, and there are no heads.)  Nothing
// is done when *stop is set.  (With whole rows per warp the aufbau determinant's
// row, connected to most of a small space, was all of the product.)
//
// Connections come from HBM, c from L2 one 32-byte sector per entry unless L1
// has it: the loads' latency bounded the product (52 cycles of stall per
// instruction, FP64 pipe 70% and HBM 60% busy at 9.7e7 connections).  So a
// batch of 128 connections is loaded while the batch before it gathers c,
// across the ends of rows, and neighbouring rows are worked on side by side
// (16 cycles, 75% and 64%; the FP64 pipe, HBM and L1 share the bound).  Rows
// are summed four at a time, so that the
// cross-lane reduction costs 1.5 FP64 additions per row instead of 8.
// Connections are read with evict-first hints so that c stays in L2.
//
// us per product, whole rows per warp / shares / shares and batches ahead:
// (24e,24o) 2.8e4 determinants 221 / 97 / 85, (22e,22o) 1.2e5 181 / 184 /
// 150, (44e,44o) 3.0e5 2940 / 2521 / 2252 and 4.3e5 3753 / 3777 / 3009.
constexpr int SIGMA_WARPS_PER_SM = 32;   // of k_sigma1, all resident
constexpr int64_t SIGMA_SHARE = 512;     // entries per warp at least
constexpr int64_t SIGMA_SUB = 16384;     // entries per share where a warp has several
// Spaces of up to SIGMA_WHOLE determinants keep their rows whole, each in the
// share where it starts, with a share of SIGMA_WHOLE_SHARE entries per warp: no
// row is longer than 16 batches, and the launch that adds the heads is saved.
// hci_sigma with cut rows / whole ones, us by determinants: 41.8 / 37.4 (33),
// 45.9 / 37.8 (443), 43.8 / 39.0 (1225), 45.7 / 41.4 (1765), 43.9 / 44.1 (2296),
// 46.7 / 47.1 (3482), 48.3 / 51.2 (3807), 57.5 / 96.3 (10020); 64 or 256 entries
// per share change nothing.
constexpr int64_t SIGMA_WHOLE = 2048, SIGMA_WHOLE_SHARE = 128;

// plan[w] = the first row that starts at or after entry w x chunk, w <= warps
__global__ void k_sigma_plan(const int64_t* __restrict__ rowptr, int64_t nV, int64_t warps, int64_t chunk,
                             int32_t* __restrict__ plan) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w > warps) return;
  int64_t lo = 0, hi = nV;
  const int64_t x = w * chunk;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (rowptr[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  plan[w] = (int32_t)(w == warps ? nV : lo);
}

// A row's entries, or those in a share
struct RowPiece {
  const int32_t* col;
  const double* val;
  int len;
};
// 128 of its entries, four per lane, zeros past its end
struct RowBatch {
  int32_t j[4];
  double v[4];
  __device__ __forceinline__ void load(const RowPiece& p, int at) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = at + 32 * u + (int)(threadIdx.x & 31);
      const bool in = k < p.len;
      j[u] = in ? __ldcs(p.col + k) : -1;
      v[u] = in ? __ldcs(p.val + k) : 0.0;
    }
  }
};

// The sum of val c[col] over row p (a lane's share), whose first batch q holds;
// leaves q with the first batch of `next`.
__device__ __forceinline__ double row_sum(const RowPiece& p, const RowPiece& next, RowBatch& q,
                                          const double* __restrict__ c) {
  double a = 0.0, a2 = 0.0;   // two chains, so consecutive FMAs do not wait on each other
  for (int at = 0;; at += 128) {
    double x[4], v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[u] = q.j[u] >= 0 ? c[q.j[u]] : 0.0;
      v[u] = q.v[u];
    }
    const bool last = at + 128 >= p.len;
    if (last) q.load(next, 0);
    else q.load(p, at + 128);
    const int left = p.len - at;
    if (left > 0) a = fma(v[0], x[0], a);
    if (left > 32) a2 = fma(v[1], x[1], a2);
    if (left > 64) a = fma(v[2], x[2], a);
    if (left > 96) a2 = fma(v[3], x[3], a2);
    if (last) return a + a2;
  }
}

template <int WARPS, bool WHOLE>
__global__ void __launch_bounds__(WARPS * 32, SIGMA_WARPS_PER_SM / WARPS) k_sigma1(const int64_t* __restrict__ rowptr,
                                                  const int64_t* __restrict__ rowstart, const int32_t* __restrict__ col,
                                               const double* __restrict__ val, const double* __restrict__ diag,
                                               int64_t nV, const int32_t* __restrict__ plan, int rounds, int64_t chunk,
                                               const double* __restrict__ c, double* __restrict__ sigma,
                                               double* __restrict__ head, const int* __restrict__ stop) {
  if (stop && *stop) return;
  const int lane = threadIdx.x & 31;
  // the block's warps take its shares in turn
  const int64_t w0 = (int64_t)blockIdx.x * WARPS * rounds + (threadIdx.x >> 5);
  for (int t = 0; t < rounds; ++t) {
    const int64_t w = w0 + WARPS * t;
    const int r0 = plan[w], r1 = plan[w + 1];
    const int64_t e0 = WHOLE ? rowptr[r0] : w * chunk, e1 = WHOLE ? rowptr[r1] : e0 + chunk;
    // row i's entries of this share
    auto piece = [&](int i) {
      const int64_t lo = rowptr[i], hi = rowptr[i + 1];
      const int64_t b = lo > e0 ? lo : e0, at = rowstart[i] + (b - lo);
      return RowPiece{col + at, val + at, (int)((hi < e1 ? hi : e1) - b)};
    };
    RowPiece next{col, val, 0};
    RowBatch q;
    const bool has_head = !WHOLE && rowptr[r0] > e0;
    const int first = has_head ? r0 - 1 : r0;
    if (first < r1) next = piece(first);
    q.load(next, 0);
    if (!WHOLE) {
      // the head: row r0 - 1 from e0 on
      double a = 0.0;
      if (has_head) {
        const RowPiece p = next;
        next = r0 < r1 ? piece(r0) : RowPiece{col, val, 0};
        a = row_sum(p, next, q, c);
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      }
      if (lane == 0) head[w] = a;
    }
    for (int g = r0; g < r1; g += 4) {
      double acc[4];
  #pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = g + r;
        acc[r] = 0.0;
        if (i < r1) {
          const RowPiece p = next;
          next = i + 1 < r1 ? piece(i + 1) : RowPiece{col, val, 0};
          acc[r] = row_sum(p, next, q, c);
        }
      }
      // four row sums at once: halve the values held per lane across lanes
      // 16 apart, then 8 apart, then a plain tree over the last 8 lanes
      const bool h16 = lane & 16, h8 = lane & 8;
      const double s0 = (h16 ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, h16 ? acc[0] : acc[2], 16);
      const double s1 = (h16 ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, h16 ? acc[1] : acc[3], 16);
      double u = (h8 ? s1 : s0) + __shfl_xor_sync(0xffffffffu, h8 ? s0 : s1, 8);
      u += __shfl_xor_sync(0xffffffffu, u, 4);
      u += __shfl_xor_sync(0xffffffffu, u, 2);
      u += __shfl_xor_sync(0xffffffffu, u, 1);
      if ((lane & 7) == 0) {
        const int i = g + (h16 ? 2 : 0) + (h8 ? 1 : 0);
        if (i < r1) sigma[i] = fma(diag[i], c[i], u);
      }
    }
  }
}

// The heads added to their rows: the first share of a run of heads of one row
// adds them all, in order.  A thread per share in a launch of its own: left to
// the last block of k_sigma1 its dependent loads took 25 us.
__global__ void __launch_bounds__(128) k_sigma_heads(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ plan,
                                                     int64_t warps, int64_t chunk, const double* __restrict__ head,
                                                     double* __restrict__ sigma, const int* __restrict__ stop) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= warps || (stop && *stop)) return;
  const int64_t row = (int64_t)plan[w] - 1;
  if (row < 0) return;
  const int64_t lo = rowptr[row], hi = rowptr[row + 1];
  if (hi <= w * chunk || lo < (w - 1) * chunk) return;      // no head, or not the row's first
  double s = sigma[row];
  for (int64_t v = w; v < warps && hi > v * chunk; ++v) s += head[v];
  sigma[row] = s;
}

// several vectors at once (one pass over the connections per 4 vectors)
__global__ void __launch_bounds__(256) k_sigma(const int64_t* __restrict__ rowptr,
                                               const int64_t* __restrict__ rowstart, const int32_t* __restrict__ col,
                                               const double* __restrict__ val, const double* __restrict__ diag,
                                               int64_t nV, const double* __restrict__ c, double* __restrict__ sigma,
                                               int nvec) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < nV; i += nwarps) {
    const int64_t b = rowstart[i], e = b + (rowptr[i + 1] - rowptr[i]);
    for (int v0 = 0; v0 < nvec; v0 += 4) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      const int nv = nvec - v0 < 4 ? nvec - v0 : 4;
      for (int64_t k = b + lane; k < e; k += 32) {
        const int64_t j = col[k];
        const double hv = val[k];
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (t < nv) acc[t] = fma(hv, c[(int64_t)(v0 + t) * nV + j], acc[t]);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        double a = acc[t];
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        acc[t] = a;
      }
      if (lane < nv) {
        double a = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3];
        const int64_t o = (int64_t)(v0 + lane) * nV + i;
        sigma[o] = fma(diag[i], c[o], a);
      }
    }
  }
}

// The stored half of row i: its entries' columns and values.
__device__ __forceinline__ void row_entries(const SegTab& T, int64_t rs, const int32_t*& col, const double*& val) {
  const int sg = (int)(rs >> GRAPH_SEG_SHIFT);
  const int64_t o = rs & GRAPH_SEG_MASK;
  col = T.col[sg] + o;
  val = T.val[sg] + o;
}

// One-orientation form: sigma = diag .* c + H_off c.  Each stored entry (i, j, v), j < i, adds
// v c_j to sigma_i (the row sum) and v c_i to sigma_j (an FP64 atomic add
// into sigma, which stays in L2); sigma is zeroed before the launch and each
// row's sum is added atomically too, since other rows scatter into it at the
// same time.  One warp per contiguous range of rows holding an equal share
// of the entries, four (col, val, c[col]) loads per lane in flight, the entry
// stream read with evict-first hints so that c and sigma stay in L2.  Rows
// are summed four at a time, as in k_sigma1: the FP64 pipe (2 operations per
// entry, 2 DFMA per clock per SM) bounds this kernel (80% busy on the
// pentacene space), and stored rows are half as long as full ones.
// blocks of k_sigma1_half per SM: all resident (64 registers, no spills), so
// the equal shares of the entries run in one wave
constexpr int SIGMA_HALF_BLOCKS_PER_SM = 4;

// PASS 0: both contributions of every entry (sigma zeroed first).  When c
// and sigma do not fit L2 together, two passes keep one random-access
// vector in L2 each: PASS 1 writes sigma_i = H_ii c_i + the row sum (plain
// stores, no atomics, no zeroing), PASS 2 then adds the scatters.
template <int PASS>
__global__ void __launch_bounds__(256, SIGMA_HALF_BLOCKS_PER_SM) k_sigma1_half(const int64_t* __restrict__ rowptr,
                                                  const int64_t* __restrict__ rowstart, const __grid_constant__ SegTab T,
                                                  const double* __restrict__ diag, int64_t nV,
                                                  const double* __restrict__ c, double* sigma) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // contiguous row ranges holding an equal share of the entries
  const int64_t tot = rowptr[nV];
  const int64_t chunk = (tot + nwarps - 1) / nwarps;
  int64_t r0, r1;
  {
    int64_t lo = 0, hi = nV, x = warp * chunk;
    while (lo < hi) { const int64_t mid = (lo + hi) >> 1; if (rowptr[mid] < x) lo = mid + 1; else hi = mid; }
    r0 = lo;
    lo = r0; hi = nV; x = (warp + 1) * chunk;
    while (lo < hi) { const int64_t mid = (lo + hi) >> 1; if (rowptr[mid] < x) lo = mid + 1; else hi = mid; }
    r1 = warp == nwarps - 1 ? nV : lo;
  }
  for (int64_t g = r0; g < r1; g += 4) {
    double acc[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      double a = 0.0;
      const int64_t i = g + r;
      if (i < r1) {
        const int64_t len = rowptr[i + 1] - rowptr[i];
        const int32_t* col;
        const double* val;
        row_entries(T, rowstart[i], col, val);
        const double ci = c[i];
        int64_t k = lane;
        if (PASS != 2 || ci != 0.0) {
          for (; k + 96 < len; k += 128) {
            const int32_t j0 = __ldcs(col + k), j1 = __ldcs(col + k + 32), j2 = __ldcs(col + k + 64),
                          j3 = __ldcs(col + k + 96);
            const double v0 = __ldcs(val + k), v1 = __ldcs(val + k + 32), v2 = __ldcs(val + k + 64),
                         v3 = __ldcs(val + k + 96);
            if (PASS != 2) {
              a = fma(v0, c[j0], a);
              a = fma(v1, c[j1], a);
              a = fma(v2, c[j2], a);
              a = fma(v3, c[j3], a);
            }
            if (PASS != 1) {
              atomicAdd(sigma + j0, v0 * ci);
              atomicAdd(sigma + j1, v1 * ci);
              atomicAdd(sigma + j2, v2 * ci);
              atomicAdd(sigma + j3, v3 * ci);
            }
          }
          for (; k < len; k += 32) {
            const int32_t j = __ldcs(col + k);
            const double v = __ldcs(val + k);
            if (PASS != 2) a = fma(v, c[j], a);
            if (PASS != 1) atomicAdd(sigma + j, v * ci);
          }
        }
      }
      acc[r] = a;
    }
    // four row sums at once (1.5 FP64 additions per row for the cross-lane
    // reduction instead of 5): halve the values held per lane across lanes
    // 16 apart, then 8 apart, then a plain tree over the last 8 lanes
    const bool h16 = lane & 16, h8 = lane & 8;
    const double w0 = (h16 ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, h16 ? acc[0] : acc[2], 16);
    const double w1 = (h16 ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, h16 ? acc[1] : acc[3], 16);
    double u = (h8 ? w1 : w0) + __shfl_xor_sync(0xffffffffu, h8 ? w0 : w1, 8);
    u += __shfl_xor_sync(0xffffffffu, u, 4);
    u += __shfl_xor_sync(0xffffffffu, u, 2);
    u += __shfl_xor_sync(0xffffffffu, u, 1);
    if (PASS != 2 && (lane & 7) == 0) {
      const int64_t i = g + (h16 ? 2 : 0) + (h8 ? 1 : 0);
      if (i < r1) {
        if (PASS == 0) atomicAdd(sigma + i, fma(diag[i], c[i], u));
        else sigma[i] = fma(diag[i], c[i], u);
      }
    }
  }
}

// Rows r0 .. nV-1 of H c for a vector that vanishes on them (the rows a
// space gained in its last extension): out[i] = sum of the row's stored
// entries times c (both forms store every connection of such a row to an
// earlier determinant in the row itself); one warp per row, batches loaded
// ahead as in k_sigma1 (the last extensions of a 4.3e5-determinant (44e,44o)
// solve: 227 -> 169 us).
__global__ void __launch_bounds__(256, 4) k_sigma_tail(const int64_t* __restrict__ rowptr,
                                                       const int64_t* __restrict__ rowstart,
                                                       const __grid_constant__ SegTab T, int64_t r0, int64_t nV,
                                                       const double* __restrict__ c, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  auto piece = [&](int64_t i) {
    RowPiece p{nullptr, nullptr, 0};
    if (i < nV) {
      row_entries(T, rowstart[i], p.col, p.val);
      p.len = (int)(rowptr[i + 1] - rowptr[i]);
    }
    return p;
  };
  RowPiece next = piece(r0 + warp);
  RowBatch q;
  q.load(next, 0);
  for (int64_t i = r0 + warp; i < nV; i += nwarps) {
    const RowPiece p = next;
    next = piece(i + nwarps);
    double a = row_sum(p, next, q, c);
    for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) out[i] = a;
  }
}

// several vectors at once (one pass over the entries per 4 vectors); sigma
// zeroed before the launch, as for k_sigma1
__global__ void __launch_bounds__(256) k_sigma_half(const int64_t* __restrict__ rowptr,
                                               const int64_t* __restrict__ rowstart, const __grid_constant__ SegTab T,
                                               const double* __restrict__ diag, int64_t nV,
                                               const double* __restrict__ c, double* sigma, int nvec) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < nV; i += nwarps) {
    const int64_t len = rowptr[i + 1] - rowptr[i];
    const int32_t* col;
    const double* val;
    row_entries(T, rowstart[i], col, val);
    for (int v0 = 0; v0 < nvec; v0 += 4) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      double cin[4] = {0.0, 0.0, 0.0, 0.0};
      const int nv = nvec - v0 < 4 ? nvec - v0 : 4;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < nv) cin[t] = c[(int64_t)(v0 + t) * nV + i];
      for (int64_t k = lane; k < len; k += 32) {
        const int64_t j = col[k];
        const double hv = val[k];
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (t < nv) {
            acc[t] = fma(hv, c[(int64_t)(v0 + t) * nV + j], acc[t]);
            atomicAdd(sigma + (int64_t)(v0 + t) * nV + j, hv * cin[t]);
          }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        double a = acc[t];
        for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        acc[t] = a;
      }
      if (lane < nv) {
        double a = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3];
        const int64_t o = (int64_t)(v0 + lane) * nV + i;
        atomicAdd(sigma + o, fma(diag[i], c[o], a));
      }
    }
  }
}

}  // namespace

// Group structures of the space in G.keys (nV determinants): alpha groups,
// beta-major order and beta groups, single-excitation neighbour lists of the
// distinct alpha and beta strings, and the (C) search cost per string.
static void space_args(hci_ctx* ctx, int64_t nV, GraphArgs& A);

static hci_status build_space(hci_ctx* ctx, int64_t nV, GraphArgs& A) {
  Graph& G = ctx->graph;
  prof_tic(ctx, HCI_PH_GRAPH_SPACE);
  const int n = ctx->n;
  const ulonglong2* V = bp<ulonglong2>(G.keys);
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, ctx->s_flags, (size_t)(2 * nV + 1) * 8));
  int64_t* flag = bp<int64_t>(ctx->s_flags);
  int64_t* excl = flag + nV;
  HCI_TRY(ensure_buf(ctx, ctx->g_ia, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, ctx->g_ua, (size_t)nV * 8));
  HCI_TRY(ensure_buf(ctx, ctx->g_ga, (size_t)(nV + 1) * 8));
  const int gb = grid_for(nV, 256);
  HCI_LAUNCH(k_run_flags, gb, 256, 0, ctx->st)(V, nV, flag);
  HCI_TRY(scan_i64(ctx, flag, excl, nV, dtot));
  HCI_LAUNCH(k_groups, gb, 256, 0, ctx->st)(V, nV, flag, excl, bp<int32_t>(ctx->g_ia), bp<uint64_t>(ctx->g_ua),
                                             bp<int64_t>(ctx->g_ga));
  HCI_LAUNCH(k_set_last, 1, 1, 0, ctx->st)(bp<int64_t>(ctx->g_ga), dtot, nV);
  int64_t nua = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&nua, dtot, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_TRY(ensure_buf(ctx, ctx->g_bkeys, (size_t)nV * 16));
  HCI_TRY(ensure_buf(ctx, ctx->g_bkeys2, (size_t)nV * 16));
  HCI_LAUNCH(k_swap_keys, gb, 256, 0, ctx->st)(V, nV, bp<ulonglong2>(ctx->g_bkeys));
  HCI_TRY(sort_keys(ctx, bp<uint64_t>(ctx->g_bkeys), bp<uint64_t>(ctx->g_bkeys2), nV, n, n));
  HCI_TRY(ensure_buf(ctx, ctx->g_ub, (size_t)nV * 8));
  HCI_TRY(ensure_buf(ctx, ctx->g_gb, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, ctx->g_ib, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, ctx->g_permb, (size_t)nV * 4));
  int32_t* bgroup_of_pos = bp<int32_t>(ctx->g_bkeys2);
  HCI_LAUNCH(k_run_flags, gb, 256, 0, ctx->st)(bp<ulonglong2>(ctx->g_bkeys), nV, flag);
  HCI_TRY(scan_i64(ctx, flag, excl, nV, dtot));
  HCI_LAUNCH(k_groups, gb, 256, 0, ctx->st)(bp<ulonglong2>(ctx->g_bkeys), nV, flag, excl, bgroup_of_pos,
                                             bp<uint64_t>(ctx->g_ub), bp<int64_t>(ctx->g_gb));
  HCI_LAUNCH(k_set_last, 1, 1, 0, ctx->st)(bp<int64_t>(ctx->g_gb), dtot, nV);
  HCI_TRY(ensure_buf(ctx, ctx->g_posb, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, ctx->g_vb, (size_t)nV * 8));
  HCI_TRY(ensure_buf(ctx, ctx->g_ba, (size_t)nV * 8));
  HCI_LAUNCH(k_perm_b, gb, 256, 0, ctx->st)(bp<ulonglong2>(ctx->g_bkeys), nV, V, bgroup_of_pos,
                                             bp<int32_t>(ctx->g_permb), bp<int32_t>(ctx->g_ib),
                                             bp<int32_t>(ctx->g_posb), bp<uint64_t>(ctx->g_ba));
  HCI_LAUNCH(k_pack_beta, gb, 256, 0, ctx->st)(V, nV, bp<uint64_t>(ctx->g_vb));
  int64_t nub = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&nub, dtot, 8, cudaMemcpyDeviceToHost, ctx->st));
  HCI_CUDA(ctx, cudaGetLastError());
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  G.nua = nua;
  G.nub = nub;
  // neighbour lists of both spins
  DevBuf* ptrs[2] = {&ctx->g_nbr_ptr, &ctx->g_bnbr_ptr};
  DevBuf* lists[2] = {&ctx->g_nbr, &ctx->g_bnbr};
  DevBuf* costs[2] = {&ctx->g_costa, &ctx->g_costb};
  const uint64_t* uniq[2] = {bp<uint64_t>(ctx->g_ua), bp<uint64_t>(ctx->g_ub)};
  const int64_t* gstart[2] = {bp<int64_t>(ctx->g_ga), bp<int64_t>(ctx->g_gb)};
  const int64_t nu[2] = {nua, nub};
  // lookups on the alpha side generate beta singles and vice versa
  const int Lside[2] = {ctx->nb * (n - ctx->nb), ctx->na * (n - ctx->na)};
  const int nel[2] = {ctx->na, ctx->nb};
  for (int s = 0; s < 2; ++s) {
    uint64_t tsize = 64;
    while (tsize < (uint64_t)(2 * nu[s] + 2)) tsize <<= 1;
    HCI_TRY(ensure_buf(ctx, ctx->g_htab, (size_t)tsize * 8));
    HCI_TRY(ensure_buf(ctx, ctx->g_hval, (size_t)tsize * 4));
    HCI_CUDA(ctx, cudaMemsetAsync(ctx->g_htab.p, 0xFF, (size_t)tsize * 8, ctx->st));
    HCI_LAUNCH(k_hash_insert, grid_for(nu[s], 256), 256, 0, ctx->st)(uniq[s], nu[s], bp<unsigned long long>(ctx->g_htab),
                                                                      bp<int32_t>(ctx->g_hval), tsize - 1);
    HCI_TRY(ensure_buf(ctx, ctx->g_cnt, (size_t)(nu[s] + 1) * 8));
    HCI_TRY(ensure_buf(ctx, *ptrs[s], (size_t)(nu[s] + 1) * 8));
    HCI_TRY(ensure_buf(ctx, *costs[s], (size_t)(nu[s] + 1) * 8));
    const int gw = grid_for(nu[s] * 32, 256);
    // one pass of hash look-ups when the padded lists (every string's
    // largest possible list) take at most 1 GB, else a count pass and a
    // fill pass
    const int Lown = nel[s] * (n - nel[s]);
    const size_t scr_bytes = (size_t)nu[s] * (size_t)(Lown > 0 ? Lown : 1) * 4;
    const bool one_pass = scr_bytes <= ((size_t)1 << 30);
    if (one_pass) HCI_TRY(ensure_buf(ctx, ctx->g_nscr, scr_bytes));
    HCI_LAUNCH(k_alpha_nbrs, gw, 256, 0, ctx->st)(n, nel[s], uniq[s], nu[s], nullptr, bp<int64_t>(ctx->g_cnt), nullptr,
                                                   bp<unsigned long long>(ctx->g_htab), bp<int32_t>(ctx->g_hval),
                                                   tsize - 1, one_pass ? bp<int32_t>(ctx->g_nscr) : nullptr);
    HCI_TRY(scan_i64(ctx, bp<int64_t>(ctx->g_cnt), bp<int64_t>(*ptrs[s]), nu[s], dtot));
    HCI_LAUNCH(k_store_at, 1, 1, 0, ctx->st)(bp<int64_t>(*ptrs[s]), nu[s], dtot);
    int64_t nn = 0;
    HCI_CUDA(ctx, cudaMemcpyAsync(&nn, dtot, 8, cudaMemcpyDeviceToHost, ctx->st));
    HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
    HCI_TRY(ensure_buf(ctx, *lists[s], (size_t)(nn + 1) * 4));
    if (one_pass)
      HCI_LAUNCH(k_compact_nbrs, gw, 256, 0, ctx->st)(bp<int32_t>(ctx->g_nscr), Lown, bp<int64_t>(*ptrs[s]), nu[s],
                                                       bp<int32_t>(*lists[s]));
    else
      HCI_LAUNCH(k_alpha_nbrs, gw, 256, 0, ctx->st)(n, nel[s], uniq[s], nu[s], bp<int64_t>(*ptrs[s]), nullptr,
                                                     bp<int32_t>(*lists[s]), bp<unsigned long long>(ctx->g_htab),
                                                     bp<int32_t>(ctx->g_hval), tsize - 1, nullptr);
    HCI_LAUNCH(k_nbr_cost, gw, 256, 0, ctx->st)(bp<int64_t>(*ptrs[s]), bp<int32_t>(*lists[s]), gstart[s], nu[s],
                                                 Lside[s], bp<int64_t>(*costs[s]));
  }
  HCI_CUDA(ctx, cudaGetLastError());
  space_args(ctx, nV, A);
  prof_toc(ctx, HCI_PH_GRAPH_SPACE);
  return HCI_OK;
}

// Traversal arguments of the space built by build_space (pointers only).
static void space_args(hci_ctx* ctx, int64_t nV, GraphArgs& A) {
  const int n = ctx->n;
  A = GraphArgs{};
  A.V = bp<ulonglong2>(ctx->graph.keys);
  A.nV = nV;
  A.n = n; A.na = ctx->na; A.nb = ctx->nb;
  A.ia = bp<int32_t>(ctx->g_ia); A.ga = bp<int64_t>(ctx->g_ga);
  A.ib = bp<int32_t>(ctx->g_ib); A.gb = bp<int64_t>(ctx->g_gb);
  A.permb = bp<int32_t>(ctx->g_permb);
  A.vb = bp<uint64_t>(ctx->g_vb);
  A.ba = bp<uint64_t>(ctx->g_ba);
  A.posb = bp<int32_t>(ctx->g_posb);
  A.anbr_ptr = bp<int64_t>(ctx->g_nbr_ptr); A.anbr = bp<int32_t>(ctx->g_nbr);
  A.bnbr_ptr = bp<int64_t>(ctx->g_bnbr_ptr); A.bnbr = bp<int32_t>(ctx->g_bnbr);
  A.costa = bp<int64_t>(ctx->g_costa); A.costb = bp<int64_t>(ctx->g_costb);
  A.H = HamView{n,
                bp<double>(ctx->h),
                bp<double>(ctx->eri),
                bp<double>(ctx->jk_same),
                bp<double>(ctx->j_opp),
                bp<double>(ctx->lists.f_ref),
                ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull),
                ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull)};
  A.queue = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 48);
  A.s2i = bp<int32_t>(ctx->graph.s2i);
}

// Entries of A's items counted into cnt.
static hci_status rows_count(hci_ctx* ctx, GraphArgs A, int64_t* cnt) {
  A.cnt = cnt;
  HCI_CUDA(ctx, cudaMemsetAsync(A.queue, 0, 8, ctx->st));
  HCI_LAUNCH(k_rows<ROWS_COUNT>, rows_grid(ctx), G_WARPS * 32, 0, ctx->st)(A);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

// The nitems items searched, item u's entries written from offs[u] of col.
static hci_status rows_fill(hci_ctx* ctx, GraphArgs A, const int4* items, int64_t nitems, const int64_t* offs,
                            int32_t* col) {
  A.items = items; A.nitems = nitems; A.offs = offs; A.col = col;
  HCI_CUDA(ctx, cudaMemsetAsync(A.queue, 0, 8, ctx->st));
  HCI_LAUNCH(k_rows<ROWS_FILL>, rows_grid(ctx), G_WARPS * 32, 0, ctx->st)(A);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

static int64_t read_i64(hci_ctx* ctx, const int64_t* d, hci_status* st) {
  int64_t v = 0;
  cudaError_t e = cudaMemcpyAsync(&v, d, 8, cudaMemcpyDeviceToHost, ctx->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->st);
  *st = e == cudaSuccess ? HCI_OK : hci_fail(ctx, HCI_ERR_CUDA, "graph: %s", cudaGetErrorString(e));
  return v;
}

// Work items of the rows in rowlist (NULL: rows 0 .. nrows-1) into
// inc.items, each row's first into inc.first.
static hci_status make_items(hci_ctx* ctx, GraphArgs& A, const int32_t* rowlist, int64_t nrows) {
  IncScratch& S = ctx->inc;
  cudaStream_t st = ctx->st;
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, S.cnt, (size_t)(nrows + 1) * 8));
  HCI_TRY(ensure_buf(ctx, S.first, (size_t)(nrows + 1) * 8));
  HCI_LAUNCH(k_item_count, grid_for(nrows, 256), 256, 0, st)(A, rowlist, nrows, bp<int64_t>(S.cnt));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(S.cnt), bp<int64_t>(S.first), nrows, dtot));
  HCI_LAUNCH(k_store_at, 1, 1, 0, st)(bp<int64_t>(S.first), nrows, dtot);
  hci_status hs = HCI_OK;
  A.nitems = read_i64(ctx, dtot, &hs);
  HCI_TRY(hs);
  HCI_TRY(ensure_buf(ctx, S.items, (size_t)A.nitems * 16));
  HCI_LAUNCH(k_item_fill, grid_for(nrows, 256), 256, 0, st)(rowlist, nrows, bp<int64_t>(S.first), bp<int4>(S.items));
  HCI_CUDA(ctx, cudaGetLastError());
  A.items = bp<int4>(S.items);
  return HCI_OK;
}

// Items' counts (inc.cnt) to offsets: inc.itp per item, inc.rpN per row
// (inc.rpN[nrows] = *total); the counts of the rows to len (or NULL).
static hci_status item_offsets(hci_ctx* ctx, const GraphArgs& A, int64_t nrows, int64_t* len) {
  IncScratch& S = ctx->inc;
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, S.itp, (size_t)(A.nitems + 1) * 8));
  HCI_TRY(ensure_buf(ctx, S.rpN, (size_t)(nrows + 1) * 8));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(S.cnt), bp<int64_t>(S.itp), A.nitems, dtot));
  HCI_LAUNCH(k_store_at, 1, 1, 0, ctx->st)(bp<int64_t>(S.itp), A.nitems, dtot);
  HCI_LAUNCH(k_row_offsets, grid_for(nrows + 1, 256), 256, 0, ctx->st)(bp<int64_t>(S.first), bp<int64_t>(S.itp), nrows,
                                                                      bp<int64_t>(S.rpN), len);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

// A's items searched once into per-warp scratch and a staging buffer (sized
// from est entries), their counts and offsets as item_offsets, items that
// outgrew the scratch or the staging space marked for a second search (*left
// of them).
static hci_status stage_search(hci_ctx* ctx, GraphArgs& A, int64_t nrows, int64_t* len, int64_t est, int64_t* total,
                               int64_t* left) {
  IncScratch& S = ctx->inc;
  cudaStream_t st = ctx->st;
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, S.cnt, (size_t)(A.nitems + 1) * 8));
  HCI_TRY(ensure_buf(ctx, S.roff, (size_t)(A.nitems + 1) * 8));
  HCI_TRY(ensure_buf(ctx, S.scr, (size_t)rows_grid(ctx) * G_WARPS * ROW_SCR * 4));
  if (S.stage.bytes < (size_t)est * 4) HCI_TRY(ensure_buf(ctx, S.stage, (size_t)est * 4));
  HCI_TRY(ensure_buf(ctx, S.ctl, 32));
  HCI_CUDA(ctx, cudaMemsetAsync(S.ctl.p, 0, 32, st));
  unsigned long long* ctl = bp<unsigned long long>(S.ctl);
  GraphArgs B = A;
  B.cnt = bp<int64_t>(S.cnt);
  B.scr = bp<int32_t>(S.scr);
  B.scr_cap = ROW_SCR;
  B.stage = bp<int32_t>(S.stage);
  B.stage_cap = (int64_t)(S.stage.bytes / 4);
  B.itoff = bp<int64_t>(S.roff);
  B.stage_ctl = ctl;
  HCI_CUDA(ctx, cudaMemsetAsync(B.queue, 0, 8, st));
  HCI_LAUNCH(k_rows<ROWS_STAGED>, rows_grid(ctx), G_WARPS * 32, 0, st)(B);
  HCI_CUDA(ctx, cudaGetLastError());
  HCI_TRY(item_offsets(ctx, A, nrows, len));
  hci_status hs = HCI_OK;
  *total = read_i64(ctx, dtot, &hs);
  HCI_TRY(hs);
  *left = read_i64(ctx, reinterpret_cast<const int64_t*>(ctl + 1), &hs);
  HCI_TRY(hs);
  return HCI_OK;
}

// Columns of the rows of stage_new_rows written to col, row q at off[q]
// (default inc.rpN[q]): staged items copied, the ones left searched again at
// their places (left < 0: nothing was staged, all are searched again).
static hci_status stage_place(hci_ctx* ctx, GraphArgs& A, int64_t left, int32_t* col, const int64_t* off = nullptr) {
  IncScratch& S = ctx->inc;
  cudaStream_t st = ctx->st;
  if (!off) off = bp<int64_t>(S.rpN);
  const bool staged = left >= 0;
  if (staged) {
    HCI_LAUNCH(k_copy_staged, grid_for(A.nitems * 32, 256), 256, 0, st)(A.items, A.nitems, bp<int64_t>(S.first),
                                                                       bp<int64_t>(S.itp), bp<int64_t>(S.roff), off,
                                                                       bp<int32_t>(S.stage), col);
    HCI_CUDA(ctx, cudaGetLastError());
    ctx->st_counts[HCI_ST_ROWS_REFILLED] += left;
  } else {
    left = A.nitems;
  }
  if (left > 0) {
    HCI_TRY(ensure_buf(ctx, S.ctl, 32));
    unsigned long long* counter = bp<unsigned long long>(S.ctl) + 2;
    HCI_CUDA(ctx, cudaMemsetAsync(counter, 0, 8, st));
    HCI_TRY(ensure_buf(ctx, S.left, (size_t)left * 24 + 16));
    int4* items = bp<int4>(S.left);
    int64_t* offs = reinterpret_cast<int64_t*>(items + left);
    HCI_LAUNCH(k_collect_left, grid_for(A.nitems, 256), 256, 0, st)(A.items, A.nitems, bp<int64_t>(S.first),
                                                                   bp<int64_t>(S.itp),
                                                                   staged ? bp<int64_t>(S.roff) : nullptr, off, counter,
                                                                   items, offs);
    HCI_TRY(rows_fill(ctx, A, items, left, offs, col));
  }
  return HCI_OK;
}

static hci_status compute_diag(hci_ctx* ctx, int64_t nrows, const ulonglong2* keys, double* out) {
  const int n = ctx->n;
  prof_tic(ctx, HCI_PH_HDIAG);
  HCI_CUDA(ctx, cudaFuncSetAttribute(k_diag, cudaFuncAttributeMaxDynamicSharedMemorySize, (2 * 64 * 64 + 128) * 8));
  // few blocks: each one gathers the 2 n^2 integrals
  if (nrows > 0)
    HCI_LAUNCH(k_diag, grid_for(nrows, 256, ctx->nsm * 2), 256, (size_t)(2 * n * n + 2 * n) * 8, ctx->st)(
        n, ctx->na == 64 ? ~0ull : ((1ull << ctx->na) - 1ull), ctx->nb == 64 ? ~0ull : ((1ull << ctx->nb) - 1ull),
        bp<double>(ctx->h), bp<double>(ctx->eri), bp<double>(ctx->lists.f_ref), ctx->ecore, keys, nrows, out);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_HDIAG);
  return HCI_OK;
}

// b grown to at least `bytes` (a quarter more, for later growth), its first
// `keep` bytes preserved
static hci_status grow_keep(hci_ctx* ctx, DevBuf& b, size_t bytes, size_t keep) {
  if (b.p && b.bytes >= bytes) return HCI_OK;
  DevBuf& t = ctx->inc.grow;
  HCI_TRY(ensure_buf(ctx, t, bytes + bytes / 4));
  if (keep > 0 && b.p) HCI_CUDA(ctx, cudaMemcpyAsync(t.p, b.p, keep, cudaMemcpyDeviceToDevice, ctx->st));
  std::swap(b, t);
  free_buf(ctx, t);
  return HCI_OK;
}

static void free_segments(hci_ctx* ctx) {
  Graph& G = ctx->graph;
  for (int k = 0; k < GRAPH_MAXSEG; ++k) {
    free_buf(ctx, G.seg_col[k]);
    free_buf(ctx, G.seg_val[k]);
  }
  G.nseg = 0;
  G.nstored = 0;
  G.nnz = 0;
  G.pool_used = G.pool_cap = 0;
}

// Buffers of stored connections: the pool grows in place up to what they
// hold, so under a budget they hold what was admitted and no more.
static hci_status conn_buf(hci_ctx* ctx, DevBuf& b, int64_t bytes) {
  return ensure_buf(ctx, b, (size_t)bytes, ctx->graph_budget > 0);
}

// A new segment of `entries` stored connections; HCI_ERR_NOMEM when the
// stored connections would exceed the context's budget.
static hci_status seg_alloc(hci_ctx* ctx, int64_t entries, int* seg) {
  Graph& G = ctx->graph;
  if (G.nseg >= GRAPH_MAXSEG) return hci_fail(ctx, HCI_ERR_INVALID, "graph: segment table full");
  const int64_t bytes = (G.nstored + entries) * 12;
  if (ctx->graph_budget > 0 && bytes > ctx->graph_budget)
    return hci_fail(ctx, HCI_ERR_NOMEM, "graph: %lld bytes of stored connections exceed the budget of %lld",
                    (long long)bytes, (long long)ctx->graph_budget);
  HCI_TRY(conn_buf(ctx, G.seg_col[G.nseg], (entries + 1) * 4));
  HCI_TRY(conn_buf(ctx, G.seg_val[G.nseg], (entries + 1) * 8));
  *seg = G.nseg++;
  return HCI_OK;
}

// The nnew rows in rowlist (NULL: all of V in order) cut into items and
// searched once (stage_search), the staging space sized from the mean count
// of a strided sample of the items (the old rows' lengths say little when
// the space grows many-fold).  When that space would exceed an eighth of
// device memory the items are only counted here (*left = -1) and stage_place
// searches them a second time, straight into place.  Rows' entries to len (or
// NULL).
static hci_status stage_new_rows(hci_ctx* ctx, GraphArgs& A, const int32_t* rowlist, int64_t nnew, int64_t nV,
                                 int64_t* len, int64_t* total, int64_t* left) {
  IncScratch& S = ctx->inc;
  cudaStream_t st = ctx->st;
  HCI_TRY(make_items(ctx, A, rowlist, nnew));
  const int64_t ns = std::min<int64_t>(A.nitems, ROW_SAMPLE);
  HCI_TRY(ensure_buf(ctx, S.samp, (size_t)ns * 24 + 16));
  int4* samp = bp<int4>(S.samp);
  int64_t* samp_cnt = reinterpret_cast<int64_t*>(samp + ns);
  HCI_LAUNCH(k_stride_sample, grid_for(ns, 256), 256, 0, st)(A.items, A.nitems, ns, samp);
  GraphArgs B = A;
  B.items = samp;
  B.nitems = ns;
  HCI_TRY(rows_count(ctx, B, samp_cnt));
  std::vector<int64_t> cnt((size_t)ns);
  HCI_CUDA(ctx, cudaMemcpyAsync(cnt.data(), samp_cnt, (size_t)ns * 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  double sum = 0.0;
  for (int64_t v : cnt) sum += (double)v;
  const double mean = ns > 0 ? SAMP_SHARE * sum / (double)ns : 0.0, rows = (double)A.nitems * mean;
  const int64_t est = (int64_t)std::min((double)nnew * (double)nV, 1.5 * rows) + ((int64_t)1 << 22);
  {
    // a graph that cannot fit device memory is refused before the search:
    // both orientations add the new rows, their transposes and slack to the
    // pool, one orientation adds the new rows
    const Graph& G = ctx->graph;
    const double need = G.half ? (double)G.nstored + rows : (double)G.pool_used + 2.5 * rows;
    if (need * 12.0 > 0.9 * (double)ctx->mem_total)
      return hci_fail(ctx, HCI_ERR_NOMEM, "graph: about %.3g bytes of stored connections would exceed device memory",
                      need * 12.0);
  }
  if ((double)est * 4.0 > (double)ctx->mem_total / 8.0) {
    // a staging buffer this large would crowd out the stored rows: count
    // the rows first and let stage_place search them again into place
    int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
    HCI_TRY(ensure_buf(ctx, S.cnt, (size_t)(A.nitems + 1) * 8));
    HCI_TRY(rows_count(ctx, A, bp<int64_t>(S.cnt)));
    HCI_TRY(item_offsets(ctx, A, nnew, len));
    hci_status hs = HCI_OK;
    *total = read_i64(ctx, dtot, &hs);
    *left = -1;
    return hs;
  }
  return stage_search(ctx, A, nnew, len, est, total, left);
}

// blocks of k_row_values: a warp per chunk, at most 16 blocks per SM
static int values_grid(int64_t entries) { return grid_for((entries + RV_CHUNK - 1) / RV_CHUNK * 32, 256); }

static hci_status graph_build_half(hci_ctx* ctx, const uint64_t* keys, int64_t nV) {
  Graph& G = ctx->graph;
  G.valid = false;
  if (nV >= ((int64_t)1 << 31) - 1) return hci_fail(ctx, HCI_ERR_INVALID, "graph: nV exceeds int32 columns");
  free_segments(ctx);
  G.half = true;
  prof_tic(ctx, HCI_PH_GRAPH);
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, G.keys, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  // a fresh space: internal ids = sorted positions
  HCI_TRY(ensure_buf(ctx, G.keys_int, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys_int.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  HCI_TRY(ensure_buf(ctx, G.s2i, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, G.i2s, (size_t)nV * 4));
  HCI_LAUNCH(k_iota, grid_for(nV, 256), 256, 0, ctx->st)(bp<int32_t>(G.s2i), bp<int32_t>(G.i2s), nV);
  GraphArgs A;
  HCI_TRY(build_space(ctx, nV, A));
  A.s2i = bp<int32_t>(G.s2i);
  A.lower = 1;
  prof_tic(ctx, HCI_PH_GRAPH_ROWS);
  // stored halves of the rows, each searched once (staged), into one segment,
  // then their elements
  int64_t nst = 0, left = 0;
  HCI_TRY(stage_new_rows(ctx, A, nullptr, nV, nV, nullptr, &nst, &left));
  HCI_TRY(ensure_buf(ctx, G.rowptr, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, G.rowstart, (size_t)(nV + 1) * 8));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.rowptr.p, ctx->inc.rpN.p, (size_t)(nV + 1) * 8, cudaMemcpyDeviceToDevice, ctx->st));
  int seg = 0;
  HCI_TRY(seg_alloc(ctx, nst, &seg));
  int32_t* col = bp<int32_t>(G.seg_col[seg]);
  double* val = bp<double>(G.seg_val[seg]);
  HCI_TRY(stage_place(ctx, A, left, col));
  HCI_LAUNCH(k_row_values, values_grid(nst), 256, 0, ctx->st)(
      nullptr, nV, bp<int64_t>(G.rowptr), nullptr, col, val, bp<ulonglong2>(G.keys), bp<ulonglong2>(G.keys_int), A.H);
  HCI_LAUNCH(k_append_rows, grid_for(nV + 1, 256), 256, 0, ctx->st)(0, nV, bp<int64_t>(G.rowptr), 0, seg,
                                                                     bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart));
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_GRAPH_ROWS);
  HCI_TRY(ensure_buf(ctx, G.diag, (size_t)nV * 8));
  HCI_TRY(compute_diag(ctx, nV, bp<ulonglong2>(G.keys_int), bp<double>(G.diag)));
  prof_toc(ctx, HCI_PH_GRAPH);
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  G.nV = nV;
  G.nstored = nst;
  G.nnz = 2 * nst;
  G.epoch += 1;
  G.parent = -1;
  ctx->st_counts[HCI_ST_GRAPH_BUILDS] += 1;
  G.valid = true;
  return HCI_OK;
}

// V' contains every determinant of the cached space.  Rows and columns of the
// graph are internal ids (insertion order): old determinants keep theirs and
// the new ones are numbered after them, so a connection between an old and a
// new determinant belongs to the new row, and the stored rows never change.
// Only the new rows are searched (once, staged), into one new segment.
static hci_status graph_extend_half(hci_ctx* ctx, const uint64_t* keys, int64_t nV, bool* done) {
  Graph& G = ctx->graph;
  IncScratch& S = ctx->inc;
  *done = false;
  const int64_t nold = G.nV;
  if (nV <= nold || nV >= ((int64_t)1 << 31) - 1 || G.nseg >= GRAPH_MAXSEG) return HCI_OK;
  cudaStream_t st = ctx->st;
  unsigned long long* missing = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 24);
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  const ulonglong2* Vn = reinterpret_cast<const ulonglong2*>(keys);
  HCI_TRY(ensure_buf(ctx, S.pos_old, (size_t)nold * 8));
  HCI_TRY(ensure_buf(ctx, S.mark, (size_t)nV * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(S.mark.p, 0, (size_t)nV * 8, st));
  HCI_CUDA(ctx, cudaMemsetAsync(missing, 0, 8, st));
  HCI_LAUNCH(k_find_old, grid_for(nold, 256), 256, 0, st)(bp<ulonglong2>(G.keys), nold, Vn, nV,
                                                          bp<int64_t>(S.pos_old), bp<int64_t>(S.mark), missing);
  unsigned long long miss = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&miss, missing, 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  if (miss) return HCI_OK;        // not an extension: full rebuild
  prof_tic(ctx, HCI_PH_GRAPH);
  const int64_t nnew = nV - nold;
  // keys and map of the old space move to the scratch side
  std::swap(G.keys, S.keys_old);
  std::swap(G.s2i, S.s2i_old);
  HCI_TRY(ensure_buf(ctx, G.keys, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, st));
  // new determinants in sorted order, their internal ids nold + q
  HCI_TRY(ensure_buf(ctx, S.flag, (size_t)(2 * nV + 1) * 8));
  int64_t* nflag = bp<int64_t>(S.flag);
  int64_t* npos = nflag + nV;
  HCI_LAUNCH(k_not, grid_for(nV, 256), 256, 0, st)(bp<int64_t>(S.mark), nV, nflag);
  HCI_TRY(scan_i64(ctx, nflag, npos, nV, dtot));
  HCI_TRY(ensure_buf(ctx, S.newrows, (size_t)nnew * 4));
  HCI_LAUNCH(k_compact_idx, grid_for(nV, 256), 256, 0, st)(nflag, npos, nV, bp<int32_t>(S.newrows));
  // maps and internal-order keys of V' (old ids and keys unchanged)
  HCI_TRY(ensure_buf(ctx, G.s2i, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, G.i2s, (size_t)nV * 4));
  HCI_TRY(grow_keep(ctx, G.keys_int, (size_t)nV * 16, (size_t)nold * 16));
  HCI_LAUNCH(k_build_perm, grid_for(nV, 256), 256, 0, st)(bp<int64_t>(S.pos_old), bp<int32_t>(S.s2i_old), nold,
                                                          bp<int32_t>(S.newrows), nnew, Vn, bp<int32_t>(G.s2i),
                                                          bp<int32_t>(G.i2s), bp<ulonglong2>(G.keys_int));
  GraphArgs A;
  HCI_TRY(build_space(ctx, nV, A));
  A.s2i = bp<int32_t>(G.s2i);
  A.lower = 1;
  prof_tic(ctx, HCI_PH_GRAPH_ROWS);
  int64_t total = 0, left = 0;
  HCI_TRY(stage_new_rows(ctx, A, bp<int32_t>(S.newrows), nnew, nV, nullptr, &total, &left));
  int seg = 0;
  HCI_TRY(seg_alloc(ctx, total, &seg));
  int32_t* col = bp<int32_t>(G.seg_col[seg]);
  double* val = bp<double>(G.seg_val[seg]);
  HCI_TRY(stage_place(ctx, A, left, col));
  HCI_LAUNCH(k_row_values, values_grid(total), 256, 0, st)(
      bp<int32_t>(S.newrows), nnew, bp<int64_t>(S.rpN), nullptr, col, val, bp<ulonglong2>(G.keys),
      bp<ulonglong2>(G.keys_int), A.H);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_GRAPH_ROWS);
  // row table: the new rows after the old ones
  prof_tic(ctx, HCI_PH_GRAPH_MERGE);
  HCI_TRY(grow_keep(ctx, G.rowptr, (size_t)(nV + 1) * 8, (size_t)(nold + 1) * 8));
  HCI_TRY(grow_keep(ctx, G.rowstart, (size_t)(nV + 1) * 8, (size_t)nold * 8));
  HCI_LAUNCH(k_append_rows, grid_for(nnew + 1, 256), 256, 0, st)(nold, nnew, bp<int64_t>(S.rpN), G.nstored, seg,
                                                                  bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart));
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_GRAPH_MERGE);
  // diagonal: old entries stay, the new ids are computed
  HCI_TRY(grow_keep(ctx, G.diag, (size_t)nV * 8, (size_t)nold * 8));
  HCI_TRY(compute_diag(ctx, nnew, bp<ulonglong2>(G.keys_int) + nold, bp<double>(G.diag) + nold));
  prof_toc(ctx, HCI_PH_GRAPH);
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  G.parent = G.epoch;
  G.epoch += 1;
  G.nold = nold;
  G.tail_entries = total;
  G.nV = nV;
  G.nstored += total;
  G.nnz = 2 * G.nstored;
  ctx->st_counts[HCI_ST_GRAPH_BUILDS] += 1;
  *done = true;
  return HCI_OK;
}

// entries the both-orientation pool (segment 0) holds
static int64_t pool_entries(const Graph& G) {
  const int64_t a = (int64_t)(G.seg_col[0].bytes / 4), b = (int64_t)(G.seg_val[0].bytes / 8);
  return a < b ? a : b;
}

static hci_status graph_build_full(hci_ctx* ctx, const uint64_t* keys, int64_t nV) {
  Graph& G = ctx->graph;
  G.valid = false;
  if (nV >= ((int64_t)1 << 31) - 1) return hci_fail(ctx, HCI_ERR_INVALID, "graph: nV exceeds int32 columns");
  free_segments(ctx);
  G.half = false;
  prof_tic(ctx, HCI_PH_GRAPH);
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  HCI_TRY(ensure_buf(ctx, G.keys, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  // a fresh space: internal ids = sorted positions
  HCI_TRY(ensure_buf(ctx, G.keys_int, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys_int.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  HCI_TRY(ensure_buf(ctx, G.s2i, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, G.i2s, (size_t)nV * 4));
  HCI_LAUNCH(k_iota, grid_for(nV, 256), 256, 0, ctx->st)(bp<int32_t>(G.s2i), bp<int32_t>(G.i2s), nV);
  GraphArgs A;
  HCI_TRY(build_space(ctx, nV, A));
  A.s2i = bp<int32_t>(G.s2i);
  prof_tic(ctx, HCI_PH_GRAPH_ROWS);
  // every row searched once (staged, as for the new rows of an extension),
  // lengths and logical offsets from it
  HCI_TRY(ensure_buf(ctx, G.rowlen, (size_t)(nV + 1) * 8));
  int64_t nnz = 0, left = 0;
  HCI_TRY(stage_new_rows(ctx, A, nullptr, nV, nV, bp<int64_t>(G.rowlen), &nnz, &left));
  HCI_TRY(ensure_buf(ctx, G.rowptr, (size_t)(nV + 1) * 8));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.rowptr.p, ctx->inc.rpN.p, (size_t)(nV + 1) * 8, cudaMemcpyDeviceToDevice, ctx->st));
  // capacities with slack, starts = their prefix sums, pool with headroom
  HCI_TRY(ensure_buf(ctx, G.rowcap, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, G.rowstart, (size_t)(nV + 1) * 8));
  HCI_LAUNCH(k_caps, grid_for(nV, 256), 256, 0, ctx->st)(bp<int64_t>(G.rowlen), nV, bp<int64_t>(G.rowcap));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(G.rowcap), bp<int64_t>(G.rowstart), nV, dtot));
  hci_status st = HCI_OK;
  const int64_t used = read_i64(ctx, dtot, &st);
  HCI_TRY(st);
  const int64_t cap = used + used / 4 + 1024;
  if (ctx->graph_budget > 0 && cap * 12 > ctx->graph_budget)
    return hci_fail(ctx, HCI_ERR_NOMEM, "graph: a pool of %lld bytes exceeds the budget of %lld", (long long)(cap * 12),
                    (long long)ctx->graph_budget);
  HCI_TRY(conn_buf(ctx, G.seg_col[0], cap * 4));
  HCI_TRY(conn_buf(ctx, G.seg_val[0], cap * 8));
  G.nseg = 1;
  HCI_TRY(stage_place(ctx, A, left, bp<int32_t>(G.seg_col[0]), bp<int64_t>(G.rowstart)));
  HCI_LAUNCH(k_row_values, values_grid(nnz), 256, 0, ctx->st)(
      nullptr, nV, bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), bp<int32_t>(G.seg_col[0]),
      bp<double>(G.seg_val[0]), bp<ulonglong2>(G.keys), bp<ulonglong2>(G.keys_int), A.H);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_GRAPH_ROWS);
  HCI_TRY(ensure_buf(ctx, G.diag, (size_t)nV * 8));
  HCI_TRY(compute_diag(ctx, nV, bp<ulonglong2>(G.keys_int), bp<double>(G.diag)));
  prof_toc(ctx, HCI_PH_GRAPH);
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  G.nV = nV;
  G.nnz = nnz;
  G.nstored = nnz;
  G.epoch += 1;
  G.parent = -1;
  G.pool_used = used;
  G.pool_cap = pool_entries(G);
  ctx->st_counts[HCI_ST_GRAPH_BUILDS] += 1;
  G.valid = true;
  return HCI_OK;
}

// V' contains every determinant of the cached space.  Rows and columns of the
// graph are internal ids (insertion order): old determinants keep theirs and
// the new ones are numbered after them, so only the new rows are searched,
// their transposes are appended to the old rows (in place where the row's
// slack allows), and no stored column changes.
static hci_status graph_extend_full(hci_ctx* ctx, const uint64_t* keys, int64_t nV, bool* done) {
  Graph& G = ctx->graph;
  IncScratch& S = ctx->inc;
  *done = false;
  const int64_t nold = G.nV;
  if (nV <= nold || nV >= ((int64_t)1 << 31) - 1 || G.nseg != 1) return HCI_OK;
  cudaStream_t st = ctx->st;
  unsigned long long* missing = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 24);
  int64_t* dtot = reinterpret_cast<int64_t*>(bp<char>(ctx->s_counter) + 40);
  const ulonglong2* Vn = reinterpret_cast<const ulonglong2*>(keys);
  HCI_TRY(ensure_buf(ctx, S.pos_old, (size_t)nold * 8));
  HCI_TRY(ensure_buf(ctx, S.mark, (size_t)nV * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(S.mark.p, 0, (size_t)nV * 8, st));
  HCI_CUDA(ctx, cudaMemsetAsync(missing, 0, 8, st));
  HCI_LAUNCH(k_find_old, grid_for(nold, 256), 256, 0, st)(bp<ulonglong2>(G.keys), nold, Vn, nV,
                                                          bp<int64_t>(S.pos_old), bp<int64_t>(S.mark), missing);
  unsigned long long miss = 0;
  HCI_CUDA(ctx, cudaMemcpyAsync(&miss, missing, 8, cudaMemcpyDeviceToHost, st));
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  if (miss) return HCI_OK;        // not an extension: full rebuild
  prof_tic(ctx, HCI_PH_GRAPH);
  hci_status hs = HCI_OK;
  const int64_t nnew = nV - nold;
  // keys, maps and row arrays of the old space move to the scratch side
  std::swap(G.keys, S.keys_old);
  std::swap(G.s2i, S.s2i_old);
  std::swap(G.rowstart, S.rp_old);
  std::swap(G.rowlen, S.len_old);
  std::swap(G.rowcap, S.cap_old);
  HCI_TRY(ensure_buf(ctx, G.keys, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, st));
  // new determinants in sorted order, their internal ids nold + q
  HCI_TRY(ensure_buf(ctx, S.flag, (size_t)(2 * nV + 1) * 8));
  int64_t* nflag = bp<int64_t>(S.flag);
  int64_t* npos = nflag + nV;
  HCI_LAUNCH(k_not, grid_for(nV, 256), 256, 0, st)(bp<int64_t>(S.mark), nV, nflag);
  HCI_TRY(scan_i64(ctx, nflag, npos, nV, dtot));
  HCI_TRY(ensure_buf(ctx, S.newrows, (size_t)nnew * 4));
  HCI_LAUNCH(k_compact_idx, grid_for(nV, 256), 256, 0, st)(nflag, npos, nV, bp<int32_t>(S.newrows));
  // maps and internal-order keys of V' (old ids and keys unchanged)
  HCI_TRY(ensure_buf(ctx, G.s2i, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, G.i2s, (size_t)nV * 4));
  HCI_TRY(grow_keep(ctx, G.keys_int, (size_t)nV * 16, (size_t)nold * 16));
  HCI_LAUNCH(k_build_perm, grid_for(nV, 256), 256, 0, st)(bp<int64_t>(S.pos_old), bp<int32_t>(S.s2i_old), nold,
                                                          bp<int32_t>(S.newrows), nnew, Vn, bp<int32_t>(G.s2i),
                                                          bp<int32_t>(G.i2s), bp<ulonglong2>(G.keys_int));
  GraphArgs A;
  HCI_TRY(build_space(ctx, nV, A));
  A.s2i = bp<int32_t>(G.s2i);
  prof_tic(ctx, HCI_PH_GRAPH_ROWS);
  // staging space from the mean length of a strided sample of the new rows
  // (the old rows' lengths say little when the space grows many-fold)
  int64_t nnzN = 0;
  {
    int64_t left = 0;
    HCI_TRY(stage_new_rows(ctx, A, bp<int32_t>(S.newrows), nnew, nV, nullptr, &nnzN, &left));
    HCI_TRY(ensure_buf(ctx, S.colN, (size_t)(nnzN + 1) * 4));
    HCI_TRY(ensure_buf(ctx, S.valN, (size_t)(nnzN + 1) * 8));
    HCI_TRY(stage_place(ctx, A, left, bp<int32_t>(S.colN)));
  }
  HCI_LAUNCH(k_row_values, values_grid(nnzN), 256, 0, st)(
      bp<int32_t>(S.newrows), nnew, bp<int64_t>(S.rpN), nullptr, bp<int32_t>(S.colN), bp<double>(S.valN),
      bp<ulonglong2>(G.keys), bp<ulonglong2>(G.keys_int), A.H);
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_GRAPH_ROWS);
  // transposed entries for the old rows, sorted by the row they go to
  prof_tic(ctx, HCI_PH_GRAPH_MERGE);
  HCI_TRY(ensure_buf(ctx, S.hist, (size_t)(nV + 1) * 8));
  HCI_CUDA(ctx, cudaMemsetAsync(S.hist.p, 0, (size_t)(nV + 1) * 8, st));
  const int gw = grid_for(nnew * 32, 256);
  HCI_TRY(ensure_buf(ctx, S.cnt, (size_t)(nnew + 1) * 8));
  HCI_LAUNCH(k_count_old_cols, gw, 256, 0, st)(bp<int64_t>(S.rpN), bp<int32_t>(S.colN), nnew, nold,
                                                bp<int64_t>(S.cnt), bp<int64_t>(S.hist));
  HCI_TRY(ensure_buf(ctx, S.tbase, (size_t)(nnew + 1) * 8));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(S.cnt), bp<int64_t>(S.tbase), nnew, dtot));
  const int64_t nT = read_i64(ctx, dtot, &hs);
  HCI_TRY(hs);
  HCI_TRY(ensure_buf(ctx, S.T, (size_t)(nT + 1) * 16));
  HCI_TRY(ensure_buf(ctx, S.T2, (size_t)(nT + 1) * 16));
  HCI_LAUNCH(k_emit_T, gw, 256, 0, st)(bp<int64_t>(S.rpN), bp<int32_t>(S.colN), nnew, nold, bp<int64_t>(S.tbase),
                                        bp<ulonglong2>(S.T));
  int bits = 1;
  while (((int64_t)1 << bits) < nold) ++bits;
  HCI_TRY(sort_keys(ctx, bp<uint64_t>(S.T), bp<uint64_t>(S.T2), nT, bits, 0));
  HCI_TRY(ensure_buf(ctx, S.tstart, (size_t)(nV + 1) * 8));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(S.hist), bp<int64_t>(S.tstart), nold, dtot));
  // plan the rows of V' (by internal id) in the pool: stay or take a new range
  HCI_TRY(ensure_buf(ctx, G.rowstart, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, G.rowlen, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, G.rowcap, (size_t)(nV + 1) * 8));
  HCI_TRY(ensure_buf(ctx, S.len, (size_t)(2 * nV + 2) * 8));
  int64_t* need = bp<int64_t>(S.len);
  int64_t* rel = need + nV + 1;
  int64_t total = 0;
  int repack = 0;
  for (int pass = 0; pass < 2; ++pass) {
    HCI_LAUNCH(k_plan_rows, grid_for(nV, 256), 256, 0, st)(
        bp<int64_t>(S.rp_old), bp<int64_t>(S.len_old), bp<int64_t>(S.cap_old), nold, bp<int64_t>(S.rpN), nnew,
        bp<int64_t>(S.hist), repack, bp<int64_t>(G.rowstart), bp<int64_t>(G.rowlen), bp<int64_t>(G.rowcap), need);
    HCI_TRY(scan_i64(ctx, need, rel, nV, dtot));
    total = read_i64(ctx, dtot, &hs);
    HCI_TRY(hs);
    if (repack || G.pool_used + total <= G.pool_cap) break;
    repack = 1;
  }
  int32_t* col_dst = bp<int32_t>(G.seg_col[0]);
  double* val_dst = bp<double>(G.seg_val[0]);
  int64_t base = G.pool_used;
  if (repack) {
    const int64_t cap = total + total / 4 + 1024;
    // the old pool stays alive while the new one is filled
    if (ctx->graph_budget > 0 && (cap + G.pool_cap) * 12 > ctx->graph_budget)
      return hci_fail(ctx, HCI_ERR_NOMEM, "graph: repacking into %lld bytes exceeds the budget of %lld",
                      (long long)(cap * 12), (long long)ctx->graph_budget);
    HCI_TRY(conn_buf(ctx, S.col_old, cap * 4));
    HCI_TRY(conn_buf(ctx, S.val_old, cap * 8));
    col_dst = bp<int32_t>(S.col_old);
    val_dst = bp<double>(S.val_old);
    base = 0;
  }
  HCI_LAUNCH(k_assign_starts, grid_for(nV, 256), 256, 0, st)(bp<int64_t>(G.rowstart), rel, nV, base);
  const auto move_grid = [&](int64_t entries) { return grid_for((entries + MOVE_CHUNK - 1) / MOVE_CHUNK * 32, 256); };
  HCI_LAUNCH(k_move_rows, move_grid(G.nnz), 256, 0, st)(bp<int64_t>(G.rowptr), nold, bp<int64_t>(S.rp_old),
                                                        bp<int32_t>(G.seg_col[0]), bp<double>(G.seg_val[0]),
                                                        bp<int64_t>(G.rowstart), col_dst, val_dst);
  if (nT > 0)
    HCI_LAUNCH(k_append_T, grid_for(nT, 256), 256, 0, st)(bp<ulonglong2>(S.T), nT, bp<int64_t>(S.tstart),
                                                         bp<int64_t>(G.rowstart), bp<int64_t>(S.len_old), nold,
                                                         bp<double>(S.valN), col_dst, val_dst);
  HCI_LAUNCH(k_move_rows, move_grid(nnzN), 256, 0, st)(bp<int64_t>(S.rpN), nnew, bp<int64_t>(S.rpN),
                                                       bp<int32_t>(S.colN), bp<double>(S.valN),
                                                       bp<int64_t>(G.rowstart) + nold, col_dst, val_dst);
  HCI_CUDA(ctx, cudaGetLastError());
  if (repack) {
    std::swap(G.seg_col[0], S.col_old);
    std::swap(G.seg_val[0], S.val_old);
    free_buf(ctx, S.col_old);
    free_buf(ctx, S.val_old);
    G.pool_cap = pool_entries(G);
    G.pool_used = total;
  } else {
    G.pool_used += total;
  }
  // logical prefix of the row lengths (internal order)
  HCI_TRY(ensure_buf(ctx, G.rowptr, (size_t)(nV + 1) * 8));
  HCI_TRY(scan_i64(ctx, bp<int64_t>(G.rowlen), bp<int64_t>(G.rowptr), nV, dtot));
  HCI_LAUNCH(k_store_at, 1, 1, 0, st)(bp<int64_t>(G.rowptr), nV, dtot);
  const int64_t nnz = read_i64(ctx, dtot, &hs);
  HCI_TRY(hs);
  prof_toc(ctx, HCI_PH_GRAPH_MERGE);
  if (nnz != G.nnz + nnzN + nT)
    return hci_fail(ctx, HCI_ERR_CUDA, "graph_extend: inconsistent sizes %lld != %lld + %lld + %lld", (long long)nnz,
                    (long long)G.nnz, (long long)nnzN, (long long)nT);
  // diagonal: old entries stay, the new ids are computed
  HCI_TRY(grow_keep(ctx, G.diag, (size_t)nV * 8, (size_t)nold * 8));
  HCI_TRY(compute_diag(ctx, nnew, bp<ulonglong2>(G.keys_int) + nold, bp<double>(G.diag) + nold));
  prof_toc(ctx, HCI_PH_GRAPH);
  HCI_CUDA(ctx, cudaStreamSynchronize(st));
  G.parent = G.epoch;
  G.epoch += 1;
  G.tail_entries = nnzN;
  G.nold = nold;
  G.nV = nV;
  G.nnz = nnz;
  G.nstored = nnz;
  ctx->st_counts[HCI_ST_GRAPH_BUILDS] += 1;
  *done = true;
  return HCI_OK;
}

// Direct form: the space's search structures and diagonal only (internal
// ids = sorted positions); every traversal searches the rows again.
static hci_status graph_build_direct(hci_ctx* ctx, const uint64_t* keys, int64_t nV) {
  Graph& G = ctx->graph;
  G.valid = false;
  free_segments(ctx);
  if (nV >= ((int64_t)1 << 31) - 1) return hci_fail(ctx, HCI_ERR_INVALID, "graph: nV exceeds int32 indices");
  prof_tic(ctx, HCI_PH_GRAPH);
  HCI_TRY(ensure_buf(ctx, ctx->s_counter, 64));
  HCI_TRY(ensure_buf(ctx, G.keys, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  HCI_TRY(ensure_buf(ctx, G.keys_int, (size_t)nV * 16));
  HCI_CUDA(ctx, cudaMemcpyAsync(G.keys_int.p, keys, (size_t)nV * 16, cudaMemcpyDeviceToDevice, ctx->st));
  HCI_TRY(ensure_buf(ctx, G.s2i, (size_t)nV * 4));
  HCI_TRY(ensure_buf(ctx, G.i2s, (size_t)nV * 4));
  HCI_LAUNCH(k_iota, grid_for(nV, 256), 256, 0, ctx->st)(bp<int32_t>(G.s2i), bp<int32_t>(G.i2s), nV);
  GraphArgs A;
  HCI_TRY(build_space(ctx, nV, A));
  // the work items of every traversal, and their shares of the rows' sums
  HCI_TRY(make_items(ctx, A, nullptr, nV));
  ctx->inc.nitems = A.nitems;
  HCI_TRY(ensure_buf(ctx, ctx->inc.itp, (size_t)A.nitems * 8));
  HCI_TRY(ensure_buf(ctx, G.diag, (size_t)nV * 8));
  HCI_TRY(compute_diag(ctx, nV, bp<ulonglong2>(G.keys_int), bp<double>(G.diag)));
  prof_toc(ctx, HCI_PH_GRAPH);
  HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
  G.nV = nV;
  G.nnz = -1;   // counted by the first direct sigma
  G.direct = true;
  G.epoch += 1;
  G.parent = -1;
  ctx->st_counts[HCI_ST_GRAPH_BUILDS] += 1;
  G.valid = true;
  return HCI_OK;
}

// the stored rows and the incremental scratch, released before a direct build
static void release_stored(hci_ctx* ctx) {
  Graph& G = ctx->graph;
  IncScratch& S = ctx->inc;
  free_segments(ctx);
  DevBuf* bufs[] = {&G.rowptr, &G.rowstart, &G.rowlen, &G.rowcap, &S.scr, &S.stage, &S.grow, &S.col_old,
                    &S.val_old, &S.colN, &S.valN, &S.T, &S.T2, &S.items, &S.first, &S.itp};
  for (DevBuf* b : bufs) free_buf(ctx, *b);
  cudaStreamSynchronize(ctx->st);
}

// Stored form of the next build: both orientations unless the context was
// set to one orientation or fell back to it.
static bool want_half(const hci_ctx* ctx) {
  return ctx->sigma_mode == HCI_SIGMA_HALF || (ctx->sigma_mode == HCI_SIGMA_AUTO && ctx->half_fallback);
}

static hci_status plan_sigma(hci_ctx* ctx);

static hci_status graph_stored(hci_ctx* ctx, const uint64_t* keys, int64_t nV) {
  Graph& G = ctx->graph;
  const bool half = want_half(ctx);
  hci_status s = HCI_OK;
  bool done = false;
  if (G.valid && !G.direct && G.half == half && ctx->incremental) {
    G.valid = false;
    s = half ? graph_extend_half(ctx, keys, nV, &done) : graph_extend_full(ctx, keys, nV, &done);
  }
  if (s == HCI_OK && !done) {
    G.direct = false;
    s = half ? graph_build_half(ctx, keys, nV) : graph_build_full(ctx, keys, nV);
  }
  if (s == HCI_OK && !half) s = plan_sigma(ctx);
  // a failure behind the build leaves a graph without its plan, and under the
  // hash of the space before it
  if (s != HCI_OK) G.valid = false;
  return s;
}

// HCI_SIGMA_AUTO: both orientations while they fit the budget (or device
// memory), then one orientation, then the direct form, each step for the
// rest of the context's life.
hci_status graph_ensure(hci_ctx* ctx, const uint64_t* keys, int64_t nV) {
  uint64_t hsh = 0;
  HCI_TRY(hash_keys(ctx, keys, nV, &hsh));
  if (ctx->graph.valid && ctx->graph.nV == nV && ctx->graph.hash == hsh) return HCI_OK;
  int ok = 0;
  HCI_TRY(check_sorted(ctx, keys, nV, &ok));
  if (!ok) return hci_fail(ctx, HCI_ERR_INVALID, "keys are not strictly ascending");
  const bool direct = ctx->sigma_mode == HCI_SIGMA_DIRECT || (ctx->sigma_mode == HCI_SIGMA_AUTO && ctx->direct_fallback);
  if (!direct) {
    hci_status s = graph_stored(ctx, keys, nV);
    if (s == HCI_ERR_NOMEM && ctx->sigma_mode == HCI_SIGMA_AUTO && !ctx->half_fallback) {
      // both orientations do not fit: store one orientation of each pair
      ctx->graph.valid = false;
      ctx->half_fallback = true;
      release_stored(ctx);
      s = graph_stored(ctx, keys, nV);
    }
    if (s == HCI_OK) {
      ctx->graph.hash = hsh;
      ctx->graph.valid = true;
      return HCI_OK;
    }
    if (s != HCI_ERR_NOMEM || ctx->sigma_mode != HCI_SIGMA_AUTO) return s;
    // the connections do not fit: search them again in every traversal
    ctx->graph.valid = false;
    ctx->direct_fallback = true;
    release_stored(ctx);
  }
  HCI_TRY(graph_build_direct(ctx, keys, nV));
  ctx->graph.hash = hsh;
  ctx->graph.valid = true;
  return HCI_OK;
}

// H c of a direct graph: every row's connections searched and evaluated
static hci_status sigma_direct(hci_ctx* ctx, const double* c, double* sigma, int nvec) {
  Graph& G = ctx->graph;
  GraphArgs A;
  space_args(ctx, G.nV, A);
  A.items = bp<int4>(ctx->inc.items);
  A.nitems = ctx->inc.nitems;
  A.dpart = bp<double>(ctx->inc.itp);
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(bp<char>(ctx->s_counter) + 56);
  for (int v = 0; v < nvec; ++v) {
    A.dc = c + (int64_t)v * G.nV;
    A.dnnz = G.nnz < 0 ? cnt : nullptr;
    if (A.dnnz) HCI_CUDA(ctx, cudaMemsetAsync(cnt, 0, 8, ctx->st));
    HCI_CUDA(ctx, cudaMemsetAsync(A.queue, 0, 8, ctx->st));
    HCI_LAUNCH(k_rows<ROWS_SIGMA>, rows_grid(ctx), G_WARPS * 32, 0, ctx->st)(A);
    HCI_LAUNCH(k_row_sums, grid_for(G.nV, 256), 256, 0, ctx->st)(bp<int64_t>(ctx->inc.first), G.nV, A.dpart,
                                                                bp<double>(G.diag), A.dc, sigma + (int64_t)v * G.nV);
    HCI_CUDA(ctx, cudaGetLastError());
    if (A.dnnz) {
      unsigned long long h = 0;
      HCI_CUDA(ctx, cudaMemcpyAsync(&h, cnt, 8, cudaMemcpyDeviceToHost, ctx->st));
      HCI_CUDA(ctx, cudaStreamSynchronize(ctx->st));
      G.nnz = (int64_t)h;
    }
  }
  return HCI_OK;
}

hci_status direct_rdm(hci_ctx* ctx, const double* c, const RdmAcc& R) {
  Graph& G = ctx->graph;
  GraphArgs A;
  space_args(ctx, G.nV, A);
  A.items = bp<int4>(ctx->inc.items);
  A.nitems = ctx->inc.nitems;
  A.dc = c;
  A.R = R;
  HCI_CUDA(ctx, cudaMemsetAsync(A.queue, 0, 8, ctx->st));
  HCI_LAUNCH(k_rows<ROWS_RDM>, rows_grid(ctx), G_WARPS * 32, 0, ctx->st)(A);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

// plan of k_sigma1 for the cached both-orientation graph: the shares' first
// rows, then the heads
static double* sig_head(Graph& G) { return reinterpret_cast<double*>(bp<char>(G.sig_plan) + ((size_t)(G.sig_warps + 2) * 4 + 7) / 8 * 8); }
static hci_status plan_sigma(hci_ctx* ctx) {
  Graph& G = ctx->graph;
  // Warps per block: with a share per warp, 8 (22 orbitals, 8e6 connections
  // 50.5 us, 16 warps 52.1; 12 orbitals, 4e5: 16.3 and 19.6).  With several,
  // a block's warps work on neighbouring rows and so find each other's c in
  // L1: 16 (44 orbitals, 1.3e9: 3302 us with 8, 3009 with 16, 3070 with 32;
  // 28 orbitals, 9.7e7: 242, 236, 241).
  const int64_t most = (int64_t)ctx->nsm * SIGMA_WARPS_PER_SM;
  const bool whole = G.nV <= SIGMA_WHOLE;
  const int block = !whole && G.nstored >= most * SIGMA_SUB ? 16 : 8;
  const int64_t share = whole ? SIGMA_WHOLE_SHARE : SIGMA_SHARE;
  const int64_t warps = std::max<int64_t>(1, std::min(most, G.nstored / share) / block) * block;
  const int64_t rounds = std::max<int64_t>(1, (G.nstored + warps * SIGMA_SUB / 2) / (warps * SIGMA_SUB));
  const int64_t shares = warps * rounds;
  HCI_TRY(ensure_buf(ctx, G.sig_plan, (size_t)(shares + 2) * 4 + 8 + (size_t)shares * 8 + 16));
  G.sig_whole = whole;
  G.sig_block = block;
  G.sig_rounds = (int)rounds;
  G.sig_warps = shares;
  G.sig_chunk = std::max<int64_t>(1, (G.nstored + shares - 1) / shares);
  HCI_LAUNCH(k_sigma_plan, (unsigned)((G.sig_warps + 256) / 256), 256, 0, ctx->st)(
      bp<int64_t>(G.rowptr), G.nV, G.sig_warps, G.sig_chunk, bp<int32_t>(G.sig_plan));
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

hci_status sigma_apply(hci_ctx* ctx, const double* c, double* sigma, int nvec, const int* stop) {
  Graph& G = ctx->graph;
  if (G.direct) {
    prof_tic(ctx, HCI_PH_SIGMA);
    HCI_TRY(sigma_direct(ctx, c, sigma, nvec));
    ctx->st_counts[HCI_ST_SIGMA_CALLS] += nvec;
    ctx->st_counts[HCI_ST_SIGMA_ROWS] += G.nV * nvec;
    ctx->st_counts[HCI_ST_SIGMA_NNZ] += G.nnz * nvec;
    prof_toc(ctx, HCI_PH_SIGMA);
    return HCI_OK;
  }
  // one orientation: two passes when c and sigma together exceed half of L2
  // (HCI_SIGMA_HALF_PASSES set at context creation overrides the choice)
  const bool two_pass = G.half && nvec == 1 &&
                        (ctx->half_passes ? ctx->half_passes == 2 : (double)G.nV * 16.0 > 0.5 * (double)ctx->l2_bytes);
  if (G.half && !two_pass) HCI_CUDA(ctx, cudaMemsetAsync(sigma, 0, (size_t)G.nV * nvec * 8, ctx->st));
  prof_tic(ctx, HCI_PH_SIGMA);
  ctx->st_counts[HCI_ST_SIGMA_CALLS] += nvec;
  ctx->st_counts[HCI_ST_SIGMA_ROWS] += G.nV * nvec;
  ctx->st_counts[HCI_ST_SIGMA_NNZ] += G.nnz * nvec;
  if (G.half) {
    const SegTab T = G.tab();
    if (nvec == 1 && two_pass) {
      HCI_LAUNCH(k_sigma1_half<1>, ctx->nsm * SIGMA_HALF_BLOCKS_PER_SM, 256, 0, ctx->st)(
          bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), T, bp<double>(G.diag), G.nV, c, sigma);
      HCI_LAUNCH(k_sigma1_half<2>, ctx->nsm * SIGMA_HALF_BLOCKS_PER_SM, 256, 0, ctx->st)(
          bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), T, bp<double>(G.diag), G.nV, c, sigma);
    } else if (nvec == 1)
      HCI_LAUNCH(k_sigma1_half<0>, ctx->nsm * SIGMA_HALF_BLOCKS_PER_SM, 256, 0, ctx->st)(
          bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), T, bp<double>(G.diag), G.nV, c, sigma);
    else
      HCI_LAUNCH(k_sigma_half, grid_for(G.nV * 32, 256, ctx->nsm * 16), 256, 0, ctx->st)(
          bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), T, bp<double>(G.diag), G.nV, c, sigma, nvec);
  } else if (nvec == 1) {
    auto* k = G.sig_whole ? k_sigma1<8, true> : G.sig_block == 16 ? k_sigma1<16, false> : k_sigma1<8, false>;
    HCI_LAUNCH(k, (unsigned)(G.sig_warps / (G.sig_block * G.sig_rounds)), G.sig_block * 32, 0, ctx->st)(
        bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), bp<int32_t>(G.seg_col[0]), bp<double>(G.seg_val[0]),
        bp<double>(G.diag), G.nV, bp<int32_t>(G.sig_plan), G.sig_rounds, G.sig_chunk, c, sigma, sig_head(G), stop);
    if (!G.sig_whole)
      HCI_LAUNCH(k_sigma_heads, (unsigned)((G.sig_warps + 127) / 128), 128, 0, ctx->st)(
          bp<int64_t>(G.rowptr), bp<int32_t>(G.sig_plan), G.sig_warps, G.sig_chunk, sig_head(G), sigma, stop);
  } else {
    HCI_LAUNCH(k_sigma, grid_for(G.nV * 32, 256, ctx->nsm * 16), 256, 0, ctx->st)(
        bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), bp<int32_t>(G.seg_col[0]), bp<double>(G.seg_val[0]),
        bp<double>(G.diag), G.nV, c, sigma, nvec);
  }
  HCI_CUDA(ctx, cudaGetLastError());
  prof_toc(ctx, HCI_PH_SIGMA);
  return HCI_OK;
}

hci_status sigma_tail(hci_ctx* ctx, int64_t r0, const double* c, double* out) {
  Graph& G = ctx->graph;
  if (G.direct || r0 >= G.nV) return HCI_OK;
  HCI_LAUNCH(k_sigma_tail, grid_for((G.nV - r0) * 32, 256), 256, 0, ctx->st)(
      bp<int64_t>(G.rowptr), bp<int64_t>(G.rowstart), G.tab(), r0, G.nV, c, out);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

hci_status to_internal(hci_ctx* ctx, const double* sorted, double* internal, int nvec) {
  const Graph& G = ctx->graph;
  HCI_LAUNCH(k_gather_vec, grid_for(G.nV * nvec, 256), 256, 0, ctx->st)(sorted, bp<int32_t>(ctx->graph.i2s), G.nV,
                                                                        nvec, internal);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

hci_status to_sorted(hci_ctx* ctx, const double* internal, double* sorted, int nvec) {
  const Graph& G = ctx->graph;
  HCI_LAUNCH(k_gather_vec, grid_for(G.nV * nvec, 256), 256, 0, ctx->st)(internal, bp<int32_t>(ctx->graph.s2i), G.nV,
                                                                        nvec, sorted);
  HCI_CUDA(ctx, cudaGetLastError());
  return HCI_OK;
}

extern "C" hci_status hci_sigma(hci_ctx* ctx, const uint64_t* keys, int64_t nV, const double* c, double* sigma,
                                int nvec) {
  if (!ctx) return hci_fail(nullptr, HCI_ERR_INVALID, "hci_sigma: null context");
  if (nV <= 0 || nvec <= 0) return hci_fail(ctx, HCI_ERR_INVALID, "hci_sigma: empty space or no vectors");
  if (!keys || !c || !sigma) return hci_fail(ctx, HCI_ERR_INVALID, "hci_sigma: null pointer");
  HCI_TRY(graph_ensure(ctx, keys, nV));
  HCI_TRY(ensure_buf(ctx, ctx->d_perm, (size_t)2 * nV * nvec * 8));
  double* ci = bp<double>(ctx->d_perm);
  double* si = ci + (int64_t)nV * nvec;
  HCI_TRY(to_internal(ctx, c, ci, nvec));
  HCI_TRY(sigma_apply(ctx, ci, si, nvec));
  return to_sorted(ctx, si, sigma, nvec);
}
