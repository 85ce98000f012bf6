// Accumulation of one connected pair <D_i| op |D_j> into the spin-summed
// 1- and 2-RDMs (Sec. IV), shared by the stored-connection and the
// recomputing traversals.
#pragma once

#include "hci_internal.cuh"

// One orientation of every connected pair (column id above the row id): the
// other orientation contributes the transpose (p,q,r,s) -> (q,p,s,r), added
// in k_rdm_finish.  A pair's operator strings are permutations of one
// another, so each pair adds to one entry and k_rdm_finish writes the
// permutations: alpha a -> c with beta b -> d to Hm[c][a][d][b], a same-spin
// double (holes a < b, particles c < d, either spin) to Hs[cd][ab] by pair
// index.  A single a -> b of spin S in D_j with weight w adds w to
// S1[S][b][a]; its spectator terms sum w n_k(D_j) are split into the aufbau
// occupation (expanded in k_rdm_finish) plus the orbitals where D_j's
// strings differ from the aufbau ones, accumulated in Ds[b][a][k] (the
// single's spin) and Do[b][a][k] (the other spin).
struct RdmAcc {
  double* Hm;
  double* Hs;
  double* S1;
  double* Ds;
  double* Do;
  uint64_t ref_a, ref_b;
};
// doubles of the accumulators, and where each starts
inline size_t rdm_acc_doubles(size_t n) {
  const size_t np = n * (n - 1) / 2;
  return n * n * n * n + np * np + 2 * n * n + 2 * n * n * n;
}
inline RdmAcc rdm_acc_at(double* base, size_t n, uint64_t ref_a, uint64_t ref_b) {
  const size_t np = n * (n - 1) / 2;
  RdmAcc R;
  R.Hm = base;
  R.Hs = R.Hm + n * n * n * n;
  R.S1 = R.Hs + np * np;
  R.Ds = R.S1 + 2 * n * n;
  R.Do = R.Ds + n * n * n;
  R.ref_a = ref_a;
  R.ref_b = ref_b;
  return R;
}
__host__ __device__ __forceinline__ int tri_index(int lo, int hi) { return hi * (hi - 1) / 2 + lo; }

// The three kinds of connected pair <ki| op |kj> with weight cc (phases flip
// the weight's sign bit).  FP64 products and L2 additions are what the
// accumulating kernels are bound by: a double takes one addition.

// alpha a -> c, beta b -> d
__device__ __forceinline__ void rdm_mixed(const RdmAcc& R, int n, ulonglong2 ki, ulonglong2 kj, double cc) {
  const uint64_t ha = kj.x & ~ki.x, hb = kj.y & ~ki.y;
  const int a = __ffsll((long long)ha) - 1, cp = __ffsll((long long)(ki.x & ~kj.x)) - 1;
  const int bh = __ffsll((long long)hb) - 1, d = __ffsll((long long)(ki.y & ~kj.y)) - 1;
  atomicAdd(&R.Hm[((cp * n + a) * n + d) * n + bh],
            flip_sign(cc, bits_between(kj.x, a, cp) + bits_between(kj.y, bh, d)));
}
// si <- sj, two electrons of one spin
__device__ __forceinline__ void rdm_same(const RdmAcc& R, int n, uint64_t si, uint64_t sj, double cc) {
  uint64_t holes = sj & ~si, parts = si & ~sj;
  const int a = __ffsll((long long)holes) - 1; holes &= holes - 1;
  const int bh = __ffsll((long long)holes) - 1;
  const int cp = __ffsll((long long)parts) - 1; parts &= parts - 1;
  const int d = __ffsll((long long)parts) - 1;
  const uint64_t t = sj ^ (1ull << a) ^ (1ull << cp);
  const int np = n * (n - 1) / 2;
  atomicAdd(&R.Hs[tri_index(cp, d) * np + tri_index(a, bh)],
            flip_sign(cc, bits_between(sj, a, cp) + bits_between(t, bh, d)));
}
// one electron of spin S
__device__ __forceinline__ void rdm_single(const RdmAcc& R, int n, ulonglong2 ki, ulonglong2 kj, double cc) {
  const int S = ki.x != kj.x ? 0 : 1;
  const uint64_t sj = S == 0 ? kj.x : kj.y, oj = S == 0 ? kj.y : kj.x, si = S == 0 ? ki.x : ki.y;
  const int a = __ffsll((long long)(sj & ~si)) - 1, bb = __ffsll((long long)(si & ~sj)) - 1;
  const double w = flip_sign(cc, bits_between(sj, a, bb));
  atomicAdd(&R.S1[(S * n + bb) * n + a], w);
  const uint64_t rs = S == 0 ? R.ref_a : R.ref_b, ro = S == 0 ? R.ref_b : R.ref_a;
  double* ds = R.Ds + (bb * n + a) * n;
  double* dt = R.Do + (bb * n + a) * n;
  // an orbital that differs is filled (+w) unless the aufbau one holds it
  for (uint64_t m = sj ^ rs; m; m &= m - 1) {
    const int k = __ffsll((long long)m) - 1;
    atomicAdd(ds + k, flip_sign(w, (int)(rs >> k)));
  }
  for (uint64_t m = oj ^ ro; m; m &= m - 1) {
    const int k = __ffsll((long long)m) - 1;
    atomicAdd(dt + k, flip_sign(w, (int)(ro >> k)));
  }
}

// any connected pair
__device__ __forceinline__ void rdm_accumulate(const RdmAcc& R, int n, ulonglong2 ki, ulonglong2 kj, double cc) {
  const int da = __popcll(ki.x ^ kj.x), db = __popcll(ki.y ^ kj.y);
  if (da == 2 && db == 2) rdm_mixed(R, n, ki, kj, cc);
  else if (da == 4) rdm_same(R, n, ki.x, kj.x, cc);
  else if (db == 4) rdm_same(R, n, ki.y, kj.y, cc);
  else rdm_single(R, n, ki, kj, cc);
}
