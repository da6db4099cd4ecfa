// Device code of libptm.so: the per-atom classification and the cell-list
// kernels (Larsen, Schmidt & Schiotz, "Robust Structural Identification via
// Polyhedral Template Matching").
//
// Device pipeline for one frame, all on the caller's stream:
//   k_bin      fractional coordinates, cell of each atom (cell list)
//   k_scan_*   exclusive scan of the cell counts
//   k_scatter  atoms copied into cell order as float4 (x, y, z, id)
//   k_knn      one thread per atom: its 14 nearest images, as a neighbour list
//              (ptm_knn.cuh; for the topological order the 18 nearest, from
//              which k_topo in ptm_topo.cuh makes the list)
//   k_knn_rest one warp per atom that k_knn left undecided
//   k_hulls    one thread per atom: hulls, graph codes, template lookup
//   k_match    one thread per atom: QCP, selection, outputs
// The phases run as separate kernels so that the warps of an SM share one
// phase of the method and its code (the instruction cache held none of the
// fused per-atom program).
#pragma once
#include "ptm_knn.cuh"

namespace ptm {

// ---------------------------------------------------------- per-atom state
// Per-atom selection state.  Plain scalars (no arrays) so that it stays in
// registers; snapshot k = 6, 12, 14 keeps its Weinberg labelling and table entry.
struct Best {
  float b1, b2;                 // best and second-best FP32 RMSD^2
  int K, cand;                  // winning snapshot (6, 12, 14) and candidate index
  int fp64;                     // the winner's eigenvalue needed the FP64 solve
  uint64_t lam6, lam12, lam14;  // Weinberg labelling per snapshot
  int ent6, ent12, ent14;       // table entry per snapshot, -1 = none
  __device__ __forceinline__ uint64_t lam(int K) const { return K == 6 ? lam6 : (K == 12 ? lam12 : lam14); }
  __device__ __forceinline__ int ent(int K) const { return K == 6 ? ent6 : (K == 12 ? ent12 : ent14); }
};

// What one atom adds to the matching counters.
struct MatchCounts { int scored, points, matched; };

// Template slots of neighbours 0 .. K - 1 (nibble j) under the correspondence given
// by the Weinberg labelling and the table candidate.
__device__ __forceinline__ uint64_t slots_of(int K, uint64_t lab, uint64_t cand) {
  uint64_t slots = 0;
#pragma unroll 2
  for (int j = K - 1; j >= 0; j--) slots = slots << 4 | (uint64_t)nib(cand, nib(lab, j) - 1);
  return slots;
}

// S_ab = sum_j w_{slot(j), a} dr_{j, b} over K neighbours, dr_{j, b} at q[(3 j + b)
// * PTM_BLOCK].  Because the template barycentre is the origin and slot 0 (the
// centre) sits at it, the data barycentre drops out of S.
__device__ __forceinline__ void cov_matrix(int K, const float *q, const float4 *tplw, uint64_t slots, float (&Sm)[3][3]) {
#pragma unroll
  for (int a = 0; a < 3; a++)
#pragma unroll
    for (int b = 0; b < 3; b++) Sm[a][b] = 0.f;
#pragma unroll 2
  for (int j = 0; j < K; j++) {
    const float4 w = __ldg(tplw + (int)(slots & 15));
    slots >>= 4;
    const float x = q[(3 * j) * PTM_BLOCK], y = q[(3 * j + 1) * PTM_BLOCK], z = q[(3 * j + 2) * PTM_BLOCK];
    Sm[0][0] = fmaf(w.x, x, Sm[0][0]); Sm[0][1] = fmaf(w.x, y, Sm[0][1]); Sm[0][2] = fmaf(w.x, z, Sm[0][2]);
    Sm[1][0] = fmaf(w.y, x, Sm[1][0]); Sm[1][1] = fmaf(w.y, y, Sm[1][1]); Sm[1][2] = fmaf(w.y, z, Sm[1][2]);
    Sm[2][0] = fmaf(w.z, x, Sm[2][0]); Sm[2][1] = fmaf(w.z, y, Sm[2][1]); Sm[2][2] = fmaf(w.z, z, Sm[2][2]);
  }
}

// Barycentre of the centre and its first K neighbours, and G_v = sum |v - mean|^2.
__device__ __forceinline__ void data_moments(int K, const Scratch &sm, float &mx, float &my, float &mz, float &Gv) {
  float sx = 0, sy = 0, sz = 0, g = 0;
#pragma unroll 1
  for (int j = 0; j < K; j++) {
    const float x = sm.DX(j), y = sm.DY(j), z = sm.DZ(j);
    sx += x; sy += y; sz += z;
    g = fmaf(x, x, fmaf(y, y, fmaf(z, z, g)));
  }
  const float inv = 1.f / (float)(K + 1);
  mx = sx * inv; my = sy * inv; mz = sz * inv;
  Gv = g - (float)(K + 1) * (mx * mx + my * my + mz * mz);
}

// RMSD^2 of one candidate from its covariance (closed form after Eq. 3); the
// FP32 Newton solution is replaced by an FP64 one when the top eigenvalue is
// not well separated (normalised P'(lambda_1) below PTM_GAP).
__device__ __noinline__ float r2_fp64(float s00, float s01, float s02, float s10, float s11, float s12, float s20,
                                      float s21, float s22, float Gv, float Gw, int N) {
  double S[3][3] = {{s00, s01, s02}, {s10, s11, s12}, {s20, s21, s22}};
  Qcp<double> o;
  qcp_solve<double>(S, (double)Gv, (double)Gw, o);
  return (float)(((double)Gw - o.lam * o.lam / (double)Gv) / N);
}

__device__ __forceinline__ float cand_r2(const float (&Sm)[3][3], float Gv, float Gw, int N, int &fp64,
                                         const FrameDesc &d) {
  Qcp<float> o;
  qcp_solve<float>(Sm, Gv, Gw, o);
  float B = sqrtf(Gv * Gw);
  float gamma = o.dP / (B * B * B);
  if (!(gamma >= PTM_GAP) || o.iters >= 60) {
    fp64 = 1;
    count(d, C_QCP64);
    return fmaxf(r2_fp64(Sm[0][0], Sm[0][1], Sm[0][2], Sm[1][0], Sm[1][1], Sm[1][2], Sm[2][0], Sm[2][1], Sm[2][2],
                         Gv, Gw, N), 0.f);
  }
  fp64 = 0;
  return fmaxf((Gw - o.lam * o.lam / Gv) / (float)N, 0.f);
}

// FP32 QCP of every admissible correspondence of the matched snapshots; keeps the
// best and second-best RMSD^2 in snapshot order (6, 12, 14) and table order (the
// first of equal values wins, Algorithm 1).
//
// The candidates of the warp's atoms form one list, scored one entry per lane per
// round: atoms have 3 to 5 candidates on average but up to 26, and one loop per
// atom ran 19 rounds at 21 % of the lanes where this takes 3 to 5.  A lane
// finds its entry's atom by bisection of the lanes' running totals, fetches that
// atom's labelling and sums by shuffles and reads its vectors in place (the rows
// of a warp's lanes are neighbouring banks, and lanes of one atom broadcast); the
// atom then takes its results back in order.  Every lane of the warp calls this,
// those without an atom too.
__device__ void score_candidates(const FrameDesc &d, const Scratch &sm, const float4 *tplw, Best &bst,
                                 MatchCounts &cnt) {
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int n6 = 0, n12 = 0, n14 = 0, f6 = 0, f12 = 0, f14 = 0;
  float Gv6 = 0.f, Gv12 = 0.f, Gv14 = 0.f, mx, my, mz;
  if (bst.ent6 >= 0) { f6 = ptm_tbl[bst.ent6].first; n6 = ptm_tbl[bst.ent6].count; data_moments(6, sm, mx, my, mz, Gv6); }
  if (bst.ent12 >= 0) { f12 = ptm_tbl[bst.ent12].first; n12 = ptm_tbl[bst.ent12].count; data_moments(12, sm, mx, my, mz, Gv12); }
  if (bst.ent14 >= 0) { f14 = ptm_tbl[bst.ent14].first; n14 = ptm_tbl[bst.ent14].count; data_moments(14, sm, mx, my, mz, Gv14); }
  const int mine = n6 + n12 + n14;
  int upto = mine;                                   // running total of the lanes' candidates
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(ALL, upto, o);
    if (lane >= o) upto += x;
  }
  const int total = __shfl_sync(ALL, upto, 31), first = upto - mine;
  const uint32_t packed = (uint32_t)n6 | (uint32_t)n12 << 8, firsts = (uint32_t)f6 | (uint32_t)f12 << 10 | (uint32_t)f14 << 20;
  for (int base = 0; base < total; base += 32) {
    const int p = base + lane;
    int owner = 0;                                   // lanes whose running total is at most p
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const int x = __shfl_sync(ALL, upto, owner + o - 1);
      if (x <= p) owner += o;
    }                                                // (entries past the list: lane 31)
    const int i = p - __shfl_sync(ALL, first, owner);
    const uint32_t np = __shfl_sync(ALL, packed, owner), fp = __shfl_sync(ALL, firsts, owner);
    const uint32_t mask = __shfl_sync(ALL, d.mask, owner);
    const int m6 = np & 255, m12 = np >> 8;
    const int K = i < m6 ? 6 : (i < m6 + m12 ? 12 : 14);
    const int c = K == 6 ? (int)(fp & 1023) + i : (K == 12 ? (int)(fp >> 10 & 1023) + i - m6 : (int)(fp >> 20) + i - m6 - m12);
    const uint64_t l6 = __shfl_sync(ALL, bst.lam6, owner), l12 = __shfl_sync(ALL, bst.lam12, owner),
                   l14 = __shfl_sync(ALL, bst.lam14, owner);
    const float g6 = __shfl_sync(ALL, Gv6, owner), g12 = __shfl_sync(ALL, Gv12, owner), g14 = __shfl_sync(ALL, Gv14, owner);
    float r2 = INFINITY;
    int fp64 = 0;
    if (p < total) {
      const uint64_t cand = __ldg((const unsigned long long *)&ptm_cand[c]);
      const int S = (int)(cand >> 60) & 7;
      if (mask >> S & 1) {
        cnt.scored++;
        cnt.points += K + 1;
        float Sm[3][3];
        const float4 *tpl = tplw + S * 15;
        cov_matrix(K, sm.q + ((threadIdx.x & ~31) | owner), tpl,
                   slots_of(K, K == 6 ? l6 : (K == 12 ? l12 : l14), cand), Sm);
        r2 = cand_r2(Sm, K == 6 ? g6 : (K == 12 ? g12 : g14), __ldg(tpl).w, K + 1, fp64, d);
      }
    }
    // the results of this lane's atom among this round's, in candidate order
    const int lo = max(first - base, 0), hi = min(upto - base, 32);
    const int trips = __reduce_max_sync(ALL, max(hi - lo, 0));
    for (int t = 0; t < trips; t++) {
      const int src = lo + t;
      const float x = __shfl_sync(ALL, r2, min(src, 31));
      const int xf = __shfl_sync(ALL, fp64, min(src, 31));
      if (src >= hi) continue;
      if (x < bst.b1) {
        const int k = base + src - first;            // candidate of this atom
        bst.b2 = bst.b1; bst.b1 = x; bst.fp64 = xf;
        bst.K = k < n6 ? 6 : (k < n6 + n12 ? 12 : 14);
        bst.cand = k < n6 ? f6 + k : (k < n6 + n12 ? f12 + k - n6 : f14 + k - n6 - n12);
      } else if (x < bst.b2) {
        bst.b2 = x;
      }
    }
  }
}

// Canonical correspondence: the paper leaves open which of the equivalent
// correspondences of a match is reported; this library reports the smallest
// member of its orbit under the template's rotation group.  Nibble 15 - s holds
// the neighbour rank of template slot s, so the orbit minimum, read slot 1
// first, is the numerically smallest packing.  A rotation brings the rank at the
// slot it maps slot 1 to into slot 1, so only the rotations that map slot 1 to
// the first neighbour's slot among slot 1's images can give the minimum: 2 of
// fcc's 24, 3 of bcc's, 1 of hcp's 6 (every packing: 0.17 ns per atom).
__device__ uint64_t canonical_corr(int S, int K, uint64_t slots) {
  const uint8_t *off = ptm_coset_off[S];
  int g0 = 0, g1 = 0;
  for (int j = 0; j < K; j++) {
    const int slot = nib(slots, j);
    g0 = __ldg(off + slot);
    g1 = __ldg(off + slot + 1);
    if (g1 > g0) break;
  }
  uint64_t best = ~0ull;
  for (int g = g0; g < g1; g++) {
    const uint64_t inv = __ldg((const unsigned long long *)&ptm_group_inv[__ldg(ptm_coset + g)]);
    uint64_t cur = 0, left = slots;
#pragma unroll 2
    for (int j = 1; j <= K; j++) {
      cur |= (uint64_t)j << (60 - 4 * nib(inv, (int)(left & 15)));
      left >>= 4;
    }
    best = cur < best ? cur : best;
  }
  return best;
}

// FP64 selection over every candidate of the matched snapshots (Algorithm 1,
// inner loops), from FP64 neighbour vectors.  Exact ties, which the paper does
// not resolve, are read as: RMSD^2 within PTM_TIE goes to the earlier template
// (SC, FCC, HCP, ICO, BCC), then to the smaller canonical correspondence.
// Returns (K << 16) | candidate index, or -1; *scored counts the candidates.
__device__ __noinline__ int select_fp64(const FrameDesc &d, const Best &bst, const double (&ex)[PTM_KNN],
                                        const double (&ey)[PTM_KNN], const double (&ez)[PTM_KNN], int *scored) {
  double best_r2 = INFINITY;
  int bK = -1, bc = -1, bS = 99, ns = 0;
  uint64_t bcp = ~0ull;
  // pass 0 finds the minimum, pass 1 picks among the candidates tied with it
  for (int pass = 0; pass < 2; pass++) {
    for (int si = 0; si < 3; si++) {
      const int K = si == 0 ? 6 : (si == 1 ? 12 : 14);
      int e = bst.ent(K);
      if (e < 0) continue;
      uint64_t lab = bst.lam(K);
      double m[3] = {0, 0, 0}, g = 0;
      for (int j = 0; j < K; j++) { m[0] += ex[j]; m[1] += ey[j]; m[2] += ez[j]; g += ex[j] * ex[j] + ey[j] * ey[j] + ez[j] * ez[j]; }
      for (int c = 0; c < 3; c++) m[c] /= (K + 1);
      double Gv = g - (K + 1) * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
      const int first = ptm_tbl[e].first, ncand = ptm_tbl[e].count;
      for (int ci = first; ci < first + ncand; ci++) {
        uint64_t cand = ptm_cand[ci];
        int S = (int)(cand >> 60) & 7;
        if (!(d.mask >> S & 1)) continue;
        if (pass == 0) ns++;
        double Sm[3][3] = {{0}}, Gw = 0;
        for (int j = 0; j < K; j++) {
          int slot = nib(cand, nib(lab, j) - 1);
          const double *w = ptm_tpl64[S][slot];
          Sm[0][0] += w[0] * ex[j]; Sm[0][1] += w[0] * ey[j]; Sm[0][2] += w[0] * ez[j];
          Sm[1][0] += w[1] * ex[j]; Sm[1][1] += w[1] * ey[j]; Sm[1][2] += w[1] * ez[j];
          Sm[2][0] += w[2] * ex[j]; Sm[2][1] += w[2] * ey[j]; Sm[2][2] += w[2] * ez[j];
        }
        for (int slot = 0; slot <= K; slot++)
          Gw += ptm_tpl64[S][slot][0] * ptm_tpl64[S][slot][0] + ptm_tpl64[S][slot][1] * ptm_tpl64[S][slot][1] +
                ptm_tpl64[S][slot][2] * ptm_tpl64[S][slot][2];
        Qcp<double> o;
        qcp_solve<double>(Sm, Gv, Gw, o);
        double r2 = fmax((Gw - o.lam * o.lam / Gv) / (K + 1), 0.0);
        if (pass == 0) {
          best_r2 = fmin(best_r2, r2);
        } else if (r2 <= best_r2 + PTM_TIE) {
          uint64_t cp = canonical_corr(S, K, slots_of(K, lab, cand));
          if (S < bS || (S == bS && cp < bcp)) { bS = S; bcp = cp; bK = K; bc = ci; }
        }
      }
    }
  }
  if (scored) *scored = ns;
  return bK > 0 ? (bK << 16) | bc : -1;
}

// FP64 neighbour vector of neighbour (sorted slot js, image img) of an atom at
// (xi, yi, zi): (x_j - x_i) + n.H with the shift exactly as the contract rounds it.
template <bool F64>
__device__ __forceinline__ void vec_fp64(const FrameDesc &d, typename RT<F64>::T xi, typename RT<F64>::T yi,
                                         typename RT<F64>::T zi, int js, int img, double &x, double &y, double &z) {
  typedef typename RT<F64>::T T;
  T xj, yj, zj;
  int idj;
  load_atom<F64>(d, js, xj, yj, zj, idj);
  int a, b, c;
  img_unpack(img, a, b, c);
  double sx, sy, sz;
  shift_f64(d, a, b, c, sx, sy, sz);
  x = ((double)xj - (double)xi) + sx;
  y = ((double)yj - (double)yi) + sy;
  z = ((double)zj - (double)zi) + sz;
}

// Rare path: the best FP32 candidates of the atom at sorted slot s lie within
// PTM_BAND.  Every candidate is scored again in FP64 from neighbour vectors
// recomputed in FP64 from the input positions, with select_fp64's result.  The warp
// does it together, a candidate per lane and neighbour t's vector in lane t: few atoms
// come here (20 of a 2^20-atom frame), but one thread took half a millisecond over two
// passes of up to 26 candidates, and the kernel waited for the last of them (calls:
// 2^20-atom polycrystal 2.44 -> 1.97 ms, 4 M atoms 7.55 -> 7.03 ms).  All lanes call
// this with the same arguments.  Returns (K << 16) | candidate index, or -1.
template <bool F64>
__device__ __noinline__ int rerank_warp(const FrameDesc *dp, int s, int e6, int e12, int e14, uint64_t lam6,
                                        uint64_t lam12, uint64_t lam14) {
  constexpr unsigned ALL = 0xffffffffu;
  typedef typename RT<F64>::T T;
  const FrameDesc &d = *dp;
  const int lane = threadIdx.x & 31;
  T xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  double ex = 0, ey = 0, ez = 0;
  if (lane < PTM_KNN) {
    const int2 e = __ldg(d.nbr + (int64_t)lane * d.n + (s - d.atom_offset));
    if (e.x >= 0) vec_fp64<F64>(d, xi, yi, zi, e.x, e.y, ex, ey, ez);
  }
  const int n6 = e6 >= 0 ? ptm_tbl[e6].count : 0, n12 = e12 >= 0 ? ptm_tbl[e12].count : 0,
            n14 = e14 >= 0 ? ptm_tbl[e14].count : 0, total = n6 + n12 + n14;
  // this lane's candidate of the round, in list order (6, 12, 14): its RMSD^2
  int K = 0, ci = -1, S = 0;
  uint64_t lab = 0, cand = 0;
  auto score = [&](int p) -> double {
    ci = -1;
    K = p < n6 ? 6 : (p < n6 + n12 ? 12 : 14);
    if (p < total) {
      const int c = K == 6 ? ptm_tbl[e6].first + p : (K == 12 ? ptm_tbl[e12].first + p - n6 : ptm_tbl[e14].first + p - n6 - n12);
      cand = __ldg((const unsigned long long *)&ptm_cand[c]);
      S = (int)(cand >> 60) & 7;
      if (d.mask >> S & 1) ci = c;
    }
    lab = K == 6 ? lam6 : (K == 12 ? lam12 : lam14);
    double m[3] = {0, 0, 0}, g = 0, Sm[3][3] = {{0}}, Gw = 0;
    for (int j = 0; j < PTM_KNN; j++) {
      const double x = __shfl_sync(ALL, ex, j), y = __shfl_sync(ALL, ey, j), z = __shfl_sync(ALL, ez, j);
      if (j >= K || ci < 0) continue;
      m[0] += x; m[1] += y; m[2] += z;
      g += x * x + y * y + z * z;
      const double *w = ptm_tpl64[S][nib(cand, nib(lab, j) - 1)];
      Sm[0][0] += w[0] * x; Sm[0][1] += w[0] * y; Sm[0][2] += w[0] * z;
      Sm[1][0] += w[1] * x; Sm[1][1] += w[1] * y; Sm[1][2] += w[1] * z;
      Sm[2][0] += w[2] * x; Sm[2][1] += w[2] * y; Sm[2][2] += w[2] * z;
    }
    if (ci < 0) return INFINITY;
    for (int c = 0; c < 3; c++) m[c] /= (K + 1);
    const double Gv = g - (K + 1) * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
    for (int slot = 0; slot <= K; slot++)
      Gw += ptm_tpl64[S][slot][0] * ptm_tpl64[S][slot][0] + ptm_tpl64[S][slot][1] * ptm_tpl64[S][slot][1] +
            ptm_tpl64[S][slot][2] * ptm_tpl64[S][slot][2];
    Qcp<double> o;
    qcp_solve<double>(Sm, Gv, Gw, o);
    return fmax((Gw - o.lam * o.lam / Gv) / (K + 1), 0.0);
  };
  double best = INFINITY, r2 = INFINITY;
  for (int base = 0; base < total; base += 32) {
    r2 = score(base + lane);
    best = fmin(best, r2);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) best = fmin(best, __shfl_xor_sync(ALL, best, o));
  // among the candidates tied with the best: earlier template, then smaller canonical
  // correspondence, then list order
  int found = -1;
  uint32_t fS = 99;
  uint64_t fcp = ~0ull;
  for (int base = 0; base < total; base += 32) {
    if (total > 32) r2 = score(base + lane);
    const bool tied = ci >= 0 && r2 <= best + PTM_TIE;
    const uint64_t cp = tied ? canonical_corr(S, K, slots_of(K, lab, cand)) : ~0ull;
    const uint32_t mS = __reduce_min_sync(ALL, tied ? (uint32_t)S : 99u);
    const bool in = tied && (uint32_t)S == mS;
    const uint32_t hi = __reduce_min_sync(ALL, in ? (uint32_t)(cp >> 32) : 0xffffffffu);
    const bool in2 = in && (uint32_t)(cp >> 32) == hi;
    const uint32_t lo = __reduce_min_sync(ALL, in2 ? (uint32_t)cp : 0xffffffffu);
    const unsigned who = __ballot_sync(ALL, in2 && (uint32_t)cp == lo);
    if (!who) continue;
    const uint64_t mcp = (uint64_t)hi << 32 | lo;
    const int pick = __shfl_sync(ALL, (K << 16) | ci, __ffs(who) - 1);
    if (mS < fS || (mS == fS && mcp < fcp)) { fS = mS; fcp = mcp; found = pick; }
  }
  return found;
}

// ------------------------------------------------------------ finalisation
// Binary alloy label (Sec. 6, Table 3) of atom a matched to template S with
// neighbour j at template slot nibble j of `slots`.  The counts below do not depend
// on which of the equivalent correspondences this is: a rotation of the template
// permutes its {100} planes (fcc) and keeps its shells (bcc).
__device__ __forceinline__ int8_t alloy_label(const FrameDesc &d, const Scratch &sm, int S, int K, uint64_t slots,
                                              int64_t a) {
  if (!d.species || (S != 1 && S != 4)) return PTM_ALLOY_NONE;
  const int8_t c = __ldg(d.species + a);
  uint32_t same = 0;                                 // slots whose atom is of the centre's species
#pragma unroll 4
  for (int j = 0; j < K; j++) {
    same |= (uint32_t)(__ldg(d.species + sm.NID(j)) == c) << (int)(slots & 15);
    slots >>= 4;
  }
  if (S == 1) {            // FCC: slots 1-4 in z = 0, 5-8 in y = 0, 9-12 in x = 0
    int sp = 0, op = 0;
#pragma unroll
    for (int p = 0; p < 3; p++) {
      const uint32_t plane = same >> (1 + 4 * p) & 15u;
      sp += plane == 15u;
      op += plane == 0u;
    }
    if (sp == 3) return PTM_ALLOY_PURE;
    if (sp == 1 && op == 2) return PTM_ALLOY_L10;
    if (sp == 2 && op == 1) return PTM_ALLOY_L12_MAJ;
    if (op == 3) return PTM_ALLOY_L12_MIN;
  } else {                 // BCC: slots 1-8 first shell, 9-14 second shell
    const uint32_t in = same >> 1 & 255u, out = same >> 9 & 63u;
    if (in == 255u && out == 63u) return PTM_ALLOY_PURE;
    if (in == 0u && out == 63u) return PTM_ALLOY_B2;
  }
  return PTM_ALLOY_NONE;
}

// Eigenvalue and quaternion of a winner whose top eigenvalue is not well
// separated, in FP64 from the same covariance (rare; out of line).
__device__ __noinline__ void winner_fp64(const float (&Sm)[3][3], float Gv, float Gw, float &lam, float (&q)[4]) {
  double S64[3][3];
  for (int a = 0; a < 3; a++) for (int b = 0; b < 3; b++) S64[a][b] = Sm[a][b];
  Qcp<double> o64;
  qcp_solve<double>(S64, (double)Gv, (double)Gw, o64);
  double q64[4];
  qcp_quat<double>(o64.K, o64.lam, q64);
  lam = (float)o64.lam;
  for (int i = 0; i < 4; i++) q[i] = (float)q64[i];
}

// Outputs of the winner; returns whether the atom is matched (Sec. 5.1).
__device__ bool finalize(const FrameDesc &d, const Scratch &sm, const float4 *tplw, const Best &bst, int idi) {
  const int K = bst.K;
  const uint64_t lab = bst.lam(K);
  const uint64_t cand = __ldg((const unsigned long long *)&ptm_cand[bst.cand]);
  const int S = (int)(cand >> 60) & 7;
  const uint64_t slots = slots_of(K, lab, cand);
  tplw += S * 15;
  float Sm[3][3];
  cov_matrix(K, sm.q + sm.t, tplw, slots, Sm);
  float mx, my, mz, Gv;
  data_moments(K, sm, mx, my, mz, Gv);
  const float Gw = __ldg(tplw).w;
  float lam, q[4];
  {
    Qcp<float> o;
    qcp_solve<float>(Sm, Gv, Gw, o);
    float B = sqrtf(Gv * Gw);
    if (bst.fp64 || !(o.dP / (B * B * B) >= PTM_GAP)) {
      float S1[3][3], lam1, q1[4];                   // copies: only this path puts them in memory
      for (int a = 0; a < 3; a++) for (int b = 0; b < 3; b++) S1[a][b] = Sm[a][b];
      winner_fp64(S1, Gv, Gw, lam1, q1);
      lam = lam1;
      for (int i = 0; i < 4; i++) q[i] = q1[i];
    } else {
      qcp_quat<float>(o.K, o.lam, q);
      lam = o.lam;
    }
  }
  const float s = lam / Gv;
  float R[3][3];
  quat_matrix<float>(q, R);
  // explicit residual of Eq. 3 at the optimum (avoids the cancellation of the
  // closed form near RMSD 0); the centre pairs with template slot 0 (origin)
  float r2 = 0.f;
  {
    float ux = -s * mx, uy = -s * my, uz = -s * mz;
    r2 = ux * ux + uy * uy + uz * uz;
  }
  float lsum = sqrtf(mx * mx + my * my + mz * mz);
#pragma unroll 1
  for (int j = 0; j < K; j++) {
    float4 w = __ldg(tplw + nib(slots, j));
    float vx = sm.DX(j) - mx, vy = sm.DY(j) - my, vz = sm.DZ(j) - mz;
    float rx = R[0][0] * w.x + R[0][1] * w.y + R[0][2] * w.z;
    float ry = R[1][0] * w.x + R[1][1] * w.y + R[1][2] * w.z;
    float rz = R[2][0] * w.x + R[2][1] * w.y + R[2][2] * w.z;
    float ex = s * vx - rx, ey = s * vy - ry, ez = s * vz - rz;
    r2 += ex * ex + ey * ey + ez * ez;
    lsum += sqrtf(vx * vx + vy * vy + vz * vz);
  }
  const float rmsd = sqrtf(r2 / (float)(K + 1));
  const int64_t a = idi;
  if (!(rmsd <= d.rmsd_max)) {
    // unmatched after the RMSD_max cut (Sec. 5.1)
    if (d.structure) d.structure[a] = PTM_NONE;
    if (d.alloy) d.alloy[a] = PTM_ALLOY_NONE;
    if (d.rmsd) d.rmsd[a] = INFINITY;
    if (d.scale) d.scale[a] = 0.f;
    if (d.quat) { d.quat[4 * a] = 1.f; d.quat[4 * a + 1] = 0.f; d.quat[4 * a + 2] = 0.f; d.quat[4 * a + 3] = 0.f; }
    if (d.strain) for (int i = 0; i < 9; i++) d.strain[9 * a + i] = 0.f;
    if (d.corr) for (int i = 0; i < 15; i++) d.corr[15 * a + i] = -1;
    if (d.vm) d.vm[a] = 0.f;
    if (d.rf) for (int i = 0; i < 3; i++) d.rf[3 * a + i] = 0.f;
    return false;
  }
  // correspondence: smallest member of its orbit (R12), atom ids per slot
  const uint64_t cp = canonical_corr(S, K, slots);
  if (d.structure) d.structure[a] = (int8_t)(S + 1);
  if (d.rmsd) d.rmsd[a] = rmsd;
  if (d.scale) d.scale[a] = s;
  if (d.corr) {
    int32_t *row = d.corr + 15 * a;
    row[0] = idi;
#pragma unroll 2
    for (int sl = 1; sl < 15; sl++) row[sl] = sl <= K ? sm.NID(nib(cp, 15 - sl) - 1) : -1;
  }
  // orientation in the fundamental zone: the equivalent rotation Q g with the
  // largest |w| (smallest angle); ties keep the earlier group element (Sec. 7)
  if (d.quat || d.rf) {
    float bw = -1.f, bq[4] = {1.f, 0.f, 0.f, 0.f};
    for (int g = ptm_group_off[S]; g < ptm_group_off[S + 1]; g++) {
      const float4 e = __ldg((const float4 *)ptm_group_quat[g]);
      const float gq[4] = {e.x, e.y, e.z, e.w};
      float o0 = q[0] * gq[0] - q[1] * gq[1] - q[2] * gq[2] - q[3] * gq[3];
      if (fabsf(o0) > bw) {
        bw = fabsf(o0);
        bq[0] = o0;
        bq[1] = q[0] * gq[1] + q[1] * gq[0] + q[2] * gq[3] - q[3] * gq[2];
        bq[2] = q[0] * gq[2] - q[1] * gq[3] + q[2] * gq[0] + q[3] * gq[1];
        bq[3] = q[0] * gq[3] + q[1] * gq[2] - q[2] * gq[1] + q[3] * gq[0];
      }
    }
    float sg = bq[0] < 0.f ? -1.f : 1.f;
    if (d.quat) for (int i = 0; i < 4; i++) d.quat[4 * a + i] = sg * bq[i];
    // Rodrigues-Frank vector of the fundamental-zone orientation (Sec. 7)
    if (d.rf) for (int i = 0; i < 3; i++) d.rf[3 * a + i] = (sg * bq[i + 1]) / (sg * bq[0]);
  }
  // strain (Sec. 8, Eq. 6-7): both sets barycentred and scaled to mean distance
  // 1; the isotropic templates give pinv(V) = V^T / (G_w / 3), so
  // A = 3 S^T / (G_w l_data); then P = (A A^T)^(1/2), U proper.
  if (d.strain || d.vm) {
    const float ldat = lsum / (float)(K + 1);
    const float f = 3.f / (Gw * ldat);
    float A[3][3], AA[3][3], X[3][3];
    for (int i = 0; i < 3; i++) for (int j = 0; j < 3; j++) A[i][j] = f * Sm[j][i];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) AA[i][j] = A[i][0] * A[j][0] + A[i][1] * A[j][1] + A[i][2] * A[j][2];
    jacobi3(AA, X);
    float s0 = sqrtf(fmaxf(AA[0][0], 0.f)), s1 = sqrtf(fmaxf(AA[1][1], 0.f)), s2 = sqrtf(fmaxf(AA[2][2], 0.f));
    if (det3<float>(A) < 0.f) {         // U must stay proper: flip the smallest singular value
      if (s0 <= s1 && s0 <= s2) s0 = -s0;
      else if (s1 <= s2) s1 = -s1;
      else s2 = -s2;
    }
    const float sig[3] = {s0, s1, s2};
    float P[3][3];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++)
        P[i][j] = X[i][0] * sig[0] * X[j][0] + X[i][1] * sig[1] * X[j][1] + X[i][2] * sig[2] * X[j][2];
    if (d.strain) for (int i = 0; i < 3; i++) for (int j = 0; j < 3; j++) d.strain[9 * a + 3 * i + j] = P[i][j];
    // von Mises shear strain (Sec. 8) in its deviatoric form, equal to
    // 3/2 sum P_ij^2 - 1/2 (tr P)^2 but free of its cancellation near P = I
    if (d.vm) {
      const float t = (P[0][0] + P[1][1] + P[2][2]) / 3.f;
      const float e0 = P[0][0] - t, e1 = P[1][1] - t, e2 = P[2][2] - t;
      const float off = P[0][1] * P[0][1] + P[0][2] * P[0][2] + P[1][2] * P[1][2] +
                        P[1][0] * P[1][0] + P[2][0] * P[2][0] + P[2][1] * P[2][1];
      d.vm[a] = sqrtf(1.5f * (e0 * e0 + e1 * e1 + e2 * e2 + off));
    }
  }
  if (d.alloy) d.alloy[a] = alloy_label(d, sm, S, K, slots, a);
  return true;
}

__device__ void write_unmatched(const FrameDesc &d, int64_t a) {
  if (d.structure) d.structure[a] = PTM_NONE;
  if (d.alloy) d.alloy[a] = PTM_ALLOY_NONE;
  if (d.rmsd) d.rmsd[a] = INFINITY;
  if (d.scale) d.scale[a] = 0.f;
  if (d.quat) { d.quat[4 * a] = 1.f; d.quat[4 * a + 1] = 0.f; d.quat[4 * a + 2] = 0.f; d.quat[4 * a + 3] = 0.f; }
  if (d.strain) for (int i = 0; i < 9; i++) d.strain[9 * a + i] = 0.f;
  if (d.corr) for (int i = 0; i < 15; i++) d.corr[15 * a + i] = -1;
  if (d.vm) d.vm[a] = 0.f;
  if (d.rf) for (int i = 0; i < 3; i++) d.rf[3 * a + i] = 0.f;
}

// Outputs of the winner in the FP64 form: the same steps as finalize, every
// metric quantity in FP64 from the FP64 neighbour vectors (results rounded to
// FP32 only when stored).
__device__ __noinline__ bool finalize_fp64(const FrameDesc &d, const Scratch &sm, int K, uint64_t lab, int ci,
                                           const double (&ex)[PTM_KNN], const double (&ey)[PTM_KNN],
                                           const double (&ez)[PTM_KNN], int idi) {
  const uint64_t cand = ptm_cand[ci];
  const int S = (int)(cand >> 60) & 7;
  double m[3] = {0, 0, 0}, g = 0;
  for (int j = 0; j < K; j++) { m[0] += ex[j]; m[1] += ey[j]; m[2] += ez[j]; g += ex[j] * ex[j] + ey[j] * ey[j] + ez[j] * ez[j]; }
  for (int c = 0; c < 3; c++) m[c] /= (K + 1);
  const double Gv = g - (K + 1) * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
  double Sm[3][3] = {{0}}, Gw = 0;
  for (int j = 0; j < K; j++) {
    const double *w = ptm_tpl64[S][nib(cand, nib(lab, j) - 1)];
    Sm[0][0] += w[0] * ex[j]; Sm[0][1] += w[0] * ey[j]; Sm[0][2] += w[0] * ez[j];
    Sm[1][0] += w[1] * ex[j]; Sm[1][1] += w[1] * ey[j]; Sm[1][2] += w[1] * ez[j];
    Sm[2][0] += w[2] * ex[j]; Sm[2][1] += w[2] * ey[j]; Sm[2][2] += w[2] * ez[j];
  }
  for (int slot = 0; slot <= K; slot++)
    Gw += ptm_tpl64[S][slot][0] * ptm_tpl64[S][slot][0] + ptm_tpl64[S][slot][1] * ptm_tpl64[S][slot][1] +
          ptm_tpl64[S][slot][2] * ptm_tpl64[S][slot][2];
  Qcp<double> o;
  qcp_solve<double>(Sm, Gv, Gw, o);
  double q[4], R[3][3];
  qcp_quat<double>(o.K, o.lam, q);
  const double s = o.lam / Gv;
  quat_matrix<double>(q, R);
  // explicit residual of Eq. 3; the centre pairs with template slot 0 (origin)
  double r2 = s * s * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
  double lsum = sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]);
  const uint64_t slots = slots_of(K, lab, cand);
  for (int j = 0; j < K; j++) {
    const double *w = ptm_tpl64[S][nib(slots, j)];
    const double vx = ex[j] - m[0], vy = ey[j] - m[1], vz = ez[j] - m[2];
    const double rx = R[0][0] * w[0] + R[0][1] * w[1] + R[0][2] * w[2];
    const double ry = R[1][0] * w[0] + R[1][1] * w[1] + R[1][2] * w[2];
    const double rz = R[2][0] * w[0] + R[2][1] * w[1] + R[2][2] * w[2];
    const double dx = s * vx - rx, dy = s * vy - ry, dz = s * vz - rz;
    r2 += dx * dx + dy * dy + dz * dz;
    lsum += sqrt(vx * vx + vy * vy + vz * vz);
  }
  const double rmsd = sqrt(r2 / (K + 1));
  const int64_t a = idi;
  if (!(rmsd <= d.rmsd_max)) { write_unmatched(d, a); return false; }
  const uint64_t cp = canonical_corr(S, K, slots);
  if (d.structure) d.structure[a] = (int8_t)(S + 1);
  if (d.rmsd) d.rmsd[a] = (float)rmsd;
  if (d.scale) d.scale[a] = (float)s;
  if (d.corr) {
    int32_t *row = d.corr + 15 * a;
    row[0] = idi;
#pragma unroll 2
    for (int sl = 1; sl < 15; sl++) row[sl] = sl <= K ? sm.NID(nib(cp, 15 - sl) - 1) : -1;
  }
  if (d.quat || d.rf) {
    double bw = -1.0, bq[4] = {1.0, 0.0, 0.0, 0.0};
    for (int gi = ptm_group_off[S]; gi < ptm_group_off[S + 1]; gi++) {
      const float *gq = ptm_group_quat[gi];
      const double o0 = q[0] * gq[0] - q[1] * gq[1] - q[2] * gq[2] - q[3] * gq[3];
      if (fabs(o0) > bw) {
        bw = fabs(o0);
        bq[0] = o0;
        bq[1] = q[0] * gq[1] + q[1] * gq[0] + q[2] * gq[3] - q[3] * gq[2];
        bq[2] = q[0] * gq[2] - q[1] * gq[3] + q[2] * gq[0] + q[3] * gq[1];
        bq[3] = q[0] * gq[3] + q[1] * gq[2] - q[2] * gq[1] + q[3] * gq[0];
      }
    }
    const double sg = bq[0] < 0.0 ? -1.0 : 1.0;
    if (d.quat) for (int i = 0; i < 4; i++) d.quat[4 * a + i] = (float)(sg * bq[i]);
    if (d.rf) for (int i = 0; i < 3; i++) d.rf[3 * a + i] = (float)((sg * bq[i + 1]) / (sg * bq[0]));
  }
  if (d.strain || d.vm) {
    const double f = 3.0 / (Gw * (lsum / (K + 1)));
    double A[3][3], AA[3][3], X[3][3];
    for (int i = 0; i < 3; i++) for (int j = 0; j < 3; j++) A[i][j] = f * Sm[j][i];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) AA[i][j] = A[i][0] * A[j][0] + A[i][1] * A[j][1] + A[i][2] * A[j][2];
    jacobi3(AA, X);
    double sg[3] = {sqrt(fmax(AA[0][0], 0.0)), sqrt(fmax(AA[1][1], 0.0)), sqrt(fmax(AA[2][2], 0.0))};
    if (det3<double>(A) < 0.0) {
      const int k = (sg[0] <= sg[1] && sg[0] <= sg[2]) ? 0 : (sg[1] <= sg[2] ? 1 : 2);
      sg[k] = -sg[k];
    }
    double P[3][3];
    for (int i = 0; i < 3; i++)
      for (int j = 0; j < 3; j++) P[i][j] = X[i][0] * sg[0] * X[j][0] + X[i][1] * sg[1] * X[j][1] + X[i][2] * sg[2] * X[j][2];
    if (d.strain) for (int i = 0; i < 3; i++) for (int j = 0; j < 3; j++) d.strain[9 * a + 3 * i + j] = (float)P[i][j];
    if (d.vm) {
      const double t = (P[0][0] + P[1][1] + P[2][2]) / 3.0;
      const double e0 = P[0][0] - t, e1 = P[1][1] - t, e2 = P[2][2] - t;
      const double off = P[0][1] * P[0][1] + P[0][2] * P[0][2] + P[1][2] * P[1][2] +
                         P[1][0] * P[1][0] + P[2][0] * P[2][0] + P[2][1] * P[2][1];
      d.vm[a] = (float)sqrt(1.5 * (e0 * e0 + e1 * e1 + e2 * e2 + off));
    }
  }
  if (d.alloy) d.alloy[a] = alloy_label(d, sm, S, K, slots, a);
  return true;
}

// Neighbour vectors for the metric steps, in rows DX / DY / DZ, and the neighbours'
// atom ids in row NID: the contract values, or for a shifted image an error-free
// FP32 sum of difference and shift.  float32 input: every neighbour's record is
// loaded in one short unrolled pass (two round trips to memory for all of them) and
// the shifted ones are redone one by one.
template <bool F64>
__device__ __forceinline__ void metric_vectors(const FrameDesc &d, const Scratch &sm, const int2 *nb, int64_t nst,
                                               typename RT<F64>::T xi, typename RT<F64>::T yi,
                                               typename RT<F64>::T zi) {
  typedef typename RT<F64>::T T;
  if constexpr (F64) {
#pragma unroll 2
    for (int t = 0; t < PTM_KNN; t++) {
      const int2 e = __ldg(nb + t * nst);
      if (e.x < 0) { sm.NID(t) = -1; sm.DX(t) = sm.DY(t) = sm.DZ(t) = 0.f; continue; }
      T xj, yj, zj;
      int idj;
      load_atom<F64>(d, e.x, xj, yj, zj, idj);
      sm.NID(t) = idj;
      int a0, a1, a2;
      img_unpack(e.y, a0, a1, a2);
      T sx, sy, sz;
      contract_shift<F64>(d, a0, a1, a2, sx, sy, sz);
      sm.DX(t) = (float)contract_dr(xj, xi, sx); sm.DY(t) = (float)contract_dr(yj, yi, sy);
      sm.DZ(t) = (float)contract_dr(zj, zi, sz);
    }
  } else {
    uint32_t shifted = 0;
    int2 e[PTM_KNN];
#pragma unroll
    for (int t = 0; t < PTM_KNN; t++) e[t] = __ldg(nb + t * nst);
#pragma unroll
    for (int t = 0; t < PTM_KNN; t++) {
      const bool none = e[t].x < 0;
      float xj, yj, zj;
      int idj;
      load_atom<F64>(d, max(e[t].x, 0), xj, yj, zj, idj);
      sm.NID(t) = none ? -1 : idj;
      sm.DX(t) = none ? 0.f : __fsub_rn(xj, xi); sm.DY(t) = none ? 0.f : __fsub_rn(yj, yi);
      sm.DZ(t) = none ? 0.f : __fsub_rn(zj, zi);
      shifted |= (uint32_t)(!none && e[t].y != img_pack(0, 0, 0)) << t;
    }
    for (; shifted; shifted &= shifted - 1) {
      const int t = __ffs(shifted) - 1;
      const int2 en = __ldg(nb + t * nst);
      float xj, yj, zj;
      int idj;
      load_atom<F64>(d, en.x, xj, yj, zj, idj);
      int a0, a1, a2;
      img_unpack(en.y, a0, a1, a2);
      float hx, hy, hz, lx, ly, lz;
      shift_f32(d, a0, a1, a2, hx, hy, hz, lx, ly, lz);
      float p, e1, q2, e2;
      two_sum(xj, -xi, p, e1); two_sum(p, hx, q2, e2); sm.DX(t) = q2 + (e1 + (e2 + lx));
      two_sum(yj, -yi, p, e1); two_sum(p, hy, q2, e2); sm.DY(t) = q2 + (e1 + (e2 + ly));
      two_sum(zj, -zi, p, e1); two_sum(p, hz, q2, e2); sm.DZ(t) = q2 + (e1 + (e2 + lz));
    }
  }
}

// FP64 contract vector of neighbour (sorted slot js, packed image img) of an atom
// at (xi, yi, zi).
template <bool F64>
__device__ __forceinline__ void vec64_row(const FrameDesc &d, typename RT<F64>::T xi, typename RT<F64>::T yi,
                                          typename RT<F64>::T zi, int js, int img, double (&v)[3]) {
  typename RT<F64>::T xj, yj, zj;
  int idj;
  load_atom<F64>(d, js, xj, yj, zj, idj);
  int a0, a1, a2;
  img_unpack(img, a0, a1, a2);
  double hx, hy, hz;
  shift_f64(d, a0, a1, a2, hx, hy, hz);
  v[0] = contract_dr((double)xj, (double)xi, hx);
  v[1] = contract_dr((double)yj, (double)yi, hy);
  v[2] = contract_dr((double)zj, (double)zi, hz);
}

// Quantisation in FP64 of the neighbours that FP32 pairs cannot decide (rare): the
// frexp exponent of their largest FP64 vector component (-100000 if all are zero),
// then q = rint(dr 2^shift) into the Q rows.  Neighbour t of the atom is the
// list entry nb[t * nst]; the Q rows are per-thread columns of shared memory
// with stride PTM_BLOCK.
template <bool F64>
__device__ __noinline__ int wide_exponent(const FrameDesc &d, typename RT<F64>::T xi, typename RT<F64>::T yi,
                                          typename RT<F64>::T zi, const int2 *nb, int64_t nst, uint32_t wide) {
  int e64 = -100000;
  for (; wide; wide &= wide - 1) {
    const int t = __ffs(wide) - 1;
    const int2 e = __ldg(nb + t * nst);
    double v[3];
    vec64_row<F64>(d, xi, yi, zi, e.x, e.y, v);
    const double m = fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2])));
    if (m > 0.0) { int et; frexp(m, &et); e64 = max(e64, et); }
  }
  return e64;
}

template <bool F64>
__device__ __noinline__ void wide_quantise(const FrameDesc &d, typename RT<F64>::T xi, typename RT<F64>::T yi,
                                           typename RT<F64>::T zi, const int2 *nb, int64_t nst, float *q,
                                           uint32_t wide, int shift) {
  const double sc = ldexp(1.0, shift);
  for (; wide; wide &= wide - 1) {
    const int t = __ffs(wide) - 1;
    const int2 e = __ldg(nb + t * nst);
    double v[3];
    vec64_row<F64>(d, xi, yi, zi, e.x, e.y, v);
    for (int c = 0; c < 3; c++) q[(3 * t + c) * PTM_BLOCK] = (float)__double2int_rn(v[c] * sc);
  }
}

// Vector of list entry e from the atom at sorted slot s, hs + ls, as FP32 pairs h + l: differences
// and shift summed without loss but for the low parts, within about 2^-44 of the
// positions and the cell.  Float64 input takes the pairs of the positions wrapped
// into the cell, float32 input the positions themselves.  Returns false for an
// image beyond the next, whose shift may be larger than that allows for.
template <bool F64>
__device__ __forceinline__ bool pair_vector(const FrameDesc &d, bool wrapped, int s, float4 hs, float2 ls, int2 e,
                                            float (&h)[3], float (&l)[3]) {
  const float4 p = __ldg((F64 ? d.hi : (const float4 *)d.sorted) + e.x);
  float2 q = make_float2(0.f, 0.f);
  int a, b, c;
  img_unpack(e.y, a, b, c);
  if constexpr (F64) {
    q = __ldg(d.lo + e.x);
    cell_image(d, wrapped, s, e.x, a, b, c);
  }
  float t0[3] = {0.f, 0.f, 0.f}, r[3] = {0.f, 0.f, 0.f};
  if (a | b | c) shift_f32(d, a, b, c, t0[0], t0[1], t0[2], r[0], r[1], r[2]);
  const float pj[3] = {p.x, p.y, p.z}, qj[3] = {F64 ? p.w : 0.f, q.x, q.y}, pi[3] = {hs.x, hs.y, hs.z},
              qi[3] = {F64 ? hs.w : 0.f, ls.x, ls.y};
#pragma unroll
  for (int k = 0; k < 3; k++) {
    float d1, e1, d2, e2;
    two_sum(pj[k], -pi[k], d1, e1);
    two_sum(d1, t0[k], d2, e2);
    const float t = __fadd_rn(e1, __fadd_rn(e2, __fadd_rn(__fsub_rn(qj[k], qi[k]), r[k])));
    h[k] = __fadd_rn(d2, t);
    l[k] = __fsub_rn(t, __fsub_rn(h[k], d2));
  }
  return max(abs(a), max(abs(b), abs(c))) <= 1;
}

// ------------------------------------------------------------ one atom
// The method for one atom runs in two kernels.  k_hulls: neighbour vectors
// from the list, their quantised copy, the incremental hull and at k = 6, 12,
// 14 the graph code and template lookup; it leaves, per atom, the matched
// snapshots' labellings and table entries (d.lam, d.ents).  k_match: QCP of
// every admissible correspondence, selection and the outputs.  `live` holds
// the lanes of this warp that entered together (all reach the warp-synchronous
// points below).

// Table entries of the snapshots k = 6, 12, 14, each + 1 in 10 bits (0 = none).
__device__ __forceinline__ uint32_t pack_ents(int e6, int e12, int e14) {
  return (uint32_t)(e6 + 1) | (uint32_t)(e12 + 1) << 10 | (uint32_t)(e14 + 1) << 20;
}

// Returns the number of orientation tests that Simulation of Simplicity decided.
template <bool F64>
__device__ int hull_atom(const FrameDesc &d, int s, const Scratch &sm, unsigned live) {
  typedef typename RT<F64>::T T;
  T xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  const int64_t sl = s - d.atom_offset;          // frame-local slot
  int nsos = 0;

  // ---- neighbours (Sec. 3): the list written by k_knn or k_topo, read in
  // place (entry t at nb[t * n]; the valid entries form a prefix).
  // Quantised copy for the exact hull predicates: q = rint(dr 2^(19 - e))
  // (half to even) on the FP64 contract vectors dr, 2^(e-1) <= max |dr_c| < 2^e
  const int2 *nb = d.nbr + sl;
  const int64_t nst = d.n;
  int cnt = 0;
  unsigned hmask;
  {
    // A float32 neighbour in the same image whose differences are exact
    // (Sterbenz: |x_j - x_i| below min(|x_i|, |x_j|)) has its FP64 vector in FP32
    // already.  The others (bit t of `wide`: shifted images, atoms near a
    // coordinate plane through the origin, every neighbour of float64 input) are
    // FP32 pairs h + l, h in the Q rows and l in rows the hull will use: scaling by a
    // power of two is exact, so rint(h 2^s) is the answer unless the rest, (h 2^s -
    // rint) + l 2^s, comes within the pair's error of one half.  Those (bit t of
    // `bad`, 3 in 1,000 atoms), and an exponent that hangs on the low parts, go to FP64
    // out of line.  (All of `wide` in FP64: quantisation 0.66 ns per float64 atom, 41 %
    // of k_hulls, and 0.22 ns per float32 atom in a 231 Angstrom box.)
    // (this thread's own words: its 24 F rows, then its 18 U rows)
    auto low = [&](int t, int c) -> uint32_t & {
      const int k = 3 * t + c;
      return k < 24 ? sm.F(k) : sm.U(k - 24);
    };
    float emaxf = 0.f, m = 0.f;
    uint32_t wide = 0, bad = 0;
    float4 hs;
    float2 ls = make_float2(0.f, 0.f);
    const bool wrapped = F64 && d.dstat[0] != 0;
    if constexpr (F64) {
      hs = __ldg(d.hi + s);
      ls = __ldg(d.lo + s);
#pragma unroll 2
      for (int t = 0; t < PTM_KNN; t++) {
        const int2 e = __ldg(nb + t * nst);
        if (e.x < 0) continue;
        cnt++;
        wide |= 1u << t;
        float h[3], l[3];
        if (!pair_vector<F64>(d, wrapped, s, hs, ls, e, h, l)) bad |= 1u << t;
#pragma unroll
        for (int c = 0; c < 3; c++) { sm.Q(t, c) = h[c]; low(t, c) = __float_as_uint(l[c]); m = fmaxf(m, fabsf(h[c])); }
      }
    } else {
      hs = make_float4(xi, yi, zi, 0.f);
#pragma unroll 7
      for (int t = 0; t < PTM_KNN; t++) {
        const int2 e = __ldg(nb + t * nst);
        if (e.x < 0) continue;
        cnt++;
        float xj, yj, zj;
        int idj;
        load_atom<false>(d, e.x, xj, yj, zj, idj);
        const float px = __fsub_rn(xj, xi), py = __fsub_rn(yj, yi), pz = __fsub_rn(zj, zi);
        const bool exact = e.y == img_pack(0, 0, 0) && fabsf(px) < fminf(fabsf(xi), fabsf(xj)) &&
                           fabsf(py) < fminf(fabsf(yi), fabsf(yj)) && fabsf(pz) < fminf(fabsf(zi), fabsf(zj));
        sm.Q(t, 0) = px; sm.Q(t, 1) = py; sm.Q(t, 2) = pz;
        if (exact) emaxf = fmaxf(emaxf, fmaxf(fabsf(px), fmaxf(fabsf(py), fabsf(pz))));
        else wide |= 1u << t;
      }
#pragma unroll 1
      for (uint32_t w = wide; w; w &= w - 1) {
        const int t = __ffs(w) - 1;
        const int2 e = __ldg(nb + t * nst);
        float h[3], l[3];
        if (!pair_vector<F64>(d, wrapped, s, hs, ls, e, h, l)) bad |= 1u << t;
#pragma unroll
        for (int c = 0; c < 3; c++) { sm.Q(t, c) = h[c]; low(t, c) = __float_as_uint(l[c]); }
        const float mt = fmaxf(fabsf(h[0]), fmaxf(fabsf(h[1]), fabsf(h[2])));
        if (e.y == img_pack(0, 0, 0) && l[0] == 0.f && l[1] == 0.f && l[2] == 0.f) {   // exact after all
          wide &= ~(1u << t);
          emaxf = fmaxf(emaxf, mt);
        }
        m = fmaxf(m, mt);
      }
      m = fmaxf(m, emaxf);
    }
    // a power of two may round up from below; far from 1 the FP32 scaling may not hold
    if (wide && ((__float_as_uint(m) & 0x7fffffu) == 0 || !(m > 0x1p-60f && m < 0x1p60f))) bad = wide;
    int e;
    frexpf(bad ? emaxf : m, &e);
    if (bad) {                                       // the exponent in FP64 then, too
      const int e64 = wide_exponent<F64>(d, xi, yi, zi, nb, nst, wide);
      if (e64 > -100000) e = emaxf > 0.f ? max(e, e64) : e64;
    }
    const float sc = ldexpf(1.f, PTM_QBITS - e);
    const float half = 0.5f - (0x1p-16f + 0x1p-42f * sc * (fabsf(hs.x) + fabsf(hs.y) + fabsf(hs.z) + 0x1p37f * d.tau));
#pragma unroll 2
    for (int t = 0; t < PTM_KNN; t++) {
      if (t >= cnt) break;
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const float y = sm.Q(t, c) * sc, r = rintf(y);
        if ((wide >> t & 1) && !(fabsf(fmaf(__uint_as_float(low(t, c)), sc, y - r)) <= half)) bad |= 1u << t;
        sm.Q(t, c) = r;
      }
    }
    if (bad) wide_quantise<F64>(d, xi, yi, zi, nb, nst, sm.q + sm.t, bad, PTM_QBITS - e);
    hmask = __ballot_sync(live, cnt >= 4);       // lanes that go on to the hulls
    if (cnt < 4) { d.ents[sl] = 0; return 0; }
  }

  // ---- hulls of the first 6, 12, 14 neighbours, built incrementally (Sec. 4)
  Best bst;
  bst.ent6 = bst.ent12 = bst.ent14 = -1;
  bst.lam6 = bst.lam12 = bst.lam14 = 0;
  const uint32_t mask = d.mask;
  int kmax = (mask & 16) ? 14 : ((mask & 14) ? 12 : 6);
  kmax = min(kmax, cnt);
  bool alive = kmax >= 6;
  int birth = 4;
  // the graphs of 12 and 14 points are looked up last: the facets of the first wait
  // in local memory until then
  bool got12 = false, got14 = false;
  uint32_t f12[20];
  if (alive) hull_init(sm, nsos);
  for (int p = 4; p <= PTM_KNN; p++) {
    // every insertion step starts warp-converged: a lane that finished (or took
    // a snapshot's longer path) waits here instead of drifting into a later
    // step alone, so the visibility tests and lookups keep full warps
    if (!__any_sync(hmask, alive)) break;
    // the hull now holds neighbours 0..p-1, all of them vertices (2 p - 4
    // facets): complete for K = 6, 12, 14.  The centre test of a snapshot rides on
    // the visibility test of point p.
    const bool want = (p == 6 && (mask & 1)) || (p == 12 && (mask & 14)) || (p == 14 && (mask & 16));
    const int nf = 2 * p - 4;
    bool centre_in = false;
    uint32_t vis = 0;
    const unsigned vmask = __ballot_sync(hmask, alive && p < kmax && !want);   // lanes testing point p,
    const unsigned bmask = __ballot_sync(hmask, alive && p < kmax && want);    // ... and the centre,
    const unsigned cmask = __ballot_sync(hmask, alive && p >= kmax && want);   // only the centre
    if (alive) {
      if (p >= kmax) { if (want) centre_in = hull_centre_inside(sm, nf, cmask, nsos); }
      else if (want) vis = hull_visibility<true>(sm, nf, p, centre_in, bmask, nsos);
      else vis = hull_visibility<false>(sm, nf, p, centre_in, vmask, nsos);
    }
    if (alive && want && centre_in) {
      if (p == 6) {
        uint64_t lab;
        int e;
        if (octahedron_lookup(sm, lab, e)) { bst.lam6 = lab; bst.ent6 = e; }
      } else if (p == 12) {
        got12 = true;
#pragma unroll 4
        for (int f = 0; f < 20; f++) f12[f] = sm.F(f);
      } else {
        got14 = true;
      }
    }
    if (!alive) continue;
    // done, p inside the hull, or a vertex swallowed
    alive = p != kmax && vis && hull_apply(sm, nf, vis, p, birth, d);
  }
#pragma unroll 1
  for (int K = 14; K >= 12; K -= 2) {
    const bool look = K == 14 ? got14 : got12;
    const unsigned lmask = __ballot_sync(hmask, look);
    if (!look) continue;
    if (K == 12) {
#pragma unroll 4
      for (int f = 0; f < 20; f++) sm.F(f) = f12[f];
    }
    uint64_t lab;
    int e;
    if (!graph_lookup(sm, K, lmask, lab, e, d)) continue;
    if (K == 12) { bst.lam12 = lab; bst.ent12 = e; }
    else { bst.lam14 = lab; bst.ent14 = e; }
  }
  d.ents[sl] = pack_ents(bst.ent6, bst.ent12, bst.ent14);
  if (bst.ent6 >= 0) d.lam[sl] = bst.lam6;
  if (bst.ent12 >= 0) d.lam[d.n + sl] = bst.lam12;
  if (bst.ent14 >= 0) d.lam[2 * d.n + sl] = bst.lam14;
  return nsos;
}

// P64 selects the FP64 form: every candidate scored and the winner's outputs
// computed in FP64 (the one-frame-per-launch comparison form).
// Every lane of the warp calls it; `active` lanes have an atom, at sorted slot s.
template <bool F64, bool P64 = false>
__device__ MatchCounts match_atom(const FrameDesc &d, int s, bool active, const Scratch &sm, const float4 *tplw) {
  typedef typename RT<F64>::T T;
  const int64_t sl = s - d.atom_offset;
  MatchCounts cnt = {0, 0, 0};
  uint32_t ents = 0;
  T xi = 0, yi = 0, zi = 0;
  int idi = 0;
  if (active) {
    ents = __ldg(d.ents + sl);
    load_atom<F64>(d, s, xi, yi, zi, idi);
  }
  if (P64 && !active) return cnt;
  if (P64 && !ents) { write_unmatched(d, idi); return cnt; }
  Best bst;
  bst.b1 = bst.b2 = INFINITY;
  bst.K = -1; bst.cand = -1; bst.fp64 = 0;
  bst.ent6 = (int)(ents & 1023) - 1;
  bst.ent12 = (int)(ents >> 10 & 1023) - 1;
  bst.ent14 = (int)(ents >> 20 & 1023) - 1;
  bst.lam6 = bst.ent6 >= 0 ? __ldg((const unsigned long long *)d.lam + sl) : 0;
  bst.lam12 = bst.ent12 >= 0 ? __ldg((const unsigned long long *)d.lam + d.n + sl) : 0;
  bst.lam14 = bst.ent14 >= 0 ? __ldg((const unsigned long long *)d.lam + 2 * d.n + sl) : 0;
  const int2 *nb = d.nbr + sl;                   // the neighbour list, entry t at nb[t * n]
  const int64_t nst = d.n;
  double ex[P64 ? PTM_KNN : 1], ey[P64 ? PTM_KNN : 1], ez[P64 ? PTM_KNN : 1];
  if constexpr (P64) {
    for (int t = 0; t < PTM_KNN; t++) {
      const int2 e = __ldg(nb + t * nst);
      if (e.x < 0) break;                          // the valid entries form a prefix
      vec_fp64<F64>(d, xi, yi, zi, e.x, e.y, ex[t], ey[t], ez[t]);
    }
  }
  if (ents) metric_vectors<F64>(d, sm, nb, nst, xi, yi, zi);
  if constexpr (!P64) {
    __syncwarp();                                  // the vectors are read across the warp
    score_candidates(d, sm, tplw, bst, cnt);
    __syncwarp();
    const bool tied = bst.K >= 0 && bst.b2 <= bst.b1 + PTM_BAND;
    if (tied) count(d, C_TIE64);
    for (unsigned m = __ballot_sync(0xffffffffu, tied); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const auto from = [&](auto x) { return __shfl_sync(0xffffffffu, x, src); };
      const FrameDesc *owner = (const FrameDesc *)from((unsigned long long)&d);
      const int w = rerank_warp<F64>(owner, from(s), from(bst.ent6), from(bst.ent12), from(bst.ent14), from(bst.lam6),
                                     from(bst.lam12), from(bst.lam14));
      if ((threadIdx.x & 31) == src && w >= 0) { bst.K = w >> 16; bst.cand = w & 0xffff; }
    }
    if (!active) return cnt;
    if (bst.K < 0) { write_unmatched(d, idi); return cnt; }     // no match, or every match masked out
  } else {
    const int w = select_fp64(d, bst, ex, ey, ez, &cnt.scored);
    if (w < 0) { write_unmatched(d, idi); return cnt; }
    const int K = w >> 16;
    cnt.matched = finalize_fp64(d, sm, K, bst.lam(K), w & 0xffff, ex, ey, ez, idi);
    return cnt;
  }
  cnt.matched = finalize(d, sm, tplw, bst, idi);
  return cnt;
}

// ------------------------------------------------------------------ kernels
// First kernel of a single-frame call: zeroes the cell counts, status words and
// counters (one launch instead of three memsets) and copies the frame's shift
// tables, passed by value, into device memory: stream ordered, so back-to-back
// asynchronous calls never share a host staging buffer.
#define PTM_STATUS_WORDS 4       // any wrap, overshoot, undecided atoms (k_knn), listed atoms (k_topo)
__global__ void k_begin(const __grid_constant__ ShiftTables t, ShiftTables *out, int *cell_count, int ncount, int *dstat,
                        unsigned long long *counters) {
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = i0; i < ncount; i += gridDim.x * blockDim.x) cell_count[i] = 0;
  if (blockIdx.x) return;
  if (threadIdx.x < PTM_STATUS_WORDS) dstat[threadIdx.x] = 0;
  if (threadIdx.x < C_NCOUNTERS) counters[threadIdx.x] = 0;
  const float *src = reinterpret_cast<const float *>(&t);
  float *dst = reinterpret_cast<float *>(out);
  for (int i = threadIdx.x; i < (int)(sizeof(ShiftTables) / 4); i += blockDim.x) dst[i] = src[i];
}

struct BinParams {
  float Hinv[9];     // fractional = x . Hinv
  float W[3];        // perpendicular cell widths
  double H[9];       // rows = cell vectors
  int nb[3];
  int pbc[3];
  int64_t n;
  int f64;
  // batches only: where this frame lives
  const void *pos;   // the frame's positions
  int *dstat;        // the frame's status words
  unsigned long long *counters;   // the call's counters (excluded atoms)
  int64_t atom_off;  // first atom of the frame in the batch order
  int cell_off;      // first cell of the frame in the batch's cell array
};

#define PTM_WRAP_TOL 1e-4f

// Cell of one atom of frame p (shared by the single-frame and batched
// binning), its lattice wrap (packed image) and how far it lies outside the
// cell (Angstrom, plus a rounding slack).  An atom with a non-finite
// coordinate, or more than PTM_FAR_PERIODS periods from the cell, is excluded:
// it gets the marker wrap PTM_EXCLUDED (no valid image packs to it), cell 0 and
// no overshoot, so it is nobody's neighbour and is itself left unmatched.
__device__ __forceinline__ int bin_atom(const BinParams &p, const void *pos, int64_t li, int &wrap, float &over) {
  float x, y, z;
  if (p.f64) {
    const double *q = (const double *)pos + 3 * li;
    x = (float)q[0]; y = (float)q[1]; z = (float)q[2];
  } else {
    const float *q = (const float *)pos + 3 * li;
    x = q[0]; y = q[1]; z = q[2];
  }
  int bc[3], w[3];
  over = 0.f;
  bool ok = true;
  for (int c = 0; c < 3; c++) {
    float f = x * p.Hinv[c] + y * p.Hinv[3 + c] + z * p.Hinv[6 + c];
    ok &= fabsf(f) < PTM_FAR_PERIODS;              // false for NaN and infinities too
    w[c] = 0;
    if (p.pbc[c] && (f < -PTM_WRAP_TOL || f >= 1.f + PTM_WRAP_TOL)) {
      w[c] = (int)floorf(f);
      f -= (float)w[c];
    }
    over = fmaxf(over, fmaxf(-f, f - 1.f) * p.W[c]);
    int b = (int)floorf(f * (float)p.nb[c]);
    bc[c] = min(max(b, 0), p.nb[c] - 1);
  }
  if (!ok) {
    wrap = PTM_EXCLUDED;
    over = 0.f;
    return 0;
  }
  // rounding of the fractional coordinates is covered by a small extra slack
  over = fmaxf(over, 0.f) + 1e-5f * fmaxf(p.W[0], fmaxf(p.W[1], p.W[2]));
  wrap = img_pack(w[0], w[1], w[2]);
  return (bc[0] * p.nb[1] + bc[1]) * p.nb[2] + bc[2];
}

__global__ void k_bin(const void *pos, BinParams p, int *cell_count, int *atom_cell, int *atom_rank,
                      int *atom_wrap, int *dstat) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  int wrap;
  float over;
  const int cell = bin_atom(p, pos, i, wrap, over);
  if (wrap == PTM_EXCLUDED) atomicAdd(p.counters + C_EXCLUDED, 1ull);
  else if (wrap != img_pack(0, 0, 0)) dstat[0] = 1;
  atomicMax(dstat + 1, __float_as_int(over));      // uniform address: the compiler aggregates per warp
  atom_cell[i] = cell;
  atom_rank[i] = atomicAdd(cell_count + cell, 1);
  atom_wrap[i] = wrap;
}

#define SCAN_BLOCK 1024
// Inclusive scan of one value per thread over a block; sh holds a word per warp.
__device__ __forceinline__ int block_scan(int v, int *sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += x;
  }
  if (lane == 31) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    int x = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    sh[lane] = x;
  }
  __syncthreads();
  return v + (w ? sh[w - 1] : 0);
}

// Exclusive scan, level 1: per-block scan of 2 elements per thread.
__global__ void k_scan_block(const int *in, int *out, int *block_sums, int n) {
  __shared__ int sh[32];
  const int a = blockIdx.x * SCAN_BLOCK * 2 + 2 * threadIdx.x, b = a + 1;
  const int va = a < n ? in[a] : 0, vb = b < n ? in[b] : 0;
  const int v = block_scan(va + vb, sh), excl = v - (va + vb);
  if (a < n) out[a] = excl;
  if (b < n) out[b] = excl + va;
  if (threadIdx.x == SCAN_BLOCK - 1) block_sums[blockIdx.x] = v;
}

// Level 2: every block sums the totals of the blocks before it (one per 2,048
// cells, a few thousand in all for 33 M atoms) and adds them to its elements; not
// launched for a single block.
__global__ void k_scan_add(int *out, const int *block_sums, int n) {
  __shared__ int sh[32];
  __shared__ int before;
  int sum = 0;
  for (int i = threadIdx.x; i < (int)blockIdx.x; i += SCAN_BLOCK) sum += block_sums[i];
  const int v = block_scan(sum, sh);
  if (threadIdx.x == SCAN_BLOCK - 1) before = v;
  __syncthreads();
  const int a = blockIdx.x * SCAN_BLOCK * 2 + 2 * threadIdx.x, b = a + 1;
  if (a < n) out[a] += before;
  if (b < n) out[b] += before;
}

// Copy of atom li of frame p into its cell-sorted slot.  Float64 input, and a
// float32 frame in which some atom lies outside the cell, also get the position
// wrapped into the cell as an FP32 pair: the neighbour search then works in FP32
// and on the 27 images, whatever the input.  An excluded atom's pair is NaN.
__device__ __forceinline__ void scatter_atom(const BinParams &p, const void *pos, int64_t li, int wrap, bool wrapped,
                                             int slot, void *sorted, float4 *hi, float2 *lo) {
  double x, y, z;
  if (p.f64) {
    const double *q = (const double *)pos + 3 * li;
    Atom64 a;
    x = a.x = q[0]; y = a.y = q[1]; z = a.z = q[2]; a.id = li;
    ((Atom64 *)sorted)[slot] = a;
  } else {
    const float *q = (const float *)pos + 3 * li;
    const float4 a = make_float4(q[0], q[1], q[2], __int_as_float((int)li));
    ((float4 *)sorted)[slot] = a;
    if (!wrapped) return;
    x = a.x; y = a.y; z = a.z;
  }
  if (wrap != img_pack(0, 0, 0)) {
    int a, b, c;
    img_unpack(wrap, a, b, c);
    x -= a * p.H[0] + b * p.H[3] + c * p.H[6];
    y -= a * p.H[1] + b * p.H[4] + c * p.H[7];
    z -= a * p.H[2] + b * p.H[5] + c * p.H[8];
    if (wrap == PTM_EXCLUDED) x = y = z = NAN;
  }
  const float hx = (float)x, hy = (float)y, hz = (float)z;
  hi[slot] = make_float4(hx, hy, hz, (float)(x - hx));
  lo[slot] = make_float2((float)(y - hy), (float)(z - hz));
}

__global__ void k_scatter(const void *pos, BinParams p, const int *atom_cell, const int *atom_rank,
                          const int *atom_wrap, const int *cell_start, const int *dstat, void *sorted, float4 *hi,
                          float2 *lo, int *sbin, int *wrapv) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const int c = atom_cell[i], wrap = atom_wrap[i];
  const int slot = cell_start[c] + atom_rank[i];
  scatter_atom(p, pos, i, wrap, dstat[0] != 0, slot, sorted, hi, lo);
  sbin[slot] = c;
  wrapv[slot] = wrap;
}

// Cell list of a small frame by one block: what k_begin, k_bin, the scan and
// k_scatter do, with the counts in shared memory.  Four launches cost more than the
// work of one block up to a few thousand atoms: 22 -> 12 us for 256 atoms, 23 -> 16
// us for 2,048; at 4,000 the block takes longer (30 against 23 us).
#define PTM_SMALL_ATOMS 2048
#define PTM_SMALL_CELLS 4096
#define PTM_SMALL_BLOCK 1024
__global__ void __launch_bounds__(PTM_SMALL_BLOCK)
    k_cells_small(const __grid_constant__ ShiftTables t, const void *pos, const __grid_constant__ BinParams p, int ncell,
                  ShiftTables *out, int *cell_start, int *dstat, unsigned long long *counters, void *sorted, float4 *hi,
                  float2 *lo, int *sbin, int *wrapv) {
  __shared__ int cells[PTM_SMALL_CELLS];
  __shared__ int sh[32];
  __shared__ int any_wrap, overs, excluded;
  constexpr int PER = PTM_SMALL_ATOMS / PTM_SMALL_BLOCK;
  const int tid = threadIdx.x;
  const float *src = reinterpret_cast<const float *>(&t);
  for (int i = tid; i < (int)(sizeof(ShiftTables) / 4); i += PTM_SMALL_BLOCK) reinterpret_cast<float *>(out)[i] = src[i];
  for (int i = tid; i < ncell; i += PTM_SMALL_BLOCK) cells[i] = 0;
  if (tid == 0) any_wrap = overs = excluded = 0;
  __syncthreads();
  int cell[PER], rank[PER], wrap[PER], omax = 0;
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int i = tid + k * PTM_SMALL_BLOCK;
    if (i >= p.n) break;
    float over;
    cell[k] = bin_atom(p, pos, i, wrap[k], over);
    rank[k] = atomicAdd(&cells[cell[k]], 1);
    if (wrap[k] == PTM_EXCLUDED) atomicAdd(&excluded, 1);
    else if (wrap[k] != img_pack(0, 0, 0)) any_wrap = 1;
    omax = max(omax, __float_as_int(over));          // over > 0: its bits order as integers
  }
  omax = __reduce_max_sync(0xffffffffu, omax);
  if ((tid & 31) == 0) atomicMax(&overs, omax);
  __syncthreads();
  // exclusive scan of the counts, a run of cells per thread
  const int run = (ncell + PTM_SMALL_BLOCK - 1) / PTM_SMALL_BLOCK, c0 = min(tid * run, ncell), c1 = min(c0 + run, ncell);
  int sum = 0;
  for (int c = c0; c < c1; c++) sum += cells[c];
  int at = block_scan(sum, sh) - sum;
  for (int c = c0; c < c1; c++) {
    const int v = cells[c];
    cells[c] = at;
    cell_start[c] = at;
    at += v;
  }
  if (tid == PTM_SMALL_BLOCK - 1) cell_start[ncell] = at;
  if (tid < C_NCOUNTERS) counters[tid] = tid == C_EXCLUDED ? excluded : 0;
  if (tid < PTM_STATUS_WORDS) dstat[tid] = tid == 0 ? any_wrap : (tid == 1 ? overs : 0);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int i = tid + k * PTM_SMALL_BLOCK;
    if (i >= p.n) break;
    const int slot = cells[cell[k]] + rank[k];
    scatter_atom(p, pos, i, wrap[k], any_wrap != 0, slot, sorted, hi, lo);
    sbin[slot] = cell[k];
    wrapv[slot] = wrap[k];
  }
}

// ------------------------------------------------------------ batched frames
// Frame of batch atom i: the last frame whose first atom is <= i.
__device__ __forceinline__ int frame_of(const int64_t *atom_off, int nframes, int64_t i) {
  int lo = 0, hi = nframes - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg((const unsigned long long *)atom_off + mid) <= (unsigned long long)i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__global__ void k_bin_batch(const BinParams *__restrict__ bp, const int64_t *__restrict__ atom_off, int nframes,
                            int64_t ntotal, int *cell_count, int *atom_cell, int *atom_rank, int *atom_wrap) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntotal) return;
  const int f = frame_of(atom_off, nframes, i);
  const BinParams &p = bp[f];
  int wrap;
  float over;
  const int cell = p.cell_off + bin_atom(p, p.pos, i - p.atom_off, wrap, over);
  if (wrap == PTM_EXCLUDED) atomicAdd(p.counters + C_EXCLUDED, 1ull);
  else if (wrap != img_pack(0, 0, 0)) p.dstat[0] = 1;
  // one atomic per frame per warp (over > 0, so its bits order as integers):
  // per-atom atomics on a frame's single status word serialise at the L2
  const unsigned same = __match_any_sync(__activemask(), f);
  const int omax = __reduce_max_sync(same, __float_as_int(over));
  if ((threadIdx.x & 31) == __ffs(same) - 1) atomicMax(p.dstat + 1, omax);
  atom_cell[i] = cell;
  atom_rank[i] = atomicAdd(cell_count + cell, 1);
  atom_wrap[i] = wrap;
}

__global__ void k_scatter_batch(const BinParams *__restrict__ bp, const int64_t *__restrict__ atom_off, int nframes,
                                int64_t ntotal, const int *atom_cell, const int *atom_rank, const int *atom_wrap,
                                const int *cell_start, void *sorted, float4 *hi, float2 *lo, int *sbin, int *wrapv) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntotal) return;
  const int f = frame_of(atom_off, nframes, i);
  const BinParams &p = bp[f];
  const int c = atom_cell[i], wrap = atom_wrap[i];
  const int slot = cell_start[c] + atom_rank[i];
  scatter_atom(p, p.pos, i - p.atom_off, wrap, p.dstat[0] != 0, slot, sorted, hi, lo);
  sbin[slot] = c - p.cell_off;
  wrapv[slot] = wrap;
}

constexpr size_t atom_smem_bytes() { return (size_t)PTM_BLOCK * SCRATCH_WORDS * 4; }
// k_match keeps only the neighbour vectors (42 words) and the neighbours' atom
// ids (14 words) per thread; the images are read from the neighbour list
constexpr int MATCH_WORDS = 42 + 14;
constexpr size_t match_smem_bytes() { return (size_t)PTM_BLOCK * MATCH_WORDS * 4; }

// Resident blocks per SM of k_hulls: 10 x (84 words x 64 threads + the 1 KB the
// driver reserves per block) fits 228 KB of shared memory, and 10 x 64 threads x
// 96 registers the register file (at 108 words and 8 blocks, 16 warps left 3 of 10
// issue slots idle: a 4 M-atom call 8.18 -> 7.49 ms, 256 frames 70.6 -> 66.7 ms).
#define PTM_ATOM_BLOCKS_PER_SM 10
// ptm_tuning.blocks_per_sm that fills the SMs with k_hulls_batch
#define PTM_TUNE_FULL 8
// k_match: 11 x (56 words x 64 threads + two descriptor copies + 1 KB) fits, at up
// to 93 registers
#define PTM_MATCH_BLOCKS_PER_SM 11
// Frames of a batch with at least this many atoms get a k_match launch of their
// own (on a 2^20-atom frame the persistent k_match_batch took 0.47 ms more than
// such a launch's 1.47 ms); the own launches alternate between the batch's stream and
// PTM_MATCH_SIDE_STREAMS side streams, so that each launch's last wave overlaps
// the next launch (the batch of 256 frames: matching 60.6 -> 48.8 ms)
#define PTM_MATCH_OWN_LAUNCH 65536
#define PTM_MATCH_SIDE_STREAMS 2

// Scratch rows of k_hulls in a block's dynamic shared memory.
__device__ __forceinline__ Scratch scratch_rows(unsigned char *smem) {
  Scratch sm;
  sm.q = (float *)smem;
  sm.nid = nullptr;                 // k_hulls reads the neighbour list in place
  sm.fac = (uint32_t *)(sm.q + 42 * PTM_BLOCK);
  sm.used = sm.fac + 24 * PTM_BLOCK;
  sm.t = threadIdx.x;
  return sm;
}

// The rows k_match uses (the others stay null).
__device__ __forceinline__ Scratch match_rows(unsigned char *smem) {
  Scratch sm;
  sm.fac = nullptr; sm.used = nullptr;
  sm.q = (float *)smem;
  sm.nid = (int *)(sm.q + 42 * PTM_BLOCK);
  sm.t = threadIdx.x;
  return sm;
}

// Normalised templates as float4 (x, y, z, .) in global memory, read through the
// read-only cache (shared memory is spent on per-thread scratch).
__device__ __forceinline__ const float4 *template_rows() { return reinterpret_cast<const float4 *>(&ptm_tpl[0][0][0]); }

// Atom of a thread in a launch that gives each warp `apw` atoms (its first lanes
// hold one each): sorted slot within the frame, -1 for a lane without an atom.
__device__ __forceinline__ int64_t spread_slot(int64_t n, int apw) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t s = w * apw + lane;
  return lane < apw && s < n ? s : -1;
}

// The frame descriptor travels by value in the kernel parameters, so back-to-back
// asynchronous calls never share a staging buffer.
template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_ATOM_BLOCKS_PER_SM) k_hulls(const __grid_constant__ FrameDesc d, int apw) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Scratch sm = scratch_rows(smem);
  const int64_t s = spread_slot(d.n, apw);
  const unsigned live = __ballot_sync(0xffffffffu, s >= 0);
  if (s < 0) return;
  const int nsos = hull_atom<F64>(d, (int)s, sm, live);
  count_warp(d, C_ATOMS, live, 1);
  count_warp(d, C_SOS, live, nsos);
}

// Bounded by instruction fetch and latency at 11 blocks per SM: its warps stand
// at different points of 50 KB of straight code, so the loops over neighbours stay
// rolled or short and the FP64 paths out of line (unrolled and inline: 80 KB; 4 M
// atoms 2.72 -> 2.48 ms).  The neighbours' loads are the exception: all in flight at
// once (-> 2.23 ms).  At 10, 9 and 8 blocks (more registers): 2.86, 2.82, 3.06 ms
// against 2.72.
template <bool F64, bool P64 = false>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_MATCH_BLOCKS_PER_SM) k_match(const __grid_constant__ FrameDesc d, int apw) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Scratch sm = match_rows(smem);
  const float4 *tplw = template_rows();
  const int64_t s = spread_slot(d.n, apw);               // frame-local slot
  const MatchCounts c = match_atom<F64, P64>(d, (int)(s + d.atom_offset), s >= 0, sm, tplw);
  count_warp(d, C_CAND, 0xffffffffu, c.scored);
  count_warp(d, C_CANDPTS, 0xffffffffu, c.points);
  count_warp(d, C_MATCHED, 0xffffffffu, c.matched);
}

// Neighbour lists of one frame, one thread per atom: NK = 14, or 18 for the
// topological order.  Measured against the insertion network and
// the FP64 arithmetic it replaced (k_knn with k_knn_rest, device time):
//   2^20-atom polycrystal, float32      1.23  -> 0.48 ms (k_knn 0.41, at 52 % of
//                                       issue; 675 -> 232 warp instructions an atom)
//   250,000 atoms, float64              6.03  -> 0.15 ms (was FP64-pipe bound)
//   202,500 atoms, unwrapped float32    4.04  -> 0.14 ms (was the general search)
//   256 frames, 31.7 M atoms            31.2  -> 15.8 ms
template <bool F64, int NK>
__global__ void __launch_bounds__(PTM_KNN_BLOCK, KnnShape<NK>::BLOCKS)
    k_knn(const __grid_constant__ FrameDesc d, int apw, int *rest, int *rest_count) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t s = spread_slot(d.n, apw);
  if (s < 0) return;
  knn_atom<F64, NK>(d, (int)s, d.n, d.nbr, smem, rest, rest_count);
}

template <bool F64, int NK>
__global__ void __launch_bounds__(PTM_KNN_BLOCK)
    k_knn_rest(const __grid_constant__ FrameDesc d, const int *rest, const int *rest_count) {
  const int n = rest ? *rest_count : (int)d.n, stride = gridDim.x * (PTM_KNN_BLOCK / 32);
  for (int i = (blockIdx.x * PTM_KNN_BLOCK + threadIdx.x) >> 5; i < n; i += stride)
    knn_rest_atom<F64, NK>(d, rest ? rest[i] : i, d.nbr);
}

// The same over a batch: each slot finds its frame; NK = 14 takes the frames in
// the Euclidean order, NK = 18 those in the topological one.
template <bool F64, int NK>
__global__ void __launch_bounds__(PTM_KNN_BLOCK, KnnShape<NK>::BLOCKS)
    k_knn_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ atom_off, int nframes,
                int64_t ntotal, int *rest, int *rest_count) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t s = (int64_t)blockIdx.x * PTM_KNN_BLOCK + threadIdx.x;
  if (s >= ntotal) return;
  const FrameDesc &d = descs[frame_of(atom_off, nframes, s)];
  if ((d.ordering == PTM_ORDER_EUCLIDEAN) != (NK == PTM_KNN)) return;
  knn_atom<F64, NK>(d, (int)s, ntotal, d.nbr, smem, rest, rest_count);
}

template <bool F64, int NK>
__global__ void __launch_bounds__(PTM_KNN_BLOCK)
    k_knn_rest_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ atom_off, int nframes,
                     const int *rest, const int *rest_count) {
  const int n = *rest_count, stride = gridDim.x * (PTM_KNN_BLOCK / 32);
  for (int i = (blockIdx.x * PTM_KNN_BLOCK + threadIdx.x) >> 5; i < n; i += stride) {
    const int s = rest[i];
    const FrameDesc &d = descs[frame_of(atom_off, nframes, s)];
    knn_rest_atom<F64, NK>(d, s, d.nbr);
  }
}

// Persistent per-atom passes over a batch: every warp pulls tiles of
// tile_atoms (a multiple of 32) consecutive slots from a global queue until the
// batch is exhausted, so uneven frames balance across the GPU and no warp waits
// for the other warp of its block.  The slots are the batch's sorted slots, or
// with a map (map_frames, map_off, nmap) a virtual numbering of the listed
// frames' atoms only: virtual slot v of listed frame k = frame_of(map_off, ...)
// is sorted slot atom_offset + v - map_off[k] of frame map_frames[k].  With
// `head` (this warp's slot of shared memory) a tile whose slots all belong to
// one frame reads that frame's descriptor from a shared copy, made when the
// frame changes.  fn(desc, slot, live): every lane, those of `live` with a slot.
template <typename Fn>
__device__ __forceinline__ void persistent_tiles(const FrameDesc *__restrict__ descs,
                                                 const int64_t *__restrict__ atom_off, int nframes, int64_t ntotal,
                                                 const int *__restrict__ map_frames, int tile_atoms,
                                                 unsigned long long *queue, FrameDesc *head, Fn &&fn) {
  const int lane = threadIdx.x & 31;
  int cached = -1;
  for (;;) {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(queue, (unsigned long long)tile_atoms);
    base = __shfl_sync(0xffffffffu, base, 0);
    if ((long long)base >= ntotal) break;
    for (int k = 0; k < tile_atoms; k += 32) {
      long long s = (long long)base + k + lane;
      const unsigned live = __ballot_sync(0xffffffffu, s < ntotal);
      if (!live) break;                  // the rest of a tile past the end (warp-uniform)
      int f = -1;
      if (s < ntotal) {
        f = frame_of(atom_off, nframes, s);
        if (map_frames) {
          s += (long long)__ldg((const long long *)&descs[__ldg(map_frames + f)].atom_offset) -
               (long long)__ldg((const long long *)atom_off + f);
          f = __ldg(map_frames + f);
        }
      }
      const int f0 = __shfl_sync(0xffffffffu, f, 0);            // lane 0 is live whenever any lane is
      if (f < 0) f = f0;
      const FrameDesc *dp = descs + f;
      if (head) {
        if (__all_sync(0xffffffffu, f == f0)) {
          if (f0 != cached) {
            const int *src = reinterpret_cast<const int *>(descs + f0);
            int *dst = reinterpret_cast<int *>(head);
            for (int w = lane; w < (int)(sizeof(FrameDesc) / 4); w += 32) dst[w] = __ldg(src + w);
            __syncwarp();
            cached = f0;
          }
          dp = head;
        }
      }
      fn(*dp, (int)s, live);
    }
  }
}

template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_ATOM_BLOCKS_PER_SM)
    k_hulls_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ atom_off, int nframes,
                  int64_t ntotal, int tile_atoms, unsigned long long *queue) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Scratch sm = scratch_rows(smem);
  persistent_tiles(descs, atom_off, nframes, ntotal, nullptr, tile_atoms, queue, nullptr,
                   [&](const FrameDesc &d, int s, unsigned live) {
                     if (!(live >> (threadIdx.x & 31) & 1)) return;
                     const int nsos = hull_atom<F64>(d, s, sm, live);
                     count_warp(d, C_ATOMS, live, 1);
                     count_warp(d, C_SOS, live, nsos);
                   });
}

// k_match over the atoms of the batch's smaller frames (the larger ones get a
// k_match launch each, with their descriptor in the kernel parameters): map_off
// is the prefix sum of the listed frames' sizes, map_frames their indices.
template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_MATCH_BLOCKS_PER_SM)
    k_match_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ map_off,
                  const int *__restrict__ map_frames, int nmap, int64_t nslots, int tile_atoms,
                  unsigned long long *queue) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Scratch sm = match_rows(smem);
  const float4 *tplw = template_rows();
  __shared__ FrameDesc heads[PTM_BLOCK / 32];
  persistent_tiles(descs, map_off, nmap, nslots, map_frames, tile_atoms, queue, &heads[threadIdx.x >> 5],
                   [&](const FrameDesc &d, int s, unsigned live) {
                     const MatchCounts c = match_atom<F64, false>(d, s, live >> (threadIdx.x & 31) & 1, sm, tplw);
                     count_warp(d, C_CAND, 0xffffffffu, c.scored);
                     count_warp(d, C_CANDPTS, 0xffffffffu, c.points);
                     count_warp(d, C_MATCHED, 0xffffffffu, c.matched);
                   });
}

}  // namespace ptm

