// Neighbour search: the NK nearest images of every atom (14 for the Euclidean
// order, 18 for the topological one) under the FP64 distance contract.
//
//   k_knn       one thread per atom: collect, sort, decide
//   k_knn_rest  one warp per atom that k_knn left undecided
//
// k_knn reads the 27 cells around the atom once.  A radius chosen from their
// occupancy admits about 24 candidates (36 for 18 neighbours), appended to a
// per-thread list in shared memory; a sorting network then orders the list in registers.  What bounds it
// is instruction issue: an insertion network run at every admitted candidate
// issued 21 k instructions per warp at 14 of 32 active lanes, because some lane
// inserts at nearly every candidate; the list costs three predicated stores per
// admitted candidate and the network runs once, with all lanes (measurements at
// the kernel).
#pragma once
#include "ptm_atom.cuh"
#include "../../include/ptm.h"

namespace ptm {

template <bool F64> struct RT { typedef float T; };
template <> struct RT<true> { typedef double T; };

__device__ __forceinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

template <bool F64>
__device__ __forceinline__ void load_atom(const FrameDesc &d, int j, typename RT<F64>::T &x,
                                          typename RT<F64>::T &y, typename RT<F64>::T &z, int &id) {
  if constexpr (F64) {
    const Atom64 *a = (const Atom64 *)d.sorted + j;
    double2 p = __ldg((const double2 *)a);
    double2 q = __ldg((const double2 *)a + 1);
    x = p.x; y = p.y; z = q.x; id = (int)__double_as_longlong(q.y);
  } else {
    float4 p = __ldg((const float4 *)d.sorted + j);
    x = p.x; y = p.y; z = p.z; id = __float_as_int(p.w);
  }
}

// Contract shift of image (a, b, c) in the input precision.
template <bool F64>
__device__ __forceinline__ void contract_shift(const FrameDesc &d, int a, int b, int c, typename RT<F64>::T &sx,
                                               typename RT<F64>::T &sy, typename RT<F64>::T &sz) {
  if constexpr (F64) {
    shift_f64(d, a, b, c, sx, sy, sz);
  } else {
    float lx, ly, lz;
    shift_f32(d, a, b, c, sx, sy, sz, lx, ly, lz);
  }
}

// The distance contract (Sec. 3 orders neighbours by distance; the paper fixes
// no precision, so the order is that of the distances between the given points
// in FP64): dr = (x_j - x_i) + shift, d2 = (dr_x^2 + dr_y^2) + dr_z^2, one
// rounded IEEE operation at a time, no fused multiply-add, float32 positions
// widened exactly.  The kernels work in FP32 with a proven error bound and
// decide in FP64 only where the FP32 values cannot order two candidates.
__device__ __forceinline__ float contract_dr(float xj, float xi, float s) { return __fadd_rn(__fsub_rn(xj, xi), s); }
__device__ __forceinline__ double contract_dr(double xj, double xi, double s) { return __dadd_rn(__dsub_rn(xj, xi), s); }
__device__ __forceinline__ float contract_d2(float a, float b, float c) {
  return __fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), __fmul_rn(c, c));
}
__device__ __forceinline__ double contract_d2(double a, double b, double c) {
  return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

// FP64 squared distance of the image (a0, a1, a2) of an atom at (xj, yj, zj):
// the ordering key.
template <typename T>
__device__ __forceinline__ double key64(const FrameDesc &d, T xj, T yj, T zj, T xi, T yi, T zi, int a0, int a1,
                                        int a2) {
  if constexpr (sizeof(T) == 4) {
    // image 0 with every FP32 difference exact (Sterbenz: |x_j - x_i| <=
    // min(|x_i|, |x_j|)): the FP64 differences are these FP32 values and the
    // zero shift adds nothing, so only the squares and sums run in FP64
    if ((a0 | a1 | a2) == 0) {
      const float px = __fsub_rn(xj, xi), py = __fsub_rn(yj, yi), pz = __fsub_rn(zj, zi);
      if (fabsf(px) <= fminf(fabsf(xi), fabsf(xj)) && fabsf(py) <= fminf(fabsf(yi), fabsf(yj)) &&
          fabsf(pz) <= fminf(fabsf(zi), fabsf(zj)))
        return contract_d2((double)px, (double)py, (double)pz);
    }
  }
  double sx, sy, sz;
  shift_f64(d, a0, a1, a2, sx, sy, sz);
  return contract_d2(contract_dr((double)xj, (double)xi, sx), contract_dr((double)yj, (double)yi, sy),
                     contract_dr((double)zj, (double)zi, sz));
}

// Key order (FP64 d2, atom id, image).  Keys are non-negative and not NaN, so
// their bit patterns order as unsigned integers: the comparisons stay off the
// FP64 pipe.
__device__ __forceinline__ bool key_less64(uint64_t ua, int ia, int ma, uint64_t ub, int ib, int mb) {
  return ua < ub || (ua == ub && (ia < ib || (ia == ib && ma < mb)));
}

__device__ __forceinline__ bool search_complete(const FrameDesc &d, int R, float d2_last) {
  const float rg = (float)R * d.min_cell_width - __int_as_float(d.dstat[1]);
  return rg > 0.f && d2_last < rg * rg * (1.f - 1e-3f);
}

// ------------------------------------------------------- sorting networks
template <int A>
__device__ __forceinline__ void cex(uint32_t (&v)[A], int i, int j) {
  const uint32_t lo = min(v[i], v[j]), hi = max(v[i], v[j]);
  v[i] = lo;
  v[j] = hi;
}

// Odd-even merge sort (Batcher) of v[L .. L + N), N a power of two.
template <int L, int N, int S, int A>
__device__ __forceinline__ void oe_merge(uint32_t (&v)[A]) {
  if constexpr (2 * S < N) {
    oe_merge<L, N, 2 * S>(v);
    oe_merge<L + S, N, 2 * S>(v);
#pragma unroll
    for (int i = L + S; i + S < L + N; i += 2 * S) cex(v, i, i + S);
  } else {
    cex(v, L, L + S);
  }
}

template <int L, int N, int A>
__device__ __forceinline__ void oe_sort(uint32_t (&v)[A]) {
  if constexpr (N > 1) {
    oe_sort<L, N / 2>(v);
    oe_sort<L + N / 2, N / 2>(v);
    oe_merge<L, N, 1>(v);
  }
}

// The H smallest of 2 H values, ascending in v[0 .. H): both halves sorted, the
// element-wise minima of one and the other reversed (a bitonic sequence of the
// H smallest), and one bitonic merge.
template <int H>
__device__ __forceinline__ void sort_low(uint32_t (&v)[2 * H]) {
  oe_sort<0, H>(v);
  oe_sort<H, H>(v);
#pragma unroll
  for (int i = 0; i < H; i++) v[i] = min(v[i], v[2 * H - 1 - i]);
#pragma unroll
  for (int k = H / 2; k > 0; k >>= 1)
#pragma unroll
    for (int i = 0; i < H; i++)
      if (!(i & k)) cex(v, i, i | k);
}

// ------------------------------------------------------------ fast search
#define PTM_KNN_BLOCK 128
// CAP: entries of the candidate list (9 bytes a thread).  AIM: candidates the
// search radius aims at (the atom itself counts), above the NK + 1 that decide an
// atom by enough for the shells of the lattices (fcc holds 12, 18, 42 atoms
// within its first shells, bcc 8, 14, 26), below the capacity.  BLOCKS: resident
// blocks per SM (36 and 72 KB of lists a block).
template <int NK> struct KnnShape {
  static constexpr int CAP = NK == PTM_KNN ? 32 : 64, AIM = NK == PTM_KNN ? 24 : 36, BLOCKS = NK == PTM_KNN ? 6 : 3;
};
constexpr size_t knn_smem_bytes(int nk) { return (size_t)PTM_KNN_BLOCK * (nk == PTM_KNN ? 32 : 64) * 9; }

// Cells hold about 7 atoms (192 in 27) where the frame fills its box.  A cluster in a box of
// vacuum has hundreds of times as many, in a few cells that are far from evenly filled: a
// radius guessed from their filling is much too wide, and two or three gathers read
// everything again.  With more than PTM_KNN_CROWDED atoms in the 27 cells
//   - up to PTM_KNN_CROWDED_LAUNCH atoms in the launch (half for float64 input), too few warps
//     to hide a thread's loads, atoms with nearly all of their frame in reach are left to
//     the warp search: 3,000 atoms in a box of 7 diameters 0.31 ms a call, 0.60 with knn_crowded;
//     8,000 0.83 and 1.28, 16,000 2.4 and 2.4; float64 3,000 0.42 and 0.60, 8,000 1.7 and 1.2;
//   - the radius is guessed from the fullest cell where the cells are filled evenly (the
//     inside of a cluster of several cells);
//   - otherwise knn_crowded reads them once, and so it does after a gather that shows the
//     guess to be far off.
// ms a call, with guesses and gathers alone and now: 64 frames of 1,500 atoms in boxes of 3
// diameters 1.09 and 0.80, 20 frames of 20,000 in 10 diameters 23.5 and 13.7, one
// frame of 24,000 in 10 diameters 7.9 and 3.9, of 60,000 in 10 22.6 and 9.8 (and 2.04,
// 59.9, 10.9 and 17.3 with all of them left to the warp search or a sampled radius).
#define PTM_KNN_CROWDED 512
#define PTM_KNN_CROWDED_LAUNCH 8192

// Per-thread candidate list in shared memory, entry i at [i][thread]: FP32
// squared distance, sorted slot, image code (m + 1 in two bits per axis).
struct KnnList {
  float *v;
  int *j;
  uint8_t *img;
  __device__ __forceinline__ float &V(int i) const { return v[i * PTM_KNN_BLOCK]; }
  __device__ __forceinline__ int &J(int i) const { return j[i * PTM_KNN_BLOCK]; }
  __device__ __forceinline__ uint8_t &M(int i) const { return img[i * PTM_KNN_BLOCK]; }
};
#define PTM_IMG_OWN (1 << 4 | 1 << 2 | 1)

template <int CAP>
__device__ __forceinline__ KnnList knn_list(unsigned char *smem) {
  KnnList l;
  l.v = (float *)smem + threadIdx.x;
  l.j = (int *)smem + CAP * PTM_KNN_BLOCK + threadIdx.x;
  l.img = smem + 8 * CAP * PTM_KNN_BLOCK + threadIdx.x;
  return l;
}

// The cells within one of cell (bx, by, bz), the own column first: visit(ca, cb,
// mx, my, mz) with ca .. cb consecutive cells of one column in image (mx, my,
// mz).  A column whose z range does not wrap is one run of the sorted order.
template <typename V>
__device__ __forceinline__ void for_cells27(const FrameDesc &d, int bx, int by, int bz, V &&visit) {
  const int nbx = d.nb[0], nby = d.nb[1], nbz = d.nb[2];
#pragma unroll 1
  for (int ix = 0; ix < 3; ix++) {
    int cx = bx + (ix == 2 ? -1 : ix), mx = 0;
    if (cx < 0) { cx += nbx; mx = -1; } else if (cx >= nbx) { cx -= nbx; mx = 1; }
    if (mx && !d.pbc[0]) continue;
#pragma unroll 1
    for (int iy = 0; iy < 3; iy++) {
      int cy = by + (iy == 2 ? -1 : iy), my = 0;
      if (cy < 0) { cy += nby; my = -1; } else if (cy >= nby) { cy -= nby; my = 1; }
      if (my && !d.pbc[1]) continue;
      int z0 = bz - 1, z1 = bz + 1;
      if (!d.pbc[2]) { z0 = max(z0, 0); z1 = min(z1, nbz - 1); }
      const bool column = z0 >= 0 && z1 < nbz;
      const int cbase = (cx * nby + cy) * nbz;
#pragma unroll 1
      for (int r = column ? 2 : 0; r < 3; r++) {
        int ca = cbase + z0, cb = cbase + z1, mz = 0;
        if (!column) {
          int cz = bz - 1 + r;
          if (cz < 0) { cz += nbz; mz = -1; } else if (cz >= nbz) { cz -= nbz; mz = 1; }
          ca = cb = cbase + cz;
        }
        visit(ca, cb, mx, my, mz);
      }
    }
  }
}

// Two candidates whose FP32 squared distances (of FP32 pairs, below) differ by more than
// this are in FP64 order, `v` the NK-th smallest: |d2_32 - d2_64| <= u (7 v) + 4 sqrt(v)
// tau, where each component is within 2 u of its FP64 value (relative) and tau
// (absolute), and the squares and sums add 3 u v.  A hundredth more covers the
// candidate after the last: one further away is not close.
__device__ __forceinline__ float knn_band(const FrameDesc &d, float v) {
  const float u = 5.9604645e-8f, vmax = 1.01f * v;
  return 2.f * (8.5f * u * vmax + 4.f * (sqrtf(vmax) + d.tau) * d.tau);
}

// Turns (a, b, c), the image of the atom at slot j as the atom at slot i sees it in the input's
// positions, into its image in positions wrapped into the cell (slots swapped: back).
// `wrapped`: whether any atom of the frame is (d.dstat[0]).
__device__ __forceinline__ void cell_image(const FrameDesc &d, bool wrapped, int i, int j, int &a, int &b, int &c) {
  if (!wrapped) return;
  int i0, i1, i2, j0, j1, j2;
  img_unpack(__ldg(d.wrapv + i), i0, i1, i2);
  img_unpack(__ldg(d.wrapv + j), j0, j1, j2);
  a += j0 - i0; b += j1 - i1; c += j2 - i2;
}

// Position at hs + ls less the shift of a lattice image (s + r, FP32 pair), as a pair h + l.
__device__ __forceinline__ void shift_pair(float hs, float ls, float s, float r, float &h, float &l) {
  float e;
  two_sum(hs, -s, h, e);
  l = (ls + e) - r;
}

// Append every candidate with d2 < T of the 27 cells to the list; returns their
// number (entries past CAP are counted, not stored).  The own atom is one of
// them, with d2 = 0.
//
// Positions are FP32 pairs h + l (SPLIT: float64 input, or wrapped into the
// cell; otherwise float32 input, l = 0).  A candidate's vector is (h_j - H) +
// (l_j - L) with H + L = h_i + l_i - shift, H the rounded difference and L its
// exact remainder with the shift's own (error-free sum): H lies beside h_j, so
// the large terms cancel exactly and a component's error is at most two
// roundings of the component, whatever the image shift, plus terms in u^2 of
// the positions (d.tau).
template <bool SPLIT, int CAP>
__device__ __forceinline__ int knn_gather(const FrameDesc &d, const float4 *__restrict__ hi, float4 hs, float2 ls,
                                          int bx, int by, int bz, float T, const KnnList &list) {
  int cnt = 0;
  for_cells27(d, bx, by, bz, [&](int ca, int cb, int mx, int my, int mz) {
    int j = __ldg(d.cell_start + ca);
    const int j1 = __ldg(d.cell_start + cb + 1);
    const float l0 = SPLIT ? hs.w : 0.f;
    float hx = hs.x, hy = hs.y, hz = hs.z, lx = l0, ly = ls.x, lz = ls.y;
    const bool shifted = (mx | my | mz) != 0;
    if (shifted) {
      const ShiftTables &t = *d.tab;
      const int i = (mx + 2) * 25 + (my + 2) * 5 + (mz + 2);
      shift_pair(hs.x, l0, t.s32[i][0], t.slo[i][0], hx, lx);
      shift_pair(hs.y, ls.x, t.s32[i][1], t.slo[i][1], hy, ly);
      shift_pair(hs.z, ls.y, t.s32[i][2], t.slo[i][2], hz, lz);
    }
    const uint8_t code = (uint8_t)((mx + 1) << 4 | (my + 1) << 2 | (mz + 1));
    auto test = [&](int jj, float x, float y, float z) {
      const float v = fmaf(x, x, fmaf(y, y, z * z));
      if (v < T) {
        if (cnt < CAP) { list.V(cnt) = v; list.J(cnt) = jj; list.M(cnt) = code; }
        cnt++;
      }
    };
    // U loads in flight: the loop's stores keep the compiler from moving the next
    // candidate's load above them (U = 1, 2, 4 for plain positions: 1.59, 1.84, 1.57
    // ms per 4 M atoms; 1, 2, 3 for pairs: 168, 180, 148 us per 200 k)
    constexpr int U = SPLIT ? 3 : 4;
    if (SPLIT || shifted) {
      for (; j < j1; j += U) {
        float4 p[U];
        float2 q[U];
#pragma unroll
        for (int k = 0; k < U; k++) {
          p[k] = __ldg(hi + min(j + k, j1 - 1));
          if constexpr (SPLIT) q[k] = __ldg(d.lo + min(j + k, j1 - 1));
        }
#pragma unroll
        for (int k = 0; k < U; k++) {
          if (k && j + k >= j1) break;
          if constexpr (SPLIT)
            test(j + k, (p[k].x - hx) + (p[k].w - lx), (p[k].y - hy) + (q[k].x - ly), (p[k].z - hz) + (q[k].y - lz));
          else
            test(j + k, (p[k].x - hx) - lx, (p[k].y - hy) - ly, (p[k].z - hz) - lz);
        }
      }
    } else {
      for (; j < j1; j += U) {
        float4 p[U];
#pragma unroll
        for (int k = 0; k < U; k++) p[k] = __ldg(hi + min(j + k, j1 - 1));
#pragma unroll
        for (int k = 0; k < U; k++) {
          if (k && j + k >= j1) break;
          test(j + k, p[k].x - hx, p[k].y - hy, p[k].z - hz);
        }
      }
    }
  });
  return cnt;
}

// The same for crowded cells, in one pass from the widest radius: when a lane's list is
// nearly full, every lane of the warp brings its radius in to the first gap after NK + 1
// candidates and drops what lies beyond.  T is the radius (squared) in the end: the
// list holds all candidates within it.  Returns their number: 0 where no gap leaves the
// list room (more than 24 or 56 atoms, 10 or 38 of them at one distance).
template <bool SPLIT, int NK>
__device__ __noinline__ int knn_crowded(const FrameDesc &d, const float4 *__restrict__ hi, float4 hs, float2 ls, int bx,
                                        int by, int bz, float &T, const KnnList &list) {
  constexpr int CAP = KnnShape<NK>::CAP, U = 8;        // U loads in flight
  const unsigned mask = __activemask();                // these lanes stay together
  const float l0 = SPLIT ? hs.w : 0.f;
  const int nbx = d.nb[0], nby = d.nb[1], nbz = d.nb[2];
  float hx = 0.f, hy = 0.f, hz = 0.f, lx = 0.f, ly = 0.f, lz = 0.f;
  uint8_t code = 0;
  int cell = 0, j = 0, j1 = 0, cnt = 0;
  for (;;) {
    while (j >= j1 && cell < 27) {                     // this lane's next cell, its own first
      const int ix = cell / 9, iy = cell / 3 % 3, iz = cell % 3;
      int cx = bx + (ix == 2 ? -1 : ix), cy = by + (iy == 2 ? -1 : iy), cz = bz + (iz == 2 ? -1 : iz), mx = 0, my = 0, mz = 0;
      cell++;
      if (cx < 0) { cx += nbx; mx = -1; } else if (cx >= nbx) { cx -= nbx; mx = 1; }
      if (cy < 0) { cy += nby; my = -1; } else if (cy >= nby) { cy -= nby; my = 1; }
      if (cz < 0) { cz += nbz; mz = -1; } else if (cz >= nbz) { cz -= nbz; mz = 1; }
      if ((mx && !d.pbc[0]) || (my && !d.pbc[1]) || (mz && !d.pbc[2])) continue;
      const int c = (cx * nby + cy) * nbz + cz, i = (mx + 2) * 25 + (my + 2) * 5 + (mz + 2);
      j = __ldg(d.cell_start + c);
      j1 = __ldg(d.cell_start + c + 1);
      const ShiftTables &t = *d.tab;
      shift_pair(hs.x, l0, t.s32[i][0], t.slo[i][0], hx, lx);
      shift_pair(hs.y, ls.x, t.s32[i][1], t.slo[i][1], hy, ly);
      shift_pair(hs.z, ls.y, t.s32[i][2], t.slo[i][2], hz, lz);
      code = (uint8_t)((mx + 1) << 4 | (my + 1) << 2 | (mz + 1));
    }
    if (!__any_sync(mask, j < j1)) break;
    if (j < j1) {
      float4 p[U];
      float2 q[U];
#pragma unroll
      for (int k = 0; k < U; k++) {
        p[k] = __ldg(hi + min(j + k, j1 - 1));
        if constexpr (SPLIT) q[k] = __ldg(d.lo + min(j + k, j1 - 1));
      }
#pragma unroll
      for (int k = 0; k < U; k++) {
        float x = (p[k].x - hx) - lx, y = (p[k].y - hy) - ly, z = (p[k].z - hz) - lz;
        if constexpr (SPLIT) { x = (p[k].x - hx) + (p[k].w - lx); y = (p[k].y - hy) + (q[k].x - ly); z = (p[k].z - hz) + (q[k].y - lz); }
        const float v = fmaf(x, x, fmaf(y, y, z * z));
        if (j + k < j1 && v < T) {                     // at most CAP - U entries before: there is room
          list.V(cnt) = v; list.J(cnt) = j + k; list.M(cnt) = code;
          cnt++;
        }
      }
      j += U;
    }
    if (!__any_sync(mask, cnt > CAP - U)) continue;
    uint32_t v[CAP];
#pragma unroll
    for (int i = 0; i < CAP; i++) v[i] = __float_as_uint(i < cnt ? list.V(i) : T);
    oe_sort<0, CAP>(v);
    uint32_t cut = 0;
#pragma unroll
    for (int c = CAP - U; c > NK; c--) cut = v[c] > v[c - 1] ? v[c] : cut;
    if (cut) T = __uint_as_float(cut);                 // (fewer candidates than that: T still)
    int kept = 0;
#pragma unroll 4
    for (int i = 0; i < cnt; i++) {
      const float x = list.V(i);
      if (!(x < T)) continue;
      list.V(kept) = x; list.J(kept) = list.J(i); list.M(kept) = list.M(i);
      kept++;
    }
    cnt = kept;
    if (cnt > CAP - U) { cnt = 0; cell = 27; j = j1 = 0; }
  }
  return cnt;
}

// NK nearest images of the atom at sorted slot s, written to out[t * n], t = 0 ..
// NK - 1; false when k_knn_rest must decide (the NK-th neighbour may lie outside
// the 27 cells, or no radius admits a fitting number of candidates).
//
// The radius is that of a sphere holding AIM atoms at the density of the 27
// cells, at most what they are sure to cover; too many or too few candidates
// rescale it, and crowded cells are read another way (PTM_KNN_CROWDED; `launch`: atoms
// of the launch, all its frames together).  The list is sorted once by its FP32
// values with the entry number in the low bits; if the NK + 1 smallest (or the NK in
// it and the radius) then differ by more than the error band, their order is the FP64
// order.  Otherwise the values are sorted again without entry numbers, close ones form runs, and a run's candidates are
// ordered by the FP64 key (d2, atom id, image); a run across slot NK takes
// every candidate within the band.
template <bool F64, bool SPLIT, int NK>
__device__ __forceinline__ bool knn_fast(const FrameDesc &d, int s, int bx, int by, int bz, bool wrapped, int2 *out,
                                         int64_t nst, const KnnList &list, int64_t launch) {
  typedef typename RT<F64>::T IN;
  constexpr int CAP = KnnShape<NK>::CAP;
  constexpr float AIM = KnnShape<NK>::AIM;
  constexpr uint32_t LOW = CAP - 1;
  const float rg = d.min_cell_width - __int_as_float(d.dstat[1]);
  if (!(rg > 0.f)) return false;
  const float Tmax = rg * rg * (1.f - 1e-3f);
  const float4 *__restrict__ hi = SPLIT ? d.hi : (const float4 *)d.sorted;
  const float4 hs = __ldg(hi + s);
  float2 ls = make_float2(0.f, 0.f);
  if constexpr (SPLIT) ls = __ldg(d.lo + s);
  int cnt = 0, atoms = 0, cells = 0;
  for_cells27(d, bx, by, bz, [&](int ca, int cb, int, int, int) {
    atoms += __ldg(d.cell_start + cb + 1) - __ldg(d.cell_start + ca);
    cells += cb - ca + 1;
  });
  float filled = (float)atoms;                       // atoms in as many cells filled evenly
  bool uneven = false;
  if (atoms > PTM_KNN_CROWDED) {
    if (launch <= PTM_KNN_CROWDED_LAUNCH >> F64 && atoms > (int)(d.n - d.n / 16)) return false;
    int most = 0;
    for_cells27(d, bx, by, bz, [&](int ca, int cb, int, int, int) {
      for (int c = ca; c <= cb; c++) most = max(most, __ldg(d.cell_start + c + 1) - __ldg(d.cell_start + c));
    });
    // (without the constant, whose weight falls as the atoms in reach grow, the surfaces of
    // large clusters leave the guess: 32,000 atoms in 2 diameters 0.68 -> 0.75 ms)
    filled = (float)most * (float)cells;
    uneven = filled > 3.f * (float)atoms + 1536.f;
  }
  const float r3 = AIM * 0.2387324f * d.cell_vol * __fdividef((float)cells, filled);
  float T = uneven ? Tmax : fminf(Tmax, exp2f(0.6666667f * __log2f(r3)));
  for (int attempt = 0; !uneven; attempt++) {
    cnt = knn_gather<SPLIT, CAP>(d, hi, hs, ls, bx, by, bz, T, list);
    if (cnt > NK && cnt <= CAP) break;
    if (cnt <= NK && (attempt == 3 || T >= Tmax)) return false;
    uneven = cnt > CAP && (attempt == 3 || (attempt ? cnt > 4 * CAP : cnt > 16 * CAP && cnt > atoms / 2));
    const float f = exp2f(0.6666667f * __log2f(__fdividef(AIM, (float)cnt)));
    if (!uneven) T = fminf(Tmax, T * (cnt > CAP ? f : fmaxf(f, 1.2f)));
  }
  if (uneven) {
    cnt = knn_crowded<SPLIT, NK>(d, hi, hs, ls, bx, by, bz, T, list);
    if (cnt <= NK) return false;
  }
  // image of list entry i: the cells' image, less the wraps of the two atoms
  auto image = [&](int j, int code, int &a, int &b, int &c) {
    a = (code >> 4) - 1; b = (code >> 2 & 3) - 1; c = (code & 3) - 1;
    if constexpr (SPLIT) cell_image(d, wrapped, j, s, a, b, c);
  };
  auto put = [&](int t, int i) {
    const int j = list.J(i);
    int a, b, c;
    image(j, list.M(i), a, b, c);
    out[t * nst] = make_int2(j, img_pack(a, b, c));
  };
  uint32_t v[CAP];
#pragma unroll 1
  for (int round = 0;; round++) {
#pragma unroll
    for (int i = 0; i < CAP; i++) {
      // past the list T stands for whatever the radius left out (with NK neighbours and no
      // more inside the widest radius, as in fcc's first two shells for NK = 18, the
      // next one need not be known)
      uint32_t x = __float_as_uint(T) | (round == 0 ? LOW : 0u);
      if (i < cnt) {
        x = __float_as_uint(list.V(i));
        if (round == 0) x = (x & ~LOW) | (uint32_t)i;
        else if (x == 0u && list.J(i) == s && list.M(i) == PTM_IMG_OWN) x = 0xffffffffu;   // the atom itself
      }
      v[i] = x;
    }
    sort_low<CAP / 2>(v);
    if (round == 1) break;
    const float band = knn_band(d, list.V(v[NK] & LOW));
    // v[0] is the atom itself (d2 = 0, unless another lies on it: then the first
    // gap is within the band); the entry after the last neighbour counts with
    // its low bits cleared, a bound for every entry beyond it
    bool decided = true;
    float prev = 0.f;
#pragma unroll
    for (int t = 1; t <= NK + 1; t++) {
      const float e = t <= NK ? list.V(v[t] & LOW) : __uint_as_float(v[t] & ~LOW);
      decided &= e - prev > band;
      prev = e;
    }
    if (decided) {
#pragma unroll
      for (int t = 0; t < NK; t++) put(t, (int)(v[t + 1] & LOW));
      return true;
    }
  }
  // ---- some ranks undecided: L[0 .. NK] ascending without the atom itself
  auto L = [&](int t) { return __uint_as_float(v[t]); };
  const float band = knn_band(d, L(NK - 1));
  uint32_t close = 0;                                // bit t: slots t and t + 1 in one run
#pragma unroll
  for (int t = 0; t < NK; t++) close |= (uint32_t)(L(t + 1) - L(t) <= band) << t;
  const bool crossing = (close >> (NK - 1)) & 1;
  const float limit = crossing ? L(NK - 1) + band : L(NK - 1);
  if (!(limit < T)) return false;                    // the list may not hold the whole last run
  if (!F64 && close) count_here(d, C_KNN64);
  IN xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  uint64_t key[CAP];                                 // local memory: indexed by entry, the same one in every lane
  uint64_t open = 0;                                 // entries placed by key
  for (int i = 0; i < cnt; i++) {
    const float x = list.V(i);
    const int j = list.J(i);
    if (!(x <= limit) || (x == 0.f && j == s && list.M(i) == PTM_IMG_OWN)) continue;
    int r0 = 0;                                      // first slot holding this value (NK - 1 beyond)
#pragma unroll
    for (int t = 0; t < NK - 1; t++) r0 += L(t) < x;
    const uint32_t below = ~close & ((1u << r0) - 1u);
    const int rs = below ? 32 - __clz(below) : 0;    // the run: slots rs .. hi - 1
    const int re = min(r0 + __ffs(~(close >> r0)), NK);
    if (re - rs == 1 && !(re == NK && crossing)) { put(rs, i); continue; }
    IN xj, yj, zj;
    int idj, a, b, c;
    load_atom<F64>(d, j, xj, yj, zj, idj);
    image(j, list.M(i), a, b, c);
    key[i] = (uint64_t)__double_as_longlong(key64(d, xj, yj, zj, xi, yi, zi, a, b, c));
    list.V(i) = __int_as_float(rs);                  // the value is not needed any more
    open |= 1ull << i;
  }
  for (uint64_t m = open; m; m &= m - 1) {
    const int i = __ffsll((long long)m) - 1, rs = __float_as_int(list.V(i));
    const uint64_t ki = key[i];
    int r = rs;
    for (uint64_t o = open; o; o &= o - 1) {
      const int k = __ffsll((long long)o) - 1;
      if (k == i || __float_as_int(list.V(k)) != rs) continue;
      const uint64_t kk = key[k];
      bool less = kk < ki;
      if (kk == ki) {                                // equal distances: by atom id, then image
        IN x, y, z;
        int ii, ik, a, b, c, p, q, w;
        load_atom<F64>(d, list.J(i), x, y, z, ii);
        load_atom<F64>(d, list.J(k), x, y, z, ik);
        image(list.J(i), list.M(i), a, b, c);
        image(list.J(k), list.M(k), p, q, w);
        less = ik < ii || (ik == ii && img_pack(p, q, w) < img_pack(a, b, c));
      }
      r += less;
    }
    if (r < NK) put(r, i);                           // beyond the NK nearest otherwise
  }
  return true;
}

// One atom of k_knn; an undecided one is appended to the list of k_knn_rest.
template <bool F64, int NK>
__device__ __forceinline__ void knn_atom(const FrameDesc &d, int s, int64_t launch, int2 *rows, unsigned char *smem,
                                         int *rest, int *rest_count) {
  const int64_t nst = d.n;
  int2 *out = rows + (s - d.atom_offset);
  if (__ldg(d.wrapv + s) == PTM_EXCLUDED) {           // excluded by the binning: no neighbours
#pragma unroll
    for (int t = 0; t < NK; t++) out[t * nst] = make_int2(-1, 0);
    return;
  }
  const int b = __ldg(d.sbin + s);
  const int bz = b % d.nb[2], byx = b / d.nb[2];
  const int by = byx % d.nb[1], bx = byx / d.nb[1];
  const KnnList list = knn_list<KnnShape<NK>::CAP>(smem);
  const bool wrapped = d.dstat[0] != 0;
  bool done;
  if (F64 || wrapped) done = knn_fast<F64, true, NK>(d, s, bx, by, bz, wrapped, out, nst, list, launch);
  else done = knn_fast<F64, false, NK>(d, s, bx, by, bz, wrapped, out, nst, list, launch);
  if (!done) rest[atomicAdd(rest_count, 1)] = s;
}

// ------------------------------------------------------- the general search
// Bound on |d2_32 - d2_64| for an FP32 contract value v whose image shift has
// length at most S (u = 2^-24).  Each component of the FP32 vector is within
// 2u (|dr_c| + |s_c|) of the FP64 one (the difference, the shift's rounding to
// FP32 and the sum each round once); squaring and the two sums add 3u v.  So
// |d2_32 - d2_64| <= u (7 v + 4 |dr| |s|) + 8 u^2 (v + S^2); the constants
// below leave room for |dr| estimated from v and for rounding in this bound.
__device__ __forceinline__ float knn_err(float v, float S) {
  const float u = 5.9604645e-8f;
  return u * (8.5f * v + 4.5f * sqrtf(v) * S + 9.f * u * S * S);
}

// The NK nearest images of atom s by the full key (FP64 d2, atom id, image), R
// growing until the NK-th distance lies inside the radius the scanned cells are
// guaranteed to cover; each R adds the cells of its shell to the list so far.  One
// warp: every lane walks a cell of its own, and lane t holds the t-th smallest key
// so far, so an insertion is a ballot and a shift by one lane.  For float32 input
// a candidate whose FP32 distance, less its error bound, exceeds the current
// NK-th key cannot enter and skips the FP64 evaluation.  Few atoms come here and
// the kernel lasts as long as its slowest: the 58 of a 2^20-atom frame took 0.40 ms
// with a thread each and lists in local memory, 0.20 ms with a warp reading column
// by column and starting over at each R, 0.06 ms now.
template <bool F64, int NK>
__device__ void knn_rest_atom(const FrameDesc &d, int s, int2 *rows) {
  typedef typename RT<F64>::T T;
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  T xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  const int b = __ldg(d.sbin + s);
  const int bz = b % d.nb[2], byx = b / d.nb[2];
  const int by = byx % d.nb[1], bx = byx / d.nb[1];
  const int wrap = __ldg(d.wrapv + s);
  if (wrap == PTM_EXCLUDED) {                            // excluded by the binning: no neighbours
    if (lane < NK) rows[(int64_t)lane * d.n + (s - d.atom_offset)] = make_int2(-1, 0);
    return;
  }
  int wi0, wi1, wi2;
  img_unpack(wrap, wi0, wi1, wi2);
  const int nbx = d.nb[0], nby = d.nb[1], nbz = d.nb[2];
  const uint64_t INF = 0x7ff0000000000000ull;
  uint64_t lk = INF, last = INF;                       // this lane's key; the NK-th key,
  float last32 = INFINITY;                             // ... and the slack, rounded up to FP32
  // float32 input keeps one key more where it is within 2^-16 of the NK-th (in units
  // of its last place; infinity turns into a NaN, which cuts nothing), to tell whether
  // FP64 was needed between the two
  constexpr int KEPT = F64 ? NK : NK + 1;
  constexpr uint64_t SLACK = F64 ? 0 : 1ull << 36;
  int lid = 0x7fffffff, lj = -1, limg = 0x7fffffff, found = -1;
  for (int R = 1; R <= PTM_RMAX; R++) {
    const int side = 2 * R + 1;
    for (int c0 = 0; c0 < side * side * side; c0 += 32) {
      // this lane's cell: offsets (ix, iy, iz) in [-R, R]^3, not in an earlier shell
      const int c = c0 + lane;
      const int iz = c % side - R, iy = c / side % side - R, ix = c / (side * side) - R;
      int cx = bx + ix, cy = by + iy, cz = bz + iz;
      const int mx = floordiv(cx, nbx), my = floordiv(cy, nby), mz = floordiv(cz, nbz);
      const bool in_shell = ix <= R && (R == 1 || max(abs(ix), max(abs(iy), abs(iz))) == R) && (d.pbc[0] || mx == 0) &&
                            (d.pbc[1] || my == 0) && (d.pbc[2] || mz == 0);
      cx -= mx * nbx; cy -= my * nby; cz -= mz * nbz;
      int j = 0, j1 = 0;
      if (in_shell) {
        const int cell = (cx * nby + cy) * nbz + cz;
        j = __ldg(d.cell_start + cell);
        j1 = __ldg(d.cell_start + cell + 1);
      }
      // A lane walks its cell, or where one cell holds more than that takes (a cluster in a
      // box of vacuum may sit in a few cells) the warp walks them one after another
      const int most = __reduce_max_sync(ALL, j1 - j), trips = __reduce_add_sync(ALL, (j1 - j + 31) >> 5);
      const bool together = most > trips;
      for (unsigned cells = together ? __ballot_sync(ALL, j < j1) : 1u; cells; cells &= cells - 1) {
        const int src0 = __ffs(cells) - 1;
        int jj = j, je = j1, nx = mx, ny = my, nz = mz;
        if (together) {
          jj = __shfl_sync(ALL, j, src0) + lane; je = __shfl_sync(ALL, j1, src0);
          nx = __shfl_sync(ALL, mx, src0); ny = __shfl_sync(ALL, my, src0); nz = __shfl_sync(ALL, mz, src0);
        }
        for (; __any_sync(ALL, jj < je); jj += together ? 32 : 1) {
          uint64_t key = INF;
          int idj = 0x7fffffff, img = 0x7fffffff;
          if (jj < je) {
            T xj, yj, zj;
            load_atom<F64>(d, jj, xj, yj, zj, idj);
            const int w = __ldg(d.wrapv + jj);
            int w0, w1, w2;
            img_unpack(w, w0, w1, w2);
            const int a0 = nx + wi0 - w0, a1 = ny + wi1 - w1, a2 = nz + wi2 - w2;
            bool in = !(jj == s && a0 == 0 && a1 == 0 && a2 == 0) && w != PTM_EXCLUDED;
            if (in) {
              T sx, sy, sz;
              contract_shift<F64>(d, a0, a1, a2, sx, sy, sz);
              const T v = contract_d2(contract_dr(xj, xi, sx), contract_dr(yj, yi, sy), contract_dr(zj, zi, sz));
              img = img_pack(a0, a1, a2);
              if constexpr (!F64) {
                const float S = sqrtf(sx * sx + sy * sy + sz * sz) * 1.0001f;
                in = !(v - 1.25f * knn_err(v, S) > last32);
              }
              if (in) {
                double k64;
                if constexpr (F64) k64 = v;
                else k64 = key64(d, xj, yj, zj, xi, yi, zi, a0, a1, a2);
                key = (uint64_t)__double_as_longlong(k64);
              }
            }
          }
          unsigned m = __ballot_sync(ALL, key < INF && key <= last + SLACK);
          while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            const uint64_t ck = __shfl_sync(ALL, key, src);
            const int cid = __shfl_sync(ALL, idj, src), cimg = __shfl_sync(ALL, img, src), cj = __shfl_sync(ALL, jj, src);
            const unsigned at = __ballot_sync(ALL, key_less64(ck, cid, cimg, lk, lid, limg)) & ((1u << KEPT) - 1u);
            if (!at) continue;                             // not below the last key kept any more
            const uint64_t uk = __shfl_up_sync(ALL, lk, 1);
            const int uid = __shfl_up_sync(ALL, lid, 1), uj = __shfl_up_sync(ALL, lj, 1),
                      uimg = __shfl_up_sync(ALL, limg, 1);
            const int first = __ffs(at) - 1;               // the keys are sorted: every lane above moves up
            if (lane == first) { lk = ck; lid = cid; lj = cj; limg = cimg; }
            else if (lane > first) { lk = uk; lid = uid; lj = uj; limg = uimg; }
            last = __shfl_sync(ALL, lk, NK - 1);
            if constexpr (!F64) last32 = __double2float_ru(__longlong_as_double((long long)(last + SLACK)));
          }
        }
      }
    }
    if (search_complete(d, R, __double2float_ru(__longlong_as_double((long long)last)))) {
      if (R > 1 && lane == 0) count(d, C_KNN_WIDE);
      found = NK;
      break;
    }
    if (!d.pbc[0] && !d.pbc[1] && !d.pbc[2] && R >= max(nbx, max(nby, nbz))) {
      found = __popc(__ballot_sync(ALL, lane < NK && lj >= 0));
      break;
    }
  }
  if (found < 0 && lane == 0) count(d, C_KNN_FAIL);
  if constexpr (!F64) {
    // counted where the FP32 values that k_knn goes by leave two neighbours within its band
    const bool split = d.dstat[0] != 0, mine = lane <= NK && lj >= 0;
    const float4 *hi = split ? d.hi : (const float4 *)d.sorted;
    const float4 hs = __ldg(hi + s);
    float v = INFINITY;
    if (mine) {
      const float4 p = __ldg(hi + lj);
      float2 ls = make_float2(0.f, 0.f), q = ls;
      int a, b, c;
      img_unpack(limg, a, b, c);
      if (split) {
        ls = __ldg(d.lo + s);
        q = __ldg(d.lo + lj);
        cell_image(d, true, s, lj, a, b, c);
      }
      const float l0 = split ? hs.w : 0.f, q0 = split ? p.w : 0.f;
      float hx = hs.x, hy = hs.y, hz = hs.z, lx = l0, ly = ls.x, lz = ls.y;
      if (a | b | c) {
        float sx, sy, sz, rx, ry, rz;
        shift_f32(d, a, b, c, sx, sy, sz, rx, ry, rz);
        shift_pair(hs.x, l0, sx, rx, hx, lx);
        shift_pair(hs.y, ls.x, sy, ry, hy, ly);
        shift_pair(hs.z, ls.y, sz, rz, hz, lz);
      }
      const float x = (p.x - hx) + (q0 - lx), y = (p.y - hy) + (q.x - ly), z = (p.z - hz) + (q.y - lz);
      v = fmaf(x, x, fmaf(y, y, z * z));
    }
    const int have = min(NK, __popc(__ballot_sync(ALL, mine)));
    const float before = __shfl_up_sync(ALL, v, 1), nk = __shfl_sync(ALL, v, max(have, 1) - 1);
    if (__any_sync(ALL, mine && lane > 0 && v - before <= knn_band(d, nk)) && lane == 0) count(d, C_KNN64);
  }
  if (lane < NK) rows[(int64_t)lane * d.n + (s - d.atom_offset)] = lane < found ? make_int2(lj, limg) : make_int2(-1, 0);
}

}  // namespace ptm
