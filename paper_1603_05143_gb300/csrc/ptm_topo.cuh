// Topological neighbour ordering (Sec. 3, Eq. 5): for every atom, its 18
// nearest images (the distance contract of the Euclidean path), the area of the
// face its Voronoi cell shares with each of them (the cell taken among those 18,
// as Sec. 9 does with the Delaunay triangulation of the centre and its 18
// nearest), and the order "larger face first, then nearer".  The first 14 in
// that order replace the 14 nearest for the rest of the method.
//
// Face area of neighbour j: the bisector plane x.v_j = |v_j|^2 / 2, clipped by
// every other neighbour's half-space x.v_i <= |v_i|^2 / 2 (one half-plane at a
// time, in plane coordinates), then the shoelace formula; 0 when nothing is
// left.  Floating point cannot reproduce exact ties between equal faces (the 12
// faces of a perfect fcc cell), so areas that follow each other in descending
// order within TOPO_BAND x the mean squared distance form one group, ordered by
// the Euclidean rank (distance, atom id, image).  FP32 areas decide unless a
// gap lies within TOPO_GUARD of the band edge; then the atom's areas are
// recomputed in FP64 from FP64 neighbour vectors, by a second kernel over just
// those atoms.

namespace ptm {

#define PTM_TOPO_N 18
#define PTM_TOPO_BAND 1e-3
#define PTM_TOPO_GUARD 2e-5
#define PTM_TOPO_NEAR 1e-6f    // of the squared half-width R = 10 x the 18th distance: 1e-4 x its square
#define PTM_TOPO_VMAX 24       // FP64 polygon buffer: 4 + 17 clips add at most 21 vertices
// FP32 pass: polygons of up to 12 vertices in shared memory (the largest polygon met
// while clipping an atom's 18 faces had 11 vertices in 6,000 atoms of crystals and
// liquid); an atom whose clipping outgrows it is left to the FP64 pass
#define PTM_TOPO_VMAX32 12
// 32-bit words per thread: FP32 vectors, two polygon buffers
#define PTM_TOPO_WORDS (3 * PTM_TOPO_N + 2 * 2 * PTM_TOPO_VMAX32)
// Resident blocks per SM that shared memory allows: 8 for the FP32 pass (102
// words x 64 threads; the neighbours' slots and images stay in their list), 3 for
// the FP64 pass (its polygon buffers).  Stating them lets the compiler give each
// thread the registers that occupancy leaves free.
#define PTM_TOPO_BLOCKS_PER_SM 8
#define PTM_TOPO64_BLOCKS_PER_SM 3

// The plane of neighbour j's face: in-plane axes e1, e2 and the foot point p.
template <typename T, typename Vec>
__device__ __forceinline__ void topo_plane(int j, Vec V, T (&e1)[3], T (&e2)[3], T (&p)[3]) {
  const T n0 = V(j, 0), n1 = V(j, 1), n2 = V(j, 2);
  const T nn = sqrt(n0 * n0 + n1 * n1 + n2 * n2);
  const T u0 = n0 / nn, u1 = n1 / nn, u2 = n2 / nn;
  // e1 = u x a with a the axis least aligned with u, e2 = u x e1
  const bool ax = fabs(u0) < (T)0.6;
  const T a0 = ax ? (T)1 : (T)0, a1 = ax ? (T)0 : (T)1;
  e1[0] = u1 * (T)0 - u2 * a1; e1[1] = u2 * a0 - u0 * (T)0; e1[2] = u0 * a1 - u1 * a0;
  const T l1 = sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
  e1[0] /= l1; e1[1] /= l1; e1[2] /= l1;
  e2[0] = u1 * e1[2] - u2 * e1[1]; e2[1] = u2 * e1[0] - u0 * e1[2]; e2[2] = u0 * e1[1] - u1 * e1[0];
  p[0] = n0 / 2; p[1] = n1 / 2; p[2] = n2 / 2;
}

// FP64 area of the Voronoi face of neighbour j among the m vectors V(i, c) (VF: the
// same rounded to FP32); P and Q are polygon buffers of 2 x vmax values, element
// e at P[e * st].  `lines` are the neighbours expected to cut the face: the polygon
// they leave is then held against every other line, and those that come near it cut
// too.  That check may run in FP32: the vertices are known, so a line's value at one is
// off by at most 130 roundings of the 18th distance squared, 8e-8 R^2, where a
// line must stay PTM_TOPO_NEAR R^2 clear of the polygon to be left out.  (Without
// it the FP32 polygon that named the lines had the last word, and of two
// neighbours within 1e-4 of a distance of each other FP32 cannot place the line that
// divides their faces: areas were off by up to the whole starting square.)
template <typename Vec, typename VecF>
__device__ double topo_face_area64(int m, int j, uint32_t lines, double R, Vec V, VecF VF, double *P, double *Q, int st,
                                   int vmax) {
  double e1[3], e2[3], p[3];
  topo_plane<double>(j, V, e1, e2, p);
  // a convex polygon gains at most one vertex per clip (4 + 17 < PTM_TOPO_VMAX);
  // rounding on a nearly degenerate polygon could emit more, so writes stop at
  // the buffer's end (the polygon then has next to no area either way)
  double *cur = P, *nxt = Q;
  int np = 4;
  cur[0] = -R; cur[st] = -R; cur[2 * st] = R; cur[3 * st] = -R;
  cur[4 * st] = R; cur[5 * st] = R; cur[6 * st] = -R; cur[7 * st] = R;
  const uint32_t all = ((1u << m) - 1u) & ~(1u << j);
  uint32_t left = lines & all, others = ~lines & all;
  for (;;) {
    for (; left && np > 0; left &= left - 1) {
      const int i = __ffs(left) - 1;
      const double w0 = V(i, 0), w1 = V(i, 1), w2 = V(i, 2);
      const double A = w0 * e1[0] + w1 * e1[1] + w2 * e1[2], B = w0 * e2[0] + w1 * e2[1] + w2 * e2[2];
      const double C = (w0 * w0 + w1 * w1 + w2 * w2) / 2 - (w0 * p[0] + w1 * p[1] + w2 * p[2]);
      int nq = 0;
      double xs = cur[0], xt = cur[st], fx = A * xs + B * xt - C;
      const double x0 = xs, t0 = xt, f0 = fx;
      for (int k = 0; k < np; k++) {
        double ys = x0, yt = t0, fy = f0;
        if (k + 1 < np) { ys = cur[2 * (k + 1) * st]; yt = cur[(2 * k + 3) * st]; fy = A * ys + B * yt - C; }
        if (fx <= 0) {
          if (nq < vmax) { nxt[2 * nq * st] = xs; nxt[(2 * nq + 1) * st] = xt; }
          nq++;
        }
        if ((fx < 0 && fy > 0) || (fx > 0 && fy < 0)) {
          const double tt = fx / (fx - fy);
          if (nq < vmax) { nxt[2 * nq * st] = xs + tt * (ys - xs); nxt[(2 * nq + 1) * st] = xt + tt * (yt - xt); }
          nq++;
        }
        xs = ys; xt = yt; fx = fy;
      }
      np = min(nq, vmax);
      double *tmp = cur; cur = nxt; nxt = tmp;
    }
    if (!others || np == 0) break;
    // cut by the others too, where they come near (a smaller polygon stays clear of
    // the lines this one is clear of: once is enough)
    float2 *X = (float2 *)nxt;
    for (int k = 0; k < np; k++) X[k * st] = make_float2((float)cur[2 * k * st], (float)cur[(2 * k + 1) * st]);
    const float a0 = (float)e1[0], a1 = (float)e1[1], a2 = (float)e1[2], b0 = (float)e2[0], b1 = (float)e2[1],
                b2 = (float)e2[2], c0 = (float)p[0], c1 = (float)p[1], c2 = (float)p[2];
    const float clear = -PTM_TOPO_NEAR * (float)R * (float)R;
    for (; others; others &= others - 1) {
      const int i = __ffs(others) - 1;
      const float w0 = VF(i, 0), w1 = VF(i, 1), w2 = VF(i, 2);
      const float A = w0 * a0 + w1 * a1 + w2 * a2, B = w0 * b0 + w1 * b1 + w2 * b2;
      const float C = (w0 * w0 + w1 * w1 + w2 * w2) / 2 - (w0 * c0 + w1 * c1 + w2 * c2);
      bool near = false;
      for (int k = 0; k < np; k++) near |= !(A * X[k * st].x + B * X[k * st].y - C <= clear);
      left |= (uint32_t)near << i;
    }
    if (!left) break;
  }
  double s2 = 0;
  for (int k = 0; k < np; k++) {
    const int k1 = k + 1 == np ? 0 : k + 1;
    s2 += cur[2 * k * st] * cur[(2 * k1 + 1) * st] - cur[2 * k1 * st] * cur[(2 * k + 1) * st];
  }
  return fabs(s2) / 2;
}

// FP32 area of the same face, polygons of at most PTM_TOPO_VMAX32 vertices at
// P[k * st] and Q[k * st].  The other planes cut the face's plane in lines; nearest
// line first, the polygon has nearly its final shape after a few cuts, and the
// first line beyond its farthest vertex ends the face, so a warp makes about 9
// cuts where the neighbours' order took all 17.  A cut marks the vertices outside
// its line: of a convex polygon one run of consecutive ones, replaced by its two
// crossings, so it copies the rest and makes two divisions however many vertices the
// other lanes' polygons have.  `over` is set when the polygon outgrows the buffer: the
// FP64 pass decides then.  With LINES the
// result is instead the set of lines (bit = neighbour) that come within PTM_TOPO_NEAR
// R of the polygon: those the FP64 area expects to be cut by (all of them when the
// polygon is empty or `over`).
template <bool LINES, typename Vec>
__device__ __forceinline__ float topo_face32(int m, int j, float R, Vec V, float2 *P, float2 *Q, int st, bool &over,
                                             uint32_t &lines) {
  float e1[3], e2[3], p[3];
  topo_plane<float>(j, V, e1, e2, p);
  // a neighbour on the centre has no plane (the axes are 0 / 0) and no face; the FP64
  // form, cut by any line at all, finds the same
  if (!(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2] > 0.f)) {
    lines = ~0u;
    return 0.f;
  }
  auto line = [&](int i, float &A, float &B, float &C) {
    const float w0 = V(i, 0), w1 = V(i, 1), w2 = V(i, 2);
    A = w0 * e1[0] + w1 * e1[1] + w2 * e1[2];
    B = w0 * e2[0] + w1 * e2[1] + w2 * e2[2];
    C = (w0 * w0 + w1 * w1 + w2 * w2) / 2 - (w0 * p[0] + w1 * p[1] + w2 * p[2]);
  };
  // signed distance of each line from the foot point, as an integer of the same
  // order with the neighbour in its low 5 bits (rounded down)
  uint32_t key[PTM_TOPO_N];
#pragma unroll
  for (int i = 0; i < PTM_TOPO_N; i++) {
    key[i] = 0xffffffffu;
    if (i < m && i != j) {
      float A, B, C;
      line(i, A, B, C);
      const float q = A * A + B * B;
      const uint32_t u = __float_as_uint(q > 0.f ? C * rsqrtf(q) : (C < 0.f ? -INFINITY : INFINITY));
      key[i] = ((u ^ ((uint32_t)((int)u >> 31) | 0x80000000u)) & ~31u) | (uint32_t)i;
    }
  }
  float2 *cur = P, *nxt = Q;
  int np = 4;
  cur[0] = make_float2(-R, -R); cur[st] = make_float2(R, -R); cur[2 * st] = make_float2(R, R); cur[3 * st] = make_float2(-R, R);
  float r2 = 2.f * R * R;                            // square of the farthest vertex's distance
#pragma unroll 1
  for (int trip = 0; trip < m; trip++) {
    uint32_t near = key[0];
#pragma unroll
    for (int i = 1; i < PTM_TOPO_N; i++) near = min(near, key[i]);
    if (near == 0xffffffffu) break;
#pragma unroll
    for (int i = 0; i < PTM_TOPO_N; i++) key[i] = key[i] == near ? 0xffffffffu : key[i];
    {
      const uint32_t u = near & ~31u;
      const float dist = __uint_as_float(u & 0x80000000u ? u ^ 0x80000000u : ~u);
      if (dist > 0.f && dist * dist > r2 * 1.00001f) break;      // it and all later lines pass outside
    }
    float A, B, C;
    line((int)(near & 31u), A, B, C);
    uint32_t out = 0;
    for (int k = 0; k < np; k++) {
      const float2 x = cur[k * st];
      out |= (uint32_t)(A * x.x + B * x.y - C > 0.f) << k;
    }
    if (!out) continue;
    const uint32_t all = (1u << np) - 1u;
    if (out == all) { np = 0; break; }
    int nq = 0;
    r2 = 0.f;
    auto put = [&](float2 x) {
      if (nq < PTM_TOPO_VMAX32) nxt[nq * st] = x;
      r2 = fmaxf(r2, x.x * x.x + x.y * x.y);
      nq++;
    };
    // the crossing from an inside vertex a to an outside one b, seen from the inside: the
    // outside one may be as far as the starting square, with its rounding.  (Largest error
    // of an area of noisy fcc, bcc and sc, of the mean squared distance: 3.1e-6; seen along
    // the edge either way 3.6e-6, cut in the neighbours' order 3.0e-6.  Faces of free
    // surfaces past the guard: 2,441 of 360,000 against 3,128 and 2,722.)
    auto cross = [&](float2 a, float fa, float2 b, float fb) {
      const float t = fa / (fa - fb);
      put(make_float2(a.x + t * (b.x - a.x), a.y + t * (b.y - a.y)));
    };
    // the run s .. e of outside vertices (cyclic)
    const uint32_t prev = (out << 1 | out >> (np - 1)) & all, begins = out & ~prev;
    if (begins & (begins - 1)) {
      // more than one run: rounding, where corners of the polygon lie on the line (the
      // faces of perfect lattices).  Vertex by vertex: left to the FP64 pass, a few such
      // atoms held k_topo64 for 0.9 ms
#pragma unroll 1
      for (int k = 0; k < np; k++) {
        const float2 x = cur[k * st], y = cur[(k + 1 == np ? 0 : k + 1) * st];
        const float fx = A * x.x + B * x.y - C, fy = A * y.x + B * y.y - C;
        if (fx <= 0.f) put(x);
        if (fx < 0.f && fy > 0.f) cross(x, fx, y, fy);
        if (fx > 0.f && fy < 0.f) cross(y, fy, x, fx);
      }
      over |= nq > PTM_TOPO_VMAX32;
      np = min(nq, PTM_TOPO_VMAX32);
      float2 *tmp = cur; cur = nxt; nxt = tmp;
      continue;
    }
    const int s = __ffs(begins) - 1, n = __popc(out);
    const int in0 = s + n >= np ? s + n - np : s + n, in1 = s ? s - 1 : np - 1, e = in0 ? in0 - 1 : np - 1;
    for (int k = in0, left = np - n; left; left--) {
      const float2 x = cur[k * st];
      nxt[nq * st] = x;
      r2 = fmaxf(r2, x.x * x.x + x.y * x.y);
      nq++;
      k = k + 1 == np ? 0 : k + 1;
    }
    // the crossings of in1 -> s and e -> in0; a vertex on the plane is its own
    const float2 a = cur[in1 * st], b = cur[s * st], c = cur[e * st], g = cur[in0 * st];
    const float fa = A * a.x + B * a.y - C, fb = A * b.x + B * b.y - C, fc = A * c.x + B * c.y - C, fg = A * g.x + B * g.y - C;
    if (fa < 0.f) cross(a, fa, b, fb);
    if (fg < 0.f) cross(g, fg, c, fc);
    over |= nq > PTM_TOPO_VMAX32;
    np = min(nq, PTM_TOPO_VMAX32);
    float2 *tmp = cur; cur = nxt; nxt = tmp;
  }
  if constexpr (LINES) {
    lines = 0;
    for (int i = 0; i < m; i++) {
      float A, B, C, f = -INFINITY;
      line(i, A, B, C);
      for (int k = 0; k < np; k++) f = fmaxf(f, A * cur[k * st].x + B * cur[k * st].y - C);
      // f is |(A, B)| <= |V(i)| times a distance, and C sums squares of such lengths
      if (f > -PTM_TOPO_NEAR * R * R) lines |= 1u << i;
    }
    if (over || np < 3) lines = ~0u;
    return 0.f;
  }
  float s2 = 0.f;
  if (np) {
    const float2 x0 = cur[0];
    float2 x = x0;
    for (int k = 1; k <= np; k++) {
      const float2 y = k < np ? cur[k * st] : x0;
      s2 += x.x * y.y - y.x * x.y;
      x = y;
    }
  }
  return fabsf(s2) / 2;
}

// Order o[0..m) of neighbour ranks by (area descending, rank ascending), then
// group by the band and order each group by rank.  Returns the faces (bit =
// neighbour rank) that may stand on either side of a gap between consecutive areas
// that lies within the guard of the band edge; 0 when every gap is clear of it.
template <typename T>
__device__ uint32_t topo_order(int m, const T *area, T mean2, int *o) {
  for (int k = 0; k < m; k++) o[k] = k;
  for (int k = 1; k < m; k++) {                       // insertion sort, stable in rank
    const int x = o[k];
    int p = k;
    while (p > 0 && area[o[p - 1]] < area[x]) { o[p] = o[p - 1]; p--; }
    o[p] = x;
  }
  const T band = (T)PTM_TOPO_BAND * mean2, guard = (T)PTM_TOPO_GUARD * mean2;
  uint32_t near = 0;
  int g0 = 0;
  for (int k = 1; k <= m; k++) {
    bool split = k == m;
    if (k < m) {
      const T gap = area[o[k - 1]] - area[o[k]];
      if (fabs(gap - band) <= guard) {
        // the two faces of the gap, and those so near to either in area that rounding may
        // have put them in its place (an area of exactly 0 is not rounding's)
        near |= (1u << o[k - 1]) | (1u << o[k]);
        for (int q = k - 1; q > 0 && area[o[q - 1]] - area[o[q]] <= guard / 2; q--) near |= 1u << o[q - 1];
        for (int q = k; q + 1 < m && area[o[q]] - area[o[q + 1]] <= guard / 2 && area[o[q + 1]] > (T)0; q++)
          near |= 1u << o[q + 1];
      }
      split = gap > band;
    }
    if (split) {                                      // group o[g0..k): order by rank
      for (int a = g0 + 1; a < k; a++) {
        const int x = o[a];
        int p = a;
        while (p > g0 && o[p - 1] > x) { o[p] = o[p - 1]; p--; }
        o[p] = x;
      }
      g0 = k;
    }
  }
  return near;
}

// What the FP32 pass leaves for the FP64 pass about a listed atom: its FP32 face
// areas and the faces to recompute in FP64 (bit = neighbour rank: those beside
// every gap at the band edge, or all).
struct TopoSide {
  float area[PTM_TOPO_N];
  uint32_t faces;
  uint32_t pad;
};

// One atom, FP32 areas.  An atom with an area gap at the band edge (or a
// polygon larger than the FP32 buffers) is appended to `list` for the FP64 pass
// instead of being decided here, so that no warp waits on one lane's FP64 work;
// the first cap_side listed atoms leave their areas and uncertain faces in
// `side`.  The 18 nearest come from k_knn (d.nbr; a slot of -1: fewer); their first 14
// rows take the order, a listed atom's by the FP64 pass.
template <bool F64>
__device__ void topo_atom(const FrameDesc &d, int s, int *tsm, int *list, int *list_count, TopoSide *side,
                          int cap_side) {
  typedef typename RT<F64>::T TI;
  const int t = threadIdx.x;
  auto VF = [&](int k, int c) -> float & { return ((float *)tsm)[(3 * k + c) * PTM_BLOCK + t]; };
  const int64_t n = d.n, sl = s - d.atom_offset;     // frame-local slot
  int2 *nb = d.nbr + sl;
  TI xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  int m = 0;
  int o[PTM_TOPO_N];
  // FP32 neighbour vectors: the difference of positions plus the image
  // shift, summed without loss (error-free sums), as the metric steps use them
  float mean2 = 0.f, dmax2 = 0.f;
#pragma unroll 2
  for (int k = 0; k < PTM_TOPO_N; k++) {
    const int2 en = nb[(int64_t)k * n];
    if (en.x < 0) break;                              // the valid entries form a prefix
    m++;
    TI xj, yj, zj;
    int idj;
    load_atom<F64>(d, en.x, xj, yj, zj, idj);
    int a0, a1, a2;
    img_unpack(en.y, a0, a1, a2);
    if constexpr (F64) {
      double hx, hy, hz;
      shift_f64(d, a0, a1, a2, hx, hy, hz);
      VF(k, 0) = (float)((xj - xi) + hx); VF(k, 1) = (float)((yj - yi) + hy); VF(k, 2) = (float)((zj - zi) + hz);
    } else {
      float hx, hy, hz, lx, ly, lz, p, e1, q2, e2;
      shift_f32(d, a0, a1, a2, hx, hy, hz, lx, ly, lz);
      two_sum(xj, -xi, p, e1); two_sum(p, hx, q2, e2); VF(k, 0) = q2 + (e1 + (e2 + lx));
      two_sum(yj, -yi, p, e1); two_sum(p, hy, q2, e2); VF(k, 1) = q2 + (e1 + (e2 + ly));
      two_sum(zj, -zi, p, e1); two_sum(p, hz, q2, e2); VF(k, 2) = q2 + (e1 + (e2 + lz));
    }
    const float r2 = VF(k, 0) * VF(k, 0) + VF(k, 1) * VF(k, 1) + VF(k, 2) * VF(k, 2);
    mean2 += r2;
    dmax2 = fmaxf(dmax2, r2);
  }
  if (m > 0) {
    mean2 /= (float)m;
    const float R = 10.f * sqrtf(dmax2);
    auto vf = [&](int i, int c) -> float { return VF(i, c); };
    // polygon buffers in shared memory, one word per thread per row
    float2 *PB = (float2 *)(tsm + 3 * PTM_TOPO_N * PTM_BLOCK) + t;
    float2 *QB = PB + PTM_TOPO_VMAX32 * PTM_BLOCK;
    float area[PTM_TOPO_N];
    bool over = false;
    for (int k = 0; k < m; k++) { uint32_t unused; area[k] = topo_face32<false>(m, k, R, vf, PB, QB, PTM_BLOCK, over, unused); }
    // a gap at the band edge, or a polygon larger than the buffer: the second pass decides
    const uint32_t near = topo_order<float>(m, area, mean2, o);
    if (near || over) {
      count(d, C_TOPO64);
      const int slot = atomicAdd(list_count, 1);
      list[slot] = s;
      if (slot < cap_side) {                      // what the FP64 pass reuses
        TopoSide &sd = side[slot];
        for (int k = 0; k < PTM_TOPO_N; k++) sd.area[k] = k < m ? area[k] : 0.f;
        sd.faces = over ? ~0u : near;
      }
      return;
    }
  }
  int2 e[PTM_KNN];
#pragma unroll
  for (int k = 0; k < PTM_KNN; k++) e[k] = k < m ? nb[(int64_t)o[k] * n] : make_int2(-1, 0);
#pragma unroll
  for (int k = 0; k < PTM_KNN; k++) nb[(int64_t)k * n] = e[k];
}

// FP64 pass for listed atom i (= list position), one thread: FP64 neighbour
// vectors, and in FP64 the areas of the faces the FP32 pass could not decide
// (those beside every gap at the band edge); the others keep their FP32
// areas, whose error (measured within 3.1e-6 of the mean squared distance) is
// far below the guard, so every gap decided from them is decided as in FP64.
// Atoms past the side buffer recompute every face.  Polygon buffers in shared
// memory, element e at P[e * PTM_BLOCK].  The lanes of `wmask` call this
// together and take their faces in step, one face per lane per trip, so a warp
// makes as many trips as its busiest lane has faces (not one per face index that
// any lane needs).  A face is first clipped again in FP32, which finds the lines that matter (about 6 of 17), so the FP64
// pipe, 2 operations a clock per SM, sees only those.
template <bool F64>
__device__ void topo_atom64(const FrameDesc &d, int s, int i, const TopoSide *side, int cap_side, double *P,
                            double *Q, float *vf32, unsigned wmask) {
  typedef typename RT<F64>::T TI;
  TI xi, yi, zi;
  int idi;
  load_atom<F64>(d, s, xi, yi, zi, idi);
  const int64_t n = d.n, sl = s - d.atom_offset;     // frame-local slot
  int jn[PTM_TOPO_N], im[PTM_TOPO_N], m = 0;
  double a64[PTM_TOPO_N];
  for (int k = 0; k < PTM_TOPO_N; k++) {
    const int2 e = d.nbr[(int64_t)k * n + sl];
    jn[k] = e.x;
    im[k] = e.y;
    m += e.x >= 0;
  }
  uint32_t faces = ~0u;
  if (i < cap_side) {
    const TopoSide &sd = side[i];
    for (int k = 0; k < PTM_TOPO_N; k++) a64[k] = (double)sd.area[k];
    faces = sd.faces;
  }
  int o[PTM_TOPO_N];
  double v64[PTM_TOPO_N][3], mean64 = 0.0, dmax64 = 0.0;
  if (m > 0) {
    for (int k = 0; k < m; k++) {
      vec_fp64<F64>(d, xi, yi, zi, jn[k], im[k], v64[k][0], v64[k][1], v64[k][2]);
      const double r2 = v64[k][0] * v64[k][0] + v64[k][1] * v64[k][1] + v64[k][2] * v64[k][2];
      mean64 += r2;
      dmax64 = fmax(dmax64, r2);
    }
    mean64 /= m;
  }
  auto vd = [&](int a, int c) -> double { return v64[a][c]; };
  auto vf = [&](int a, int c) -> float & { return vf32[(3 * a + c) * PTM_BLOCK]; };
  for (int k = 0; k < m; k++)
    for (int c = 0; c < 3; c++) vf(k, c) = (float)v64[k][c];
  uint32_t todo = m > 0 ? faces & ((1u << m) - 1u) : 0u;
  while (__any_sync(wmask, todo != 0)) {
    if (!todo) continue;
    const int k = __ffs(todo) - 1;
    todo &= todo - 1;
    const double R = 10.0 * sqrt(dmax64);
    bool over = false;
    uint32_t lines;
    topo_face32<true>(m, k, (float)R, vf, (float2 *)P, (float2 *)Q, PTM_BLOCK, over, lines);
    a64[k] = topo_face_area64(m, k, lines, R, vd, vf, P, Q, PTM_BLOCK, PTM_TOPO_VMAX);
  }
  if (m > 0) topo_order<double>(m, a64, mean64, o);
  for (int k = 0; k < PTM_KNN; k++) d.nbr[(int64_t)k * n + sl] = k < m ? make_int2(jn[o[k]], im[o[k]]) : make_int2(-1, 0);
}

// Bounded by instruction issue (60 % of the slots; 2,000 warp instructions an atom).  262 k
// atoms: 1.69 ms with every plane clipping every vertex, 1.35 ms with marks and one copy
// per cut, 1.01 ms nearest line first and at 8 blocks per SM.
template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_TOPO_BLOCKS_PER_SM) k_topo(const __grid_constant__ FrameDesc d, int *list,
                                                    int *list_count, TopoSide *side, int cap_side) {
  extern __shared__ __align__(16) unsigned char tsm_raw[];
  const int64_t s = (int64_t)blockIdx.x * PTM_BLOCK + threadIdx.x;
  if (s >= d.n) return;
  topo_atom<F64>(d, (int)s, (int *)tsm_raw, list, list_count, side, cap_side);
}

// Second pass over the listed atoms, one thread per atom (grid-stride over the
// list: its length is read on the device): fn(position in the list, lanes of the
// warp that call together).  (Spreading a short list thinner, 8 atoms per warp, made
// 3 times the FP64 warp instructions: 0.37 -> 0.44 ms for 7,800 atoms; clipping by
// the lines that matter only: 0.24 ms, 0.27 with the lines left out checked in FP32.)
template <typename Fn>
__device__ __forceinline__ void topo64_list(int cnt, Fn &&fn) {
  for (int i0 = blockIdx.x * PTM_BLOCK + (threadIdx.x & ~31); i0 < cnt; i0 += gridDim.x * PTM_BLOCK) {
    const int i = i0 + (threadIdx.x & 31);
    const unsigned wmask = __ballot_sync(0xffffffffu, i < cnt);
    if (i < cnt) fn(i, wmask);
  }
}

template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_TOPO64_BLOCKS_PER_SM) k_topo64(const __grid_constant__ FrameDesc d,
                                                      const int *list, const int *list_count, const TopoSide *side,
                                                      int cap_side) {
  extern __shared__ __align__(16) unsigned char tsm_raw[];
  double *P = (double *)tsm_raw + threadIdx.x, *Q = P + 2 * PTM_TOPO_VMAX * PTM_BLOCK;
  float *vf = (float *)((double *)tsm_raw + 4 * PTM_TOPO_VMAX * PTM_BLOCK) + threadIdx.x;
  topo64_list(*list_count, [&](int i, unsigned wmask) {
    topo_atom64<F64>(d, list[i], i, side, cap_side, P, Q, vf, wmask);
  });
}

// The same two passes over a batch: every slot finds its frame (frames in the
// Euclidean order are skipped); each frame's list is its own segment of the batch's
// (FrameDesc::nbr).
template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_TOPO_BLOCKS_PER_SM)
    k_topo_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ atom_off, int nframes,
                 int64_t ntotal, int *list, int *list_count, TopoSide *side, int cap_side) {
  extern __shared__ __align__(16) unsigned char tsm_raw[];
  const int64_t s = (int64_t)blockIdx.x * PTM_BLOCK + threadIdx.x;
  if (s >= ntotal) return;
  const FrameDesc &d = descs[frame_of(atom_off, nframes, s)];
  if (d.ordering != PTM_ORDER_TOPOLOGICAL) return;
  topo_atom<F64>(d, (int)s, (int *)tsm_raw, list, list_count, side, cap_side);
}

template <bool F64>
__global__ void __launch_bounds__(PTM_BLOCK, PTM_TOPO64_BLOCKS_PER_SM)
    k_topo64_batch(const FrameDesc *__restrict__ descs, const int64_t *__restrict__ atom_off, int nframes,
                   const int *list, const int *list_count, const TopoSide *side, int cap_side) {
  extern __shared__ __align__(16) unsigned char tsm_raw[];
  double *P = (double *)tsm_raw + threadIdx.x, *Q = P + 2 * PTM_TOPO_VMAX * PTM_BLOCK;
  float *vf = (float *)((double *)tsm_raw + 4 * PTM_TOPO_VMAX * PTM_BLOCK) + threadIdx.x;
  topo64_list(*list_count, [&](int i, unsigned wmask) {
    const int s = list[i];
    const FrameDesc &d = descs[frame_of(atom_off, nframes, s)];
    topo_atom64<F64>(d, s, i, side, cap_side, P, Q, vf, wmask);
  });
}

// Listed atoms whose areas and uncertain faces the FP32 pass keeps for the FP64
// pass (a quarter of the atoms: 3.6 % were listed in the hot polycrystal, 2.6 %
// in the mixed-phase frame, up to 15 % in cold crystals; the rest recompute every
// face).
constexpr size_t topo_side_cap(size_t n) { return n / 4 + 256; }
constexpr size_t topo_side_bytes(size_t n) { return topo_side_cap(n) * sizeof(TopoSide); }
// FP64 pass: two polygon buffers of 2 x PTM_TOPO_VMAX doubles (FP32 polygons use
// them too) and the FP32 vectors per thread; 3 blocks of 61.5 KB + 1 KB per SM
constexpr size_t topo64_smem_bytes() {
  return (size_t)PTM_BLOCK * (4 * PTM_TOPO_VMAX * sizeof(double) + 3 * PTM_TOPO_N * sizeof(float));
}

constexpr size_t topo_smem_bytes() { return (size_t)PTM_BLOCK * PTM_TOPO_WORDS * 4; }

}  // namespace ptm
