// Tensor assembly (FP64) and packing into the tile-blocked storage.
//
// Sec. 3 of the paper: the field of every uniformly magnetised cuboid or
// tetrahedral tile is evaluated analytically at the centre of every other tile; the tensor is
// computed once, at the start (Sec. 3.1), and stored in a reduced precision
// (FP32 in the paper, Sec. 3.2).  One thread evaluates one 3x3 block in FP64
// and stores its 6 unique entries directly in the requested precision.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "mt_internal.cuh"

namespace {

// Tensor of the cuboid (centre c, full edges e) at the point r, from the
// Newtonian potential Phi of the box:  N = -(1/4 pi) grad grad Phi, so that
// H = -N M.  Faces are numbered low (0) / high (1) on each axis; a corner's
// sign is s = -(-1)^(f_x + f_y + f_z): +1 when an odd number of its faces are
// high faces.
//   N_xx = -(1/4 pi) sum_corners s atan(dy dz / (dx R))
//   N_xy = +(1/4 pi) sum_corners s log(dz + R)         (xz: dy, yz: dx)
// The FP64 pipe bounds assembly (GB300 executes ~2 FP64 operations per clock
// and SM), so the 24 arctangents and 24 logarithms of the sums are not taken
// one by one: the arctangents of an entry are the arguments of complex
// numbers dx R + i dy dz, which are multiplied, and the logarithms of an
// entry are one logarithm of a ratio of products: 3 + 3 transcendental
// functions per block instead of 48.  The rounding of the products is a few
// ulps of the angle or of the ratio, as much as that of the sums it replaces
// (whose logarithms of lengths in metres are of order 20); against 128-bit
// arithmetic distant blocks come out 7 to 13 times closer, touching ones as
// before.  n = 6,000 graded film, tensor and first field: 150.1 -> 39.3 ms, and
// 33.6 with signs and sizes tested on the high words and pairs that do not
// touch told apart by that test alone.
__device__ __forceinline__ double small_series(double t, double z) {
  // t (1 + z/3 + z^2/5 + z^3/7 + z^4/9 + z^5/11): atan t with z = -t^2,
  // atanh t with z = t^2; |t| < 2^-5 leaves z^6 / 13 < 7e-20
  return t * fma(z, fma(z, fma(z, fma(z, fma(z, 1.0 / 11, 1.0 / 9), 1.0 / 7), 1.0 / 5), 1.0 / 3), 1.0);
}
constexpr double kSmallArg = 0.03125;

// Tests of signs and sizes on the high words: a comparison of doubles costs
// the FP64 pipe as much as a product, and a block has about forty of them.
__device__ __forceinline__ bool is_zero(double a) { return (__double_as_longlong(a) << 1) == 0; }
__device__ __forceinline__ bool is_neg(double a) { return __double2hiint(a) < 0; }
__device__ __forceinline__ double flip_sign(double a, double of) {  // -a where of is negative
  return __hiloint2double(__double2hiint(a) ^ (__double2hiint(of) & (int)0x80000000), __double2loint(a));
}
// |a| 32 < b by the high words (b >= 0): |a| < kSmallArg b follows
__device__ __forceinline__ bool is_small(double a, double b) {
  return (unsigned)(__double2hiint(a) & 0x7fffffff) + (5u << 20) < (unsigned)__double2hiint(b);
}

// Arguments p of one face pair: theta_1 - theta_0 with theta = atan(b / a),
// a > 0, as a complex number (its argument is in (-pi, pi)).
struct Cplx {
  double re, im;
};
__device__ __forceinline__ Cplx arg_diff(double a1, double b1, double a0, double b0) {
  return {fma(a1, a0, b1 * b0), fma(b1, a0, -(a1 * b0))};
}
__device__ __forceinline__ Cplx cmul(Cplx p, Cplx q) {
  return {fma(p.re, q.re, -(p.im * q.im)), fma(p.re, q.im, p.im * q.re)};
}

// Sum over the corners of s atan(v w / (u R)) for the axis u: the faces
// u[0], u[1]; vw[fv | fw << 1] the products of the other two offsets;
// R(fu, fv, fw) the distances.  For a face u = 0 (the point in its plane,
// outside the face) the arctangents count 0: their +-pi/2 limits cancel.
template <typename RF>
__device__ __forceinline__ double angle_sum(const double u[2], const double vw[4], RF R) {
  Cplx pa[2], pb[2], f[2];
  int least = 1;  // > 0: every partial argument within (-pi/2, pi/2), the products keep the branch
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double a = fabs(u[k]);
    if (is_zero(a)) {
      pa[k] = pb[k] = f[k] = {1.0, 0.0};
      continue;
    }
    pa[k] = arg_diff(a * R(k, 1, 0), vw[1], a * R(k, 0, 0), vw[0]);
    pb[k] = arg_diff(a * R(k, 0, 1), vw[2], a * R(k, 1, 1), vw[3]);
    f[k] = cmul(pa[k], pb[k]);
    pa[k].im = flip_sign(pa[k].im, u[k]);
    pb[k].im = flip_sign(pb[k].im, u[k]);
    f[k].im = flip_sign(f[k].im, u[k]);
    least = min(min(least, __double2hiint(f[k].re)), min(__double2hiint(pa[k].re), __double2hiint(pb[k].re)));
  }
  if (least > 0) {
    const Cplx t = cmul(f[0], {f[1].re, -f[1].im});
    if (!is_neg(t.re) && is_small(t.im, t.re)) {
      const double q = t.im / t.re;
      return small_series(q, -q * q);
    }
    return atan2(t.im, t.re);
  }
  return (atan2(pa[0].im, pa[0].re) + atan2(pb[0].im, pb[0].re)) -
         (atan2(pa[1].im, pa[1].re) + atan2(pb[1].im, pb[1].re));
}

// Sum over the corners of s log(w + R) for the log's axis w: w[0], w[1] its
// offsets; R(f1, f2, fw).  Where both offsets are negative, log(R - w) of the
// swapped faces takes its place: exact, and free of the cancellation of
// w + R for a point far on the negative side.
template <typename RF>
__device__ __forceinline__ double log_sum(const double w[2], RF R) {
  const bool neg = is_neg(w[0]) && is_neg(w[1]);
  const double w0 = neg ? -w[0] : w[0], w1 = neg ? -w[1] : w[1];
  const double n = ((R(0, 0, 1) + w1) * (R(1, 1, 1) + w1)) * ((R(1, 0, 0) + w0) * (R(0, 1, 0) + w0));
  const double d = ((R(0, 0, 0) + w0) * (R(1, 1, 0) + w0)) * ((R(1, 0, 1) + w1) * (R(0, 1, 1) + w1));
  const double diff = n - d, sum = n + d;
  double v;
  if (is_small(diff, sum)) {
    const double q = diff / sum;
    v = 2.0 * small_series(q, q * q);  // log(n / d) = 2 atanh((n - d) / (n + d))
  } else {
    v = log(n / d);
  }
  return neg ? -v : v;
}

__device__ __forceinline__ void cuboid_tensor(const double *r, const double *c, const double *e, double out[6]) {
  // offsets r - face in units of a power of two near the tile's size (exact):
  // the products below stay far from under- and overflow in any unit of length
  const double unit = scalbn(1.0, -ilogb(e[0] + e[1] + e[2]));
  double d[3][2], R[8];  // [axis][face]; corner distance, index fx | fy << 1 | fz << 2
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double ur = unit * r[a];
    d[a][0] = ur - unit * (c[a] - 0.5 * e[a]);
    d[a][1] = ur - unit * (c[a] + 0.5 * e[a]);
  }
  double xy[4], xz[4], yz[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    xy[q] = d[0][q & 1] * d[1][q >> 1];
    xz[q] = d[0][q & 1] * d[2][q >> 1];
    yz[q] = d[1][q & 1] * d[2][q >> 1];
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double x = d[0][q & 1], y = d[1][(q >> 1) & 1], z = d[2][(q >> 2) & 1];
    R[q] = sqrt(x * x + y * y + z * z);
  }
  const double k = 0.25 / MT_PI;
  out[0] = -k * angle_sum(d[0], yz, [&](int x, int y, int z) { return R[x | (y << 1) | (z << 2)]; });
  out[3] = -k * angle_sum(d[1], xz, [&](int y, int x, int z) { return R[x | (y << 1) | (z << 2)]; });
  out[5] = -k * angle_sum(d[2], xy, [&](int z, int x, int y) { return R[x | (y << 1) | (z << 2)]; });
  out[1] = k * log_sum(d[2], [&](int x, int y, int z) { return R[x | (y << 1) | (z << 2)]; });
  out[2] = k * log_sum(d[1], [&](int x, int z, int y) { return R[x | (y << 1) | (z << 2)]; });
  out[4] = k * log_sum(d[0], [&](int y, int z, int x) { return R[x | (y << 1) | (z << 2)]; });
}

// Tensor of a uniformly magnetised tetrahedron at r.  The body's field is that
// of its face charges sigma_f = M.n_f, so with H = -N M,
//   N = (1/4 pi) sum_f g_f n_f^T,  g_f = grad_r int_f dS / |r - r'|.
// For a plane triangle the gradient splits into a part along n_f, minus the
// signed solid angle of the face, and an in-plane part from the 2-D
// divergence theorem: minus the sum over its edges of the edge's outward
// in-plane normal u times l_e = int_e dl / |r - r'|.  Each edge belongs to
// two faces and l_e is the same for both, so
//   N = (1/4 pi) [ sum_f -omega_f n_f n_f^T - sum_e l_e (u n^T + u' n'^T) ]
// with dyads that depend on the tetrahedron only (the polyhedron form of
// Werner and Scheeres, 1997): they are formed once per tile (tetra_geom), and
// a block takes 4 distances, 4 solid angles (atan2 form of Van Oosterom and
// Strackee, 1983; the triple product as (a - r).(b - a) x (c - a)) and 6 edge
// integrals, l_e = 2 atanh(|e| / (R_a + R_b)).  FP64 throughout; the FP64 pipe bounds it
// (per-pair face geometry and every edge twice took three times the
// operations): 5,760 tetrahedra, tensor and first field, 153.8 -> 34.2 ms; errors
// against 128-bit arithmetic 0.3 to 0.65 of the per-face form's.
__device__ __forceinline__ void sub3(const double *a, const double *b, double *c) {
  c[0] = a[0] - b[0];
  c[1] = a[1] - b[1];
  c[2] = a[2] - b[2];
}
__device__ __forceinline__ double dot3(const double *a, const double *b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}
__device__ __forceinline__ void crs3(const double *a, const double *b, double *c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

// per-tile geometry of a tetrahedron (doubles): vertices 4 x 3, outward face
// normals (b - a) x (c - a) 4 x 3, face dyads n n^T 4 x 6, edge dyads 6 x 6
// (symmetrised: the exact ones are symmetric), edge lengths 6, the largest
// distance of a vertex from the centroid, the centroid.  Face f lies opposite
// vertex f; edges 01, 02, 03, 12, 13, 23.  Dyad entries xx xy xz yy yz zz.
constexpr int kTgVert = 0, kTgNorm = 12, kTgFace = 24, kTgEdge = 48, kTgLen = 84, kTgRad = 90, kTgCen = 91,
              kTgSize = 94;
__device__ __forceinline__ int tetra_edge(int a, int b) {  // a < b
  return a == 0 ? b - 1 : a + b;
}

__device__ void tetra_geom(const double *c, const double *v, double *G) {
  for (int q = 0; q < 12; ++q) G[kTgVert + q] = v[q];
  for (int q = kTgEdge; q < kTgLen; ++q) G[q] = 0.0;
  double rad = 0.0;
  for (int a = 0; a < 4; ++a) {
    double d[3];
    sub3(v + 3 * a, c, d);
    rad = fmax(rad, sqrt(dot3(d, d)));
    for (int b = a + 1; b < 4; ++b) {
      sub3(v + 3 * b, v + 3 * a, d);
      G[kTgLen + tetra_edge(a, b)] = sqrt(dot3(d, d));
    }
  }
  G[kTgRad] = rad;
  for (int q = 0; q < 3; ++q) G[kTgCen + q] = c[q];
#pragma unroll 1
  for (int f = 0; f < 4; ++f) {
    // face (a, b, c) opposite vertex f, made counter-clockwise about its
    // outward normal
    int id[3] = {f == 0 ? 1 : 0, f <= 1 ? 2 : 1, f <= 2 ? 3 : 2};
    double ab[3], ac[3], nf[3], to_f[3];
    sub3(v + 3 * id[1], v + 3 * id[0], ab);
    sub3(v + 3 * id[2], v + 3 * id[0], ac);
    crs3(ab, ac, nf);
    sub3(v + 3 * f, v + 3 * id[0], to_f);
    if (dot3(nf, to_f) > 0.0) {
      const int t = id[1];
      id[1] = id[2];
      id[2] = t;
      for (int q = 0; q < 3; ++q) nf[q] = -nf[q];
    }
    for (int q = 0; q < 3; ++q) G[kTgNorm + 3 * f + q] = nf[q];
    const double inv = 1.0 / sqrt(dot3(nf, nf));
    for (int q = 0; q < 3; ++q) nf[q] *= inv;
    int k = 0;
    for (int a = 0; a < 3; ++a)
      for (int b = a; b < 3; ++b) G[kTgFace + 6 * f + k++] = nf[a] * nf[b];
    for (int e = 0; e < 3; ++e) {
      const int p = id[e], q = id[(e + 1) % 3];
      double t[3], u[3];
      sub3(v + 3 * q, v + 3 * p, t);
      const double len = sqrt(dot3(t, t));
      for (int a = 0; a < 3; ++a) t[a] /= len;
      crs3(t, nf, u);  // in-plane, out of the face
      double *D = G + kTgEdge + 6 * tetra_edge(p < q ? p : q, p < q ? q : p);
      k = 0;
      for (int a = 0; a < 3; ++a)
        for (int b = a; b < 3; ++b) D[k++] += 0.5 * (u[a] * nf[b] + u[b] * nf[a]);
    }
  }
}

__global__ void k_tetra_geom(int64_t n, const double *centre, const double *vert, double *geo) {
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j < n) tetra_geom(centre + 3 * j, vert + 12 * j, geo + kTgSize * j);
}

__device__ __forceinline__ void tetra_tensor(const double *r, const double *G, double out[6]) {
  double D[4][3], L[4], num[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double *d = D[a];
    sub3(G + kTgVert + 3 * a, r, d);
    L[a] = sqrt(dot3(d, d));
    // the faces that hold vertex a: any of a face's vertices gives its triple
    // product; faces 1, 2, 3 take vertex 0, face 0 vertex 1
    if (a == 0) {
#pragma unroll
      for (int f = 1; f < 4; ++f) num[f] = dot3(d, G + kTgNorm + 3 * f);
    } else if (a == 1) {
      num[0] = dot3(d, G + kTgNorm);
    }
  }
  double N[6] = {0, 0, 0, 0, 0, 0}, dots[6];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a + 1; b < 4; ++b) {
      const int e = tetra_edge(a, b);
      const double len = G[kTgLen + e];
      dots[e] = dot3(D[a], D[b]);
      const double s = L[a] + L[b];
      double li;
      // 8 len < s by the high words; 2 atanh(q), q = len / s: 10 terms leave q^20 / 21 < 5e-20
      if (__double2hiint(len) + (3 << 20) < __double2hiint(s)) {
        const double q = len / s, z = q * q;
        li = 2.0 * q *
             fma(z, fma(z, fma(z, fma(z, fma(z, fma(z, fma(z, fma(z, fma(z, 1.0 / 19, 1.0 / 17), 1.0 / 15), 1.0 / 13),
                                                   1.0 / 11), 1.0 / 9), 1.0 / 7), 1.0 / 5), 1.0 / 3), 1.0);
      } else if (dots[e] >= 0.0) {
        li = log((s + len) / (s - len));
      } else {
        // near the edge s - len would cancel:
        // s^2 - len^2 = 2 (R_a R_b + dot) = 2 |a x b|^2 / (R_a R_b - dot)
        double x[3];
        crs3(D[a], D[b], x);
        li = log((s + len) * (s + len) * fma(L[a], L[b], -dots[e]) / (2.0 * dot3(x, x)));
      }
#pragma unroll
      for (int q = 0; q < 6; ++q) N[q] = fma(-li, G[kTgEdge + 6 * e + q], N[q]);
    }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int a = f == 0 ? 1 : 0, b = f <= 1 ? 2 : 1, c = f <= 2 ? 3 : 2;
    const double den = fma(L[a] * L[b], L[c], fma(dots[tetra_edge(a, b)], L[c],
                                                  fma(dots[tetra_edge(a, c)], L[b], dots[tetra_edge(b, c)] * L[a])));
    double half;  // half the solid angle
    if (!is_neg(den) && is_small(num[f], den)) {
      const double q = num[f] / den;
      half = small_series(q, -q * q);
    } else {
      half = atan2(num[f], den);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) N[q] = fma(2.0 * half, G[kTgFace + 6 * f + q], N[q]);
  }
  const double k = 0.25 / MT_PI;
#pragma unroll
  for (int q = 0; q < 6; ++q) out[q] = k * N[q];
}

// One block per lattice offset (dx, dy, dz): the tensor of the tile at the
// origin seen from (dx ex, dy ey, dz ez).  Index ((dx + Lx - 1)(2Ly - 1) +
// dy + Ly - 1)(2Lz - 1) + dz + Lz - 1.
__global__ void k_offset_table(int Lx, int Ly, int Lz, double ex, double ey, double ez, double *table) {
  const int64_t Ny = 2 * Ly - 1, Nz = 2 * Lz - 1;
  const int64_t tot = (int64_t)(2 * Lx - 1) * Ny * Nz;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= tot) return;
  const int dz = (int)(t % Nz) - (Lz - 1);
  const int dy = (int)((t / Nz) % Ny) - (Ly - 1);
  const int dx = (int)(t / (Ny * Nz)) - (Lx - 1);
  const double r[3] = {dx * ex, dy * ey, dz * ez};
  const double c[3] = {0.0, 0.0, 0.0};
  const double e[3] = {ex, ey, ez};
  cuboid_tensor(r, c, e, table + 6 * t);
}

// Relations of tetrahedra i and j (i != j), as pair_relation: bit 0 = the
// centroid of i lies in or on tetrahedron j (barycentric coordinates all
// >= -eps), bit 1 = they share a vertex (a "near" pair).
__device__ int tetra_relation(const double *ci, const double *vi, const double *vj) {
  bool touch = false;
#pragma unroll 1
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b)
      touch = touch || (vi[3 * a] == vj[3 * b] && vi[3 * a + 1] == vj[3 * b + 1] && vi[3 * a + 2] == vj[3 * b + 2]);
  // barycentric coordinates of ci in j: solve [v1-v0, v2-v0, v3-v0] x = ci - v0
  double e1[3], e2[3], e3[3], d[3], c23[3], c31[3], c12[3];
  sub3(vj + 3, vj, e1);
  sub3(vj + 6, vj, e2);
  sub3(vj + 9, vj, e3);
  sub3(ci, vj, d);
  crs3(e2, e3, c23);
  crs3(e3, e1, c31);
  crs3(e1, e2, c12);
  const double det = dot3(e1, c23);
  const double x = dot3(d, c23) / det, y = dot3(d, c31) / det, z = dot3(d, c12) / det;
  const double eps = 1e-12;
  const bool in = x >= -eps && y >= -eps && z >= -eps && (1.0 - x - y - z) >= -eps;
  return (in ? 1 : 0) | (touch ? 2 : 0);
}

// Geometry relations of tiles i and j (i != j): bit 0 = volumes overlap or
// the centre of i lies in/on tile j (invalid), bit 1 = the closed boxes touch
// (a "near" pair, kept in FP64 for the BF16 precisions).
__device__ __forceinline__ int pair_relation(const double *ci, const double *ei, const double *cj,
                                             const double *ej) {
  // boxes that do not touch share no volume and hold no centre either (their
  // bounds lie 1e-9 inside the touching one's): most pairs end here
  bool vol = true, pt = true, touch = true;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    touch = touch && (fabs(ci[a] - cj[a]) <= 0.5 * (ei[a] + ej[a]) * (1.0 + 1e-9));
  if (!touch) return 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double d = fabs(ci[a] - cj[a]);
    const double half = 0.5 * (ei[a] + ej[a]);
    const double tol = 1e-12 * (ei[a] + ej[a]);
    vol = vol && (d < half - tol);
    pt = pt && (d <= 0.5 * ej[a] + tol);
  }
  return ((vol || pt) ? 1 : 0) | (touch ? 2 : 0);
}

__device__ __forceinline__ int64_t scale_index(int64_t i, int64_t j, int TR, int TC, int64_t Q) {
  const int64_t p = i / TR, q = j / TC;
  const int r = (int)(i - p * TR), c = (int)(j - q * TC);
  return ((p * Q + q) * TR + r) * (int64_t)TC + c;
}

struct AsmArgs {
  const double *centre, *edge;
  const double *vert;  // 12n, tetrahedral tiles
  const double *geo;   // kTgSize n, tetrahedral tiles (tetra_geom)
  // uniform lattice: block (i, j) = table[offset lat_i - lat_j] (nullptr: evaluate)
  const double *table;
  const int32_t *lat;
  int Lx, Ly, Lz;
  int64_t n;
  int TR, TC, nplane;
  int64_t Q;
  int prec;
  void *data;
  int8_t *scale;
  int *bad;           // set to 1 on overlap
  int *planar_bad;    // set to 1 if a 4- or 3-plane (single-layer) tensor meets |N_xz| or |N_yz| >
                      // kPlanarTol, or (3 or 5 planes) a block's trace off delta_ij by more than kTraceTol
  int dense;          // 1: tensor-core planes (dense_a_index), else the streaming layout
  int half;           // 1: streaming FP32 tensor of one tile shape, upper triangle of chunks only
  int64_t Kp;
  int *near_fill;     // per-row fill counter (BF16 precisions)
  const int32_t *near_ptr;
  int32_t *near_col;
  double *near_val;
  int count_only;     // 1: only count near blocks per row into near_fill
};

// Block (i, j) into the storage: apart, in FP64, if it is a touching pair of a
// BF16 precision, else in the tensor's layout and precision.
__device__ __forceinline__ void store_block(const AsmArgs &A, int64_t i, int64_t j, bool near, const double N6[6]) {
  if (near) {
    const int slot = atomicAdd(&A.near_fill[i], 1);
    const int64_t at = A.near_ptr[i] + slot;
    A.near_col[at] = (int32_t)j;
#pragma unroll
    for (int e = 0; e < 6; ++e) A.near_val[6 * at + e] = N6[e];
    return;  // dense store keeps zeros there
  }
  if (A.dense) {
    __nv_bfloat16 *D = (__nv_bfloat16 *)A.data;
    const bool split = A.prec == MT_BF16_SPLIT;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      const int pl = stream_plane(e, A.nplane);
      if (pl < 0) {
        if (!(fabs(N6[e]) <= kPlanarTol)) *A.planar_bad = 1;
        continue;
      }
      const size_t at = dense_a_index(i, j, pl, A.Kp / 64, A.nplane, split);
      const __nv_bfloat16 hi = __double2bfloat16(N6[e]);
      D[at] = hi;
      if (split) D[at + kDenseLo] = __double2bfloat16(N6[e] - (double)__bfloat162float(hi));
    }
    return;
  }
  switch (A.prec) {
    case MT_F64: {
      double *D = (double *)A.data;
#pragma unroll
      for (int e = 0; e < 6; ++e) D[layout_index(i, j, e, A.TR, A.TC, 6, A.Q)] = N6[e];
    } break;
    case MT_F32: {
      float *D = (float *)A.data;
#pragma unroll
      for (int e = 0; e < 6; ++e) {
        const int pl = stream_plane(e, A.nplane);
        if (pl >= 0) D[layout_index_h(i, j, pl, A.TR, A.TC, A.nplane, A.Q, A.half)] = (float)N6[e];
        else if (traceless(A.nplane) && e == 5) {
          // zz is not stored: the identity that gives it must hold here
          const double tr = N6[0] + N6[3] + N6[5] - (i == j ? 1.0 : 0.0);
          if (!(fabs(tr) <= kTraceTol * (fabs(N6[0]) + fabs(N6[3]) + fabs(N6[5])) + kPlanarTol))
            *A.planar_bad = 1;
        } else if (!(fabs(N6[e]) <= kPlanarTol)) *A.planar_bad = 1;
      }
    } break;
    case MT_BF16_SCALED: {
      // power-of-two scale of the block: 2^s with s = exponent of max |N|
      double mx = 0.0;
#pragma unroll
      for (int e = 0; e < 6; ++e) mx = fmax(mx, fabs(N6[e]));
      int s = 0;
      if (mx > 0.0) {
        frexp(mx, &s);
        s = max(-126, min(126, s));
      }
      __nv_bfloat16 *D = (__nv_bfloat16 *)A.data;
#pragma unroll
      for (int e = 0; e < 6; ++e) {
        const int pl = stream_plane(e, A.nplane);
        if (pl >= 0) D[layout_index(i, j, pl, A.TR, A.TC, A.nplane, A.Q)] = __double2bfloat16(ldexp(N6[e], -s));
        else if (!(fabs(N6[e]) <= kPlanarTol)) *A.planar_bad = 1;
      }
      A.scale[scale_index(i, j, A.TR, A.TC, A.Q)] = (int8_t)s;
    } break;
    case MT_BF16_SPLIT: {
      __nv_bfloat16 *D = (__nv_bfloat16 *)A.data;
      const int half = A.nplane / 2;  // hi planes, then as many lo planes
#pragma unroll
      for (int e = 0; e < 6; ++e) {
        const int pl = stream_plane(e, half);
        if (pl < 0) {
          if (!(fabs(N6[e]) <= kPlanarTol)) *A.planar_bad = 1;
          continue;
        }
        const __nv_bfloat16 hi = __double2bfloat16(N6[e]);
        const __nv_bfloat16 lo = __double2bfloat16(N6[e] - (double)__bfloat162float(hi));
        D[layout_index(i, j, pl, A.TR, A.TC, A.nplane, A.Q)] = hi;
        D[layout_index(i, j, half + pl, A.TR, A.TC, A.nplane, A.Q)] = lo;
      }
    } break;
  }
}

__device__ __forceinline__ bool kept_apart(const AsmArgs &A, int rel) {
  return (rel & 2) && (A.prec == MT_BF16_SCALED || A.prec == MT_BF16_SPLIT);
}

// Cuboids: grid (Q, P); TC threads; thread = column j of the chunk, loop over
// the panel's TR rows i.
__global__ void k_assemble(AsmArgs A) {
  const int64_t q = blockIdx.x, p = blockIdx.y;
  const int64_t j = q * A.TC + threadIdx.x;
  if (j >= A.n) return;
  double cj[3], ej[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cj[a] = A.centre[3 * j + a];
    ej[a] = A.edge[3 * j + a];
  }
  for (int r = 0; r < A.TR; ++r) {
    const int64_t i = p * A.TR + r;
    if (i >= A.n) break;
    double ci[3], ei[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      ci[a] = A.centre[3 * i + a];
      ei[a] = A.edge[3 * i + a];
    }
    int rel;
    int64_t toff = 0;
    if (A.table) {
      // lattice: the offset decides everything (a repeated index = overlap,
      // touching = at most one step on every axis)
      const int dx = A.lat[3 * i] - A.lat[3 * j], dy = A.lat[3 * i + 1] - A.lat[3 * j + 1];
      const int dz = A.lat[3 * i + 2] - A.lat[3 * j + 2];
      const bool same = dx == 0 && dy == 0 && dz == 0;
      const bool touch = dx >= -1 && dx <= 1 && dy >= -1 && dy <= 1 && dz >= -1 && dz <= 1;
      rel = (i == j) ? 2 : ((same ? 1 : 0) | (touch ? 2 : 0));
      toff = ((int64_t)(dx + A.Lx - 1) * (2 * A.Ly - 1) + (dy + A.Ly - 1)) * (2 * A.Lz - 1) + (dz + A.Lz - 1);
    } else {
      rel = (i == j) ? 2 : pair_relation(ci, ei, cj, ej);
    }
    if (rel & 1) atomicExch(A.bad, 1);
    // half storage: block (i, j) of an omitted chunk is block (j, i), which
    // its own chunk stores (the relation above is still checked for all pairs)
    if (A.half && half_q0(p, A.TC / A.TR) > q) continue;
    const bool near = kept_apart(A, rel);
    if (A.count_only) {
      if (near) atomicAdd(&A.near_fill[i], 1);
      continue;
    }
    double N6[6];
    if (A.table) {
#pragma unroll
      for (int e = 0; e < 6; ++e) N6[e] = A.table[6 * toff + e];
    } else {
      cuboid_tensor(ci, cj, ej, N6);
    }
    store_block(A, i, j, near, N6);
  }
}

// Tetrahedra: a block needs the source tile's ~90 doubles of geometry, so the
// roles are turned round: a CTA stages kTetCols source tiles in shared memory
// (read by all its threads at once: broadcasts) and thread t takes field
// point i = kTetRows blockIdx.y + t.
constexpr int kTetCols = 16, kTetRows = 128;
__global__ void __launch_bounds__(kTetRows) k_assemble_tetra(AsmArgs A) {
  __shared__ double sg[kTetCols * kTgSize];
  const int64_t j0 = blockIdx.x * (int64_t)kTetCols;
  const int cols = (int)(A.n - j0 < kTetCols ? A.n - j0 : kTetCols);
  for (int q = threadIdx.x; q < cols * kTgSize; q += kTetRows) sg[q] = A.geo[j0 * kTgSize + q];
  __syncthreads();
  const int64_t i = blockIdx.y * (int64_t)kTetRows + threadIdx.x;
  if (i >= A.n) return;
  double ci[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) ci[a] = A.centre[3 * i + a];
  const double rad = A.geo[i * kTgSize + kTgRad];
  for (int k = 0; k < cols; ++k) {
    const int64_t j = j0 + k;
    const double *G = sg + k * kTgSize;
    int rel = 2;
    if (i != j) {
      // tiles further apart than their vertices reach from the centroids
      // neither share a vertex nor hold each other's centroid
      double d[3];
      sub3(ci, G + kTgCen, d);
      const double reach = (rad + G[kTgRad]) * (1.0 + 1e-9);
      rel = dot3(d, d) > reach * reach ? 0 : tetra_relation(ci, A.vert + 12 * i, G + kTgVert);
    }
    if (rel & 1) atomicExch(A.bad, 1);
    const bool near = kept_apart(A, rel);
    if (A.count_only) {
      if (near) atomicAdd(&A.near_fill[i], 1);
      continue;
    }
    double N6[6];
    tetra_tensor(ci, G, N6);
    store_block(A, i, j, near, N6);
  }
}

void launch_assemble(const AsmArgs &A, const mt_layout &L) {
  if (A.geo)
    k_assemble_tetra<<<dim3((unsigned)((A.n + kTetCols - 1) / kTetCols), (unsigned)((A.n + kTetRows - 1) / kTetRows)),
                       kTetRows>>>(A);
  else
    k_assemble<<<dim3((unsigned)L.Q, (unsigned)L.P), L.TC>>>(A);
}

// sort each row's near blocks by column so that the FP64 near sum has a
// fixed order (one thread per row; rows hold at most 27 entries for cuboid
// grids, a few dozen for tetrahedral meshes)
__global__ void k_sort_near(int64_t n, const int32_t *ptr, int32_t *col, double *val) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t b = ptr[i], e = ptr[i + 1];
  for (int32_t a = b + 1; a < e; ++a) {
    const int32_t cj = col[a];
    double v[6];
    for (int q = 0; q < 6; ++q) v[q] = val[6 * a + q];
    int32_t z = a - 1;
    while (z >= b && col[z] > cj) {
      col[z + 1] = col[z];
      for (int q = 0; q < 6; ++q) val[6 * (z + 1) + q] = val[6 * z + q];
      --z;
    }
    col[z + 1] = cj;
    for (int q = 0; q < 6; ++q) val[6 * (z + 1) + q] = v[q];
  }
}

// near blocks times the source tile's Ms as FP32 hi + lo pairs
// (N_ij Ms_j = hi + lo to ~2^-48 relative; Ms_j as the FP32 value every
// product uses), so that the near product multiplies plain m
__global__ void k_near_split(int64_t count6, const double *val, const int32_t *col, const float *Ms, float2 *hl) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count6) return;
  const double v = val[t] * (double)Ms[col[t / 6]];
  const float hi = (float)v;
  hl[t] = make_float2(hi, (float)(v - (double)hi));
}

__global__ void k_blocks(const double *centre, const double *edge, const double *vert, int kind, int64_t count,
                         const int64_t *pairs, double *out) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= count) return;
  const int64_t i = pairs[2 * p], j = pairs[2 * p + 1];
  if (kind == MT_TILE_TETRA) {
    double G[kTgSize];
    tetra_geom(&centre[3 * j], &vert[12 * j], G);
    tetra_tensor(&centre[3 * i], G, &out[6 * p]);
  } else
    cuboid_tensor(&centre[3 * i], &centre[3 * j], &edge[3 * j], &out[6 * p]);
}

// stored value -> double, rows [i0, i1), all columns; out[((i-i0)*n + j)*6 + e]
__global__ void k_read_rows(const void *data, const int8_t *scale, int prec, int64_t n, int TR, int TC,
                            int nplane, int64_t Q, bool hs, int64_t i0, int64_t i1, double *out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t rows = i1 - i0;
  if (t >= rows * n) return;
  const int64_t i = i0 + t / n, j = t % n;
  for (int e = 0; e < 6; ++e) {
    double v = 0.0;
    switch (prec) {
      case MT_F64: v = ((const double *)data)[layout_index(i, j, e, TR, TC, 6, Q)]; break;
      case MT_F32: {
        auto stored = [&](int ee) {
          const int pl = stream_plane(ee, nplane);
          int64_t at = pl < 0 ? -1 : layout_index_h(i, j, pl, TR, TC, nplane, Q, hs);
          if (pl >= 0 && at < 0) at = layout_index_h(j, i, pl, TR, TC, nplane, Q, hs);  // N_ij = N_ji
          return pl < 0 ? 0.0 : (double)((const float *)data)[at];
        };
        if (traceless(nplane) && e == 5)  // zz from the trace: delta_ij - xx - yy of the stored values, in FP32
          v = (double)((i == j ? 1.0f : 0.0f) - ((float)stored(0) + (float)stored(3)));
        else
          v = stored(e);
      } break;
      case MT_BF16_SCALED: {
        const int pl = stream_plane(e, nplane);
        v = pl < 0 ? 0.0
                   : ldexp((double)__bfloat162float(
                               ((const __nv_bfloat16 *)data)[layout_index(i, j, pl, TR, TC, nplane, Q)]),
                           (int)scale[scale_index(i, j, TR, TC, Q)]);
      } break;
      case MT_BF16_SPLIT: {
        const int half = nplane / 2, pl = stream_plane(e, half);
        const __nv_bfloat16 *d = (const __nv_bfloat16 *)data;
        v = pl < 0 ? 0.0
                   : (double)__bfloat162float(d[layout_index(i, j, pl, TR, TC, nplane, Q)]) +
                         (double)__bfloat162float(d[layout_index(i, j, half + pl, TR, TC, nplane, Q)]);
      } break;
    }
    out[t * 6 + e] = v;
  }
}

// dense layout -> double, rows [i0, i1)
__global__ void k_read_rows_dense(const __nv_bfloat16 *D, bool split, int64_t n, int64_t KB, int np, int64_t i0,
                                  int64_t i1, double *out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t rows = i1 - i0;
  if (t >= rows * n) return;
  const int64_t i = i0 + t / n, j = t % n;
  for (int e = 0; e < 6; ++e) {
    const int pl = stream_plane(e, np);
    double v = 0.0;
    if (pl >= 0) {
      const size_t at = dense_a_index(i, j, pl, KB, np, split);
      v = (double)__bfloat162float(D[at]);
      if (split) v += (double)__bfloat162float(D[at + kDenseLo]);
    }
    out[t * 6 + e] = v;
  }
}

// merge the FP64 near blocks of rows [i0, i1) into out
__global__ void k_merge_near(int64_t n, int64_t i0, int64_t i1, const int32_t *ptr, const int32_t *col,
                             const double *val, double *out) {
  const int64_t i = i0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= i1) return;
  for (int32_t a = ptr[i]; a < ptr[i + 1]; ++a) {
    const int64_t j = col[a];
    for (int e = 0; e < 6; ++e) out[((i - i0) * n + j) * 6 + e] = val[6 * a + e];
  }
}

}  // namespace

namespace mt {

mt_status assemble(mt_tensor *T) {
  mt_tiles *t = T->tiles;
  const int64_t n = T->n;
  const mt_layout &L = T->L;
  DevTemp<int> bad_flag;
  MT_CUDA(bad_flag.alloc(2));
  int *d_bad = bad_flag.p;
  MT_CUDA(cudaMemset(d_bad, 0, 2 * sizeof(int)));
  AsmArgs A{};
  A.centre = t->d_centre;
  A.edge = t->d_edge;
  A.vert = t->d_vert;
  A.n = n;
  A.TR = L.TR;
  A.TC = L.TC;
  A.nplane = L.nplane;
  A.Q = L.Q;
  A.prec = T->prec;
  A.data = T->d_data;
  A.scale = T->d_scale;
  A.bad = d_bad;
  A.planar_bad = d_bad + 1;
  A.dense = T->layout == MT_LAYOUT_DENSE;
  A.half = T->L.half ? 1 : 0;
  A.Kp = T->Kp;
  DevTemp<double> table;
  double *d_table = nullptr;
  if (t->lattice && t->kind == MT_TILE_CUBOID) {
    const int64_t cnt = (int64_t)(2 * t->Lx - 1) * (2 * t->Ly - 1) * (2 * t->Lz - 1);
    MT_CUDA(table.alloc(6 * cnt));
    d_table = table.p;
    k_offset_table<<<(unsigned)((cnt + 127) / 128), 128>>>(t->Lx, t->Ly, t->Lz, t->lat_edge[0], t->lat_edge[1],
                                                          t->lat_edge[2], d_table);
    MT_CUDA(cudaGetLastError());
    A.table = d_table;
    A.lat = t->d_lat;
    A.Lx = t->Lx;
    A.Ly = t->Ly;
    A.Lz = t->Lz;
  }
  DevTemp<double> geo;
  if (t->kind == MT_TILE_TETRA) {
    MT_CUDA(geo.alloc((size_t)kTgSize * n));
    k_tetra_geom<<<(unsigned)((n + 127) / 128), 128>>>(n, t->d_centre, t->d_vert, geo.p);
    MT_CUDA(cudaGetLastError());
    A.geo = geo.p;
  }
  const bool has_near = (T->prec == MT_BF16_SCALED || T->prec == MT_BF16_SPLIT);
  DevTemp<int> fill;  // per-row counters of the blocks kept apart
  if (has_near) {
    MT_CUDA(fill.alloc(n));
    MT_CUDA(cudaMemset(fill.p, 0, sizeof(int) * n));
    A.near_fill = fill.p;
    A.count_only = 1;
    launch_assemble(A, L);
    MT_CUDA(cudaGetLastError());
    std::vector<int> cnt(n);
    MT_CUDA(cudaMemcpy(cnt.data(), fill.p, sizeof(int) * n, cudaMemcpyDeviceToHost));
    std::vector<int32_t> ptr(n + 1, 0);
    for (int64_t i = 0; i < n; ++i) ptr[i + 1] = ptr[i] + cnt[i];
    T->near_count = ptr[n];
    MT_CUDA(cudaMalloc(&T->d_near_ptr, sizeof(int32_t) * (n + 1)));
    MT_CUDA(cudaMalloc(&T->d_near_col, sizeof(int32_t) * std::max<int64_t>(1, T->near_count)));
    MT_CUDA(cudaMalloc(&T->d_near_val, sizeof(double) * 6 * std::max<int64_t>(1, T->near_count)));
    MT_CUDA(cudaMalloc(&T->d_near_hl, sizeof(float2) * 6 * std::max<int64_t>(1, T->near_count)));
    MT_CUDA(cudaMemcpy(T->d_near_ptr, ptr.data(), sizeof(int32_t) * (n + 1), cudaMemcpyHostToDevice));
    A.near_ptr = T->d_near_ptr;
    A.near_col = T->d_near_col;
    A.near_val = T->d_near_val;
    A.count_only = 0;
  }
  // every block into its place (again with another layout, should the first
  // turn out not to hold the tensor)
  auto fill_all = [&]() -> mt_status {
    if (has_near) MT_CUDA(cudaMemset(fill.p, 0, sizeof(int) * n));
    launch_assemble(A, T->L);
    MT_CUDA(cudaGetLastError());
    if (T->near_count > 0) {
      k_sort_near<<<(unsigned)((n + 127) / 128), 128>>>(n, T->d_near_ptr, T->d_near_col, T->d_near_val);
      k_near_split<<<(unsigned)((6 * T->near_count + 255) / 256), 256>>>(6 * T->near_count, T->d_near_val,
                                                                        T->d_near_col, t->d_Ms, T->d_near_hl);
      MT_CUDA(cudaGetLastError());
    }
    MT_CUDA(cudaDeviceSynchronize());
    return MT_OK;
  };
  mt_status st = fill_all();
  if (st != MT_OK) return st;
  int bad[2] = {0, 0};
  MT_CUDA(cudaMemcpy(bad, d_bad, 2 * sizeof(int), cudaMemcpyDeviceToHost));
  MT_CHECK(!bad[0], MT_EOVERLAP, "mt_demag_assemble: tiles overlap or a tile centre lies on another tile");
  if (bad[1] && (T->L.nplane == 4 || traceless(T->L.nplane))) {
    // an xz or yz entry of the single-layer set is not round-off, or (3
    // planes) a block's trace is off its identity: store all 6 planes after
    // all (within the budget reserved for them)
    mt_ctx *ctx = t->ctx;
    const bool half = T->L.half;
    size_t data_bytes;
    if (A.dense) {
      T->L.nplane = 6;
      data_bytes = dense_tensor_bytes(n, T->prec, 6);
    } else {
      layout_for(T->prec, &T->L);
      T->L.P = (n + T->L.TR - 1) / T->L.TR;
      T->L.Q = (n + T->L.TC - 1) / T->L.TC;
      T->L.half = half;
      T->L.CH = half ? half_chunks(T->L.P, T->L.Q, T->L.TC / T->L.TR) : T->L.P * T->L.Q;
      data_bytes = (size_t)T->L.CH * T->L.chunk_bytes();
    }
    const size_t bytes = data_bytes + (A.dense ? 0 : (size_t)T->L.CH * T->L.scale_bytes_per_chunk);
    {
      std::lock_guard<std::mutex> lk(ctx->mu);
      MT_CHECK(ctx->in_use - T->bytes + bytes <= ctx->budget, MT_ENOMEM,
               "mt_demag_assemble: %zu bytes exceed the context budget", bytes);
      ctx->in_use += bytes - T->bytes;
      T->bytes = bytes;
    }
    MT_CUDA(cudaFree(T->d_data));
    T->d_data = nullptr;
    MT_CUDA(cudaMalloc(&T->d_data, data_bytes));
    MT_CUDA(cudaMemset(T->d_data, 0, data_bytes));
    A.data = T->d_data;
    A.TR = T->L.TR;
    A.TC = T->L.TC;
    A.nplane = T->L.nplane;
    A.Q = T->L.Q;
    return fill_all();
  }
  return MT_OK;
}

mt_status blocks_fp64(mt_tiles *t, int64_t count, const int64_t *pairs, double *out) {
  if (count == 0) return MT_OK;
  for (int64_t p = 0; p < 2 * count; ++p)
    MT_CHECK(pairs[p] >= 0 && pairs[p] < t->n, MT_EINVAL, "mt_demag_blocks: pair index out of range");
  int64_t *d_pairs = nullptr;
  double *d_out = nullptr;
  MT_CUDA(cudaMalloc(&d_pairs, sizeof(int64_t) * 2 * count));
  MT_CUDA(cudaMalloc(&d_out, sizeof(double) * 6 * count));
  MT_CUDA(cudaMemcpy(d_pairs, pairs, sizeof(int64_t) * 2 * count, cudaMemcpyHostToDevice));
  k_blocks<<<(unsigned)((count + 127) / 128), 128>>>(t->d_centre, t->d_edge, t->d_vert, t->kind, count, d_pairs,
                                                     d_out);
  MT_CUDA(cudaGetLastError());
  MT_CUDA(cudaMemcpy(out, d_out, sizeof(double) * 6 * count, cudaMemcpyDeviceToHost));
  cudaFree(d_pairs);
  cudaFree(d_out);
  return MT_OK;
}

mt_status read_rows(const mt_tensor *T, int64_t i0, int64_t i1, double *out) {
  const int64_t n = T->n;
  const int64_t rows = i1 - i0;
  if (rows <= 0) return MT_OK;
  double *d_out = nullptr;
  MT_CUDA(cudaMalloc(&d_out, sizeof(double) * 6 * rows * n));
  const int64_t tot = rows * n;
  if (T->layout == MT_LAYOUT_DENSE)
    k_read_rows_dense<<<(unsigned)((tot + 255) / 256), 256>>>((const __nv_bfloat16 *)T->d_data,
                                                              T->prec == MT_BF16_SPLIT, n, T->Kp / 64, T->L.nplane,
                                                              i0, i1, d_out);
  else
    k_read_rows<<<(unsigned)((tot + 255) / 256), 256>>>(T->d_data, T->d_scale, T->prec, n, T->L.TR, T->L.TC,
                                                         T->L.nplane, T->L.Q, T->L.half, i0, i1, d_out);
  MT_CUDA(cudaGetLastError());
  if (T->near_count > 0) {
    k_merge_near<<<(unsigned)((rows + 127) / 128), 128>>>(n, i0, i1, T->d_near_ptr, T->d_near_col,
                                                          T->d_near_val, d_out);
    MT_CUDA(cudaGetLastError());
  }
  MT_CUDA(cudaMemcpy(out, d_out, sizeof(double) * 6 * rows * n, cudaMemcpyDeviceToHost));
  cudaFree(d_out);
  return MT_OK;
}

}  // namespace mt
