// k_refine.cu — near-wall refinement of one grid level, child compaction and
// the finest level's adjacent-face lists.
//
// Paper (Sec. "Identification of Cells Near the Boundary", "Face Detection",
// "Spatial Binning Algorithm"): every cell of every block of the level checks
// the faces stored in the bins around it; a block with an adjacent cell is
// marked and M_RefineAndCoarsenBlocks subdivides it.  The paper maps one
// thread to one cell (thread block = cell block) and tests the cell centre
// against the face with Alg. 1.
//
// Here one warp owns one block of 4^D cells (two cells per lane in 3D).  The
// warp walks the bins overlapped by the block's query box (block inflated by
// d_L); each lane takes one bin entry, visits it only in its canonical bin
// (so a face seen in several bins is tested once), and runs the separating-axis
// test of the face against the whole inflated block.  Survivors leave their
// per-axis projection intervals in shared memory and every lane tests its
// cells against them.  The adjacency bits are combined with warp ballots.
//
// Decisions are exact: each FP32 axis test carries a forward error bound; a
// (cell, face) pair whose sign is not certified on every axis is re-evaluated
// in FP64 (and counted).  Block-level culls only use certified separations.
#include <algorithm>
#include <type_traits>

#include "internal.cuh"

namespace amr {

namespace {

constexpr float kEpsK = 16.0f;  // safety factor over the forward error bound (see axis_bound)

template <int D>
struct Surv;

// Per-survivor data in the block frame (origin = the block's lower corner).
// Axis order (3D): 0..2 box axes, 3 face normal, 4 + 3k + i = e_i x edge_k.
// Per axis the cell-centre projection x is tested against four thresholds
// t = (lo - eps, hi + eps, lo + eps, hi - eps), [lo, hi] being the face's
// projection widened by the cell's: x < t.x or x > t.y certifies separation,
// t.z < x < t.w certifies overlap, anything else is not certified.
template <>
struct Surv<3> {
  float4 en[3];  // e0.xyz e1.x | e1.yz e2.xy | e2.z n.xyz
  float4 t[13];
  uint32_t face;
  uint32_t pad[3];
};
// 2D: 0..1 box axes, 2 segment normal (-e_y, e_x).
template <>
struct Surv<2> {
  float4 t[3];
  float e[2];
  uint32_t face;
  uint32_t pad[1];
};

// FP64 decision of the separating-axis test of the box [x_c - r, x_c + r]^3
// and the closed triangle (vertices absolute FP32).  The margin of the
// definition is max over the 13 axes of gap_a / |a| (gap_a = the FP64 gap
// between the projected intervals); its sign is that of the largest gap_a, so
// the pair is adjacent exactly when no axis has gap_a > 0, and no square root
// or division is needed (a quotient of normal magnitudes does not underflow).
// *band: the margin lies within tol of 0, tested as gap_a^2 <= tol^2 |a|^2 on
// the deciding axes (a diagnostic count).  An axis with gap_a > tol |a| settles
// the pair at once: separated, outside the band.
__device__ __noinline__ bool sat_adjacent_fp64_3(const float* V, const double* xc, double r, double tol,
                                                 bool* band) {
  double p[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) p[k][c] = __dsub_rn((double)V[3 * k + c], xc[c]);
  const double tol2 = tol * tol;
  bool sep = false;        // some axis with a positive gap
  bool pos_small = true;   // every positive gap within tol |a|
  bool near0 = false;      // some axis with gap >= -tol |a|
  // false: the pair is settled (separated beyond the band)
  auto axis = [&](double a0, double a1, double a2) -> bool {
    const double l2sq = __dadd_rn(__dadd_rn(__dmul_rn(a0, a0), __dmul_rn(a1, a1)), __dmul_rn(a2, a2));
    if (l2sq == 0.0) return true;
    double lo = 1e300, hi = -1e300;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double s = __dadd_rn(__dadd_rn(__dmul_rn(p[k][0], a0), __dmul_rn(p[k][1], a1)), __dmul_rn(p[k][2], a2));
      lo = fmin(lo, s);
      hi = fmax(hi, s);
    }
    const double R = __dmul_rn(r, __dadd_rn(__dadd_rn(fabs(a0), fabs(a1)), fabs(a2)));
    const double g = fmax(__dsub_rn(lo, R), __dsub_rn(-R, hi));
    const bool small = __dmul_rn(g, g) <= __dmul_rn(tol2, l2sq);
    if (g > 0.0) {
      sep = true;
      if (!small) {
        pos_small = false;
        return false;
      }
    } else if (small) {
      near0 = true;
    }
    return true;
  };
  *band = false;
  if (!axis(1.0, 0.0, 0.0) || !axis(0.0, 1.0, 0.0) || !axis(0.0, 0.0, 1.0)) return false;
  const double u0 = __dsub_rn(p[1][0], p[0][0]), u1 = __dsub_rn(p[1][1], p[0][1]), u2 = __dsub_rn(p[1][2], p[0][2]);
  const double w0 = __dsub_rn(p[2][0], p[0][0]), w1 = __dsub_rn(p[2][1], p[0][1]), w2 = __dsub_rn(p[2][2], p[0][2]);
  if (!axis(__dsub_rn(__dmul_rn(u1, w2), __dmul_rn(u2, w1)), __dsub_rn(__dmul_rn(u2, w0), __dmul_rn(u0, w2)),
            __dsub_rn(__dmul_rn(u0, w1), __dmul_rn(u1, w0))))
    return false;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3;
    const double ex = __dsub_rn(p[k1][0], p[k][0]), ey = __dsub_rn(p[k1][1], p[k][1]),
                 ez = __dsub_rn(p[k1][2], p[k][2]);
    if (!axis(0.0, -ez, ey) || !axis(ez, 0.0, -ex) || !axis(-ey, ex, 0.0)) return false;
  }
  *band = sep ? pos_small : near0;
  return !sep;
}

__device__ __noinline__ double margin_fp64_2(const float* V, const double* xc, double r) {
  double p[2][2];
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int c = 0; c < 2; ++c) p[k][c] = __dsub_rn((double)V[2 * k + c], xc[c]);
  double m = -1e300;
  auto axis = [&](double a0, double a1) {
    const double l2 = sqrt(__dadd_rn(__dmul_rn(a0, a0), __dmul_rn(a1, a1)));
    if (l2 == 0.0) return;
    const double s0 = __dadd_rn(__dmul_rn(p[0][0], a0), __dmul_rn(p[0][1], a1));
    const double s1 = __dadd_rn(__dmul_rn(p[1][0], a0), __dmul_rn(p[1][1], a1));
    const double lo = fmin(s0, s1), hi = fmax(s0, s1);
    const double R = __dmul_rn(r, __dadd_rn(fabs(a0), fabs(a1)));
    m = fmax(m, fmax(__dsub_rn(lo, R), __dsub_rn(-R, hi)) / l2);
  };
  axis(1.0, 0.0);
  axis(0.0, 1.0);
  const double e0 = __dsub_rn(p[1][0], p[0][0]), e1 = __dsub_rn(p[1][1], p[0][1]);
  axis(-e1, e0);
  return m;
}

// FP64 distance from the point xc to the closed face (vertices absolute FP32):
// the plane distance when the projection lies in the closed triangle, else the
// smallest distance to the three edges (the point predicate of Alg. 1).
__device__ __forceinline__ double seg_dist2_fp64(const double* a, const double* b, int dim) {
  double e[3] = {0, 0, 0}, ae = 0.0, ee = 0.0;
  for (int c = 0; c < dim; ++c) {
    e[c] = __dsub_rn(b[c], a[c]);
    ae = __fma_rn(-a[c], e[c], ae);
    ee = __fma_rn(e[c], e[c], ee);
  }
  const double t = ee > 0.0 ? fmin(1.0, fmax(0.0, ae / ee)) : 0.0;
  double d2 = 0.0;
  for (int c = 0; c < dim; ++c) {
    const double q = __fma_rn(t, e[c], a[c]);
    d2 = __fma_rn(q, q, d2);
  }
  return d2;
}

__device__ __noinline__ double point_dist_fp64(const float* V, const double* xc, int dim) {
  double p[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  for (int k = 0; k < dim; ++k)
    for (int c = 0; c < dim; ++c) p[k][c] = __dsub_rn((double)V[dim * k + c], xc[c]);
  if (dim == 2) return sqrt(seg_dist2_fp64(p[0], p[1], 2));
  const double u[3] = {p[1][0] - p[0][0], p[1][1] - p[0][1], p[1][2] - p[0][2]};
  const double w[3] = {p[2][0] - p[0][0], p[2][1] - p[0][1], p[2][2] - p[0][2]};
  const double n[3] = {u[1] * w[2] - u[2] * w[1], u[2] * w[0] - u[0] * w[2], u[0] * w[1] - u[1] * w[0]};
  const double nn = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
  if (nn > 0.0) {
    bool neg = true, pos = true;
    for (int k = 0; k < 3; ++k) {
      const double* a = p[k];
      const double* b = p[(k + 1) % 3];
      const double e[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
      const double m[3] = {e[1] * n[2] - e[2] * n[1], e[2] * n[0] - e[0] * n[2], e[0] * n[1] - e[1] * n[0]};
      const double sk = -(a[0] * m[0] + a[1] * m[1] + a[2] * m[2]);
      if (sk > 0.0) neg = false;
      if (sk < 0.0) pos = false;
    }
    if (neg || pos) return fabs(p[0][0] * n[0] + p[0][1] * n[1] + p[0][2] * n[2]) / sqrt(nn);
  }
  return sqrt(fmin(seg_dist2_fp64(p[0], p[1], 3), fmin(seg_dist2_fp64(p[1], p[2], 3), seg_dist2_fp64(p[2], p[0], 3))));
}

// Block-frame quantities shared by all lanes of the warp for one block.
template <int D>
struct BlockFrame {
  float Xb[3];     // block corner rounded to FP32 (the frame origin)
  float cB[3];     // block centre in the frame
  float h, r, rb;  // cell size, cell and block half-widths (inflated) in FP32
  float O;         // bound on |cell centre offsets| and |block centre| in the frame
};

// Per-face setup (one lane): edges, projections of the face on every axis in
// the block frame, the cell-level intervals [tmin - r|a|_1, tmax + r|a|_1] and
// their error bounds.  Returns false when some axis certifiably separates the
// face from the whole inflated block.  Without kCull (face-by-face marking, which has no block) the face is
// kept whatever the block would say.
//
// Error bound per axis a: every computed projection, interval end and cell
// coordinate differs from its exact value by at most a few unit roundoffs of
// (P + O + r) |a|_1, where P bounds the vertex offsets in the frame (this also
// covers the rounding of the frame origin, of the edges when they are not
// exact and of the FP32 normal relative to the FP64 one).  eps = 16 u (P+O+r)|a|_1.
template <int D, bool kCull = true>
__device__ __forceinline__ bool setup_face(const float* V, const float* nh, const BlockFrame<D>& F, Surv<D>& S) {
  float p[3][3];
  float P = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int c = 0; c < D; ++c) {
      p[k][c] = V[D * k + c] - F.Xb[c];
      P = fmaxf(P, fabsf(p[k][c]));
    }
  const float scale = kEpsK * kU32 * (P + F.O + F.r);
  // one axis: false when it certifiably separates the face from the whole inflated block
  auto axis = [&](int ai, float ax, float ay, float az) -> bool {
    const float A1 = fabsf(ax) + fabsf(ay) + fabsf(az);
    if (A1 == 0.0f) {
      S.t[ai] = make_float4(-INFINITY, INFINITY, -INFINITY, INFINITY);
      return true;
    }
    float tmin = INFINITY, tmax = -INFINITY;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const float s = D == 3 ? fmaf(p[k][2], az, fmaf(p[k][1], ay, p[k][0] * ax)) : fmaf(p[k][1], ay, p[k][0] * ax);
      tmin = fminf(tmin, s);
      tmax = fmaxf(tmax, s);
    }
    const float eps = scale * A1;
    if constexpr (!kCull) {
      const float R = F.r * A1;
      const float lo = tmin - R, hi = tmax + R;
      S.t[ai] = make_float4(lo - eps, hi + eps, lo + eps, hi - eps);
      return true;
    }
    const float xb = D == 3 ? fmaf(F.cB[2], az, fmaf(F.cB[1], ay, F.cB[0] * ax)) : fmaf(F.cB[1], ay, F.cB[0] * ax);
    const float RB = F.rb * A1;
    // block interval [xb - RB, xb + RB] vs face interval [tmin, tmax]
    if (xb - RB - tmax > eps || tmin - (xb + RB) > eps) return false;
    const float R = F.r * A1;
    const float lo = tmin - R, hi = tmax + R;
    S.t[ai] = make_float4(lo - eps, hi + eps, lo + eps, hi - eps);
    return true;
  };
  if constexpr (D == 3) {
    float e[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int k1 = (k + 1) % 3;
#pragma unroll
      for (int c = 0; c < 3; ++c) e[k][c] = V[3 * k1 + c] - V[3 * k + c];
    }
    // box axes first: the cheap AABB cull
    if (!axis(0, 1.f, 0.f, 0.f) || !axis(1, 0.f, 1.f, 0.f) || !axis(2, 0.f, 0.f, 1.f)) return false;
    if (!axis(3, nh[0], nh[1], nh[2])) return false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
      if (!axis(4 + 3 * k, 0.f, -ez, ey)) return false;
      if (!axis(5 + 3 * k, ez, 0.f, -ex)) return false;
      if (!axis(6 + 3 * k, -ey, ex, 0.f)) return false;
    }
    S.en[0] = make_float4(e[0][0], e[0][1], e[0][2], e[1][0]);
    S.en[1] = make_float4(e[1][1], e[1][2], e[2][0], e[2][1]);
    S.en[2] = make_float4(e[2][2], nh[0], nh[1], nh[2]);
  } else {
    const float e0 = V[2] - V[0], e1 = V[3] - V[1];
    if (!axis(0, 1.f, 0.f, 0.f) || !axis(1, 0.f, 1.f, 0.f)) return false;
    if (!axis(2, -e1, e0, 0.f)) return false;
    S.e[0] = e0;
    S.e[1] = e1;
  }
  return true;
}

// Cell tests of the lane's two cells against one survivor: 0 = separated,
// 1 = intersecting, 2 = not certified (needs FP64).  o0 / o1 are the cell
// centres in the block frame.  All axes are evaluated (the warp runs the
// longest lane anyway); the thresholds come as one 16-byte load per axis.
template <int D>
__device__ __forceinline__ void cell_test2(const Surv<D>& S, const float* o0, const float* o1, int& r0, int& r1) {
  bool sep0 = false, in0 = true, sep1 = false, in1 = true;
  auto upd = [](float x, const float4& t, bool& sep, bool& in) {
    sep |= (x < t.x) | (x > t.y);
    in &= (x > t.z) & (x < t.w);
  };
  if constexpr (D == 3) {
#pragma unroll
    for (int ai = 0; ai < 3; ++ai) {
      const float4 t = S.t[ai];
      upd(o0[ai], t, sep0, in0);
      upd(o1[ai], t, sep1, in1);
    }
    const float4 q0 = S.en[0], q1 = S.en[1], q2 = S.en[2];
    const float e[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
    {
      const float4 t = S.t[3];
      upd(fmaf(o0[2], q2.w, fmaf(o0[1], q2.z, o0[0] * q2.y)), t, sep0, in0);
      upd(fmaf(o1[2], q2.w, fmaf(o1[1], q2.z, o1[0] * q2.y)), t, sep1, in1);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
      const float4 ta = S.t[4 + 3 * k], tb = S.t[5 + 3 * k], tc = S.t[6 + 3 * k];
      upd(fmaf(o0[2], ey, -o0[1] * ez), ta, sep0, in0);
      upd(fmaf(o1[2], ey, -o1[1] * ez), ta, sep1, in1);
      upd(fmaf(o0[0], ez, -o0[2] * ex), tb, sep0, in0);
      upd(fmaf(o1[0], ez, -o1[2] * ex), tb, sep1, in1);
      upd(fmaf(o0[1], ex, -o0[0] * ey), tc, sep0, in0);
      upd(fmaf(o1[1], ex, -o1[0] * ey), tc, sep1, in1);
    }
  } else {
#pragma unroll
    for (int ai = 0; ai < 2; ++ai) upd(o0[ai], S.t[ai], sep0, in0);
    upd(fmaf(o0[1], S.e[0], -o0[0] * S.e[1]), S.t[2], sep0, in0);
    sep1 = true;
  }
  r0 = sep0 ? 0 : (in0 ? 1 : 2);
  r1 = sep1 ? 0 : (in1 ? 1 : 2);
}

// Point predicate: survivor data in the block frame, stored over the
// thresholds of the box predicate.  3D layout: t[0..2] = vertex k (xyz) with
// 1/|n|^2 (0: zero-area face) and the error scale in .w of t[0] / t[1];
// t[3..5] = edge e_k = p_{k+1} - p_k with 1/|e_k|^2; t[6..8] = m_k = e_k x n
// with the edge-function error scale in t[6].w; t[9] = n.
// Error analysis (u = 2^-24, L = bound on |coordinates| in the frame, vertex
// offsets plus cell-centre offsets): every difference w = x - p_k carries one
// rounding (<= 2uL per component), the squared edge and plane distances are
// sums of a few products of such terms and are within 64 u (2 sqrt(3) L)^2 of
// their exact values; an edge function m_k . w_k is within 96 u L |e_k|_1 |n|_1.
template <int D>
__device__ __forceinline__ void setup_point(const float* V, const float* nh, const BlockFrame<D>& F, Surv<D>& S) {
  float p[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  float P = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int c = 0; c < D; ++c) {
      p[k][c] = V[D * k + c] - F.Xb[c];
      P = fmaxf(P, fabsf(p[k][c]));
    }
  const float L = P + F.O;
  const float E = 64.0f * kU32 * 12.0f * L * L;
  if constexpr (D == 3) {
    float e[3][3], m[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) e[k][c] = p[(k + 1) % 3][c] - p[k][c];
    const float nn = nh[0] * nh[0] + nh[1] * nh[1] + nh[2] * nh[2];
    const float n1 = fabsf(nh[0]) + fabsf(nh[1]) + fabsf(nh[2]);
    float m1 = 0.f;  // bound on |m_k|_1 and on its rounding, max_k |e_k|_1 |n|_1
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      m[k][0] = e[k][1] * nh[2] - e[k][2] * nh[1];
      m[k][1] = e[k][2] * nh[0] - e[k][0] * nh[2];
      m[k][2] = e[k][0] * nh[1] - e[k][1] * nh[0];
      m1 = fmaxf(m1, (fabsf(e[k][0]) + fabsf(e[k][1]) + fabsf(e[k][2])) * n1);
    }
    S.t[0] = make_float4(p[0][0], p[0][1], p[0][2], nn > 0.f ? 1.0f / nn : 0.f);
    S.t[1] = make_float4(p[1][0], p[1][1], p[1][2], E);
    S.t[2] = make_float4(p[2][0], p[2][1], p[2][2], 0.f);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ee = e[k][0] * e[k][0] + e[k][1] * e[k][1] + e[k][2] * e[k][2];
      S.t[3 + k] = make_float4(e[k][0], e[k][1], e[k][2], ee > 0.f ? 1.0f / ee : 0.f);
      S.t[6 + k] = make_float4(m[k][0], m[k][1], m[k][2], k == 0 ? 96.0f * kU32 * m1 * L : 0.f);
    }
    S.t[9] = make_float4(nh[0], nh[1], nh[2], 0.f);
  } else {
    const float e0 = p[1][0] - p[0][0], e1 = p[1][1] - p[0][1];
    const float ee = e0 * e0 + e1 * e1;
    S.t[0] = make_float4(p[0][0], p[0][1], e0, e1);
    S.t[1] = make_float4(ee > 0.f ? 1.0f / ee : 0.f, E, 0.f, 0.f);
  }
}

// Squared distance from w (= x - p) to the segment p + s e, s in [0, 1].
__device__ __forceinline__ float seg_dist2(float wx, float wy, float wz, const float4& e) {
  const float s = fminf(1.0f, fmaxf(0.0f, (wx * e.x + wy * e.y + wz * e.z) * e.w));
  const float qx = fmaf(-s, e.x, wx), qy = fmaf(-s, e.y, wy), qz = fmaf(-s, e.z, wz);
  return qx * qx + qy * qy + qz * qz;
}

// Point-predicate test of one cell centre o: 0 = farther than d, 1 = within
// d, 2 = not certified (FP64).  The plane distance A is a lower bound of the
// distance and the nearest edge distance Bv an upper bound; A applies when the
// projection is certainly inside the triangle, Bv when it is certainly outside.
template <int D>
__device__ __forceinline__ int point_test(const Surv<D>& S, const float* o, float R2) {
  if constexpr (D == 3) {
    const float4 t0 = S.t[0], t1 = S.t[1], t2 = S.t[2];
    const float E = t1.w;
    const float w[3][3] = {{o[0] - t0.x, o[1] - t0.y, o[2] - t0.z},
                           {o[0] - t1.x, o[1] - t1.y, o[2] - t1.z},
                           {o[0] - t2.x, o[1] - t2.y, o[2] - t2.z}};
    float Bv = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) Bv = fminf(Bv, seg_dist2(w[k][0], w[k][1], w[k][2], S.t[3 + k]));
    if (Bv <= R2 - E) return 1;
    const float4 n = S.t[9];
    const float pn = w[0][0] * n.x + w[0][1] * n.y + w[0][2] * n.z;
    const float A = t0.w > 0.f ? pn * pn * t0.w : 0.f;
    if (A > R2 + E) return 0;
    const float es = S.t[6].w;
    bool neg = true, pos = true, lo = false, hi = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 m = S.t[6 + k];
      const float sk = w[k][0] * m.x + w[k][1] * m.y + w[k][2] * m.z;
      if (!(sk < -es)) neg = false;
      if (!(sk > es)) pos = false;
      if (sk < -es) lo = true;
      if (sk > es) hi = true;
    }
    const bool inside = t0.w > 0.f && (neg || pos);
    const bool outside = t0.w == 0.f || (lo && hi);
    if (inside) return A < R2 - E ? 1 : 2;
    if (outside) return Bv > R2 + E ? 0 : 2;
    return 2;
  } else {
    const float4 t0 = S.t[0], t1 = S.t[1];
    const float d2 = seg_dist2(o[0] - t0.x, o[1] - t0.y, 0.f, make_float4(t0.z, t0.w, 0.f, t1.x));
    if (d2 <= R2 - t1.y) return 1;
    if (d2 > R2 + t1.y) return 0;
    return 2;
  }
}

// Point predicate, quick test: the face's centroid c (in the frame) and the squares of the radii within which
// a cell centre is certainly within d of the face (c is a point of it) and beyond which it certainly is not
// (every point of the face lies within rho of c).  Stored behind setup_point's data.  False when no cell centre
// of the block can be within d.  The radii leave 16 u (P + O) + 8 u d for the rounding of the offsets and of d.
// A face that is small against d settles nearly every cell this way: 8 operations instead of about 100.
// Bound by: issue slots.  3D, 112,500 faces, d = 0.05 of the domain (3 to 12 cells), masks of three levels: 10.98 ->
// 5.50 ms per pass (88.5 million candidates, 7.3 million survivors); sampled bins and own-bin candidates 3.71 ->
// 2.91 ms.  The separating axes (about 100 operations per face and block) are left to faces whose radius passes a
// quarter of the block's: a smaller one leaves the sphere little that the axes could take out.
struct FaceCentre {
  float c[3], in2, out2, rho, P;
};
template <int D>
__device__ __forceinline__ FaceCentre face_centre(const float* V, const BlockFrame<D>& F, float d) {
  FaceCentre C;
  float p[3][3];
  C.P = 0.f;
  C.c[0] = C.c[1] = C.c[2] = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int q = 0; q < D; ++q) {
      p[k][q] = V[D * k + q] - F.Xb[q];
      C.P = fmaxf(C.P, fabsf(p[k][q]));
      C.c[q] += p[k][q];
    }
  float r2 = 0.f;
#pragma unroll
  for (int q = 0; q < D; ++q) C.c[q] *= D == 3 ? 1.0f / 3.0f : 0.5f;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < D; ++q) s = fmaf(p[k][q] - C.c[q], p[k][q] - C.c[q], s);
    r2 = fmaxf(r2, s);
  }
  const float e = 16.0f * kU32 * (C.P + F.O) + 8.0f * kU32 * d;
  C.rho = sqrtf(r2) + e;
  const float in = fmaxf(d - e, 0.f), out = d + C.rho + e;
  // squares that would leave FP32's range: within is left to point_test, beyond starts at a safe one
  C.in2 = in > 1e-15f && in < 1e18f ? in * in * (1.0f - 8.0f * kU32) : -1.0f;
  C.out2 = fmaxf(out * out * (1.0f + 8.0f * kU32), 1e-30f);
  return C;
}

// Squared distance from the centroid to the box ctr +- half (in the frame): beyond out2, no point of the box is
// within d of the face.
template <int D>
__device__ __forceinline__ float centre_to_box2(const FaceCentre& C, const float* ctr, const float* half) {
  float b2 = 0.f;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    const float x = fmaxf(fabsf(C.c[q] - ctr[q]) - half[q], 0.f);
    b2 = fmaf(x, x, b2);
  }
  return b2;
}

template <int D>
__device__ __forceinline__ bool setup_centre(const float* V, const BlockFrame<D>& F, float d, float& rho, Surv<D>& S) {
  const FaceCentre C = face_centre<D>(V, F, d);
  rho = C.rho;
  if constexpr (D == 3) {
    S.t[10] = make_float4(C.c[0], C.c[1], C.c[2], C.out2);
    S.t[11].x = C.in2;
  } else {
    S.t[2] = make_float4(C.c[0], C.c[1], C.out2, C.in2);
  }
  const float half[3] = {1.5f * F.h, 1.5f * F.h, 1.5f * F.h};  // the cell centres' box
  return centre_to_box2<D>(C, F.cB, half) <= C.out2;
}

// A face whose bounding box or plane (line) lies certainly farther than d from the box ctr +- half: differences of
// frame coordinates are within 4 u (P + O), their products with the normal within 32 u |n|_1 (P + O).
template <int D>
__device__ __forceinline__ bool face_beyond(const float* V, const float* nh, const BlockFrame<D>& F, float d, float P,
                                            const float* ctr, const float* half) {
  const float w = P + F.O, e = 8.0f * kU32 * (w + d);
  bool far = false;
  float p0[3], p1[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int q = 0; q < D; ++q) {
    p0[q] = V[q] - F.Xb[q];
    p1[q] = V[D + q] - F.Xb[q];
    float lo = fminf(p0[q], p1[q]), hi = fmaxf(p0[q], p1[q]);
    if (D == 3) {
      const float p2 = V[2 * D + q] - F.Xb[q];
      lo = fminf(lo, p2);
      hi = fmaxf(hi, p2);
    }
    far |= lo - (ctr[q] + half[q]) > d + e || (ctr[q] - half[q]) - hi > d + e;
  }
  float n[3] = {nh[0], nh[1], nh[2]};
  if (D == 2) {
    n[0] = p0[1] - p1[1];
    n[1] = p1[0] - p0[0];
    n[2] = 0.f;
  }
  float s = 0.f, reach = 0.f, n1 = 0.f, n2 = 0.f;
#pragma unroll
  for (int q = 0; q < D; ++q) {
    s = fmaf(n[q], ctr[q] - p0[q], s);
    reach = fmaf(fabsf(n[q]), half[q], reach);
    n1 += fabsf(n[q]);
    n2 = fmaf(n[q], n[q], n2);
  }
  // (2D: the normal is a rounded difference, within 4 u w per component)
  const float en = 32.0f * kU32 * w * (D == 3 ? n1 : n1 + w);
  const float slab = (sqrtf(n2) * d + reach) * (1.0f + 8.0f * kU32) + en;
  return far || (slab < 1e30f && fabsf(s) > slab);
}

// 0 farther than d, 1 within d, 3 left to point_test.
template <int D>
__device__ __forceinline__ int quick_test(const Surv<D>& S, const float* o) {
  float q, out2, in2;
  if constexpr (D == 3) {
    const float4 t = S.t[10];
    const float x = o[0] - t.x, y = o[1] - t.y, z = o[2] - t.z;
    q = fmaf(z, z, fmaf(y, y, x * x));
    out2 = t.w;
    in2 = S.t[11].x;
  } else {
    const float4 t = S.t[2];
    const float x = o[0] - t.x, y = o[1] - t.y;
    q = fmaf(y, y, x * x);
    out2 = t.z;
    in2 = t.w;
  }
  return q > out2 ? 0 : (q <= in2 ? 1 : 3);
}

struct WarpCounters {
  unsigned long long fb = 0, band = 0, cand = 0, surv = 0, big = 0;
};

template <int D>
__device__ __noinline__ bool resolve_fp64(const RefineLevel& a, uint32_t gid, uint32_t face, const int* b,
                                          int cell_local, unsigned long long* fb, unsigned long long* band) {
  const LevelGeom G = level_geom(a.table ? a.table[gid] : a.g0, a.level);
  float V[D * D];
#pragma unroll
  for (int j = 0; j < D * D; ++j) V[j] = a.X[(int64_t)j * a.nf + face];
  double xc[3];
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const int li = (cell_local >> (2 * c)) & 3;
    xc[c] = __dadd_rn(G.origin[c], __dmul_rn((double)(4 * b[c] + li) + 0.5, G.h));
  }
  const double r = __dadd_rn(0.5 * G.h, G.d);
  ++*fb;
  if (D == 3 && a.pred != 1) {
    bool in_band = false;
    const bool adj = sat_adjacent_fp64_3(V, xc, r, kBandRel * G.h, &in_band);
    if (in_band) ++*band;
    return adj;
  }
  const double m = a.pred == 1 ? point_dist_fp64(V, xc, D) - G.d : margin_fp64_2(V, xc, r);
  if (fabs(m) <= kBandRel * G.h) ++*band;
  return m <= 0.0;
}

// FP64 decisions that go one by one by the whole warp (resolve_sat_warp), at most; more of them go a lane each (a
// warp's DP instructions serve 13 axes of one pair there, and here 32 pairs).  A box of 49,152 faces on cell planes,
// 4 levels, 21 M pairs, nearly all exact contacts: marks 146 ms one by one, 26.5 so (walk and marks before: 53.6);
// 768 wide faces of the same box: walk 35.4 and 16.1.  82 K faces with 70 K exact contacts: marks 2.16 and 1.21.
constexpr int kFewFp64 = 6;

// sat_adjacent_fp64_3 by a whole warp, an axis per lane (the same operations in the same order per axis,
// so the same decision and band): an FP64 operation takes tens of cycles here, and one pair's 13 axes in
// a row held its warp for tens of microseconds, which on a small mesh is longer than the rest of a level.
// Every lane passes the same arguments and gets the decision (bit 0; bit 1: in the band).
__device__ __noinline__ uint32_t resolve_sat_warp(const RefineLevel& a, uint32_t gid, uint32_t face, int b0, int b1,
                                                  int b2, int cell_local) {
  const int lane = threadIdx.x & 31;
  const GeomParams& P = a.table ? a.table[gid] : a.g0;
  const double h = scalbn(P.h0, -a.level);
  const double d = __dadd_rn(P.d_abs, __dmul_rn(P.d_rel, h));
  const double r = __dadd_rn(0.5 * h, d), tol = kBandRel * h;
  const int b[3] = {b0, b1, b2};
  double p[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double xc = __dadd_rn(P.origin[c], __dmul_rn((double)(4 * b[c] + ((cell_local >> (2 * c)) & 3)) + 0.5, h));
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k][c] = __dsub_rn((double)a.X[(int64_t)(3 * k + c) * a.nf + face], xc);
  }
  double a0 = lane == 0 ? 1.0 : 0.0, a1 = lane == 1 ? 1.0 : 0.0, a2 = lane == 2 ? 1.0 : 0.0;
  if (lane == 3) {
    const double u0 = __dsub_rn(p[1][0], p[0][0]), u1 = __dsub_rn(p[1][1], p[0][1]), u2 = __dsub_rn(p[1][2], p[0][2]);
    const double w0 = __dsub_rn(p[2][0], p[0][0]), w1 = __dsub_rn(p[2][1], p[0][1]), w2 = __dsub_rn(p[2][2], p[0][2]);
    a0 = __dsub_rn(__dmul_rn(u1, w2), __dmul_rn(u2, w1));
    a1 = __dsub_rn(__dmul_rn(u2, w0), __dmul_rn(u0, w2));
    a2 = __dsub_rn(__dmul_rn(u0, w1), __dmul_rn(u1, w0));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3;
    if (lane >= 4 + 3 * k && lane < 7 + 3 * k) {
      const double ex = __dsub_rn(p[k1][0], p[k][0]), ey = __dsub_rn(p[k1][1], p[k][1]),
                   ez = __dsub_rn(p[k1][2], p[k][2]);
      const int i = lane - 4 - 3 * k;
      a0 = i == 0 ? 0.0 : (i == 1 ? ez : -ey);
      a1 = i == 0 ? -ez : (i == 1 ? 0.0 : ex);
      a2 = i == 0 ? ey : (i == 1 ? -ex : 0.0);
    }
  }
  const double l2sq = __dadd_rn(__dadd_rn(__dmul_rn(a0, a0), __dmul_rn(a1, a1)), __dmul_rn(a2, a2));
  double lo = 1e300, hi = -1e300;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double s = __dadd_rn(__dadd_rn(__dmul_rn(p[k][0], a0), __dmul_rn(p[k][1], a1)), __dmul_rn(p[k][2], a2));
    lo = fmin(lo, s);
    hi = fmax(hi, s);
  }
  const double R = __dmul_rn(r, __dadd_rn(__dadd_rn(fabs(a0), fabs(a1)), fabs(a2)));
  const double g = fmax(__dsub_rn(lo, R), __dsub_rn(-R, hi));
  const bool axis = lane < 13 && l2sq != 0.0;
  const bool small = __dmul_rn(g, g) <= __dmul_rn(tol * tol, l2sq);
  const unsigned sep = __ballot_sync(0xffffffffu, axis && g > 0.0);
  const unsigned big = __ballot_sync(0xffffffffu, axis && g > 0.0 && !small);
  const unsigned near0 = __ballot_sync(0xffffffffu, axis && !(g > 0.0) && small);
  return (sep == 0u ? 1u : 0u) | ((sep ? big == 0u : near0 != 0u) ? 2u : 0u);
}

// Per-warp shared memory of the walk: survivor data, a double buffer of bin
// entries filled by TMA bulk copies with one mbarrier per buffer, and the
// block's survivor records.
template <int D>
struct WarpSmem {
  Surv<D> surv[32];
  typename EntryT<D>::type buf[2][32];
  uint64_t bar[2];
  uint64_t rm[kRecCap];  // survivor records of the block: cell-hit masks ...
  uint32_t rf[kRecCap];  // ... and face ids
};

template <int D>
__device__ __forceinline__ void warp_smem_init(WarpSmem<D>& sm, int lane) {
  if (lane == 0) {
    mbar_init(&sm.bar[0], 1);
    mbar_init(&sm.bar[1], 1);
    mbar_fence_init();
  }
  __syncwarp();
}

// The entries of the query box's x-rows (y, z fixed, x in [qlo_x, qhi_x]) are
// contiguous in the bin payload.  Lane i holds row i of the current group of
// (up to) 32 rows: its first entry `s`, its length `n` and the row's start
// `v` in the group's concatenated entry list.  Chunk c = entries [32c, 32c+32)
// of that list; every lane copies its row's part of the chunk into the buffer
// (lane 0 first announces the chunk's bytes on the buffer's mbarrier).
template <typename E>
__device__ __forceinline__ void issue_chunk(const E* payload, uint32_t s, uint32_t n, uint32_t v, uint32_t c,
                                            uint32_t T, E* buf, uint64_t* bar, int lane) {
  const uint32_t c0 = 32u * c, c1 = c0 + 32u < T ? c0 + 32u : T;
  if (lane == 0) mbar_arrive_expect_tx(bar, (c1 - c0) * (uint32_t)sizeof(E));
  __syncwarp();
  const uint32_t a0 = v > c0 ? v : c0, a1 = v + n < c1 ? v + n : c1;
  if (a0 < a1) {
    fence_proxy_async_smem();  // this warp's earlier reads of the buffer come first
    bulk_copy_g2s(buf + (a0 - c0), payload + s + (a0 - v), (a1 - a0) * (uint32_t)sizeof(E), bar);
  }
}

// Mark-only walk, point predicate: the cells of a block not yet marked (bits of um) that one of the ns faces which
// the warp gathered reaches (3D query box: their entries, listed in the entry buffer; else vertices at the front of
// the slots); returns what is left of um.  A lane per face, a row of four cells at a time: where some face's quick
// test is sure the cell is done; what the quick tests leave open is queued as (face, cell) pairs in the record stage,
// which only runs the closest-point test, 32 pairs at a time, for cells that nothing else has marked by then.
// Bound by: issue slots, at 16 warps per SM (128 registers).  3D, 112,500 faces, d = 0.05 (3 to 12 cells), the two
// walked levels: 4.92 ms one face at a time over the lanes' cells (any open cell cost the whole warp a closest-point
// test) -> 2.68 with 32 faces at a time -> 2.20 with the bins beyond d left out and the nearest rows first (90 -> 49
// million candidates) -> 1.79 in rows of four cells -> 1.57 with the cull by spheres; own-bin candidates 2.46 -> 0.87.
// Few or wide faces, and faces in many bins, are better taken one at a time (gather_pays in api.cu).
template <int D, int PRED>
__device__ __forceinline__ uint64_t mark_batch(const RefineLevel& a, uint32_t gid, const int* b, WarpSmem<D>& sm,
                                               uint32_t ns, uint64_t um, const BlockFrame<D>& F, const FastGeom& g,
                                               const float* shift, uint32_t own0, uint32_t own1, uint32_t oz0,
                                               uint32_t oz1, int lane, WarpCounters& wc) {
  constexpr bool kOwnBin = PRED == 2;
  constexpr uint32_t kQueue = (sizeof(sm.rm) + sizeof(sm.rf)) / 2;
  uint16_t* pairs = reinterpret_cast<uint16_t*>(sm.rm);
  const float R2 = g.d * g.d;
  FaceCentre C{};
  uint32_t bin = 0, binz = 0;
  const bool have = (uint32_t)lane < ns;
  if (have) {
    Surv<D>& S = sm.surv[lane];
    float V[D * D], nh[3] = {0.f, 0.f, 0.f};
    float4 v0 = S.t[0], v1{}, v2{};
    if constexpr (D == 3 && !kOwnBin) {
      const float4* E = static_cast<const float4*>(a.payload) + 4ull * reinterpret_cast<const uint32_t*>(sm.buf)[lane];
      v0 = __ldg(E), v1 = __ldg(E + 1), v2 = __ldg(E + 2);
      S.face = __float_as_uint(__ldg(E + 3).x) & kIdMask;
    } else {
      if constexpr (D == 3) v1 = S.t[1], v2 = S.t[2];
      if constexpr (kOwnBin) bin = S.pad[0];
      if constexpr (kOwnBin && D == 3) binz = S.pad[1];
    }
    V[0] = v0.x, V[1] = v0.y, V[2] = v0.z, V[3] = v0.w;
    if constexpr (D == 3) {
      V[4] = v1.x, V[5] = v1.y, V[6] = v1.z, V[7] = v1.w, V[8] = v2.x;
      nh[0] = v2.y, nh[1] = v2.z, nh[2] = v2.w;
    }
    C = face_centre<D>(V, F, g.d);
    setup_point<D>(V, nh, F, S);
  }
  __syncwarp();
  auto place = [&](int l, int c) {  // of cell l along axis c
    const float k = (float)l + 0.5f;
    return fmaf(k, g.h_hi, fmaf(k, g.h_lo, shift[c]));
  };
  float dx2[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const float dx = place(l, 0) - C.c[0];
    dx2[l] = dx * dx;
  }
  uint32_t nq = 0;
  for (uint64_t u = um; u;) {
    // a row of four cells
    const int row = (__ffsll((long long)u) - 1) >> 2;
    const uint32_t cells = (uint32_t)(u >> (4 * row)) & 15u;
    u &= ~(15ull << (4 * row));
    const float dy = place(row & 3, 1) - C.c[1];
    float yz = dy * dy;
    if constexpr (D == 3) {
      const float dz = place(row >> 2, 2) - C.c[2];
      yz = fmaf(dz, dz, yz);
    }
    uint32_t done = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      if (!((cells >> l) & 1u)) continue;
      const int cell = 4 * row + l;
      bool want = have;
      if constexpr (kOwnBin) {
        // (every lane takes part in the exchange)
        const uint32_t cb = __shfl_sync(0xffffffffu, cell < 32 ? own0 : own1, cell & 31);
        const uint32_t cz = D == 3 ? __shfl_sync(0xffffffffu, cell < 32 ? oz0 : oz1, cell & 31) : 0u;
        want = want && bin == cb && binz == cz;
      }
      const float q = yz + dx2[l];
      if (__any_sync(0xffffffffu, want && q <= C.in2)) {
        done |= 1u << l;
      } else {
        const bool open = want && !(q > C.out2);
        const unsigned ob = __ballot_sync(0xffffffffu, open);
        if (open) pairs[nq + __popc(ob & ((1u << lane) - 1u))] = (uint16_t)(lane | cell << 5);
        nq += __popc(ob);
      }
    }
    um &= ~((uint64_t)done << (4 * row));
    if (nq > kQueue - 128u || !u) {
      __syncwarp();
      for (uint32_t q0 = 0; q0 < nq; q0 += 32) {
        const uint32_t e = q0 + lane < nq ? pairs[q0 + lane] : 0u;
        const int c = (int)(e >> 5);
        int t = 0;
        if (q0 + lane < nq && ((um >> c) & 1ull)) {
          const Surv<D>& S = sm.surv[e & 31u];
          float x[3];
#pragma unroll
          for (int k = 0; k < D; ++k) x[k] = place((c >> (2 * k)) & 3, k);
          t = point_test<D>(S, x, R2);
          if (t == 2) t = resolve_fp64<D>(a, gid, S.face, b, c, &wc.fb, &wc.band) ? 1 : 0;
        }
        const uint32_t lo = __reduce_or_sync(0xffffffffu, t && c < 32 ? 1u << c : 0u);
        const uint32_t hi = D == 3 ? __reduce_or_sync(0xffffffffu, t && c >= 32 ? 1u << (c - 32) : 0u) : 0u;
        um &= ~((uint64_t)hi << 32 | lo);
      }
      nq = 0;
      u &= um;
      __syncwarp();
    }
  }
  return um;
}

// Shared walk of one block: bins of the query box, canonical-bin dedup,
// block-level cull, cell tests.  For every surviving face the whole warp calls
// `on_surv(face, r0, r1)`, r0 / r1 = whether the face meets the lane's cell
// `lane` / `lane + 32`; h0 / h1 accumulate them.  kMarkOnly: only the mask is
// wanted, so marked cells skip further tests and the walk ends as soon as every
// cell of the block is marked.
//
// The block frame is built in FP32 from the geometry row's double-float h0 and
// origin: the block corner origin + 4 b h is formed as hi + lo (hi = the frame
// origin, lo = its rounding error, carried into the cell and block centres),
// so no FP64 instruction runs per block.  The bin query range is widened by
// a margin that covers the FP32 error of the bin coordinate (a superset of
// bins only adds candidates the block test rejects).
//
// The bin ranges of all x-rows of the box are read in parallel (one lane per
// row); entries then arrive in shared memory by TMA bulk copies in chunks of
// 32, double-buffered: the next chunk is requested before the warp tests the
// current one.
constexpr uint32_t kFirstBatch = 8;  // faces of a block's first mark_batch
template <int D, int PRED, bool kMarkOnly, bool kGather, typename OnSurv>
__device__ __forceinline__ void walk_block(const RefineLevel& a, const GeomParams& P, uint32_t gid, const int* b,
                                           WarpSmem<D>& sm, uint32_t& phase, int lane, WarpCounters& wc, bool& h0,
                                           bool& h1, OnSurv on_surv) {
  using E = typename EntryT<D>::type;
  const FastGeom g = fast_geom(P, a.level);
  const float hf = g.h_hi;
  BlockFrame<D> F;
  int qlo[3] = {0, 0, 0}, qhi[3] = {0, 0, 0};
  float O = 4.0f * hf;
  float shift[3] = {0.f, 0.f, 0.f};
  const int Bn = P.B;
  const float margin = 1e-6f * (float)Bn + 1e-3f;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    float lo;
    df_position(P.org_hi[c], P.org_lo[c], (float)(4 * b[c]), g.h_hi, g.h_lo, F.Xb[c], lo);
    shift[c] = lo;
    F.cB[c] = fmaf(2.0f, g.h_hi, lo);
    O = fmaxf(O, 4.0f * hf + 2.0f * fabsf(lo));
    // bin coordinates of the inflated block's ends relative to the domain origin
    const float k0 = (float)(4 * b[c]);
    const float xlo = fmaf(k0, g.h_hi, fmaf(k0, g.h_lo, -g.d));
    const float xhi = fmaf(k0 + 4.0f, g.h_hi, fmaf(k0 + 4.0f, g.h_lo, g.d));
    const float tlo = floorf(xlo * P.scale32[c] - margin);
    const float thi = floorf(xhi * P.scale32[c] + margin);
    qlo[c] = tlo < 0.f ? 0 : (tlo > (float)(Bn - 1) ? Bn - 1 : (int)tlo);
    qhi[c] = thi < 0.f ? 0 : (thi > (float)(Bn - 1) ? Bn - 1 : (int)thi);
  }
  F.h = hf;
  F.r = fmaf(0.5f, hf, g.d);
  // block-level cull: the box around the block centre that holds every cell's
  // test region (point predicate: the cell centres' box, 1.5 h, inflated by d)
  constexpr bool kPoint = PRED >= 1;   // point predicate (Alg. 1)
  constexpr bool kOwnBin = PRED == 2;  // the paper's binned search: each cell only sees its own bin
  F.rb = kPoint ? fmaf(1.5f, hf, g.d) : fmaf(2.0f, hf, g.d);
  const float R2 = g.d * g.d;
  F.O = O;
  // the paper's binned search: the query box is the bins of the block's cell
  // centres, and each cell only takes the entries of its own bin (bins of the
  // FP64 cell centres, as the definition computes them)
  uint32_t own0 = 0, own1 = 0, oz0 = 0, oz1 = 0;
  if constexpr (kOwnBin) {
    const double hL = scalbn(P.h0, -a.level);
    auto centre_bin = [&](int c, int l) {
      const double x = __dadd_rn(P.origin[c], __dmul_rn((double)(4 * b[c] + l) + 0.5, hL));
      return bin_coord(x, P.origin[c], P.bin_scale[c], P.B);
    };
    uint32_t cb0[3] = {0, 0, 0}, cb1[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < D; ++c) {
      qlo[c] = centre_bin(c, 0);
      qhi[c] = centre_bin(c, 3);
      cb0[c] = (uint32_t)centre_bin(c, (lane >> (2 * c)) & 3);
      if (D == 3) cb1[c] = (uint32_t)centre_bin(c, ((lane + 32) >> (2 * c)) & 3);
    }
    own0 = cb0[0] | (cb0[1] << 16);
    oz0 = cb0[2];
    own1 = cb1[0] | (cb1[1] << 16);
    oz1 = cb1[2];
  }
  // cell centres of this lane in the frame: lo + (l + 1/2) h
  float o0[3] = {0, 0, 0}, o1[3] = {0, 0, 0};
  const bool lane_cell = D == 3 || lane < 16;
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const float l0 = (float)((lane >> (2 * c)) & 3) + 0.5f;
    o0[c] = fmaf(l0, g.h_hi, fmaf(l0, g.h_lo, shift[c]));
    if (D == 3) {
      const float l1 = (float)(((lane + 32) >> (2 * c)) & 3) + 0.5f;
      o1[c] = fmaf(l1, g.h_hi, fmaf(l1, g.h_lo, shift[c]));
    }
  }
  // marks of the point predicate: the unmarked cells, their centres' box, the faces gathered for mark_batch
  constexpr bool kMarkPoint = kPoint && kMarkOnly && kGather;
  uint64_t um = D == 3 ? ~0ull : 0xffffull;
  float ctr[3] = {F.cB[0], F.cB[1], D == 3 ? F.cB[D - 1] : 0.f}, half[3] = {1.5f * hf, 1.5f * hf, 1.5f * hf};
  uint32_t ns = 0, most = kFirstBatch;
  const int64_t B = Bn;
  const E* payload = static_cast<const E*>(a.payload);
  constexpr bool kSpheres = kMarkPoint && D == 3 && !kOwnBin;  // (own bin: most candidates stay, 1.38 / 1.40 ms)
  constexpr bool kTrim = kMarkPoint && !kOwnBin;  // (marks: a face may come twice)
  const int ny = qhi[1] - qlo[1] + 1;
  [[maybe_unused]] float bc[3] = {0.f, 0.f, 0.f};  // block centre relative to the domain's origin
#pragma unroll
  for (int c = 0; c < D; ++c) {
    const float k = (float)(4 * b[c] + 2);
    bc[c] = fmaf(k, g.h_hi, k * g.h_lo);
  }
  const int nrows = ny * (D == 3 ? qhi[2] - qlo[2] + 1 : 1);
  // the gathered faces against the unmarked cells; then the box of those that are left
  [[maybe_unused]] auto work_off = [&]() {
    um = mark_batch<D, PRED>(a, gid, b, sm, ns, um, F, g, shift, own0, own1, oz0, oz1, lane, wc);
    ns = 0;
    most = 32u;
    if (!um) return;
    // the box of the cells that are left
    auto span = [&](uint32_t any, int c) {  // any: 4 bits, one per cell coordinate
      const float lo = (float)(__ffs(any) - 1), hi = (float)(31 - __clz(any));
      ctr[c] = fmaf(0.5f * (lo + hi + 1.0f), g.h_hi, shift[c]);
      half[c] = 0.5f * (hi - lo) * g.h_hi;
    };
    const uint64_t pz = um | um >> 32, pl = pz | pz >> 16;      // over z
    const uint32_t xy = (uint32_t)pl & 0xffffu, x2 = xy | xy >> 8;
    span((x2 | x2 >> 4) & 15u, 0);
    uint32_t any = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) any |= ((xy >> (4 * l)) & 15u) ? 1u << l : 0u;
    span(any, 1);
    if constexpr (D == 3) {
      any = 0;
#pragma unroll
      for (int l = 0; l < 4; ++l) any |= ((um >> (16 * l)) & 0xffffull) ? 1u << l : 0u;
      span(any, 2);
    }
  };
  for (int rg = 0; rg < nrows; rg += 32) {
    // this group's rows: one lane each
    uint32_t rs = 0, rn = 0;
    const int ri = rg + lane;
    float far2 = 0.f;  // a row's distance from the block's centre, squared
    if (ri < nrows) {
      const int y = qlo[1] + ri % ny, z = D == 3 ? qlo[2] + ri / ny : 0;
      int x0 = qlo[0], x1 = qhi[0];
      if constexpr (kTrim) {
        // the bins within d of the cell centres' box: a face that reaches a centre has its nearest point in one of
        // them (bins at the domain's sides go on outside it); margins in bins as above
        float left2 = g.d * g.d * (1.0f + 1e-4f);
#pragma unroll
        for (int c = 1; c < D; ++c) {
          const int i = c == 1 ? y : z;
          const float inv = 1.0f / P.scale32[c];
          const float lo = i == 0 ? -INFINITY : ((float)i - margin) * inv;
          const float hi = i == Bn - 1 ? INFINITY : ((float)(i + 1) + margin) * inv;
          const float gap = fmaxf(0.f, fmaxf(lo - bc[c] - 1.5f * hf, bc[c] - 1.5f * hf - hi));
          left2 -= gap * gap;
          const float off = ((float)i + 0.5f) * inv - bc[c];
          far2 = fmaf(off, off, far2);
        }
        if (left2 < 0.f) {
          x1 = x0 - 1;
        } else {
          const float reach = sqrtf(left2) * (1.0f + 1e-4f) + 1.5f * hf;
          const float tl = floorf((bc[0] - reach) * P.scale32[0] - margin);
          const float th = floorf((bc[0] + reach) * P.scale32[0] + margin);
          x0 = max(x0, tl > (float)(Bn - 1) ? Bn - 1 : (int)fmaxf(tl, 0.f));
          x1 = min(x1, th < 0.f ? 0 : (int)fminf(th, (float)(Bn - 1)));
        }
      }
      if (!kTrim || x1 >= x0) {
        const int64_t b0 = P.bin_base + x0 + B * (y + B * (int64_t)z);
        rs = a.offsets[b0];
        rn = a.offsets[b0 + (x1 - x0 + 1)] - rs;
      }
    }
    if constexpr (kTrim) {
      // the nearest rows first: a face close to the block marks all of it and ends the walk
      const float key = rn ? far2 : INFINITY;
      const int n = nrows - rg < 32 ? nrows - rg : 32;
      int rank = 0, src = lane;
      for (int i = 0; i < n; ++i) {
        const float k = __shfl_sync(0xffffffffu, key, i);
        rank += k < key || (k == key && i < lane) ? 1 : 0;
      }
      for (int i = 0; i < n; ++i)
        if (__shfl_sync(0xffffffffu, rank, i) == lane) src = i;
      rs = __shfl_sync(0xffffffffu, rs, src);
      rn = __shfl_sync(0xffffffffu, rn, src);
    }
    const uint32_t incl = warp_inclusive_scan<uint32_t>(rn);
    const uint32_t T = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t rv = incl - rn;
    const uint32_t nch = (T + 31u) / 32u;
    if (nch == 0) continue;
    if constexpr (kSpheres) {
      uint32_t* list = reinterpret_cast<uint32_t*>(sm.buf);
      // the group's item k: the last row that starts at or before it, and its place there
      auto entry_of = [&](uint32_t k) {
        int l = 0;
#pragma unroll
        for (int st = 16; st > 0; st >>= 1)
          if (__shfl_sync(0xffffffffu, rv, l + st) <= k) l += st;
        return __shfl_sync(0xffffffffu, rs, l) + k - __shfl_sync(0xffffffffu, rv, l);
      };
      uint32_t e = entry_of((uint32_t)lane);
      float4 ball = (uint32_t)lane < T ? __ldg(a.spheres + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      for (uint32_t c = 0; c < nch; ++c) {
        const bool more = c + 1 < nch;
        const uint32_t e1 = entry_of(32u * (c + 1) + lane);
        const float4 ball1 = 32u * (c + 1) + lane < T ? __ldg(a.spheres + e1) : make_float4(0.f, 0.f, 0.f, 0.f);
        bool surv = false;
        if (32u * c + lane < T) {
          wc.cand++;
          FaceCentre C;
          C.c[0] = ball.x - F.Xb[0], C.c[1] = ball.y - F.Xb[1], C.c[2] = ball.z - F.Xb[2];
          const float m = fmaxf(fmaxf(fabsf(C.c[0]), fabsf(C.c[1])), fabsf(C.c[2]));
          const float out = g.d + ball.w + 16.0f * kU32 * (m + F.O) + 8.0f * kU32 * g.d;
          surv = centre_to_box2<D>(C, ctr, half) <= fmaxf(out * out * (1.0f + 8.0f * kU32), 1e-30f);
          if (surv && ball.w > 0.25f * F.rb) {
            const E& ent = payload[e];
            float V[9], nh[3];
#pragma unroll
            for (int j = 0; j < 9; ++j) V[j] = ent.v[j];
#pragma unroll
            for (int j = 0; j < 3; ++j) nh[j] = ent.n[j];
            surv = !face_beyond<D>(V, nh, F, g.d, m + 2.0f * ball.w, ctr, half);
          }
        }
        unsigned left = __ballot_sync(0xffffffffu, surv);
        wc.surv += __popc(left);
        // into the free places; a full list (a short one at first: near faces settle whole blocks) is worked off
        while (left || (!more && ns)) {
          const uint32_t at = ns + __popc(left & ((1u << lane) - 1u));
          const bool put = ((left >> lane) & 1u) && at < 32u;
          if (put) list[at] = e;
          const unsigned got = __ballot_sync(0xffffffffu, put);
          left &= ~got;
          ns += __popc(got);
          __syncwarp();
          if (ns < most && more) continue;
          work_off();
          if (!um) break;
        }
        if (!um) break;
        e = e1;
        ball = ball1;
      }
      h0 = !((um >> lane) & 1ull);
      h1 = !((um >> (lane + 32)) & 1ull);
      if (!um) return;
      continue;
    }
    int cb = 0;
    issue_chunk<E>(payload, rs, rn, rv, 0u, T, sm.buf[0], &sm.bar[0], lane);
    for (uint32_t c = 0; c < nch; ++c) {
      const int nb = cb ^ 1;
      const bool more = c + 1 < nch;
      if (more) issue_chunk<E>(payload, rs, rn, rv, c + 1, T, sm.buf[nb], &sm.bar[nb], lane);
      mbar_wait_bounded(&sm.bar[cb], (phase >> cb) & 1u, a.err);
      phase ^= 1u << cb;
      const uint32_t n = T - 32u * c < 32u ? T - 32u * c : 32u;
      bool surv = false;
      if ((uint32_t)lane < n) {
        const E& ent = sm.buf[cb][lane];
        const uint32_t id = ent.id;
        // visit a face only in the first bin of its range inside the query box
        bool canon = kOwnBin || ((id >> 29) & 1u) || (int)ent.bin[0] == qlo[0];
        canon = canon && (kOwnBin || ((id >> 30) & 1u) || (int)ent.bin[1] == qlo[1]);
        if (D == 3) canon = canon && (kOwnBin || ((id >> 31) & 1u) || (int)ent.bin[2] == qlo[2]);
        wc.cand += canon ? 1u : 0u;
        if (kTrim || canon) {
          const uint32_t f = id & kIdMask;
          float nh[3] = {0.f, 0.f, 0.f};
          if constexpr (D == 3) {
            nh[0] = ent.n[0];
            nh[1] = ent.n[1];
            nh[2] = ent.n[2];
          }
          float V[D * D];
#pragma unroll
          for (int j = 0; j < D * D; ++j) V[j] = ent.v[j];
          if constexpr (kMarkPoint) {
            const FaceCentre C = face_centre<D>(V, F, g.d);
            surv = centre_to_box2<D>(C, ctr, half) <= C.out2;
            if (surv && C.rho > 0.25f * F.rb) surv = !face_beyond<D>(V, nh, F, g.d, C.P, ctr, half);
          } else if constexpr (kPoint) {
            // the separating axes only for a face that is large against the block's reach
            float rho;
            surv = setup_centre<D>(V, F, g.d, rho, sm.surv[lane]);
            if (surv && rho > 0.25f * F.rb) {
              surv = setup_face<D>(V, nh, F, sm.surv[lane]);
              if (surv) setup_centre<D>(V, F, g.d, rho, sm.surv[lane]);
            }
            if (surv) setup_point<D>(V, nh, F, sm.surv[lane]);
          } else {
            surv = setup_face<D>(V, nh, F, sm.surv[lane]);
          }
          if constexpr (!kMarkPoint) {
            if constexpr (kOwnBin) {
              sm.surv[lane].pad[0] = ent.bin[0] | (ent.bin[1] << 16);
              if constexpr (D == 3) sm.surv[lane].pad[1] = ent.bin[2];
            }
            sm.surv[lane].face = f;
          }
        }
      }
      if constexpr (kMarkPoint && !kSpheres) {
        // survivors into the free slots; a full set (a small one at first: near faces settle whole blocks) is worked off
        unsigned left = __ballot_sync(0xffffffffu, surv);
        wc.surv += __popc(left);
        while (left || (!more && ns)) {
          const uint32_t at = ns + __popc(left & ((1u << lane) - 1u));
          const bool put = ((left >> lane) & 1u) && at < 32u;
          if (put) {
            const E& ent = sm.buf[cb][lane];
            Surv<D>& S = sm.surv[at];
            S.t[0] = make_float4(ent.v[0], ent.v[1], ent.v[2], ent.v[3]);
            if constexpr (D == 3) {
              S.t[1] = make_float4(ent.v[4], ent.v[5], ent.v[6], ent.v[7]);
              S.t[2] = make_float4(ent.v[8], ent.n[0], ent.n[1], ent.n[2]);
            }
            if constexpr (kOwnBin) {
              S.pad[0] = ent.bin[0] | (ent.bin[1] << 16);
              if constexpr (D == 3) S.pad[1] = ent.bin[2];
            }
            S.face = ent.id & kIdMask;
          }
          const unsigned got = __ballot_sync(0xffffffffu, put);
          left &= ~got;
          ns += __popc(got);
          __syncwarp();
          if (ns < most && more) continue;
          work_off();
          if (!um) break;
        }
        h0 = !((um >> lane) & 1ull) && lane_cell;
        h1 = D == 3 && !((um >> (lane + 32)) & 1ull);
      } else {
      unsigned m = __ballot_sync(0xffffffffu, surv);
      __syncwarp();
      wc.surv += __popc(m);
      while (m) {
        const int s = __ffs(m) - 1;
        m &= m - 1;
        const Surv<D>& S = sm.surv[s];
        int t0 = 0, t1 = 0;
        if constexpr (kPoint) {
          // cells that the face can count for: the lane's own, unmarked, in the entry's bin
          bool w0 = lane_cell && !(kMarkOnly && h0), w1 = D == 3 && !(kMarkOnly && h1);
          if constexpr (kOwnBin) {
            const uint32_t sz = D == 3 ? S.pad[1] : 0u;
            w0 = w0 && own0 == S.pad[0] && oz0 == sz;
            w1 = w1 && own1 == S.pad[0] && oz1 == sz;
          }
          t0 = w0 ? quick_test<D>(S, o0) : 0;
          t1 = w1 ? quick_test<D>(S, o1) : 0;
          if (__any_sync(0xffffffffu, t0 == 3 || t1 == 3)) {
            if (t0 == 3) t0 = point_test<D>(S, o0, R2);
            if (t1 == 3) t1 = point_test<D>(S, o1, R2);
          }
        } else if (!(kMarkOnly && h0 && h1)) {
          cell_test2<D>(S, o0, o1, t0, t1);
        }
        if constexpr (D == 3 && !kPoint) {
          if (__any_sync(0xffffffffu, (!(kMarkOnly && h0) && t0 == 2) || (!(kMarkOnly && h1) && t1 == 2))) {
            uint64_t u = (uint64_t)__ballot_sync(0xffffffffu, !(kMarkOnly && h0) && t0 == 2) |
                         ((uint64_t)__ballot_sync(0xffffffffu, !(kMarkOnly && h1) && t1 == 2) << 32);
            if (__popcll(u) > kFewFp64) u = 0;  // (a lane each, below)
            for (; u; u &= u - 1) {
              const int cell = __ffsll((long long)u) - 1;
              const uint32_t w = resolve_sat_warp(a, gid, S.face, b[0], b[1], b[2], cell);
              if (lane == 0) {
                ++wc.fb;
                wc.band += w >> 1;
              }
              if (cell == lane) t0 = (int)(w & 1u);
              if (cell == lane + 32) t1 = (int)(w & 1u);
            }
          }
        }
        bool r0 = false, r1 = false;
        if (lane_cell && !(kMarkOnly && h0)) {
          if (t0 == 2) t0 = resolve_fp64<D>(a, gid, S.face, b, lane, &wc.fb, &wc.band) ? 1 : 0;
          r0 = t0 != 0;
        }
        if (D == 3 && !(kMarkOnly && h1)) {
          if (t1 == 2) t1 = resolve_fp64<D>(a, gid, S.face, b, lane + 32, &wc.fb, &wc.band) ? 1 : 0;
          r1 = t1 != 0;
        }
        h0 |= r0;
        h1 |= r1;
        on_surv(S.face, r0, r1);
      }
      }
      __syncwarp();
      // marking only: once every cell of the block is marked, the rest of the walk cannot change the mask
      if (kMarkOnly && __all_sync(0xffffffffu, (h0 || !lane_cell) && (D == 2 || h1))) {
        if (more) {
          mbar_wait_bounded(&sm.bar[nb], (phase >> nb) & 1u, a.err);  // the copy already in flight
          phase ^= 1u << nb;
          __syncwarp();
        }
        return;
      }
      cb = nb;
    }
  }
}

// One survivor record past the shared-memory stage, into the warp's spill area
// (out of line: it is rare, and the walk's registers stay with the common case).
// The area of the calling warp: kSpillCap records per warp of the launch.
__device__ __forceinline__ SurvRec* warp_spill(SurvRec* spill) {
  return spill + ((uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kSpillCap;
}

__device__ __noinline__ void spill_record(SurvRec* spill, uint32_t i, uint32_t face, uint64_t cells) {
  SurvRec r;
  r.face = face;
  r.pad = 0u;
  r.cells = cells;
  warp_spill(spill)[i] = r;
}

// The block's K survivor records (staged in shared memory, past kRecCap in the
// warp's spill area) into a contiguous range of the level's record array, and
// its descriptor: offset << kInfoShift | K, 0 for none, ~0 when they are incomplete (the
// adjacency pass then walks the block again).  Whole warp.
template <int D>
__device__ __forceinline__ void store_records(const RefineLevel& a, WarpSmem<D>& sm, uint32_t K, unsigned blk,
                                              int lane);

template <int D>
__device__ __forceinline__ void store_records(const RefineLevel& a, WarpSmem<D>& sm, uint32_t K, unsigned blk,
                                              int lane) {
  __syncwarp();  // the staged and spilled records are visible to the whole warp
  const uint32_t kmax = (uint32_t)kRecCap + (a.spill ? (uint32_t)kSpillCap : 0u);
  uint64_t base = ~0ull;
  if (K > 0 && K <= kmax) {
    if (lane == 0) base = atomicAdd(reinterpret_cast<unsigned long long*>(a.rec_count), (unsigned long long)K);
    base = __shfl_sync(0xffffffffu, base, 0);
    if ((int64_t)(base + K) > a.cap_recs) base = ~0ull;
  }
  if (base != ~0ull) {
    for (uint32_t i = lane; i < K; i += 32) {
      SurvRec r;
      if (i < (uint32_t)kRecCap) {
        r.face = sm.rf[i];
        r.pad = 0u;
        r.cells = sm.rm[i];
      } else {
        r = warp_spill(a.spill)[i - kRecCap];
      }
      a.recs[base + i] = r;
    }
  }
  if (lane == 0) a.rec_desc[blk] = K == 0 ? 0ull : (base == ~0ull ? ~0ull : (base << kInfoShift) | K);
  __syncwarp();
}

// A sphere about every bin entry's face, in bin order: centroid (rounded; the radius is taken from the rounded one)
// and a radius that covers the face.  The marks of the point predicate cull by it: 16 bytes and 15 operations per
// candidate instead of the entry's 64 (read with bank conflicts) and about 90.  112,500 faces: built in
// 7.5 us, and a pass of 2.36 ms took 2.17.
__global__ void __launch_bounds__(256) k_entry_spheres(const Entry3* __restrict__ entries, const uint32_t* n_entries,
                                                       float4* __restrict__ out) {
  const uint32_t n = *n_entries;
  for (uint64_t i = blockIdx.x * 256ull + threadIdx.x; i < n; i += gridDim.x * 256ull) {
    const float4* E = reinterpret_cast<const float4*>(entries + i);
    const float4 a = __ldg(E), b = __ldg(E + 1), c = __ldg(E + 2);
    const float V[9] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x};
    float m[3], r2 = 0.f, X = 0.f;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      m[q] = (V[q] + V[3 + q] + V[6 + q]) * (1.0f / 3.0f);
      X = fmaxf(fmaxf(X, fabsf(V[q])), fmaxf(fabsf(V[3 + q]), fabsf(V[6 + q])));
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < 3; ++q) s = fmaf(V[3 * k + q] - m[q], V[3 * k + q] - m[q], s);
      r2 = fmaxf(r2, s);
    }
    out[i] = make_float4(m[0], m[1], m[2], sqrtf(r2) * (1.0f + 8.0f * kU32) + 8.0f * kU32 * X);
  }
}

// ENDS: 0 no geometry of the launch ends at this level, 1 all do, 2 some may (the point predicate's two walks share
// no code: one kernel with both held 112 registers, and the walk that keeps records took 0.386 instead of 0.341 ms).
template <int D, int PRED, int ENDS, bool GATHER>
__global__ void __launch_bounds__(256) k_refine(RefineLevel a) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  WarpSmem<D>& sm = reinterpret_cast<WarpSmem<D>*>(s_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  warp_smem_init<D>(sm, lane);
  uint32_t phase = 0;
  const int64_t n = launch_count(a.n_blocks, a.n_dev, a.err);
  constexpr int NC = D == 3 ? 64 : 16;
  WarpCounters wc;
  // work in batches of a.batch consecutive blocks: one atomic and one coalesced
  // load of the batch's coordinates and geometry ids per batch
  const int batch = a.batch > 0 ? (a.batch < kMaxBatch ? a.batch : kMaxBatch) : 1;
  for (;;) {
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(a.work, (unsigned)batch);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= n) break;
    int cv = 0;
    uint32_t gv = 0;
    if (lane < batch * D && (int64_t)base + lane / D < n) cv = a.blocks[(int64_t)base * D + lane];
    if (a.gid && lane < batch && (int64_t)base + lane < n) gv = a.gid[base + lane];
  for (int q = 0; q < batch; ++q) {
    const unsigned blk = base + (unsigned)q;
    if (blk >= n) break;
    int b[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < D; ++c) b[c] = __shfl_sync(0xffffffffu, cv, q * D + c);
    const uint32_t gid = __shfl_sync(0xffffffffu, gv, q);
    const GeomParams& P = a.table ? a.table[gid] : a.g0;
    // per-cell face counts and survivor records only where the block's geometry ends here
    const bool fin = ENDS == 2 ? a.blockcnt && a.level == P.n_levels - 1 : ENDS == 1;
    if (a.skip_mark_only && ((P.face_levels >> a.level) & 1u)) continue;  // marked face by face
    uint32_t cnt0 = 0, cnt1 = 0;
    bool h0 = false, h1 = false;
    if (ENDS == 1 || (ENDS == 2 && fin)) {
      if constexpr (ENDS != 0) {
      uint32_t K = 0;  // records of this block (warp-uniform); past kRecCap into the warp's spill area
      walk_block<D, PRED, false, false>(a, P, gid, b, sm, phase, lane, wc, h0, h1, [&](uint32_t f, bool r0, bool r1) {
        cnt0 += r0 ? 1u : 0u;
        cnt1 += r1 ? 1u : 0u;
        if (a.recs) {
          const uint64_t cm = (uint64_t)__ballot_sync(0xffffffffu, r0) |
                              ((uint64_t)__ballot_sync(0xffffffffu, r1) << 32);
          if (cm) {
            if (lane == 0) {
              if (K < (uint32_t)kRecCap) {
                sm.rf[K] = f;
                sm.rm[K] = cm;
              } else if (a.spill && K < (uint32_t)(kRecCap + kSpillCap)) {
                spill_record(a.spill, K - kRecCap, f, cm);
              }
            }
            ++K;
          }
        }
      });
      if (a.recs) {
        if (K > (uint32_t)kRecCap) wc.big += 1;
        store_records<D>(a, sm, K, blk, lane);
      }
      }
    } else if constexpr (ENDS != 1) {
      walk_block<D, PRED, true, GATHER>(a, P, gid, b, sm, phase, lane, wc, h0, h1, [](uint32_t, bool, bool) {});
      cnt0 = h0 ? 1u : 0u;
      cnt1 = h1 ? 1u : 0u;
    }
    const uint64_t mask = (uint64_t)__ballot_sync(0xffffffffu, cnt0 > 0) |
                          ((uint64_t)__ballot_sync(0xffffffffu, cnt1 > 0) << 32);
    const uint64_t m = D == 3 ? mask : (mask & 0xffffull);
    if (lane == 0) {
      a.mask[blk] = m;
      a.flag[blk] = m != 0 ? 1 : 0;
    }
    if (a.blockcnt) {
      if (fin && a.cellcnt) {
        if (cnt0 > 0xffffu || cnt1 > 0xffffu) atomicOr(a.err, ERR_OVERFLOW);
        if (lane < NC) a.cellcnt[(int64_t)blk * NC + lane] = (uint16_t)min(cnt0, 0xffffu);
        if (D == 3) a.cellcnt[(int64_t)blk * NC + 32 + lane] = (uint16_t)min(cnt1, 0xffffu);
      }
      uint32_t pairs = fin ? cnt0 + cnt1 : 0u;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
      if (lane == 0) a.blockcnt[blk] = fin ? ((uint64_t)pairs | ((uint64_t)__popcll(m) << 32)) : 0ull;
    }
  }
  }
  // flush warp counters
  unsigned long long v[5] = {wc.fb, wc.band, wc.cand, wc.surv, wc.big};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  }
  if (lane == 0) {
    if (v[0]) atomicAdd(&a.counters[CNT_FALLBACK], v[0]);
    if (v[1]) atomicAdd(&a.counters[CNT_BAND], v[1]);
    atomicAdd(&a.counters[CNT_CANDIDATES], v[2]);       // per-lane counts
    atomicAdd(&a.counters[CNT_SURVIVORS], v[3] / 32);   // every lane counted the same survivors
    if (v[4]) atomicAdd(&a.counters[CNT_BIG_BLOCKS], v[4] / 32);
  }
}

// ---------------------------------------------------------------------------
// Refinement by parent groups (3D box predicate, levels below the roots).
//
// Every block of such a level is one of the 8 children of a marked parent,
// and the children of a parent are consecutive (slot order).  One warp takes a
// parent's 8 children together: it walks the bins of the parent box inflated
// by d_L once (the union of the children's query boxes), deduplicates, and
// culls each candidate against the whole inflated parent box; every survivor
// is then culled against each child's box (lane-parallel, certified, all 13
// axes), and only the remaining (face, child) pairs run the cell tests.  The
// bins are walked once per 8 children instead of once per child.
//
// The frame is the parent's corner (= child 0's corner); the cell thresholds
// of a survivor hold for all 512 cells of the group (its error bound takes
// the group's extent, 8 cells, as the bound on the cell-centre offsets).  The
// decisions are the per-block walk's (certified FP32 or the same FP64
// resolution), so the masks, counts and records are identical.
// ---------------------------------------------------------------------------
constexpr int kGroupPool = 24;  // survivor records of a group staged in shared memory (more: spill area)

struct GroupSmem {
  Surv<3> surv[32];
  Entry3 buf[2][32];
  uint64_t bar[2];
  SurvRec pool[kGroupPool];  // face, child (pad), cell mask
  uint16_t cnt[8][64];       // per child and cell: faces that meet the cell (finest level)
  uint8_t sidx[32];          // lanes of the chunk's survivors, in lane order
};

// Child j of the group may meet the face: no axis certifiably separates the
// projections of its cell centres (a box of half-width 1.5 h around the child
// centre cj) from the face's cell-level interval.  The widening by
// (t.z - t.x) = 2 eps absorbs the rounding of the child-centre projection and
// of the additions, so a culled child has no cell that meets the face.
__device__ __forceinline__ bool child_may_meet(const Surv<3>& S, const float* cj, float h15) {
  const float4 q0 = S.en[0], q1 = S.en[1], q2 = S.en[2];
  auto sep = [&](float x, float A1, const float4& t) {
    const float w = fmaf(h15, A1, t.z - t.x);
    return (x + w < t.x) | (x - w > t.y);
  };
  bool out = sep(cj[0], 1.f, S.t[0]) | sep(cj[1], 1.f, S.t[1]) | sep(cj[2], 1.f, S.t[2]);
  out |= sep(fmaf(cj[2], q2.w, fmaf(cj[1], q2.z, cj[0] * q2.y)), fabsf(q2.y) + fabsf(q2.z) + fabsf(q2.w), S.t[3]);
  const float e[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
    out |= sep(fmaf(cj[2], ey, -cj[1] * ez), fabsf(ey) + fabsf(ez), S.t[4 + 3 * k]);
    out |= sep(fmaf(cj[0], ez, -cj[2] * ex), fabsf(ex) + fabsf(ez), S.t[5 + 3 * k]);
    out |= sep(fmaf(cj[1], ex, -cj[0] * ey), fabsf(ex) + fabsf(ey), S.t[6 + 3 * k]);
  }
  return !out;
}

// Per-warp counters of the group kernel (32-bit: a warp's counts stay far below 2^32).
struct GroupCounters {
  uint32_t fb = 0, band = 0, cand = 0, surv = 0, big = 0;
};

// FP64 decision of one (cell, face) pair of a group (the per-block walk's resolution).
__device__ __noinline__ bool resolve_group(const RefineLevel& a, uint32_t gid, uint32_t face, const int* b,
                                           int cell_local, GroupCounters& wc) {
  unsigned long long fb = 0, band = 0;
  const bool r = resolve_fp64<3>(a, gid, face, b, cell_local, &fb, &band);
  wc.fb += (uint32_t)fb;
  wc.band += (uint32_t)band;
  return r;
}

// One parent group: walk, culls and cell tests.  kMark: only the masks are
// wanted (the walk ends once every cell of the 8 children is marked); else the
// per-cell counts and the survivor records of the finest level are kept.
// hb0 / hb1: bit j = the lane's cell `lane` / `lane + 32` of child j is adjacent.
template <bool kMark>
__device__ __forceinline__ void walk_group(const RefineLevel& a, const GeomParams& P, uint32_t gid, const int* c0,
                                           GroupSmem& sm, uint32_t& phase, int lane, GroupCounters& wc,
                                           uint32_t& hb0, uint32_t& hb1, uint32_t& K, SurvRec* spill) {
  const FastGeom g = fast_geom(P, a.level);
  const float hf = g.h_hi;
  BlockFrame<3> F;
  int qlo[3], qhi[3];
  float O = 8.0f * hf;
  float shift[3];
  const int Bn = P.B;
  const float margin = 1e-6f * (float)Bn + 1e-3f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float lo;
    df_position(P.org_hi[c], P.org_lo[c], (float)(4 * c0[c]), g.h_hi, g.h_lo, F.Xb[c], lo);
    shift[c] = lo;
    F.cB[c] = fmaf(4.0f, g.h_hi, lo);
    O = fmaxf(O, 8.0f * hf + 2.0f * fabsf(lo));
    const float k0 = (float)(4 * c0[c]);
    const float xlo = fmaf(k0, g.h_hi, fmaf(k0, g.h_lo, -g.d));
    const float xhi = fmaf(k0 + 8.0f, g.h_hi, fmaf(k0 + 8.0f, g.h_lo, g.d));
    const float tlo = floorf(xlo * P.scale32[c] - margin);
    const float thi = floorf(xhi * P.scale32[c] + margin);
    qlo[c] = tlo < 0.f ? 0 : (tlo > (float)(Bn - 1) ? Bn - 1 : (int)tlo);
    qhi[c] = thi < 0.f ? 0 : (thi > (float)(Bn - 1) ? Bn - 1 : (int)thi);
  }
  F.h = hf;
  F.r = fmaf(0.5f, hf, g.d);
  F.rb = fmaf(4.0f, hf, g.d);  // the union of the 512 inflated cells: the parent box inflated by d
  F.O = O;
  const float h15 = 1.5f * hf;
  uint32_t full = 0;  // children whose 64 cells are all marked (kMark)
  const int64_t B = Bn;
  const Entry3* payload = static_cast<const Entry3*>(a.payload);
  const int nx = qhi[0] - qlo[0] + 1, ny = qhi[1] - qlo[1] + 1;
  const int nrows = ny * (qhi[2] - qlo[2] + 1);
  for (int rg = 0; rg < nrows; rg += 32) {
    uint32_t rs = 0, rn = 0;
    const int ri = rg + lane;
    if (ri < nrows) {
      const int y = qlo[1] + ri % ny, z = qlo[2] + ri / ny;
      const int64_t b0 = P.bin_base + qlo[0] + B * (y + B * (int64_t)z);
      rs = a.offsets[b0];
      rn = a.offsets[b0 + nx] - rs;
    }
    const uint32_t incl = warp_inclusive_scan<uint32_t>(rn);
    const uint32_t T = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t rv = incl - rn;
    const uint32_t nch = (T + 31u) / 32u;
    if (nch == 0) continue;
    int cb = 0;
    issue_chunk<Entry3>(payload, rs, rn, rv, 0u, T, sm.buf[0], &sm.bar[0], lane);
    for (uint32_t c = 0; c < nch; ++c) {
      const int nb = cb ^ 1;
      const bool more = c + 1 < nch;
      if (more) issue_chunk<Entry3>(payload, rs, rn, rv, c + 1, T, sm.buf[nb], &sm.bar[nb], lane);
      mbar_wait_bounded(&sm.bar[cb], (phase >> cb) & 1u, a.err);
      phase ^= 1u << cb;
      const uint32_t n = T - 32u * c < 32u ? T - 32u * c : 32u;
      bool surv = false;
      if ((uint32_t)lane < n) {
        const Entry3& ent = sm.buf[cb][lane];
        const uint32_t id = ent.id;
        // visit a face only in the first bin of its range inside the query box
        const bool canon = (((id >> 29) & 1u) || (int)ent.bin[0] == qlo[0]) &&
                           (((id >> 30) & 1u) || (int)ent.bin[1] == qlo[1]) &&
                           (((id >> 31) & 1u) || (int)ent.bin[2] == qlo[2]);
        if (canon) {
          wc.cand++;
          const float nh[3] = {ent.n[0], ent.n[1], ent.n[2]};
          float V[9];
#pragma unroll
          for (int j = 0; j < 9; ++j) V[j] = ent.v[j];
          surv = setup_face<3>(V, nh, F, sm.surv[lane]);
          sm.surv[lane].face = id & kIdMask;
        }
      }
      unsigned m = __ballot_sync(0xffffffffu, surv);
      if (surv) sm.sidx[__popc(m & ((1u << lane) - 1u))] = (uint8_t)lane;
      __syncwarp();
      // child culls: lane = (survivor, child) pair
      const int ns = __popc(m);
      for (int base = 0; base < 8 * ns; base += 32) {
        const int p = base + lane;
        bool keep = false;
        int s = 0;
        if (p < 8 * ns) {
          s = sm.sidx[p >> 3];
          const int j = p & 7;
          float cj[3];
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float l = (float)(4 * ((j >> q) & 1) + 2);
            cj[q] = fmaf(l, g.h_hi, fmaf(l, g.h_lo, shift[q]));
          }
          keep = child_may_meet(sm.surv[s], cj, h15);
        }
        const unsigned kb = __ballot_sync(0xffffffffu, keep);
        if ((lane & 7) == 0 && p < 8 * ns) sm.surv[s].pad[0] = (kb >> (lane & 24)) & 0xffu;
      }
      __syncwarp();
      while (m) {
        const int s = __ffs(m) - 1;
        m &= m - 1;
        const Surv<3>& S = sm.surv[s];
        uint32_t cm = S.pad[0];
        if (kMark) cm &= ~full;
        wc.surv += __popc(cm);
        while (cm) {
          const int j = __ffs(cm) - 1;
          cm &= cm - 1;
          // read the survivor's thresholds from shared memory per child (not held in registers
          // across the children, which spills)
          asm volatile("" ::: "memory");
          const int cx = j & 1, cy = (j >> 1) & 1, cz = (j >> 2) & 1;
          // the lane's cells `lane` and `lane + 32` of child j, centres in the frame
          float o0[3], o1[3];
          {
            const int d0[3] = {4 * cx, 4 * cy, 4 * cz};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const float a0 = (float)(d0[q] + ((lane >> (2 * q)) & 3)) + 0.5f;
              const float a1 = (float)(d0[q] + (((lane + 32) >> (2 * q)) & 3)) + 0.5f;
              o0[q] = fmaf(a0, g.h_hi, fmaf(a0, g.h_lo, shift[q]));
              o1[q] = fmaf(a1, g.h_hi, fmaf(a1, g.h_lo, shift[q]));
            }
          }
          const bool m0 = kMark && ((hb0 >> j) & 1u), m1 = kMark && ((hb1 >> j) & 1u);
          int t0 = 0, t1 = 0;
          cell_test2<3>(S, o0, o1, t0, t1);
          const int bj[3] = {c0[0] + cx, c0[1] + cy, c0[2] + cz};  // child j's block coordinates
          // pairs not certified in FP32: many a lane each, a few one after another by the whole warp (one vote first,
          // for few faces have any; by value, for the walk's registers are full)
          if (__any_sync(0xffffffffu, (!m0 && t0 == 2) || (!m1 && t1 == 2))) {
            uint32_t u0 = __ballot_sync(0xffffffffu, !m0 && t0 == 2), u1 = __ballot_sync(0xffffffffu, !m1 && t1 == 2);
            if (__popc(u0) + __popc(u1) > kFewFp64) {
              if (!m0 && t0 == 2) t0 = resolve_group(a, gid, S.face, bj, lane, wc) ? 1 : 0;
              if (!m1 && t1 == 2) t1 = resolve_group(a, gid, S.face, bj, lane + 32, wc) ? 1 : 0;
            } else {
              while (u0 | u1) {
                const int cell = u0 ? __ffs(u0) - 1 : 31 + __ffs(u1);
                if (u0) u0 &= u0 - 1; else u1 &= u1 - 1;
                const uint32_t w = resolve_sat_warp(a, gid, S.face, bj[0], bj[1], bj[2], cell);
                if (lane == 0) {
                  ++wc.fb;
                  wc.band += w >> 1;
                }
                if (cell == lane) t0 = (int)(w & 1u);
                if (cell == lane + 32) t1 = (int)(w & 1u);
              }
            }
          }
          const bool r0 = !m0 && t0 != 0, r1 = !m1 && t1 != 0;
          hb0 |= (uint32_t)r0 << j;
          hb1 |= (uint32_t)r1 << j;
          if constexpr (kMark) {
            if (__all_sync(0xffffffffu, ((hb0 & hb1) >> j) & 1u)) full |= 1u << j;
          } else {
            const uint32_t n0 = sm.cnt[j][lane], n1 = sm.cnt[j][lane + 32];
            if ((r0 && n0 == 0xffffu) || (r1 && n1 == 0xffffu)) atomicOr(a.err, ERR_OVERFLOW);
            sm.cnt[j][lane] = (uint16_t)min(n0 + (uint32_t)r0, 0xffffu);
            sm.cnt[j][lane + 32] = (uint16_t)min(n1 + (uint32_t)r1, 0xffffu);
            if (a.recs) {
              const uint64_t cells = (uint64_t)__ballot_sync(0xffffffffu, r0) |
                                     ((uint64_t)__ballot_sync(0xffffffffu, r1) << 32);
              if (cells) {
                if (lane == 0) {
                  SurvRec r;
                  r.face = S.face;
                  r.pad = (uint32_t)j;
                  r.cells = cells;
                  if (K < (uint32_t)kGroupPool)
                    sm.pool[K] = r;
                  else if (spill && K < (uint32_t)(kGroupPool + kSpillCap))
                    spill[K - kGroupPool] = r;
                }
                ++K;
              }
            }
          }
        }
      }
      __syncwarp();
      if (kMark && full == 0xffu) {
        if (more) {
          mbar_wait_bounded(&sm.bar[nb], (phase >> nb) & 1u, a.err);  // the copy already in flight
          phase ^= 1u << nb;
          __syncwarp();
        }
        return;
      }
      cb = nb;
    }
  }
}

// The group's K records into a contiguous range of the level's record array,
// grouped by child (each child's records in the order they were found), and
// every child's descriptor: offset << kInfoShift | count, 0 for none, ~0 when the
// records are incomplete (the adjacency pass then walks the block again).
__device__ __noinline__ void store_group_records(const RefineLevel& a, GroupSmem& sm, const SurvRec* spill,
                                                  uint32_t K, unsigned blk0, int lane) {
  __syncwarp();  // the staged and spilled records are visible to the whole warp
  const uint32_t kmax = (uint32_t)kGroupPool + (spill ? (uint32_t)kSpillCap : 0u);
  uint64_t base = ~0ull;
  if (K > 0 && K <= kmax) {
    if (lane == 0) base = atomicAdd(reinterpret_cast<unsigned long long*>(a.rec_count), (unsigned long long)K);
    base = __shfl_sync(0xffffffffu, base, 0);
    if ((int64_t)(base + K) > a.cap_recs) base = ~0ull;
  }
  if (K == 0 || base == ~0ull) {
    if (lane < 8) a.rec_desc[blk0 + lane] = K == 0 ? 0ull : ~0ull;
    __syncwarp();
    return;
  }
  auto rec = [&](uint32_t i) { return i < (uint32_t)kGroupPool ? sm.pool[i] : spill[i - kGroupPool]; };
  // records per child, then the child's first position
  uint32_t cntj = 0;  // lane j < 8: records of child j
  for (uint32_t i0 = 0; i0 < K; i0 += 32) {
    const uint32_t i = i0 + (uint32_t)lane;
    const uint32_t j = i < K ? rec(i).pad : 8u;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint32_t n = __popc(__ballot_sync(0xffffffffu, j == (uint32_t)q));
      if (lane == q) cntj += n;
    }
  }
  const uint32_t incl = warp_inclusive_scan<uint32_t>(lane < 8 ? cntj : 0u);
  const uint32_t first = incl - (lane < 8 ? cntj : 0u);
  if (lane < 8) a.rec_desc[blk0 + lane] = cntj == 0 ? 0ull : ((base + first) << kInfoShift) | cntj;
  uint32_t run = first;  // lane j < 8: next position of child j
  for (uint32_t i0 = 0; i0 < K; i0 += 32) {
    const uint32_t i = i0 + (uint32_t)lane;
    SurvRec r;
    r.pad = 8u;
    if (i < K) r = rec(i);
    uint32_t pos = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const unsigned bq = __ballot_sync(0xffffffffu, r.pad == (uint32_t)q);
      const uint32_t rq = __shfl_sync(0xffffffffu, run, q);
      if (r.pad == (uint32_t)q) pos = rq + __popc(bq & ((1u << lane) - 1u));
      if (lane == q) run += __popc(bq);
    }
    if (i < K) {
      SurvRec o;
      o.face = r.face;
      o.pad = 0u;
      o.cells = r.cells;
      a.recs[base + pos] = o;
    }
  }
  __syncwarp();
}

constexpr int kGroupWarps = 4;  // warps per CTA of k_refine_groups (4 CTAs per SM by registers and shared memory)

__global__ void __launch_bounds__(kGroupWarps * 32, 4) k_refine_groups(RefineLevel a) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  GroupSmem& sm = reinterpret_cast<GroupSmem*>(s_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    mbar_init(&sm.bar[0], 1);
    mbar_init(&sm.bar[1], 1);
    mbar_fence_init();
  }
  __syncwarp();
  uint32_t phase = 0;
  const int64_t n = launch_count(a.n_blocks, a.n_dev, a.err);
  if ((n & 7) != 0 && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, ERR_BADINDEX);  // children in eights
  const int64_t ng = n >> 3;
  SurvRec* spill = a.spill ? warp_spill(a.spill) : nullptr;
  GroupCounters wc;
  for (;;) {
    unsigned gi = 0;
    if (lane == 0) gi = atomicAdd(a.work, 1u);
    gi = __shfl_sync(0xffffffffu, gi, 0);
    if ((int64_t)gi >= ng) break;
    const unsigned blk0 = gi * 8u;
    int cv = lane < 3 ? a.blocks[(int64_t)blk0 * 3 + lane] : 0;
    int c0[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) c0[c] = __shfl_sync(0xffffffffu, cv, c);
    const uint32_t gid = a.gid ? a.gid[blk0] : 0u;
    const GeomParams& P = a.table ? a.table[gid] : a.g0;
    if (a.skip_mark_only && ((P.face_levels >> a.level) & 1u)) continue;  // marked face by face
    const bool fin = a.blockcnt && a.level == P.n_levels - 1;
    uint32_t hb0 = 0, hb1 = 0, K = 0;
    if (fin) {
      reinterpret_cast<uint4*>(sm.cnt)[lane] = make_uint4(0u, 0u, 0u, 0u);
      reinterpret_cast<uint4*>(sm.cnt)[lane + 32] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
      walk_group<false>(a, P, gid, c0, sm, phase, lane, wc, hb0, hb1, K, spill);
      if (a.recs) {
        if (K > (uint32_t)kGroupPool) wc.big += 1;
        store_group_records(a, sm, spill, K, blk0, lane);
      }
    } else {
      walk_group<true>(a, P, gid, c0, sm, phase, lane, wc, hb0, hb1, K, spill);
    }
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      const unsigned blk = blk0 + (unsigned)j;
      const uint64_t m = (uint64_t)__ballot_sync(0xffffffffu, (hb0 >> j) & 1u) |
                         ((uint64_t)__ballot_sync(0xffffffffu, (hb1 >> j) & 1u) << 32);
      if (lane == 0) {
        a.mask[blk] = m;
        a.flag[blk] = m != 0 ? 1 : 0;
      }
      if (a.blockcnt) {
        uint32_t pairs = 0;
        if (fin) {
          const uint32_t n0 = sm.cnt[j][lane], n1 = sm.cnt[j][lane + 32];
          if (a.cellcnt) {
            a.cellcnt[(int64_t)blk * 64 + lane] = (uint16_t)n0;
            a.cellcnt[(int64_t)blk * 64 + 32 + lane] = (uint16_t)n1;
          }
          pairs = n0 + n1;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        }
        if (lane == 0) a.blockcnt[blk] = fin ? ((uint64_t)pairs | ((uint64_t)__popcll(m) << 32)) : 0ull;
      }
    }
  }
  // fb, band and cand are per-lane counts; surv and big, warp-uniform ones
  unsigned long long v[5] = {wc.fb, wc.band, wc.cand, wc.surv, wc.big};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  }
  if (lane == 0) {
    if (v[0]) atomicAdd(&a.counters[CNT_FALLBACK], v[0]);
    if (v[1]) atomicAdd(&a.counters[CNT_BAND], v[1]);
    atomicAdd(&a.counters[CNT_CANDIDATES], v[2]);
    atomicAdd(&a.counters[CNT_SURVIVORS], v[3]);  // (face, child) pairs that ran the cell tests
    if (v[4]) atomicAdd(&a.counters[CNT_BIG_BLOCKS], v[4]);
  }
}

// Ascending sort of P keys in shared memory (P a power of two from 64 up; pad the
// tail with ~0) by the whole warp: the bitonic network, each lane taking every
// 32nd compare-exchange of a stage, four of them in flight.
template <typename T>
__device__ __noinline__ void warp_bitonic(T* k, uint32_t P, int lane) {
  for (uint32_t s = 2; s <= P; s <<= 1)
    for (uint32_t j = s >> 1; j > 0; j >>= 1) {
#pragma unroll 4
      for (uint32_t t = (uint32_t)lane; t < P / 2; t += 32) {
        const uint32_t low = t & (j - 1), i = ((t - low) << 1) | low;
        const T x = k[i], y = k[i + j];
        const bool swap = ((i & s) == 0) == (x > y);
        k[i] = swap ? y : x;
        k[i + j] = swap ? x : y;
      }
      __syncwarp();
    }
}

// Ascending face ids in each of a block's cell lists (cell c's count and offset
// held by lane c, or lane c - 32 in n1 / off1): the warp sorts one list at a time
// in the shared memory at sf (room for cap keys); a longer list is sorted in
// place by one lane.  Out of line: only blocks walked again need it.
__device__ __noinline__ void sort_cell_lists(uint32_t* adj_ids, int NC, uint32_t n0, uint32_t n1, uint64_t off0,
                                             uint64_t off1, uint32_t* sf, uint32_t cap, int lane) {
  for (int c = 0; c < NC; ++c) {
    const uint32_t cnt = c < 32 ? __shfl_sync(0xffffffffu, n0, c) : __shfl_sync(0xffffffffu, n1, c - 32);
    const uint64_t off = c < 32 ? __shfl_sync(0xffffffffu, off0, c) : __shfl_sync(0xffffffffu, off1, c - 32);
    if (cnt <= 1) continue;
    uint32_t* L = adj_ids + off;
    if (cnt <= cap) {
      uint32_t P = 64;
      while (P < cnt) P <<= 1;
      for (uint32_t i = lane; i < P; i += 32) sf[i] = i < cnt ? L[i] : 0xffffffffu;
      __syncwarp();
      warp_bitonic(sf, P, lane);
      for (uint32_t i = lane; i < cnt; i += 32) L[i] = sf[i];
      __syncwarp();
    } else if (lane == 0) {
      for (uint32_t i = 1; i < cnt; ++i) {
        const uint32_t v = L[i];
        uint32_t k = i;
        while (k > 0 && L[k - 1] > v) {
          L[k] = L[k - 1];
          --k;
        }
        L[k] = v;
      }
    }
    __syncwarp();
  }
}

// A block's K survivor records in ascending order of face id, by the whole warp: face id and place of each in sk.
__device__ __noinline__ void sort_records(const SurvRec* recs, uint32_t K, uint64_t* sk, int lane) {
  uint32_t P = 64;
  while (P < K) P <<= 1;
  for (uint32_t i = lane; i < P; i += 32) sk[i] = i < K ? (uint64_t)recs[i].face << 32 | i : ~0ull;
  __syncwarp();
  warp_bitonic(sk, P, lane);
}

// Shared memory of a warp of the adjacency's second pass: room to sort kSortRecs records (8 bytes each), over
// which the walk's memory is laid so that only the part before its mbarriers is shared.  Bound by: the sort's chain
// of shared memory exchanges.  2D, 4,832 blocks of about 260 records, 16.9 million pairs: 2.35 ms with room for 256
// records (the walk's memory; blocks with more were walked again and their lists sorted one by one) -> 0.28 with
// room for all and whole cells written side by side -> 0.14 with four exchanges in flight, the masks left in place
// and blocks handed out singly.
constexpr uint32_t kSortRecs = 1024;  // what the refine pass keeps of a block at most
static_assert(kRecCap + kSpillCap <= (int)kSortRecs, "every block that kept its records is sorted");
constexpr uint32_t kSortRegion = 8 * kSortRecs;
template <int D>
__host__ __device__ constexpr uint32_t walk_offset() {
  constexpr uint32_t walk = (uint32_t)(sizeof(Surv<D>) * 32 + sizeof(typename EntryT<D>::type) * 64);
  return walk < kSortRegion ? kSortRegion - walk : 0u;
}
template <int D>
__host__ __device__ constexpr uint32_t second_pass_bytes() {  // (a multiple of 16 for each warp's copies)
  static_assert(walk_offset<D>() % 16 == 0 && sizeof(WarpSmem<D>) % 16 == 0, "16-byte aligned walk memory");
  return walk_offset<D>() + (uint32_t)sizeof(WarpSmem<D>);
}
template <int D>
__device__ __forceinline__ uint32_t* sort_area(WarpSmem<D>& sm) {
  return reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(&sm) - walk_offset<D>());
}
// Largest power of two P with P keys (and P payloads of 8 bytes) in the region.
__host__ __device__ constexpr uint32_t pow2_floor(uint32_t x) {
  uint32_t p = 1;
  while (p * 2 <= x) p *= 2;
  return p;
}

// Emit the adjacent-face lists of the blocks whose geometry ends at this
// level, in two passes.  MODE 0 takes every block: it writes the block's rows
// (adjacent cells and their list offsets, from the block-level scan and the
// per-cell counts) and, when the refine pass kept at most kRecCap survivor
// records, ranks them by face id and lists each cell's faces in that order; it
// needs only a little shared memory, so many warps stay resident.  Other blocks
// go to a list that MODE 1 takes, with the walk's shared memory: more records
// are sorted there, and blocks without records are walked again (the same
// decisions as k_refine) and their lists sorted.  Rows and pairs continue after
// the running totals of earlier levels.
template <int D, int PRED, int MODE>
__device__ __forceinline__ void emit_block(const EmitArgs& a, unsigned blk, uint32_t gid, WarpSmem<D>& sm,
                                           uint32_t& phase, WarpCounters& wc, uint64_t* rm, uint32_t* rf,
                                           int lane, uint64_t run_cells, uint64_t run_pairs,
                                           const uint64_t* pre = nullptr) {
  // pre (MODE 0): the block's base and record descriptor, loaded with its batch
  constexpr int NC = D == 3 ? 64 : 16;
    const GeomParams& P = a.lv.table ? a.lv.table[gid] : a.lv.g0;
    if (a.lv.level != P.n_levels - 1) return;
    int b[3] = {0, 0, 0};
#pragma unroll
    for (int c = 0; c < D; ++c) b[c] = a.lv.blocks[(int64_t)blk * D + c];
    const uint64_t base = pre ? pre[0] : a.block_base[blk];
    const uint64_t pair_base = run_pairs + (base & 0xffffffffull);
    const uint64_t cell_base = run_cells + (base >> 32);
    const uint64_t desc = pre ? pre[1] : (a.lv.recs ? a.lv.rec_desc[blk] : ~0ull);
    const uint32_t K = (uint32_t)(desc & kInfoMask);  // (desc != ~0: the block's records)
    const uint64_t rec0 = desc >> kInfoShift;
    // MODE 0: its records, two per lane
    uint32_t f[2] = {0xffffffffu, 0xffffffffu};
    uint64_t cm[2] = {0ull, 0ull};
    const bool held = MODE == 0 && desc != ~0ull && K <= (uint32_t)kRecCap;
    if (held) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t i = (uint32_t)lane + 32u * h;
        if (i < K) {
          const SurvRec r = a.lv.recs[rec0 + i];
          f[h] = r.face;
          cm[h] = r.cells;
        }
      }
    }
    // faces per cell: as the walk counted them, or (a level marked from the faces) from the records
    uint32_t n0 = 0, n1 = 0;
    auto count = [&](uint64_t m) {
      n0 += (uint32_t)(m >> lane) & 1u;
      n1 += D == 3 ? (uint32_t)(m >> (lane + 32)) & 1u : 0u;
    };
    if (a.lv.cellcnt) {
      n0 = lane < NC ? a.lv.cellcnt[(int64_t)blk * NC + lane] : 0u;
      n1 = D == 3 ? (uint32_t)a.lv.cellcnt[(int64_t)blk * NC + 32 + lane] : 0u;
    } else if (held) {
      for (uint32_t j = 0; j < K; ++j) count(__shfl_sync(0xffffffffu, j < 32 ? cm[0] : cm[1], (int)(j & 31u)));
    } else {
      for (uint32_t j = 0; j < K; ++j) count(a.lv.recs[rec0 + j].cells);
    }
    // exclusive prefixes over cells in bit order (cells 0..31 then 32..63)
    const uint32_t i0 = warp_inclusive_scan<uint32_t>(n0);
    const uint32_t tot0 = __shfl_sync(0xffffffffu, i0, 31);
    const uint32_t i1 = warp_inclusive_scan<uint32_t>(n1);
    const uint64_t off0 = pair_base + i0 - n0;
    const uint64_t off1 = pair_base + tot0 + i1 - n1;
    const uint32_t a0 = n0 > 0, a1 = n1 > 0;
    const uint32_t j0 = warp_inclusive_scan<uint32_t>(a0);
    const uint32_t atot0 = __shfl_sync(0xffffffffu, j0, 31);
    const uint32_t j1 = warp_inclusive_scan<uint32_t>(a1);
    bool bad = (int64_t)(off1 + n1) > a.cap_pairs || (int64_t)(off0 + n0) > a.cap_pairs;
    if (MODE == 0 && a0) {
      const uint64_t row = cell_base + j0 - 1;
      if ((int64_t)row < a.cap_cells) {
        a.adj_cell[row] = blk * (uint32_t)NC + lane;
        a.adj_off[row] = (uint32_t)off0;
      } else {
        bad = true;
      }
    }
    if (MODE == 0 && a1) {
      const uint64_t row = cell_base + atot0 + j1 - 1;
      if ((int64_t)row < a.cap_cells) {
        a.adj_cell[row] = blk * (uint32_t)NC + 32 + lane;
        a.adj_off[row] = (uint32_t)off1;
      } else {
        bad = true;
      }
    }
    uint32_t c0 = 0, c1 = 0;
    const bool can0 = (int64_t)(off0 + n0) <= a.cap_pairs, can1 = (int64_t)(off1 + n1) <= a.cap_pairs;
    auto put = [&](bool r0, bool r1, uint32_t f) {
      if (r0) {
        if (c0 < n0 && can0)
          a.adj_ids[off0 + c0] = f;
        else
          bad = true;
        ++c0;
      }
      if constexpr (D == 3) {
        if (r1) {
          if (c1 < n1 && can1)
            a.adj_ids[off1 + c1] = f;
          else
            bad = true;
          ++c1;
        }
      }
    };
    constexpr uint32_t kSortKeys = pow2_floor(kSortRegion / 4);
    if constexpr (MODE == 0) {
    if (held) {
      // the refine pass left this block's surviving faces with their cell masks:
      // rank them by face id, then every lane lists its cells' faces in that order
      uint32_t rank[2] = {0u, 0u};
      for (uint32_t j = 0; j < K; ++j) {
        const uint32_t fj = __shfl_sync(0xffffffffu, j < 32 ? f[0] : f[1], (int)(j & 31u));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t i = (uint32_t)lane + 32u * h;
          rank[h] += (fj < f[h] || (fj == f[h] && j < i)) ? 1u : 0u;
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t i = (uint32_t)lane + 32u * h;
        if (i < K) {
          rf[rank[h]] = f[h];
          rm[rank[h]] = cm[h];
        }
      }
      __syncwarp();
      for (uint32_t j = 0; j < K; ++j) {
        const uint64_t mj = rm[j];
        put(lane < NC && ((mj >> lane) & 1ull), D == 3 && ((mj >> (lane + 32)) & 1ull), rf[j]);
      }
      __syncwarp();
      if (bad || c0 != n0 || c1 != n1) atomicOr(a.lv.err, ERR_OVERFLOW);
      return;
    }
      // more records than staged in shared memory, or none kept: the second pass takes the block
      if (lane == 0) {
        const unsigned pos = atomicAdd(a.defer_n, 1u);
        if ((int64_t)pos < a.defer_cap)
          a.defer[pos] = blk;
        else
          atomicOr(a.lv.err, ERR_OVERFLOW);
      }
      return;
    } else {
    if (desc != ~0ull && K > (uint32_t)kRecCap && K <= kSortRecs) {
      // many records: sort them by face id in shared memory, then list the cells' faces in that order
      uint64_t* sk = reinterpret_cast<uint64_t*>(sort_area<D>(sm));
      const SurvRec* recs = a.lv.recs + rec0;
      sort_records(recs, K, sk, lane);
      if constexpr (D == 3) {
        for (uint32_t j0 = 0; j0 < K; j0 += 32) {
          const uint64_t key = j0 + lane < K ? sk[j0 + lane] : 0ull;
          const uint64_t my = j0 + lane < K ? recs[(uint32_t)key].cells : 0ull;
          const uint32_t n = K - j0 < 32u ? K - j0 : 32u;
          for (uint32_t j = 0; j < n; ++j) {
            const uint64_t mj = __shfl_sync(0xffffffffu, my, (int)j);
            put((mj >> lane) & 1ull, (mj >> (lane + 32)) & 1ull,
                __shfl_sync(0xffffffffu, (uint32_t)(key >> 32), (int)j));
          }
        }
      } else if (__all_sync(0xffffffffu, can0)) {
        // 32 records and one cell at a time: the cell's faces leave side by side
        uint32_t at = (uint32_t)off0;  // (offsets are 32 bits, as adj_off holds them)
        for (uint32_t j0 = 0; j0 < K; j0 += 32) {
          const uint64_t key = j0 + lane < K ? sk[j0 + lane] : 0ull;
          const uint32_t mj = j0 + lane < K ? (uint32_t)recs[(uint32_t)key].cells : 0u, fj = (uint32_t)(key >> 32);
          uint32_t any = __reduce_or_sync(0xffffffffu, mj);
          while (any) {
            const int c = __ffs(any) - 1;
            any &= any - 1;
            const bool r = (mj >> c) & 1u;
            const uint32_t who = __ballot_sync(0xffffffffu, r);
            const uint32_t to = __shfl_sync(0xffffffffu, at, c);
            const uint32_t i = to + __popc(who & ((1u << lane) - 1u));
            if (r && (int64_t)i < a.cap_pairs) a.adj_ids[i] = fj;
            if (lane == c) at += __popc(who);
          }
        }
        c0 = at - (uint32_t)off0;
      } else {
        bad = true;
      }
      __syncwarp();
      if (bad || c0 != n0 || c1 != n1) atomicOr(a.lv.err, ERR_OVERFLOW);
      return;
    }
    bool h0 = false, h1 = false;
    walk_block<D, PRED, false, false>(a.lv, P, gid, b, sm, phase, lane, wc, h0, h1,
                         [&](uint32_t fc, bool r0, bool r1) { put(r0, r1, fc); });
    if (bad || c0 != n0 || c1 != n1) atomicOr(a.lv.err, ERR_OVERFLOW);
    if (!__all_sync(0xffffffffu, can0 && can1)) return;  // lists beyond the capacity (reported)
    // ascending face ids per cell
    sort_cell_lists(a.adj_ids, NC, n0, n1, off0, off1, sort_area<D>(sm), kSortKeys, lane);
    }
}

template <int D, int PRED, int MODE>
__global__ void __launch_bounds__(256) k_adjacency(EmitArgs a) {
  constexpr int kW = 8;  // warps per CTA at most
  __shared__ uint64_t s_rm[MODE == 0 ? kW : 1][kRecCap];
  __shared__ uint32_t s_rf[MODE == 0 ? kW : 1][kRecCap];
  extern __shared__ __align__(16) unsigned char s_raw[];  // MODE 1: the walk's per-warp memory
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  WarpSmem<D>& sm = *reinterpret_cast<WarpSmem<D>*>(
      s_raw + (MODE == 0 ? 0u : (uint32_t)wid * second_pass_bytes<D>() + walk_offset<D>()));
  uint32_t phase = 0;
  if constexpr (MODE == 1) warp_smem_init<D>(sm, lane);
  uint64_t* rm = s_rm[MODE == 0 ? wid : 0];
  uint32_t* rf = s_rf[MODE == 0 ? wid : 0];
  const uint64_t run_cells = a.run ? a.run[0] : 0ull, run_pairs = a.run ? a.run[1] : 0ull;
  WarpCounters wc;
  if constexpr (MODE == 0) {
    const int64_t n = launch_count(a.lv.n_blocks, a.lv.n_dev, a.lv.err);
    // Up to 32 blocks per atomic: each lane reads one block's mask, the warp then takes the marked blocks of the
    // group one after another.  Fewer where every warp of the launch would not get 32 (a block costs about 1.5 us of
    // one warp's time: 396 blocks took 0.057 ms as 13 groups of 32, 0.030 as 396 of one).
    const int64_t share = n / ((int64_t)gridDim.x * (blockDim.x >> 5));
    const unsigned batch = share < 1 ? 1u : (share < 32 ? (unsigned)share : 32u);
    for (;;) {
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(a.lv.work, batch);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base >= n) break;
      const bool in_range = (unsigned)lane < batch && (int64_t)base + lane < n;
      const uint64_t my_mask = in_range ? a.lv.mask[base + lane] : 0ull;
      const uint32_t my_gid = in_range && a.lv.gid ? a.lv.gid[base + lane] : 0u;
      // the marked blocks' row bases and record descriptors, one coalesced load for the batch
      const bool marked = my_mask != 0;
      const uint64_t my_base = marked ? a.block_base[base + lane] : 0ull;
      const uint64_t my_desc = marked && a.lv.recs ? a.lv.rec_desc[base + lane] : ~0ull;
      unsigned todo = __ballot_sync(0xffffffffu, marked);
      while (todo) {
        const int q = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t gid = __shfl_sync(0xffffffffu, my_gid, q);
        const uint64_t pre[2] = {__shfl_sync(0xffffffffu, my_base, q), __shfl_sync(0xffffffffu, my_desc, q)};
        emit_block<D, PRED, MODE>(a, base + (unsigned)q, gid, sm, phase, wc, rm, rf, lane, run_cells, run_pairs,
                                  pre);
      }
    }
  } else {
    const int64_t nd = (int64_t)*a.defer_n;
    const int64_t n = nd < a.defer_cap ? nd : a.defer_cap;
    for (;;) {
      unsigned i = 0;
      if (lane == 0) i = atomicAdd(a.lv.work, 1u);
      i = __shfl_sync(0xffffffffu, i, 0);
      if ((int64_t)i >= n) break;
      const unsigned blk = a.defer[i];
      const uint32_t gid = a.lv.gid ? a.lv.gid[blk] : 0u;
      emit_block<D, PRED, MODE>(a, blk, gid, sm, phase, wc, rm, rf, lane, run_cells, run_pairs);
    }
  }
}

// Children of the marked blocks whose geometry continues below this level,
// canonical order, single pass with look-back over ticketed tiles.
constexpr int kChThreads = 256;
constexpr int kChItems = 4;

template <int D>
__global__ void __launch_bounds__(kChThreads) k_children(ChildrenArgs a, uint64_t* state, unsigned* ticket) {
  __shared__ unsigned s_tile;
  __shared__ uint32_t s_warp[kChThreads / 32];
  __shared__ uint64_t s_prefix;
  const int64_t n = launch_count(a.n, a.n_dev, a.err);
  const int64_t ntiles = (n + (int64_t)kChThreads * kChItems - 1) / ((int64_t)kChThreads * kChItems);
  constexpr int NCH = D == 3 ? 8 : 4;
  if (ntiles == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.total = 0;
    return;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= ntiles) break;
    const int64_t base = tile * (int64_t)kChThreads * kChItems + (int64_t)threadIdx.x * kChItems;
    uint32_t fl[kChItems];
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < kChItems; ++i) {
      const int64_t j = base + i;
      bool emit = false;
      if (j < n && (a.flag ? a.flag[j] != 0 : a.mask[j] != 0)) {
        const GeomParams P = geom_row(a.g0, a.table, a.gid, j);
        emit = a.level < P.n_levels - 1;
      }
      fl[i] = emit ? 1u : 0u;
      sum += fl[i];
    }
    const uint32_t incl = warp_inclusive_scan<uint32_t>(sum);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      uint32_t w = lane < kChThreads / 32 ? s_warp[lane] : 0u;
      w = warp_inclusive_scan<uint32_t>(w);
      if (lane < kChThreads / 32) s_warp[lane] = w;
    }
    __syncthreads();
    const uint32_t wex = wid > 0 ? s_warp[wid - 1] : 0u;
    if (wid == 0) {
      const uint64_t agg = s_warp[kChThreads / 32 - 1];
      const uint64_t pre = lookback_warp(state, tile, agg, a.err);
      if (lane == 0) {
        s_prefix = pre;
        if (tile == ntiles - 1) {
          const uint64_t tot = (pre + agg) * NCH;
          *a.total = tot;
          if ((int64_t)tot > a.cap_out) atomicOr(a.err, ERR_OVERFLOW);
        }
      }
    }
    __syncthreads();
    uint64_t k = s_prefix + wex + incl - sum;
    if (a.first_child) {
      uint64_t kk = k;
#pragma unroll
      for (int i = 0; i < kChItems; ++i) {
        const int64_t j = base + i;
        if (j < n) {
          const uint64_t o = kk * NCH;
          if (fl[i] && o >= 0x7fffffffull) atomicOr(a.err, ERR_OVERFLOW);
          // children past the level's capacity (reported below) do not exist: the block lookups descend by this index
          a.first_child[j] = fl[i] && (int64_t)(o + NCH) <= a.cap_out ? (int32_t)o : -1;
        }
        kk += fl[i];
      }
    }
#pragma unroll
    for (int i = 0; i < kChItems; ++i) {
      if (fl[i]) {
        const int64_t p = base + i;
        int bc[3] = {0, 0, 0};
#pragma unroll
        for (int c = 0; c < D; ++c) bc[c] = a.blocks[p * D + c];
        const uint32_t g = a.gid ? a.gid[p] : 0u;
#pragma unroll
        for (int s = 0; s < NCH; ++s) {
          const int64_t o = (int64_t)k * NCH + s;
          if (o >= a.cap_out) break;
          a.child_blocks[o * D + 0] = 2 * bc[0] + (s & 1);
          a.child_blocks[o * D + 1] = 2 * bc[1] + ((s >> 1) & 1);
          if (D == 3) a.child_blocks[o * D + 2] = 2 * bc[2] + ((s >> 2) & 1);
          a.child_parent[o] = (int32_t)p;
          if (a.child_gid) a.child_gid[o] = g;
        }
        ++k;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Face-centric marking of a level whose masks are the only output (no
// adjacency lists): one warp per face tests the cells of the level whose test
// region can meet the face (the face's AABB widened by d, in cells) and ORs
// the hits into their blocks' masks.  Coarse levels are where this pays: a
// block there sees hundreds of faces, each of which the block walk tests
// against all of the block's cells, while a face covers only a few cells.
// The decisions are the block walk's: the same certified FP32 tests, in a
// frame at the lower corner of the face's cell range (the error bounds need
// only the frame's offset bounds P and O), and the same FP64 resolution.
// ---------------------------------------------------------------------------

// One cell's SAT test against a survivor: the projections of cell_test2, the box axes and the face
// normal (in 2D, all) first, then the edge axes.
__device__ __forceinline__ void cell_axis(float x, const float4& t, bool& sep, bool& in) {
  sep |= (x < t.x) | (x > t.y);
  in &= (x > t.z) & (x < t.w);
}

template <int D>
__device__ __forceinline__ void cell_axes_face(const Surv<D>& S, const float* o, bool& sep, bool& in) {
#pragma unroll
  for (int ai = 0; ai < D; ++ai) cell_axis(o[ai], S.t[ai], sep, in);
  if constexpr (D == 3) {
    const float4 q2 = S.en[2];
    cell_axis(fmaf(o[2], q2.w, fmaf(o[1], q2.z, o[0] * q2.y)), S.t[3], sep, in);
  } else {
    cell_axis(fmaf(o[1], S.e[0], -o[0] * S.e[1]), S.t[2], sep, in);
  }
}

template <int D>
__device__ __forceinline__ void cell_axes_edges(const Surv<D>& S, const float* o, bool& sep, bool& in) {
  if constexpr (D == 3) {
    const float4 q0 = S.en[0], q1 = S.en[1], q2 = S.en[2];
    const float e[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
      cell_axis(fmaf(o[2], ey, -o[1] * ez), S.t[4 + 3 * k], sep, in);
      cell_axis(fmaf(o[0], ez, -o[2] * ex), S.t[5 + 3 * k], sep, in);
      cell_axis(fmaf(o[1], ex, -o[0] * ey), S.t[6 + 3 * k], sep, in);
    }
  }
}

template <int D>
__device__ __forceinline__ int cell_test1(const Surv<D>& S, const float* o) {
  bool sep = false, in = true;
  cell_axes_face<D>(S, o, sep, in);
  cell_axes_edges<D>(S, o, sep, in);
  return sep ? 0 : (in ? 1 : 2);
}

// setup_face without the block cull, lane-parallel: lane ai < 13 (2D: 3)
// computes axis ai with setup_face's arithmetic; lane 0 stores the edges.
template <int D>
__device__ __forceinline__ void setup_face_lanes(const float* V, const float* nh, const BlockFrame<D>& F, Surv<D>& S,
                                                 int lane) {
  constexpr int NA = D == 3 ? 13 : 3;
  float p[3][3];
  float P = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int c = 0; c < D; ++c) {
      p[k][c] = V[D * k + c] - F.Xb[c];
      P = fmaxf(P, fabsf(p[k][c]));
    }
  const float scale = kEpsK * kU32 * (P + F.O + F.r);
  if (lane < NA) {
    float ax = 0.f, ay = 0.f, az = 0.f;
    if constexpr (D == 3) {
      if (lane < 3) {
        ax = lane == 0 ? 1.f : 0.f;
        ay = lane == 1 ? 1.f : 0.f;
        az = lane == 2 ? 1.f : 0.f;
      } else if (lane == 3) {
        ax = nh[0];
        ay = nh[1];
        az = nh[2];
      } else {
        const int k = (lane - 4) / 3, i = (lane - 4) % 3;
        float ex = 0.f, ey = 0.f, ez = 0.f;
#pragma unroll
        for (int kk = 0; kk < 3; ++kk)
          if (kk == k) {
            const int kn = (kk + 1) % 3;
            ex = V[3 * kn + 0] - V[3 * kk + 0];
            ey = V[3 * kn + 1] - V[3 * kk + 1];
            ez = V[3 * kn + 2] - V[3 * kk + 2];
          }
        if (i == 0) {
          ax = 0.f;
          ay = -ez;
          az = ey;
        } else if (i == 1) {
          ax = ez;
          ay = 0.f;
          az = -ex;
        } else {
          ax = -ey;
          ay = ex;
          az = 0.f;
        }
      }
    } else {
      if (lane < 2) {
        ax = lane == 0 ? 1.f : 0.f;
        ay = lane == 1 ? 1.f : 0.f;
      } else {
        ax = -(V[3] - V[1]);
        ay = V[2] - V[0];
      }
    }
    const float A1 = fabsf(ax) + fabsf(ay) + fabsf(az);
    float4 t = make_float4(-INFINITY, INFINITY, -INFINITY, INFINITY);
    if (A1 != 0.0f) {
      float tmin = INFINITY, tmax = -INFINITY;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float s = D == 3 ? fmaf(p[k][2], az, fmaf(p[k][1], ay, p[k][0] * ax)) : fmaf(p[k][1], ay, p[k][0] * ax);
        tmin = fminf(tmin, s);
        tmax = fmaxf(tmax, s);
      }
      const float eps = scale * A1;
      const float R = F.r * A1;
      const float lo = tmin - R, hi = tmax + R;
      t = make_float4(lo - eps, hi + eps, lo + eps, hi - eps);
    }
    S.t[lane] = t;
  }
  if (lane == 0) {
    if constexpr (D == 3) {
      float e[3][3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int k1 = (k + 1) % 3;
#pragma unroll
        for (int c = 0; c < 3; ++c) e[k][c] = V[3 * k1 + c] - V[3 * k + c];
      }
      S.en[0] = make_float4(e[0][0], e[0][1], e[0][2], e[1][0]);
      S.en[1] = make_float4(e[1][1], e[1][2], e[2][0], e[2][1]);
      S.en[2] = make_float4(e[2][2], nh[0], nh[1], nh[2]);
    } else {
      S.e[0] = V[2] - V[0];
      S.e[1] = V[3] - V[1];
    }
  }
}

constexpr int kMarkWarps = 4;  // warps per CTA of k_mark_faces
constexpr int kMarkSlots = 64;  // blocks of a face's range looked up once per face (more: per cell)

template <int D, int PRED, bool MULTI>
__global__ void __launch_bounds__(kMarkWarps * 32, 6) k_mark_faces(MarkArgs m) {
  const RefineLevel& a = m.lv;
  __shared__ Surv<D> s_surv[kMarkWarps];
  __shared__ int32_t s_bi[kMarkWarps][kMarkSlots];    // block index of each slot of the range (-1: absent)
  __shared__ uint64_t s_mk[kMarkWarps][kMarkSlots];   // its mask when the face started (skips marked cells)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Surv<D>& S = s_surv[wid];
  const int64_t nblk = launch_count(a.n_blocks, a.n_dev, a.err);
  // cell i meets the face's AABB [vmin, vmax] only if its test region does: box,
  // origin + [i h - d, (i + 1) h + d]; point, its centre origin + (i + 1/2) h
  // within [vmin - d, vmax + d]
  constexpr bool kPoint = PRED == 1;
  const int batch = m.batch > 0 ? (m.batch < kFaceBatch ? m.batch : kFaceBatch) : 1;
  WarpCounters wc;
  unsigned long long n_tests = 0;
  for (;;) {
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(a.work, (unsigned)batch);
    base = __shfl_sync(0xffffffffu, base, 0);
    const int64_t first = m.faces.begin + base;
    if (first >= m.faces.end) break;
    for (int q = 0; q < batch; ++q) {
      const int64_t f = first + q;
      if (f >= m.faces.end) break;
      // the face's geometry: only geometries marked face by face on this level (their blocks of the
      // level have the mask as the only output; the walk does the others)
      const uint32_t gid = MULTI ? __ldg(m.face_gid + f) : 0u;
      const GeomParams& P = row<MULTI>(a, gid);
      if (!((P.face_levels >> a.level) & 1u) || (P.face_levels & kFaceUnit)) continue;
      const FastGeom g = fast_geom(P, a.level);
      const float hf = g.h_hi;
      const float inv_h = 1.0f / hf;
      const float R2 = g.d * g.d;
      int ncell[3] = {1, 1, 1};
#pragma unroll
      for (int c = 0; c < D; ++c) ncell[c] = (4 * P.root[c]) << a.level;
      float V[D * D], nh[3] = {0.f, 0.f, 0.f};
      if constexpr (D == 3) {
        const float4* R = reinterpret_cast<const float4*>(m.rec + f);
        const float4 r0 = __ldg(R), r1 = __ldg(R + 1), r2 = __ldg(R + 2);
        V[0] = r0.x; V[1] = r0.y; V[2] = r0.z; V[3] = r0.w; V[4] = r1.x;
        V[5] = r1.y; V[6] = r1.z; V[7] = r1.w; V[8] = r2.x;
        nh[0] = r2.y; nh[1] = r2.z; nh[2] = r2.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) V[j] = __ldg(a.X + (int64_t)j * a.nf + f);
      }
      // cell range per axis: cells whose test region can meet the face's AABB
      // (a superset: the margin covers the FP32 error of the cell coordinate)
      int lo[3] = {0, 0, 0}, n[3] = {1, 1, 1};
      BlockFrame<D> F;
      float shift[3] = {0.f, 0.f, 0.f};
      float O = 0.f;
      bool empty = false;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        float vmin = V[c], vmax = V[c];
#pragma unroll
        for (int k = 1; k < D; ++k) {
          vmin = fminf(vmin, V[D * k + c]);
          vmax = fmaxf(vmax, V[D * k + c]);
        }
        const float margin = 1e-3f + 16.0f * kU32 * (fmaxf(fabsf(vmin), fabsf(vmax)) + fabsf(P.org_hi[c])) * inv_h;
        const float xl = (vmin - P.org_hi[c] - g.d) * inv_h - (kPoint ? 0.5f : 1.0f);
        const float xh = (vmax - P.org_hi[c] + g.d) * inv_h - (kPoint ? 0.5f : 0.0f);
        if (!(xl <= xh)) empty = true;  // also a non-finite coordinate
        const float tl = floorf(xl - margin), th = floorf(xh + margin);
        const int il = tl < 0.f ? 0 : (tl > (float)(ncell[c] - 1) ? ncell[c] : (int)tl);
        const int ih = th < 0.f ? -1 : (th > (float)(ncell[c] - 1) ? ncell[c] - 1 : (int)th);
        if (ih < il) empty = true;
        lo[c] = il;
        n[c] = ih - il + 1;
        float flo;
        df_position(P.org_hi[c], P.org_lo[c], (float)il, g.h_hi, g.h_lo, F.Xb[c], flo);
        shift[c] = flo;
        F.cB[c] = 0.f;
        O = fmaxf(O, (float)(n[c] + 1) * hf + 2.0f * fabsf(flo));
      }
      if (empty) continue;
      F.h = hf;
      F.r = fmaf(0.5f, hf, g.d);
      F.rb = 0.f;
      F.O = O;
      wc.cand++;
      __syncwarp();  // the previous face's tests are done with S
      if constexpr (kPoint) {
        if (lane == 0) setup_point<D>(V, nh, F, S);
      } else {
        setup_face_lanes<D>(V, nh, F, S, lane);
      }
      __syncwarp();
      // the host keeps every range below 2^15 cells (largest face of the binning); a
      // larger one here means inconsistent inputs: reported, not tested
      const int64_t total = (int64_t)n[0] * n[1] * (D == 3 ? n[2] : 1);
      if (total > (1 << 20)) {
        if (lane == 0) atomicOr(a.err, ERR_OVERFLOW);
        continue;
      }
      // index of the level's block with coordinates b, or -1 when the level does not have it: its
      // root by the root order, then per level the ancestor's first child plus the slot (the
      // coordinates' bit of that level per axis); the upper levels' arrays stay in cache
      auto find = [&](const int* b) -> int64_t {
        const int L = a.level;
        int64_t i = P.root_base + (b[0] >> L) + (int64_t)P.root[0] * ((b[1] >> L) + (int64_t)P.root[1] * (b[2] >> L));
        for (int l = 1; l <= L && i >= 0; ++l) {
          const int sh = L - l;
          const int slot = ((b[0] >> sh) & 1) | (((b[1] >> sh) & 1) << 1) | (D == 3 ? ((b[2] >> sh) & 1) << 2 : 0);
          const int32_t c = __ldg(m.first_child[l - 1] + i);
          i = c >= 0 ? (int64_t)c + slot : -1;
        }
        return i < nblk ? i : -1;
      };
      // the range's blocks: looked up once, one lane per block, when they fit the slots
      int blo[3] = {0, 0, 0}, nbk[3] = {1, 1, 1};
#pragma unroll
      for (int c = 0; c < D; ++c) {
        blo[c] = lo[c] >> 2;
        nbk[c] = ((lo[c] + n[c] - 1) >> 2) - blo[c] + 1;
      }
      const int nslot = nbk[0] * nbk[1] * nbk[2];
      const bool slots = nslot <= kMarkSlots;
      // k = a + n b (0 <= a < n, k < 2^20): b = floor((k + 1/2) / n), exactly, from an FP32
      // reciprocal (the quotient is at least 1/(2n) from an integer; the error is below 2^-21 k / n)
      auto divn = [](int k, float inv) { return (int)(((float)k + 0.5f) * inv); };
      const float inv_b0 = 1.0f / (float)nbk[0], inv_b1 = 1.0f / (float)nbk[1];
      if (slots) {
        for (int k = lane; k < nslot; k += 32) {
          const int k1 = divn(k, inv_b0), k2 = divn(k1, inv_b1);
          const int b[3] = {blo[0] + k - k1 * nbk[0], blo[1] + k1 - k2 * nbk[1], blo[2] + k2};
          const int64_t bi = find(b);
          s_bi[wid][k] = (int32_t)bi;
          s_mk[wid][k] = bi >= 0 ? a.mask[bi] : ~0ull;  // absent: every cell skipped
        }
        __syncwarp();
      }
      const float inv_n0 = 1.0f / (float)n[0], inv_n1 = 1.0f / (float)n[1];
      for (int j = lane; j < (int)total; j += 32) {
        const int j1 = divn(j, inv_n0), j2 = D == 3 ? divn(j1, inv_n1) : 0;
        const int i0 = j - j1 * n[0];
        const int i1 = D == 3 ? j1 - j2 * n[1] : j1, i2 = j2;
        const int cell[3] = {lo[0] + i0, lo[1] + i1, D == 3 ? lo[2] + i2 : 0};
        int b[3] = {cell[0] >> 2, cell[1] >> 2, D == 3 ? cell[2] >> 2 : 0};
        const int local = (cell[0] & 3) | ((cell[1] & 3) << 2) | (D == 3 ? (cell[2] & 3) << 4 : 0);
        const uint64_t bit = 1ull << local;
        int64_t bi;
        uint64_t mk;
        if (slots) {
          const int k = (b[0] - blo[0]) + nbk[0] * ((b[1] - blo[1]) + nbk[1] * (b[2] - blo[2]));
          bi = s_bi[wid][k];
          mk = s_mk[wid][k];
        } else {
          bi = find(b);
          mk = bi >= 0 ? a.mask[bi] : ~0ull;
        }
        if (mk & bit) continue;  // absent block or already marked (a stale mask only costs a test)
        ++n_tests;
        const float l[3] = {(float)i0 + 0.5f, (float)i1 + 0.5f, (float)i2 + 0.5f};
        float o[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < D; ++c) o[c] = fmaf(l[c], g.h_hi, fmaf(l[c], g.h_lo, shift[c]));
        int t = kPoint ? point_test<D>(S, o, R2) : cell_test1<D>(S, o);
        if (t == 2) {
          // not certified in FP32: FP64, unless another face has marked the cell meanwhile
          if (__ldcg(reinterpret_cast<const unsigned long long*>(a.mask + bi)) & bit) continue;
          t = resolve_fp64<D>(a, gid, (uint32_t)f, b, local, &wc.fb, &wc.band) ? 1 : 0;
        }
        if (t) {
          atomicOr(reinterpret_cast<unsigned long long*>(a.mask + bi), (unsigned long long)bit);
          a.flag[bi] = 1;
        }
      }
    }
  }
  unsigned long long v[4] = {wc.fb, wc.band, wc.cand, n_tests};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  }
  if (lane == 0) {
    if (v[0]) atomicAdd(&a.counters[CNT_FALLBACK], v[0]);
    if (v[1]) atomicAdd(&a.counters[CNT_BAND], v[1]);
    if (v[2]) atomicAdd(&a.counters[CNT_FACE_SETUPS], v[2] / 32);  // every lane counted the same faces
    if (v[3]) atomicAdd(&a.counters[CNT_FACE_TESTS], v[3]);
  }
}

// ---------------------------------------------------------------------------
// The same marking where d is the cell size itself (d_abs = 0, d_rel = 1, the
// default) and the predicate the box one.  A cell's inflated box is then the
// 3^D block of cells around it, so a face meets it exactly when the face meets
// one of those cells: a face is tested against the few cells that its own AABB
// reaches (r = h / 2), and the cells it meets are widened by one cell with bit
// operations on the block masks.  On the largest workload that leaves 16 cells
// per face and level to test instead of 84.
//
// The decisions stay those of the definition.  A certified overlap with a cell
// is far beyond FP64's rounding, so the inflated boxes of its neighbours meet
// the face; a face certified apart from all 3^D cells of an inflated box has a
// distance from it that FP64 sees.  Where the test of a cell is not certified,
// those of its 3^D neighbours that no certified cell marks are tested with their
// own inflated boxes, each once, as everywhere else (FP32, then FP64).  Cells of one layer outside the domain are tested as
// well, for they widen into it.  A cell that a face meets lies in a block of
// the level: the cell above it was marked.
//
// A warp takes up to kCellFaces faces in steps, each packed over all the faces: a
// lane per face (cell range, axis thresholds), a lane per block of the ranges
// (index), where the ranges are long a lane per x-row (the part of it that no
// axis separates), a lane per cell, a lane per block again (widening, then one
// atomic for its new marks).  A face with more blocks than kCellPool is taken in
// tiles.  Bound by instructions and the latency of the block lookups.  Against a
// warp per face testing every inflated cell (k_mark_faces): the five levels of
// 1.3 M faces 10.6 -> 2.36 ms, the four of 82 K 0.76 -> 0.29, the three of 20 K
// 0.22 -> 0.13 (the uncertified cells' tests by one lane in a row: 4.5, 1.0 and
// 0.53 ms).
//
// REC: the level is the last of its geometries and their adjacency is wanted.  A
// face's widened cells of a block are then the block's survivor record, so the
// face leaves it (staged, with its rank among the block's records) and
// k_place_records brings the records together by block: no block walks its bins.
// Marks and records of the finest level, 1.3 M faces of 9 cells edge on 11 M
// blocks: 15.5 ms by the parents' walk (k_refine_groups), 4.3 + 1.1 ms; 82 K on
// 0.76 M: 0.98 -> 0.41 + 0.05.  Without the rows' cut the faces took 5.6 ms; 8
// faces per warp and 7 blocks per SM 5.9.
// ---------------------------------------------------------------------------
template <int D>
struct MarkFace {
  float shift[3];              // frame corner's rounding error
  float h_hi, h_lo;
  float inv_n0, inv_n1, inv_b0, inv_b1;
  int lo[3], off[3];           // first cell of the range; its place from the frame's corner, in cells
  int blo[3];                  // first block of the widened range
  int n0, n1, nb0, nb1, nb2;   // cells and blocks per axis
  int total, nslot;
  uint32_t slot, face, gid;    // first slot of the range's blocks
  uint8_t c0[3], c1[3];        // blocks of the range (from blo) whose marks are sent
};

constexpr int kCellWarps = 4;    // warps per CTA of k_mark_cells
constexpr int kCellBlocks = 5;   // CTAs per SM (shared memory)
constexpr int kCellFaces = 16;   // faces a warp takes per work fetch
constexpr int kCellPool = 160;   // blocks of the ranges of a group of faces
constexpr uint32_t kCellRow = 3; // mean cells per x-row above which rows are cut first
constexpr int kCellTile = 3;     // a face with more blocks is taken in tiles of 3 per axis and their rims
static_assert((kCellTile + 2) * (kCellTile + 2) * (kCellTile + 2) <= kCellPool, "a tile and its rim fit");

template <int D>
struct CellSmem {
  Surv<D> surv[kCellFaces];
  MarkFace<D> f[kCellFaces];
  alignas(8) uint32_t met[kCellPool][2];  // per block: its cells that the face meets, then widened
  uint64_t tmp[kCellPool];
  uint32_t open[kCellPool][2];   // cells whose test was not certified
  int32_t bi[kCellPool];         // the block's index (-1: absent)
  uint8_t own[kCellPool];        // its face
  int whole[4][3];               // a face taken in tiles: lo, n, blo, nb of its range
};

// cell_test1 for the cell's box widened by grow: the thresholds move by grow |a|_1, and the
// certificates by the rounding of that.
template <int D>
__device__ __noinline__ int cell_test_grown(const Surv<D>& S, const float* o, float grow) {
  bool sep = false, in = true;
  auto upd = [&](float x, float A1, const float4& t) {
    const float g = grow * A1, e = kEpsK * kU32 * g;
    sep |= (x < (t.x - g) - e) | (x > (t.y + g) + e);
    in &= (x > (t.z - g) + e) & (x < (t.w + g) - e);
  };
  if constexpr (D == 3) {
#pragma unroll
    for (int ai = 0; ai < 3; ++ai) upd(o[ai], 1.f, S.t[ai]);
    const float4 q0 = S.en[0], q1 = S.en[1], q2 = S.en[2];
    const float e[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
    upd(fmaf(o[2], q2.w, fmaf(o[1], q2.z, o[0] * q2.y)), fabsf(q2.y) + fabsf(q2.z) + fabsf(q2.w), S.t[3]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
      upd(fmaf(o[2], ey, -o[1] * ez), fabsf(ey) + fabsf(ez), S.t[4 + 3 * k]);
      upd(fmaf(o[0], ez, -o[2] * ex), fabsf(ex) + fabsf(ez), S.t[5 + 3 * k]);
      upd(fmaf(o[1], ex, -o[0] * ey), fabsf(ex) + fabsf(ey), S.t[6 + 3 * k]);
    }
  } else {
    upd(o[0], 1.f, S.t[0]);
    upd(o[1], 1.f, S.t[1]);
    upd(fmaf(o[1], S.e[0], -o[0] * S.e[1]), fabsf(S.e[0]) + fabsf(S.e[1]), S.t[2]);
  }
  return sep ? 0 : (in ? 1 : 2);
}

// The part of an x-row (iy, iz) of a face's range that no axis separates from the face: first cell and
// count.  The projection of a cell centre on an axis is linear along the row, so each axis leaves an
// interval; it is kept a little too wide (the cells left are tested), which also covers the rounding of
// the projection at the row's start.  An axis with hardly any x part cuts nothing.
__device__ __forceinline__ void row_part(const Surv<3>& S, const MarkFace<3>& Q, int iy, int iz, int& ix, uint32_t& n) {
  const float lx = (float)Q.off[0] + 0.5f, ly = (float)(Q.off[1] + iy) + 0.5f, lz = (float)(Q.off[2] + iz) + 0.5f;
  const float ox = fmaf(lx, Q.h_hi, fmaf(lx, Q.h_lo, Q.shift[0])), oy = fmaf(ly, Q.h_hi, fmaf(ly, Q.h_lo, Q.shift[1])),
              oz = fmaf(lz, Q.h_hi, fmaf(lz, Q.h_lo, Q.shift[2]));
  float lo = 0.f, hi = (float)(Q.n0 - 1);
  auto cut = [&](float s, float ax, const float4& t) {
    const float g = ax * Q.h_hi;
    if (fabsf(g) > 1e-35f) {
      const float r = __fdividef(1.0f, g), a = (t.x - s) * r, b = (t.y - s) * r;
      lo = fmaxf(lo, fminf(a, b));
      hi = fminf(hi, fmaxf(a, b));
    }
  };
  cut(ox, 1.f, S.t[0]);
  const float4 q0 = S.en[0], q1 = S.en[1], q2 = S.en[2];
  cut(fmaf(oz, q2.w, fmaf(oy, q2.z, ox * q2.y)), q2.y, S.t[3]);
  const float e[3][3] = {{q0.x, q0.y, q0.z}, {q0.w, q1.x, q1.y}, {q1.z, q1.w, q2.x}};
  bool out = (oy < S.t[1].x) | (oy > S.t[1].y) | (oz < S.t[2].x) | (oz > S.t[2].y);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float ex = e[k][0], ey = e[k][1], ez = e[k][2];
    const float s = fmaf(oz, ey, -oy * ez);
    const float4 t = S.t[4 + 3 * k];
    out |= (s < t.x) | (s > t.y);
    cut(fmaf(ox, ez, -oz * ex), ez, S.t[5 + 3 * k]);
    cut(fmaf(oy, ex, -ox * ey), -ey, S.t[6 + 3 * k]);
  }
  const int i0 = (int)fmaxf(0.f, ceilf(lo - 1e-3f)), i1 = (int)fminf((float)(Q.n0 - 1), floorf(hi + 1e-3f));
  ix = i0;
  n = !out && i1 >= i0 ? (uint32_t)(i1 - i0 + 1) : 0u;
}
__device__ __forceinline__ void row_part(const Surv<2>&, const MarkFace<2>&, int, int, int&, uint32_t&) {}

// A block mask widened by one cell along axis AX: its own cells, and the neighbours' facing layers
// (prev / next: the masks of the blocks before and after it on that axis).
template <int AX>
__device__ __forceinline__ uint64_t widen(uint64_t m, uint64_t prev, uint64_t next) {
  constexpr int s = 2 * AX == 0 ? 1 : (AX == 1 ? 4 : 16);
  constexpr uint64_t first = AX == 0 ? 0x1111111111111111ull : (AX == 1 ? 0x000f000f000f000full : 0xffffull);
  constexpr uint64_t last = first << (3 * s);
  return m | ((m << s) & ~first) | ((m >> s) & ~last) | ((prev >> (3 * s)) & first) | ((next << (3 * s)) & last);
}

template <int D, bool MULTI, bool REC>
__global__ void __launch_bounds__(kCellWarps * 32, kCellBlocks) k_mark_cells(MarkArgs m) {
  const RefineLevel& a = m.lv;
  __shared__ __align__(16) CellSmem<D> s_all[kCellWarps];
  const int lane = threadIdx.x & 31;
  CellSmem<D>& sm = s_all[threadIdx.x >> 5];
  const int64_t nblk = launch_count(a.n_blocks, a.n_dev, a.err);
  const int batch = m.batch > 0 ? (m.batch < kCellFaces ? m.batch : kCellFaces) : 1;
  // k = a + n b (0 <= a < n, k < 2^20): b = floor((k + 1/2) / n), exactly, from an FP32
  // reciprocal (the quotient is at least 1/(2n) from an integer; the error is below 2^-21 k / n)
  auto divn = [](int k, float inv) { return (int)(((float)k + 0.5f) * inv); };
  // index of the level's block with coordinates b, or -1 when the level does not have it: its
  // root by the root order, then per level the ancestor's first child plus the slot (the
  // coordinates' bit of that level per axis); the upper levels' arrays stay in cache
  auto find = [&](uint32_t g, const int* b) -> int32_t {
    const GeomParams& Q = row<MULTI>(a, g);
    const int L = a.level;
#pragma unroll
    for (int c = 0; c < D; ++c)
      if (b[c] < 0 || b[c] >= (Q.root[c] << L)) return -1;
    int64_t i = Q.root_base + (b[0] >> L) + (int64_t)Q.root[0] * ((b[1] >> L) + (int64_t)Q.root[1] * (b[2] >> L));
    for (int l = 1; l <= L && i >= 0; ++l) {
      const int sh = L - l;
      const int slot = ((b[0] >> sh) & 1) | (((b[1] >> sh) & 1) << 1) | (D == 3 ? ((b[2] >> sh) & 1) << 2 : 0);
      const int32_t c = __ldg(m.first_child[l - 1] + i);
      i = c >= 0 ? (int64_t)c + slot : -1;
    }
    return i < nblk ? (int32_t)i : -1;
  };
  auto set_range = [](MarkFace<D>& M, const int* n, const int* nb) {
    M.total = n[0] * n[1] * n[2];
    M.nslot = nb[0] * nb[1] * nb[2];
    M.n0 = n[0], M.n1 = n[1], M.nb0 = nb[0], M.nb1 = nb[1], M.nb2 = nb[2];
    M.inv_n0 = 1.0f / (float)n[0], M.inv_n1 = 1.0f / (float)n[1];
    M.inv_b0 = 1.0f / (float)nb[0], M.inv_b1 = 1.0f / (float)nb[1];
  };
  WarpCounters wc;
  unsigned long long n_tests = 0;
  for (;;) {
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(a.work, (unsigned)batch);
    base = __shfl_sync(0xffffffffu, base, 0);
    const int64_t first = m.faces.begin + base;
    if (first >= m.faces.end) break;
    // a lane per face: its cell range and thresholds
    const int64_t f = first + lane;
    bool use = lane < batch && f < m.faces.end;
    const uint32_t gid = MULTI && use ? __ldg(m.face_gid + f) : 0u;
    const GeomParams& P = row<MULTI>(a, gid);
    use = use && ((P.face_levels >> a.level) & 1u) && (P.face_levels & kFaceUnit);
    MarkFace<D> M;
    BlockFrame<D> F;
    float V[D * D], nh[3] = {0.f, 0.f, 0.f};
    if (use) {
      const FastGeom g = fast_geom(P, a.level);
      const float hf = g.h_hi, inv_h = 1.0f / hf;
      if constexpr (D == 3) {
        const float4* R = reinterpret_cast<const float4*>(m.rec + f);
        const float4 r0 = __ldg(R), r1 = __ldg(R + 1), r2 = __ldg(R + 2);
        V[0] = r0.x; V[1] = r0.y; V[2] = r0.z; V[3] = r0.w; V[4] = r1.x;
        V[5] = r1.y; V[6] = r1.z; V[7] = r1.w; V[8] = r2.x;
        nh[0] = r2.y; nh[1] = r2.z; nh[2] = r2.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) V[j] = __ldg(a.X + (int64_t)j * a.nf + f);
      }
      // cells that can meet the face's AABB (a superset: the margin covers the FP32 error of the
      // cell coordinate), down to one layer outside the domain; the blocks of that range widened
      int n[3] = {1, 1, 1}, nb[3] = {1, 1, 1};
      float O = 0.f;
      M.lo[2] = M.blo[2] = 0;
      M.shift[2] = 0.f;
#pragma unroll
      for (int c = 0; c < D; ++c) {
        const int ncell = (4 * P.root[c]) << a.level;
        float vmin = V[c], vmax = V[c];
#pragma unroll
        for (int k = 1; k < D; ++k) {
          vmin = fminf(vmin, V[D * k + c]);
          vmax = fmaxf(vmax, V[D * k + c]);
        }
        const float margin = 1e-3f + 16.0f * kU32 * (fmaxf(fabsf(vmin), fabsf(vmax)) + fabsf(P.org_hi[c])) * inv_h;
        const float xl = (vmin - P.org_hi[c]) * inv_h, xh = (vmax - P.org_hi[c]) * inv_h;
        if (!(xl <= xh)) use = false;  // also a non-finite coordinate
        const float tl = floorf(xl - margin), th = floorf(xh + margin);
        const int il = tl < -1.f ? -1 : (tl > (float)ncell ? ncell + 1 : (int)tl);
        const int ih = th < -1.f ? -2 : (th > (float)ncell ? ncell : (int)th);
        if (ih < il) use = false;
        M.lo[c] = il;
        n[c] = ih - il + 1;
        M.blo[c] = (il - 1) >> 2;
        nb[c] = ((ih + 1) >> 2) - M.blo[c] + 1;
        float flo;
        df_position(P.org_hi[c], P.org_lo[c], (float)il, g.h_hi, g.h_lo, F.Xb[c], flo);
        M.shift[c] = flo;
        F.cB[c] = 0.f;
        // the frame holds the range and the neighbours of its cells
        O = fmaxf(O, (float)(n[c] + 2) * hf + 2.0f * fabsf(flo));
      }
      F.h = hf;
      F.r = 0.5f * hf;
      F.rb = 0.f;
      F.O = O;
      // the host keeps every range below 2^15 cells (largest face of the binning); a
      // larger one here means inconsistent inputs: reported, not tested
      const int64_t wide = (int64_t)(n[0] + 2) * (n[1] + 2) * (D == 3 ? n[2] + 2 : 1);
      if (use && wide > (1 << 20)) {
        atomicOr(a.err, ERR_OVERFLOW);
        use = false;
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        M.off[c] = 0;
        M.c0[c] = 0;
        M.c1[c] = (uint8_t)(nb[c] < 255 ? nb[c] : 255);
      }
      M.h_hi = g.h_hi, M.h_lo = g.h_lo;
      M.slot = 0u, M.face = (uint32_t)f, M.gid = gid;
      set_range(M, n, nb);
    }
    const unsigned valid = __ballot_sync(0xffffffffu, use);
    const int nv = __popc(valid);
    if (use) {
      wc.cand++;
      const int i = __popc(valid & ((1u << lane) - 1u));
      setup_face<D, false>(V, nh, F, sm.surv[i]);
      sm.f[i] = M;
    }
    __syncwarp();
    int my_total = lane < nv ? sm.f[lane].total : 0;
    int my_slots = lane < nv ? sm.f[lane].nslot : 0;
    int tile = 0;            // tiles of the face g0 already taken, where it has too many blocks
    for (int g0 = 0; g0 < nv;) {
      // a run of faces whose blocks fit the slots, or a tile of one face with more
      bool big = tile > 0;
      if (tile == 0) {
        const MarkFace<D>& Q = sm.f[g0];
        big = Q.nslot > kCellPool;
        if (big) {
          const int wn[3] = {Q.n0, Q.n1, Q.total / (Q.n0 * Q.n1)}, wb[3] = {Q.nb0, Q.nb1, Q.nb2};
          if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              sm.whole[0][q] = Q.lo[q];
              sm.whole[1][q] = wn[q];
              sm.whole[2][q] = Q.blo[q];
              sm.whole[3][q] = wb[q];
            }
          }
          __syncwarp();
        }
      }
      int g1 = g0 + 1;
      if (big) {
        int nt[3], t[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) nt[q] = (sm.whole[3][q] + kCellTile - 1) / kCellTile;
        t[0] = tile % nt[0], t[1] = tile / nt[0] % nt[1], t[2] = tile / (nt[0] * nt[1]);
        __syncwarp();
        MarkFace<D> M = sm.f[g0];
        int n[3], nb[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          // its blocks, one more around them (for the cells that widen into them), and of the face's
          // range the cells within one of its own
          const int b0 = t[q] * kCellTile, b1 = min(b0 + kCellTile, sm.whole[3][q]);
          const int h0 = max(b0 - 1, 0), h1 = min(b1 + 1, sm.whole[3][q]);
          const int lo = max(sm.whole[0][q], 4 * (sm.whole[2][q] + b0) - 1);
          const int hi = min(sm.whole[0][q] + sm.whole[1][q] - 1, 4 * (sm.whole[2][q] + b1));
          M.lo[q] = q < D ? lo : 0;
          n[q] = q < D ? hi - lo + 1 : 1;
          M.off[q] = q < D ? lo - sm.whole[0][q] : 0;
          M.blo[q] = sm.whole[2][q] + h0;
          nb[q] = h1 - h0;
          M.c0[q] = (uint8_t)(b0 - h0), M.c1[q] = (uint8_t)(b1 - h0);
        }
        if (n[0] <= 0 || n[1] <= 0 || n[2] <= 0) n[0] = n[1] = n[2] = 0;
        set_range(M, n, nb);
        __syncwarp();  // every lane has read the face
        if (lane == 0) sm.f[g0] = M;
        __syncwarp();
        if (lane == g0) my_total = M.total, my_slots = M.nslot;
        if (++tile == nt[0] * nt[1] * nt[2]) tile = 0;
      }
      const bool last_tile = tile == 0;
      const uint32_t ns = lane >= g0 && lane < nv ? (uint32_t)min(my_slots, kCellPool + 1) : 0u;
      const uint32_t sincl = warp_inclusive_scan<uint32_t>(ns);
      if (!big) g1 = g0 + __popc(__ballot_sync(0xffffffffu, ns && sincl <= (uint32_t)kCellPool));
      const bool own = lane >= g0 && lane < g1;
      const uint32_t nsl = __shfl_sync(0xffffffffu, sincl, g1 - 1);
      const uint32_t sfirst = sincl - ns;
      if (own) sm.f[lane].slot = sfirst;
      __syncwarp();
      for (uint32_t k0 = 0; k0 < nsl; k0 += 32) {
        const int j = range_owner(sfirst, own, g0, k0, lane);
        const uint32_t s = k0 + lane;
        if (s < nsl) {
          const MarkFace<D>& Q = sm.f[j];
          const int k = (int)(s - Q.slot);
          const int k1 = divn(k, Q.inv_b0), k2 = divn(k1, Q.inv_b1);
          const int b[3] = {Q.blo[0] + k - k1 * Q.nb0, Q.blo[1] + k1 - k2 * Q.nb1, Q.blo[2] + k2};
          sm.bi[s] = find(Q.gid, b);
          sm.own[s] = (uint8_t)j;
          sm.met[s][0] = sm.met[s][1] = 0u;
          sm.open[s][0] = sm.open[s][1] = 0u;
        }
      }
      __syncwarp();
      const uint32_t nc = own ? (uint32_t)my_total : 0u;
      const uint32_t cincl = warp_inclusive_scan<uint32_t>(nc);
      const uint32_t cfirst = cincl - nc, ncell = __shfl_sync(0xffffffffu, cincl, 31);
      // cell (i + dd) of face j's range: its coordinates and its centre in the face's frame
      auto centre = [&](const MarkFace<D>& Q, const int* i, int d0, int d1, int d2, int* x, float* o) {
        const int dd[3] = {d0, d1, d2};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          x[q] = Q.lo[q] + i[q] + dd[q];
          const float l = (float)(Q.off[q] + i[q] + dd[q]) + 0.5f;
          o[q] = q < D ? fmaf(l, Q.h_hi, fmaf(l, Q.h_lo, Q.shift[q])) : 0.f;
        }
      };
      auto cell_of = [&](const MarkFace<D>& Q, int idx, int* i) {
        const int j1 = divn(idx, Q.inv_n0), j2 = D == 3 ? divn(j1, Q.inv_n1) : 0;
        i[0] = idx - j1 * Q.n0;
        i[1] = D == 3 ? j1 - j2 * Q.n1 : j1;
        i[2] = j2;
      };
      auto local_of = [](const int* x) { return (x[0] & 3) | ((x[1] & 3) << 2) | (D == 3 ? (x[2] & 3) << 4 : 0); };
      auto slot_of = [](const MarkFace<D>& Q, const int* x) {
        return Q.slot + (uint32_t)(((x[0] >> 2) - Q.blo[0]) +
                                   Q.nb0 * (((x[1] >> 2) - Q.blo[1]) + Q.nb1 * ((x[2] >> 2) - Q.blo[2])));
      };
      // the cells' tests, 32 at a time: of whole ranges, or (ranges with long x-rows) of the part of each
      // row that no axis separates, a lane per row finding it first
      const uint32_t nr = own && nc ? (uint32_t)(nc / sm.f[lane].n0) : 0u;
      const uint32_t rincl = warp_inclusive_scan<uint32_t>(nr);
      const uint32_t rfirst = rincl - nr, nrow = __shfl_sync(0xffffffffu, rincl, 31);
      const bool by_row = D == 3 && ncell > kCellRow * nrow;
      bool any_open = false;
      for (uint32_t r0 = 0; r0 < (by_row ? nrow : 1u); r0 += 32) {
        int jr = 0, iy = 0, iz = 0, ix = 0;
        uint32_t rc = 0;  // cells of the lane's row, from ix on
        if (by_row) {
          jr = range_owner(rfirst, own && nc, g0, r0, lane);
          const int k = (int)(r0 + lane - __shfl_sync(0xffffffffu, rfirst, jr));
          if (r0 + lane < nrow) {
            const MarkFace<D>& Q = sm.f[jr];
            iz = divn(k, Q.inv_n1);
            iy = k - iz * Q.n1;
            row_part(sm.surv[jr], Q, iy, iz, ix, rc);
          }
        }
        const uint32_t tincl = warp_inclusive_scan<uint32_t>(rc);
        const uint32_t tfirst = tincl - rc;
        const uint32_t items = by_row ? __shfl_sync(0xffffffffu, tincl, 31) : ncell;
        for (uint32_t k0 = 0; k0 < items; k0 += 32) {
          const bool valid_cell = k0 + lane < items;
          int j, ci[3] = {0, 0, 0};
          if (by_row) {
            int l = 0;  // the last row that starts at or before the item
#pragma unroll
            for (int st = 16; st > 0; st >>= 1) {
              const uint32_t fs = __shfl_sync(0xffffffffu, tfirst, l + st);
              if (fs <= k0 + lane) l += st;
            }
            j = __shfl_sync(0xffffffffu, jr, l);
            ci[0] = __shfl_sync(0xffffffffu, ix, l) + (int)(k0 + lane - __shfl_sync(0xffffffffu, tfirst, l));
            ci[1] = __shfl_sync(0xffffffffu, iy, l);
            ci[2] = __shfl_sync(0xffffffffu, iz, l);
          } else {
            j = range_owner(cfirst, own && nc, g0, k0, lane);  // (a tile may have no cells)
            const int idx = (int)(k0 + lane - __shfl_sync(0xffffffffu, cfirst, j));
            if (valid_cell) cell_of(sm.f[j], idx, ci);
          }
          const MarkFace<D>& C = sm.f[j];
          int cx[3];
          float co[3];
          bool sep = !valid_cell, in = true;
          if (valid_cell) {
            centre(C, ci, 0, 0, 0, cx, co);
            ++n_tests;
            cell_axes_face<D>(sm.surv[j], co, sep, in);
          }
          // in some rounds the face's plane passes by every cell: no edge axes then
          if (D == 3 && __any_sync(0xffffffffu, !sep) && valid_cell) cell_axes_edges<D>(sm.surv[j], co, sep, in);
          if (!sep && in) atomicOr(&sm.met[slot_of(C, cx)][local_of(cx) >> 5], 1u << (local_of(cx) & 31));
          const bool unsure = !sep && !in;
          // a cell whose test is not certified is settled after the widening
          if (unsure) atomicOr(&sm.open[slot_of(C, cx)][local_of(cx) >> 5], 1u << (local_of(cx) & 31));
          any_open |= __any_sync(0xffffffffu, unsure);
        }
      }
      __syncwarp();
      // widen along each axis, a lane per block (met -> tmp -> met -> tmp)
      uint64_t* met = reinterpret_cast<uint64_t*>(&sm.met[0][0]);
      auto at_of = [&](uint32_t s, int* at) {  // a slot's place in its face's blocks
        const MarkFace<D>& Q = sm.f[sm.own[s]];
        const int k = (int)(s - Q.slot), k1 = divn(k, Q.inv_b0), k2 = divn(k1, Q.inv_b1);
        at[0] = k - k1 * Q.nb0, at[1] = k1 - k2 * Q.nb1, at[2] = k2;
      };
      auto sends = [&](uint32_t s) {  // a block of the level, and of the tile itself
        const MarkFace<D>& Q = sm.f[sm.own[s]];
        int at[3];
        at_of(s, at);
        bool send = sm.bi[s] >= 0;
#pragma unroll
        for (int q = 0; q < D; ++q) send = send && at[q] >= Q.c0[q] && at[q] < Q.c1[q];
        return send;
      };
      auto pass = [&](auto ax, const uint64_t* in, uint64_t* out, bool last) {
        constexpr int AX = decltype(ax)::value;
        for (uint32_t s = lane; s < nsl; s += 32) {
          const MarkFace<D>& Q = sm.f[sm.own[s]];
          int at[3];
          at_of(s, at);
          const int n = AX == 0 ? Q.nb0 : (AX == 1 ? Q.nb1 : Q.nb2);
          const int step = AX == 0 ? 1 : (AX == 1 ? Q.nb0 : Q.nb0 * Q.nb1);
          uint64_t w = widen<AX>(in[s], at[AX] > 0 ? in[s - step] : 0ull, at[AX] + 1 < n ? in[s + step] : 0ull);
          if (last) w = sends(s) ? w & (D == 3 ? ~0ull : 0xffffull) : 0ull;
          out[s] = w;
        }
        __syncwarp();
      };
      pass(std::integral_constant<int, 0>{}, met, sm.tmp, false);
      pass(std::integral_constant<int, 1>{}, sm.tmp, met, D == 2);
      if constexpr (D == 3) pass(std::integral_constant<int, 2>{}, met, sm.tmp, true);
      uint64_t* res = D == 3 ? sm.tmp : met;
      if (any_open) {
        // the neighbours of open cells that no certain cell has marked: each once, by its own inflated box, a lane
        // per neighbour; then FP64, in 3D a few by the whole warp, more of them a lane each
        uint32_t* out = reinterpret_cast<uint32_t*>(res);
        uint32_t* seen = reinterpret_cast<uint32_t*>(D == 3 ? met : sm.tmp);
        for (uint32_t k = lane; k < 2 * nsl; k += 32) seen[k] = 0u;
        __syncwarp();
        uint32_t pend = 0;  // lane i: the i-th neighbour (slot << 6 | cell) left to FP64
        int np = 0;
        auto decide = [&]() {
          auto cell_at = [&](uint32_t e, int* z) {
            const MarkFace<D>& Q = sm.f[sm.own[e >> 6]];
            int at[3];
            at_of(e >> 6, at);
#pragma unroll
            for (int q = 0; q < 3; ++q) z[q] = q < D ? 4 * (Q.blo[q] + at[q]) + (int)((e >> (2 * q)) & 3u) : 0;
            return &Q;
          };
          if (D == 2 || np > kFewFp64) {
            if (lane < np) {
              int z[3];
              const MarkFace<D>& Q = *cell_at(pend, z);
              const int b[3] = {z[0] >> 2, z[1] >> 2, z[2] >> 2};
              if (resolve_fp64<D>(a, Q.gid, Q.face, b, (int)(pend & 63u), &wc.fb, &wc.band))
                atomicOr(out + 2 * (pend >> 6) + ((pend >> 5) & 1u), 1u << (pend & 31u));
            }
          } else if constexpr (D == 3) {
            for (int k = 0; k < np; ++k) {
              const uint32_t e = __shfl_sync(0xffffffffu, pend, k);
              int z[3];
              const MarkFace<D>& Q = *cell_at(e, z);
              const uint32_t w = resolve_sat_warp(a, Q.gid, Q.face, z[0] >> 2, z[1] >> 2, z[2] >> 2, (int)(e & 63u));
              if (lane == 0) {
                ++wc.fb;
                wc.band += w >> 1;
                if (w & 1u) atomicOr(out + 2 * (e >> 6) + ((e >> 5) & 1u), 1u << (e & 31u));
              }
            }
          }
          np = 0;
          __syncwarp();
        };
        for (uint32_t s = 0; s < nsl; ++s) {
          for (uint64_t u = sm.open[s][0] | (uint64_t)sm.open[s][1] << 32; u; u &= u - 1) {
            const int cell = __ffsll((long long)u) - 1;
            const MarkFace<D>& Q = sm.f[sm.own[s]];
            int t = 0, x[3] = {0, 0, 0};
            uint32_t y = 0;
            if (lane < (D == 3 ? 27 : 9)) {
              int at[3], i[3] = {0, 0, 0};
              float o[3];
              at_of(s, at);
#pragma unroll
              for (int q = 0; q < D; ++q) i[q] = 4 * (Q.blo[q] + at[q]) + ((cell >> (2 * q)) & 3) - Q.lo[q];
              centre(Q, i, lane % 3 - 1, lane / 3 % 3 - 1, D == 3 ? lane / 9 - 1 : 0, x, o);
              const uint32_t sy = slot_of(Q, x);
              y = 2 * sy + (local_of(x) >> 5);
              const uint32_t bit = 1u << (local_of(x) & 31);
              if (sends(sy) && !(out[y] & bit) && !(atomicOr(seen + y, bit) & bit)) {
                // (a record wants every cell of its face, a mask only the cells that are not marked yet)
                const uint64_t now = REC ? 0ull : __ldcg(reinterpret_cast<const unsigned long long*>(a.mask + sm.bi[sy]));
                if (!((now >> local_of(x)) & 1ull)) t = cell_test_grown<D>(sm.surv[sm.own[s]], o, Q.h_hi);
              }
            }
            if (t == 1) atomicOr(out + y, 1u << (local_of(x) & 31));
            for (unsigned vb = __ballot_sync(0xffffffffu, t == 2); vb; vb &= vb - 1) {
              const uint32_t e = __shfl_sync(0xffffffffu, (y >> 1) << 6 | (uint32_t)local_of(x), __ffs(vb) - 1);
              if (lane == np) pend = e;
              if (++np == 32) decide();
            }
            __syncwarp();
          }
        }
        if (np) decide();
      }
      // a block's new marks with one atomic; a face of a geometry that ends here leaves a record for the block
      auto ends_here = [&](uint32_t s) {
        return !MULTI || row<MULTI>(a, sm.f[sm.own[s]].gid).n_levels - 1 == a.level;
      };
      uint32_t nrec = 0;
      for (uint32_t s0 = 0; s0 < nsl; s0 += 32) {
        const uint32_t s = s0 + lane;
        const uint64_t w = s < nsl ? res[s] : 0ull;
        if (w) {
          const int32_t bi = sm.bi[s];
          const uint64_t now = __ldcg(reinterpret_cast<const unsigned long long*>(a.mask + bi));
          if (w & ~now) {
            atomicOr(reinterpret_cast<unsigned long long*>(a.mask + bi), (unsigned long long)w);
            if (now == 0) a.flag[bi] = 1;
          }
        }
        if constexpr (REC) nrec += __popc(__ballot_sync(0xffffffffu, w && ends_here(s)));
      }
      if constexpr (REC) {
        if (nrec) {
          uint64_t at = 0;
          if (lane == 0) at = atomicAdd(reinterpret_cast<unsigned long long*>(a.rec_count), (unsigned long long)nrec);
          at = __shfl_sync(0xffffffffu, at, 0);
          for (uint32_t s0 = 0; s0 < nsl; s0 += 32) {
            const uint32_t s = s0 + lane;
            const uint64_t w = s < nsl ? res[s] : 0ull;
            const bool emit = w && ends_here(s);
            const unsigned eb = __ballot_sync(0xffffffffu, emit);
            const uint64_t pos = at + __popc(eb & ((1u << lane) - 1u));
            at += __popc(eb);
            if (emit && (int64_t)pos < a.cap_recs) {
              StagedRec r;
              r.cells = w;
              r.face = sm.f[sm.own[s]].face;
              r.block = (uint32_t)sm.bi[s];
              r.rank = (uint32_t)(atomicAdd(reinterpret_cast<unsigned long long*>(a.info + sm.bi[s]),
                                            1ull | (unsigned long long)__popcll(w) << kInfoShift) & kInfoMask);
              r.pad = 0u;
              a.staged[pos] = r;
            }
          }
        }
      }
      __syncwarp();
      if (last_tile) g0 = g1;
    }
    __syncwarp();  // the next faces reuse the records
  }
  unsigned long long v[4] = {wc.fb, wc.band, wc.cand, n_tests};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  }
  if (lane == 0) {
    if (v[0]) atomicAdd(&a.counters[CNT_FALLBACK], v[0]);
    if (v[1]) atomicAdd(&a.counters[CNT_BAND], v[1]);
    if (v[2]) atomicAdd(&a.counters[CNT_FACE_SETUPS], v[2]);
    if (v[3]) atomicAdd(&a.counters[CNT_FACE_TESTS], v[3]);
  }
}

// After the faces have left their records (staged in any order, each with its rank within its block): per block its
// pairs | adjacent cells << 32 for the row scan, and the place of its records, claimed by 1,024 blocks at a time (the
// order does not matter, every block's lists are sorted).  With a scan of the counts instead, counting and row scan
// took 35 us on 0.76 M blocks and 23 on 0.23 M, so 24 and 16 (placing the records 28 and 11, now 31 and 11).
__global__ void __launch_bounds__(1024) k_record_counts(RefineLevel a, uint64_t* first, unsigned long long* placed) {
  __shared__ uint64_t s_warp[32];
  __shared__ uint64_t s_base;
  const int64_t n = launch_count(a.n_blocks, a.n_dev, a.err);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t b0 = blockIdx.x * 1024ll; b0 < n; b0 += gridDim.x * 1024ll) {
    const int64_t b = b0 + threadIdx.x;
    const uint64_t info = b < n ? a.info[b] : 0ull;
    const uint64_t c = info & kInfoMask, incl = warp_inclusive_scan<uint64_t>(c);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      const uint64_t w = s_warp[lane], upto = warp_inclusive_scan<uint64_t>(w);
      s_warp[lane] = upto - w;
      if (lane == 31) s_base = upto ? atomicAdd(placed, (unsigned long long)upto) : 0ull;
    }
    __syncthreads();
    if (b < n) {
      a.blockcnt[b] = info ? (info >> kInfoShift) | ((uint64_t)__popcll(a.mask[b]) << 32) : 0ull;
      first[b] = s_base + s_warp[wid] + incl - c;
    }
    __syncthreads();  // the next blocks reuse the sums
  }
}

// The staged records into their blocks' runs (first[b]: their places), and each block's descriptor; `placed` is zero
// again for the next level.
// More records than were staged (a replay whose capacities were outgrown; the caller runs again with more
// room): the level is left without records, cells and pairs, so that the kernels after this one find nothing
// to read (rows without their offsets would lead the link kernel out of its tables).
__global__ void __launch_bounds__(256) k_place_records(RefineLevel a, const uint64_t* first, unsigned long long* placed,
                                                       uint64_t* level_tot) {
  const int64_t n = (int64_t)*a.rec_count;
  if (blockIdx.x == 0 && threadIdx.x == 0) *placed = 0ull;
  if (n > a.cap_recs) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      *level_tot = 0;
      atomicOr(a.err, ERR_OVERFLOW);
    }
    const int64_t nb = launch_count(a.n_blocks, a.n_dev, a.err);
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x)
      a.rec_desc[b] = 0ull;
    return;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const StagedRec r = a.staged[i];
    const uint64_t at = first[r.block];
    SurvRec o;
    o.face = r.face;
    o.pad = 0u;
    o.cells = r.cells;
    a.recs[at + r.rank] = o;
    if (r.rank == 0) {
      a.rec_desc[r.block] = (at << kInfoShift) | (a.info[r.block] & kInfoMask);
    }
  }
}

// Warps per SM kept resident: 32 (CTAs of `warps` warps).
int grid_warps(int num_sms, int64_t n, int warps, bool persistent) {
  const int64_t cap = (int64_t)num_sms * (32 / warps > 0 ? 32 / warps : 1);
  if (persistent) return (int)cap;
  int64_t need = (n + warps - 1) / warps;
  if (need < 1) need = 1;
  return (int)(need < cap ? need : cap);
}

template <typename K>
void allow_smem(K kernel, size_t bytes) {
  if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

int launch_refine(const RefineLevel& a, int num_sms, cudaStream_t st) {
  if (!a.n_dev && a.n_blocks <= 0) return 0;
  const int warps = a.warps > 0 ? a.warps : 4;
  const int g = grid_warps(num_sms, a.n_blocks, warps, a.n_dev != nullptr);
  const size_t smem = (size_t)warps * (a.dim == 3 ? sizeof(WarpSmem<3>) : sizeof(WarpSmem<2>));
  auto go = [&](auto kernel) {
    allow_smem(kernel, smem);
    kernel<<<g, warps * 32, smem, st>>>(a);
  };
  const int mode = a.search == 1 ? 2 : (a.pred == 1 ? 1 : 0);
  if (refine_by_groups(a.dim, a.level, a.pred, a.search)) {
    // one warp per parent group of 8 children
    const int gg = grid_warps(num_sms, a.n_blocks / 8, kGroupWarps, a.n_dev != nullptr);
    const size_t gsm = (size_t)kGroupWarps * sizeof(GroupSmem);
    allow_smem(k_refine_groups, gsm);
    k_refine_groups<<<gg, kGroupWarps * 32, gsm, st>>>(a);
    return 1;
  }
  // one geometry: every block ends here or none does
  const int ends = mode == 0 ? 2 : (!a.blockcnt ? 0 : (a.table ? 2 : 1));
  auto pick = [&](auto k0, auto g0, auto k1, auto k2, auto g2) {
    ends == 0 ? (a.gather ? go(g0) : go(k0)) : (ends == 1 ? go(k1) : (a.gather ? go(g2) : go(k2)));
  };
  if (a.dim == 3) {
    if (mode == 2)
      pick(k_refine<3, 2, 0, false>, k_refine<3, 2, 0, true>, k_refine<3, 2, 1, false>, k_refine<3, 2, 2, false>,
           k_refine<3, 2, 2, true>);
    else if (mode == 1)
      pick(k_refine<3, 1, 0, false>, k_refine<3, 1, 0, true>, k_refine<3, 1, 1, false>, k_refine<3, 1, 2, false>,
           k_refine<3, 1, 2, true>);
    else
      go(k_refine<3, 0, 2, false>);
  } else {
    if (mode == 2)
      pick(k_refine<2, 2, 0, false>, k_refine<2, 2, 0, true>, k_refine<2, 2, 1, false>, k_refine<2, 2, 2, false>,
           k_refine<2, 2, 2, true>);
    else if (mode == 1)
      pick(k_refine<2, 1, 0, false>, k_refine<2, 1, 0, true>, k_refine<2, 1, 1, false>, k_refine<2, 1, 2, false>,
           k_refine<2, 1, 2, true>);
    else
      go(k_refine<2, 0, 2, false>);
  }
  return 1;
}

int launch_entry_spheres(const void* payload, const uint32_t* n_entries, float4* out, int num_sms, cudaStream_t st) {
  k_entry_spheres<<<num_sms * 8, 256, 0, st>>>(static_cast<const Entry3*>(payload), n_entries, out);
  return 1;
}

int launch_adjacency(const EmitArgs& a, int num_sms, cudaStream_t st) {
  if (!a.lv.n_dev && a.lv.n_blocks <= 0) return 0;
  const int warps = a.lv.warps > 0 ? a.lv.warps : 4;
  const int mode = a.lv.search == 1 ? 2 : (a.lv.pred == 1 ? 1 : 0);
  // first pass: little shared memory, so up to 64 warps per SM
  {
    const int64_t cap = (int64_t)num_sms * (64 / warps > 0 ? 64 / warps : 1);
    int64_t g = a.lv.n_dev ? cap : (a.lv.n_blocks + warps - 1) / warps;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    auto go = [&](auto kernel) { kernel<<<(unsigned)g, warps * 32, 0, st>>>(a); };
    if (a.lv.dim == 3)
      mode == 2 ? go(k_adjacency<3, 2, 0>) : (mode == 1 ? go(k_adjacency<3, 1, 0>) : go(k_adjacency<3, 0, 0>));
    else
      mode == 2 ? go(k_adjacency<2, 2, 0>) : (mode == 1 ? go(k_adjacency<2, 1, 0>) : go(k_adjacency<2, 0, 0>));
  }
  // second pass over the listed blocks (its count on the device): the walk's shared memory
  cudaMemsetAsync(a.lv.work, 0, sizeof(unsigned), st);
  {
    const int g = grid_warps(num_sms, 0, warps, true);
    const size_t smem = (size_t)warps * (a.lv.dim == 3 ? second_pass_bytes<3>() : second_pass_bytes<2>());
    auto go = [&](auto kernel) {
      allow_smem(kernel, smem);
      kernel<<<g, warps * 32, smem, st>>>(a);
    };
    if (a.lv.dim == 3)
      mode == 2 ? go(k_adjacency<3, 2, 1>) : (mode == 1 ? go(k_adjacency<3, 1, 1>) : go(k_adjacency<3, 0, 1>));
    else
      mode == 2 ? go(k_adjacency<2, 2, 1>) : (mode == 1 ? go(k_adjacency<2, 1, 1>) : go(k_adjacency<2, 0, 1>));
  }
  return 2;
}

int launch_mark_faces(const MarkArgs& m, int num_sms, cudaStream_t st) {
  const int64_t nf = m.faces.end - m.faces.begin;
  if (nf <= 0) return 0;
  const bool point = m.lv.pred == 1, multi = m.lv.table != nullptr;
  int k = 0;
  auto go = [&](auto kernel, int batch, int64_t resident, int warps) {
    MarkArgs x = m;
    x.batch = batch;
    const int64_t need = (nf + (int64_t)x.batch * warps - 1) / ((int64_t)x.batch * warps);
    if (k++) cudaMemsetAsync(m.lv.work, 0, sizeof(unsigned), st);
    kernel<<<(unsigned)std::min<int64_t>(need, resident), warps * 32, 0, st>>>(x);
  };
  auto cells = [&](auto kernel) {
    const int64_t grid = (int64_t)num_sms * kCellBlocks;
    go(kernel, m.faces.fetch(grid * kCellWarps, kCellFaces), grid, kCellWarps);
  };
  auto faces = [&](auto kernel) {
    const int64_t few = m.faces.used / ((int64_t)num_sms * 48);  // two fetches for each of 24 warps per SM
    go(kernel, (int)std::max<int64_t>(1, std::min<int64_t>(kFaceBatch, few)), (int64_t)num_sms * 8, kMarkWarps);
  };
  if (m.unit) {
    const bool rec = m.lv.staged != nullptr;
    if (m.lv.dim == 3)
      multi ? (rec ? cells(k_mark_cells<3, true, true>) : cells(k_mark_cells<3, true, false>))
            : (rec ? cells(k_mark_cells<3, false, true>) : cells(k_mark_cells<3, false, false>));
    else
      multi ? cells(k_mark_cells<2, true, false>) : cells(k_mark_cells<2, false, false>);
  }
  if (m.plain) {
    if (m.lv.dim == 3)
      point ? (multi ? faces(k_mark_faces<3, 1, true>) : faces(k_mark_faces<3, 1, false>))
            : (multi ? faces(k_mark_faces<3, 0, true>) : faces(k_mark_faces<3, 0, false>));
    else
      point ? (multi ? faces(k_mark_faces<2, 1, true>) : faces(k_mark_faces<2, 1, false>))
            : (multi ? faces(k_mark_faces<2, 0, true>) : faces(k_mark_faces<2, 0, false>));
  }
  return k;
}

int launch_record_counts(const RefineLevel& a, uint64_t* first, uint64_t* placed, int num_sms, cudaStream_t st) {
  const int64_t g = std::min<int64_t>((a.n_blocks + 1023) / 1024, (int64_t)num_sms * 2);
  k_record_counts<<<(unsigned)std::max<int64_t>(1, g), 1024, 0, st>>>(a, first,
                                                                      reinterpret_cast<unsigned long long*>(placed));
  return 1;
}

int launch_place_records(const RefineLevel& a, const uint64_t* first, uint64_t* placed, uint64_t* level_tot,
                         int num_sms, cudaStream_t st) {
  const int64_t g = std::min<int64_t>((a.cap_recs + 255) / 256, (int64_t)num_sms * 8);
  k_place_records<<<(unsigned)std::max<int64_t>(1, g), 256, 0, st>>>(
      a, first, reinterpret_cast<unsigned long long*>(placed), level_tot);
  return 1;
}

size_t children_scratch_bytes(int64_t n) {
  const int64_t tiles = (n + (int64_t)kChThreads * kChItems - 1) / ((int64_t)kChThreads * kChItems);
  return 16 + (size_t)(tiles > 0 ? tiles : 1) * 8;
}

int launch_children(const ChildrenArgs& a, void* scratch, int num_sms, cudaStream_t st) {
  cudaMemsetAsync(scratch, 0, children_scratch_bytes(a.n), st);
  int64_t tiles = (a.n + (int64_t)kChThreads * kChItems - 1) / ((int64_t)kChThreads * kChItems);
  if (tiles < 1) tiles = 1;
  if (a.n_dev && tiles > (int64_t)num_sms * 4) tiles = (int64_t)num_sms * 4;
  unsigned* ticket = reinterpret_cast<unsigned*>(scratch);
  uint64_t* state = reinterpret_cast<uint64_t*>(static_cast<char*>(scratch) + 16);
  if (a.dim == 3)
    k_children<3><<<(unsigned)tiles, kChThreads, 0, st>>>(a, state, ticket);
  else
    k_children<2><<<(unsigned)tiles, kChThreads, 0, st>>>(a, state, ticket);
  return 1;
}

}  // namespace amr
