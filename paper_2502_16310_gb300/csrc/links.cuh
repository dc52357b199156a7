// links.cuh — the FP64 definition of a D3Q19 link's crossing of a face, shared by the link kernels.
#pragma once

#include "internal.cuh"

namespace amr {

namespace {

__device__ __forceinline__ void d3q19_dir(int i, int& cx, int& cy, int& cz) {
  cx = d3q19_c(i, 0);
  cy = d3q19_c(i, 1);
  cz = d3q19_c(i, 2);
}

struct LinkHit {
  bool hit;
  bool band;
  double t;
};

__device__ __noinline__ LinkHit link_fp64_3(const float* V, const double* xc, const int* ci, double h);

// FP64 evaluation of direction di for the cell (block coordinates blk3, cell bit),
// with the cell centre formed in FP64 (the slow path of undecided signs).
__device__ __noinline__ LinkHit link_fallback_3(const float* V, const int* blk3, uint32_t bit, const double* origin,
                                                double h, int di) {
  int ci[3];
  d3q19_dir(di, ci[0], ci[1], ci[2]);
  double xc[3];
  for (int c = 0; c < 3; ++c) {
    const int gc = 4 * blk3[c] + (int)((bit >> (2 * c)) & 3u);
    xc[c] = __dadd_rn(origin[c], __dmul_rn((double)gc + 0.5, h));
  }
  return link_fp64_3(V, xc, ci, h);
}

// FP64 evaluation of one (link, face) pair, same definition as the FP32 path.
__device__ __noinline__ LinkHit link_fp64_3(const float* V, const double* xc, const int* ci, double h) {
  LinkHit r{false, false, 0.0};
  double p[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) p[k][c] = (double)V[3 * k + c] - xc[c];
  const double d[3] = {ci[0] * h, ci[1] * h, ci[2] * h};
  const double u[3] = {p[1][0] - p[0][0], p[1][1] - p[0][1], p[1][2] - p[0][2]};
  const double w[3] = {p[2][0] - p[0][0], p[2][1] - p[0][1], p[2][2] - p[0][2]};
  const double n[3] = {u[1] * w[2] - u[2] * w[1], u[2] * w[0] - u[0] * w[2], u[0] * w[1] - u[1] * w[0]};
  const double ln = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
  if (ln == 0.0) return r;
  const double den = d[0] * n[0] + d[1] * n[1] + d[2] * n[2];
  if (den == 0.0) return r;
  const double ld = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
  if (fabs(den) <= kBandRel * ld * ln) r.band = true;
  auto vol = [&](const double* a, const double* b) {
    const double c0 = a[1] * b[2] - a[2] * b[1], c1 = a[2] * b[0] - a[0] * b[2], c2 = a[0] * b[1] - a[1] * b[0];
    return d[0] * c0 + d[1] * c1 + d[2] * c2;
  };
  const double l0 = vol(p[1], p[2]) / den, l1 = vol(p[2], p[0]) / den, l2 = vol(p[0], p[1]) / den;
  const double t = (p[0][0] * n[0] + p[0][1] * n[1] + p[0][2] * n[2]) / den;
  const double mu = fmin(fmin(fmin(l0, l1), l2), fmin(t, 1.0 - t));
  if (fabs(mu) <= kBandRel) r.band = true;
  r.hit = mu >= 0.0;
  r.t = t;
  return r;
}

// One link of one (cell, face) pair with k_links' tests and arithmetic: -1 no hit, 1 hit (q), 2 undecided
// in FP32 (FP64 decides).  R: the face's record; x: the cell.
__device__ __noinline__ int link_pair_3(const FaceRec3* R, const int* x, const GeomParams& P, float h_hi, float h_lo,
                                        int di, float* q) {
  const float4* r = reinterpret_cast<const float4*>(R);
  const float4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3);
  const float V[9] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x};
  const float nh[3] = {r2.y, r2.z, r2.w}, nl[3] = {r3.x, r3.y, r3.z};
  float p[3][3], ph0[3], pl0[3], pmax = 0.f, xmax = 0.f;
  for (int c = 0; c < 3; ++c) {
    float ohi, olo;
    df_position(P.org_hi[c], P.org_lo[c], (float)(2 * x[c] + 1), 0.5f * h_hi, 0.5f * h_lo, ohi, olo);
    xmax = fmaxf(xmax, fabsf(ohi));
    for (int k = 0; k < 3; ++k) {
      float s, e;
      df_two_sum(V[3 * k + c], -ohi, s, e);
      const float l = e - olo;
      if (k == 0) {
        ph0[c] = s;
        pl0[c] = l;
      }
      p[k][c] = s + l;
      pmax = fmaxf(pmax, fabsf(p[k][c]));
    }
  }
  float ns, ne;
  df_two_prod(nh[0], ph0[0], ns, ne);
  for (int c = 1; c < 3; ++c) {
    float pp, pe, s, t;
    df_two_prod(nh[c], ph0[c], pp, pe);
    df_two_sum(ns, pp, s, t);
    ns = s;
    ne += t + pe;
  }
  const float n1 = fabsf(nh[0]) + fabsf(nh[1]) + fabsf(nh[2]);
  for (int c = 0; c < 3; ++c) ne = fmaf(nh[c], pl0[c], fmaf(nl[c], ph0[c], ne));
  const float num = ns + ne;
  const float eps_num = 16.0f * kU32 * kU32 * n1 * (xmax + pmax) + 4.0f * kU32 * fabsf(ne);
  const float nn2 = sqrtf(nh[0] * nh[0] + nh[1] * nh[1] + nh[2] * nh[2]);
  const float cx = dir_comp(kDirX, di), cy = dir_comp(kDirY, di), cz = dir_comp(kDirZ, di);
  const float cl = fabsf(cx) + fabsf(cy) + fabsf(cz);
  {
    // the line's reach of the plane, and on which side
    const float D = cx * nh[0] + cy * nh[1] + cz * nh[2];
    const float eD = 4.0f * kU32 * (fabsf(cx * nh[0]) + fabsf(cy * nh[1]) + fabsf(cz * nh[2]));
    const float reach = h_hi * (fabsf(D) + eD) * (1.0f + 16.0f * kU32);
    if (fabsf(num) - eps_num > reach) return -1;
    if (!((num >= -eps_num && D >= -eD) || (num <= eps_num && D <= eD))) return -1;
  }
  float s1, e1, dh, e2;
  df_two_sum(cx * nh[0], cy * nh[1], s1, e1);
  df_two_sum(s1, cz * nh[2], dh, e2);
  const float den = dh + ((e1 + e2) + (cx * nl[0] + cy * nl[1] + cz * nl[2]));
  if (den == 0.0f && dh == 0.0f) return -1;
  const float ad = fabsf(den), sg = den > 0.f ? 1.f : -1.f;
  const bool unc = ad <= (cl == 1.0f ? 1e-5f : 1.41421356e-5f) * nn2;
  const float sn = sg * num, hd = h_hi * ad;
  if (!unc && (sn < -eps_num || sn - eps_num > hd * (1.0f + 8.0f * kU32))) return -1;
  bool out = false, all_in = true;
  for (int k = 0; k < 3; ++k) {
    const float* A = p[(k + 1) % 3];
    const float* B = p[(k + 2) % 3];
    const float C0 = fmaf(A[1], B[2], -A[2] * B[1]), C1 = fmaf(A[2], B[0], -A[0] * B[2]),
                C2 = fmaf(A[0], B[1], -A[1] * B[0]);
    const float M = fmaxf(fmaxf(fabsf(A[1] * B[2]) + fabsf(A[2] * B[1]), fabsf(A[2] * B[0]) + fabsf(A[0] * B[2])),
                          fabsf(A[0] * B[1]) + fabsf(A[1] * B[0]));
    const float u = sg * (cx * C0 + cy * C1 + cz * C2), eu = 8.0f * kU32 * cl * M;
    if (u < -eu) out = true;
    if (!(u > eu)) all_in = false;
  }
  if (out && !unc) return -1;
  if (!unc && all_in && sn > eps_num && sn + eps_num < hd * (1.0f - 8.0f * kU32)) {
    *q = num / (h_hi * den);
    return 1;
  }
  return 2;
}

}  // namespace

}  // namespace amr
