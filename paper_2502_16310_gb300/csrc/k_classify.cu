// k_classify.cu — node classification of the finest adjacent cells and the
// restriction of the wall links to fluid nodes.
//
// Paper (Sec. "Conclusions": node classification is the next step towards the
// boundary conditions of the LBM): a node is solid when it lies inside the closed
// boundary mesh.  Each adjacent cell casts a ray from its centre along +x
// through its own row of bins and counts the faces the ray crosses: odd = solid
// (a closed mesh, any orientation).  A face is counted once, in the first of its
// bins along the walked row.  A face whose yz bounding box certainly misses the
// ray is skipped in FP32; the others are tested (point in the projected
// triangle, crossing beyond the centre), in FP64 where FP32 is not certain.  A ray that passes exactly through an
// edge or a vertex, or a crossing at the centre itself, is not decided by the
// crossing count: such a cell is classified by the generalized winding number
// of the whole mesh (sum of the signed solid angles / 4 pi; 2D: angles / 2 pi),
// |w| > 1/2 = solid, and counted.
#include "internal.cuh"

namespace amr {

namespace {

constexpr int kCThreads = 128;

// 0 = no crossing, 1 = crossing beyond the centre, 2 = undecided
template <int D>
__device__ int ray_cross(const float* v, const double* p) {
  if constexpr (D == 2) {
    // segment a-b against the ray y = p.y, x > p.x; the half-open rule (lower end in,
    // upper end out) counts a ray through a shared vertex exactly once
    const double ay = v[1], by = v[3];
    if (!((ay <= p[1] && p[1] < by) || (by <= p[1] && p[1] < ay))) return 0;
    const double ax = v[0], bx = v[2];
    const double t = __ddiv_rn(__dsub_rn(p[1], ay), __dsub_rn(by, ay));
    const double xh = __fma_rn(t, __dsub_rn(bx, ax), ax);
    if (fabs(xh - p[0]) <= 1e-12 * (fabs(xh) + fabs(p[0]))) return 2;  // the centre on the segment
    return xh > p[0] ? 1 : 0;
  } else {
    // projection onto the yz plane: edge functions of (p.y, p.z), each with a bound on
    // its rounding error; a sign within that bound is not decided
    constexpr double u64 = 1.1102230246251565e-16;
    double e[3];
    bool tie = false;
    for (int k = 0; k < 3; ++k) {
      const int k1 = (k + 1) % 3;
      const double ay = v[3 * k + 1], az = v[3 * k + 2], by = v[3 * k1 + 1], bz = v[3 * k1 + 2];
      const double t1 = __dmul_rn(__dsub_rn(by, ay), __dsub_rn(p[2], az));
      const double t2 = __dmul_rn(__dsub_rn(bz, az), __dsub_rn(p[1], ay));
      e[k] = __dsub_rn(t1, t2);
      if (fabs(e[k]) <= 8.0 * u64 * (fabs(t1) + fabs(t2))) tie = true;
    }
    if (tie) {
      // decided only when another edge function certainly puts the point outside
      const bool out = (e[0] > 0.0 || e[1] > 0.0 || e[2] > 0.0) && (e[0] < 0.0 || e[1] < 0.0 || e[2] < 0.0);
      return out ? 0 : 2;
    }
    const bool pos = e[0] > 0.0 && e[1] > 0.0 && e[2] > 0.0;
    const bool neg = e[0] < 0.0 && e[1] < 0.0 && e[2] < 0.0;
    if (!pos && !neg) {
      // outside unless an edge function is zero while the others agree in sign
      const bool maybe = (e[0] >= 0.0 && e[1] >= 0.0 && e[2] >= 0.0) || (e[0] <= 0.0 && e[1] <= 0.0 && e[2] <= 0.0);
      return maybe ? 2 : 0;
    }
    // crossing point: x on the face plane at (p.y, p.z), by barycentric weights e_k / sum
    const double s = __dadd_rn(__dadd_rn(e[0], e[1]), e[2]);
    const double xh = (e[1] * (double)v[0] + e[2] * (double)v[3] + e[0] * (double)v[6]) / s;
    if (fabs(xh - p[0]) <= 1e-12 * (fabs(xh) + fabs(p[0]))) return 2;  // the centre on the face
    return xh > p[0] ? 1 : 0;
  }
}

// Signed solid angle of face f seen from p (2D: angle).
template <int D>
__device__ double face_angle(const float* X, int64_t nf, int64_t f, const double* p) {
  if constexpr (D == 2) {
    const double a0 = (double)X[f] - p[0], a1 = (double)X[nf + f] - p[1];
    const double b0 = (double)X[2 * nf + f] - p[0], b1 = (double)X[3 * nf + f] - p[1];
    return atan2(a0 * b1 - a1 * b0, a0 * b0 + a1 * b1);
  } else {
    double a[3], b[3], c[3];
    for (int k = 0; k < 3; ++k) {
      a[k] = (double)X[(int64_t)k * nf + f] - p[k];
      b[k] = (double)X[(int64_t)(3 + k) * nf + f] - p[k];
      c[k] = (double)X[(int64_t)(6 + k) * nf + f] - p[k];
    }
    const double la = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
    const double lb = sqrt(b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
    const double lc = sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
    const double det = a[0] * (b[1] * c[2] - b[2] * c[1]) - a[1] * (b[0] * c[2] - b[2] * c[0]) +
                       a[2] * (b[0] * c[1] - b[1] * c[0]);
    const double ab = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
    const double ac = a[0] * c[0] + a[1] * c[1] + a[2] * c[2];
    const double bc = b[0] * c[0] + b[1] * c[1] + b[2] * c[2];
    return 2.0 * atan2(det, la * lb * lc + ab * lc + ac * lb + bc * la);
  }
}

// The generalized winding number of the whole mesh around p is beyond 1/2 (whole warp, a share of the faces
// per lane, the shares added by a fixed tree).
template <int D>
__device__ __noinline__ bool winding_solid(const float* X, int64_t nf, double p0, double p1, double p2) {
  const double p[3] = {p0, p1, p2};
  double w = 0.0;
  for (int64_t f = threadIdx.x & 31; f < nf; f += 32) w += face_angle<D>(X, nf, f, p);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
  const double pi = 3.14159265358979323846;
  return fabs(D == 2 ? w / (2.0 * pi) : w / (4.0 * pi)) > 0.5;
}

// 2D: a thread per adjacent cell walks the bins of its ray.
__global__ void __launch_bounds__(kCThreads) k_classify_2(ClassifyArgs a) {
  const Entry2* payload = static_cast<const Entry2*>(a.payload);
  unsigned long long n_fb = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // warp-uniform trip count: undecided cells go to the whole warp
  for (int64_t r0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); r0 < a.n_rows; r0 += stride) {
    const int64_t row = r0 + (threadIdx.x & 31);
    double p[3] = {0, 0, 0};
    uint32_t cross = 0;
    bool undecided = false;
    if (row < a.n_rows) {
      const uint32_t id = a.adj_cell[a.row0 + row];
      const uint32_t blk = id / 16, bit = id % 16;
      const GeomParams& P = a.g0;
      const double hL = scalbn(P.h0, -a.level);
      int cb[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int gc = 4 * a.blocks[(int64_t)blk * 2 + c] + (int)((bit >> (2 * c)) & 3u);
        p[c] = __dadd_rn(P.origin[c], __dmul_rn((double)gc + 0.5, hL));
        cb[c] = bin_coord(p[c], P.origin[c], P.bin_scale[c], P.B);
      }
      const float py = (float)p[1], tol = 1e-6f * (fabsf(py) + 1.0f);
      for (int xb = cb[0]; xb < P.B && !undecided; ++xb) {
        const int64_t bin = P.bin_base + xb + (int64_t)P.B * cb[1];
        const uint32_t j1 = a.offsets[bin + 1];
        for (uint32_t j = a.offsets[bin]; j < j1; ++j) {
          const Entry2& ent = payload[j];
          // count each face once: in its first bin of the walked row
          if (!(((ent.id >> 29) & 1u) || (int)ent.bin[0] == cb[0])) continue;
          const float v[4] = {ent.v[0], ent.v[1], ent.v[2], ent.v[3]};
          // the y range certainly misses the ray
          if (py < fminf(v[1], v[3]) - tol || py > fmaxf(v[1], v[3]) + tol) continue;
          const int r = ray_cross<2>(v, p);
          if (r == 2) {
            undecided = true;
            break;
          }
          cross += (uint32_t)r;
        }
      }
    }
    bool solid = (cross & 1u) != 0;
    for (unsigned ub = __ballot_sync(0xffffffffu, undecided); ub; ub &= ub - 1) {
      const int src = __ffs(ub) - 1;
      const bool s = winding_solid<2>(a.X, a.nf, __shfl_sync(0xffffffffu, p[0], src), __shfl_sync(0xffffffffu, p[1], src), 0.0);
      if ((int)(threadIdx.x & 31) == src) {
        solid = s;
        ++n_fb;
      }
    }
    if (row < a.n_rows) a.cls[a.row0 + row] = solid ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n_fb += __shfl_xor_sync(0xffffffffu, n_fb, o);
  if ((threadIdx.x & 31) == 0 && n_fb) atomicAdd(&a.counters[CNT_CLASS_FALLBACK], n_fb);
}

// 3D: a warp per block with adjacent cells.  The block's 4 x 4 lines of cells along x share their rays, and
// each (y, z) row of bins is one run of payload entries, so the warp loads the run 32 entries at a time, keeps
// those whose yz box comes near the block's rays, and tests them against the 16 rays (two entries at once,
// half a warp each).  A crossing toggles the cells of its line that lie before it.
//
// An entry counts for a cell as it did when the cell walked alone: from the cell's own bin on, once per face
// (its first bin, or the cell's own).  The test is FP32 on offsets from the ray with error bounds that cover
// the FP64 test's own thresholds, so what it decides FP64 decides alike; the rest is decided in FP64.
//
// Bound by the walk of the runs.  A thread per cell, all in FP64, took 4.37 ms for 3.7 M cells of a sphere of
// 20 K triangles; now 0.24 ms.
constexpr int kKWarps = 4;       // warps per CTA
struct RayEntry {
  float v[9];
  float lo1, hi1, lo2, hi2;      // yz box
  uint32_t cells;                // cells along the line that it counts for
};

__global__ void __launch_bounds__(kKWarps * 32) k_classify_3(ClassifyArgs a) {
  __shared__ RayEntry s_ent[kKWarps][32];
  const Entry3* payload = static_cast<const Entry3*>(a.payload);
  const int lane = threadIdx.x & 31, ray = lane & 15, half = lane >> 4;
  RayEntry* ents = s_ent[threadIdx.x >> 5];
  const GeomParams& P = a.g0;
  const double hL = scalbn(P.h0, -a.level);
  const FastGeom g = fast_geom(P, a.level);
  const float h = g.h_hi;
  const int64_t nw = (int64_t)gridDim.x * kKWarps;
  for (int64_t blk = (int64_t)blockIdx.x * kKWarps + (threadIdx.x >> 5); blk < a.n_blocks; blk += nw) {
    const uint64_t mask = a.mask[blk];
    if (mask == 0) continue;
    const uint64_t row0 = a.block_base[blk] >> 32;
    int b[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) b[c] = a.blocks[blk * 3 + c];
    auto centre = [&](int c, int i) { return __dadd_rn(P.origin[c], __dmul_rn((double)(4 * b[c] + i) + 0.5, hL)); };
    // the same centre as FP32 hi + lo, and its bin: FP32 where that is certain (FP64 for every block's lanes
    // had the kernel wait for the FP64 pipe 80% of its time, 0.40 ms)
    auto split = [&](int c, int i, float& hi, float& lo) {
      df_position(P.org_hi[c], P.org_lo[c], (float)(2 * (4 * b[c] + i) + 1), 0.5f * g.h_hi, 0.5f * g.h_lo, hi, lo);
    };
    auto bin_of = [&](int c, int i) {
      float hi, lo;
      split(c, i, hi, lo);
      const float t = (((hi - P.org_hi[c]) - P.org_lo[c]) + lo) * P.scale32[c], k = floorf(t);
      const float err = 8.0f * kU32 * (fabsf(hi) + fabsf(P.org_hi[c])) * fabsf(P.scale32[c]);
      if (t - k > err && (k + 1.0f) - t > err) return k < 0.f ? 0 : (k > (float)(P.B - 1) ? P.B - 1 : (int)k);
      return bin_coord(centre(c, i), P.origin[c], P.bin_scale[c], P.B);
    };
    float pxh, pxl, pyh, pyl, pzh, pzl;
    split(0, 0, pxh, pxl);
    split(1, ray & 3, pyh, pyl);
    split(2, ray >> 2, pzh, pzl);
    const int yb = bin_of(1, ray & 3), zb = bin_of(2, ray >> 2);
    // bins of the line's cells along x (lane i < 4: cell i), and of the rays' ends
    const int my_xb = bin_of(0, lane & 3);
    int xb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) xb[i] = __shfl_sync(0xffffffffu, my_xb, i);
    const float by0 = __shfl_sync(0xffffffffu, pyh, 0), by1 = __shfl_sync(0xffffffffu, pyh, 3);
    const float bz0 = __shfl_sync(0xffffffffu, pzh, 0), bz1 = __shfl_sync(0xffffffffu, pzh, 12);
    const float tol = 1e-6f * (fmaxf(fabsf(by0), fabsf(by1)) + fmaxf(fabsf(bz0), fabsf(bz1)) + 1.0f);
    const float d0 = 5.7e-14f * (fabsf(pyh) + fabsf(pzh) + fabsf(P.org_hi[1]) + fabsf(P.org_hi[2]));  // 2^-44: hi + lo
    uint32_t solid = 0, open = 0;  // of the lane's line, from its half of the entries: parity, undecided
    // the rows of bins that hold a ray, each once (where bins are finer than cells, most rows between them hold none:
    // 180 faces on 16^3 cells, 128^3 bins 0.69 ms with all rows walked, now 0.07)
    int zp = -1;
#pragma unroll 1
    for (int iz = 0; iz < 4; ++iz) {
      const int z = __shfl_sync(0xffffffffu, zb, 4 * iz);
      if (z == zp) continue;
      zp = z;
      int yp = -1;
#pragma unroll 1
      for (int iy = 0; iy < 4; ++iy) {
        const int y = __shfl_sync(0xffffffffu, yb, iy);
        if (y == yp) continue;
        yp = y;
        const int64_t bin = P.bin_base + (int64_t)P.B * (y + (int64_t)P.B * z);
        const uint32_t j0 = a.offsets[bin + xb[0]], j1 = a.offsets[bin + P.B];
        const bool mine = yb == y && zb == z;  // the lane's ray lies in this row of bins
        for (uint32_t jj = j0; jj < j1; jj += 32) {
          bool near = false;
          if (jj + lane < j1) {
            const float4* q = reinterpret_cast<const float4*>(payload + jj + lane);
            const float4 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3);
            RayEntry e;
            e.v[0] = q0.x, e.v[1] = q0.y, e.v[2] = q0.z, e.v[3] = q0.w, e.v[4] = q1.x;
            e.v[5] = q1.y, e.v[6] = q1.z, e.v[7] = q1.w, e.v[8] = q2.x;
            e.lo1 = fminf(fminf(e.v[1], e.v[4]), e.v[7]), e.hi1 = fmaxf(fmaxf(e.v[1], e.v[4]), e.v[7]);
            e.lo2 = fminf(fminf(e.v[2], e.v[5]), e.v[8]), e.hi2 = fmaxf(fmaxf(e.v[2], e.v[5]), e.v[8]);
            const bool first = (__float_as_uint(q3.x) >> 29) & 1u;  // the face's first bin along x
            const int x = (int)__float_as_uint(q3.y);
            e.cells = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (xb[i] == x || (first && xb[i] < x)) e.cells |= 1u << i;
            near = e.cells && by1 >= e.lo1 - tol && by0 <= e.hi1 + tol && bz1 >= e.lo2 - tol && bz0 <= e.hi2 + tol;
            if (near) ents[lane] = e;
          }
          unsigned nb = __ballot_sync(0xffffffffu, near);
          __syncwarp();
          while (nb) {
            const int e0 = __ffs(nb) - 1;
            nb &= nb - 1;
            const int e1 = nb ? __ffs(nb) - 1 : -1;
            nb &= nb - 1;
            const int ei = half ? e1 : e0;
            if (ei < 0 || !mine) continue;
            const RayEntry& E = ents[ei];
            if (pyh < E.lo1 - tol || pyh > E.hi1 + tol || pzh < E.lo2 - tol || pzh > E.hi2 + tol) continue;
            // offsets from the ray; the edge functions of its point in the yz projection
            float ey[3], ez[3], ex[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              ex[k] = (E.v[3 * k] - pxh) - pxl;
              ey[k] = (E.v[3 * k + 1] - pyh) - pyl;
              ez[k] = (E.v[3 * k + 2] - pzh) - pzl;
            }
            float u[3], err[3];
            bool pos = true, neg = true, some_pos = false, some_neg = false;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const int k1 = (k + 1) % 3;
              const float t1 = ey[k] * ez[k1], t2 = ez[k] * ey[k1];
              u[k] = t1 - t2;
              const float ay = fabsf(ey[k]) + fabsf(ey[k1]), az = fabsf(ez[k]) + fabsf(ez[k1]);
              err[k] = 8.0f * kU32 * (fabsf(t1) + fabsf(t2)) + 2.0f * d0 * (ay + az) + 4e-15f * ay * az;
              pos = pos && u[k] > err[k];
              neg = neg && u[k] < -err[k];
              some_pos = some_pos || u[k] > err[k];
              some_neg = some_neg || u[k] < -err[k];
            }
            if (some_pos && some_neg) continue;  // certainly outside
            uint32_t todo = E.cells;             // cells left to FP64
            if (pos || neg) {
              const float s = u[0] + u[1] + u[2];
              const float xr = (u[1] * ex[0] + u[2] * ex[1] + u[0] * ex[2]) / s;  // crossing from cell 0's centre
              const float X = fmaxf(fmaxf(fabsf(ex[0]), fabsf(ex[1])), fabsf(ex[2]));
              const float eb = 2.0f * (err[0] + err[1] + err[2]) * X / fabsf(s) + 16.0f * kU32 * (X + 3.0f * h) +
                               4e-12f * (fabsf(pxh) + fabsf(P.org_hi[0]) + X + 3.0f * h);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float d = xr - (float)i * h;
                if (((todo >> i) & 1u) && fabsf(d) > eb) {
                  solid ^= d > 0.f ? 1u << i : 0u;
                  todo &= ~(1u << i);
                }
              }
            }
            for (; todo; todo &= todo - 1) {
              const int i = __ffs(todo) - 1;
              const double p[3] = {centre(0, i), centre(1, ray & 3), centre(2, ray >> 2)};
              const int r = ray_cross<3>(E.v, p);
              if (r == 2) open |= 1u << i;
              if (r == 1) solid ^= 1u << i;
            }
          }
          __syncwarp();  // the next entries reuse the places
        }
      }
    }
    solid ^= __shfl_xor_sync(0xffffffffu, solid, 16);
    open |= __shfl_xor_sync(0xffffffffu, open, 16);
    // the lane's half of its line: cells 2 half and 2 half + 1
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = 2 * half + k, cell = i | (ray << 2);
      const bool adj = (mask >> cell) & 1ull;
      bool in = (solid >> i) & 1u;
      const uint64_t row = row0 + __popcll(mask & ((1ull << cell) - 1ull));
      const bool undecided = adj && ((open >> i) & 1u);
      const unsigned ob = __ballot_sync(0xffffffffu, undecided);
      unsigned late = 0;  // beyond the list's room: by this warp, at once
      if (ob) {
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&a.counters[CNT_CLASS_FALLBACK], (unsigned long long)__popc(ob));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(ob & ((1u << lane) - 1u));
        if (undecided && (int64_t)at < a.open_cap) a.open_rows[at] = (uint32_t)row;
        late = __ballot_sync(0xffffffffu, undecided && (int64_t)at >= a.open_cap);
      }
      for (unsigned ub = late; ub; ub &= ub - 1) {
        const int src = __ffs(ub) - 1;
        const int ci = 2 * (src >> 4) + k, r = src & 15;
        const bool w = winding_solid<3>(a.X, a.nf, centre(0, ci), centre(1, r & 3), centre(2, r >> 2));
        if (lane == src) in = w;
      }
      if (adj) a.cls[row] = in ? 1 : 0;  // (a listed cell's is settled by k_classify_open)
    }
  }
}

// 3D: the cells whose rays met an edge, a warp each, by the winding number.  They come in clusters (a mesh on cell
// planes has them in whole blocks), so deciding them where they were found left most warps idle: 6,964 such cells on
// a box of 17,328 faces 79 ms by a thread per cell, 115 by the warp of the block, now 30.
__global__ void __launch_bounds__(kKWarps * 32) k_classify_open(ClassifyArgs a) {
  const int lane = threadIdx.x & 31;
  const GeomParams& P = a.g0;
  const double hL = scalbn(P.h0, -a.level);
  const int64_t listed = (int64_t)a.counters[CNT_CLASS_FALLBACK], n = listed < a.open_cap ? listed : a.open_cap;
  for (int64_t i = (int64_t)blockIdx.x * kKWarps + (threadIdx.x >> 5); i < n; i += (int64_t)gridDim.x * kKWarps) {
    const uint32_t row = a.open_rows[i], id = a.adj_cell[row];
    double p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      p[c] = __dadd_rn(P.origin[c], __dmul_rn((double)(4 * a.blocks[(int64_t)(id / 64) * 3 + c] +
                                                       (int)((id >> (2 * c)) & 3u)) + 0.5, hL));
    const bool in = winding_solid<3>(a.X, a.nf, p[0], p[1], p[2]);
    if (lane == 0) a.cls[row] = in ? 1 : 0;
  }
}

// Stable compaction of the links to those whose cell is fluid: keep flags and
// the per-block counts, then a scan gives the positions.
constexpr int kFThreads = 256;

__global__ void k_fluid_count(const uint32_t* link_cell, const uint8_t* cls, int64_t n, uint32_t* cnt) {
  __shared__ uint32_t s;
  if (threadIdx.x == 0) s = 0;
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)kFThreads + threadIdx.x;
  const bool keep = i < n && cls[link_cell[i]] == 0;
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(&s, (uint32_t)__popc(m));
  __syncthreads();
  if (threadIdx.x == 0) cnt[blockIdx.x] = s;
}

__global__ void k_fluid_move(const uint32_t* link_cell, const uint8_t* link_dir, const float* link_q,
                             const uint32_t* link_face, const uint8_t* cls, int64_t n, const uint32_t* base,
                             uint32_t* o_cell, uint8_t* o_dir, float* o_q, uint32_t* o_face) {
  __shared__ uint32_t s_warp[kFThreads / 32];
  const int64_t i = blockIdx.x * (int64_t)kFThreads + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool keep = i < n && cls[link_cell[i]] == 0;
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if (lane == 0) s_warp[wid] = (uint32_t)__popc(m);
  __syncthreads();
  uint32_t off = base[blockIdx.x];
  for (int w = 0; w < wid; ++w) off += s_warp[w];
  if (keep) {
    const uint32_t pos = off + (uint32_t)__popc(m & ((1u << lane) - 1u));
    o_cell[pos] = link_cell[i];
    o_dir[pos] = link_dir[i];
    o_q[pos] = link_q[i];
    o_face[pos] = link_face[i];
  }
}

}  // namespace

int launch_classify(const ClassifyArgs& a, cudaStream_t st) {
  if (a.n_rows <= 0) return 0;
  const int sms = current_sm_count();
  if (a.dim == 3) {
    const int64_t need = (a.n_blocks + kKWarps - 1) / kKWarps, cap = (int64_t)sms * 16;
    k_classify_3<<<(unsigned)(need < cap ? need : cap), kKWarps * 32, 0, st>>>(a);
    k_classify_open<<<(unsigned)(sms * 8), kKWarps * 32, 0, st>>>(a);
    return 2;
  }
  const int64_t need = (a.n_rows + kCThreads - 1) / kCThreads, cap = (int64_t)sms * 16;
  k_classify_2<<<(unsigned)(need < cap ? need : cap), kCThreads, 0, st>>>(a);
  return 1;
}

int64_t fluid_blocks(int64_t n) { return (n + kFThreads - 1) / kFThreads; }

int launch_fluid_count(const uint32_t* link_cell, const uint8_t* cls, int64_t n, uint32_t* cnt, cudaStream_t st) {
  if (n <= 0) return 0;
  k_fluid_count<<<(unsigned)fluid_blocks(n), kFThreads, 0, st>>>(link_cell, cls, n, cnt);
  return 1;
}

int launch_fluid_move(const uint32_t* link_cell, const uint8_t* link_dir, const float* link_q,
                      const uint32_t* link_face, const uint8_t* cls, int64_t n, const uint32_t* base,
                      uint32_t* o_cell, uint8_t* o_dir, float* o_q, uint32_t* o_face, cudaStream_t st) {
  if (n <= 0) return 0;
  k_fluid_move<<<(unsigned)fluid_blocks(n), kFThreads, 0, st>>>(link_cell, link_dir, link_q, link_face, cls, n, base,
                                                                o_cell, o_dir, o_q, o_face);
  return 1;
}

}  // namespace amr
