// k_flinks.cu — wall links found from the faces: a 3D level below the roots, either predicate, any d that puts every
// face a link can cross into its cell's list (0.5 h; point predicate sqrt(2) h), faces up to 26 cells wide.
//
// A lattice line (a row of cell centres along one of the 9 lines of D3Q19) that crosses a face at one
// point gives at most two links of the face: the cell before the point links forward across it with
// q = t, the cell after it backward.  So a face needs the lattice lines inside its projection along each
// of the 9 directions and two plane offsets per crossing, where the pair-by-pair kernel (k_links.cu)
// tests 9 lines for each of the face's 340 adjacent cells.  A cell whose link meets a face is adjacent
// to it, so no list is needed.
//
//   k_face_links    up to 3 faces of a warp together.  A lane per (face, direction): the projection; a
//                   lane per row of lines: the part inside it; a lane per line: the three edge functions
//                   (2D cross products with an error bound) and, inside, the offsets of the two cells
//                   around the crossing, in double-float with k_links' operations.  What is not
//                   certified goes through that kernel's test of each pair around it, so the links and
//                   every bit of q are the same.  Hits are gathered in shared memory and leave as runs,
//                   one per (face, group), a group being the 8 consecutive blocks of one parent.
//   k_place_runs    the runs' descriptors by group (their counts scanned).
//   k_count_links   per group the links it has (several faces may meet one link), for the output's scan.
//   k_write_links   per group: every hit to its place in (cell, direction) order, the least (t, face)
//                   where faces compete, through shared memory so that the output is written in runs.
//
// Bound by instructions (about 700 warp instructions per 32 links in all, 400 of them in k_face_links, at 16
// warps per SM) and by the latency of the group kernels' loads.  465 M links of 1.3 M faces: 24.2 ms by pairs,
// 14.9 here; 31.5 M of 82 K: 1.61, 1.19; 9.5 M of 20 K: 0.49, 0.45.  k_write_links with a word less per cell, so
// that 8 CTAs fit an SM instead of 6: 1.25 -> 1.19 (1.28 at 7).
// Direction by direction over 16 faces, the hits of a (face, group) left in pieces: 19.7 and 1.54 ms;
// each cell's position worked out per crossing instead of taken from a table: 1.54.  At 5 blocks per SM
// (96 registers, spills) 16.7 and 1.34 ms.
#include <algorithm>

#include "links.cuh"

namespace amr {

namespace {

constexpr int kFWarps = 4;       // warps per CTA of k_face_links
constexpr int kFBlocks = 4;      // CTAs per SM
constexpr int kFFaces = 8;       // faces a warp takes per work fetch
constexpr int kFTogether = 3;    // faces whose lines are worked on together, at most
constexpr int kFPool = 128;      // groups in reach of them
constexpr int kFTab = 128;       // entries of their offset tables
constexpr int kFBuf = 512;       // hits gathered before they leave

struct LineFace {
  float p[9];                    // vertices in the frame (corner of the range's first cell)
  float v0[3];
  float nh[3], nl[3];
  float shift[3];
  float h_hi, h_lo;
  float L, nn2;                  // bound on offsets in the frame; |n|
  float inv_g0, inv_g1;
  int lo[3], n[3];               // the face's cells: first, count
  int g[3], ng[3];               // groups (parents) of the range widened by one cell
  float xmax;                    // bound on the cell centres' coordinates
  int est;                       // about how many hits it will have
  int tab[3];                    // per axis: place of cell -1's entry in LineSmem::tab (n + 3 entries)
  uint32_t slot, face, gid;
};

struct LineDir {                 // one lattice direction of one face
  int face, l;
  float P[3], Q[3];              // the vertices in the projection along it
  float Pb, Qb, e;               // line (0, 0) there; error bound of an edge function
  float s0, su, sv, ds;          // crossing along line (u, v), in steps from its first cell; error bound
  float dh, dl, inv;             // c . n as hi + lo; 1 / (h c . n)
  float n1, ih, mg;              // |n|_1; 1 / h; margin of a line's place in the projection, in cells
  int u0, u1, v0;                // lines: u in [u0, u1], rows from v0
  int par;                       // c nearly parallel to the face
};

struct LineSmem {
  LineFace f[kFFaces];
  LineDir d[9 * kFTogether];
  int32_t bi[kFPool];            // group of each slot (-1: not in the level)
  uint32_t cnt[kFPool];          // hits gathered per slot
  uint32_t off[kFPool];
  uint8_t own[kFPool];
  float2 tab[kFTab];             // first vertex minus cell centre along an axis, hi + lo
  float bq[kFBuf];               // gathered hits: q, slot << 16 | direction << 9 | cell of the group, rank
  uint32_t bc[kFBuf];
  uint16_t br[kFBuf];
};

// Lattice line l: axes a (and b), sign of b's part, the third axis w.
struct Line {
  int a, b, w;
  float sg;
  int si;
};
__device__ __forceinline__ Line line_axes(int l) {
  Line r;
  if (l < 3) {
    r.a = l;
    r.b = l == 0 ? 1 : 0;
    r.w = l == 2 ? 1 : 2;
    r.si = 0;
  } else {
    const int p = (l - 3) >> 1;
    r.a = p == 2 ? 1 : 0;
    r.b = p == 0 ? 1 : 2;
    r.w = 2 - p;
    r.si = (l - 3) & 1 ? -1 : 1;
  }
  r.sg = (float)r.si;
  return r;
}
static_assert(d3q19_c(9, 0) == 1 && d3q19_c(9, 1) == -1 && d3q19_c(11, 0) == 1 && d3q19_c(11, 2) == 1 &&
              d3q19_c(17, 1) == 1 && d3q19_c(17, 2) == -1, "line l: directions 2l + 1 and 2l + 2");

__device__ __forceinline__ float frame_at(const LineFace& F, int c, float i) {
  return fmaf(i + 0.5f, F.h_hi, fmaf(i + 0.5f, F.h_lo, F.shift[c]));
}

template <bool MULTI>
__device__ __forceinline__ const GeomParams& geom_of(const FaceLinkArgs& a, uint32_t gid) {
  if constexpr (MULTI) return a.table[gid];
  return a.g0;
}

// Lines of row v of a projection that can lie inside it: u from `u` on, `n` of them (a superset).  The row cuts
// the triangle in the interval between its edges' crossings; each is widened by what the rounding of the
// row's place can move it along its edge.
__device__ __forceinline__ void row_lines(const LineFace& F, const LineDir& T, int v, int& u, uint32_t& n) {
  const float q0 = fmaf((float)v, F.h_hi, fmaf((float)v, F.h_lo, T.Qb));
  const float d = 16.0f * kU32 * F.L;
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const int m1 = (m + 1) % 3;
    const float a = T.Q[m] - q0, b = T.Q[m1] - q0;
    if (fminf(a, b) <= d && fmaxf(a, b) >= -d) {
      const float P0 = T.P[m], P1 = T.P[m1], w = fabsf(a - b);
      // the crossing, within 2 d / w of the edge; an edge within d of the row counts whole
      const float s = w > 0.f ? __fdividef(a, a - b) : 0.f, es = w > 0.f ? __fdividef(2.0f * d, w) + 1e-6f : 1.f;
      const float s0 = fminf(1.f, fmaxf(0.f, s - es)), s1 = fminf(1.f, fmaxf(0.f, s + es));
      const float x0 = fmaf(P1 - P0, s0, P0), x1 = fmaf(P1 - P0, s1, P0);
      lo = fminf(lo, fminf(x0, x1));
      hi = fmaxf(hi, fmaxf(x0, x1));
    }
  }
  const int u0 = max(T.u0, (int)fmaxf(-1e6f, ceilf((lo - T.Pb) * T.ih - T.mg)));
  const int u1 = min(T.u1, (int)fminf(1e6f, floorf((hi - T.Pb) * T.ih + T.mg)));
  u = u0;
  n = lo <= hi && u1 >= u0 ? (uint32_t)(u1 - u0 + 1) : 0u;
}

// The last lane whose first item (ascending, exclusive prefix sums) is at or before `item`: its owner, for
// items of the warp's lanes of which some have none.
__device__ __forceinline__ int last_at(uint32_t first, uint32_t item) {
  int l = 0;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1) {
    const uint32_t f = __shfl_sync(0xffffffffu, first, l + st);
    if (f <= item) l += st;
  }
  return l;
}

// Gathered hits out: a run per slot with hits.  Out of line (as is link_pair_3): the kernel's loop has to stay
// in the instruction cache.
__device__ __noinline__ void flush_hits(const FaceLinkArgs& a, LineSmem& sm, uint32_t nsl, uint32_t nbuf) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  uint32_t run = 0, runs = 0;
  for (uint32_t s0 = 0; s0 < nsl; s0 += 32) {
    const uint32_t s = s0 + lane, c = s < nsl ? sm.cnt[s] : 0u;
    const uint32_t incl = warp_inclusive_scan<uint32_t>(c);
    if (s < nsl) sm.off[s] = run + incl - c;
    run += __shfl_sync(0xffffffffu, incl, 31);
    runs += __popc(__ballot_sync(0xffffffffu, c != 0));
  }
  unsigned long long base = 0, rb = 0;
  if (lane == 0) {
    base = atomicAdd(a.hit_count, (unsigned long long)nbuf);
    rb = atomicAdd(a.run_count, (unsigned long long)runs);
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  rb = __shfl_sync(0xffffffffu, rb, 0);
  __syncwarp();
  for (uint32_t i = lane; i < nbuf; i += 32) {
    const uint32_t c = sm.bc[i];
    const unsigned long long at = base + sm.off[c >> 16] + sm.br[i];
    if ((int64_t)at < a.cap_hits) {
      a.hit_q[at] = sm.bq[i];
      a.hit_code[at] = (uint16_t)c;
    }
  }
  for (uint32_t s0 = 0; s0 < nsl; s0 += 32) {
    const uint32_t s = s0 + lane, c = s < nsl ? sm.cnt[s] : 0u;
    const unsigned cb = __ballot_sync(0xffffffffu, c != 0);
    const unsigned long long at = rb + __popc(cb & ((1u << lane) - 1u));
    rb += __popc(cb);
    if (c) {
      if ((int64_t)at < a.cap_runs) {
        StagedRun r;
        r.start = base + sm.off[s];
        r.n = c;
        r.face = sm.f[sm.own[s]].face;
        r.group = (uint32_t)sm.bi[s];
        r.rank = (uint32_t)atomicAdd(a.group_runs + sm.bi[s], 1ull);
        a.staged[at] = r;
      }
      sm.cnt[s] = 0u;
    }
  }
  __syncwarp();
}

template <bool MULTI>
__global__ void __launch_bounds__(kFWarps * 32, kFBlocks) k_face_links(FaceLinkArgs a) {
  __shared__ __align__(16) LineSmem s_all[kFWarps];
  const int lane = threadIdx.x & 31;
  LineSmem& sm = s_all[threadIdx.x >> 5];
  const int64_t nblk = launch_count(a.n_blocks, a.n_dev, a.err);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.n_groups = (uint64_t)(nblk >> 3);
  auto divn = [](int k, float inv) { return (int)(((float)k + 0.5f) * inv); };  // k / n, k < 2^20
  // the group of the level's blocks below parent b (coordinates on the level above), or -1
  auto find = [&](uint32_t gid, const int* b) -> int32_t {
    const GeomParams& Q = geom_of<MULTI>(a, gid);
    const int U = a.level - 1;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (b[c] < 0 || b[c] >= (Q.root[c] << U)) return -1;
    int64_t i = Q.root_base + (b[0] >> U) + (int64_t)Q.root[0] * ((b[1] >> U) + (int64_t)Q.root[1] * (b[2] >> U));
    for (int l = 0; l <= U; ++l) {
      const int32_t c = __ldg(a.first_child[l] + i);
      if (c < 0) return -1;
      if (l == U) return (int64_t)c + 8 <= nblk ? c >> 3 : -1;
      const int sh = U - l - 1;
      i = (int64_t)c + (((b[0] >> sh) & 1) | (((b[1] >> sh) & 1) << 1) | (((b[2] >> sh) & 1) << 2));
    }
    return -1;
  };
  unsigned long long n_fb = 0, n_band = 0, n_hit = 0;  // n_hit: warp-uniform
  uint32_t nbuf = 0, nsl = 0;
  auto flush = [&]() {
    if (nbuf) flush_hits(a, sm, nsl, nbuf);
    n_hit += nbuf;
    nbuf = 0;
  };
  for (;;) {
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(a.work, (unsigned)a.batch);
    base = __shfl_sync(0xffffffffu, base, 0);
    const int64_t first = a.faces.begin + base;
    if (first >= a.faces.end) break;
    // a lane per face: its cells (down to one layer outside the domain), their frame, the groups in reach
    const int64_t f = first + lane;
    bool use = lane < a.batch && f < a.faces.end;
    const uint32_t gid = MULTI && use ? __ldg(a.face_gid + f) : 0u;
    const GeomParams& P = geom_of<MULTI>(a, gid);
    use = use && P.n_levels - 1 == a.level;
    LineFace M;
    int my_slots = 0;
    if (use) {
      const FastGeom g = fast_geom(P, a.level);
      const float4* R = reinterpret_cast<const float4*>(a.rec + f);
      const float4 r0 = __ldg(R), r1 = __ldg(R + 1), r2 = __ldg(R + 2), r3 = __ldg(R + 3);
      const float V[9] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w, r2.x};
      M.nh[0] = r2.y, M.nh[1] = r2.z, M.nh[2] = r2.w;
      M.nl[0] = r3.x, M.nl[1] = r3.y, M.nl[2] = r3.z;
      M.h_hi = g.h_hi, M.h_lo = g.h_lo;
      const float inv_h = 1.0f / g.h_hi;
      float O = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int ncell = (4 * P.root[c]) << a.level;
        const float vmin = fminf(fminf(V[c], V[3 + c]), V[6 + c]), vmax = fmaxf(fmaxf(V[c], V[3 + c]), V[6 + c]);
        const float margin = 1e-3f + 16.0f * kU32 * (fmaxf(fabsf(vmin), fabsf(vmax)) + fabsf(P.org_hi[c])) * inv_h;
        const float xl = (vmin - P.org_hi[c]) * inv_h, xh = (vmax - P.org_hi[c]) * inv_h;
        if (!(xl <= xh)) use = false;
        const float tl = floorf(xl - margin), th = floorf(xh + margin);
        const int il = tl < -1.f ? -1 : (tl > (float)ncell ? ncell + 1 : (int)tl);
        const int ih = th < -1.f ? -2 : (th > (float)ncell ? ncell : (int)th);
        if (ih < il) use = false;
        M.lo[c] = il;
        M.n[c] = ih - il + 1;
        M.g[c] = (il - 1) >> 3;
        M.ng[c] = ((ih + 1) >> 3) - M.g[c] + 1;
        float corner, flo;
        df_position(P.org_hi[c], P.org_lo[c], (float)il, g.h_hi, g.h_lo, corner, flo);
        M.shift[c] = flo;
        M.v0[c] = V[c];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          M.p[3 * k + c] = V[3 * k + c] - corner;
          O = fmaxf(O, fabsf(M.p[3 * k + c]));
        }
        O = fmaxf(O, (float)(M.n[c] + 3) * g.h_hi + 2.0f * fabsf(flo));
      }
      M.L = O;
      M.xmax = 0.f;
      {
        // one hit each way per crossing; lines of direction d_l cross the face about |d_l . n| / (2 h^2) times
        const float x = M.nh[0], y = M.nh[1], z = M.nh[2];
        const float all = fabsf(x) + fabsf(y) + fabsf(z) + fabsf(x + y) + fabsf(x - y) + fabsf(x + z) + fabsf(x - z) +
                          fabsf(y + z) + fabsf(y - z);
        M.est = (int)fminf(1e6f, 1.15f * all * inv_h * inv_h) + 16;
      }
      int ne = 0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        M.xmax = fmaxf(M.xmax, fabsf(M.v0[c]) + O + 2.0f * g.h_hi);  // centres lie within L of the vertex
        M.tab[c] = ne;
        ne += M.n[c] + 3;
      }
      M.nn2 = sqrtf(M.nh[0] * M.nh[0] + M.nh[1] * M.nh[1] + M.nh[2] * M.nh[2]);
      M.inv_g0 = 1.0f / (float)M.ng[0], M.inv_g1 = 1.0f / (float)M.ng[1];
      M.slot = 0u, M.face = (uint32_t)f, M.gid = gid;
      const int64_t wide = (int64_t)M.ng[0] * M.ng[1] * M.ng[2];
      if (use && (wide > kFPool || ne > kFTab)) {  // the host keeps the largest face's range below 2^15 cells
        atomicOr(a.err, ERR_OVERFLOW);
        use = false;
      }
      my_slots = use ? (int)wide : 0;
    }
    const unsigned valid = __ballot_sync(0xffffffffu, use);
    const int nv = __popc(valid);
    if (use) sm.f[__popc(valid & ((1u << lane) - 1u))] = M;
    __syncwarp();
    my_slots = lane < nv ? sm.f[lane].ng[0] * sm.f[lane].ng[1] * sm.f[lane].ng[2] : 0;
    const uint32_t my_tab = lane < nv ? (uint32_t)(sm.f[lane].tab[2] + sm.f[lane].n[2] + 3) : 0u;
    for (int g0 = 0; g0 < nv;) {
      // a few faces whose groups, tables and hits fit
      const uint32_t ns = lane >= g0 && lane < nv ? (uint32_t)my_slots : 0u;
      const uint32_t sincl = warp_inclusive_scan<uint32_t>(ns);
      const uint32_t nt = lane >= g0 && lane < nv ? my_tab : 0u, tincl = warp_inclusive_scan<uint32_t>(nt);
      // (one face always fits; its hits may leave in several parts)
      const uint32_t he = lane >= g0 && lane < nv ? (uint32_t)sm.f[lane].est : 0u, hincl = warp_inclusive_scan<uint32_t>(he);
      const bool fits = ns && sincl <= (uint32_t)kFPool && tincl <= (uint32_t)kFTab && lane < g0 + kFTogether &&
                        (lane == g0 || hincl <= (uint32_t)kFBuf - 64u);
      const int g1 = g0 + __popc(__ballot_sync(0xffffffffu, fits));
      const bool own = lane >= g0 && lane < g1;
      const uint32_t tfirst0 = tincl - nt, ntab = __shfl_sync(0xffffffffu, tincl, g1 - 1);
      nsl = __shfl_sync(0xffffffffu, sincl, g1 - 1);
      const uint32_t sfirst = sincl - ns;
      if (own) sm.f[lane].slot = sfirst;
      __syncwarp();
      // the offset of the first vertex from every cell coordinate in reach (k_links' operations)
      for (uint32_t k0 = 0; k0 < ntab; k0 += 32) {
        const int j = range_owner(tfirst0, own, g0, k0, lane);
        const int k = (int)(k0 + lane - __shfl_sync(0xffffffffu, tfirst0, j));
        if (k0 + lane < ntab) {
          const LineFace& Q = sm.f[j];
          const GeomParams& G = geom_of<MULTI>(a, Q.gid);
          const int c = k >= Q.tab[2] ? 2 : (k >= Q.tab[1] ? 1 : 0);
          const int x = Q.lo[c] + k - Q.tab[c] - 1;
          float ohi, olo, p, e;
          df_position(G.org_hi[c], G.org_lo[c], (float)(2 * x + 1), 0.5f * Q.h_hi, 0.5f * Q.h_lo, ohi, olo);
          df_two_sum(Q.v0[c], -ohi, p, e);
          sm.tab[k0 + lane] = make_float2(p, e - olo);
        }
      }
      __syncwarp();
      if (own) {
#pragma unroll
        for (int c = 0; c < 3; ++c) sm.f[lane].tab[c] += (int)tfirst0;
      }
      for (uint32_t k0 = 0; k0 < nsl; k0 += 32) {
        const int j = range_owner(sfirst, own, g0, k0, lane);
        const uint32_t s = k0 + lane;
        if (s < nsl) {
          const LineFace& Q = sm.f[j];
          const int k = (int)(s - Q.slot), k1 = divn(k, Q.inv_g0), k2 = divn(k1, Q.inv_g1);
          const int b[3] = {Q.g[0] + k - k1 * Q.ng[0], Q.g[1] + k1 - k2 * Q.ng[1], Q.g[2] + k2};
          sm.bi[s] = find(Q.gid, b);
          sm.own[s] = (uint8_t)j;
          sm.cnt[s] = 0u;
        }
      }
      __syncwarp();
      // slot of the group that holds cell x (absolute) of face Q: of a cell in reach, or of any (-1: none)
      auto slot_in = [&](const LineFace& Q, const int* x) -> int {
        return (int)Q.slot + ((x[0] >> 3) - Q.g[0]) + Q.ng[0] * (((x[1] >> 3) - Q.g[1]) + Q.ng[1] * ((x[2] >> 3) - Q.g[2]));
      };
      auto slot_of = [&](const LineFace& Q, const int* x) -> int {
        const int q[3] = {(x[0] >> 3) - Q.g[0], (x[1] >> 3) - Q.g[1], (x[2] >> 3) - Q.g[2]};
        if (q[0] < 0 || q[0] >= Q.ng[0] || q[1] < 0 || q[1] >= Q.ng[1] || q[2] < 0 || q[2] >= Q.ng[2]) return -1;
        const int s = (int)Q.slot + q[0] + Q.ng[0] * (q[1] + Q.ng[1] * q[2]);
        return sm.bi[s] >= 0 ? s : -1;
      };
      // cell of its group: child slot, then the cell of the block
      auto code_of = [](const int* x, int dir) {
        const uint32_t child = ((x[0] >> 2) & 1) | (((x[1] >> 2) & 1) << 1) | (((x[2] >> 2) & 1) << 2);
        const uint32_t cell = (x[0] & 3) | ((x[1] & 3) << 2) | ((x[2] & 3) << 4);
        return child << 6 | cell | (uint32_t)dir << 9;
      };
      // every lane with h adds a hit (whole warp; there is room for 32)
      auto append = [&](bool h, int slot, uint32_t code, float q) {
        const unsigned hb = __ballot_sync(0xffffffffu, h);
        if (h) {
          const uint32_t at = nbuf + __popc(hb & ((1u << lane) - 1u));
          sm.bq[at] = !(q > 0.0f) ? 0.0f : fminf(q, 1.0f);
          sm.bc[at] = (uint32_t)slot << 16 | code;
          sm.br[at] = (uint16_t)atomicAdd(&sm.cnt[slot], 1u);
        }
        nbuf += __popc(hb);
      };
      {
        // a lane per (face, direction): the projection along the direction and its rows of lines
        uint32_t nr = 0;
        if (lane < 9 * (g1 - g0)) {
          const int fi = g0 + lane / 9, l = lane % 9;
          const Line ln = line_axes(l);
          const LineFace& F = sm.f[fi];
          LineDir& T = sm.d[lane];
          T.face = fi;
          T.l = l;
          const float oa = frame_at(F, ln.a, 0.f), ob = frame_at(F, ln.b, 0.f), ow = frame_at(F, ln.w, 0.f);
          float pmin = INFINITY, pmax = -INFINITY, qmin = INFINITY, qmax = -INFINITY;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const float p = F.p[3 * k + ln.b] - ln.sg * F.p[3 * k + ln.a], q = F.p[3 * k + ln.w];
            T.P[k] = p;
            T.Q[k] = q;
            pmin = fminf(pmin, p), pmax = fmaxf(pmax, p);
            qmin = fminf(qmin, q), qmax = fmaxf(qmax, q);
          }
          const float Pb = ob - ln.sg * oa;
          T.Pb = Pb;
          T.Qb = ow;
          // Beyond this k_links certifies the edge, too.  Offsets of a line inside the projection are at most 2 L in P
          // and L in Q, and within 8.2 u L (a difference of two vertex coordinates, the line's place, their difference,
          // each rounded) and 3 u L of their values, so an edge function is within 2 (2 L 3 u L + L 8.2 u L) + 6 u L^2 <
          // 35 u L^2.  k_links asks for 8 u |c|_1 M and is itself within 4 u |c|_1 M, M <= 2 L^2: 48 u L^2 more.
          T.e = 96.0f * kU32 * F.L * F.L;
          // c . n and the crossing's place along line (u, v)
          float dh, de;
          df_two_sum(F.nh[ln.a], ln.sg * F.nh[ln.b], dh, de);
          const float dl = de + (F.nl[ln.a] + ln.sg * F.nl[ln.b]), den = dh + dl;
          T.dh = dh, T.dl = dl;
          T.par = fabsf(den) <= (ln.si == 0 ? 1e-5f : 1.41421356e-5f) * F.nn2;
          T.n1 = fabsf(F.nh[0]) + fabsf(F.nh[1]) + fabsf(F.nh[2]);
          const float inv = 1.0f / (F.h_hi * den);
          const float num = F.nh[0] * F.p[0] + F.nh[1] * F.p[1] + F.nh[2] * F.p[2] -
                            (F.nh[ln.a] * oa + F.nh[ln.b] * ob + F.nh[ln.w] * ow);
          T.inv = inv;
          T.s0 = num * inv;
          T.su = -F.nh[ln.b] * F.h_hi * inv;
          T.sv = -F.nh[ln.w] * F.h_hi * inv;
          T.ds = 64.0f * kU32 * T.n1 * F.L * fabsf(inv);
          // lines that can meet the projection (a superset), within reach of the range's cells
          const float ih = 1.0f / F.h_hi, mg = 1e-3f + 16.0f * kU32 * F.L * ih;
          const int na = F.n[ln.a], nb = F.n[ln.b], nw = F.n[ln.w];
          const int ul = ln.si == 0 ? -1 : (ln.si > 0 ? -1 - na : -2), uh = ln.si == 0 ? nb : (ln.si > 0 ? nb + 1 : na + nb);
          const int u0 = max(ul, (int)fmaxf(-1e6f, ceilf((pmin - Pb) * ih - mg)));
          const int u1 = min(uh, (int)fminf(1e6f, floorf((pmax - Pb) * ih + mg)));
          const int v0 = max(-1, (int)fmaxf(-1e6f, ceilf((qmin - ow) * ih - mg)));
          const int v1 = min(nw, (int)fminf(1e6f, floorf((qmax - ow) * ih + mg)));
          T.u0 = u0, T.u1 = u1, T.v0 = v0;
          T.ih = ih, T.mg = mg;
          if (u1 >= u0 && v1 >= v0 && !(den == 0.0f && dh == 0.0f)) nr = (uint32_t)(v1 - v0 + 1);
        }
        __syncwarp();
        const uint32_t rincl = warp_inclusive_scan<uint32_t>(nr);
        const uint32_t rfirst = rincl - nr, nrow = __shfl_sync(0xffffffffu, rincl, 31);
        // cell i of line (u, v)
        auto cell_at = [&](const LineFace& F, const Line& ln, int u, int v, int i, int* x) {
#pragma unroll
          for (int c = 0; c < 3; ++c) x[c] = F.lo[c] + (c == ln.a ? i : (c == ln.b ? u + ln.si * i : v));
        };
        for (uint32_t r0 = 0; r0 < nrow; r0 += 32) {
          // a lane per row of lines: the part of it inside the projection
          int jr = last_at(rfirst, r0 + lane), vr = 0, ur = 0;
          const int kr = (int)(r0 + lane - __shfl_sync(0xffffffffu, rfirst, jr));
          uint32_t rc = 0;
          if (r0 + lane < nrow) {
            vr = sm.d[jr].v0 + kr;
            row_lines(sm.f[sm.d[jr].face], sm.d[jr], vr, ur, rc);
          }
          const uint32_t tincl = warp_inclusive_scan<uint32_t>(rc);
          const uint32_t tfirst = tincl - rc, items = __shfl_sync(0xffffffffu, tincl, 31);
          for (uint32_t k0 = 0; k0 < items; k0 += 32) {
            // a lane per line: inside by its edge functions; then the cells before and after the crossing
            const int rl = last_at(tfirst, k0 + lane);
            const int j = __shfl_sync(0xffffffffu, jr, rl), v = __shfl_sync(0xffffffffu, vr, rl);
            const int u = __shfl_sync(0xffffffffu, ur, rl) + (int)(k0 + lane - __shfl_sync(0xffffffffu, tfirst, rl));
            if (nbuf > (uint32_t)kFBuf - 64u) flush();
            bool redo = false, ha = false, hb = false;
            int ilo = 0, ihi = -1, sa = -1, sb = -1;
            uint32_t ca = 0, cb = 0;
            float qa = 0.f, qb = 0.f;
            if (k0 + lane < items) {
              const LineDir& T = sm.d[j];
              const LineFace& F = sm.f[T.face];
              const Line ln = line_axes(T.l);
              const float p0 = fmaf((float)u, F.h_hi, fmaf((float)u, F.h_lo, T.Pb));
              const float q0 = fmaf((float)v, F.h_hi, fmaf((float)v, F.h_lo, T.Qb));
              const float Pd[3] = {T.P[0] - p0, T.P[1] - p0, T.P[2] - p0};
              const float Qd[3] = {T.Q[0] - q0, T.Q[1] - q0, T.Q[2] - q0};
              float lo = INFINITY, hi = -INFINITY;
#pragma unroll
              for (int m = 0; m < 3; ++m) {
                const int m1 = (m + 1) % 3;
                const float U = fmaf(Pd[m], Qd[m1], -Qd[m] * Pd[m1]);
                lo = fminf(lo, U);
                hi = fmaxf(hi, U);
              }
              const bool outside = hi > T.e && lo < -T.e;
              const bool in = (lo > T.e || hi < -T.e) && !T.par;
              const float sc = fmaf((float)u, T.su, fmaf((float)v, T.sv, T.s0));
              const int na = F.n[ln.a];
              if (in) {
                const float den = T.dh + T.dl, sg = den > 0.f ? 1.f : -1.f, hd = F.h_hi * fabsf(den);
                const float eps0 = 16.0f * kU32 * kU32 * T.n1 * (F.xmax + 2.0f * F.L);
                // num = n . (v0 - x) in double-float with k_links' operations, from the tables, and its error bound
                auto offset = [&](int i, float& eps) {
                  float2 d[3];
#pragma unroll
                  for (int c = 0; c < 3; ++c) d[c] = sm.tab[F.tab[c] + 1 + (c == ln.a ? i : (c == ln.b ? u + ln.si * i : v))];
                  float ns, ne;
                  df_two_prod(F.nh[0], d[0].x, ns, ne);
#pragma unroll
                  for (int c = 1; c < 3; ++c) {
                    float pp, pe, s, t;
                    df_two_prod(F.nh[c], d[c].x, pp, pe);
                    df_two_sum(ns, pp, s, t);
                    ns = s;
                    ne += t + pe;
                  }
#pragma unroll
                  for (int c = 0; c < 3; ++c) ne = fmaf(F.nh[c], d[c].y, fmaf(F.nl[c], d[c].x, ne));
                  eps = eps0 + 4.0f * kU32 * fabsf(ne);
                  return ns + ne;
                };
                auto certified = [&](float sn, float e) { return sn > e && sn + e < hd * (1.0f - 8.0f * kU32); };
                // the cell before the crossing; it and the next lie in the widened range, on both axes
                const int nb = F.n[ln.b];
                const int i0 = max(-1, ln.si == 0 ? -1 : (ln.si > 0 ? -1 - u : u - nb));
                const int i1 = min(na - 1, ln.si == 0 ? na : (ln.si > 0 ? nb - u - 1 : u));
                int i = (int)fminf((float)i1, fmaxf((float)i0, floorf(sc)));
                bool ok = false;
                float eps, num = 0.f;
#pragma unroll 1
                for (int tries = 0; tries < 2 && i0 <= i1; ++tries) {
                  num = offset(i, eps);
                  ok = certified(sg * num, eps);
                  const float t = num * T.inv;
                  if (ok || (t >= 0.f && t < 1.f)) break;
                  i = (int)fminf((float)i1, fmaxf((float)i0, (float)i + floorf(t)));  // the estimate was off
                }
                if (ok) {
                  qa = num / (F.h_hi * den);
                  num = offset(i + 1, eps);
                  ok = certified(-sg * num, eps);
                  qb = num / (F.h_hi * -den);
                }
                if (ok) {
                  int x[3];
                  cell_at(F, ln, u, v, i, x);
                  sa = slot_in(F, x);
                  ca = code_of(x, 2 * T.l + 1);
                  cell_at(F, ln, u, v, i + 1, x);
                  sb = slot_in(F, x);
                  cb = code_of(x, 2 * T.l + 2);
                  ha = sm.bi[sa] >= 0;
                  hb = sm.bi[sb] >= 0;
                }
                redo = !ok;
                ilo = i0 <= i1 ? max(-1, i - 1) : -1;
                ihi = i0 <= i1 ? min(na, i + 2) : na;
              } else if (!outside) {
                if (T.par) {
                  redo = !(fabsf(sc) > (float)(na + 3) + T.ds);
                  ilo = -1;
                  ihi = na;
                } else {
                  ilo = (int)fminf((float)na, fmaxf(-1.f, floorf(sc - T.ds) - 1.f));
                  ihi = (int)fmaxf(-1.f, fminf((float)na, floorf(sc + T.ds) + 2.f));
                  redo = true;
                }
              }
            }
            append(ha, sa, ca, qa);
            append(hb, sb, cb, qb);
            // lines not certified: both senses of cells [ilo, ihi] by k_links' own test of the pair (FP64
            // where that is not certified), eight lanes per line
            for (unsigned rb = __ballot_sync(0xffffffffu, redo); rb;) {
              unsigned mine = rb;
#pragma unroll
              for (int k = 0; k < 3; ++k)
                if (k < lane >> 3) mine &= mine - 1u;
#pragma unroll
              for (int k = 0; k < 4; ++k) rb &= rb - 1u;
              const int src = mine ? __ffs(mine) - 1 : 0;
              const int js = __shfl_sync(0xffffffffu, j, src), us = __shfl_sync(0xffffffffu, u, src),
                        vs = __shfl_sync(0xffffffffu, v, src), i0 = __shfl_sync(0xffffffffu, ilo, src),
                        i1 = __shfl_sync(0xffffffffu, ihi, src);
              const int ne = mine ? 2 * (i1 - i0 + 1) : 0, most = __reduce_max_sync(0xffffffffu, ne);
              for (int t0 = 0; t0 < most; t0 += 8) {
                if (nbuf > (uint32_t)kFBuf - 32u) flush();
                const LineFace& F = sm.f[sm.d[mine ? js : 0].face];
                const int l = sm.d[mine ? js : 0].l;
                const Line ln = line_axes(l);
                const int t = t0 + (lane & 7), dir = 2 * l + 1 + (t & 1);
                bool h = false;
                int slot = -1, x[3] = {0, 0, 0};
                float q = 0.f;
                if (t < ne) {
                  cell_at(F, ln, us, vs, i0 + (t >> 1), x);
                  slot = slot_of(F, x);
                  if (slot >= 0) {
                    const GeomParams& G = geom_of<MULTI>(a, F.gid);
                    const int st = link_pair_3(a.rec + F.face, x, G, F.h_hi, F.h_lo, dir, &q);
                    h = st == 1;
                    if (st == 2) {
                      const double o3[3] = {G.origin[0], G.origin[1], G.origin[2]};
                      const float4* R = reinterpret_cast<const float4*>(a.rec + F.face);
                      const float4 w0 = __ldg(R), w1 = __ldg(R + 1), w2 = __ldg(R + 2);
                      const float V[9] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w, w2.x};
                      const int blk[3] = {x[0] >> 2, x[1] >> 2, x[2] >> 2};
                      const uint32_t bit = (x[0] & 3) | ((x[1] & 3) << 2) | ((x[2] & 3) << 4);
                      const LinkHit r = link_fallback_3(V, blk, bit, o3, scalbn(G.h0, -a.level), dir);
                      ++n_fb;
                      if (r.band) ++n_band;
                      h = r.hit;
                      q = (float)r.t;
                    }
                  }
                }
                append(h, slot, code_of(x, dir), q);
              }
            }
          }
        }
        __syncwarp();
      }
      flush();
      g0 = g1;
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n_fb += __shfl_xor_sync(0xffffffffu, n_fb, o);
    n_band += __shfl_xor_sync(0xffffffffu, n_band, o);
  }
  if (lane == 0) {
    if (n_fb) atomicAdd(&a.counters[CNT_LINK_FALLBACK], n_fb);
    if (n_band) atomicAdd(&a.counters[CNT_LINK_BAND], n_band);
    if (n_hit) atomicAdd(&a.counters[CNT_LINK_CAND], n_hit);
  }
}

// The runs by group (first[g] = scan of the groups' counts).
__global__ void __launch_bounds__(256) k_place_runs(FaceLinkArgs a) {
  const int64_t n = (int64_t)*a.run_count;
  if (n > a.cap_runs || (int64_t)*a.hit_count > a.cap_hits) {  // not all were kept: the caller runs again with more room
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, ERR_OVERFLOW);
    return;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const StagedRun r = a.staged[i];
    HitRun o;
    o.start = r.start;
    o.n = r.n;
    o.face = r.face;
    a.runs[a.first[r.group] + r.rank] = o;
  }
}

constexpr int kGWarps = 4;       // warps per CTA of the group kernels
constexpr int kGBlocks = 8;      // CTAs of k_write_links per SM (shared memory)
constexpr int kGWindow = 448;    // links of a group gathered in shared memory at a time

// Visit a group's hits, 4 a lane at a time (their loads overlap): fn(valid, code, q, face); returns their
// number.  WITH_Q: also read q.
template <bool WITH_Q, typename F>
__device__ __forceinline__ uint32_t for_hits(const FaceLinkArgs& a, int64_t g, uint32_t n_run, int lane, F&& fn) {
  constexpr int U = 4;
  const HitRun* runs = a.runs + a.first[g];
  uint32_t all = 0;
  for (uint32_t r0 = 0; r0 < n_run; r0 += 32) {
    HitRun r{};
    if (r0 + lane < n_run) r = runs[r0 + lane];
    const uint32_t incl = warp_inclusive_scan<uint32_t>(r.n);
    const uint32_t first = incl - r.n, total = __shfl_sync(0xffffffffu, incl, 31);
    all += total;
    for (uint32_t k0 = 0; k0 < total; k0 += 32 * U) {
      uint32_t code[U], face[U];
      float q[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const uint32_t k = k0 + 32 * i;
        const int j = range_owner(first, r.n != 0u, 0, k, lane);  // (every run has hits)
        const unsigned long long at = __shfl_sync(0xffffffffu, r.start - first, j) + k + lane;
        face[i] = __shfl_sync(0xffffffffu, r.face, j);
        const bool ok = k + lane < total;
        code[i] = ok ? (uint32_t)a.hit_code[at] : 0xffffffffu;
        q[i] = WITH_Q && ok ? a.hit_q[at] : 0.f;
      }
#pragma unroll
      for (int i = 0; i < U; ++i) fn(code[i] != 0xffffffffu, code[i], q[i], face[i]);
    }
  }
  return all;
}

// Per-cell tables have one pad word per 16 cells: a lane owns 16 cells in a row.
constexpr int kGCells = 512 + 32;
__device__ __forceinline__ uint32_t cell_word(uint32_t cell) { return cell + (cell >> 4); }

// A group's directions hit per cell; returns its hits.
__device__ __forceinline__ uint32_t mark_hits(const FaceLinkArgs& a, int64_t g, uint32_t n_run, uint32_t* dirs, int lane) {
#pragma unroll
  for (int i = 0; i < kGCells / 32; ++i) dirs[lane + 32 * i] = 0u;
  __syncwarp();
  const uint32_t n = for_hits<false>(a, g, n_run, lane, [&](bool ok, uint32_t code, float, uint32_t) {
    if (ok) atomicOr(dirs + cell_word(code & 511u), 1u << (code >> 9));
  });
  __syncwarp();
  return n;
}

// The lane's 16 cells of the group (lane >> 2 = block): adjacent cells among them.
__device__ __forceinline__ uint32_t lane_cells(const FaceLinkArgs& a, int64_t g, int lane) {
  return (uint32_t)(a.mask[8 * g + (lane >> 2)] >> (16 * (lane & 3))) & 0xffffu;
}

__global__ void __launch_bounds__(kGWarps * 32) k_count_links(FaceLinkArgs a) {
  __shared__ uint32_t s_dirs[kGWarps][kGCells];
  const int lane = threadIdx.x & 31;
  uint32_t* dirs = s_dirs[threadIdx.x >> 5];
  const int64_t n = (int64_t)*a.n_groups, nw = (int64_t)gridDim.x * kGWarps;
  // not all were kept (reported by k_place_runs): the level has no links then
  const bool kept = (int64_t)*a.run_count <= a.cap_runs && (int64_t)*a.hit_count <= a.cap_hits;
  for (int64_t g = (int64_t)blockIdx.x * kGWarps + (threadIdx.x >> 5); g < n; g += nw) {
    const uint32_t n_run = (uint32_t)a.group_runs[g];
    uint32_t c = 0;
    if (n_run && kept) {
      mark_hits(a, g, n_run, dirs, lane);
      const uint32_t cells = lane_cells(a, g, lane);
#pragma unroll
      for (int i = 0; i < 16; ++i) c += (cells >> i) & 1u ? __popc(dirs[17 * lane + i]) : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      __syncwarp();
    }
    if (lane == 0) a.group_links[g] = c;
  }
}

struct WriteSmem {
  uint32_t dirs[kGCells];                // per cell: directions hit (1 to 18) << 13 | its first link in the group (14 bits)
  uint32_t cells[32];                    // per lane's 16 cells: the adjacent ones | row of the first << 16
  unsigned long long key[kGWindow];      // q bits << 34 | direction << 29 | face
  uint16_t row[kGWindow];
};

__global__ void __launch_bounds__(kGWarps * 32, kGBlocks) k_write_links(FaceLinkArgs a) {
  __shared__ __align__(16) WriteSmem s_all[kGWarps];
  const int lane = threadIdx.x & 31;
  WriteSmem& sm = s_all[threadIdx.x >> 5];
  const int64_t n = (int64_t)*a.n_groups, nw = (int64_t)gridDim.x * kGWarps;
  const uint64_t row0 = a.run[0], link0 = a.run[2];
  if (link0 + *a.n_links > (uint64_t)a.link_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, ERR_OVERFLOW);
    return;
  }
  if ((int64_t)*a.run_count > a.cap_runs || (int64_t)*a.hit_count > a.cap_hits) return;  // reported by k_place_runs
  for (int64_t g = (int64_t)blockIdx.x * kGWarps + (threadIdx.x >> 5); g < n; g += nw) {
    const uint32_t n_run = (uint32_t)a.group_runs[g];
    if (!n_run) continue;
    const uint32_t n_hit = mark_hits(a, g, n_run, sm.dirs, lane);
    // each cell's first link and row
    const uint32_t cells = lane_cells(a, g, lane);
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) c += (cells >> i) & 1u ? __popc(sm.dirs[17 * lane + i]) : 0;
    const uint32_t rows = __popc(cells);
    const uint32_t cincl = warp_inclusive_scan<uint32_t>(c), rincl = warp_inclusive_scan<uint32_t>(rows);
    const uint32_t total = __shfl_sync(0xffffffffu, cincl, 31);
    sm.cells[lane] = cells | (rincl - rows) << 16;
    {
      uint32_t at = cincl - c;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        // (a hit cell is adjacent: others have no hits)
        const uint32_t d = (cells >> i) & 1u ? sm.dirs[17 * lane + i] : 0u;
        sm.dirs[17 * lane + i] = d << 13 | at;
        at += __popc(d);
      }
    }
    __syncwarp();
    const uint64_t grow = row0 + (a.block_base[8 * g] >> 32), out0 = link0 + a.link_base[g];
    for (uint32_t w0 = 0; w0 < total; w0 += kGWindow) {
      const uint32_t nw0 = total - w0 < (uint32_t)kGWindow ? total - w0 : (uint32_t)kGWindow;
      const bool once = n_hit == total;  // one face per link: plain stores
      if (!once) {
        for (uint32_t i = lane; i < nw0; i += 32) sm.key[i] = ~0ull;
        __syncwarp();
      }
      for_hits<true>(a, g, n_run, lane, [&](bool ok, uint32_t code, float q, uint32_t face) {
        if (!ok) return;
        const uint32_t cell = code & 511u, dir = code >> 9, w = sm.dirs[cell_word(cell)], d = (w >> 13) & ~1u;
        const uint32_t pos = (w & 0x3fffu) + __popc(d & ((1u << dir) - 1u)) - w0;
        if (pos >= nw0 || !((d >> dir) & 1u)) return;
        const uint32_t t = sm.cells[cell >> 4];
        const unsigned long long k = (unsigned long long)__float_as_uint(q) << 34 | (unsigned long long)dir << 29 | face;
        if (once)
          sm.key[pos] = k;
        else
          atomicMin(&sm.key[pos], k);
        sm.row[pos] = (uint16_t)((t >> 16) + __popc(t & ((1u << (cell & 15u)) - 1u)));
      });
      __syncwarp();
      for (uint32_t i = lane; i < nw0; i += 32) {
        const unsigned long long k = sm.key[i];
        const uint64_t o = out0 + w0 + i;
        a.link_cell[o] = (uint32_t)(grow + sm.row[i]);
        a.link_dir[o] = (uint8_t)((k >> 29) & 31u);
        a.link_q[o] = __uint_as_float((uint32_t)(k >> 34));
        a.link_face[o] = (uint32_t)(k & ((1ull << 29) - 1));
      }
      __syncwarp();
    }
  }
}

}  // namespace

int launch_face_links(const FaceLinkArgs& a0, void* scan_scratch, int num_sms, cudaStream_t st) {
  FaceLinkArgs a = a0;
  const int64_t groups = std::max<int64_t>(1, a.n_blocks / 8);
  cudaMemsetAsync(a.hit_count, 0, 2 * sizeof(unsigned long long), st);  // and run_count, which follows it
  cudaMemsetAsync(a.group_runs, 0, sizeof(uint64_t) * (size_t)groups, st);
  cudaMemsetAsync(a.work, 0, sizeof(unsigned), st);
  const int64_t grid = (int64_t)num_sms * kFBlocks;
  a.batch = a.faces.fetch(grid * kFWarps, kFFaces);
  const int64_t nf = a.faces.end - a.faces.begin;
  const int64_t need = std::max<int64_t>(1, (nf + (int64_t)a.batch * kFWarps - 1) / ((int64_t)a.batch * kFWarps));
  if (a.table)
    k_face_links<true><<<(unsigned)std::min(need, grid), kFWarps * 32, 0, st>>>(a);
  else
    k_face_links<false><<<(unsigned)std::min(need, grid), kFWarps * 32, 0, st>>>(a);
  int k = 1;
  k += launch_scan_u64(reinterpret_cast<const uint64_t*>(a.group_runs), a.first, groups, a.n_groups, a.scan_total,
                       scan_scratch, a.err, num_sms, st);
  k_place_runs<<<(unsigned)std::min<int64_t>((a.cap_runs + 255) / 256, (int64_t)num_sms * 8), 256, 0, st>>>(a);
  const unsigned gg = (unsigned)std::min<int64_t>((groups + kGWarps - 1) / kGWarps, (int64_t)num_sms * 16);
  k_count_links<<<gg, kGWarps * 32, 0, st>>>(a);
  k += 2 + launch_scan_u64(a.group_links, a.link_base, groups, a.n_groups, a.n_links, scan_scratch, a.err, num_sms, st);
  const unsigned gw = (unsigned)std::min<int64_t>((groups + kGWarps - 1) / kGWarps, (int64_t)num_sms * kGBlocks);
  k_write_links<<<gw, kGWarps * 32, 0, st>>>(a);
  return k + 1;
}

}  // namespace amr
