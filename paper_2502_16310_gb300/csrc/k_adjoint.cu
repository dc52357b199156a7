// k_adjoint.cu — vertex adjoint of the wall-link fractions q, deterministic.
//
// q of a link is the hit parameter t of the plane through its face (links are
// only formed on hits, Sec. "Identification of Cells Near the Boundary"):
//   t = ((v0 - x) . n) / (d . n),  n = (v1 - v0) x (v2 - v0),  d = c_i h.
// With w = (v0 - x - t d) / (d . n):
//   dt/dv1 = (v2 - v0) x w,  dt/dv2 = w x (v1 - v0),  dt/dv0 = n / (d . n) - dt/dv1 - dt/dv2
// (2D: t = ((v0 - x) x e) / (d x e), e = v1 - v0, dt/dv1 = (-w_y, w_x),
//  dt/dv0 = (e_y, -e_x) / (d x e) - dt/dv1).  The flags and the adjacency are
// not differentiated: gradients flow only through q of the hit face.
//
// Determinism without float atomics: a tile's links are grouped by face in shared
// memory and added in a fixed order (double-float), and the tiles' sums of a face
// are added as integers (fixed point, a scale per face), whose order does not
// matter.  For indexed input the face corners are grouped by vertex with a stable
// LSD radix sort (once per load) and one thread per vertex sums its corners in
// ascending (face, corner) order.
#include "internal.cuh"

namespace amr {

namespace {

constexpr int kRThreads = 256;
constexpr int kRWarps = kRThreads / 32;
constexpr int kRItems = 16;                       // keys per thread
constexpr int kRTile = kRThreads * kRItems;       // 4096 keys per tile
constexpr int kRBits = 8;
constexpr int kRDigits = 1 << kRBits;

// Per tile: digit histogram, written digit-major so that one exclusive scan
// over [digit][tile] gives every (digit, tile) its output base.
__global__ void __launch_bounds__(kRThreads) k_radix_hist(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                          uint32_t* __restrict__ hist, int64_t n_tiles) {
  __shared__ uint32_t h[kRDigits];
  for (int i = threadIdx.x; i < kRDigits; i += kRThreads) h[i] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kRTile;
  for (int i = threadIdx.x; i < kRTile; i += kRThreads) {
    const int64_t j = base + i;
    if (j < n) atomicAdd(&h[(keys[j] >> shift) & (kRDigits - 1)], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kRDigits; i += kRThreads) hist[(int64_t)i * n_tiles + blockIdx.x] = h[i];
}

// Stable scatter of one tile: warp w owns keys [w*512, (w+1)*512) of the tile;
// per-warp digit counts are prefixed across warps, then each warp walks its
// keys 32 at a time in order, ranking equal digits with __match_any_sync.
// vals_in null: the values are the keys' indices; keys_out null: keys not kept.
__global__ void __launch_bounds__(kRThreads) k_radix_scatter(const uint32_t* __restrict__ keys_in,
                                                             const uint32_t* __restrict__ vals_in, int64_t n, int shift,
                                                             const uint32_t* __restrict__ offs, int64_t n_tiles,
                                                             uint32_t* __restrict__ keys_out,
                                                             uint32_t* __restrict__ vals_out) {
  __shared__ uint32_t cnt[kRWarps][kRDigits];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kRWarps * kRDigits; i += kRThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  const int64_t wbase = (int64_t)blockIdx.x * kRTile + (int64_t)wid * (kRTile / kRWarps);
  constexpr int kChunks = kRTile / kRWarps / 32;
  for (int c = 0; c < kChunks; ++c) {
    const int64_t j = wbase + c * 32 + lane;
    if (j < n) atomicAdd(&cnt[wid][(keys_in[j] >> shift) & (kRDigits - 1)], 1u);
  }
  __syncthreads();
  // exclusive prefix over warps per digit, plus the global base of (digit, tile)
  for (int d = threadIdx.x; d < kRDigits; d += kRThreads) {
    uint32_t run = offs[(int64_t)d * n_tiles + blockIdx.x];
    for (int w = 0; w < kRWarps; ++w) {
      const uint32_t c = cnt[w][d];
      cnt[w][d] = run;
      run += c;
    }
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  for (int c = 0; c < kChunks; ++c) {
    const int64_t j = wbase + c * 32 + lane;
    const bool ok = j < n;
    const unsigned active = __ballot_sync(0xffffffffu, ok);
    uint32_t k = 0, v = 0, d = 0;
    if (ok) {
      k = keys_in[j];
      v = vals_in ? vals_in[j] : (uint32_t)j;  // no input values: the key's own index
      d = (k >> shift) & (kRDigits - 1);
    }
    const unsigned peers = __match_any_sync(0xffffffffu, ok ? d : 0xffffffffu) & active;
    if (ok) {
      const uint32_t pos = cnt[wid][d] + __popc(peers & lt);
      if (keys_out) keys_out[pos] = k;
      vals_out[pos] = v;
    }
    __syncwarp();
    if (ok && (peers & lt) == 0) cnt[wid][d] += __popc(peers);
    __syncwarp();
  }
}

__global__ void k_count_keys(const uint32_t* __restrict__ keys, int64_t n, uint32_t* __restrict__ cnt) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&cnt[keys[i]], 1u);
}

__device__ __forceinline__ void acc2(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  lo += (hi - (s - bb)) + (x - bb);
  hi = s;
}

// ---------------------------------------------------------------------------
// Face sums.  A link's gradient is linear in w = (v0 - x - t d) / (d . n) and in
// 1 / (d . n), so a face needs only W = sum of grad_q w and S = sum of
// grad_q / (d . n) over its links (4 numbers in 3D, 3 in 2D); the cross products
// with its edges follow once per face, in FP64.
//
// Links come in (cell, direction) order, in which a face's links are near one
// another: 256 consecutive links name about 10 different faces on the largest
// workload.  A warp groups its 256 links by face in shared memory (a hash of the
// face ids, ranks by __match_any_sync), adds each face's terms in double-float
// and sends one set of sums per face to global memory.  There the sums of a
// face's tiles are added as integers: the terms are fixed point with a scale per
// face and axis (the largest |grad_q / (c . n)| of its links, which a first kernel finds, the face's extent
// along the axis and a bound on its number of links), so the result does not depend on the order of the
// tiles.  With b bits for the number the spacing is 2^-(62 - b) of the bound: 2^-51 for a face of 10 cells
// across (b = 11; 22 for one of 600 cells).  With the number of all links and the largest axis for every face it was
// 2^-33 at 5e8 links: less than the double-float sums of a tile hold.  What depends on the face alone (the 9
// lines' 1 / (c . n), the bounds) is worked out once per face.
//
// Bound by instructions (the grouping, the positions, the double-float sums), at
// 9 bytes a link in the first kernel and 17 and the cell's in the second.  Before,
// a three-pass radix sort grouped all links by face and every face gathered its
// links from six arrays: 19.9 ms for 465 M links on 1.3 M faces (1.62 ms for
// 31.5 M on 82 K), now 7.6 ms (0.55 ms: 0.09 the scales, 0.42 the sums).  Tiles of
// 1,024 links per block of 8 warps lost to the barriers between the steps of the
// grouping (0.60 ms for the sums), and a sub-warp per face to the uneven numbers
// of links (0.69 ms).
// ---------------------------------------------------------------------------
constexpr int kSWarps = 4;                        // warps per block
constexpr int kSBlocks = 9;                       // blocks per SM (shared memory)
constexpr int kSItems = 8;                        // links per lane
constexpr int kSTile = 32 * kSItems;              // links per tile (a warp's)
constexpr uint32_t kSChunk = 12;                  // terms a lane adds in a row
constexpr int kSHashBits = 9;
constexpr int kSHash = 1 << kSHashBits;           // hash slots: a tile's faces always fit
static_assert(kSHash >= 2 * kSTile, "half of the slots stay free");
constexpr uint32_t kNonFinite = 1023u;            // scale key of a face with a non-finite term

// Lattice line of direction dir (its index in FaceLines::inv) and the sense along it.
template <int D>
__device__ __forceinline__ int line_of(int dir, bool& minus) {
  if constexpr (D == 3) {  // 2l + 1 and 2l + 2
    minus = (dir & 1) == 0;
    return (dir - 1) >> 1;
  } else {  // (1, 3), (2, 4), (5, 7), (6, 8)
    minus = ((dir - 1) & 2) != 0;
    return ((dir - 1) & 1) + (dir > 4 ? 2 : 0);
  }
}
static_assert(d3q19_c(1, 0) == -d3q19_c(2, 0) && d3q19_c(9, 1) == -d3q19_c(10, 1), "opposite directions are neighbours");
static_assert(d2q9_c(1, 0) == -d2q9_c(3, 0) && d2q9_c(6, 0) == -d2q9_c(8, 0) && d2q9_c(6, 1) == -d2q9_c(8, 1), "pairs");

// Power of two that brings the face normal's largest component to [1, 2).
__device__ __forceinline__ float normal_scale(float m) {
  const uint32_t eb = __float_as_uint(m) >> 23;
  return __uint_as_float((eb < 254u ? 254u - eb : 1u) << 23);
}

template <int D>
__device__ __forceinline__ void face_normal(const AdjointArgs& a, int64_t f, float* hi, float* lo) {
  if constexpr (D == 3) {
    const float4* R = reinterpret_cast<const float4*>(a.rec + f);
    const float4 r2 = __ldg(R + 2), r3 = __ldg(R + 3);
    hi[0] = r2.y, hi[1] = r2.z, hi[2] = r2.w;
    lo[0] = r3.x, lo[1] = r3.y, lo[2] = r3.z;
  } else {  // (e_y, -e_x): d x e = d . n
    hi[0] = a.X[3 * a.nf + f] - a.X[a.nf + f];
    hi[1] = a.X[f] - a.X[2 * a.nf + f];
    hi[2] = lo[0] = lo[1] = lo[2] = 0.f;
  }
}

template <bool MULTI>
__device__ __forceinline__ const GeomParams& face_geom(const AdjointArgs& a, int64_t f) {
  if constexpr (MULTI) return a.table[a.face_gid ? a.face_gid[f] : 0u];
  return a.g0;
}

// Per face what its links' terms need: v0, the lines' 1 / (c . n) of the scaled normal (0: parallel,
// no link), per axis the exponent r with |v0 - x - t d| < 2^r for every point x + t d of the face (twice its
// extent, since a certified hit may lie outside it by its rounding, and the rounding of t d), and the bits b
// of its number of links: a lattice line meets the face in at most four (the cells before and after the
// crossing, two of each where it is a node), and a convex region of area A and perimeter U holds at most
// A + U / 2 + 1 points of a unit lattice (Nosarzewska's bound; the face projected along the line, in units of h).
template <int D, bool MULTI>
__global__ void __launch_bounds__(256) k_face_lines(AdjointArgs a) {
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < a.nf; f += (int64_t)gridDim.x * blockDim.x) {
    const GeomParams& P = face_geom<MULTI>(a, f);
    const float h = fast_geom(P, P.n_levels - 1).h_hi;
    float hi[3], lo[3];
    face_normal<D>(a, f, hi, lo);
    const float scale = normal_scale(fmaxf(fmaxf(fabsf(hi[0]), fabsf(hi[1])), fabsf(hi[2])));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      hi[c] *= scale;
      lo[c] *= scale;
    }
    FaceLines L{};
    float e[2][3] = {};  // the edges from v0
#pragma unroll
    for (int c = 0; c < D; ++c) {
      L.v0[c] = a.X[(int64_t)c * a.nf + f];
      float m = 0.f;
#pragma unroll
      for (int k = 1; k < D; ++k) {
        e[k - 1][c] = a.X[(int64_t)(D * k + c) * a.nf + f] - L.v0[c];
        m = fmaxf(m, fabsf(e[k - 1][c]));
      }
      L.scale |= (__float_as_uint(fmaf(3.8e-6f, h, 2.0f * m)) >> 23) << (8 * c);
    }
    const float ih = 1.0f / h;
    float lines = 0.f;  // lattice lines through the face
    constexpr int kPlus3[9] = {1, 3, 5, 7, 9, 11, 13, 15, 17}, kPlus2[4] = {1, 2, 5, 6};
#pragma unroll
    for (int l = 0; l < (D == 3 ? 9 : 4); ++l) {
      float c[3];
#pragma unroll
      for (int q = 0; q < 3; ++q)
        c[q] = D == 3 ? (float)d3q19_c(kPlus3[l], q) : (q < 2 ? (float)d2q9_c(kPlus2[l < 4 ? l : 0], q) : 0.f);
      const float den = (c[0] * hi[0] + c[1] * hi[1] + c[2] * hi[2]) + (c[0] * lo[0] + c[1] * lo[1] + c[2] * lo[2]);
      L.inv[l] = den == 0.f ? 0.f : 1.0f / den;
      // the projection along the line: axes i < j with a part of c (i: the first of them or the only one), w the third
      if constexpr (D == 3) {
        const int n_axes = (c[0] != 0.f) + (c[1] != 0.f) + (c[2] != 0.f);
        const int i = c[0] != 0.f ? 0 : (c[1] != 0.f ? 1 : 2);
        const int j = n_axes == 2 ? (c[2] != 0.f ? 2 : 1) : (i + 1) % 3, w = 3 - i - j;
        const float s = n_axes == 2 ? c[i] * c[j] : 0.f;
        const float p0 = e[0][j] - s * e[0][i], p1 = e[1][j] - s * e[1][i], q0 = e[0][w], q1 = e[1][w];
        const float area = 0.5f * fabsf(p0 * q1 - q0 * p1), rim = fabsf(p0) + fabsf(q0) + fabsf(p1) + fabsf(q1) +
                                                                  fabsf(p1 - p0) + fabsf(q1 - q0);
        lines += area * ih * ih + 0.5f * rim * ih + 1.0f;
      } else if (l < 4) {
        lines += fabsf(c[0] * e[0][1] - c[1] * e[0][0]) * ih + 1.0f;
      }
    }
    const int bits = (int)(__float_as_uint(4.1f * lines + 4.0f) >> 23) - 126;
    L.scale |= (uint32_t)min(a.count_bits, bits) << 24;
    reinterpret_cast<FaceLines*>(a.face_lines)[f] = L;
  }
}

// Per face the largest bound on |grad_q / (c . n)|: key k > 0 says < 2^(k - 253), 0: no term but zero.
// Four links per thread, so that their chains of three loads overlap.
template <int D>
__global__ void __launch_bounds__(256) k_face_scale(AdjointArgs a) {
  constexpr int U = 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * U;
  for (int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) * U; w0 < a.n_links; w0 += stride) {
    const int64_t l0 = w0 + (threadIdx.x & 31);
    uint32_t f[U], key[U], old[U];
    float gq[U], inv[U];
    int dir[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t l = l0 + 32 * u;
      const bool ok = l < a.n_links;
      f[u] = ok ? a.link_face[l] : 0xffffffffu;
      gq[u] = ok ? a.grad_q[l] : 0.f;
      dir[u] = ok ? a.link_dir[l] : 1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      bool minus;
      const int line = line_of<D>(dir[u], minus);
      inv[u] = gq[u] != 0.f ? __ldg(a.face_lines[f[u]].inv + line) : 0.f;  // not zero: a link of this round
      old[u] = f[u] != 0xffffffffu ? __ldcg(a.face_key + f[u]) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t eg = (__float_as_uint(gq[u]) >> 23) & 255u, ei = (__float_as_uint(inv[u]) >> 23) & 255u;
      key[u] = inv[u] == 0.f ? 0u : (eg == 255u || ei == 255u || eg + ei > 504u ? kNonFinite : eg + ei + 1u);
      // one atomic per face and round: the links of a face come together, before any has raised its key
      const unsigned peers = __match_any_sync(0xffffffffu, f[u]);
      const uint32_t m = __reduce_max_sync(peers, key[u]);
      if ((threadIdx.x & 31) == __ffs(peers) - 1 && m > old[u]) atomicMax(a.face_key + f[u], m);
    }
  }
}

// The scale 2^-(key - 253) of a face's terms in two factors (both normal numbers): a term grad_q / (c . n)
// of the face is below 1 once multiplied by both.
__device__ __forceinline__ void term_scale(uint32_t key, float& s1, float& s2) {
  const int e = (int)key - 253, e1 = e >> 1;
  s1 = __uint_as_float((uint32_t)(127 - e1) << 23);
  s2 = __uint_as_float((uint32_t)(127 - (e - e1)) << 23);
}

struct SumSmem {
  // the hash (face ids, then their numbers in the tile) lives until every link knows its face's
  // number; the terms, ordered by face, then take its place
  float4 term[kSTile];
  uint32_t face[kSTile];
  uint16_t at[kSTile + 2];  // per face: its links so far, then its first place
};

template <int D, bool MULTI>
__global__ void __launch_bounds__(kSWarps * 32, kSBlocks) k_face_sums(AdjointArgs a) {
  constexpr int NC = D == 3 ? 64 : 16;
  constexpr int NV = D + 1;  // W and S
  __shared__ __align__(16) SumSmem s_all[kSWarps];
  const int lane = threadIdx.x & 31;
  SumSmem& sm = s_all[threadIdx.x >> 5];
  uint32_t* s_key = reinterpret_cast<uint32_t*>(sm.term);
  uint16_t* s_id = reinterpret_cast<uint16_t*>(s_key + kSHash);
  static_assert(sizeof(sm.term) >= kSHash * 6, "the hash fits the terms' place");
  const unsigned lt = (1u << lane) - 1u;
  const int64_t ntiles = (a.n_links + kSTile - 1) / kSTile;
  const int64_t nw = (int64_t)gridDim.x * kSWarps;
  for (int64_t tile = (int64_t)blockIdx.x * kSWarps + (threadIdx.x >> 5); tile < ntiles; tile += nw) {
    const int64_t l0 = tile * kSTile + lane;
#pragma unroll
    for (int i = 0; i < kSHash / 128; ++i)
      reinterpret_cast<uint4*>(s_key)[lane + 32 * i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncwarp();
    // each round's faces into the hash, one lane per face; kept: the face's number in the tile and the
    // link's rank among the face's links
    uint32_t pk[kSItems], nd = 0;
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
      const int64_t l = l0 + 32 * r;
      pk[r] = l < a.n_links ? a.link_face[l] : 0xffffffffu;
    }
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
      const uint32_t f = pk[r];
      const unsigned peers = __match_any_sync(0xffffffffu, f);
      const int lead = __ffs(peers) - 1;
      uint32_t h = 0;
      bool fresh = false;
      const bool ask = f != 0xffffffffu && lane == lead;
      if (ask) {
        h = (f * 2654435761u) >> (32 - kSHashBits);
        for (;;) {  // ends: at most kSTile of the kSHash slots are taken
          const uint32_t prev = atomicCAS(s_key + h, 0xffffffffu, f);
          fresh = prev == 0xffffffffu;
          if (fresh || prev == f) break;
          h = (h + 1) & (kSHash - 1);
        }
      }
      const unsigned fb = __ballot_sync(0xffffffffu, fresh);
      uint32_t id = 0, n = 0;
      if (ask) {
        if (fresh) {
          id = nd + __popc(fb & lt);
          s_id[h] = (uint16_t)id;
          sm.face[id] = f;
        } else {
          id = s_id[h];
          n = sm.at[id];
        }
        sm.at[id] = (uint16_t)(n + __popc(peers));
      }
      nd += __popc(fb);
      const uint32_t both = __shfl_sync(0xffffffffu, id | n << 16, lead);
      pk[r] = f == 0xffffffffu ? 0xffffffffu : both + ((uint32_t)__popc(peers & lt) << 16);
      __syncwarp();
    }
    // first place of each face
    uint32_t run = 0;
    for (uint32_t i0 = 0; i0 < nd; i0 += 32) {
      const uint32_t i = i0 + lane, n = i < nd ? sm.at[i] : 0u;
      const uint32_t incl = warp_inclusive_scan<uint32_t>(n);
      if (i < nd) sm.at[i] = (uint16_t)(run + incl - n);
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) sm.at[nd] = (uint16_t)run;
    __syncwarp();
    // the links' terms, in (face, link) order
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
      if (pk[r] == 0xffffffffu) continue;
      const int64_t l = l0 + 32 * r;
      const float gq = a.grad_q[l], t = a.link_q[l];
      const uint32_t cell = a.adj_cell[a.link_cell[l]];
      const int dir = a.link_dir[l];
      const uint32_t id = pk[r] & 0xffffu, f = sm.face[id];
      const GeomParams& P = face_geom<MULTI>(a, f);
      const int Lf = P.n_levels - 1;  // a face's links lie on the finest level of its geometry
      const FastGeom fg = fast_geom(P, Lf);
      const uint32_t blk = cell / NC, bit = cell % NC;
      const int32_t* bc = (MULTI ? a.level_blocks[Lf] : a.blocks) + (int64_t)blk * D;
      const FaceLines* FL = a.face_lines + f;
      const float4 v0 = __ldg(reinterpret_cast<const float4*>(FL));
      bool minus;
      const int line = line_of<D>(dir, minus);
      float inv = __ldg(FL->inv + line);
      inv = minus ? -inv : inv;
      float s1, s2;
      term_scale(__ldg(a.face_key + f), s1, s2);
      const float ginv = (gq * s1) * (inv * s2);
      const float V0[3] = {v0.x, v0.y, v0.z};
      const float hh = 0.5f * fg.h_hi, hl = 0.5f * fg.h_lo;
      float term[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < D; ++q) {
        // v0 - x with x = origin + k h / 2: the difference of the leading parts is as exact as the
        // result, the roundings of the parts follow it
        const float k = (float)(8 * bc[q] + 2 * (int)((bit >> (2 * q)) & 3u) + 1);
        float u, e, p, pe;
        df_two_sum(V0[q], -P.org_hi[q], u, e);
        df_two_prod(k, hh, p, pe);
        const float d = (u - p) + ((e - P.org_lo[q]) - fmaf(k, hl, pe));
        const float c = dir_comp(D == 3 ? (q == 0 ? kDirX : q == 1 ? kDirY : kDirZ) : (q == 0 ? kDir2X : kDir2Y), dir);
        term[q] = (d - t * (c * fg.h_hi)) * ginv;
      }
      term[D] = ginv;
      sm.term[sm.at[id] + (pk[r] >> 16)] = make_float4(term[0], term[1], term[2], term[3]);
    }
    __syncwarp();
    // the faces' terms in chunks of kSChunk, a lane per chunk (most tiles fit one round of 32): the lane
    // adds its terms in double-float, a segmented shuffle adds the chunks of a face into its first lane,
    // and that lane sends the sums
    for (uint32_t g0 = 0; g0 < nd; g0 += 32) {
      const uint32_t i = g0 + lane;
      const uint32_t nc = i < nd ? ((uint32_t)sm.at[i + 1] - sm.at[i] + kSChunk - 1) / kSChunk : 0u;
      const uint32_t incl = warp_inclusive_scan<uint32_t>(nc);
      const uint32_t first = incl - nc, total = __shfl_sync(0xffffffffu, incl, 31);
      for (uint32_t k0 = 0; k0 < total; k0 += 32) {
        // faces whose chunks start before / in this round
        const unsigned before = __popc(__ballot_sync(0xffffffffu, nc && first < k0));
        const unsigned heads = __reduce_or_sync(0xffffffffu, nc && first - k0 < 32u ? 1u << (first - k0) : 0u);
        const int j = (int)(before + __popc(heads & (lt | (1u << lane)))) - 1;
        const uint32_t fj = __shfl_sync(0xffffffffu, first, j);
        const bool ok = k0 + lane < total;
        float hi[NV], lo[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) hi[v] = lo[v] = 0.f;
        if (ok) {
          const uint32_t end = sm.at[g0 + j + 1];
          const uint32_t e0 = sm.at[g0 + j] + (k0 + lane - fj) * kSChunk;
          const uint32_t e1 = e0 + kSChunk < end ? e0 + kSChunk : end;
          for (uint32_t e = e0; e < e1; ++e) {
            const float4 x = sm.term[e];
            const float y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int v = 0; v < NV; ++v) acc2(hi[v], lo[v], y[v]);
          }
        }
        // lanes [lane, last] hold chunks of this lane's face
        const uint32_t after = heads & ~(lt | (1u << lane));
        const uint32_t n_here = total - k0 < 32u ? total - k0 : 32u;
        const int last = (after ? __ffs(after) - 1 : (int)n_here) - 1;
        for (int o = 1; o < 32; o <<= 1) {
          if (!__any_sync(0xffffffffu, lane + o <= last)) break;
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float ph = __shfl_down_sync(0xffffffffu, hi[v], o);
            const float pl = __shfl_down_sync(0xffffffffu, lo[v], o);
            if (lane + o <= last) {
              acc2(hi[v], lo[v], ph);
              lo[v] += pl;
            }
          }
        }
        if (ok && (lane == 0 || ((heads >> lane) & 1u))) {
          const uint32_t f = sm.face[g0 + j], key = __ldg(a.face_key + f);
          if (key != 0u && key != kNonFinite) {
            const uint32_t sc = __ldg(&a.face_lines[f].scale);
            const int b = (int)(sc >> 24), k = 62 - b;
            // no more than so many bounds (t of a face nearly along its line may be off): the sums stay below 2^63
            const uint32_t cnt = min((uint32_t)(sm.at[g0 + j + 1] - sm.at[g0 + j]), 1u << min(b, 16));
            const long long lim = (long long)cnt << k;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
              // terms below 1 (W: below 2^r)
              const int r = v < D ? (int)((sc >> (8 * v)) & 255u) - 126 : 0;
              const double x = ((double)hi[v] + (double)lo[v]) * __hiloint2double((1023 + k - r) << 20, 0);
              const long long n = min(max(__double2ll_rn(x), -lim), lim);
              if (n) atomicAdd(a.face_acc + (int64_t)f * NV + v, (unsigned long long)n);
            }
          }
        }
      }
    }
    __syncwarp();
  }
}

// grad_face[f][k][c] from the face's sums, in FP64.
template <int D, bool MULTI>
__global__ void __launch_bounds__(256) k_face_grad(AdjointArgs a) {
  constexpr int NV = D + 1;
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < a.nf; f += (int64_t)gridDim.x * blockDim.x) {
    float* out = a.grad_face + f * D * D;
    const uint32_t key = a.n_links > 0 ? a.face_key[f] : 0u;
    if (key == 0u || key == kNonFinite) {
#pragma unroll
      for (int j = 0; j < D * D; ++j) out[j] = key == 0u ? 0.f : __int_as_float(0x7fffffff);
      continue;
    }
    const GeomParams& P = face_geom<MULTI>(a, f);
    const FastGeom fg = fast_geom(P, P.n_levels - 1);
    float nh[3], nl[3];
    face_normal<D>(a, f, nh, nl);
    const float scale = normal_scale(fmaxf(fmaxf(fabsf(nh[0]), fabsf(nh[1])), fabsf(nh[2])));
    // grad_q / (d . n) of the sums: the terms left out h, the power of two of the scaled normal and the key's
    const double unit = scalbn((double)scale / ((double)fg.h_hi + (double)fg.h_lo), (int)key - 253);
    const uint32_t sc = a.face_lines[f].scale;
    const int k = 62 - (int)(sc >> 24);
    double v[4];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int r = j < D ? (int)((sc >> (8 * j)) & 255u) - 126 : 0;
      v[j] = (double)(long long)a.face_acc[f * NV + j] * __hiloint2double((1023 - k + r) << 20, 0) * unit;
    }
    double X[D][D];
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int c = 0; c < D; ++c) X[k][c] = (double)a.X[(int64_t)(D * k + c) * a.nf + f];
    if constexpr (D == 3) {
      const double e1[3] = {X[1][0] - X[0][0], X[1][1] - X[0][1], X[1][2] - X[0][2]};
      const double e2[3] = {X[2][0] - X[0][0], X[2][1] - X[0][1], X[2][2] - X[0][2]};
      const double g1[3] = {e2[1] * v[2] - e2[2] * v[1], e2[2] * v[0] - e2[0] * v[2], e2[0] * v[1] - e2[1] * v[0]};
      const double g2[3] = {v[1] * e1[2] - v[2] * e1[1], v[2] * e1[0] - v[0] * e1[2], v[0] * e1[1] - v[1] * e1[0]};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        out[c] = (float)(((double)nh[c] + (double)nl[c]) * v[3] - g1[c] - g2[c]);
        out[3 + c] = (float)g1[c];
        out[6 + c] = (float)g2[c];
      }
    } else {
      const double e0 = X[1][0] - X[0][0], e1 = X[1][1] - X[0][1];
      out[0] = (float)(e1 * v[2] + v[1]);
      out[1] = (float)(-e0 * v[2] - v[0]);
      out[2] = (float)-v[1];
      out[3] = (float)v[0];
    }
  }
}

// One thread per vertex: sum of its face corners' gradients in ascending (face, corner) order.
template <int D>
__global__ void k_vertex_grad(const float* __restrict__ grad_face, const uint32_t* __restrict__ vert_off,
                              const uint32_t* __restrict__ vert_corners, int64_t nv, float* __restrict__ out) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
    float hi[D], lo[D];
#pragma unroll
    for (int c = 0; c < D; ++c) hi[c] = lo[c] = 0.f;
    for (uint32_t s = vert_off[v]; s < vert_off[v + 1]; ++s) {
      const uint32_t corner = vert_corners[s];  // f * D + k
#pragma unroll
      for (int c = 0; c < D; ++c) acc2(hi[c], lo[c], grad_face[(int64_t)corner * D + c]);
    }
#pragma unroll
    for (int c = 0; c < D; ++c) out[v * D + c] = hi[c] + lo[c];
  }
}

inline int grid_1d(int64_t n, int threads = 256) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  const int64_t cap = (int64_t)current_sm_count() * 32;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace

size_t radix_sort_scratch_bytes(int64_t n) {
  const int64_t tiles = (n + kRTile - 1) / kRTile;
  const int64_t nh = (tiles > 0 ? tiles : 1) * kRDigits;
  // hist + offsets (nh + 1 each) + ping-pong keys/values (2n each) + scan scratch
  return (size_t)(2 * (nh + 1)) * 4 + (size_t)(4 * (n > 0 ? n : 1)) * 4 + scan_u32_scratch_bytes(nh) + 256;
}

int launch_stable_sort(const uint32_t* keys, int64_t n, int key_bits, uint32_t* sorted_keys, uint32_t* sorted_vals,
                       const uint32_t* vals_in, void* scratch, uint64_t* total, unsigned* err, cudaStream_t st) {
  // vals_in == nullptr: values are 0..n-1
  if (n <= 0) return 0;
  const int64_t tiles = (n + kRTile - 1) / kRTile;
  const int64_t nh = tiles * kRDigits;
  char* s = static_cast<char*>(scratch);
  uint32_t* hist = reinterpret_cast<uint32_t*>(s);
  uint32_t* offs = hist + (nh + 1);
  uint32_t* ka = offs + (nh + 1);
  uint32_t* va = ka + n;
  uint32_t* kb = va + n;
  uint32_t* vb = kb + n;
  void* scan_scr = reinterpret_cast<void*>(((uintptr_t)(vb + n) + 255) & ~(uintptr_t)255);
  int launches = 0;
  int passes = (key_bits + kRBits - 1) / kRBits;
  if (passes < 1) passes = 1;
  // the first pass reads the caller's keys (and values, or the indices), the last writes the
  // caller's outputs; the passes between ping-pong through the scratch
  const uint32_t* kin = keys;
  const uint32_t* vin = vals_in;
  for (int p = 0; p < passes; ++p) {
    const int shift = p * kRBits;
    const bool last = p == passes - 1;
    uint32_t* kout = last ? sorted_keys : (p % 2 == 0 ? kb : ka);
    uint32_t* vout = last ? sorted_vals : (p % 2 == 0 ? vb : va);
    k_radix_hist<<<(unsigned)tiles, kRThreads, 0, st>>>(kin, n, shift, hist, tiles);
    launches += 1 + launch_scan_u32(hist, offs, nh, total, scan_scr, err, st);
    k_radix_scatter<<<(unsigned)tiles, kRThreads, 0, st>>>(kin, vin, n, shift, offs, tiles, kout, vout);
    ++launches;
    kin = kout;
    vin = vout;
  }
  return launches;
}

int launch_count_keys(const uint32_t* keys, int64_t n, uint32_t* cnt, cudaStream_t st) {
  if (n <= 0) return 0;
  k_count_keys<<<grid_1d(n), 256, 0, st>>>(keys, n, cnt);
  return 1;
}

namespace {
template <int D, bool MULTI>
int face_grad(const AdjointArgs& a, cudaStream_t st) {
  int k = 1;
  if (a.n_links > 0) {
    cudaMemsetAsync(a.face_key, 0, sizeof(uint32_t) * (size_t)a.nf, st);
    cudaMemsetAsync(a.face_acc, 0, sizeof(unsigned long long) * (size_t)(D + 1) * (size_t)a.nf, st);
    const int64_t cap = (int64_t)current_sm_count() * kSBlocks;  // resident at once
    const int64_t blocks = (a.n_links + kSTile * kSWarps - 1) / (kSTile * kSWarps);
    k_face_lines<D, MULTI><<<grid_1d(a.nf), 256, 0, st>>>(a);
    k_face_scale<D><<<grid_1d((a.n_links + 3) / 4), 256, 0, st>>>(a);
    k_face_sums<D, MULTI><<<(unsigned)(blocks < cap ? blocks : cap), kSWarps * 32, 0, st>>>(a);
    k += 3;
  }
  k_face_grad<D, MULTI><<<grid_1d(a.nf), 256, 0, st>>>(a);
  return k;
}
}  // namespace

int launch_face_grad(const AdjointArgs& a, cudaStream_t st) {
  if (a.nf <= 0) return 0;
  if (a.dim == 3) return a.table ? face_grad<3, true>(a, st) : face_grad<3, false>(a, st);
  return a.table ? face_grad<2, true>(a, st) : face_grad<2, false>(a, st);
}

int launch_vertex_grad(int dim, const float* grad_face, const uint32_t* vert_off, const uint32_t* vert_corners,
                       int64_t nv, float* out, cudaStream_t st) {
  if (nv <= 0) return 0;
  if (dim == 3)
    k_vertex_grad<3><<<grid_1d(nv), 256, 0, st>>>(grad_face, vert_off, vert_corners, nv, out);
  else
    k_vertex_grad<2><<<grid_1d(nv), 256, 0, st>>>(grad_face, vert_off, vert_corners, nv, out);
  return 1;
}

}  // namespace amr
