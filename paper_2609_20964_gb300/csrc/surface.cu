// Iso-value (Sec. 2.4, Eq. 27), marching cubes (Eq. 28), exact signed distance
// to the triangles (Eqs. 29-34) and stencil normals (after Eq. 32).
//
// Iso-value: c = mean over the finite input points of chi interpolated
// trilinearly between cell centres (positions clamped into the node hull),
// accumulated in FP64 with a fixed-order two-pass reduction.
//
// Marching cubes on the (res-1)^3 cubes between cell centres; a node is inside
// iff chi < c.  Cubes are processed in 4^3 bricks (one CTA each): a count pass,
// a scan over bricks, and an emit pass that writes each brick's triangles
// contiguously.  Each triangle stores its three vertices and the global ids of
// the edges they sit on (3 * linear index of the lower node + axis).  A shared
// edge's vertex is computed from the same two chi values by every cube, so it
// is bit-identical across cubes (watertight).
//
// The case table is derived at load time from the face-consistent rule: on a
// face with four crossed edges every inside corner is cut off by its own
// segment; segments are directed with the inside corners on their right seen
// from outside the cube, chained into loops (listed by smallest edge id) and
// fanned from their first edge, so triangles face from inside to outside.
//
// Distance: exact minimum over all triangles of the point-to-triangle distance
// (closest point by Voronoi regions of the triangle: vertices, edges, face —
// the method of Ericson, Real-Time Collision Detection, 5.1.5), found through
// an implicit octree over the bricks whose nodes bound their triangles by
// fitted solid cylinders (pucks), pruned only by lower bounds of them.  Grid
// nodes are searched on nested lattices, by blocks of nodes that share a walk;
// off-grid queries 32 a warp.  Sign: +1 where
// chi >= c, -1 where chi < c (the marching-cubes surface separates the two node
// classes, so this is the parity of crossings of any ray from the node).
#include <math.h>
#include <stddef.h>

#include <algorithm>

#include "wgeo_internal.cuh"

namespace wgeo {

__constant__ int c_mc_count[256];
__constant__ signed char c_mc_tris[256][kMaxTriPerCube][3];

// ---------------------------------------------------------------- host: table
namespace {

struct EdgeGeo {
  int axis;
  int c0, c1;  // lower / upper corner
};

void corner_xyz(int k, double* p) {
  p[0] = k & 1;
  p[1] = (k >> 1) & 1;
  p[2] = (k >> 2) & 1;
}

EdgeGeo edge_geo(int e) {
  EdgeGeo g;
  g.axis = e / 4;
  const int a = e % 4;
  int lo[3] = {0, 0, 0};
  const int o0 = (g.axis == 0) ? 1 : 0;
  const int o1 = (g.axis == 2) ? 1 : 2;
  lo[o0] = a & 1;
  lo[o1] = a >> 1;
  g.c0 = lo[0] + 2 * lo[1] + 4 * lo[2];
  lo[g.axis] = 1;
  g.c1 = lo[0] + 2 * lo[1] + 4 * lo[2];
  return g;
}

int table_for_case(int cs, int tris[kMaxTriPerCube * 2][3]) {
  bool in[8];
  for (int k = 0; k < 8; ++k) in[k] = (cs >> k) & 1;
  bool crossed[12];
  for (int e = 0; e < 12; ++e) {
    EdgeGeo g = edge_geo(e);
    crossed[e] = in[g.c0] != in[g.c1];
  }
  int next[12];
  for (int e = 0; e < 12; ++e) next[e] = -1;
  for (int axis = 0; axis < 3; ++axis) {
    for (int side = 0; side < 2; ++side) {
      double nrm[3] = {0, 0, 0};
      nrm[axis] = side ? 1.0 : -1.0;
      int fe[4], nfe = 0;
      for (int e = 0; e < 12; ++e) {
        EdgeGeo g = edge_geo(e);
        double p0[3];
        corner_xyz(g.c0, p0);
        if (g.axis != axis && (int)p0[axis] == side && crossed[e]) fe[nfe++] = e;
      }
      auto mid = [](int e, double* m) {
        EdgeGeo g = edge_geo(e);
        double a[3], b[3];
        corner_xyz(g.c0, a);
        corner_xyz(g.c1, b);
        for (int i = 0; i < 3; ++i) m[i] = 0.5 * (a[i] + b[i]);
      };
      auto add_seg = [&](int a, int b, const double* ref) {
        double pa[3], pb[3];
        mid(a, pa);
        mid(b, pb);
        const double d[3] = {pb[0] - pa[0], pb[1] - pa[1], pb[2] - pa[2]};
        const double left[3] = {nrm[1] * d[2] - nrm[2] * d[1], nrm[2] * d[0] - nrm[0] * d[2],
                                nrm[0] * d[1] - nrm[1] * d[0]};
        double s = 0;
        for (int i = 0; i < 3; ++i) s += left[i] * (ref[i] - 0.5 * (pa[i] + pb[i]));
        if (s > 0) std::swap(a, b);
        next[a] = b;
      };
      if (nfe == 2) {
        double ref[3] = {0, 0, 0};
        int cnt = 0;
        for (int k = 0; k < 8; ++k) {
          double p[3];
          corner_xyz(k, p);
          if ((int)p[axis] == side && in[k]) {
            for (int i = 0; i < 3; ++i) ref[i] += p[i];
            ++cnt;
          }
        }
        for (int i = 0; i < 3; ++i) ref[i] /= cnt;
        add_seg(fe[0], fe[1], ref);
      } else if (nfe == 4) {
        for (int k = 0; k < 8; ++k) {
          double p[3];
          corner_xyz(k, p);
          if ((int)p[axis] != side || !in[k]) continue;
          int adj[2], na = 0;
          for (int q = 0; q < 4; ++q) {
            EdgeGeo g = edge_geo(fe[q]);
            if (g.c0 == k || g.c1 == k) adj[na++] = fe[q];
          }
          add_seg(adj[0], adj[1], p);
        }
      }
    }
  }
  int nt = 0;
  bool seen[12] = {false};
  for (int e = 0; e < 12; ++e) {
    if (!crossed[e] || seen[e]) continue;
    int loop[12], nl = 0;
    int f = e;
    do {
      loop[nl++] = f;
      seen[f] = true;
      f = next[f];
    } while (f != e && f >= 0 && nl < 12);
    for (int k = 1; k + 1 < nl; ++k) {
      tris[nt][0] = loop[0];
      tris[nt][1] = loop[k];
      tris[nt][2] = loop[k + 1];
      ++nt;
    }
  }
  return nt;
}

}  // namespace

void host_mc_table(int* counts, int* tris) {
  for (int cs = 0; cs < 256; ++cs) {
    int t[kMaxTriPerCube * 2][3];
    const int nt = table_for_case(cs, t);
    counts[cs] = nt;
    for (int k = 0; k < kMaxTriPerCube; ++k)
      for (int v = 0; v < 3; ++v) tris[(cs * kMaxTriPerCube + k) * 3 + v] = (k < nt) ? t[k][v] : -1;
  }
}

int upload_mc_table() {
  int counts[256];
  int tris[256 * kMaxTriPerCube * 3];
  host_mc_table(counts, tris);
  signed char t8[256 * kMaxTriPerCube * 3];
  for (int i = 0; i < 256 * kMaxTriPerCube * 3; ++i) t8[i] = (signed char)tris[i];
  for (int i = 0; i < 256; ++i)
    if (counts[i] > kMaxTriPerCube) return WGEO_ERR_INVALID_ARG;
  WGEO_CUDA_TRY(cudaMemcpyToSymbol(c_mc_count, counts, sizeof(counts)));
  WGEO_CUDA_TRY(cudaMemcpyToSymbol(c_mc_tris, t8, sizeof(t8)));
  return WGEO_OK;
}

// ---------------------------------------------------------------- device
namespace {

struct SurfParams {
  double lo[3];
  double h;
  int res;
  int nb;        // bricks per axis
  float sc, us;  // box units -> the search's units (search_scale), and back
};

SurfParams surf_params(const wgeo_handle* h, int res) {
  SurfParams g;
  for (int a = 0; a < 3; ++a) g.lo[a] = h->lo[a];
  g.h = h->h;
  g.res = res;
  g.nb = div_up(res - 1, kBrick);
  g.sc = search_scale(h->h);
  g.us = 1.f / g.sc;
  return g;
}

__device__ __forceinline__ int64_t lin3(int i, int j, int k, int n) {
  return ((int64_t)k * n + j) * n + i;
}

__global__ void isovalue_kernel(const float* __restrict__ pts, int64_t n, const int* __restrict__ pcell,
                                const float* __restrict__ chi, SurfParams g,
                                double* __restrict__ partials) {
  __shared__ double red[32];
  double s = 0.0, cnt = 0.0;
  const int res = g.res;
  // lo and 1/h as float-float pairs: the cells and weights come from
  // node_coord_ff, the FP64 pipe only sums
  float lo_hi[3], lo_lo[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo_hi[a] = (float)g.lo[a];
    lo_lo[a] = (float)(g.lo[a] - (double)lo_hi[a]);
  }
  const double ih = 1.0 / g.h;
  const float ih_hi = (float)ih, ih_lo = (float)(ih - (double)ih_hi);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (pcell[i] < 0) continue;
    int i0[3];
    float t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      node_cell_ff(node_coord_ff(pts[3 * i + a], lo_hi[a], lo_lo[a], ih_hi, ih_lo), res, i0[a], t[a]);
    // the interpolated value in float-float (weights and products in float)
    float2 v = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
      const float w = (dx ? t[0] : 1.f - t[0]) * (dy ? t[1] : 1.f - t[1]) * (dz ? t[2] : 1.f - t[2]);
      v = ff_add_f(v, w * chi[lin3(i0[0] + dx, i0[1] + dy, i0[2] + dz, res)]);
    }
    s += (double)v.x + (double)v.y;
    cnt += 1.0;
  }
  s = block_sum<256>(s, red);
  cnt = block_sum<256>(cnt, red);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = s;
    partials[2 * blockIdx.x + 1] = cnt;
  }
}

__global__ void isovalue_finalize_kernel(const double* __restrict__ partials, int nblocks, DevState* st) {
  __shared__ double red[32];
  double s = 0.0, cnt = 0.0;
  for (int i = threadIdx.x; i < nblocks; i += blockDim.x) {
    s += partials[2 * i];
    cnt += partials[2 * i + 1];
  }
  s = block_sum<1024>(s, red);
  cnt = block_sum<1024>(cnt, red);
  if (threadIdx.x == 0) {
    st->c = cnt > 0.0 ? s / cnt : 0.0;
    float cu = (float)st->c;
    if ((double)cu < st->c) cu = nextafterf(cu, INFINITY);
    st->c_up = cu;
    st->npts = (long long)cnt;
  }
}

// Case code of a cube: bit q set when corner q is inside (chi < c, tested as
// chi < c_up, the smallest float >= c).
__device__ __forceinline__ int cube_code(const float* __restrict__ chi, int i, int j, int k, int n, float c_up) {
  int code = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float v = chi[lin3(i + (q & 1), j + ((q >> 1) & 1), k + (q >> 2), n)];
    code |= (v < c_up) ? (1 << q) : 0;
  }
  return code;
}

// Cube (i,j,k) of a 4^3 brick handled by thread t: Morton order inside the
// brick, so the 8 cubes of each 2^3 sub-brick (an octree leaf) are the
// contiguous threads 8k..8k+7 and their triangles are contiguous in memory.
__device__ __forceinline__ void brick_cube(int t, int& lx, int& ly, int& lz) {
  lx = (t & 1) | (((t >> 3) & 1) << 1);
  ly = ((t >> 1) & 1) | (((t >> 4) & 1) << 1);
  lz = ((t >> 2) & 1) | (((t >> 5) & 1) << 1);
}

// Inside bits of the nodes (chi < c, tested as chi < c_up), 32 per word
// along x: word w of row (j, k) holds x = 32 w .. 32 w + 31 (bits past the
// grid's edge clear), at bits[(k n + j) nw + w], nw = ceil(n / 32).  One warp
// per word: coalesced reads of chi, one ballot.
constexpr int kBitRows = 8;   // rows per warp in mc_bits_kernel (loads in flight per lane)
__global__ void __launch_bounds__(256) mc_bits_kernel(const float* __restrict__ chi, int n, int nw,
                                                      const DevState* __restrict__ st,
                                                      unsigned* __restrict__ bits) {
  // block (32, 8): warp y takes word blockIdx.x of kBitRows consecutive rows
  // (k n + j), their loads issued together
  const int row0 = (blockIdx.y * 8 + threadIdx.y) * kBitRows;
  const int x = 32 * blockIdx.x + threadIdx.x;
  const float c_up = st->c_up;
  float v[kBitRows];
#pragma unroll
  for (int r = 0; r < kBitRows; ++r)
    v[r] = (x < n && row0 + r < n * n) ? chi[(int64_t)(row0 + r) * n + x] : INFINITY;
#pragma unroll
  for (int r = 0; r < kBitRows; ++r) {
    const unsigned m = __ballot_sync(0xffffffffu, v[r] < c_up);
    if (threadIdx.x == 0 && row0 + r < n * n) bits[(row0 + r) * nw + blockIdx.x] = m;
  }
}

// Four 4^3 bricks of cubes per CTA (consecutive brick indices), 64 threads
// (two warps) per brick.
constexpr int kMcBricks = 4;

// Triangles per 4^3 brick from the inside bits.  A thread takes 32 cubes
// along x (one word) of one cube row: the cube's 8 corner bits are bit b and
// bit b + 1 of the four node rows (j, k), (j + 1, k), (j, k + 1), (j + 1,
// k + 1), so the cubes that the surface crosses (corners neither all inside
// nor all outside) come out of eight word operations, and only those look up
// their case.  The 16 threads of one word and brick row (j, k mod 4) are 16
// consecutive lanes; their counts for the word's 8 bricks are summed by
// shuffles (only where a cube is crossed) and written by the first.
__global__ void mc_count_kernel(const unsigned* __restrict__ bits, SurfParams g, int nw,
                                int* __restrict__ brick_count) {
  const int n = g.res, m = n - 1, nb = g.nb;
  const int cw = (m + 31) / 32;              // cube words per row
  const int64_t groups = (int64_t)cw * nb * nb;
  const int lane = threadIdx.x & 31, sub = lane & 15;
  // warp-uniform trip count (two groups per warp): every lane reaches the shuffles
  for (int64_t wb = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; 2 * wb < groups;
       wb += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t gi = 2 * wb + (lane >> 4);   // (w, by, bz) of this half-warp
    const bool ok = gi < groups;
    const int w = ok ? (int)(gi % cw) : 0;
    const int by = ok ? (int)((gi / cw) % nb) : 0, bz = ok ? (int)(gi / ((int64_t)cw * nb)) : 0;
    const int j = 4 * by + (sub & 3), k = 4 * bz + (sub >> 2);
    // triangle counts of the word's 8 bricks, 16 bits each (at most 320 per
    // brick after the half-warp sum): bricks 0-3 in c03, 4-7 in c47
    unsigned long long c03 = 0ull, c47 = 0ull;
    bool any = false;
    if (ok && j < m && k < m) {
      unsigned A[4], B[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int64_t row = (int64_t)(k + (r >> 1)) * n + (j + (r & 1));
        const unsigned lo = bits[row * nw + w];
        const unsigned hi = (w + 1 < nw) ? bits[row * nw + w + 1] : 0u;
        A[r] = lo;
        B[r] = (lo >> 1) | (hi << 31);
      }
      const unsigned all_in = A[0] & A[1] & A[2] & A[3] & B[0] & B[1] & B[2] & B[3];
      const unsigned all_out = ~(A[0] | A[1] | A[2] | A[3] | B[0] | B[1] | B[2] | B[3]);
      const int xv = m - 32 * w;             // cubes of this word inside the grid
      const unsigned valid = xv >= 32 ? 0xffffffffu : ((1u << xv) - 1u);
      unsigned mixed = ~(all_in | all_out) & valid;
      any = mixed != 0u;
      while (mixed) {
        const int b = __ffs(mixed) - 1;
        mixed &= mixed - 1u;
        // corner q = (x offset q & 1, y offset q >> 1 & 1, z offset q >> 2)
        int code = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const unsigned word = (q & 1) ? B[q >> 1] : A[q >> 1];
          code |= (int)((word >> b) & 1u) << q;
        }
        const unsigned long long add = (unsigned long long)c_mc_count[code] << (16 * ((b >> 2) & 3));
        if (b < 16) c03 += add; else c47 += add;
      }
    }
    // sum over the 16 lanes of the half-warp (both halves take part)
    if (__any_sync(0xffffffffu, any)) {
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        c03 += __shfl_xor_sync(0xffffffffu, c03, o);
        c47 += __shfl_xor_sync(0xffffffffu, c47, o);
      }
    }
    if (ok && sub == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int bx = 8 * w + q;
        const unsigned long long v = q < 4 ? c03 : c47;
        if (bx < nb) brick_count[((int64_t)bz * nb + by) * nb + bx] = (int)((v >> (16 * (q & 3))) & 0xffffull);
      }
    }
  }
}

// The triangle total and its status, and the node coordinates per axis in the
// search's units (it reads them instead of forming them in FP64 at every node).
__global__ void mc_total_kernel(const int* __restrict__ brick_off, int nbricks, int64_t cap,
                                int* __restrict__ leaf_off, DevState* st, SurfParams g, float* __restrict__ axis) {
  for (int t = threadIdx.x; t < 3 * g.res; t += blockDim.x) {
    const int a = t / g.res, i = t - a * g.res;
    axis[t] = (float)(g.lo[a] + (i + 0.5) * g.h) * g.sc;
  }
  if (threadIdx.x != 0) return;
  const long long T = brick_off[nbricks];
  st->ntris = T;
  leaf_off[8 * (int64_t)nbricks] = brick_off[nbricks];
  if (T > cap) atomicOr(&st->status, WGEO_STATUS_MESH_CAPACITY);
  if (T == 0) atomicOr(&st->status, WGEO_STATUS_EMPTY_SURFACE);
}

__device__ __forceinline__ void edge_lower_offset(int e, int& ox, int& oy, int& oz, int& axis) {
  axis = e >> 2;
  const int a = e & 3;
  int o[3] = {0, 0, 0};
  const int o0 = (axis == 0) ? 1 : 0;
  const int o1 = (axis == 2) ? 1 : 2;
  o[o0] = a & 1;
  o[o1] = a >> 1;
  ox = o[0];
  oy = o[1];
  oz = o[2];
}

// Edges of a brick's cubes, by the local coordinates (0..kBrick) of their
// lower end node: along the edge's axis 0..kBrick-1, across it 0..kBrick.
constexpr int kEdgesPerAxis = kBrick * (kBrick + 1) * (kBrick + 1);
constexpr int kBrickEdges = 3 * kEdgesPerAxis;
constexpr int div_up_c(int a, int b) { return (a + b - 1) / b; }
__device__ __forceinline__ int brick_edge_slot(int ax, int ex, int ey, int ez) {
  const int u = ax == 0 ? ex : (ax == 1 ? ey : ez);   // along the axis
  const int v = ax == 0 ? ey : ex;                     // the first other axis
  const int w = ax == 2 ? ey : ez;                     // the second
  return ax * kEdgesPerAxis + (w * (kBrick + 1) + v) * kBrick + u;
}
__device__ __forceinline__ void brick_edge_of_slot(int sl, int& ax, int& ex, int& ey, int& ez) {
  ax = sl / kEdgesPerAxis;
  const int r = sl - ax * kEdgesPerAxis;
  const int u = r % kBrick, v = (r / kBrick) % (kBrick + 1), w = r / (kBrick * (kBrick + 1));
  ex = ax == 0 ? u : v;
  ey = ax == 1 ? u : (ax == 0 ? v : w);
  ez = ax == 2 ? u : w;
}

// Emits each brick's triangles contiguously (Morton cube order) and the
// triangle offset of each of its 8 sub-bricks (octree leaves).  A vertex is
// placed in FP64 from the cube edge's two indicator values (Eq. 28); with
// `chiff` (the refined float-float indicator, current buffer chosen by the
// solve's index) those values carry the float-float low parts, so the vertex
// follows the refined solution rather than its float32 copy.  tris holds the
// vertices rounded to float32; tris_lo (may be null) their residuals
// (double vertex - float vertex, rounded to float), so that hi + lo keeps
// about 48 bits: near-tie decisions and the adjoint's closest points use it.
// The bricks with triangles, listed (one atomic per warp); an empty brick
// writes its 8 leaf offsets here (all equal to its triangle offset).
__global__ void mc_live_kernel(const int* __restrict__ brick_off, int nbr, int* __restrict__ leaf_off,
                               int* __restrict__ list, unsigned* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  // warp-uniform trip count: every lane reaches the ballot
  for (int b0 = blockIdx.x * blockDim.x; b0 < nbr; b0 += gridDim.x * blockDim.x) {
    const int br = b0 + threadIdx.x;
    bool live = false;
    if (br < nbr) {
      const int base = brick_off[br];
      live = brick_off[br + 1] != base;
      if (!live) {
        int4* lo4 = reinterpret_cast<int4*>(leaf_off + 8 * (int64_t)br);
        lo4[0] = make_int4(base, base, base, base);
        lo4[1] = make_int4(base, base, base, base);
      }
    }
    const unsigned mk = __ballot_sync(0xffffffffu, live);
    if (mk) {
      const int leader = __ffs(mk) - 1;
      unsigned at = 0;
      if (lane == leader) at = atomicAdd(count, (unsigned)__popc(mk));
      at = __shfl_sync(0xffffffffu, at, leader);
      if (live) list[at + __popc(mk & ((1u << lane) - 1u))] = br;
    }
  }
}

__global__ void __launch_bounds__(64 * kMcBricks) mc_emit_kernel(const float* __restrict__ chi, ChiFF chiff,
                                                                 SurfParams g, const DevState* __restrict__ st,
                                                                 const int* __restrict__ brick_off, int64_t cap,
                                                                 const int* __restrict__ live_list,
                                                                 const unsigned* __restrict__ nlive,
                                                                 Tri* __restrict__ tris, Tri* __restrict__ tris_lo,
                                                                 int* __restrict__ leaf_off,
                                                                 unsigned* __restrict__ leaf_cnt) {
  const int grp = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = g.res, m = n - 1;
  const double c = st->c;
  const float c_up = st->c_up;
  const float2* __restrict__ xff = chiff.p[0] ? chiff.p[st->fwd.xidx] : nullptr;
  __shared__ int wt[2 * kMcBricks];
  // the brick's crossing edges (listed first, so that the FP64 placement
  // runs on full warps), and its vertices, one per crossing edge (hi with
  // the edge id in .w; lo)
  __shared__ short s_cross[kMcBricks][kBrickEdges];
  __shared__ int s_ncross[kMcBricks];
  __shared__ float4 s_vh[kMcBricks][kBrickEdges], s_vl[kMcBricks][kBrickEdges];
  const unsigned count = *nlive;
  // persistent: kMcBricks listed bricks per iteration (the same trip count in
  // the whole CTA: every thread reaches the barriers)
  for (unsigned b0 = blockIdx.x * kMcBricks; b0 < count; b0 += gridDim.x * kMcBricks) {
    const bool live = b0 + grp < count;
    const int br = live ? live_list[b0 + grp] : 0;
    const int base = live ? brick_off[br] : 0;
    const int bx = br % g.nb, by = (br / g.nb) % g.nb, bz = br / (g.nb * g.nb);
    int i = 0, j = 0, k = 0;
    int code = 0, cnt = 0;
    if (live) {
      int lx, ly, lz;
      brick_cube(t, lx, ly, lz);
      i = bx * kBrick + lx;
      j = by * kBrick + ly;
      k = bz * kBrick + lz;
      if (i < m && j < m && k < m) {
        code = cube_code(chi, i, j, k, n, c_up);
        cnt = c_mc_count[code];
      }
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int tt = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += tt;
    }
    // the 8 cubes' triangle counts of each leaf (8 consecutive threads), 4 bits each
    unsigned pk = (unsigned)cnt << (4 * (t & 7));
    pk |= __shfl_xor_sync(0xffffffffu, pk, 1);
    pk |= __shfl_xor_sync(0xffffffffu, pk, 2);
    pk |= __shfl_xor_sync(0xffffffffu, pk, 4);
    if (live && leaf_cnt && (t & 7) == 0) leaf_cnt[8 * (int64_t)br + (t >> 3)] = pk;
    if (lane == 31) wt[w] = incl;
    if (t == 0) s_ncross[grp] = 0;
    __syncthreads();
    if (live) {
      for (int r = 0; r < div_up_c(kBrickEdges, 64); ++r) {   // the same trip count in both warps
        const int e = t + 64 * r;
        bool cross = false;
        if (e < kBrickEdges) {
          int ax, ex, ey, ez;
          brick_edge_of_slot(e, ax, ex, ey, ez);
          const int pi = bx * kBrick + ex, pj = by * kBrick + ey, pk = bz * kBrick + ez;
          if (pi + (ax == 0) < n && pj + (ax == 1) < n && pk + (ax == 2) < n) {
            const int64_t p = lin3(pi, pj, pk, n);
            const int64_t stride = (ax == 0) ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
            // crossing exactly when the two corner bits of the cube codes differ
            cross = (chi[p] < c_up) != (chi[p + stride] < c_up);
          }
        }
        const unsigned mk = __ballot_sync(0xffffffffu, cross);
        if (mk) {
          const int leader = __ffs(mk) - 1;
          int at = 0;
          if (lane == leader) at = atomicAdd(&s_ncross[grp], __popc(mk));
          at = __shfl_sync(0xffffffffu, at, leader);
          if (cross) s_cross[grp][at + __popc(mk & ((1u << lane) - 1u))] = (short)e;
        }
      }
    }
    __syncthreads();
    if (live) {
      const int nc = s_ncross[grp];
      for (int ci = t; ci < nc; ci += 64) {
        const int e = s_cross[grp][ci];
        int ax, ex, ey, ez;
        brick_edge_of_slot(e, ax, ex, ey, ez);
        const int pi = bx * kBrick + ex, pj = by * kBrick + ey, pk = bz * kBrick + ez;
        const int64_t p = lin3(pi, pj, pk, n);
        const int64_t stride = (ax == 0) ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
        double c1, c2;
        if (xff) {
          const float2 f1 = xff[p], f2 = xff[p + stride];
          c1 = (double)f1.x + (double)f1.y;
          c2 = (double)f2.x + (double)f2.y;
        } else {
          c1 = (double)chi[p];
          c2 = (double)chi[p + stride];
        }
        const double eta = (c - c1) / (c2 - c1);
        // node centre, moved by eta h along the edge's axis
        double px = fma(pi + 0.5, g.h, g.lo[0]), py = fma(pj + 0.5, g.h, g.lo[1]), pz = fma(pk + 0.5, g.h, g.lo[2]);
        if (ax == 0) px = fma(eta, g.h, px);
        else if (ax == 1) py = fma(eta, g.h, py);
        else pz = fma(eta, g.h, pz);
        const int gid = (int)(3 * p + ax);
        const float hx = (float)px, hy = (float)py, hz = (float)pz;
        s_vh[grp][e] = make_float4(hx, hy, hz, __int_as_float(gid));
        s_vl[grp][e] = make_float4((float)(px - (double)hx), (float)(py - (double)hy), (float)(pz - (double)hz), 0.f);
      }
    }
    __syncthreads();
    if (live) {
      const int excl = incl - cnt + ((w & 1) ? wt[w - 1] : 0);
      if ((t & 7) == 0) leaf_off[8 * (int64_t)br + (t >> 3)] = base + excl;
      const int li = i - bx * kBrick, lj = j - by * kBrick, lk = k - bz * kBrick;
      for (int q = 0; q < cnt; ++q) {
        const int64_t idx = (int64_t)base + excl + q;
        if (idx >= cap) break;
        auto slot = [&](int v) {
          int ox, oy, oz, ax;
          edge_lower_offset(c_mc_tris[code][q][v], ox, oy, oz, ax);
          return brick_edge_slot(ax, li + ox, lj + oy, lk + oz);
        };
        const int s0 = slot(0), s1 = slot(1), s2 = slot(2);
        tris[idx] = Tri{s_vh[grp][s0], s_vh[grp][s1], s_vh[grp][s2]};
        if (tris_lo) tris_lo[idx] = Tri{s_vl[grp][s0], s_vl[grp][s1], s_vl[grp][s2]};
      }
    }
    __syncthreads();   // the shared arrays are reused by the next bricks
  }
}

// ---- octree of "pucks" over the leaves (2^3-cube sub-bricks).  A puck is a
// solid cylinder (centre c, unit axis n, radius r, half-thickness t) holding
// every vertex of the node's triangles, hence (by convexity) the triangles
// themselves; its exact distance is a lower bound on their distance.  For a
// smooth patch the cylinder is thin and oriented along the surface normal, so
// the bound stays tight even for far, oblique queries.  Empty node: r < 0.
struct PyrInfo {
  int nlev;
  int dim[12];
  long long off[12];
};

__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

__device__ __forceinline__ int leaf_index(int lx, int ly, int lz, int nb) {
  const int br = ((lz >> 1) * nb + (ly >> 1)) * nb + (lx >> 1);
  return 8 * br + ((lx & 1) | ((ly & 1) << 1) | ((lz & 1) << 2));
}

// Inflation of a puck's radius and half-thickness, for the float rounding of
// the offsets they are the largest of (relative) and of the ~48-bit vertices
// behind the float32 ones (of the coordinates' magnitude).  What the distance
// of a query rounds is left to puck_dist2.
constexpr float kPuckRel = 2e-6f;
constexpr float kPuckAbs = 2e-7f;

// Search record of a triangle for the distance search: vertex a and the edge
// vectors ab, ac with the Gram entries |ab|^2, ab.ac and |ac|^2, and the
// reciprocals the Voronoi regions divide by (0 for a zero-length edge or a
// collapsed triangle), all in the search's units (sc).
// With the vertices' low parts (lo, may be null) the edge vectors are the
// float32 roundings of the differences of the ~48-bit vertices, not the
// differences of the float32 vertices: their directions then carry float32
// rounding (~6e-8 relative) instead of the vertices' absolute rounding,
// which a far node's closest point would amplify by distance / edge length.
__device__ __forceinline__ void write_search_record(const Tri& tr, const Tri* lo, float sc,
                                                    float4* __restrict__ rec) {
  float3 a = f3(tr.a);
  const float3 b = f3(tr.b), c = f3(tr.c);
  float3 ab = sub3(b, a), ac = sub3(c, a), bc = sub3(c, b);
  if (lo) {
    const float3 al = f3(lo->a), bl = f3(lo->b), cl = f3(lo->c);
    ab = make_float3(ab.x + (bl.x - al.x), ab.y + (bl.y - al.y), ab.z + (bl.z - al.z));
    ac = make_float3(ac.x + (cl.x - al.x), ac.y + (cl.y - al.y), ac.z + (cl.z - al.z));
    bc = make_float3(bc.x + (cl.x - bl.x), bc.y + (cl.y - bl.y), bc.z + (cl.z - bl.z));
  }
  a = make_float3(a.x * sc, a.y * sc, a.z * sc);
  ab = make_float3(ab.x * sc, ab.y * sc, ab.z * sc);
  ac = make_float3(ac.x * sc, ac.y * sc, ac.z * sc);
  bc = make_float3(bc.x * sc, bc.y * sc, bc.z * sc);
  const float e00 = dot3(ab, ab), e11 = dot3(ac, ac), ebc = dot3(bc, bc);
  const float3 cr = cross3(ab, ac);
  const float det = dot3(cr, cr);   // = |ab|^2 |ac|^2 - (ab.ac)^2, without the cancellation
  rec[0] = make_float4(a.x, a.y, a.z, e00);
  rec[1] = make_float4(ab.x, ab.y, ab.z, dot3(ab, ac));
  rec[2] = make_float4(ac.x, ac.y, ac.z, e11);
  rec[3] = make_float4(e00 > 0.f ? 1.f / e00 : 0.f, e11 > 0.f ? 1.f / e11 : 0.f, ebc > 0.f ? 1.f / ebc : 0.f,
                       det > 0.f ? 1.f / det : 0.f);
}

// Leaf pucks, pass 1 (every leaf): an empty leaf gets the empty puck; a
// leaf with triangles goes to the list of live leaves (one atomic per warp),
// which the fitting passes then take with full warps.
__global__ void puck_leaf_scan_kernel(const int* __restrict__ leaf_off, int nb, int64_t cap,
                                      float4* __restrict__ pyr, int* __restrict__ live, DevState* __restrict__ st) {
  const int nl = 2 * nb;
  const int64_t nleaf = (int64_t)nl * nl * nl;
  const int lane = threadIdx.x & 31;
  // warp-uniform trip count: every lane reaches the ballot
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < nleaf; base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = base + threadIdx.x;
    bool full = false;
    if (t < nleaf) {
      const int lx = (int)(t % nl), ly = (int)((t / nl) % nl), lz = (int)(t / ((int64_t)nl * nl));
      const int li = leaf_index(lx, ly, lz, nb);
      full = min((int64_t)leaf_off[li + 1], cap) > (int64_t)leaf_off[li];
      if (!full) {
        pyr[2 * t] = make_float4(0.f, 0.f, 0.f, -1.f);
        pyr[2 * t + 1] = make_float4(0.f, 0.f, 1.f, 0.f);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, full);
    if (m) {
      const int leader = __ffs(m) - 1;
      unsigned at = 0;
      if (lane == leader) at = atomicAdd(&st->nleaf_live, (unsigned)__popc(m));
      at = __shfl_sync(0xffffffffu, at, leader);
      if (full) live[at + __popc(m & ((1u << lane) - 1u))] = (int)t;
    }
  }
}

// v / |v|, (0, 0, 1) for no direction, by way of a power of two that brings v's
// largest component near 1: a sum of area normals is a square of the box's
// units, and its square can leave the float range.
__device__ __forceinline__ float3 unit_normal(float3 v) {
  const unsigned e = __float_as_uint(fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fabsf(v.z))) >> 23;
  const float k = __uint_as_float((254u - min(e, 253u)) << 23);
  v = make_float3(v.x * k, v.y * k, v.z * k);
  const float nn = sqrtf(dot3(v, v));
  return nn > 0.f ? make_float3(v.x / nn, v.y / nn, v.z / nn) : make_float3(0.f, 0.f, 1.f);
}

// Puck (centre + radius, axis + half-thickness, in the search's units) fitted to
// the vertices of triangles [q0, q1): centroid and mean area normal, then the largest radial
// and axial vertex offsets in that frame, padded so the bound stays
// conservative under float rounding.
__device__ __forceinline__ void fit_puck(const Tri* __restrict__ tris, int64_t q0, int64_t q1, float sc, float4& A,
                                         float4& B) {
  float3 cs = make_float3(0.f, 0.f, 0.f), ns = make_float3(0.f, 0.f, 0.f);
  for (int64_t q = q0; q < q1; ++q) {
    const Tri tr = tris[q];
    const float3 a = f3(tr.a), b = f3(tr.b), c = f3(tr.c);
    cs.x += a.x + b.x + c.x;
    cs.y += a.y + b.y + c.y;
    cs.z += a.z + b.z + c.z;
    const float3 cr = cross3(sub3(b, a), sub3(c, a));
    ns.x += cr.x;
    ns.y += cr.y;
    ns.z += cr.z;
  }
  const float inv = 1.f / (3.f * (float)(q1 - q0));
  const float3 cc = make_float3(cs.x * inv, cs.y * inv, cs.z * inv);
  const float3 nv = unit_normal(ns);
  float r = 0.f, th = 0.f;
  for (int64_t q = q0; q < q1; ++q) {
    const Tri tr = tris[q];
    const float4 vv[3] = {tr.a, tr.b, tr.c};
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const float3 d = sub3(f3(vv[v]), cc);
      const float z = dot3(d, nv);
      const float rho2 = fmaxf(dot3(d, d) - z * z, 0.f);
      th = fmaxf(th, fabsf(z));
      r = fmaxf(r, sqrtf(rho2));
    }
  }
  const float pad = kPuckRel * (r + th) + kPuckAbs * (fabsf(cc.x) + fabsf(cc.y) + fabsf(cc.z));
  A = make_float4(cc.x * sc, cc.y * sc, cc.z * sc, (r + pad) * sc);
  B = make_float4(nv.x, nv.y, nv.z, (th + pad) * sc);
}

// Rank of the q-th triangle of a leaf in a depth-first walk of the octree that
// takes children from the last to the first (the leaf's Morton code, 9 bits an
// axis, descending): the order in which the search ranks equal distances.
__device__ __forceinline__ unsigned walk_rank(int lx, int ly, int lz, int q) {
  auto spread = [](unsigned v) {   // nine bits, two zeros between each
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    return (v | (v << 2)) & 0x09249249u;
  };
  const unsigned m = spread((unsigned)lx) | (spread((unsigned)ly) << 1) | (spread((unsigned)lz) << 2);
  return ((0x07ffffffu - m) << 5) | (unsigned)min(q, 31);
}

// Leaf pucks, pass 2 (live leaves): the triangles' search records, the
// leaf's puck fitted to its vertices, and (cell_pyr non-null) one puck per
// cube of the leaf that holds triangles, stored at the slot of the cube's
// first triangle (cell_pyr[2 q0], [2 q0 + 1]); leaf_cnt packs the cubes'
// triangle counts, 4 bits per cube in the leaf's cube order.
__global__ void puck_leaf_kernel(const Tri* __restrict__ tris, Tri* __restrict__ tris_lo,
                                 const int* __restrict__ leaf_off, const unsigned* __restrict__ leaf_cnt, int nb,
                                 int64_t cap, const int* __restrict__ live, const DevState* __restrict__ st,
                                 float4* __restrict__ pyr, float4* __restrict__ tris_s,
                                 float4* __restrict__ cell_pyr, float sc) {
  const int nl = 2 * nb;
  const int64_t nlive = st->nleaf_live;
  for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < nlive;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = live[it];
    const int lx = (int)(t % nl), ly = (int)((t / nl) % nl), lz = (int)(t / ((int64_t)nl * nl));
    const int li = leaf_index(lx, ly, lz, nb);
    const int64_t s0 = leaf_off[li];
    const int64_t s1 = min((int64_t)leaf_off[li + 1], cap);
    for (int64_t q = s0; q < s1; ++q) {
      const Tri tr = tris[q];
      if (tris_lo) {
        const Tri tl = tris_lo[q];
        write_search_record(tr, &tl, sc, tris_s + kTriRec * q);
        tris_lo[q].a.w = __uint_as_float(walk_rank(lx, ly, lz, (int)(q - s0)));
      } else {
        write_search_record(tr, nullptr, sc, tris_s + kTriRec * q);
      }
    }
    float4 A, B;
    fit_puck(tris, s0, s1, sc, A, B);
    pyr[2 * t] = A;
    pyr[2 * t + 1] = B;
    if (cell_pyr) {
      unsigned cn = leaf_cnt[li];
      int64_t q0 = s0;
      for (; cn != 0u; cn >>= 4) {
        const int64_t q1 = min(q0 + (int64_t)(cn & 15u), s1);
        if (q0 < q1) {
          fit_puck(tris, q0, q1, sc, A, B);
          cell_pyr[2 * q0] = A;
          cell_pyr[2 * q0 + 1] = B;
        }
        q0 += cn & 15u;
      }
    }
  }
}

// Tight puck of an internal node at level l >= 1 (dim d_l; level 1 = bricks):
// axis and centre from its own triangles, radius and half-thickness from
// their vertices (two passes over the bricks it covers).
// Squared distance from p to the solid cylinder of a puck (INF when empty),
// from below: every term that p's distance d to the centre rounds (z and the
// hardware reciprocal square root, a few 1e-7 d; the difference d^2 - z^2, a
// few 1e-7 d^2) is taken low by 1e-6 of it.  (An inflation of the pucks by 1e-5
// of the coordinates covered the same: 0.008 cells of thickness at 512^3,
// which at 150 cells from the surface admits 1.5 cells more on every side.)
__device__ __forceinline__ float puck_dist2(const float3 p, const float4 A, const float4 B) {
  if (A.w < 0.f) return INFINITY;
  const float3 d = make_float3(p.x - A.x, p.y - A.y, p.z - A.z);
  const float z = d.x * B.x + d.y * B.y + d.z * B.z;
  const float x2 = fmaxf(fmaf(d.x * d.x + d.y * d.y + d.z * d.z, 1.f - 1e-6f, -z * z), 0.f);
  const float rho = x2 * rsqrtf(fmaxf(x2, 1e-30f));
  const float dz = fmaxf(fmaf(fabsf(z), 1.f - 1e-6f, -B.w), 0.f);
  const float dr = fmaxf(fmaf(rho, 1.f - 1e-6f, -A.w), 0.f);
  return dz * dz + dr * dr;
}

// Vertex-fitted pucks for every octree level above the leaves.  A node's
// frame is its vertex centroid and mean area normal (in the box's units; the
// finished pucks are brought to the search's); both come from sums
// that add up the tree (per brick first: a level-1 node is one brick).  The
// radius and half-thickness are the largest radial and axial vertex offsets
// in that frame, taken in one pass over the leaves for all levels at once
// (warp-aggregated atomic maxima on the bits of non-negative floats).  Aux
// slots cover the nodes of levels >= 1: aux index = pyramid index - off[1].
__device__ __forceinline__ void node_frame(const float4 s0, const float4 s1, float3& c, float3& ax) {
  const float inv = 1.f / (3.f * s0.w);
  c = make_float3(s0.x * inv, s0.y * inv, s0.z * inv);
  ax = unit_normal(f3(s1));
}

__global__ void puck_sums_brick_kernel(const Tri* __restrict__ tris, const int* __restrict__ brick_off, int nb,
                                       int64_t cap, float4* __restrict__ sums, unsigned* __restrict__ rth) {
  const int64_t nbr = (int64_t)nb * nb * nb;
  for (int64_t br = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; br < nbr;
       br += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q0 = brick_off[br];
    const int64_t q1 = min((int64_t)brick_off[br + 1], cap);
    float3 cs = make_float3(0.f, 0.f, 0.f), ns = make_float3(0.f, 0.f, 0.f);
    for (int64_t q = q0; q < q1; ++q) {
      const Tri tr = tris[q];
      const float3 a = f3(tr.a), b = f3(tr.b), c = f3(tr.c);
      cs.x += a.x + b.x + c.x;
      cs.y += a.y + b.y + c.y;
      cs.z += a.z + b.z + c.z;
      const float3 cr = cross3(sub3(b, a), sub3(c, a));
      ns.x += cr.x;
      ns.y += cr.y;
      ns.z += cr.z;
    }
    sums[2 * br] = make_float4(cs.x, cs.y, cs.z, (float)(q1 > q0 ? q1 - q0 : 0));
    sums[2 * br + 1] = make_float4(ns.x, ns.y, ns.z, 0.f);
    rth[2 * br] = 0u;
    rth[2 * br + 1] = 0u;
  }
}

__global__ void puck_sums_up_kernel(float4* __restrict__ sums, unsigned* __restrict__ rth, int64_t a_child,
                                    int dchild, int64_t a_parent, int dparent) {
  const int64_t np = (int64_t)dparent * dparent * dparent;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < np;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(t % dparent), y = (int)((t / dparent) % dparent), z = (int)(t / ((int64_t)dparent * dparent));
    float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = 0; q < 8; ++q) {
      const int cx = 2 * x + (q & 1), cy = 2 * y + ((q >> 1) & 1), cz = 2 * z + (q >> 2);
      if (cx >= dchild || cy >= dchild || cz >= dchild) continue;
      const int64_t ci = a_child + ((int64_t)cz * dchild + cy) * dchild + cx;
      const float4 c0 = sums[2 * ci], c1 = sums[2 * ci + 1];
      s0 = make_float4(s0.x + c0.x, s0.y + c0.y, s0.z + c0.z, s0.w + c0.w);
      s1 = make_float4(s1.x + c1.x, s1.y + c1.y, s1.z + c1.z, 0.f);
    }
    sums[2 * (a_parent + t)] = s0;
    sums[2 * (a_parent + t) + 1] = s1;
    rth[2 * (a_parent + t)] = 0u;
    rth[2 * (a_parent + t) + 1] = 0u;
  }
}

__global__ void puck_rth_kernel(const Tri* __restrict__ tris, const int* __restrict__ leaf_off, int nb, int64_t cap,
                                PyrInfo pi, const int* __restrict__ live, const DevState* __restrict__ st,
                                const float4* __restrict__ sums, unsigned* __restrict__ rth) {
  const int dl = pi.dim[0];
  const int64_t nlive = st->nleaf_live;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // the live leaves (list order keeps a warp's leaves together); warp-uniform
  // trip count: every lane reaches the warp-wide reductions
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nlive; base += stride) {
    const int64_t it = base + threadIdx.x;
    const bool in = it < nlive;
    const int64_t t = in ? live[it] : 0;
    const int lx = in ? (int)(t % dl) : 0, ly = in ? (int)((t / dl) % dl) : 0,
              lz = in ? (int)(t / ((int64_t)dl * dl)) : 0;
    int64_t q0 = 0, q1 = 0;
    if (in) {
      const int li = leaf_index(lx, ly, lz, nb);
      q0 = leaf_off[li];
      q1 = min((int64_t)leaf_off[li + 1], cap);
    }
#pragma unroll 1
    for (int l = 1; l < pi.nlev; ++l) {
      const int d = pi.dim[l];
      const int64_t node = ((int64_t)(lz >> l) * d + (ly >> l)) * d + (lx >> l);
      const int64_t a = pi.off[l] - pi.off[1] + node;
      float r = 0.f, th = 0.f;
      if (q1 > q0) {
        float3 c, ax;
        node_frame(sums[2 * a], sums[2 * a + 1], c, ax);
        for (int64_t q = q0; q < q1; ++q) {
          const Tri tr = tris[q];
          const float4 vv[3] = {tr.a, tr.b, tr.c};
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            const float3 dv = sub3(f3(vv[v]), c);
            const float zz = dot3(dv, ax);
            th = fmaxf(th, fabsf(zz));
            r = fmaxf(r, sqrtf(fmaxf(dot3(dv, dv) - zz * zz, 0.f)));
          }
        }
      }
      const long long key = (q1 > q0) ? (long long)a : -1ll;
      const unsigned peers = __match_any_sync(0xffffffffu, key);
      const unsigned rm = __reduce_max_sync(peers, __float_as_uint(r));
      const unsigned tm = __reduce_max_sync(peers, __float_as_uint(th));
      if (key >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) {
        atomicMax(&rth[2 * a], rm);
        atomicMax(&rth[2 * a + 1], tm);
      }
    }
  }
}

__global__ void puck_finalize_kernel(float4* __restrict__ pyr, const float4* __restrict__ sums,
                                     const unsigned* __restrict__ rth, int64_t naux, int64_t pyr_base, float sc) {
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < naux; a += (int64_t)gridDim.x * blockDim.x) {
    const float4 s0 = sums[2 * a], s1 = sums[2 * a + 1];
    const int64_t gi = pyr_base + a;
    if (!(s0.w > 0.f)) {
      pyr[2 * gi] = make_float4(0.f, 0.f, 0.f, -1.f);
      pyr[2 * gi + 1] = make_float4(0.f, 0.f, 1.f, 0.f);
      continue;
    }
    float3 c, ax;
    node_frame(s0, s1, c, ax);
    const float r = __uint_as_float(rth[2 * a]), th = __uint_as_float(rth[2 * a + 1]);
    const float pad = kPuckRel * (r + th) + kPuckAbs * (fabsf(c.x) + fabsf(c.y) + fabsf(c.z));
    pyr[2 * gi] = make_float4(c.x * sc, c.y * sc, c.z * sc, (r + pad) * sc);
    pyr[2 * gi + 1] = make_float4(ax.x, ax.y, ax.z, (th + pad) * sc);
  }
}

// Child-occupancy masks of the internal nodes (levels >= 1): bit q set when
// child q (x + (q & 1), y + (q >> 1 & 1), z + (q >> 2), at twice the
// coordinates) exists and holds triangles.  The mask sits in the low 8 bits of
// the node's radius, rounded up first so that the stored radius never
// shrinks (the bound stays conservative; at most 2^-14 relative).
__global__ void puck_mask_kernel(float4* __restrict__ pyr, PyrInfo pi) {
  const int64_t total = pi.off[pi.nlev - 1] + 1 - pi.off[1];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t gi = pi.off[1] + t;
    int l = 1;
    while (l + 1 < pi.nlev && gi >= pi.off[l + 1]) ++l;
    const float4 A = pyr[2 * gi];
    if (A.w < 0.f) continue;
    const int64_t r = gi - pi.off[l];
    const int d = pi.dim[l], dc = pi.dim[l - 1];
    const int x = (int)(r % d), y = (int)((r / d) % d), z = (int)(r / ((int64_t)d * d));
    unsigned mask = 0;
    for (int q = 0; q < 8; ++q) {
      const int cx = 2 * x + (q & 1), cy = 2 * y + ((q >> 1) & 1), cz = 2 * z + (q >> 2);
      if (cx >= dc || cy >= dc || cz >= dc) continue;
      const int64_t cg = pi.off[l - 1] + ((int64_t)cz * dc + cy) * dc + cx;
      if (pyr[2 * cg].w >= 0.f) mask |= 1u << q;
    }
    const unsigned up = (__float_as_uint(A.w) + 0xffu) & ~0xffu;
    pyr[2 * gi].w = __uint_as_float(up | mask);
  }
}

}  // namespace

namespace {

constexpr int kWarps = 4;          // warps per CTA
constexpr int kStack = 96;         // per-warp traversal stack (exact queries)

// Float32 rounding of one point-triangle distance, as a bound used to detect
// near-ties: relative to the distance, plus an absolute part for the rounding
// of the node and vertex coordinates (of magnitude up to the coordinate scale).
constexpr float kTieRel = 4e-7f;
constexpr float kTieAbs = 1.5e-7f;
constexpr int kCand = 4;           // smallest float32 distances kept per node

struct TieSlots {
  int2* p[2];   // the two float-float iterate buffers; the one not current is free
};

// Squared distance from p to a triangle given by its search record (see
// write_search_record): the Voronoi region picks the closest point
// y = a + v ab + w ac (Ericson's case analysis, with the six dot products
// reduced to d1 = ab.ap and d2 = ac.ap through the stored Gram entries and
// the divisions replaced by the stored reciprocals), and the residual
// p - y = ap - v ab - w ac is formed relative to a, so its rounding scales
// with the distance and the edge length rather than with the coordinates.

__device__ __forceinline__ float tri_dist2_rec(const float3 p, const float4* __restrict__ rec, float& v, float& w) {
  const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
  const float3 ap = make_float3(p.x - r0.x, p.y - r0.y, p.z - r0.z);
  const float d1 = r1.x * ap.x + r1.y * ap.y + r1.z * ap.z;   // ab . ap
  const float d2 = r2.x * ap.x + r2.y * ap.y + r2.z * ap.z;   // ac . ap
  rec_weights(ap, d1, d2, r0, r1, r2, r3, v, w);
  const float rx = ap.x - v * r1.x - w * r2.x;
  const float ry = ap.y - v * r1.y - w * r2.y;
  const float rz = ap.z - v * r1.z - w * r2.z;
  return rx * rx + ry * ry + rz * rz;
}
__device__ __forceinline__ float tri_dist2_rec(const float3 p, const float4* __restrict__ rec) {
  float v, w;
  return tri_dist2_rec(p, rec, v, w);
}

// Key (32-bit hash) of a node's closest feature on triangle t, from the weights
// (v, w) of its closest point y = a + v ab + w ac and the edge ids of the
// triangle's vertices: a vertex (weights 0 / 1) by its id, an edge (one weight
// 0, or v = 1 - w) by its two, a face by the triangle.  Triangles that share
// the closest vertex or edge give the same key; vertices never collide, other
// pairs with probability 2^-32.
__device__ __forceinline__ unsigned feature_key(float v, float w, const Tri* __restrict__ tri, int t) {
  auto mix = [](unsigned x) {
    x *= 0x9E3779B1u;
    return x ^ (x >> 15);
  };
  const bool onb = v == 1.f && w == 0.f, onc = w == 1.f && v == 0.f, ona = v == 0.f && w == 0.f;
  const bool face = !(w == 0.f || v == 0.f || v == 1.f - w);
  if (face) return mix(mix((unsigned)t) + 0x7F4A7C15u);
  const unsigned ga = mix(__float_as_uint(tri[t].a.w)), gb = mix(__float_as_uint(tri[t].b.w)),
                 gc = mix(__float_as_uint(tri[t].c.w));
  if (ona || onb || onc) return ona ? ga : onb ? gb : gc;
  const unsigned p = w == 0.f ? ga : v == 0.f ? ga : gb, q = w == 0.f ? gb : gc;
  return mix((min(p, q) * 0x85EBCA6Bu) ^ max(p, q));
}

// Class of the same feature: a hash of ten bits per vertex (sdf_tie_kernel).
__device__ __forceinline__ unsigned feature_class(float v, float w, const Tri* __restrict__ tri, int t) {
  auto hash10 = [](float gid) { return (__float_as_uint(gid) * 0x9E3779B1u) >> 22; };
  auto edge = [](unsigned p, unsigned q) { return (1u << 20) | (min(p, q) << 10) | max(p, q); };
  const unsigned ha = hash10(tri[t].a.w), hb = hash10(tri[t].b.w), hc = hash10(tri[t].c.w);
  unsigned x;
  if (w == 0.f) {
    x = (v == 0.f) ? ha : (v == 1.f ? hb : edge(ha, hb));
  } else if (v == 0.f) {
    x = (w == 1.f) ? hc : edge(ha, hc);
  } else if (v == 1.f - w) {
    x = edge(hb, hc);
  } else {
    x = (2u << 20) ^ (unsigned)t;
  }
  return ((x * 0x9E3779B1u) ^ 0x7F4A7C15u) * 0x85EBCA6Bu;
}

// The same distance in float-float for the near-tie decisions, on the ~48-bit
// vertices (float32 vertex + its low part, see mc_emit_kernel): a, ab, ac and
// ap in float-float, so the distance is that of the refined surface to ~1e-14
// relative and two candidates are ranked as the exact (FP64) mesh ranks them
// unless they tie to that level.  The Voronoi region and the weights (v, w)
// come from the float32 record: a region chosen wrongly near a region boundary,
// and rounding of the weights, change |p - y| only to second order (the
// residual is normal to the directions they move y in).
__device__ __forceinline__ Ff tri_dist2_ff_exact(const Vec3<Ff> p, const float4* __restrict__ rec, const Tri& hi,
                                                 const Tri& lo, float sc) {
  const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
  const float3 ah = f3(hi.a, sc), bh = f3(hi.b, sc), ch = f3(hi.c, sc);
  const float3 al = f3(lo.a, sc), bl = f3(lo.b, sc), cl = f3(lo.c, sc);
  const Ff ax = Ff(ah.x) + Ff(al.x), ay = Ff(ah.y) + Ff(al.y), az = Ff(ah.z) + Ff(al.z);
  const Ff abx = (Ff(bh.x) + Ff(bl.x)) - ax, aby = (Ff(bh.y) + Ff(bl.y)) - ay, abz = (Ff(bh.z) + Ff(bl.z)) - az;
  const Ff acx = (Ff(ch.x) + Ff(cl.x)) - ax, acy = (Ff(ch.y) + Ff(cl.y)) - ay, acz = (Ff(ch.z) + Ff(cl.z)) - az;
  const Ff apx = p.x - ax, apy = p.y - ay, apz = p.z - az;
  const float3 ap = make_float3(apx.hi, apy.hi, apz.hi);
  const float d1 = r1.x * ap.x + r1.y * ap.y + r1.z * ap.z;
  const float d2 = r2.x * ap.x + r2.y * ap.y + r2.z * ap.z;
  float v, w;
  rec_weights(ap, d1, d2, r0, r1, r2, r3, v, w);
  const Ff fv(v), fw(w);
  const Ff rx = apx - (fv * abx + fw * acx);
  const Ff ry = apy - (fv * aby + fw * acy);
  const Ff rz = apz - (fv * abz + fw * acz);
  return rx * rx + ry * ry + rz * rz;
}

// Octree entry: level in bits 27..31, node coordinates (< 512 per axis) in bits
// 0..8 (x), 9..17 (y), 18..26 (z).  sdf_node_kernel stacks this word beside the
// node's child mask; sdf_query_kernel with the node's pyramid index, so that a
// pop loads the node's puck at once instead of first looking up its level's
// offset and dimension; sdf_patch_kernel's fronts hold the coordinates alone.
__device__ __forceinline__ unsigned pack_node(int lev, int x, int y, int z) {
  return ((unsigned)lev << 27) | ((unsigned)z << 18) | ((unsigned)y << 9) | (unsigned)x;
}

// ---- Exact distance search over the grid nodes.
//
// Exactness at near-ties: two triangles whose distances differ by less than
// the float32 rounding may be ranked either way, and the closest point (and
// with it the vertex gradient of Eqs. 35-36) differs between them.  Each node
// keeps its kCand smallest float32 distances, one per closest feature, and
// prunes against the best plus a rounding margin; when the second lies within
// that margin the node is a near-tie: it is appended to tie_list, the ids of
// the candidates within the margin go to tie_a, tie_b and tie_cd at the same
// list position (-1 for none), and sdf_tie_kernel re-decides it in
// float-float.  Without TIES (no closest triangle is kept) the search keeps
// the float32 minimum alone, which is within the same rounding of the exact
// distance.
//
// Nested lattices, coarse to fine: sdf_node_kernel searches the nodes of the
// coarsest lattice, a warp per node; sdf_patch_kernel then takes the lattices
// of half the stride in turn, a block per 8 x 8 x 4 nodes, seeded with the
// closest triangles of the coarser lattice's nodes around them; blocks with too
// many candidates (around a point far from everything, like a sphere's centre,
// every triangle is one) leave their nodes on a list that sdf_node_kernel
// takes at the end.
//
// Bound: instruction issue (72% of the slots; a node's answer is 60 flops, the
// proof that no other triangle is nearer the rest).  Per warp of 32 nodes at
// 128^3 (star body, 76,000 triangles) the finest pass runs 12,000 instructions
// against 25,000 of a warp that walks the octree for its 32 nodes by itself,
// testing each popped puck and each triangle for all of them: 0.7 for the
// seeds, 2 for the block's walk, 1 + 2.5 for the patch's cubes (of 240 in the
// block's reach, 74 in the patch's and 6.7 in a node's), 3 for 19 triangle
// tests a node and 2 for its 3 exact ones.  Search stage before -> now, ms, of
// star bodies: 0.79 -> 0.32 (64^3, 16,384 points), 2.79 -> 1.61 (128^3, 100,000),
// 16.4 -> 11.9 (256^3, 200,000), 137 -> 90 (512^3, 500,000); 1.47 -> 0.30 on a 64^3
// sphere, whose centre kept one warp busy for all of it.

// What the search reads and writes (device pointers of the handle).
struct Search {
  const float4* tris_s;
  const Tri* tris;
  const Tri* tris_lo;       // a.w: walk_rank
  const int* leaf_off;
  const unsigned* leaf_cnt;
  const float4* pyr;
  const float4* cell_pyr;
  const float* axis;        // node coordinates, [3][res]
  const float* chi;
  DevState* st;
  int64_t cap;
  int n;                    // nodes per axis
  int nb;                   // bricks per axis
  float h;                  // cell size and
  float coord;              // largest |coordinate| of the box, in the search's units
  float sc, us;             // box units -> the search's, and back
  float* phi;
  float* sdf_out;
  int* ctri;
  int* tie_a;
  int* tie_b;
  TieSlots tie_cd;
  int* tie_list;
  int* seed_ids;            // closest triangle of every node of the lattices done so far
  int* defer;               // nodes left to sdf_node_kernel
};

// The candidate list of one node: the NC smallest distances, one entry per
// closest feature (by feature_key; with TIES alone), in registers.  Triangles
// sharing the closest vertex (often six of them) or edge tie exactly and would
// otherwise fill the list and push out a distinct surface point at the same
// distance (a node on the medial axis), which the tie pass must see.  Entries
// are ordered by distance, equal ones with the node's seeds first (s: its eight
// of them, may be null) and then by walk_rank, so the list does not depend on
// the order in which triangles come; each comes once.
__device__ __forceinline__ bool comes_first(int t, int u, const Tri* __restrict__ tris_lo, const int* s) {
  if (s) {
    int st = 8, su = 8;
#pragma unroll
    for (int q = 7; q >= 0; --q) {
      if (s[q] == t) st = q;
      if (s[q] == u) su = q;
    }
    if (st != su) return st < su;
  }
  const unsigned rt = __float_as_uint(tris_lo[t].a.w), ru = __float_as_uint(tris_lo[u].a.w);
  return rt < ru || (rt == ru && t < u);
}

template <bool TIES>
struct Cands {
  static constexpr int NC = TIES ? kCand : 1;
  float cd[NC];
  int ct[NC];
  unsigned ck[NC];
  float cut;        // a near-tie's squared distance is at most this
  __device__ __forceinline__ void init(bool valid) {
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      cd[q] = INFINITY;
      ct[q] = -1;
      ck[q] = 0u;
    }
    cut = valid ? INFINITY : -INFINITY;
  }
  // the exact test of triangle t against p, and its place in the list
  __device__ __forceinline__ void offer(const float3 p, int t, const Search& S, const int* seeds) {
    float v, w;
    const float d2 = tri_dist2_rec(p, S.tris_s + kTriRec * (int64_t)t, v, w);
    if (!TIES) {
      if (d2 < cd[0] || (d2 == cd[0] && t < ct[0])) {
        cd[0] = d2;
        ct[0] = t;
      }
      return;
    }
    if (!(d2 <= cd[NC - 1])) return;
    const unsigned key = feature_key(v, w, S.tris, t);
    bool before[NC];   // whether t comes before entry q (false, ..., true, ...)
    int at = NC - 1;   // the entry it replaces: its feature's, else the last
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      before[q] = d2 < cd[q];
      if (d2 == cd[q] && ct[q] != -1) before[q] = comes_first(t, ct[q], S.tris_lo, seeds);
      if (ct[q] != -1 && ck[q] == key) at = q;
    }
#pragma unroll
    for (int q = NC - 1; q >= 0; --q) {
      if (q > at || !before[q]) continue;
      const bool down = q > 0 && before[q > 0 ? q - 1 : 0];   // the entry above moves here
      cd[q] = down ? cd[q > 0 ? q - 1 : 0] : d2;
      ct[q] = down ? ct[q > 0 ? q - 1 : 0] : t;
      ck[q] = down ? ck[q > 0 ? q - 1 : 0] : key;
    }
  }
  __device__ __forceinline__ void swap(int a, int b) {
    const float tf = cd[a];
    cd[a] = cd[b];
    cd[b] = tf;
    const int ti = ct[a];
    ct[a] = ct[b];
    ct[b] = ti;
    const unsigned tk = ck[a];
    ck[a] = ck[b];
    ck[b] = tk;
  }
  // the cut that goes with the best distance
  __device__ __forceinline__ float reach(float mabs) const {
    if (!TIES) return cd[0];
    const float r = sqrtf(cd[0]) * (1.f + kTieRel) + mabs;
    return r * r;
  }
};

// Results of the warp's nodes (lane with `valid`: linear node o): distance and
// sign, closest triangle, and the near-tie list (one atomic per warp; the
// candidates at the same list position, so that the tie pass reads them
// coalesced).
template <bool COUNT, bool TIES>
__device__ __forceinline__ void store_nodes(const Search& S, const Cands<TIES>& c, bool valid, int64_t o, bool seed,
                                            int lane) {
  constexpr int NC = Cands<TIES>::NC;
  const bool tie = TIES && valid && c.ct[NC > 1 ? 1 : 0] != -1 && c.cd[NC > 1 ? 1 : 0] <= c.cut;
  int tie_at = 0;
  if (TIES) {
    const unsigned m = __ballot_sync(0xffffffffu, tie);
    if (m) {
      const int leader = __ffs(m) - 1;
      unsigned base = 0;
      if (lane == leader) {
        base = atomicAdd(&S.st->ntie, (unsigned)__popc(m));
        if (COUNT) atomicAdd(&S.st->sdf_cnt[3], (unsigned long long)__popc(m));
      }
      base = __shfl_sync(0xffffffffu, base, leader);
      tie_at = (int)(base + __popc(m & ((1u << lane) - 1u)));
      if (tie) S.tie_list[tie_at] = (int)o;
    }
  }
  if (!valid) return;
  const int bt = c.ct[0];
  const float val = (S.chi[o] >= S.st->c_up ? 1.f : -1.f) * sqrtf(c.cd[0]) * S.us;
  S.phi[o] = val;
  if (S.sdf_out) S.sdf_out[o] = val;
  if (S.ctri) S.ctri[o] = bt;
  if (seed) S.seed_ids[o] = bt;
  if (TIES && tie) {
    S.tie_a[tie_at] = bt;
    S.tie_b[tie_at] = c.ct[NC > 1 ? 1 : 0];
    int more[2] = {-1, -1};
#pragma unroll
    for (int q = 2; q < NC; ++q)
      if (c.cd[q] <= c.cut && c.ct[q] != -1) more[q - 2] = c.ct[q];
    S.tie_cd.p[S.st->fwd.xidx ^ 1][tie_at] = make_int2(more[0], more[1]);
  }
}

// Octree entries waiting on a warp's stack: pack_node's word and the node's
// child-occupancy mask, known when the node was bounded, so a pop needs no
// memory.  Up to four nodes are popped at a time, their 32 children bounded one
// per lane.  Four are taken only while the stack holds kPopFour entries or
// fewer, then one by one: a pop of one node of level l leaves at most 7 more
// entries per level below it, so the stack stays below kPopFour - 4 + 32 + 7 *
// 9 (at most 10 levels).
constexpr int kPopFour = 60;
constexpr int kSrchStack = 160;
static_assert(kPopFour - 4 + 32 + 7 * 9 <= kSrchStack, "search stack");

// One leaf's cube of a lane: its first triangle and triangle count, from the
// leaf's triangle offset and its cubes' counts (4 bits each).
__device__ __forceinline__ void leaf_cube(const Search& S, int li, int cube, int& q0, int& cnt) {
  const unsigned cn = S.leaf_cnt[li];
  const unsigned below = cn & ((1u << (4 * cube)) - 1u);
  const unsigned pairs = (below & 0x0f0f0f0fu) + ((below >> 4) & 0x0f0f0f0fu);
  q0 = S.leaf_off[li] + (int)((pairs * 0x01010101u) >> 24);
  cnt = (int)((cn >> (4 * cube)) & 15u);
  if ((int64_t)q0 + cnt > S.cap) cnt = max((int)(S.cap - q0), 0);
}

// Whether some point of a box may have its closest surface point, or a near-tie
// with it, in a puck.  With y a surface point, p0 the box's centre and e its
// half extents, any point p of the box is at most |p - y| from the surface,
// and for a point c of the puck |p - c|^2 - |p - y|^2 is linear in p: its
// least value over the box is |p0 - c|^2 - |p0 - y|^2 - 2 sum_a e_a |c - y|_a.
// So the puck is out when its distance to p0 exceeds |p0 - y| by more than
// that sum's bound over the puck's bounding sphere.  Unlike a bound from the
// distance to the box alone, whose slack grows with the distance to the
// surface, this one depends on the lateral offset c - y only.  Each of the
// box's reference points y (the closest points of its corner nodes) has to
// admit the puck: over a flat surface one of them alone admits offsets of
// twice the box's extent on the far side, and the opposite corners' together
// leave just the box's own footprint.
// refs: y and |p0 - y|^2 widened by reach_of; N of them, at the indices of
// ref_at (all eight corners, or four that share no edge).
__device__ __forceinline__ constexpr int ref_at(int n, int q) { return n == 8 ? q : q == 0 ? 0 : q == 1 ? 3 : q == 2 ? 5 : 6; }
template <int N>
__device__ __forceinline__ bool puck_reaches(const float3 p0, const float4* refs, const float3 e, float elen,
                                             const float4 A, const float4 B) {
  const float d = puck_dist2(p0, A, B) * (1.f - 1e-6f) - 2.00002f * elen * (A.w + B.w);
  bool in = true;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const float4 y = refs[ref_at(N, q)];
    const float s = e.x * fabsf(A.x - y.x) + e.y * fabsf(A.y - y.y) + e.z * fabsf(A.z - y.z);
    in = in && d <= fmaf(2.00002f, s, y.w);
  }
  return in;
}

// |p0 - y|^2 widened by the margin of a near-tie at the box's farthest point
// from y (kTieRel, kTieAbs) and by the float rounding of y, p0 and the
// squares.
__device__ __forceinline__ float reach_of(const float3 p0, const float3 y, float elen, float coord) {
  const float3 d = sub3(p0, y);
  const float u = dot3(d, d);
  const float m = sqrtf(u) + elen;
  return u + 2.f * m * (1e-6f * m + 5e-7f * coord);
}

// Squared distance d^2 from p to a triangle without branches, to rank triangles:
// the least of the three clamped edges and, when the projection falls inside,
// the face, each as a quadratic form about vertex a (stationary in the
// weights, so their rounding enters to second order).  Its error is the
// cancellation against |p - a|^2, which tri_dist2_rec avoids, below 1e-6 (d +
// sqrt(3) h)^2 (edges are at most the cube's diagonal; 4e-7 (d^2 + 3 h^2)
// measured), and on thin triangles that of the face weights: they are off by
// about the rounding times (edge / height)^2, and the smaller of the face at
// such weights and the edges exceeds d^2 by up to 4.0e-5 h^2 (worst of 6e7
// triangles tried, at a height of 0.007 edges).
__device__ __forceinline__ float tri_dist2_fast(const float3 p, const float4* __restrict__ rec) {
  const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
  const float3 ap = make_float3(p.x - r0.x, p.y - r0.y, p.z - r0.z);
  const float s = ap.x * ap.x + ap.y * ap.y + ap.z * ap.z;
  const float d1 = r1.x * ap.x + r1.y * ap.y + r1.z * ap.z;
  const float d2 = r2.x * ap.x + r2.y * ap.y + r2.z * ap.z;
  const float e00 = r0.w, e01 = r1.w, e11 = r2.w;
  const float m1 = -2.f * d1, m2 = -2.f * d2;
  const float t1 = __saturatef(d1 * r3.x), t2 = __saturatef(d2 * r3.y);
  const float q1 = fmaf(t1, fmaf(t1, e00, m1), s), q2 = fmaf(t2, fmaf(t2, e11, m2), s);
  const float g = e00 - e01, db = (d2 - d1) + g;            // bc . bp
  const float t3 = __saturatef(db * r3.z);
  const float q3 = fmaf(t3, fmaf(t3, g + (e11 - e01), -2.f * db), (s + m1) + e00);
  const float v = (e11 * d1 - e01 * d2) * r3.w, w = (e00 * d2 - e01 * d1) * r3.w;
  const float qf = fmaf(v, fmaf(v, e00, fmaf(2.f * w, e01, m1)), fmaf(w, fmaf(w, e11, m2), s));
  const bool in = fminf(fminf(v, w), 1.f - (v + w)) >= 0.f;
  const float q = fminf(fminf(q1, q2), q3);
  return fmaxf(in ? fminf(q, qf) : q, 0.f);
}

// The cut that goes with a distance of tri_dist2_fast: the near-tie margin
// (Cands::reach) widened by the errors of this distance and of the one to be
// admitted, 2e-6 (d + sqrt(3) h)^2 <= 3e-6 d^2 + 1.8e-5 h^2 of cancellation and
// 4e-5 h^2 of thin triangles (the square root by the hardware's approximation,
// from above).
constexpr float kFastRel = 4e-6f;   // of d^2, 8e-7 of it the near-tie margin's
constexpr float kFastAbs = 1e-4f;   // of h^2
__device__ __forceinline__ float fast_cut(float q, float mabs, float h2) {
  const float m = 2.f * mabs;
  return fmaf(q, 1.f + kFastRel, fmaf(2.001f * m, q * rsqrtf(fmaxf(q, 1e-30f)), fmaf(m, m, kFastAbs * h2)));
}

// Closest point to p on triangle t (its search record).
__device__ __forceinline__ float3 closest_on(const float3 p, const float4* __restrict__ rec) {
  const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
  const float3 ap = make_float3(p.x - r0.x, p.y - r0.y, p.z - r0.z);
  float v, w;
  rec_weights(ap, r1.x * ap.x + r1.y * ap.y + r1.z * ap.z, r2.x * ap.x + r2.y * ap.y + r2.z * ap.z, r0, r1, r2, r3, v,
              w);
  return make_float3(r0.x + (v * r1.x + w * r2.x), r0.y + (v * r1.y + w * r2.y), r0.z + (v * r1.z + w * r2.z));
}

// ---- a warp per node: the coarsest lattice (LIST false: every stride-th node
// from nothing, after a descent to the nearest leaf) or the deferred nodes
// (LIST true: from the closest triangle found so far).  The 32 lanes bound 32
// octree children, then 32 cubes, then test 32 triangles at a time against the
// one node by tri_dist2_fast; the cut is the warp's smallest, and the triangles
// within it wait for the exact test.
constexpr int kNodeTris = 192;   // triangles waiting: below 32, plus 32 cubes of at most 5
template <bool COUNT, bool TIES, bool LIST>
__global__ void __launch_bounds__(kWarps * 32) sdf_node_kernel(const __grid_constant__ Search S,
                                                               const __grid_constant__ PyrInfo pi, int stride) {
  __shared__ unsigned s_stk[kWarps][kSrchStack];
  __shared__ unsigned char s_msk[kWarps][kSrchStack];
  __shared__ int s_leaf[kWarps][40];
  __shared__ int s_tri[kWarps][kNodeTris];
  __shared__ int s_hit[kWarps][64];
  __shared__ float s_hq[kWarps][64];
  __shared__ int s_off[12], s_dim[12];
  if (threadIdx.x < 12) {
    s_off[threadIdx.x] = (int)pi.off[threadIdx.x];
    s_dim[threadIdx.x] = pi.dim[threadIdx.x];
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned* stk = s_stk[w];
  unsigned char* msk = s_msk[w];
  int* leaf = s_leaf[w];
  int* tri = s_tri[w];
  int* hit = s_hit[w];
  float* hq = s_hq[w];
  const int n = S.n;
  const int nl = (n + stride - 1) / stride;
  const unsigned total = LIST ? S.st->ndefer : (unsigned)nl * nl * nl;
  const int top = pi.nlev - 1;
  const unsigned root_mask = __float_as_uint(S.pyr[2 * (int64_t)s_off[top]].w) & 0xffu;
  const bool empty = S.pyr[2 * (int64_t)s_off[top]].w < 0.f;
  const float mabs = TIES ? kTieAbs * S.coord : 0.f, h2 = S.h * S.h;
  for (unsigned it = blockIdx.x * kWarps + w; it < total; it += gridDim.x * kWarps) {
    int i, j, k;
    if (LIST) {
      const unsigned o = (unsigned)S.defer[it];
      const unsigned row = o / (unsigned)n;
      i = (int)(o - row * n), j = (int)(row % n), k = (int)(row / n);
    } else {
      const unsigned row = it / (unsigned)nl;
      i = stride * (int)(it - row * nl), j = stride * (int)(row % nl), k = stride * (int)(row / nl);
    }
    const int64_t o = lin3(i, j, k, n);
    const float3 p = make_float3(S.axis[i], S.axis[n + j], S.axis[2 * n + k]);
    Cands<TIES> c;
    c.init(true);
    unsigned long long c_nodes = 0, c_leaves = 0, c_tests = 0;
    float cut = INFINITY;   // of the fast distances
    int nhit = 0;
    // the waiting triangles still within the cut, moved together
    auto drop_hits = [&]() {
      int kept = 0;
#pragma unroll
      for (int q = 0; q < 64; q += 32) {
        const int t = hit[q + lane];
        const float d = hq[q + lane];
        const bool in = q + lane < nhit && d < cut;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
          hit[kept + __popc(m & below)] = t;
          hq[kept + __popc(m & below)] = d;
        }
        kept += __popc(m);
        __syncwarp();
      }
      nhit = kept;
    };
    // ... into the lanes' candidate lists
    auto run_hits = [&]() {
      for (int q = lane; q < nhit; q += 32) c.offer(p, hit[q], S, nullptr);
      nhit = 0;
      __syncwarp();
    };
    auto test = [&](bool on, int t) {
      if (COUNT) c_tests += (unsigned)__popc(__ballot_sync(0xffffffffu, on));
      float q = INFINITY;
      if (on) q = tri_dist2_fast(p, S.tris_s + kTriRec * (int64_t)t);
      const bool in = q < cut;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (m) {
        cut = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(in ? fminf(cut, fast_cut(q, mabs, h2)) : cut)));
        if (in) {
          hit[nhit + __popc(m & below)] = t;
          hq[nhit + __popc(m & below)] = q;
        }
        nhit += __popc(m);
        __syncwarp();
        if (nhit > 32) {
          drop_hits();
          if (nhit > 32) run_hits();
        }
      }
    };
    if (LIST) {
      // its cube finds the seed again: only the cut is kept
      const int seed = S.seed_ids[o];
      test(lane == 0 && seed >= 0, seed);
      nhit = 0;
    } else if (!empty) {
      // descent by the children's bounds; the leaf's triangles give the first cut
      int x = 0, y = 0, z = 0;
      unsigned mask = root_mask;
      for (int lev = top; lev > 0; --lev) {
        const int dc = s_dim[lev - 1];
        float key = INFINITY;
        unsigned cm = 0;
        if (lane < 8 && ((mask >> lane) & 1u)) {
          const int cx = 2 * x + (lane & 1), cy = 2 * y + ((lane >> 1) & 1), cz = 2 * z + (lane >> 2);
          const int64_t cg = s_off[lev - 1] + ((int64_t)cz * dc + cy) * dc + cx;
          const float4 A = S.pyr[2 * cg];
          key = puck_dist2(p, A, S.pyr[2 * cg + 1]);
          cm = __float_as_uint(A.w) & 0xffu;
        }
        const unsigned kb = __float_as_uint(key);
        const int at = __ffs(__ballot_sync(0xffffffffu, kb == __reduce_min_sync(0xffffffffu, kb))) - 1;
        mask = __shfl_sync(0xffffffffu, cm, at);
        x = 2 * x + (at & 1), y = 2 * y + ((at >> 1) & 1), z = 2 * z + ((at >> 2) & 1);
      }
      const int li = leaf_index(x, y, z, S.nb);
      const int q0 = S.leaf_off[li], q1 = (int)min((int64_t)S.leaf_off[li + 1], S.cap);
      for (int q = q0; q < q1; q += 32) test(q + lane < q1, min(q + lane, q1 - 1));
      nhit = 0;   // the leaf's cubes come again
    }
    int sp = 0, nlf = 0, nt = 0;
    if (!empty) {
      if (lane == 0) {
        stk[0] = pack_node(top, 0, 0, 0);
        msk[0] = (unsigned char)root_mask;
      }
      sp = 1;
    }
    __syncwarp();
    while (sp > 0 || nlf > 0 || nt > 0) {
      if (nt >= 32 || (sp == 0 && nlf == 0)) {
        // 32 triangles
        const int m = min(nt, 32);
        nt -= m;
        const int t = tri[nt + min(lane, m - 1)];
        test(lane < m, t);
        __syncwarp();
      } else if (nlf >= 4 || sp == 0) {
        // the cubes of four leaves
        const int m = min(nlf, 4);
        nlf -= m;
        if (COUNT) c_leaves += m;
        int q0 = 0, cnt = 0;
        if ((lane >> 3) < m) leaf_cube(S, leaf[nlf + (lane >> 3)], lane & 7, q0, cnt);
        if (cnt > 0 && !(puck_dist2(p, S.cell_pyr[2 * (int64_t)q0], S.cell_pyr[2 * (int64_t)q0 + 1]) < cut)) cnt = 0;
        int at = cnt;   // inclusive prefix sum of the counts
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, at, d);
          if (lane >= d) at += v;
        }
        const int all = __shfl_sync(0xffffffffu, at, 31);
        at += nt - cnt;
        for (int q = 0; q < cnt; ++q) tri[at + q] = q0 + q;
        nt += all;
        __syncwarp();
      } else {
        // the children of up to four nodes
        const int m = sp <= kPopFour ? min(sp, 4) : 1;
        sp -= m;
        const int sl = lane >> 3, ch = lane & 7;
        unsigned e = 0, mask = 0;
        if (sl < m) {
          e = stk[sp + sl];
          mask = msk[sp + sl];
        }
        __syncwarp();
        if (COUNT) c_nodes += m;
        bool keep = false;
        const int lev = (int)(e >> 27);
        const int cx = 2 * (int)(e & 511u) + (ch & 1), cy = 2 * (int)((e >> 9) & 511u) + ((ch >> 1) & 1),
                  cz = 2 * (int)((e >> 18) & 511u) + (ch >> 2);
        unsigned cm = 0;
        if ((mask >> ch) & 1u) {
          const int dc = s_dim[lev - 1];
          const int64_t cg = s_off[lev - 1] + ((int64_t)cz * dc + cy) * dc + cx;
          const float4 A = S.pyr[2 * cg];
          keep = puck_dist2(p, A, S.pyr[2 * cg + 1]) < cut;
          cm = __float_as_uint(A.w) & 0xffu;
        }
        const bool lf = keep && lev == 1;
        const unsigned mn = __ballot_sync(0xffffffffu, keep && !lf), ml = __ballot_sync(0xffffffffu, lf);
        if (lf) {
          leaf[nlf + __popc(ml & below)] = leaf_index(cx, cy, cz, S.nb);
        } else if (keep) {
          const int at = sp + __popc(mn & below);
          stk[at] = pack_node(lev - 1, cx, cy, cz);
          msk[at] = (unsigned char)cm;
        }
        sp += __popc(mn);
        nlf += __popc(ml);
        __syncwarp();
      }
    }
    drop_hits();
    Cands<TIES> r;
    r.init(true);
    constexpr int NC = Cands<TIES>::NC;
    run_hits();
    // the lanes' lists merged: the smallest entry of all, its feature (and its
    // triangle) dropped everywhere, and again
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const unsigned kb = __float_as_uint(c.cd[0]);
      const unsigned best = __reduce_min_sync(0xffffffffu, kb);
      // equal distances: as in the list (without ranks by the triangle index)
      const bool head = kb == best && c.ct[0] != -1;
      const unsigned order = !head ? 0xffffffffu : TIES ? __float_as_uint(S.tris_lo[c.ct[0]].a.w) : (unsigned)c.ct[0];
      const unsigned least = __reduce_min_sync(0xffffffffu, order);
      const unsigned id = __reduce_min_sync(0xffffffffu, head && order == least ? (unsigned)c.ct[0] : 0xffffffffu);
      const int own = __ffs(__ballot_sync(0xffffffffu, id != 0xffffffffu && c.ct[0] == (int)id)) - 1;
      const unsigned key = __shfl_sync(0xffffffffu, c.ck[0], max(own, 0));
      if (id != 0xffffffffu) {
        r.cd[q] = __uint_as_float(best);
        r.ct[q] = (int)id;
      }
#pragma unroll
      for (int a = 0; a < NC; ++a) {
        if (c.ct[a] != -1 && id != 0xffffffffu &&
            (c.ct[a] == (int)id || (TIES && c.ck[a] == key))) {
          c.cd[a] = INFINITY;
          c.ct[a] = -1;
        }
      }
      // the dropped entry (at most one: a lane lists a feature once) moves to the end
#pragma unroll
      for (int a = 0; a + 1 < NC; ++a)
        if (c.cd[a + 1] < c.cd[a]) c.swap(a, a + 1);
    }
    r.cut = r.reach(mabs);
    if (COUNT && lane == 0) {
      atomicAdd(&S.st->sdf_cnt[0], c_nodes);
      atomicAdd(&S.st->sdf_cnt[1], c_leaves);
      atomicAdd(&S.st->sdf_cnt[2], c_tests);
    }
    store_nodes<COUNT, TIES>(S, r, lane == 0, o, true, lane);
    __syncwarp();
  }
}

// ---- a block per 8 x 8 x 4 nodes of the lattice of `stride` S (those whose
// coordinates are not all multiples of 2 S), a warp per patch of 4 x 4 x 2.  A
// 2 x 2 x 2 group of nodes (8 lanes) shares the eight nodes of the coarser
// lattice's cell that holds it, whose closest triangles seed its nodes; a
// node's cut is then near its final value and the rest is certification:
//   the block walks the octree level by level, one child per thread, then the
//     leaves' cubes, against its box (puck_reaches): a list of cubes;
//   each warp passes the list against its patch's box, one cube per lane, and
//     the cubes left against its 32 nodes' own cuts, one cube per lane and
//     one node at a time: a queue of (node, cube) pairs;
//   the lanes take the pairs as they come free and test their triangles by
//     tri_dist2_fast; a triangle within its node's cut waits at the node's
//     lane for the exact test and the candidate list.
constexpr int kPatchWarps = 8;
constexpr int kFront = 1024;      // octree nodes of a level within reach of a block (more: its nodes are deferred)
constexpr int kChunk = 128;       // leaves whose cubes are taken at a time
constexpr int kBlockCubes = 8 * kChunk;
constexpr int kCubes = 64;        // a warp's cubes: taken 32 at a time, below 32 left plus one step's 32
constexpr int kQueue = 512;       // a warp's (node, cube) pairs: flushed above kQueue - 32, plus one node's 32
constexpr int kHits = 8;          // triangles within a node's cut, waiting for the exact test
template <bool COUNT, bool TIES>
__global__ void __launch_bounds__(kPatchWarps * 32, 4) sdf_patch_kernel(const __grid_constant__ Search S,
                                                                        const __grid_constant__ PyrInfo pi,
                                                                        int stride, int leaf_max) {
  __shared__ float4 s_bref[8];                            // the block's reference points
  __shared__ float4 s_ref[kPatchWarps][8];                // the patches'
  __shared__ float4 s_node[kPatchWarps][32];              // node position and cut (of the fast distances)
  __shared__ unsigned s_leaf[kFront];                     // the block's walk: even levels, the leaves last
  union Walk {
    unsigned front[kFront];                               // odd levels
    unsigned short queue[kPatchWarps][kQueue];            // then the warps' pairs: node << 11 | block cube
  };
  __shared__ Walk s_w;
  __shared__ int s_bcube[kBlockCubes];                    // first triangle
  __shared__ int s_hit[kPatchWarps][kHits][32];
  __shared__ int s_nhit[kPatchWarps][32];
  __shared__ int s_seed[kPatchWarps][32];                 // per group: the closest triangles of its cell's corners
  __shared__ unsigned short s_hq[kPatchWarps][kHits][32]; // the hits' distances, the top half of the float
  __shared__ unsigned short s_cube[kPatchWarps][kCubes];  // block cubes
  __shared__ unsigned char s_fmask[2][kFront];
  __shared__ unsigned char s_bcnt[kBlockCubes];
  __shared__ int s_off[12], s_dim[12], s_num[13];
  __shared__ unsigned s_has;
  static_assert(kBlockCubes <= 2048, "pairs hold 11 bits of cube");
  const int tid = threadIdx.x;
  if (tid < 12) {
    s_off[tid] = (int)pi.off[tid];
    s_dim[tid] = pi.dim[tid];
  }
  if (tid < 13) s_num[tid] = 0;   // per level: the front's nodes; 12: the cubes
  if (tid == 0) s_has = 0u;
  __syncthreads();
  const int n = S.n;
  const int w = tid >> 5, lane = tid & 31, grp = lane >> 3, sub = lane & 7;
  const unsigned below = (1u << lane) - 1u;
  const int nl = (n + stride - 1) / stride;
  const int ntx = (nl + 7) / 8;
  const int bx = blockIdx.x % ntx, by = (blockIdx.x / ntx) % ntx;
  // the middle slabs first: the blocks with the most candidates lie inside the
  // body, and what runs last should be short
  const int zq = blockIdx.x / (ntx * ntx), nz = gridDim.x / (ntx * ntx);
  const int bz = nz / 2 + ((zq & 1) ? -((zq + 1) >> 1) : (zq >> 1));
  const int i = stride * (bx * 8 + 4 * (w & 1) + 2 * (grp & 1) + (sub & 1));
  const int j = stride * (by * 8 + 4 * ((w >> 1) & 1) + 2 * (grp >> 1) + ((sub >> 1) & 1));
  const int k = stride * (bz * 4 + 2 * (w >> 2) + (sub >> 2));
  const bool here = i < n && j < n && k < n;
  const bool valid = here && ((i | j | k) & stride);
  const unsigned vmask = __ballot_sync(0xffffffffu, valid);
  const int64_t o = lin3(i, j, k, n);
  // positions past the grid's edge only place the boxes
  auto pos = [&](int a, int q) { return q < n ? S.axis[a * n + q] : S.axis[a * n + n - 1] + (float)(q - n + 1) * S.h; };
  const float3 p = make_float3(pos(0, i), pos(1, j), pos(2, k));
  const float mabs = TIES ? kTieAbs * S.coord : 0.f, h2 = S.h * S.h;
  Cands<TIES> c;
  c.init(valid);
  int bt = -1;
  unsigned c_tests = 0;
  // waiting triangles that a later, nearer one has put out of reach leave
  // their slots
  auto drop_hits = [&]() {
    const int mine = min(s_nhit[w][lane], kHits);
    const float cut = s_node[w][lane].w;
    int kept = 0;
#pragma unroll
    for (int q = 0; q < kHits; ++q) {
      if (q < mine) {
        const unsigned short hq = s_hq[w][q][lane];
        if (__uint_as_float((unsigned)hq << 16) < cut) {
          s_hit[w][kept][lane] = s_hit[w][q][lane];
          s_hq[w][kept][lane] = hq;
          ++kept;
        }
      }
    }
    s_nhit[w][lane] = kept;
    return kept;
  };
  // the waiting triangles into the candidate lists
  auto run_hits = [&]() {
    const int mine = drop_hits();
    const int most = __reduce_max_sync(0xffffffffu, mine);
#pragma unroll 1
    for (int q = 0; q < most; ++q) {
      if (q < mine) c.offer(p, s_hit[w][q][lane], S, &s_seed[w][8 * grp]);
    }
    s_nhit[w][lane] = 0;
    __syncwarp();
  };
  {
    // seeds: lane `sub` of a group reads the closest triangle of its corner of
    // the coarser lattice's cell; each distinct one is tested once, for the
    // node's first cut (within which its cube finds it again)
    const int s2 = 2 * stride;
    const int ci = (i & ~(s2 - 1)) + s2 * (sub & 1), cj = (j & ~(s2 - 1)) + s2 * ((sub >> 1) & 1),
              ck = (k & ~(s2 - 1)) + s2 * (sub >> 2);
    int t = -1;
    if (ci < n && cj < n && ck < n) t = S.seed_ids[lin3(ci, cj, ck, n)];
    const unsigned same = __match_any_sync(0xffffffffu, t) & (0xffu << (8 * grp));
    unsigned left = (__ballot_sync(0xffffffffu, t >= 0 && lane == __ffs(same) - 1) >> (8 * grp)) & 0xffu;
    float bq = INFINITY;
    while (__any_sync(0xffffffffu, left != 0u)) {
      const int tq = __shfl_sync(0xffffffffu, t, left ? 8 * grp + __ffs(left) - 1 : lane);
      if (here && left != 0u) {
        const float q = tri_dist2_fast(p, S.tris_s + kTriRec * (int64_t)tq);
        if (q < bq) {
          bq = q;
          bt = tq;
        }
      }
      left &= left - 1u;
    }
    s_nhit[w][lane] = 0;
    s_seed[w][lane] = t;
    s_node[w][lane] = make_float4(p.x, p.y, p.z, !valid ? -INFINITY : bt < 0 ? INFINITY : fast_cut(bq, mabs, h2));
  }
  // the boxes of the patch and of the block: half extents (plus the rounding
  // of the positions), centres, and reference points: the closest points of
  // their eight corner nodes (a corner past the grid's edge takes another's)
  const float eg = 0.5f * (float)stride * S.h * (1.f + 1e-5f) + 2e-7f * S.coord;
  const float3 ep = make_float3(3.f * eg, 3.f * eg, eg), eb = make_float3(7.f * eg, 7.f * eg, 3.f * eg);
  const float epl = 4.3588995f * eg, ebl = 10.344085f * eg;   // sqrt(19), sqrt(107)
  auto mid = [&](float v) {
    return 0.5f * (__shfl_sync(0xffffffffu, v, 0) + __shfl_sync(0xffffffffu, v, 31));
  };
  const float3 pp = make_float3(mid(p.x), mid(p.y), mid(p.z));
  const float3 pb = make_float3(0.5f * (pos(0, stride * 8 * bx) + pos(0, stride * (8 * bx + 7))),
                                0.5f * (pos(1, stride * 8 * by) + pos(1, stride * (8 * by + 7))),
                                0.5f * (pos(2, stride * 4 * bz) + pos(2, stride * (4 * bz + 3))));
  const unsigned with = __ballot_sync(0xffffffffu, here && bt >= 0);
  {
    // corner q of a patch: the node of group (q & 3) at the same corner; the
    // block's corner w lies at the corner w of its patch w
    const int cl = 8 * (lane & 3) + (lane & 7);
    const int ref = (with >> cl) & 1u ? cl : 31 - __clz(with | 1u);
    const float3 rp = make_float3(__shfl_sync(0xffffffffu, p.x, ref), __shfl_sync(0xffffffffu, p.y, ref),
                                  __shfl_sync(0xffffffffu, p.z, ref));
    const int rt = __shfl_sync(0xffffffffu, bt, ref);
    if (lane < 8 && with != 0u) {
      const float3 y = closest_on(rp, S.tris_s + kTriRec * (int64_t)rt);
      s_ref[w][lane] = make_float4(y.x, y.y, y.z, reach_of(pp, y, epl, S.coord));
      if (lane == w) {
        s_bref[w] = make_float4(y.x, y.y, y.z, reach_of(pb, y, ebl, S.coord));
        atomicOr(&s_has, 1u << w);
      }
    }
  }
  // the walk begins at the first level of at most 4 nodes per axis
  int l0 = pi.nlev - 1;
  while (l0 > 1 && s_dim[l0 - 1] <= 4) --l0;
  if (tid < s_dim[l0] * s_dim[l0] * s_dim[l0]) {
    const int d = s_dim[l0];
    const int z = tid / (d * d), r = tid - z * d * d, y = r / d, x = r - y * d;
    const float rad = S.pyr[2 * (int64_t)(s_off[l0] + tid)].w;
    (l0 & 1 ? s_w.front : s_leaf)[tid] = ((unsigned)z << 18) | ((unsigned)y << 9) | (unsigned)x;
    s_fmask[l0 & 1][tid] = rad < 0.f ? 0 : (unsigned char)(__float_as_uint(rad) & 0xffu);   // empty: no children
    if (tid == 0) s_num[l0] = d * d * d;
  }
  __syncthreads();
  const unsigned has = s_has;
  if (has != 0xffu && has != 0u) {   // a patch without nodes leaves its corner to another's reference
    if (tid < 8 && !((has >> tid) & 1u)) s_bref[tid] = s_bref[__ffs(has) - 1];
    __syncthreads();
  }
  bool heavy = false;
  int m = 0;
  if (has != 0u) {
    // the octree, a level at a time; level 0 are the leaves (their indices)
    for (int lev = l0; lev > 0; --lev) {
      m = s_num[lev];
      if (m > kFront) break;
      const unsigned* cur = lev & 1 ? s_w.front : s_leaf;
      unsigned* nxt = lev & 1 ? s_leaf : s_w.front;
      const int dc = s_dim[lev - 1];
      for (int b0 = 0; b0 < 8 * m; b0 += kPatchWarps * 32) {
        const int q = b0 + tid, ch = q & 7;
        bool keep = false;
        unsigned cm = 0, ent = 0;
        if (q < 8 * m && (s_fmask[lev & 1][q >> 3] >> ch) & 1u) {
          const unsigned e = cur[q >> 3];
          const int cx = 2 * (int)(e & 511u) + (ch & 1), cy = 2 * (int)((e >> 9) & 511u) + ((ch >> 1) & 1),
                    cz = 2 * (int)(e >> 18) + (ch >> 2);
          const int64_t cg = s_off[lev - 1] + ((int64_t)cz * dc + cy) * dc + cx;
          const float4 A = S.pyr[2 * cg];
          keep = puck_reaches<8>(pb, s_bref, eb, ebl, A, S.pyr[2 * cg + 1]);
          cm = __float_as_uint(A.w) & 0xffu;
          ent = lev == 1 ? (unsigned)leaf_index(cx, cy, cz, S.nb)
                         : ((unsigned)cz << 18) | ((unsigned)cy << 9) | (unsigned)cx;
        }
        const unsigned b = __ballot_sync(0xffffffffu, keep);
        int at = 0;
        if (lane == 0 && b) at = atomicAdd(&s_num[lev - 1], __popc(b));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & below);
        if (keep && at < kFront) {
          nxt[at] = ent;
          s_fmask[(lev & 1) ^ 1][at] = (unsigned char)cm;
        }
      }
      __syncthreads();
      m = s_num[lev - 1];
    }
    heavy = m > leaf_max;
  }
  if (heavy) {
    if (!vmask) return;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&S.st->ndefer, (unsigned)__popc(vmask));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (valid) {
      S.defer[base + __popc(vmask & below)] = (int)o;
      S.seed_ids[o] = bt;
    }
    return;
  }
  int ncube = 0, nq = 0;
  unsigned short* queue = s_w.queue[w];
  // the queued pairs' triangles, a lane taking the next pair when it is
  // through with one
  auto run_queue = [&]() {
    __syncwarp();
    int next = 0, t = 0, t1 = 0, v = 0;
    float3 x = p;
    while (true) {
      const unsigned free = __ballot_sync(0xffffffffu, t == t1);
      if (t == t1) {
        const int at = next + __popc(free & below);
        if (at < nq) {
          const unsigned e = queue[at];
          v = (int)(e >> 11);
          t = s_bcube[e & 2047u];
          t1 = t + s_bcnt[e & 2047u];
          x = f3(s_node[w][v]);
        }
      }
      next += __popc(free);
      const bool on = t < t1;
      if (!__any_sync(0xffffffffu, on)) break;
      if (COUNT) c_tests += (unsigned)__popc(__ballot_sync(0xffffffffu, on));
      bool hit = false;
      float q = 0.f;
      const int tq = t;
      if (on) {
        q = tri_dist2_fast(x, S.tris_s + kTriRec * (int64_t)t);
        hit = q < *reinterpret_cast<volatile float*>(&s_node[w][v].w);
        ++t;
      }
      while (__any_sync(0xffffffffu, hit)) {
        if (hit) {
          atomicMin(reinterpret_cast<int*>(&s_node[w][v].w), __float_as_int(fast_cut(q, mabs, h2)));
          const int at = atomicAdd(&s_nhit[w][v], 1);
          if (at < kHits) {
            s_hit[w][at][v] = tq;
            s_hq[w][at][v] = (unsigned short)(__float_as_uint(q) >> 16);
            hit = false;
          }
        }
        if (__any_sync(0xffffffffu, hit)) {   // a node's slots are full
          __syncwarp();
          if (__any_sync(0xffffffffu, drop_hits() > kHits - 2)) run_hits();
          __syncwarp();
        }
      }
    }
    nq = 0;
    __syncwarp();
  };
  // up to 32 listed cubes against each node's own cut
  auto run_cubes = [&](bool last) {
    const int take = min(ncube, 32);
    ncube -= take;
    const bool done = last && ncube == 0;
    // 16 cubes or fewer: two lanes share a cube, each with half of the nodes
    const bool halves = take <= 16;
    const int at0 = halves ? lane & 15 : lane;
    const int bi = at0 < take ? s_cube[w][ncube + at0] : 0;
    const int64_t q0 = s_bcube[bi];
    const float4 A = S.cell_pyr[2 * q0], B = S.cell_pyr[2 * q0 + 1];
    unsigned mine = 0;   // the cube's nodes
    const int v0 = halves ? lane & 16 : 0, v1 = halves ? 16 : 32;
#pragma unroll 8
    for (int v = 0; v < v1; ++v) {
      const float4 nd = s_node[w][v0 + v];
      if (puck_dist2(f3(nd), A, B) < nd.w) mine |= 1u << v;
    }
    mine = mine << v0;
    if (at0 >= take) mine = 0;
    // the pairs, cube by cube (the lanes that take them share triangles); what
    // does not fit waits for the queue to be worked off
    while (true) {
      int at = __popc(mine);   // inclusive prefix sum over the lanes
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, at, d);
        if (lane >= d) at += x;
      }
      const int all = __shfl_sync(0xffffffffu, at, 31);
      at += nq - __popc(mine);
      while (mine != 0u && at < kQueue) {
        queue[at++] = (unsigned short)(((__ffs(mine) - 1) << 11) | bi);
        mine &= mine - 1u;
      }
      nq = min(nq + all, kQueue);
      const bool more = __any_sync(0xffffffffu, mine != 0u);
      if (more || done) run_queue();
      if (!more) break;
    }
    __syncwarp();
  };
  for (int c0 = 0; c0 < m; c0 += kChunk) {
    if (c0 > 0) {
      __syncthreads();
      if (tid == 0) s_num[12] = 0;
      __syncthreads();
    }
    const int leaves = min(m - c0, kChunk);
    for (int b0 = 0; b0 < 8 * leaves; b0 += kPatchWarps * 32) {
      const int q = b0 + tid;
      int q0 = 0, cnt = 0;
      if (q < 8 * leaves) leaf_cube(S, (int)s_leaf[c0 + (q >> 3)], q & 7, q0, cnt);
      const bool in = cnt > 0 && puck_reaches<8>(pb, s_bref, eb, ebl, S.cell_pyr[2 * (int64_t)q0],
                                                 S.cell_pyr[2 * (int64_t)q0 + 1]);
      const unsigned b = __ballot_sync(0xffffffffu, in);
      int at = 0;
      if (lane == 0 && b) at = atomicAdd(&s_num[12], __popc(b));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & below);
      if (in) {
        s_bcube[at] = q0;
        s_bcnt[at] = (unsigned char)cnt;
      }
    }
    __syncthreads();
    if (!vmask) continue;
    const int nbc = s_num[12];
    for (int b0 = 0; b0 < nbc; b0 += 32) {
      const int q = b0 + lane;
      bool in = false;
      if (q < nbc) {
        const int64_t q0 = s_bcube[q];
        in = puck_reaches<4>(pp, s_ref[w], ep, epl, S.cell_pyr[2 * q0], S.cell_pyr[2 * q0 + 1]);
      }
      const unsigned b = __ballot_sync(0xffffffffu, in);
      if (in) s_cube[w][ncube + __popc(b & below)] = (unsigned short)q;
      ncube += __popc(b);
      __syncwarp();
      const bool last = b0 + 32 >= nbc;
      while (ncube >= 32 || (last && (ncube > 0 || nq > 0))) run_cubes(last);
    }
  }
  if (!vmask) return;
  run_hits();
  if (COUNT && lane == 0) {
    if (w == 0) {
      for (int l = 1; l < pi.nlev; ++l) atomicAdd(&S.st->sdf_cnt[0], (unsigned long long)s_num[l]);
      atomicAdd(&S.st->sdf_cnt[1], (unsigned long long)m);
    }
    atomicAdd(&S.st->sdf_cnt[2], (unsigned long long)c_tests);
  }
  c.cut = c.reach(mabs);
  store_nodes<COUNT, TIES>(S, c, valid, o, stride > 1, lane);
}

// Float-float decision between the float32 near-tie candidates of a node:
// distances (tri_dist2_ff_exact on the ~48-bit vertices) from the node position
// rounded once from double, the smaller wins; equal distances (a shared edge or
// vertex: the same closest point) take the smaller triangle index.  The node
// coordinates come from per-axis float-float tables built once per block, and
// chi >= c (c double) is tested as chi >= the smallest float not below c, so no
// node needs FP64.
//
// Candidates of one class (the top 32 - id_bits bits of feature_class) are not
// told apart here: the float32 distance, and where that is equal the order of
// the candidate list, decides between them beforehand.  Candidates that share
// their closest vertex or edge are of one class and the same closest point;
// distinct features meet in one by chance, two vertices about once in 1000
// (their ten bits), others once in 2^(32 - id_bits).  At such a node (50 of 16.8
// million at 256^3) the float32 choice stands, right to 4e-7 of the distance but
// not always the nearer one.  Deciding those in float-float too lowers the
// error of a dense 120^3 gradient against 64 bits by 0.2 to 8% (3.92e-4 -> 3.91e-4,
// 1.73e-6 -> 1.60e-6) but moves gradients of 256^3 grids by up to 4e-5 of their
// norm, past the 1e-5 that results are kept to from version to version: the
// rule stays.  id_bits comes from the grid, so that the choice does not depend on
// the handle's capacities.  The seeds are the triangles of the stride-2 lattice
// around the node.  The nodes of that lattice (even != 0) take their own pass,
// after the others have read their triangles.
__global__ void sdf_tie_kernel(const __grid_constant__ Search S, SurfParams g, int id_bits, int even) {
  __shared__ float2 s_ax[3][kMaxRes];
  const int n = g.res;
  for (int t = threadIdx.x; t < 3 * n; t += blockDim.x) {
    const int a = t / n, i = t % n;
    const double v = (g.lo[a] + (i + 0.5) * g.h) * (double)g.sc;
    const float hi = (float)v;
    s_ax[a][i] = make_float2(hi, (float)(v - (double)hi));
  }
  __syncthreads();
  const float cf = S.st->c_up;
  const unsigned un = (unsigned)n;
  const unsigned count = S.st->ntie;
  const int xi = S.st->fwd.xidx ^ 1;
  for (unsigned it = blockIdx.x * blockDim.x + threadIdx.x; it < count; it += gridDim.x * blockDim.x) {
    const unsigned o = (unsigned)S.tie_list[it];
    const unsigned row = o / un;
    const int i = (int)(o - row * un), j = (int)(row % un), k = (int)(row / un);
    if ((((i | j | k) & 1) == 0) != (even != 0)) continue;
    const int2 t23 = S.tie_cd.p[xi][it];
    int cand[kCand] = {S.tie_a[it], S.tie_b[it], t23.x, t23.y};
    const float2 px = s_ax[0][i], py = s_ax[1][j], pz = s_ax[2][k];
    const float3 p = make_float3(px.x, py.x, pz.x);
    int left = 0;
    float d2[kCand];
    unsigned cls[kCand];
#pragma unroll 1
    for (int q = 0; q < kCand; ++q) {
      if (cand[q] < 0) continue;
      float v, w;
      d2[q] = tri_dist2_rec(p, S.tris_s + kTriRec * (int64_t)cand[q], v, w);
      cls[q] = feature_class(v, w, S.tris, cand[q]) >> id_bits;
      for (int r = 0; r < q && cand[q] >= 0; ++r) {
        if (cand[r] < 0 || cls[r] != cls[q]) continue;
        bool stays = d2[r] < d2[q];
        if (d2[r] == d2[q]) {
          int seeds[8];
          for (int c = 0; c < 8; ++c) {
            const int ci = (i & ~1) + 2 * (c & 1), cj = (j & ~1) + 2 * ((c >> 1) & 1), ck = (k & ~1) + 2 * (c >> 2);
            seeds[c] = !even && ci < n && cj < n && ck < n ? S.ctri[lin3(ci, cj, ck, n)] : -1;
          }
          stays = comes_first(cand[r], cand[q], S.tris_lo, seeds);
        }
        cand[stays ? q : r] = -1;
      }
    }
#pragma unroll
    for (int q = 0; q < kCand; ++q) left += cand[q] >= 0;
    const Vec3<Ff> pf = {Ff(px.x, px.y), Ff(py.x, py.y), Ff(pz.x, pz.y)};
    Ff bd(INFINITY);
    int bi = -1;
    // one copy of the float-float distance in the loop: unrolled, the four
    // copies overflow the instruction cache
#pragma unroll 1
    for (int q = 0; q < kCand; ++q) {
      if (cand[q] < 0) continue;
      if (left == 1) {   // decided by its class: the distance stays the search's
        bi = cand[q];
        break;
      }
      const Ff d2 = tri_dist2_ff_exact(pf, S.tris_s + kTriRec * (int64_t)cand[q], S.tris[cand[q]], S.tris_lo[cand[q]],
                                       S.sc);
      if (bi < 0 || d2 < bd || (!(bd < d2) && cand[q] < bi)) {
        bd = d2;
        bi = cand[q];
      }
    }
    S.ctri[o] = bi;
    if (left == 1) continue;
    const float sgn = (S.chi[o] >= cf) ? 1.f : -1.f;
    const float val = sgn * sqrtf(__fadd_rn(bd.hi, bd.lo)) * S.us;
    S.phi[o] = val;
    if (S.sdf_out) S.sdf_out[o] = val;
  }
}

// n = grad phi / |grad phi|: central differences inside, second-order one-sided
// on the first and last node of each axis; 0 where |grad| is 0 or not finite.
// One thread per (x, y) column marches kNrmZ planes in z, keeping the
// column's previous, current and next phi in registers; x and y neighbours
// come through L1 from the warp's own row and the block's neighbouring rows.
// No index division, coalesced loads and stores of every plane.
constexpr int kNrmZ = 16;
__global__ void __launch_bounds__(256) normals_kernel(const float* __restrict__ phi, int n, double h,
                                                      float* __restrict__ nrm) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y;
  const int k0 = blockIdx.z * kNrmZ;
  if (i >= n || j >= n || k0 >= n) return;
  const int64_t nn = (int64_t)n * n, N = nn * n;
  const float inv2h = (float)(0.5 / h);
  const int k1 = min(k0 + kNrmZ, n);
  int64_t t = (int64_t)k0 * nn + (int64_t)j * n + i;
  float zm = k0 > 0 ? phi[t - nn] : 0.f;
  float zc = phi[t];
  for (int k = k0; k < k1; ++k, t += nn) {
    const float zp = k + 1 < n ? phi[t + nn] : 0.f;
    float gr[3];
    if (i == 0)
      gr[0] = -3.f * zc + 4.f * phi[t + 1] - phi[t + 2];
    else if (i == n - 1)
      gr[0] = 3.f * zc - 4.f * phi[t - 1] + phi[t - 2];
    else
      gr[0] = phi[t + 1] - phi[t - 1];
    if (j == 0)
      gr[1] = -3.f * zc + 4.f * phi[t + n] - phi[t + 2 * n];
    else if (j == n - 1)
      gr[1] = 3.f * zc - 4.f * phi[t - n] + phi[t - 2 * n];
    else
      gr[1] = phi[t + n] - phi[t - n];
    if (k == 0)
      gr[2] = -3.f * zc + 4.f * zp - phi[t + 2 * nn];
    else if (k == n - 1)
      gr[2] = 3.f * zc - 4.f * zm + phi[t - 2 * nn];
    else
      gr[2] = zp - zm;
#pragma unroll
    for (int a = 0; a < 3; ++a) gr[a] *= inv2h;
    const float m2 = gr[0] * gr[0] + gr[1] * gr[1] + gr[2] * gr[2];
    const bool ok = isfinite(m2) && m2 > 0.f;
    const float inv = ok ? rsqrtf(m2) : 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) nrm[a * N + t] = ok ? gr[a] * inv : 0.f;
    zm = zc;
    zc = zp;
  }
}

// ---- exact signed distance at arbitrary query points (Sec. 2.4, Eqs. 29-34,
// evaluated off the grid).  Two kernels: the distance search over queries
// sorted by cell, then the sign, one thread per query.

// Distance search: a warp of 32 neighbouring queries walks the octree depth
// first.  A popped node's puck is bounded by every lane against its own query
// and entered when it beats some lane's cut; children are pushed farthest first
// by the bound of the warp's first query, and a leaf's triangles are tested by
// all lanes, each the same (broadcast) triangle against its own query.
//
// The cut starts from an upper bound: the nearest node's |phi| plus the node's
// distance to q (triangle inequality), widened for the float rounding of both;
// with the nodes' closest triangles kept (SEEDS), those of the 8 nodes around q
// are offered first.  Writes the unsigned distance and the unit direction (q -
// y) / |q - y| to the closest surface point y (zero when q is on the surface,
// infinite distance when the mesh is empty).
//
// Bound: instruction issue and latency (10^6 uniform queries at 256^3, 2.61 ms:
// 1.48 10^9 warp instructions, 62% of the issue slots at 40% occupancy, waits on
// global loads 4.5 of 11 cycles an instruction; DRAM 1%).
template <bool SEEDS>
__global__ void __launch_bounds__(kWarps * 32, 8) sdf_query_kernel(const float* __restrict__ phi, SurfParams g,
                                                                const Tri* __restrict__ tris,
                                                                const float4* __restrict__ tris_s,
                                                                const int* __restrict__ leaf_off, int64_t cap,
                                                                const float4* __restrict__ pyr, PyrInfo pi,
                                                                const float4* __restrict__ sorted,
                                                                const int* __restrict__ total,
                                                                const int* __restrict__ ctri,
                                                                float* __restrict__ dist_out,
                                                                float* __restrict__ dir_out,
                                                                int* __restrict__ tri_out) {
  __shared__ uint2 s_node[kWarps][kStack];   // (packed level and coordinates, pyramid index)
  __shared__ int s_off[12];
  __shared__ int s_dim[12];
  if (threadIdx.x < 12) {
    s_off[threadIdx.x] = pi.off[threadIdx.x];
    s_dim[threadIdx.x] = pi.dim[threadIdx.x];
  }
  __syncthreads();
  const int m = *total;
  const int n = g.res;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float coord = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    coord = fmaxf(coord, (float)fmax(fabs(g.lo[a]), fabs(g.lo[a] + n * g.h)));
  coord *= g.sc;
  const int top = pi.nlev - 1;
  const int nb = (s_dim[0] + 1) / 2;
  uint2* stk = s_node[w];
  const int nwarps = gridDim.x * kWarps;
  for (int base = (blockIdx.x * kWarps + w) * 32; base < m; base += nwarps * 32) {
    const int k = base + lane;
    const bool valid = k < m;
    const float4 e = sorted[valid ? k : base];
    const float3 p = f3(e, g.sc);
    // nearest node and the bound |phi(node)| + |q - node|
    int ni[3];
    const float pq[3] = {e.x, e.y, e.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double f = ((double)pq[a] - g.lo[a]) / g.h - 0.5;
      ni[a] = (int)fmin(fmax(rint(f), 0.0), (double)(n - 1));
    }
    const int64_t o = lin3(ni[0], ni[1], ni[2], n);
    const float3 nd = make_float3((float)(g.lo[0] + (ni[0] + 0.5) * g.h) * g.sc,
                                  (float)(g.lo[1] + (ni[1] + 0.5) * g.h) * g.sc,
                                  (float)(g.lo[2] + (ni[2] + 0.5) * g.h) * g.sc);
    const float dn = sqrtf((p.x - nd.x) * (p.x - nd.x) + (p.y - nd.y) * (p.y - nd.y) + (p.z - nd.z) * (p.z - nd.z));
    const float bnd = (fabsf(phi[o]) * g.sc + dn) * (1.f + 1e-5f) + 1e-6f * coord;
    float cut = valid ? bnd * bnd : -INFINITY;
    float cd = INFINITY;
    int ct = -1;
    auto offer = [&](float d2, int t) {
      if (d2 < cut && d2 < cd) {
        cd = d2;
        ct = t;
        cut = d2;
      }
    };
    if (SEEDS && valid) {
      // the closest triangles of the 8 nodes around q
      int c0[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double f = ((double)pq[a] - g.lo[a]) / g.h - 0.5;
        c0[a] = (int)fmin(fmax(floor(f), 0.0), (double)(n - 2));
      }
#pragma unroll 1
      for (int qn = 0; qn < 8; ++qn) {
        const int t = ctri[lin3(c0[0] + (qn & 1), c0[1] + ((qn >> 1) & 1), c0[2] + (qn >> 2), n)];
        if (t >= 0) offer(tri_dist2_rec(p, tris_s + kTriRec * (int64_t)t), t);
      }
    }
    int sp = 1;
    if (lane == 0) stk[0] = make_uint2(pack_node(top, 0, 0, 0), (unsigned)s_off[top]);
    __syncwarp();
    while (sp > 0) {
      --sp;
      const uint2 ew = stk[sp];
      __syncwarp();
      const unsigned en = ew.x;
      const int gi = (int)ew.y;
      const int lev = (int)(en >> 27);
      const int x = (int)(en & 511u), y = (int)((en >> 9) & 511u), z = (int)((en >> 18) & 511u);
      const float4 An = pyr[2 * gi];
      const float lb = puck_dist2(p, An, pyr[2 * gi + 1]);
      if (!__any_sync(0xffffffffu, lb < cut)) continue;
      if (lev == 0) {
        const int li = leaf_index(x, y, z, nb);
        const int64_t s0 = leaf_off[li];
        const int64_t s1 = min((int64_t)leaf_off[li + 1], cap);
        for (int64_t t = s0; t < s1; ++t) offer(tri_dist2_rec(p, tris_s + kTriRec * t), (int)t);
        continue;
      }
      const int dc = s_dim[lev - 1];
      const int cbase = s_off[lev - 1];
      float key[8];
      uint2 ent[8];
      int nc = 0;
      const unsigned cmask = __float_as_uint(An.w) & 0xffu;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (!((cmask >> q) & 1u)) continue;
        const int cx = 2 * x + (q & 1), cy = 2 * y + ((q >> 1) & 1), cz = 2 * z + (q >> 2);
        const int cg = cbase + (cz * dc + cy) * dc + cx;
        const float d = puck_dist2(p, pyr[2 * cg], pyr[2 * cg + 1]);
        if (!__any_sync(0xffffffffu, d < cut)) continue;
        const float dm = __shfl_sync(0xffffffffu, d, 0);
        int q2 = nc;
        while (q2 > 0 && key[q2 - 1] < dm) {
          key[q2] = key[q2 - 1];
          ent[q2] = ent[q2 - 1];
          --q2;
        }
        key[q2] = dm;
        ent[q2] = make_uint2(pack_node(lev - 1, cx, cy, cz), (unsigned)cg);
        ++nc;
      }
      if (lane == 0)
        for (int q = 0; q < nc && sp + q < kStack; ++q) stk[sp + q] = ent[q];
      sp = min(sp + nc, kStack);
      __syncwarp();
    }
    if (!valid) continue;
    const int idx = __float_as_int(e.w);
    float3 dir = make_float3(0.f, 0.f, 0.f);
    if (ct >= 0 && cd > 0.f) {
      // residual q - y of the closest point y, as in the distance itself
      const float4* rec = tris_s + kTriRec * (int64_t)ct;
      const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
      const float3 ap = make_float3(p.x - r0.x, p.y - r0.y, p.z - r0.z);
      const float d1 = r1.x * ap.x + r1.y * ap.y + r1.z * ap.z;
      const float d2 = r2.x * ap.x + r2.y * ap.y + r2.z * ap.z;
      float v, wt;
      rec_weights(ap, d1, d2, r0, r1, r2, r3, v, wt);
      const float3 r = make_float3(ap.x - v * r1.x - wt * r2.x, ap.y - v * r1.y - wt * r2.y,
                                   ap.z - v * r1.z - wt * r2.z);
      const float len = sqrtf(r.x * r.x + r.y * r.y + r.z * r.z);
      if (len > 0.f) dir = make_float3(r.x / len, r.y / len, r.z / len);
      if (!(r0.w * r2.w * r3.w < kSliverKappa)) {
        // a sliver: the closest point's direction in FP64
        const Tri tr = tris[ct];
        const double pd[3] = {e.x, e.y, e.z}, ad[3] = {tr.a.x, tr.a.y, tr.a.z}, bd[3] = {tr.b.x, tr.b.y, tr.b.z},
                     cdv[3] = {tr.c.x, tr.c.y, tr.c.z};
        double bw64[3], dir64[3];
        closest_point_fp64(pd, ad, bd, cdv, bw64, dir64);
        dir = make_float3((float)dir64[0], (float)dir64[1], (float)dir64[2]);
      }
    }
    dist_out[idx] = ct >= 0 ? sqrtf(cd) * g.us : INFINITY;
    if (tri_out) tri_out[idx] = ct;
    if (dir_out) {
      dir_out[3 * (int64_t)idx] = dir.x;
      dir_out[3 * (int64_t)idx + 1] = dir.y;
      dir_out[3 * (int64_t)idx + 2] = dir.z;
    }
  }
}

__device__ __forceinline__ float orient3(float3 a, float3 b, float3 c, float3 d) {
  // (a - d) . ((b - d) x (c - d))
  const float3 ad = make_float3(a.x - d.x, a.y - d.y, a.z - d.z);
  const float3 bd = make_float3(b.x - d.x, b.y - d.y, b.z - d.z);
  const float3 cd = make_float3(c.x - d.x, c.y - d.y, c.z - d.z);
  return ad.x * (bd.y * cd.z - bd.z * cd.y) + ad.y * (bd.z * cd.x - bd.x * cd.z) + ad.z * (bd.x * cd.y - bd.y * cd.x);
}

// Squared distance from p to triangle (a, b, c): the closest point by Voronoi
// regions (Ericson, Real-Time Collision Detection, 5.1.5), in float.
__device__ float pt_tri_dist2(float3 p, float3 a, float3 b, float3 c) {
  const float3 ab = sub3(b, a), ac = sub3(c, a), ap = sub3(p, a);
  const float d1 = dot3(ab, ap), d2 = dot3(ac, ap);
  float3 y;
  if (d1 <= 0.f && d2 <= 0.f) {
    y = a;
  } else {
    const float3 bp = sub3(p, b);
    const float d3 = dot3(ab, bp), d4 = dot3(ac, bp);
    const float3 cp = sub3(p, c);
    const float d5 = dot3(ab, cp), d6 = dot3(ac, cp);
    const float vc = d1 * d4 - d3 * d2, vb = d5 * d2 - d1 * d6, va = d3 * d6 - d5 * d4;
    if (d3 >= 0.f && d4 <= d3) {
      y = b;
    } else if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) {
      const float t = d1 / (d1 - d3);
      y = make_float3(a.x + t * ab.x, a.y + t * ab.y, a.z + t * ab.z);
    } else if (d6 >= 0.f && d5 <= d6) {
      y = c;
    } else if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) {
      const float t = d2 / (d2 - d6);
      y = make_float3(a.x + t * ac.x, a.y + t * ac.y, a.z + t * ac.z);
    } else if (va <= 0.f && (d4 - d3) >= 0.f && (d5 - d6) >= 0.f) {
      const float t = (d4 - d3) / ((d4 - d3) + (d5 - d6));
      y = make_float3(b.x + t * (c.x - b.x), b.y + t * (c.y - b.y), b.z + t * (c.z - b.z));
    } else {
      const float den = va + vb + vc;
      const float v = den != 0.f ? vb / den : 0.f, ww = den != 0.f ? vc / den : 0.f;
      y = make_float3(a.x + v * ab.x + ww * ac.x, a.y + v * ab.y + ww * ac.y, a.z + v * ab.z + ww * ac.z);
    }
  }
  const float3 r = sub3(p, y);
  return dot3(r, r);
}

// Sign of every query by a parity test local to the cube that holds it (the
// query clamped into the node hull, where no triangle lies between it and its
// clamp): the segment from q to a corner v of the cube stays in the cube, so
// only that cube's marching-cubes triangles, regenerated from chi exactly as
// mc_emit_kernel writes them, can cross it; v's class is known (chi < c
// inside), and an odd number of crossings gives q the other class.  v is the
// corner farthest from the cube's triangles, so no triangle passes within
// rounding of it, among the corners off every cube face that q lies on (so
// the open segment avoids the faces, where triangles of the neighbouring cubes
// meet this cube's); q exactly at a corner takes that node's class.  A crossing needs q and v strictly on opposite sides of the
// triangle's plane and the line qv inside the triangle: the three orientations
// of the line against the triangle's edges agree in sign.  Each edge's
// orientation is evaluated once, in the order of its endpoints' global edge
// ids, and negated for the triangle that runs it the other way, so a line
// through an edge shared by two triangles counts for exactly one of them.  A
// float orientation can be wrong only when q lies within rounding of a
// triangle, where |phi| is of rounding size.  Non-finite queries get NaN and a
// zero gradient.
__global__ void query_sign_kernel(const float* __restrict__ q, int64_t m, const float* __restrict__ chi,
                                  ChiFF chiff, SurfParams g, const DevState* __restrict__ st,
                                  float* __restrict__ sdf_q, float* __restrict__ nrm_q) {
  const int n = g.res;
  const double c = st->c;
  const float c_up = st->c_up;
  const float2* __restrict__ xff = chiff.p[0] ? chiff.p[st->fwd.xidx] : nullptr;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    const float x0 = q[3 * t], x1 = q[3 * t + 1], x2 = q[3 * t + 2];
    if (!(isfinite(x0) && isfinite(x1) && isfinite(x2))) {
      sdf_q[t] = __int_as_float(0x7fc00000);
      if (nrm_q) nrm_q[3 * t] = nrm_q[3 * t + 1] = nrm_q[3 * t + 2] = 0.f;
      continue;
    }
    const float xs[3] = {x0, x1, x2};
    float qc[3];
    int cc[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double lo = g.lo[a] + 0.5 * g.h, hi = g.lo[a] + (n - 0.5) * g.h;
      const double v = fmin(fmax((double)xs[a], lo), hi);
      qc[a] = (float)v;
      cc[a] = min((int)floor((v - g.lo[a]) / g.h - 0.5), n - 2);
      cc[a] = max(cc[a], 0);
    }
    const int code = cube_code(chi, cc[0], cc[1], cc[2], n, c_up);
    // faces of the cube that q lies on: the segment's corner must be on the
    // opposite face, so that the open segment runs inside the cube (where only
    // this cube's triangles are); at a corner q takes that node's class
    int need_hi = 0, need_lo = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float flo = (float)(g.lo[a] + (cc[a] + 0.5) * g.h), fhi = (float)(g.lo[a] + (cc[a] + 1.5) * g.h);
      if (qc[a] == flo) need_hi |= 1 << a;
      if (qc[a] == fhi) need_lo |= 1 << a;
    }
    bool inside;
    if ((need_hi | need_lo) == 7) {
      const int corner = (need_lo & 1) | (((need_lo >> 1) & 1) << 1) | (((need_lo >> 2) & 1) << 2);
      inside = ((code >> corner) & 1) != 0;
    } else if (code == 0 || code == 255) {
      inside = code == 255;
    } else {
      // the cube's triangles
      float3 vt[kMaxTriPerCube][3];
      int gid[kMaxTriPerCube][3];
      const int ntri = c_mc_count[code];
      for (int tr = 0; tr < ntri; ++tr)
        for (int v = 0; v < 3; ++v) {
          const int ed = c_mc_tris[code][tr][v];
          int ox, oy, oz, ax;
          edge_lower_offset(ed, ox, oy, oz, ax);
          const int pi = cc[0] + ox, pj = cc[1] + oy, pk = cc[2] + oz;
          const int64_t pl = lin3(pi, pj, pk, n);
          const int64_t stride = (ax == 0) ? 1 : (ax == 1 ? (int64_t)n : (int64_t)n * n);
          double c1, c2;
          if (xff) {
            const float2 f1 = xff[pl], f2 = xff[pl + stride];
            c1 = (double)f1.x + (double)f1.y;
            c2 = (double)f2.x + (double)f2.y;
          } else {
            c1 = (double)chi[pl];
            c2 = (double)chi[pl + stride];
          }
          const double eta = (c - c1) / (c2 - c1);
          double pos[3] = {g.lo[0] + (pi + 0.5) * g.h, g.lo[1] + (pj + 0.5) * g.h, g.lo[2] + (pk + 0.5) * g.h};
          pos[ax] += eta * g.h;
          vt[tr][v] = make_float3((float)pos[0], (float)pos[1], (float)pos[2]);
          gid[tr][v] = (int)(3 * pl + ax);
        }
      // the corner farthest from the triangles
      int best_c = 0;
      float best_d = -1.f;
      float3 vpos = make_float3(0.f, 0.f, 0.f);
      for (int qn = 0; qn < 8; ++qn) {
        if ((qn & need_hi) != need_hi || (qn & need_lo) != 0) continue;
        const float3 cp = make_float3((float)(g.lo[0] + (cc[0] + (qn & 1) + 0.5) * g.h),
                                      (float)(g.lo[1] + (cc[1] + ((qn >> 1) & 1) + 0.5) * g.h),
                                      (float)(g.lo[2] + (cc[2] + (qn >> 2) + 0.5) * g.h));
        float dmin = INFINITY;
        for (int tr = 0; tr < ntri; ++tr) dmin = fminf(dmin, pt_tri_dist2(cp, vt[tr][0], vt[tr][1], vt[tr][2]));
        if (dmin > best_d) {
          best_d = dmin;
          best_c = qn;
          vpos = cp;
        }
      }
      const float3 qp = make_float3(qc[0], qc[1], qc[2]);
      int cross = 0;
      for (int tr = 0; tr < ntri; ++tr) {
        const float sq = orient3(vt[tr][0], vt[tr][1], vt[tr][2], qp);
        const float sv = orient3(vt[tr][0], vt[tr][1], vt[tr][2], vpos);
        if (!((sq > 0.f && sv < 0.f) || (sq < 0.f && sv > 0.f))) continue;
        int sg[3];
        for (int ei = 0; ei < 3; ++ei) {
          const int a = ei, b = (ei + 1) % 3;
          const bool fwd = gid[tr][a] < gid[tr][b];
          const float3 A = fwd ? vt[tr][a] : vt[tr][b], B = fwd ? vt[tr][b] : vt[tr][a];
          const int sgn = orient3(qp, vpos, A, B) >= 0.f ? 1 : -1;
          sg[ei] = fwd ? sgn : -sgn;
        }
        cross += (sg[0] == sg[1] && sg[1] == sg[2]) ? 1 : 0;
      }
      inside = (((code >> best_c) & 1) != 0) != ((cross & 1) != 0);
    }
    if (inside) {
      sdf_q[t] = -sdf_q[t];
      if (nrm_q) {
        nrm_q[3 * t] = -nrm_q[3 * t];
        nrm_q[3 * t + 1] = -nrm_q[3 * t + 1];
        nrm_q[3 * t + 2] = -nrm_q[3 * t + 2];
      }
    }
  }
}

PyrInfo pyramid_info(int nl) {
  PyrInfo pi;
  int d = nl;
  long long off = 0;
  pi.nlev = 0;
  while (true) {
    pi.dim[pi.nlev] = d;
    pi.off[pi.nlev] = off;
    off += (long long)d * d * d;
    ++pi.nlev;
    if (d == 1) break;
    d = (d + 1) / 2;
  }
  return pi;
}

}  // namespace

// nb = bricks per axis; the octree's leaves are the 2 nb sub-bricks per axis
size_t pyramid_nodes(int nb) {
  PyrInfo pi = pyramid_info(2 * nb);
  return (size_t)(pi.off[pi.nlev - 1] + 1);
}

size_t pyramid_aux_nodes(int nb) {
  PyrInfo pi = pyramid_info(2 * nb);
  return (size_t)(pi.off[pi.nlev - 1] + 1 - pi.off[1]);
}

int launch_isovalue(wgeo_handle* h, const float* points, int64_t n, int res, cudaStream_t s) {
  const SurfParams g = surf_params(h, res);
  const int nbk = grid_blocks(n, 256, kPartials);
  if (n > 0) {
    isovalue_kernel<<<nbk, 256, 0, s>>>(points, n, h->pcell, h->chi32, g, h->partials);
    WGEO_LAUNCH_CHECK();
  } else {
    WGEO_CUDA_TRY(cudaMemsetAsync(h->partials, 0, 2 * sizeof(double), s));
  }
  isovalue_finalize_kernel<<<1, 1024, 0, s>>>(h->partials, n > 0 ? nbk : 1, h->dstate);
  WGEO_LAUNCH_CHECK();
  return WGEO_OK;
}

int launch_mc_sdf_normals(wgeo_handle* h, int res, float* sdf_out, float* nrm_out, cudaStream_t s) {
  const SurfParams g = surf_params(h, res);
  const int nbricks = g.nb * g.nb * g.nb;
  int slot = stage_begin(h, kStMC, s);
  {
    // inside bits of the nodes (in the solver's idle correction buffer), then
    // the triangles per brick from them
    const int nw = div_up(res, 32);
    unsigned* bits = reinterpret_cast<unsigned*>(h->e32);
    mc_bits_kernel<<<dim3(nw, div_up((int64_t)res * res, 8 * kBitRows)), dim3(32, 8), 0, s>>>(h->chi32, res, nw,
                                                                                               h->dstate, bits);
    WGEO_LAUNCH_CHECK();
    const int64_t groups = (int64_t)div_up(res - 1, 32) * g.nb * g.nb;
    mc_count_kernel<<<grid_blocks(16 * groups, 256, h->num_sms * 16), 256, 0, s>>>(bits, g, nw, h->brick_count);
    WGEO_LAUNCH_CHECK();
  }
  int rc = exclusive_scan(h->brick_count, h->brick_off, nbricks, h->scan_tmp, s);
  if (rc) return rc;
  mc_total_kernel<<<1, 256, 0, s>>>(h->brick_off, nbricks, h->mesh_cap, h->leaf_off, h->dstate, g, h->axis);
  WGEO_LAUNCH_CHECK();
  // the bricks with triangles, listed in the solver's idle residual buffer
  int* live_bricks = reinterpret_cast<int*>(h->r32);
  WGEO_CUDA_TRY(cudaMemsetAsync(&h->dstate->nbrick_live, 0, sizeof(unsigned), s));
  mc_live_kernel<<<grid_blocks(nbricks, 256, h->num_sms * 16), 256, 0, s>>>(h->brick_off, nbricks, h->leaf_off,
                                                                            live_bricks, &h->dstate->nbrick_live);
  WGEO_LAUNCH_CHECK();
  // vertices from the refined float-float indicator (MIXED precision) and
  // their low parts for the near-tie decisions and the adjoint (when kept)
  mc_emit_kernel<<<std::min(div_up(nbricks, kMcBricks), h->num_sms * 8), 64 * kMcBricks, 0, s>>>(
      h->chi32, chiff_of(h), g, h->dstate, h->brick_off, h->mesh_cap, live_bricks, &h->dstate->nbrick_live,
      h->tris, h->tris_lo, h->leaf_off, h->leaf_cnt);
  WGEO_LAUNCH_CHECK();
  const PyrInfo pi = pyramid_info(2 * g.nb);
  const int64_t nleaf = (int64_t)pi.dim[0] * pi.dim[0] * pi.dim[0];
  // the live leaves, listed in the correction buffer (its inside bits are consumed)
  int* live = reinterpret_cast<int*>(h->e32);
  WGEO_CUDA_TRY(cudaMemsetAsync(&h->dstate->nleaf_live, 0, sizeof(unsigned), s));
  puck_leaf_scan_kernel<<<grid_blocks(nleaf, 256, h->num_sms * 16), 256, 0, s>>>(h->leaf_off, g.nb, h->mesh_cap,
                                                                                 h->pyramid, live, h->dstate);
  WGEO_LAUNCH_CHECK();
  const int live_grid = grid_blocks(nleaf, 256, h->num_sms * 8);
  puck_leaf_kernel<<<live_grid, 256, 0, s>>>(h->tris, h->tris_lo, h->leaf_off, h->leaf_cnt, g.nb, h->mesh_cap, live,
                                             h->dstate, h->pyramid, h->tris_s, h->cell_pyr, g.sc);
  WGEO_LAUNCH_CHECK();
  {
    // levels >= 1: sums per brick, sums up the tree, vertex maxima, pucks
    const int64_t nbr = (int64_t)g.nb * g.nb * g.nb;
    puck_sums_brick_kernel<<<grid_blocks(nbr, 128, 152 * 16), 128, 0, s>>>(h->tris, h->brick_off, g.nb,
                                                                           h->mesh_cap, h->pyr_sums, h->pyr_rth);
    WGEO_LAUNCH_CHECK();
    for (int l = 2; l < pi.nlev; ++l) {
      const int64_t np = (int64_t)pi.dim[l] * pi.dim[l] * pi.dim[l];
      puck_sums_up_kernel<<<grid_blocks(np, 128, 152 * 16), 128, 0, s>>>(
          h->pyr_sums, h->pyr_rth, pi.off[l - 1] - pi.off[1], pi.dim[l - 1], pi.off[l] - pi.off[1], pi.dim[l]);
      WGEO_LAUNCH_CHECK();
    }
    puck_rth_kernel<<<live_grid, 256, 0, s>>>(h->tris, h->leaf_off, g.nb, h->mesh_cap, pi, live, h->dstate,
                                              h->pyr_sums, h->pyr_rth);
    WGEO_LAUNCH_CHECK();
    const int64_t naux = pi.off[pi.nlev - 1] + 1 - pi.off[1];
    puck_finalize_kernel<<<grid_blocks(naux, 256, 152 * 16), 256, 0, s>>>(h->pyramid, h->pyr_sums, h->pyr_rth,
                                                                          naux, pi.off[1], g.sc);
    WGEO_LAUNCH_CHECK();
    puck_mask_kernel<<<grid_blocks(naux, 256, 152 * 16), 256, 0, s>>>(h->pyramid, pi);
    WGEO_LAUNCH_CHECK();
  }
  stage_end(h, kStMC, slot, s);
  slot = stage_begin(h, kStSDF, s);
  // the solver's residual / correction scratch is idle until the next solve:
  // it holds the near-tie candidates between the two kernels, and so does the
  // float-float iterate buffer that is not the current one (its index is on
  // the device); the near-tie list and the deferred nodes lie in the adjoint's
  // dL/dchi buffer, which is idle until a backward clears it
  const int64_t N = (int64_t)res * res * res;
  int* ctri = h->opt.keep_for_backward ? h->ctri : nullptr;
  Search S;
  S.tris_s = h->tris_s;
  S.tris = h->tris;
  S.tris_lo = h->tris_lo;
  S.leaf_off = h->leaf_off;
  S.leaf_cnt = h->leaf_cnt;
  S.pyr = h->pyramid;
  S.cell_pyr = h->cell_pyr;
  S.axis = h->axis;
  S.chi = h->chi32;
  S.st = h->dstate;
  S.cap = h->mesh_cap;
  S.n = res;
  S.nb = g.nb;
  S.h = (float)g.h * g.sc;
  S.coord = 0.f;
  for (int a = 0; a < 3; ++a)
    S.coord = std::max(S.coord, (float)std::max(fabs(g.lo[a]), fabs(g.lo[a] + res * g.h)));
  S.coord *= g.sc;
  S.sc = g.sc;
  S.us = g.us;
  S.phi = h->phi;
  S.sdf_out = sdf_out;
  S.ctri = ctri;
  S.tie_a = reinterpret_cast<int*>(h->r32);
  S.tie_b = reinterpret_cast<int*>(h->e32);
  S.tie_cd.p[0] = reinterpret_cast<int2*>(h->chiff[0]);
  S.tie_cd.p[1] = reinterpret_cast<int2*>(h->chiff[1]);
  S.tie_list = ctri ? reinterpret_cast<int*>(h->dchi64) : nullptr;
  S.defer = ctri ? S.tie_list + N : S.tie_b;
  // closest triangles of the coarser lattices, read by the finer ones as seeds
  S.seed_ids = ctri ? ctri : S.tie_a;
  static_assert(offsetof(DevState, ndefer) == offsetof(DevState, ntie) + sizeof(unsigned), "cleared together");
  WGEO_CUDA_TRY(cudaMemsetAsync(&h->dstate->ntie, 0, 2 * sizeof(unsigned), s));
  const bool count = h->opt.stage_timing == 2;
  const int threads = kWarps * 32;
  auto node_pass = [&](bool list, int stride) -> int {
    const int64_t nl = (res + stride - 1) / stride;
    const int blocks = list ? h->num_sms * 8 : grid_blocks(32 * nl * nl * nl, threads, h->num_sms * 64);
#define WGEO_NODE_PASS(C, T)                                                          \
  if (list)                                                                           \
    sdf_node_kernel<C, T, true><<<blocks, threads, 0, s>>>(S, pi, stride);            \
  else                                                                                \
    sdf_node_kernel<C, T, false><<<blocks, threads, 0, s>>>(S, pi, stride);
    if (ctri) {
      if (count) { WGEO_NODE_PASS(true, true) } else { WGEO_NODE_PASS(false, true) }
    } else {
      if (count) { WGEO_NODE_PASS(true, false) } else { WGEO_NODE_PASS(false, false) }
    }
#undef WGEO_NODE_PASS
    WGEO_LAUNCH_CHECK();
    return WGEO_OK;
  };
  // stride of the coarsest lattice.  A coarser one costs fewer searches from
  // nothing (4,300 warp instructions a node at 128^3, 7,200 at 256^3), but its
  // patch passes have too few blocks to fill the chip and boxes with many
  // candidates.  Search stage, us, star body / sphere / small sphere / points
  // that fill the box: stride 2 against 4 at 72^3 425 447 233 646 / 445 464 181
  // 734, at 80^3 595 569 325 857 / 587 555 239 929, at 96^3 981 954 577 1265 /
  // 776 858 397 1176; 4 against 8 at 160^3 2840 3279 1458 4495 / 3055 3781 1404
  // 5490, at 176^3 3745 4511 1889 5198 / 3907 4965 1831 6115, at 224^3 7744 9110
  // 4227 12161 / 7603 9827 3946 13069.  Above 160^3 the shape decides, up to 10%
  // either way (the swimming ellipsoid at 192^3 3.8 / 3.6 ms); at 256^3 11.8 /
  // 11.5 ms (star body), at 512^3 102 / 85.
  const int coarse = res < 80 ? 2 : res <= 160 ? 4 : 8;
  rc = node_pass(false, coarse);
  if (rc) return rc;
  for (int stride = coarse / 2; stride >= 1; stride /= 2) {
    const int nl = (res + stride - 1) / stride;
    const int nblk = ((nl + 7) / 8) * ((nl + 7) / 8) * ((nl + 3) / 4);
    // leaves in a block's reach above which its nodes are searched one by one:
    // cheaper in a block (a third of the instructions), but where the blocks
    // are few the longest decides.  Search stage, us, star body / sphere / two
    // shells / points that fill the box: 256 against 512 at 72^3 423 447 326 642 /
    // 405 505 328 563, at 88^3 698 717 443 1192 / 670 781 545 993, at 96^3 827 859
    // 506 1403 / 774 856 611 1170, at 128^3 1708 1919 1075 2997 / 1515 1747 1147
    // 2367; 512 against kFront at 160^3 (16,000 blocks) 2842 3285 2115 4509 / 2819
    // 3342 2419 4181, at 176^3 (21,296) 3910 5005 2719 6659 / 3816 4706 3050 6008.
    const int leaf_max = res <= 80 ? 256 : nblk <= 16384 ? 512 : kFront;
    if (ctri) {
      if (count)
        sdf_patch_kernel<true, true><<<nblk, kPatchWarps * 32, 0, s>>>(S, pi, stride, leaf_max);
      else
        sdf_patch_kernel<false, true><<<nblk, kPatchWarps * 32, 0, s>>>(S, pi, stride, leaf_max);
    } else {
      if (count)
        sdf_patch_kernel<true, false><<<nblk, kPatchWarps * 32, 0, s>>>(S, pi, stride, leaf_max);
      else
        sdf_patch_kernel<false, false><<<nblk, kPatchWarps * 32, 0, s>>>(S, pi, stride, leaf_max);
    }
    WGEO_LAUNCH_CHECK();
  }
  rc = node_pass(true, 1);
  if (rc) return rc;
  stage_end(h, kStSDF, slot, s);
  if (ctri) {
    slot = stage_begin(h, kStSDFTie, s);
    // bits of a triangle id under the default capacity of this grid (at least
    // 4096 triangles; at most 24 bits, 16 * 800^2)
    int id_bits = 13;
    while (((int64_t)1 << id_bits) - 1 < (int64_t)16 * res * res) ++id_bits;
    sdf_tie_kernel<<<152 * 8, 256, 0, s>>>(S, g, id_bits, 0);
    WGEO_LAUNCH_CHECK();
    sdf_tie_kernel<<<152 * 8, 256, 0, s>>>(S, g, id_bits, 1);
    WGEO_LAUNCH_CHECK();
    stage_end(h, kStSDFTie, slot, s);
  }
  if (nrm_out) {
    slot = stage_begin(h, kStNormals, s);
    normals_kernel<<<dim3(div_up(res, 32), div_up(res, 8), div_up(res, kNrmZ)), dim3(32, 8), 0, s>>>(
        h->phi, res, h->h, nrm_out);
    WGEO_LAUNCH_CHECK();
    stage_end(h, kStNormals, slot, s);
  }
  return WGEO_OK;
}

int launch_query_exact_chunk(wgeo_handle* h, const float* q, int nq, float* sdf_q, float* nrm_q, int* tri,
                             cudaStream_t s) {
  if (nq == 0) return WGEO_OK;
  const SurfParams g = surf_params(h, h->res);
  const PyrInfo pi = pyramid_info(2 * g.nb);
  const int* ctri = h->opt.keep_for_backward ? h->ctri : nullptr;
  // queries sorted by (cell of 8 h, sub-cell key), so that a warp's 32
  // queries lie close together
  const float box[6] = {(float)g.lo[0], (float)g.lo[1], (float)g.lo[2], (float)(g.lo[0] + g.res * g.h),
                        (float)(g.lo[1] + g.res * g.h), (float)(g.lo[2] + g.res * g.h)};
  PointGrid pg;
  int rc = build_point_grid(h, q, nq, box, 8.0 * g.h, true, nullptr, &pg, s);
  if (rc) return rc;
  const int* total = h->dp_off + pg.ncell;
  const int nblk = grid_blocks((int64_t)nq, kWarps * 32, 152 * 8);
  if (ctri)
    sdf_query_kernel<true><<<nblk, kWarps * 32, 0, s>>>(h->phi, g, h->tris, h->tris_s, h->leaf_off, h->mesh_cap, h->pyramid,
                                                        pi, h->dp_sorted, total, ctri, sdf_q, nrm_q, tri);
  else
    sdf_query_kernel<false><<<nblk, kWarps * 32, 0, s>>>(h->phi, g, h->tris, h->tris_s, h->leaf_off, h->mesh_cap,
                                                         h->pyramid, pi, h->dp_sorted, total, nullptr, sdf_q, nrm_q,
                                                         tri);
  WGEO_LAUNCH_CHECK();
  query_sign_kernel<<<grid_blocks(nq, 128, 152 * 16), 128, 0, s>>>(q, nq, h->chi32, chiff_of(h), g, h->dstate,
                                                                    sdf_q, nrm_q);
  WGEO_LAUNCH_CHECK();
  return WGEO_OK;
}

int launch_query_exact(wgeo_handle* h, const float* q, int64_t m, float* sdf_q, float* nrm_q, cudaStream_t s) {
  // in chunks the point-grid workspace can sort
  for (int64_t c0 = 0; c0 < m; c0 += h->dp_points) {
    const int nq = (int)std::min<int64_t>(h->dp_points, m - c0);
    int rc = launch_query_exact_chunk(h, q + 3 * c0, nq, sdf_q + c0, nrm_q ? nrm_q + 3 * c0 : nullptr, nullptr, s);
    if (rc) return rc;
  }
  return WGEO_OK;
}

}  // namespace wgeo
