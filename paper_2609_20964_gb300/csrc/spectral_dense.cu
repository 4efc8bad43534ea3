// Spectral correction of the adjoint solve on grids that the FFT passes do not
// take (n not a power of two, or below 32), up to dense_limit: the same direct solve of L e = r -
// mean(r) in the cosine basis (solver.cu), each one-dimensional transform as a
// dense product folded by the basis' symmetry.  The forward solves of these
// grids stay with their V-cycles: chi decides which of two nearly equidistant
// triangles a node takes, and a chi that differs by the V-cycles' own 1e-7
// moves a few such nodes to the other one.
//
// Q[k][i] = s_k cos(pi k (2 i + 1) / 2n) (orthonormal) is even in i about the
// middle of the line for even k and odd for odd k, so with s_i = x_i +
// x_{n-1-i} and d_i = x_i - x_{n-1-i} over the first half of the line
//   X_{2k}   = sum_i Q[2k][i] s_i,     X_{2k+1} = sum_i Q[2k+1][i] d_i,
// and back, with E_i = sum_k Q[2k][i] X_{2k} and O_i = sum_k Q[2k+1][i] X_{2k+1},
//   x_i = E_i + O_i,  x_{n-1-i} = E_i - O_i:
// n^2 / 2 multiply-adds per line and transform instead of n^2.  For odd n the
// middle value belongs to the even part alone (Q[odd][middle] = 0).
//
// Why dense: the sizes here are m 2^k with m <= 16, m odd or not, so an FFT
// would need radices 3, 5, 7, 11 and 13 and its shared-memory passes, while a
// product of this size is a few tens of microseconds at the FP32 rate of this
// GPU.  Bound: FP32 issue, 32 FMA per 4 shared 16-byte loads.  Adjoint solve
// (two corrections and residuals) against the V-cycles, ms: 0.20 / 0.80 at
// 88^3, 0.30 / 1.8 (unlumped operator) at 96^3, 0.30 / 1.0 at 120^3; where the
// n^4 operations catch up with the V-cycles' n^3 is dense_limit.  Line numbers
// (n^2 of them) fit 32 bits, element offsets are 64-bit.
#include "wgeo_internal.cuh"

namespace wgeo {

namespace {

constexpr int kLines = 32;       // lines per block
constexpr int kLS = 36;          // row stride of the folded tile (16-byte rows, four lines apart in the banks)
constexpr int kChunk = 8;        // reduction rows of the basis staged at a time
constexpr int kOut = 4;          // outputs of each parity per thread (times 4 lines)

__host__ __device__ constexpr int half_of(int n) { return (n + 1) / 2; }
__host__ __device__ constexpr int half_pad(int n) { return (half_of(n) + kOut - 1) / kOut * kOut; }
__host__ __device__ constexpr int red_pad(int n) { return (half_of(n) + kChunk - 1) / kChunk * kChunk; }
// a table row holds the even outputs, then the odd ones
__host__ __device__ constexpr int table_row(int n) { return 2 * half_pad(n); }

size_t tile_floats(int n) { return (size_t)2 * red_pad(n) * kLS; }
size_t smem_bytes(int n) { return sizeof(float) * (tile_floats(n) + 2 * (size_t)kChunk * table_row(n)); }

// fwd[r = i][o = k'] and inv[r = k'][o = i], zero outside the basis; sk[k] =
// 4 sin^2(pi k / 2n).
__global__ void dense_tables_kernel(int n, float* __restrict__ fwd, float* __restrict__ inv, float* __restrict__ sk) {
  const int h = half_of(n), hp = half_pad(n), rp = red_pad(n);
  const int total = rp * 2 * hp;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int r = t / (2 * hp), c = t - r * 2 * hp;
    const int odd = c >= hp ? 1 : 0, o = c - odd * hp;
    auto basis = [&](int kk, int i) {
      const int k = 2 * kk + odd;
      if (kk >= h || i >= h || k >= n || (odd && 2 * i + 1 == n)) return 0.f;
      const int m = (int)(((long long)k * (2 * i + 1)) % (4 * n));   // the angle's whole turns dropped exactly
      return (float)(sqrt((k ? 2.0 : 1.0) / n) * cospi((double)m / (2.0 * n)));
    };
    fwd[t] = basis(o, r);
    inv[t] = basis(r, o);
  }
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const double s = sinpi((double)k / (2.0 * n));
    sk[k] = (float)(4.0 * s * s);
  }
}

__device__ __forceinline__ void copy16_async(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

// acc_e / acc_o [output][line] of one thread: both parities' products over the
// whole reduction, the basis streamed through shared memory in two buffers.
// Every thread of the block calls it; those past the outputs only copy.
__device__ __forceinline__ void dense_product(const float* __restrict__ table, int n, const float* U, const float* V,
                                              float* W, int lq, int og, float (&ae)[kOut][4], float (&ao)[kOut][4]) {
  const int hp = half_pad(n), row = table_row(n), chunks = red_pad(n) / kChunk;
  const int vec = kChunk * row / 4;
  const bool mine = og * kOut < hp;
#pragma unroll
  for (int a = 0; a < kOut; ++a)
#pragma unroll
    for (int l = 0; l < 4; ++l) ae[a][l] = ao[a][l] = 0.f;
  for (int q = threadIdx.x; q < vec; q += blockDim.x) copy16_async(W + 4 * q, table + 4 * q);
  copy_commit();
  for (int c = 0; c < chunks; ++c) {
    float* cur = W + (c & 1) * kChunk * row;
    if (c + 1 < chunks) {
      float* nxt = W + ((c + 1) & 1) * kChunk * row;
      const float* src = table + (size_t)(c + 1) * kChunk * row;
      for (int q = threadIdx.x; q < vec; q += blockDim.x) copy16_async(nxt + 4 * q, src + 4 * q);
      copy_commit();
      copy_wait<1>();
    } else {
      copy_wait<0>();
    }
    __syncthreads();
    if (mine) {
#pragma unroll
      for (int r = 0; r < kChunk; ++r) {
        const int rr = c * kChunk + r;
        const float4 s = *reinterpret_cast<const float4*>(U + rr * kLS + 4 * lq);
        const float4 d = *reinterpret_cast<const float4*>(V + rr * kLS + 4 * lq);
        const float4 we = *reinterpret_cast<const float4*>(cur + r * row + kOut * og);
        const float4 wo = *reinterpret_cast<const float4*>(cur + r * row + hp + kOut * og);
        const float sl[4] = {s.x, s.y, s.z, s.w}, dl[4] = {d.x, d.y, d.z, d.w};
        const float el[4] = {we.x, we.y, we.z, we.w}, ol[4] = {wo.x, wo.y, wo.z, wo.w};
#pragma unroll
        for (int a = 0; a < kOut; ++a)
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            ae[a][l] = fmaf(el[a], sl[l], ae[a][l]);
            ao[a][l] = fmaf(ol[a], dl[l], ao[a][l]);
          }
      }
    }
    __syncthreads();   // the buffer is refilled by the next copy but one; U and V may be rewritten after the last
  }
}

// MODE 0: forward transform along `axis`; 1: its inverse; 2 (axis z): forward,
// division by the eigenvalue, inverse.  A block takes kLines lines: along x,
// consecutive rows of the grid; along y, neighbouring x columns of one plane;
// along z, consecutive positions of the flattened (x, y) plane.  `in` may be
// `out`: a block reads and writes its own lines only.
template <int MODE>
__global__ void __launch_bounds__(800) dense_pass_kernel(const float* in, float* out, int n, int axis,
                                                         const float* __restrict__ fwd,
                                                         const float* __restrict__ inv,
                                                         const float* __restrict__ sk, int q1,
                                                         const int* __restrict__ gate) {
  if (*gate) return;
  extern __shared__ float4 dsm4[];
  float* U = reinterpret_cast<float*>(dsm4);   // even part [reduction row][line]
  float* V = U + red_pad(n) * kLS;             // odd part
  float* W = V + red_pad(n) * kLS;             // two chunks of the basis
  const int h = half_of(n), rp = red_pad(n);
  const int64_t nn = (int64_t)n * n;
  const int tiles = axis == 1 ? (n + kLines - 1) / kLines : 1;
  const int fixed = axis == 1 ? blockIdx.x / tiles : 0;
  const int t0 = (axis == 1 ? blockIdx.x - fixed * tiles : blockIdx.x) * kLines;
  const int lines = (int)min((int64_t)kLines, (axis == 1 ? n : nn) - t0);
  // element i of line l: base + l * lstep + i * istep
  const int64_t base = axis == 0 ? (int64_t)t0 * n : axis == 1 ? fixed * nn + t0 : t0;
  const int64_t lstep = axis == 0 ? n : 1, istep = axis == 0 ? 1 : axis == 1 ? n : nn;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  // the tile: along y and z a warp reads rows of 32 neighbouring lines; along
  // x it reads 8 elements of 4 lines (whole sectors, all banks)
  const int i_per = axis == 0 ? 8 : 1, l_per = axis == 0 ? 4 : 32;
  const int li = axis == 0 ? (lane & 7) : 0, ll = axis == 0 ? (lane >> 3) : lane;
  const int irow = (rp + i_per - 1) / i_per, lgrp = kLines / l_per;
  for (int q = warp; q < irow * lgrp; q += nwarp) {
    const int r = (q / lgrp) * i_per + li, l = (q % lgrp) * l_per + ll;
    if (r >= rp) continue;
    float u = 0.f, v = 0.f;
    if (r < h && l < lines) {
      const float* p = in + base + l * lstep;
      if (MODE == 1) {
        u = p[(2 * r) * istep];
        if (2 * r + 1 < n) v = p[(2 * r + 1) * istep];
      } else {
        const float a = p[r * istep];
        const int m = n - 1 - r;
        if (m == r) {
          u = a;
        } else {
          const float b = p[m * istep];
          u = a + b;
          v = a - b;
        }
      }
    }
    U[r * kLS + l] = u;
    V[r * kLS + l] = v;
  }
  const int lq = threadIdx.x & 7, og = threadIdx.x >> 3;
  float ae[kOut][4], ao[kOut][4];
  dense_product(MODE == 1 ? inv : fwd, n, U, V, W, lq, og, ae, ao);
  const bool mine = og * kOut < half_pad(n);
  if (MODE == 2) {
    // divide by the eigenvalue of mode (kx, ky, kz); the zero mode (the mean) is dropped
    if (mine) {
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const int p = min(t0 + 4 * lq + l, (int)(nn - 1));
        const int ky = p / n, kx = p - ky * n;
        const float sx = sk[kx], sy = sk[ky];
        const float mx = 1.f - sx * (1.f / 6.f), my = 1.f - sy * (1.f / 6.f);
#pragma unroll
        for (int a = 0; a < kOut; ++a) {
          const int kk = og * kOut + a;
#pragma unroll
          for (int odd = 0; odd < 2; ++odd) {
            const int kz = 2 * kk + odd;
            const float sz = kz < n ? sk[kz] : 1.f;
            float lam;
            if (q1) {
              const float mz = 1.f - sz * (1.f / 6.f);
              lam = -(float)kQ1Scale * (sx * my * mz + mx * (sy * mz + my * sz));
            } else {
              lam = -(sx + sy + sz);
            }
            const bool drop = kz >= n || (kx | ky | kz) == 0;
            float& x = odd ? ao[a][l] : ae[a][l];
            x = drop ? 0.f : x / lam;
          }
        }
      }
    }
    if (mine) {
#pragma unroll
      for (int a = 0; a < kOut; ++a) {
        const int kk = og * kOut + a;
        if (kk < rp) {
          *reinterpret_cast<float4*>(U + kk * kLS + 4 * lq) = make_float4(ae[a][0], ae[a][1], ae[a][2], ae[a][3]);
          *reinterpret_cast<float4*>(V + kk * kLS + 4 * lq) = make_float4(ao[a][0], ao[a][1], ao[a][2], ao[a][3]);
        }
      }
    }
    __syncthreads();
    dense_product(inv, n, U, V, W, lq, og, ae, ao);
  }
  if (!mine) return;
  // element pairs of a thread: (2 o, 2 o + 1) of the forward transform,
  // (o, n - 1 - o) of the inverse
  if (axis == 0) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      if (4 * lq + l >= lines) break;
      float* p = out + base + (4 * lq + l) * lstep;
#pragma unroll
      for (int a = 0; a < kOut; ++a) {
        const int o = og * kOut + a;
        if (o >= h) break;
        if (MODE == 0) {
          p[2 * o] = ae[a][l];
          if (2 * o + 1 < n) p[2 * o + 1] = ao[a][l];
        } else {
          p[o] = ae[a][l] + ao[a][l];
          if (n - 1 - o != o) p[n - 1 - o] = ae[a][l] - ao[a][l];
        }
      }
    }
  } else {
    const bool vec = 4 * lq + 4 <= lines && (n & 3) == 0;
#pragma unroll
    for (int a = 0; a < kOut; ++a) {
      const int o = og * kOut + a;
      if (o >= h) break;
      const int first = MODE == 0 ? 2 * o : o, second = MODE == 0 ? 2 * o + 1 : n - 1 - o;
      const bool two = MODE == 0 ? second < n : second != o;
      float* p = out + base + 4 * lq;
      float x[4], y[4];
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        x[l] = MODE == 0 ? ae[a][l] : ae[a][l] + ao[a][l];
        y[l] = MODE == 0 ? ao[a][l] : ae[a][l] - ao[a][l];
      }
      if (vec) {
        *reinterpret_cast<float4*>(p + first * istep) = make_float4(x[0], x[1], x[2], x[3]);
        if (two) *reinterpret_cast<float4*>(p + second * istep) = make_float4(y[0], y[1], y[2], y[3]);
      } else {
#pragma unroll
        for (int l = 0; l < 4; ++l)
          if (4 * lq + l < lines) {
            p[first * istep + l] = x[l];
            if (two) p[second * istep + l] = y[l];
          }
      }
    }
  }
}

}  // namespace

// Floats of the basis and eigenvalue tables of every grid up to max_res.
size_t dense_table_floats(int max_res) {
  return 2 * (size_t)red_pad(max_res) * table_row(max_res) + (size_t)max_res;
}

// Under the caller's capture a solve's tables are part of what is captured, and
// a replay may come between any two calls, on another grid than the last one's:
// from then on every call of the handle makes its own (`held`, the grid that the
// tables are known to hold, stays -1).
int tables_for_capture(int& held, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  WGEO_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
  if (cap != cudaStreamCaptureStatusNone) held = -1;
  return WGEO_OK;
}

// The tables for n, and the shared-memory opt-in of the pass kernels (kept out
// of any capture of the handle's own).
int dense_setup(wgeo_handle* h, int n, cudaStream_t s) {
  if (!h->dense_attr) {
    const int most = (int)smem_bytes(kMaxRes);
    WGEO_CUDA_TRY(cudaFuncSetAttribute(dense_pass_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    WGEO_CUDA_TRY(cudaFuncSetAttribute(dense_pass_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    WGEO_CUDA_TRY(cudaFuncSetAttribute(dense_pass_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    h->dense_attr = true;
  }
  int rc = tables_for_capture(h->dense_n, s);
  if (rc) return rc;
  if (h->dense_n == n) return WGEO_OK;
  float* fwd = h->dense_tab;
  float* inv = fwd + (size_t)red_pad(n) * table_row(n);
  float* sk = inv + (size_t)red_pad(n) * table_row(n);
  dense_tables_kernel<<<grid_blocks((int64_t)red_pad(n) * table_row(n), 256), 256, 0, s>>>(n, fwd, inv, sk);
  WGEO_LAUNCH_CHECK();
  if (h->dense_n >= 0) h->dense_n = n;
  return WGEO_OK;
}

// e = the solution of L e = r - mean(r) (L the handle's operator), zero mean.
int dense_solve(wgeo_handle* h, int n, float* e, const float* r, const int* gate, cudaStream_t s) {
  const float* fwd = h->dense_tab;
  const float* inv = fwd + (size_t)red_pad(n) * table_row(n);
  const float* sk = inv + (size_t)red_pad(n) * table_row(n);
  const int threads = (8 * (half_pad(n) / kOut) + 31) / 32 * 32;
  const size_t smem = smem_bytes(n);
  const int rows = div_up((int64_t)n * n, kLines), cols = n * div_up(n, kLines);
  const int q1 = h->opt.galerkin ? 1 : 0;
#define WGEO_DENSE_PASS(MODE, SRC, AXIS, BLOCKS)                                                        \
  dense_pass_kernel<MODE><<<BLOCKS, threads, smem, s>>>(SRC, e, n, AXIS, fwd, inv, sk, q1, gate);       \
  WGEO_LAUNCH_CHECK();
  WGEO_DENSE_PASS(0, r, 0, rows)
  WGEO_DENSE_PASS(0, e, 1, cols)
  WGEO_DENSE_PASS(2, e, 2, rows)
  WGEO_DENSE_PASS(1, e, 1, cols)
  WGEO_DENSE_PASS(1, e, 0, rows)
#undef WGEO_DENSE_PASS
  return WGEO_OK;
}

}  // namespace wgeo
