// Gradients of the interaction energy (Sec. II.A with Eq. (EQForce)):
//   E = mu0 V Ms_t sum_i m_t(i) . grad phi_s(x_i),  phi_s = spline of (S * M_s).
// E is linear in m_s, so dE/dm_s is the transposed forward path applied to
// the target's weights, run backwards:
//   1. transposed gradient evaluation (k_adj_scatter): every coefficient node
//      collects mu0 V Ms_t m_t,a / d_a times the derivative weights of axis a
//      from the targets whose 64 taps cover it;
//   2. transposed prefilter on the whole box (k_pref_T), per axis: with the
//      mirror band matrix B of the prefilter P = B^-1, B^T = W B W^-1 for
//      W = diag(1/2, 1, ..., 1, 1/2), so P^T = W P W^-1: scale the two end
//      samples by 2, run the mirror recursion, scale the ends by 1/2;
//   3. transposed potential sum Mbar_c(j) = sum_b S_c(b - j) phibar(b): the
//      box is laid on the circular grid at its nodes (k_place), transformed by
//      the x and y forward passes, multiplied by the conjugate S spectra and
//      summed over box planes per source layer (k_zadj), and transformed back
//      by the y and x inverse passes.
// The recursion of step 2 is Unser's exact mirror-boundary one (causal start
// from the mirrored periodic extension, anticausal start in closed form).
#include <cuda_runtime.h>

#include "mm_internal.h"
#include "spline_w.cuh"

namespace mm {

// ------------------------------------------------------------------ 1. scatter
__global__ void __launch_bounds__(256) k_adj_scatter(const AdjScatterJob J) {
  __shared__ float w_s[3][12];
  __shared__ int sh_s[3];
  if (threadIdx.x < 3) {
    // the gather's split of sigma u into a whole-cell shift and weights
    const int a = threadIdx.x;
    const double su = J.sigma * J.u[a];
    const double fl = floor(su);
    bspline_w((float)(su - fl), w_s[a]);
    int sh = J.guard[a] + ((int)fl - J.U0[a]);
    const int need = (a == 0 ? J.nx : a == 1 ? J.ny : J.nz) + 3;
    if (sh < 0 || sh + need > J.r[a]) {
      atomicOr(J.err, 1);
      sh = 0x7fffffff;
    }
    sh_s[a] = sh;
  }
  __syncthreads();
  if (sh_s[0] == 0x7fffffff || sh_s[1] == 0x7fffffff || sh_s[2] == 0x7fffffff) return;
  const size_t nr = (size_t)J.r[0] * J.r[1] * J.r[2];
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nr) return;
  const int xr = (int)(idx % J.r[0]);
  const int yr = (int)((idx / J.r[0]) % J.r[1]);
  const int zr = (int)(idx / ((size_t)J.r[0] * J.r[1]));
  const size_t N = (size_t)J.nx * J.ny * J.nz;
  const float gx = J.escale * J.inv_d[0], gy = J.escale * J.inv_d[1], gz = J.escale * J.inv_d[2];
  float s = 0.f;
  for (int kz = 0; kz < 4; ++kz) {
    const int iz = zr - sh_s[2] - kz;
    if (iz < 0 || iz >= J.nz) continue;
    for (int ky = 0; ky < 4; ++ky) {
      const int iy = yr - sh_s[1] - ky;
      if (iy < 0 || iy >= J.ny) continue;
#pragma unroll
      for (int kx = 0; kx < 4; ++kx) {
        const int ix = xr - sh_s[0] - kx;
        if (ix < 0 || ix >= J.nx) continue;
        const size_t cell = ((size_t)iz * J.ny + iy) * J.nx + ix;
        const float mx = __ldg(J.m + cell), my = __ldg(J.m + N + cell), mz = __ldg(J.m + 2 * N + cell);
        s += gx * mx * w_s[0][4 + kx] * w_s[1][ky] * w_s[2][kz] +
             gy * my * w_s[0][kx] * w_s[1][4 + ky] * w_s[2][kz] +
             gz * mz * w_s[0][kx] * w_s[1][ky] * w_s[2][4 + kz];
      }
    }
  }
  J.box[((size_t)(zr + J.start[2]) * J.bdim[1] + (yr + J.start[1])) * J.bdim[0] + (xr + J.start[0])] = s;
}

cudaError_t launch_adj_scatter(const AdjScatterJob& J, cudaStream_t st) {
  const size_t nr = (size_t)J.r[0] * J.r[1] * J.r[2];
  if (nr == 0) return cudaSuccess;
  k_adj_scatter<<<(unsigned)((nr + 255) / 256), 256, 0, st>>>(J);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ 2. prefilter transpose
constexpr float kZ1a = -0.26794919243112270f;  // sqrt(3) - 2

// P^T = W P W^-1 in place on the box lines along `axis`.  A CTA brings `lines`
// of them into shared memory, sample k of line l at k (lines + 1) + l (whole
// coalesced runs from memory, consecutive banks for the recursions), and one
// thread each runs the two recursions there: straight from memory they waited
// on every load of a serial chain (75^3 box: 36 us an axis, now 14 us).
__global__ void __launch_bounds__(256) k_pref_T(float* box, int bx, int by, int bz, int axis, int lines) {
  extern __shared__ float ps[];
  const int L = axis == 0 ? bx : (axis == 1 ? by : bz);
  const size_t nlines = (size_t)bx * by * bz / L;
  const size_t l0 = (size_t)blockIdx.x * lines;
  const int nl = (int)(nlines - l0 < (size_t)lines ? nlines - l0 : (size_t)lines);
  const int pitch = lines + 1;
  // address of sample k of line l
  auto at = [&](size_t l, int k) -> size_t {
    if (axis == 0) return l * bx + k;
    if (axis == 1) return (l / bx) * ((size_t)bx * by) + l % bx + (size_t)k * bx;
    return l + (size_t)k * ((size_t)bx * by);
  };
  const int n = nl * L;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int l = axis == 0 ? i / L : i % nl, k = axis == 0 ? i % L : i / nl;
    ps[k * pitch + l] = box[at(l0 + l, k)];
  }
  __syncthreads();
  if ((int)threadIdx.x < nl) {
    float* x = ps + threadIdx.x;
    const float z = kZ1a;
    auto y = [&](int k) {  // W^-1 x: end samples doubled
      const float v = x[k * pitch];
      return (k == 0 || k == L - 1) ? 2.f * v : v;
    };
    // causal start: sum_k z^k of the mirrored periodic extension (period 2L - 2)
    const int P = 2 * L - 2;
    const int K = P < 48 ? P : 48;  // |z|^48 ~ 3e-28
    float c0 = 0.f, zk = 1.f;
    for (int k = 0; k < K; ++k) {
      const int kk = k < L ? k : P - k;
      c0 += zk * y(kk);
      zk *= z;
    }
    if (K == P) c0 /= (1.f - zk);  // zk = z^P
    // causal pass, c+ stored in place
    float cp = c0;
    float yprev_cp = 0.f;
    x[0] = cp;
    for (int k = 1; k < L; ++k) {
      const float v = y(k);
      yprev_cp = cp;
      cp = v + z * cp;
      x[k * pitch] = cp;
    }
    // anticausal pass: c-[L-1] = z / (z^2 - 1) (c+[L-1] + z c+[L-2]); c = 6 c-; W: ends halved
    float cm = z / (z * z - 1.f) * (cp + z * yprev_cp);
    x[(L - 1) * pitch] = 0.5f * 6.f * cm;
    for (int k = L - 2; k >= 0; --k) {
      cm = z * (cm - x[k * pitch]);
      x[k * pitch] = (k == 0 ? 0.5f : 1.f) * 6.f * cm;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int l = axis == 0 ? i / L : i % nl, k = axis == 0 ? i % L : i / nl;
    box[at(l0 + l, k)] = ps[k * pitch + l];
  }
}

cudaError_t launch_pref_T(float* box, const int bdim[3], cudaStream_t st) {
  for (int axis = 0; axis < 3; ++axis) {
    const int L = bdim[axis];
    if (L < 2) continue;
    const size_t nlines = (size_t)bdim[0] * bdim[1] * bdim[2] / L;
    // 32 lines a CTA, fewer when they are long (a plan's axis has at most a few thousand nodes)
    int lines = 32;
    while (lines > 1 && sizeof(float) * (size_t)(lines + 1) * L > 200 * 1024) lines /= 2;
    const size_t smem = sizeof(float) * (size_t)(lines + 1) * L;
    // one limit for every launch: a limit of each launch's own would be lowered
    // under a longer box's launch by another thread's shorter one
    cudaError_t e = allow_smem((const void*)k_pref_T, 227 * 1024);
    if (e != cudaSuccess) return e;
    k_pref_T<<<(unsigned)((nlines + lines - 1) / lines), 256, smem, st>>>(box, bdim[0], bdim[1], bdim[2], axis, lines);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ------------------------------------------------------------------ 3. place, z sum, scale
// box node (xb, yb, zb) -> grid[zb][(lo_y + yb) mod Qy][(lo_x + xb) mod Qx]
__global__ void k_place(const float* box, int bx, int by, int bz, int lo_x, int lo_y, float* grid, int Qx,
                        int Qy) {
  const size_t n = (size_t)bx * by * bz;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int xb = (int)(i % bx);
  const int yb = (int)((i / bx) % by);
  const int zb = (int)(i / ((size_t)bx * by));
  int gx = (lo_x + xb) % Qx, gy = (lo_y + yb) % Qy;
  if (gx < 0) gx += Qx;
  if (gy < 0) gy += Qy;
  grid[((size_t)zb * Qy + gy) * Qx + gx] = box[i];
}

cudaError_t launch_place(const float* box, const int bdim[3], const int box_lo[3], float* grid, int Qx, int Qy,
                         cudaStream_t st) {
  const size_t n = (size_t)bdim[0] * bdim[1] * bdim[2];
  k_place<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(box, bdim[0], bdim[1], bdim[2], box_lo[0], box_lo[1], grid,
                                                       Qx, Qy);
  return cudaGetLastError();
}

// CTA -> (kx, a chunk of 32 frequency pairs ky, Qy - ky, one per lane): the box
// planes of the chunk are staged in shared memory a block of planes at a time,
// and each warp takes kZAdjOut consecutive source layers of one component.  The
// spectra depend on the layer difference alone, so a warp reads one new plane of
// them per box plane and shifts the rest along in registers; a staged value
// serves kZAdjOut sums.  (A thread per output plane, every box plane read again
// from L2 for each: 379 us for the 64^3 cubes; now 62 us.)  The stored S_x, S_y
// are imaginary parts, S_z real; conjugation flips the imaginary ones, and S_y
// is odd in y.
constexpr int kZAdjThreads = 256;
constexpr int kZAdjOut = 8;     // source layers per warp
constexpr int kZAdjStage = 32;  // box planes staged at a time
__global__ void __launch_bounds__(kZAdjThreads) k_zadj(const ZAdjJob J) {
  __shared__ float4 zs[kZAdjStage][32];  // (in at ky, in at Qy - ky)
  const int nch = (J.kyq + 31) / 32;
  const int kx = blockIdx.x / nch;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = (blockIdx.x - kx * nch) * 32 + lane;
  const int kc = min(k, J.kyq - 1);  // lanes past the end compute the last frequency and store nothing
  const int Qy = J.Qy, nz = J.nz;
  const bool two = kc != 0 && 2 * kc != Qy;
  const int k1 = two ? Qy - kc : kc;
  const size_t pstride = (size_t)J.kxh * Qy;
  const size_t kstride = (size_t)J.kxh * J.kyq;
  const float2* in = J.in + (size_t)kx * Qy;
  const int groups = (nz + kZAdjOut - 1) / kZAdjOut;  // of one component
  // tasks (component, group of layers) in rounds of one per warp; the block
  // stages the box planes once a round
  for (int t0 = 0; t0 < 3 * groups; t0 += kZAdjThreads / 32) {
    const int task = t0 + warp;
    const bool mine = task < 3 * groups;
    const int c = mine ? task / groups : 0;
    const int j0 = mine ? (task - c * groups) * kZAdjOut : 0;
    const float* Sq = J.Sq + (size_t)c * kstride + (size_t)kx * J.kyq + kc;
    float w[kZAdjOut];  // w[j]: S at layer difference zb - (j0 + j)
    float4 acc[kZAdjOut];
#pragma unroll
    for (int j = 0; j < kZAdjOut; ++j) {
      acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      w[j] = 0.f;
    }
    // before box plane 0: the differences -1 - (j0 + j), shifted in below
    if (mine) {
#pragma unroll
      for (int j = 0; j + 1 < kZAdjOut; ++j) {
        const int p = nz - 2 - (j0 + j);
        if (p >= 0) w[j] = __ldg(Sq + (size_t)p * 3 * kstride);
      }
    }
    for (int z0 = 0; z0 < J.bz; z0 += kZAdjStage) {
      const int nzb = min(kZAdjStage, J.bz - z0);
      __syncthreads();
      for (int p = warp; p < nzb; p += kZAdjThreads / 32) {
        const float2 a = in[(size_t)(z0 + p) * pstride + kc], b = in[(size_t)(z0 + p) * pstride + k1];
        zs[p][lane] = make_float4(a.x, a.y, b.x, b.y);
      }
      __syncthreads();
      if (!mine) continue;
      // plane index of difference zb - j0 is zb - j0 + nz - 1 >= 0
      const float* s = Sq + (size_t)(z0 - j0 + nz - 1) * 3 * kstride;
#pragma unroll 4
      for (int p = 0; p < nzb; ++p) {
#pragma unroll
        for (int j = kZAdjOut - 1; j > 0; --j) w[j] = w[j - 1];
        w[0] = __ldg(s + (size_t)p * 3 * kstride);
        const float4 v = zs[p][lane];
#pragma unroll
        for (int j = 0; j < kZAdjOut; ++j) {
          acc[j].x = fmaf(w[j], v.x, acc[j].x);
          acc[j].y = fmaf(w[j], v.y, acc[j].y);
          acc[j].z = fmaf(w[j], v.z, acc[j].z);
          acc[j].w = fmaf(w[j], v.w, acc[j].w);
        }
      }
    }
    if (!mine || k >= J.kyq) continue;
#pragma unroll
    for (int j = 0; j < kZAdjOut; ++j) {
      if (j0 + j >= nz) break;
      float2* dst = J.out + (size_t)(c * nz + j0 + j) * pstride + (size_t)kx * Qy;
      const float4 a = acc[j];
      // real: S_z; else conj(i v) = -i v, with S_y negated at Qy - ky
      const float s1 = c == 1 ? -1.f : 1.f;
      dst[k] = c == 2 ? make_float2(a.x, a.y) : make_float2(a.y, -a.x);
      if (two) dst[k1] = c == 2 ? make_float2(a.z, a.w) : make_float2(s1 * a.w, -s1 * a.z);
    }
  }
}

cudaError_t launch_zadj(const ZAdjJob& J, cudaStream_t st) {
  const int grid = J.kxh * ((J.kyq + 31) / 32);
  if (grid == 0) return cudaSuccess;
  k_zadj<<<grid, kZAdjThreads, 0, st>>>(J);
  return cudaGetLastError();
}

__global__ void k_scale(const float* in, float* out, size_t n, float s) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = s * in[i];
}

cudaError_t launch_scale(const float* in, float* out, size_t n, float s, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_scale<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, out, n, s);
  return cudaGetLastError();
}

}  // namespace mm
